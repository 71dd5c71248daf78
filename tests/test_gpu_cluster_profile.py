"""Counters of the per-pass timing where a solve is one launch (GPU): the iterations that are timed are those of
the solves since the last reset, also where a system has nothing left to do and its cluster returns at once."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if torch.cuda.is_available():
    from paper_1411_0330_gb300 import lsh


def handle(precision, batch=False):
    rng = np.random.default_rng(5)
    ph = rng.integers(0, 2, (12, 14, 10)).astype(np.uint8)
    if batch:
        ph = np.stack([ph, np.zeros_like(ph), np.roll(ph, 3, 0)])  # a homogeneous cell converges at once
    h = lsh.Handle(torch.from_numpy(ph).cuda(), np.array([np.eye(3), 20.0 * np.eye(3)]), green=lsh.FILTERED,
                   precision=precision, batch=batch)
    h.profile_enable(1)
    return h


@pytest.mark.parametrize("precision", [0, 1])
def test_a_solve_with_nothing_to_do_counts_nothing(precision):
    h = handle(precision)
    tau, info = h.solve(np.array([1.0, 0.0, 0.5]), tol=1e-10)
    first = h.profile_read(reset=True)
    assert first["timed_sys_iters"] == info["iters"] == first["timed_iters"]
    _, again = h.solve(np.array([1.0, 0.0, 0.5]), tau=tau.clone(), tol=1e-6, warm_start=True)
    second = h.profile_read(reset=True)
    assert again["iters"] == 0
    assert second["timed_sys_iters"] == second["timed_iters"] == 0


@pytest.mark.parametrize("precision", [0, 1])
def test_systems_that_are_done_count_nothing_in_later_steps(precision):
    h = handle(precision, batch=True)
    _, infos = h.effective(tol=1e-11)
    got = h.profile_read(reset=True)
    assert got["timed_sys_iters"] == sum(i["iters"] for i in infos)
