"""CG solves in one thread-block cluster per system (small grids) against the same solves by separate
passes (LSH_NO_CLUSTER=1) and the oracle, over what reaches them: 2D and 3D, lengths that leave CTAs
without slices or positions, odd rows and row counts, every operator, phases outside I0, indefinite
operators, voxel fields, batches, warm starts, iteration limits.

Both paths run the same recurrences with sums taken in another order: FP64 fields after the same number of
iterations agree to 1e-9 of their largest value, effective tensors to 1e-10 (FP64) and 1e-8 (mixed) of the
oracle's, iteration counts to 2 per solve."""
import numpy as np
import pytest

import oracle
from helpers import k_mu

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if torch.cuda.is_available():
    from paper_1411_0330_gb300 import lsh

KM, MUM = k_mu(1.0, 0.3)
KI, MUI = k_mu(10.0, 0.2)


def rel(a, b):
    return np.abs(np.asarray(a) - np.asarray(b)).max() / np.abs(np.asarray(b)).max()


def handles(monkeypatch, *args, **kw):
    h = lsh.Handle(*args, **kw)
    monkeypatch.setenv("LSH_NO_CLUSTER", "1")
    g = lsh.Handle(*args, **kw)
    monkeypatch.delenv("LSH_NO_CLUSTER")
    return h, g


def launches(h):
    return h.profile_read(reset=True)["launches"]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("green", [0, 1, 2])
@pytest.mark.parametrize("shape", [(32, 32), (9, 7), (35, 20), (3, 64), (6, 5, 7), (16, 4, 9), (10, 12, 14)])
def test_scalar(shape, green, precision, monkeypatch):
    d = len(shape)
    rng = np.random.default_rng(sum(shape) + green)
    ph = rng.integers(0, 3, shape).astype(np.uint8)
    ref = 0.5 * np.eye(d)
    mods = np.array([np.diag(rng.uniform(1.0, 6.0, d)), ref, np.diag(rng.uniform(1.0, 6.0, d))])  # phase 1: off I0
    h, g = handles(monkeypatch, torch.from_numpy(ph).cuda(), mods, green=green, precision=precision, ref=ref)
    launches(h), launches(g)
    A, I = h.effective(tol=1e-11)
    B, J = g.effective(tol=1e-11)
    assert launches(h) < launches(g)  # the path under test ran
    Ao, _ = oracle.effective(oracle.Problem(ph, mods, green=green, ref=ref), tol=1e-13)
    assert rel(A, Ao) < (1e-8 if precision else 1e-10), rel(A, Ao)
    assert all(i["status"] == 0 and i["relres"] <= 1e-11 for i in I)
    for a, b in zip(I, J):
        assert abs(a["iters"] - b["iters"]) <= 2 * max(1, a["outer"])


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kind", ["phase", "scale", "fraction"])
@pytest.mark.parametrize("shape,green", [((5, 7, 9), 0), ((8, 6, 10), 1), ((12, 12, 12), 1)])
def test_elastic(shape, green, kind, precision, monkeypatch):
    rng = np.random.default_rng(sum(shape) + green)
    ph = np.zeros(shape, np.uint8) if kind == "fraction" else (rng.random(shape) < 0.3).astype(np.uint8)
    mods, ref = np.array([[KM, MUM], [KI, MUI]]), np.array([0.25 * KM, 0.25 * MUM])
    kw, ok = {}, {}
    if kind != "phase":
        f = (rng.uniform(0.5, 2.0, shape) if kind == "scale" else rng.uniform(0.0, 1.0, shape)).astype(np.float32)
        kw, ok = {kind: torch.from_numpy(f).cuda()}, {"scale" if kind == "scale" else "frac": f.astype(np.float64)}
    h, g = handles(monkeypatch, torch.from_numpy(ph).cuda(), mods, physics=lsh.ELASTIC, green=green,
                   precision=precision, ref=ref, **kw)
    launches(h), launches(g)
    A, I = h.effective(tol=1e-11)
    B, J = g.effective(tol=1e-11)
    assert launches(h) < launches(g)
    Ao, _ = oracle.effective(oracle.Problem(ph, mods, physics=1, green=green, ref=ref, **ok), tol=1e-13)
    assert rel(A, Ao) < (1e-8 if precision else 1e-10), rel(A, Ao)
    for a, b in zip(I, J):
        assert a["status"] == 0 and abs(a["iters"] - b["iters"]) <= 2 * max(1, a["outer"])


def test_limit_warm_start_batch_and_indefinite(monkeypatch):
    rng = np.random.default_rng(8)
    ph = rng.integers(0, 2, (3, 20, 18)).astype(np.uint8)
    mods = np.array([np.eye(2), 10 * np.eye(2)])
    h, g = handles(monkeypatch, torch.from_numpy(ph).cuda(), mods, green=0, batch=True)
    load = np.array([0.3, -1.0])
    t1, i1 = h.solve(load, maxit=7, tol=1e-12, raise_on_fail=False)
    t2, i2 = g.solve(load, maxit=7, tol=1e-12, raise_on_fail=False)
    assert all(a["iters"] == 7 and a["status"] == lsh.ERR_NOT_CONVERGED for a in i1)
    assert rel(t1.cpu().numpy(), t2.cpu().numpy()) < 1e-9
    t3, i3 = h.solve(load, tau=t1.clone(), tol=1e-12, warm_start=True)
    t4, _ = g.solve(load, tol=1e-12)
    assert rel(t3.cpu().numpy(), t4.cpu().numpy()) < 1e-9
    again, _ = h.solve(load, tau=t1.clone(), tol=1e-12, warm_start=True)
    assert torch.equal(t3, again)
    # reference between the phases: plain CG on an indefinite operator
    k, m = handles(monkeypatch, torch.from_numpy(ph).cuda(), mods, green=0, batch=True, ref=5.5 * np.eye(2))
    A, _ = k.effective(tol=1e-10, solver=lsh.SOLVER_CG)
    B, _ = m.effective(tol=1e-10, solver=lsh.SOLVER_CG)
    assert rel(A, B) < 1e-9
