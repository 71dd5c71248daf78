"""Solves whose kernels are chained by programmatic dependent launches (GPU) against the same kernels launched one
after the other (per-pass timing puts events between them): the same bits, over separate passes in both
precisions, plane passes and 2D grids, with few blocks and with many."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if torch.cuda.is_available():
    from paper_1411_0330_gb300 import lsh


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("graphs", [False, True])
@pytest.mark.parametrize("shape", [(20, 24, 28), (32, 32, 32), (40, 48, 45), (60, 50), (300, 250), (64, 64, 64)])
def test_same_bits(shape, precision, graphs, monkeypatch):
    monkeypatch.setenv("LSH_NO_CLUSTER", "1")
    d = len(shape)
    ph = (np.random.default_rng(sum(shape)).random(shape) < 0.3).astype(np.uint8)
    h = lsh.Handle(torch.from_numpy(ph).cuda(), np.array([np.eye(d), 8.0 * np.eye(d)]), precision=precision)
    load = np.arange(1.0, d + 1.0)
    chained, info = h.solve(load, tol=1e-9, graphs=graphs)
    again, _ = h.solve(load, tol=1e-9, graphs=graphs)
    h.profile_enable(1)
    apart, other = h.solve(load, tol=1e-9, graphs=False)
    assert info["iters"] == other["iters"]
    assert torch.equal(chained, apart) and torch.equal(chained, again)
