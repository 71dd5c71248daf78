"""Elasticity on grids of one z layer (GPU): the mixed solver, whose z pass leaves (p, Gamma p) block by block of
its shared-memory tiles there, against FP64 CG on the same problem and, on a small grid, the oracle.  The grids
reach from one tile per row to more blocks than any other pass has."""
import numpy as np
import pytest

import oracle
from helpers import k_mu

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if torch.cuda.is_available():
    from paper_1411_0330_gb300 import lsh

MODS = np.array([k_mu(1.0, 0.3), k_mu(10.0, 0.2)])


def effective(ph, green, precision, **kw):
    h = lsh.Handle(torch.from_numpy(ph).cuda(), MODS, physics=lsh.ELASTIC, green=green, precision=precision, **kw)
    A, infos = h.effective(tol=1e-10)
    assert all(i["status"] == 0 and i["relres"] <= 1e-10 for i in infos)
    return A


# C* of the mixed solver to 1e-8, the accuracy it is held to
@pytest.mark.parametrize("shape,systems", [((1, 30, 12), 0), ((1, 96, 600), 0), ((1, 256, 256), 0), ((1, 256, 256), 1),
                                           ((1, 300, 250), 4), ((1, 600, 600), 0)])
@pytest.mark.parametrize("green", [0, 1])
def test_mixed_against_fp64(shape, systems, green, monkeypatch):
    monkeypatch.setenv("LSH_NO_CLUSTER", "1")
    ph = (np.random.default_rng(sum(shape) + green).random(shape) < 0.3).astype(np.uint8)
    A = effective(ph, green, lsh.MIXED, max_systems=systems)
    B = effective(ph, green, lsh.FP64)
    assert np.abs(A - B).max() < 1e-8 * np.abs(B).max()
    if ph.size < 1000:
        Ao, _ = oracle.effective(oracle.Problem(ph, MODS, physics=1, green=green), tol=1e-12)
        assert np.abs(A - Ao).max() < 1e-8 * np.abs(Ao).max()
