"""Shared-memory passes whose blocks take more than 48 KB (GPU): long lines along x or z with systems enough to
fill the blocks, in both precisions; the inverse x pass and the z pass hold static tables beside their tiles.
One application of each microstructure of a stack against the oracle's, and the solvers against one another."""
import numpy as np
import pytest

import oracle
from helpers import k_mu

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if torch.cuda.is_available():
    from paper_1411_0330_gb300 import lsh

SHAPES = [((600, 600), 0), ((500, 1000), 0), ((24, 20, 600), 0), ((20, 24, 500), 1), ((125, 40, 42), 1),
          ((126, 45, 40), 1), ((144, 40, 42), 1), ((600, 30, 42), 0)]


def problem(shape, physics, batch):
    d = len(shape)
    rng = np.random.default_rng(sum(shape))
    ph = rng.integers(0, 2, (batch,) * (batch > 0) + shape).astype(np.uint8)
    return ph, np.array([k_mu(1.0, 0.3), k_mu(4.0, 0.2)]) if physics else np.array([np.eye(d), 4.0 * np.eye(d)])


def rel(a, b):
    return np.abs(np.asarray(a) - np.asarray(b)).max() / np.abs(np.asarray(b)).max()


# one FP64 application to 1e-12, one FP32 application to 2e-5, as for the other passes
@pytest.mark.parametrize("shape,physics", SHAPES)
@pytest.mark.parametrize("precision", [0, 1])
def test_apply_of_a_stack(shape, physics, precision):
    ph, mods = problem(shape, physics, 6)
    h = lsh.Handle(torch.from_numpy(ph).cuda(), mods, physics=physics, green=1, precision=precision, batch=True)
    x = np.random.default_rng(1).standard_normal(h.field_shape)
    y = h.apply(torch.from_numpy(x).to(torch.float32 if precision else torch.float64).cuda()).cpu().numpy()
    for b in (0, 5):
        yo = oracle.apply(oracle.Problem(ph[b], mods, physics=physics, green=1), x[b])
        assert rel(y[b], yo) < (2e-5 if precision else 1e-12)


# C* of the mixed solver to 1e-8, the accuracy it is held to
@pytest.mark.parametrize("shape,physics", SHAPES)
def test_effective(shape, physics):
    ph, mods = problem(shape, physics, 0)
    got = []
    for precision in (lsh.FP64, lsh.MIXED):
        h = lsh.Handle(torch.from_numpy(ph).cuda(), mods, physics=physics, green=1, precision=precision)
        A, infos = h.effective(tol=1e-10)
        assert all(i["status"] == 0 and i["relres"] <= 1e-10 for i in infos)
        got.append(A)
    assert rel(got[1], got[0]) < 1e-8
