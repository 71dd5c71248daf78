"""The register inverse x passes with the CG update of z in them (GPU) against the oracle's solutions: every
length, both block sizes, phases outside I0, per-voxel scale fields, tabulated and finite-difference operators."""
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


# C* tolerance 1e-8, the accuracy the mixed solver is held to, solves at 1e-11
@pytest.mark.parametrize("variant", [1, 3])
@pytest.mark.parametrize("shape", [(8, 16, 16), (8, 16, 32), (4, 16, 64), (4, 8, 128), (2, 8, 256), (16, 8, 256)])
def test_elastic_with_voxels_outside_I0(shape, variant):
    rng = np.random.default_rng(sum(shape))
    ph = rng.integers(0, 3, shape).astype(np.uint8)
    ref = np.array([0.5 * KM, 0.5 * MUM])
    mods = np.array([[KM, MUM], list(ref), [KI, MUI]])
    h = lsh.Handle(torch.from_numpy(ph).cuda(), mods, physics=lsh.ELASTIC, green=lsh.FILTERED, precision=lsh.MIXED,
                   ref=ref)
    h.set_variants(0, variant, 0, 0)
    A, infos = h.effective(tol=1e-11)
    Ao, _ = oracle.effective(oracle.Problem(ph, mods, physics=1, green=1, ref=ref), tol=1e-13)
    assert all(i["status"] == 0 and i["relres"] <= 1e-11 for i in infos)
    assert rel(A, Ao) < 1e-8, rel(A, Ao)


@pytest.mark.parametrize("variant", [1, 3])
@pytest.mark.parametrize("shape,green", [((8, 16, 16), 0), ((8, 16, 64), 2), ((8, 16, 256), 1), ((128, 128), 1)])
@pytest.mark.parametrize("scaled", [False, True])
def test_scalar(shape, green, scaled, variant):
    d = len(shape)
    rng = np.random.default_rng(sum(shape) + green)
    ph = rng.integers(0, 2, shape).astype(np.uint8)
    mods = np.array([np.diag(rng.uniform(1.0, 6.0, d)) for _ in range(2)])
    f = rng.uniform(0.5, 2.0, shape).astype(np.float32)
    ref = 0.25 * np.eye(d)
    h = lsh.Handle(torch.from_numpy(ph).cuda(), mods, green=green, precision=lsh.MIXED, ref=ref,
                   scale=torch.from_numpy(f).cuda() if scaled else None)
    h.set_variants(0, variant, 0, 0)
    A, infos = h.effective(tol=1e-11)
    kw = {"scale": f.astype(np.float64)} if scaled else {}
    Ao, _ = oracle.effective(oracle.Problem(ph, mods, green=green, ref=ref, **kw), tol=1e-13)
    assert all(i["status"] == 0 and i["relres"] <= 1e-11 for i in infos)
    assert rel(A, Ao) < 1e-8, rel(A, Ao)
