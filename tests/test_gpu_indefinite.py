"""CG asked for on an indefinite operator (reference between the phases) with the mixed solver (GPU): its inner
iterations stay near those of FP64 CG on the same problem, over the paths that FP32 solves take (small grids,
plane and separate passes), and the effective tensor agrees to 1e-8, the accuracy the mixed solver is held to."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if torch.cuda.is_available():
    from paper_1411_0330_gb300 import lsh


def spheres(shape, share):
    rng, g = np.random.default_rng(1), np.zeros(shape, bool)
    axes = np.meshgrid(*[np.arange(n) + 0.5 for n in shape], indexing="ij", sparse=True)
    while g.mean() < share:
        d2 = 0
        for x, n in zip(axes, shape):
            a = np.abs(x - rng.uniform(0, n))
            d2 = d2 + np.minimum(a, n - a) ** 2
        g |= d2 <= max(1.5, min(shape) / 6) ** 2
    return g.astype(np.uint8)


@pytest.mark.parametrize("shape", [(32, 32), (60, 50), (16, 16, 16), (20, 24, 28), (32, 32, 32), (48, 48, 48)])
@pytest.mark.parametrize("green", [0, 1])
@pytest.mark.parametrize("contrast", [20.0, 100.0])
@pytest.mark.parametrize("scaled", [False, True])
@pytest.mark.parametrize("tune", [False, True])
def test_mixed_cg_near_fp64_cg(shape, green, contrast, scaled, tune):
    """At most twice the iterations of FP64: the mixed solver starts two or three inner solves from nothing."""
    d = len(shape)
    ph = torch.from_numpy(spheres(shape, 0.3)).cuda()
    mods, ref = np.array([np.eye(d), contrast * np.eye(d)]), 0.5 * (1.0 + contrast) * np.eye(d)
    kw = dict(green=green, ref=ref)
    if scaled:
        kw["scale"] = torch.ones(shape, dtype=torch.float32, device="cuda")
    got = []
    for precision in (lsh.FP64, lsh.MIXED):
        h = lsh.Handle(ph, mods, precision=precision, tune=tune, **kw)
        A, infos = h.effective(tol=1e-10, solver=lsh.SOLVER_CG)
        assert all(i["status"] == 0 and i["relres"] <= 1e-10 for i in infos)
        got.append((A, max(i["iters"] for i in infos)))
    assert np.abs(got[1][0] - got[0][0]).max() < 1e-8 * np.abs(got[0][0]).max()
    assert got[1][1] <= 2 * got[0][1], (got[0][1], got[1][1])
