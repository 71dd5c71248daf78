"""FP64 cluster solves whose transforms are radix-2 stages on two lanes per butterfly (GPU): counts of butterflies
that fill a warp, a part of one, and one warp and a part of the next, against the oracle; runs repeated on the
same data give the same bits."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if torch.cuda.is_available():
    from paper_1411_0330_gb300 import lsh


# C* to 1e-10 of the oracle's, the accuracy FP64 solves are held to, solves at 1e-11
@pytest.mark.parametrize("shape", [(2, 2), (2, 6), (4, 10), (16, 2), (32, 32), (64, 14), (2, 4, 8), (4, 6, 16)])
def test_solve(shape):
    d = len(shape)
    rng = np.random.default_rng(sum(shape))
    ph = rng.integers(0, 2, shape).astype(np.uint8)
    mods = np.array([np.eye(d), 6.0 * np.eye(d)])
    h = lsh.Handle(torch.from_numpy(ph).cuda(), mods, green=lsh.FILTERED)
    A, infos = h.effective(tol=1e-11)
    Ao, _ = oracle.effective(oracle.Problem(ph, mods, green=1), tol=1e-13)
    assert np.abs(A - Ao).max() < 1e-10 * np.abs(Ao).max()
    assert all(i["status"] == 0 for i in infos)
    for _ in range(20):
        assert np.array_equal(h.effective(tol=1e-11)[0], A)
