"""Iterations enqueued between two readings of the solver's state (GPU): with the default interval no more than
have run already, so that the launches of a solve stay within those of twice its iterations and one interval of
eight, also where the residual stands still at first and then drops."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if torch.cuda.is_available():
    from paper_1411_0330_gb300 import lsh


def discs(n, share):
    rng, g, x = np.random.default_rng(3), np.zeros((n, n), bool), np.arange(n) + 0.5
    while g.mean() < share:
        d = [np.minimum(np.abs(x - c), n - np.abs(x - c)) for c in rng.uniform(0, n, 2)]
        g |= d[0][:, None] ** 2 + d[1][None] ** 2 <= (n / 10) ** 2
    return g.astype(np.uint8)


@pytest.mark.parametrize("green", [0, 1, 2])
@pytest.mark.parametrize("contrast", [1e-4, 1e-2, 10.0, 1e3])
@pytest.mark.parametrize("graphs", [False, True])
def test_launches_of_a_solve(green, contrast, graphs, monkeypatch):
    monkeypatch.setenv("LSH_NO_CLUSTER", "1")
    h = lsh.Handle(torch.from_numpy(discs(64, 0.3)).cuda(), np.array([np.eye(2), contrast * np.eye(2)]), green=green)
    h.profile_read(reset=True)
    _, info = h.solve(np.array([1.0, 0.0]), tol=1e-10, graphs=graphs)
    launches = h.profile_read()["launches"]
    assert info["status"] == 0
    # six kernels an iteration, the start and the end of the solve four
    assert 6 * info["iters"] <= launches <= 6 * (2 * info["iters"] + 8) + 4
