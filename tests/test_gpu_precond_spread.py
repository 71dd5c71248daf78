"""Where (A - A0)^{-1} spreads far (GPU): the preconditioned CG iterations against iterations without one, on
media with many values of M (random volume fractions, graded phases, stiffness factors evenly spaced in their
inverse) and on two phases of extreme contrast.  The yardsticks are MINRES (never preconditioned, the same
Krylov space as plain CG) and FP64 CG on phase maps (plain); the mixed solver reaches 1e-10 in refinement steps
whose inner solves start from nothing, worth up to half as many iterations again and some eight a step."""
import numpy as np
import pytest

from helpers import k_mu

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if torch.cuda.is_available():
    from paper_1411_0330_gb300 import lsh

SHAPES = [(64, 64), (20, 24, 28), (16, 16, 16)]


def most(infos):
    assert all(i["status"] == 0 and i["relres"] <= 1e-10 for i in infos)
    return max(i["iters"] for i in infos)


def field(shape, kind, contrast):
    u = np.random.default_rng(sum(shape)).random(shape)
    f = u if kind == "fraction" else 1.0 / (1.0 + (contrast - 1.0) * u)
    return {kind: torch.from_numpy(f.astype(np.float32)).cuda()}


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("green", [0, 1, 2])
@pytest.mark.parametrize("kind", ["fraction", "scale"])
@pytest.mark.parametrize("contrast", [10.0, 1e3])
def test_voxel_fields(shape, green, kind, contrast):
    d = len(shape)
    ph = torch.zeros(shape, dtype=torch.uint8, device="cuda")
    mods = np.array([np.eye(d), contrast * np.eye(d)]) if kind == "fraction" else np.array([contrast * np.eye(d)])
    kw = dict(green=green, ref=0.25 * np.eye(d), **field(shape, kind, contrast))
    h = lsh.Handle(ph, mods, precision=lsh.FP64, **kw)
    plain = most(h.effective(tol=1e-10, solver=lsh.SOLVER_MINRES)[1])
    assert most(h.effective(tol=1e-10)[1]) <= plain
    assert most(lsh.Handle(ph, mods, precision=lsh.MIXED, **kw).effective(tol=1e-10)[1]) <= 1.5 * plain + 16


def phase_map_counts(ph, mods, green):
    return [most(lsh.Handle(torch.from_numpy(ph).cuda(), mods, green=green, precision=p).effective(tol=1e-10)[1])
            for p in (lsh.FP64, lsh.MIXED)]


@pytest.mark.parametrize("shape", SHAPES[:2])
@pytest.mark.parametrize("green", [0, 2])
@pytest.mark.parametrize("phases,contrast", [(2, 10.0), (2, 1e3), (3, 1e3), (16, 1e3), (64, 1e4)])
def test_phase_maps(shape, green, phases, contrast):
    d = len(shape)
    ph = np.random.default_rng(phases).integers(0, phases, shape).astype(np.uint8)
    inv = np.linspace(1.0, 1.0 / contrast, phases)  # even steps in the resistivity
    count = phase_map_counts(ph, np.array([np.eye(d) / v for v in inv]), green)
    assert count[1] <= 1.5 * count[0] + 16, count


@pytest.mark.parametrize("contrast", [1e4, 1e5, 1e6])
@pytest.mark.parametrize("share", [0.05, 0.3])
def test_stiff_voxels_under_finite_differences(contrast, share):
    ph = (np.random.default_rng(2).random((64, 64)) < share).astype(np.uint8)
    count = phase_map_counts(ph, np.array([np.eye(2), contrast * np.eye(2)]), lsh.FD)
    assert count[1] <= 1.5 * count[0] + 16, count


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("cluster", [False, True])
def test_scale_fields_that_follow_one_another(precision, cluster, monkeypatch):
    """A handle whose scale field goes from a narrow one to a wide one and back solves as new handles do."""
    if not cluster:
        monkeypatch.setenv("LSH_NO_CLUSTER", "1")
    shape = (12, 14, 10)
    ph = torch.zeros(shape, dtype=torch.uint8, device="cuda")
    fields = [field(shape, "scale", c)["scale"] for c in (2.0, 1e3, 2.0)]
    mods, kw = np.array([4.0 * np.eye(3)]), dict(green=lsh.TRUNCATED, precision=precision, ref=1e-3 * np.eye(3))
    h = lsh.Handle(ph, mods, scale=fields[0], **kw)
    for f in fields:
        h.set_microstructure(ph, f)
        got, infos = h.effective(tol=1e-9)
        want, fresh = lsh.Handle(ph, mods, scale=f, **kw).effective(tol=1e-9)
        assert np.array_equal(got, want)
        assert [i["iters"] for i in infos] == [i["iters"] for i in fresh]


@pytest.mark.parametrize("share,contrast", [(0.7, 1e-2), (0.7, 1e-3), (0.3, 1e3)])
@pytest.mark.parametrize("green", [0, 1])
def test_elastic_voxels_of_two_kinds(share, contrast, green):
    ph = (np.random.default_rng(2).random((16, 16, 16)) < share).astype(np.uint8)
    mods = np.array([k_mu(1.0, 0.3), k_mu(contrast, 0.2)])
    count = [most(lsh.Handle(torch.from_numpy(ph).cuda(), mods, physics=lsh.ELASTIC, green=green,
                             precision=p).effective(tol=1e-10)[1]) for p in (lsh.FP64, lsh.MIXED)]
    assert count[1] <= 1.2 * count[0] + 16, count


def spheres(shape, share):
    rng, g = np.random.default_rng(3), np.zeros(shape, bool)
    axes = np.meshgrid(*[np.arange(n) + 0.5 for n in shape], indexing="ij", sparse=True)
    while g.mean() < share:
        d2 = 0
        for x, n in zip(axes, shape):
            a = np.abs(x - rng.uniform(0, n))
            d2 = d2 + np.minimum(a, n - a) ** 2
        g |= d2 <= (min(shape) / 6) ** 2
    return g.astype(np.uint8)


@pytest.mark.parametrize("shape", [(8, 64, 64), (24, 20, 60), (16, 32, 64), (200, 30)])
@pytest.mark.parametrize("contrast", [10.0, 1e-3])
def test_filtered_operator_on_boxes_of_unequal_lengths(shape, contrast):
    d = len(shape)
    mods = np.array([np.eye(d), contrast * np.eye(d)])
    count = phase_map_counts(spheres(shape, 0.3), mods, lsh.FILTERED)
    assert count[1] <= 1.2 * count[0] + 16, count
