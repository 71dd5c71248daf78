"""Shared-memory FFT passes over the radices of their plans (GPU) against the oracle: lengths with every
radix 2..12 alone and in products of two and three stages, odd and even row lengths (vector widths 1, 2 and
4), grids of one z plane, caller buffers that do not start on a vector boundary.

Tolerances as for the other passes: one FP64 application to 1e-12, one FP32 application to 2e-5 of the
output's largest value."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if torch.cuda.is_available():
    from paper_1411_0330_gb300 import lsh


def rel(a, b):
    return np.abs(np.asarray(a) - np.asarray(b)).max() / np.abs(np.asarray(b)).max()


# numpy shapes: slowest axis first
SHAPES = [(7, 9, 10), (12, 14, 15), (18, 20, 21), (25, 24, 27), (28, 6, 30), (3, 35, 36), (40, 2, 42), (45, 49, 4),
          (5, 54, 50), (8, 63, 70), (2, 72, 75), (81, 3, 80), (1, 90, 84), (6, 5, 98), (2, 3, 108), (4, 112, 1),
          (105, 2, 126), (3, 144, 2), (7, 1, 150), (630, 4), (5, 343), (243, 6), (2, 600), (500, 3), (64, 96), (48, 35),
          (1, 256), (9, 1)]


@pytest.mark.parametrize("shape", SHAPES)
def test_apply_over_the_plans(shape):
    d = len(shape)
    rng = np.random.default_rng(sum(shape))
    ph = rng.integers(0, 3, shape).astype(np.uint8)
    mods = np.array([np.diag(rng.uniform(1.0, 10.0, d)) for _ in range(3)])
    for green in (0, 1, 2):
        P = oracle.Problem(ph, mods, green=green)
        x = rng.standard_normal(P.field_shape)
        yo = oracle.apply(P, x)
        h = lsh.Handle(torch.from_numpy(ph).cuda(), mods, green=green, precision=lsh.MIXED)
        assert rel(h.apply(torch.from_numpy(x).cuda()).cpu().numpy(), yo) < 1e-12, green
        assert rel(h.apply(torch.from_numpy(x).float().cuda()).cpu().numpy(), yo) < 2e-5, green


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("shape", [(6, 10), (4, 6, 12), (3, 5, 7)])
def test_unaligned_caller_buffers(shape, dtype):
    rng = np.random.default_rng(3)
    ph = rng.integers(0, 2, shape).astype(np.uint8)
    mods = np.array([np.eye(len(shape)), 4.0 * np.eye(len(shape))])
    h = lsh.Handle(torch.from_numpy(ph).cuda(), mods, green=1, precision=lsh.MIXED)
    t = torch.float32 if dtype == "f32" else torch.float64
    n = int(np.prod(h.field_shape))
    x = torch.randn(n + 1, dtype=t, device="cuda")
    y = torch.zeros(n + 1, dtype=t, device="cuda")
    xu, yu = x[1:].view(h.field_shape), y[1:].view(h.field_shape)
    h.apply(xu, out=yu)
    assert torch.equal(yu, h.apply(xu.clone()))


@pytest.mark.parametrize("shape", [(16, 16, 16), (32, 48, 48), (16, 64, 64), (128, 16, 16), (16, 128, 128)])
@pytest.mark.parametrize("kind", ["phase", "scale", "fraction"])
@pytest.mark.parametrize("green", [0, 1])
def test_elastic_apply_in_mandel_components(shape, kind, green):
    """FP32 apply whose fields stay in Mandel components (z variant 11) against the one through the internal
    basis (variant 10), two microstructures, voxels outside I0: both are the operator to FP32 rounding, each
    2e-5 of the largest value from the oracle's, and from each other by the FFT's rounding (2e-6)."""
    rng = np.random.default_rng(sum(shape) + green)
    K, mu = 0.8333, 0.3846
    ref = np.array([0.25 * K, 0.25 * mu])
    mods = np.array([[K, mu], [6.7 * K, 10.8 * mu]] if kind == "fraction" else [[K, mu], list(ref), [6.7 * K, 10.8 * mu]])
    ph = rng.integers(0, len(mods), (2,) + shape).astype(np.uint8)
    kw = {}
    if kind != "phase":
        f = rng.uniform(0.5, 2.0, ph.shape) if kind == "scale" else rng.uniform(0.0, 1.0, ph.shape)
        kw = {kind: torch.from_numpy(f.astype(np.float32)).cuda()}
    h = lsh.Handle(torch.from_numpy(ph).cuda(), mods, physics=lsh.ELASTIC, green=green, precision=lsh.MIXED, ref=ref,
                   batch=True, **kw)
    x = torch.randn(h.field_shape, dtype=torch.float32, device="cuda")
    h.set_variants(0, 0, 2, 11)
    a = h.apply(x).double()
    h.set_variants(0, 0, 2, 10)
    b = h.apply(x).double()
    assert float((a - b).abs().max()) < 2e-6 * float(b.abs().max())
