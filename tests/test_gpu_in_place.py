"""lsh_apply with y == x (GPU): the values of an apply to another buffer, bit for bit, over the passes that take
a caller's buffers directly (plane passes in Mandel components, plane and separate passes of scalar fields,
double-float, 2D) and those that go through the handle's own (rotations, buffers off the vector boundary)."""
import numpy as np
import pytest

from helpers import k_mu

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if torch.cuda.is_available():
    from paper_1411_0330_gb300 import lsh

MODS = {1: np.array([k_mu(1.0, 0.3), k_mu(10.0, 0.2)])}


def problem(shape, physics, dtype, batch, **kw):
    rng = np.random.default_rng(sum(shape) + physics)
    lead = (2,) if batch else ()
    ph = torch.from_numpy(rng.integers(0, 2, lead + shape).astype(np.uint8)).cuda()
    d = len(shape)
    mods = MODS[1] if physics else np.array([np.eye(d), 5.0 * np.eye(d)])
    h = lsh.Handle(ph, mods, physics=physics, green=lsh.FILTERED, precision=lsh.MIXED, batch=batch, **kw)
    return h, torch.from_numpy(rng.standard_normal(h.field_shape)).to(dtype).cuda()


@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("shape,physics", [((16, 16, 16), 1), ((32, 48, 48), 1), ((32, 128, 128), 1), ((16, 64, 64), 0),
                                           ((10, 12, 18), 1), ((10, 12, 18), 0), ((20, 36), 0)])
def test_apply_in_place(shape, physics, dtype, batch):
    h, x = problem(shape, physics, dtype, batch)
    want = h.apply(x)
    y = x.clone()
    h.apply(y, out=y)
    assert torch.equal(y, want)


@pytest.mark.parametrize("z", [0, 10, 11])
def test_apply_in_place_over_the_z_variants(z):
    h, x = problem((32, 32, 32), 1, torch.float32, True, max_systems=1)
    h.set_variants(0, 0, 2, z)
    want = h.apply(x)
    y = x.clone()
    h.apply(y, out=y)
    assert torch.equal(y, want)


@pytest.mark.parametrize("physics", [0, 1])
def test_double_float_apply_in_place(physics):
    h, x = problem((16, 32, 32), physics, torch.float64, False)
    want = h.apply(x, double_float=True)
    y = x.clone()
    h.apply(y, out=y, double_float=True)
    assert torch.equal(y, want)


@pytest.mark.parametrize("offset", [4, 1])
def test_elastic_apply_to_a_buffer_that_overlaps_in_part(offset):
    """Not promised, but it gave these values before the elastic fields stayed in the caller's buffers."""
    h, x = problem((16, 32, 32), 1, torch.float32, False)
    want = h.apply(x)
    both = torch.zeros(x.numel() + offset, dtype=x.dtype, device="cuda")
    xv, yv = both[:x.numel()].view(x.shape), both[offset:].view(x.shape)
    xv.copy_(x)
    h.apply(xv, out=yv)
    assert torch.equal(yv, want)
