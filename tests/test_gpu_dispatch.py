"""Choices by size: blocks launched directly or from graphs, and the default
launch shape of the LB kernel.  Every choice runs the same operations per site,
so the fields must be equal to the last bit."""
import numpy as np
import pytest

from paper_2503_06610_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nh():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_06610_gb300 import nh as mod
    mod.load_library()
    return mod


def _channel(nh, dims, **kw):
    nx, ny, nz = dims
    p = dict(nx=nx, ny=ny, nz=nz, walls_z=True, anchoring="homeotropic", shifted=True, tau=0.8, g=(1e-5, 3e-6, 0.0),
             K=0.005, q0=0.2, W0=0.0, dt_fd=4, precision="fp32", storage="f32", **I.LESLIE_ALIGN_09)
    p.update(kw)
    ch = nh.Channel(p)
    rng = np.random.Generator(np.random.PCG64(3))
    ch.set_fields(I.tilted_director(nx, ny, nz, amplitude=0.5, seed=1),
                  rng.uniform(-0.02, 0.02, size=(3, nx * ny * nz)), 1.0 + rng.uniform(-0.01, 0.01, size=nx * ny * nz))
    return ch


# the last directly launched block length, the first two replayed from graphs (an even and an odd count of steps)
@pytest.mark.parametrize("dt_fd", [11, 12, 13])
@pytest.mark.parametrize("paper_order", [False, True])
def test_blocks_with_and_without_graphs(nh, dt_fd, paper_order):
    a, b = (_channel(nh, (33, 18, 9), dt_fd=dt_fd, paper_order=paper_order) for _ in range(2))
    b.set_graphs(False)
    for steps in (2 * dt_fd + 1, 1, dt_fd - 2, 2 * dt_fd):
        a.step(steps)
        b.step(steps)
        for x, y in zip(a.get_fields(), b.get_fields()):
            assert np.array_equal(x, y)
        assert np.array_equal(a.get_populations(), b.get_populations())


# on both sides of the lines between the shapes: 32 768 sites; 1e5 sites and rows of four (16-bit stores); odd rows;
# rows of 256 sites with 4096 rows
@pytest.mark.parametrize("dims,storage", [((32, 32, 32), "f32"), ((32, 32, 33), "f32"), ((33, 32, 32), "f32"),
                                          ((33, 32, 32), "f16s"), ((64, 56, 28), "f16s"), ((64, 55, 28), "bf16s"),
                                          ((66, 50, 32), "bf16s"), ((256, 64, 64), "f16s"), ((256, 65, 63), "bf16s")])
def test_default_shape_equals_one_site_shape(nh, dims, storage):
    a, b = (_channel(nh, dims, storage=storage) for _ in range(2))
    b.set_lb_variant(1)
    for ch in (a, b):
        ch.step(9)
    for x, y in zip(a.get_fields(), b.get_fields()):
        assert np.array_equal(x, y)
    assert np.array_equal(a.get_populations(), b.get_populations())
