"""Tiles of the kernel that takes two LB steps in one pass, in domains whose width
is no multiple of 32: against single steps, bit for bit."""
import numpy as np
import pytest

from paper_2503_06610_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# a tile as wide as the domain (of few and of many rows), two and three shares of the width, ragged last ones
NARROW = [(9, 330, 260), (2, 700, 540), (7, 300, 400), (16, 512, 128), (33, 38, 600), (47, 131, 131), (64, 64, 200),
          (65, 200, 64), (70, 71, 160), (100, 100, 80), (131, 97, 60)]


@pytest.fixture(scope="module")
def nh():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_06610_gb300 import nh as mod
    mod.load_library()
    return mod


def _channel(nh, dims, walls=True, seed=3):
    nx, ny, nz = dims
    ch = nh.Channel(dict(nx=nx, ny=ny, nz=nz, walls_z=walls, anchoring="homeotropic", shifted=True, tau=0.8,
                         g=(1e-5, 3e-6, -2e-6), K=0.005, q0=0.2, W0=0.0, dt_fd=100, precision="fp32", storage="f32",
                         **I.LESLIE_ALIGN_09))
    rng = np.random.Generator(np.random.PCG64(seed))
    N = nx * ny * nz
    n = rng.normal(size=(3, N)) * 0.1
    n[2] += 1.0
    ch.set_fields(n / np.linalg.norm(n, axis=0), rng.uniform(-0.02, 0.02, size=(3, N)), 1.0 + rng.uniform(-0.01, 0.01, size=N))
    return ch


def _equal(a, b):
    for x, y in zip(a.get_fields(), b.get_fields()):
        assert np.array_equal(x, y)
    assert np.array_equal(a.get_populations(), b.get_populations())


@pytest.mark.parametrize("dims", NARROW)
@pytest.mark.parametrize("walls", [True, False])
def test_narrow_domains_equal_single_steps(nh, dims, walls):
    a, b = _channel(nh, dims, walls), _channel(nh, dims, walls)
    before = a.launch_count()
    a.step(5)
    assert a.launch_count() - before == 3
    for _ in range(5):
        b.step(1)
    _equal(a, b)
    assert a.diagnostics()["mass"] == pytest.approx(b.diagnostics()["mass"], rel=2e-6)
    a.step(2)  # a pair that ends a call leaves the diagnostics' sums
    b.step(1)
    b.step(1)
    _equal(a, b)
    assert a.diagnostics()["mass"] == pytest.approx(b.diagnostics()["mass"], rel=2e-6)


def test_tiles_of_different_widths_in_one_launch(nh):
    dims = [(9, 330, 260), (128, 128, 48), (47, 131, 131), (256, 64, 47)]
    batch = [_channel(nh, d, seed=k) for k, d in enumerate(dims)]
    before = batch[0].launch_count()
    nh.batch_step(batch, 4)
    assert batch[0].launch_count() - before == 2, "two pairs of all channels"
    nh.batch_step(batch, 3)
    for k, d in enumerate(dims):
        one = _channel(nh, d, seed=k)
        for _ in range(7):
            one.step(1)
        _equal(batch[k], one)


def test_thin_channels_take_single_steps(nh):
    ch = _channel(nh, (1024, 750, 1))
    before = ch.launch_count()
    ch.step(4)
    assert ch.launch_count() - before == 4
