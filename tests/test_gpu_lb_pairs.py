"""Two LB steps in one pass (FP32 stores) against single steps, bit for bit.

A call of one step runs the single-step kernel; a longer call takes its steps in
pairs where it can.  Both collide every site with the same operations, so
populations, u, rho, n and the force must be equal to the last bit."""
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
    p = dict(nx=nx, ny=ny, nz=nz, walls_z=True, anchoring="homeotropic", shifted=True, tau=0.8, g=(1e-5, 3e-6, -2e-6),
             K=0.005, q0=0.2, W0=0.0, dt_fd=100, precision="fp32", storage="f32", **I.LESLIE_ALIGN_09)
    p.update(kw)
    ch = nh.Channel(p)
    ch.set_diag_fold(False)  # the stress kernel with the diagnostics' sums is another kernel
    rng = np.random.Generator(np.random.PCG64(3))
    n = I.tilted_director(nx, ny, nz, amplitude=0.5, seed=1)
    u = rng.uniform(-0.02, 0.02, size=(3, nx * ny * nz))
    ch.set_fields(n, u, 1.0 + rng.uniform(-0.01, 0.01, size=nx * ny * nz))
    return ch


def _state(ch):
    return [ch.get_populations(), ch.get_force(), *ch.get_fields()]


# at least 7.5e5 sites: ragged tiles in x and y, odd sizes, one and two layers, thin channels
DIMS = [(256, 128, 23), (256, 256, 64), (151, 117, 45), (131, 97, 60), (1024, 750, 1), (768, 512, 2), (33, 1000, 23),
        (9, 330, 260), (2000, 6, 64), (33, 38, 600)]


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("walls,shifted", [(True, True), (False, True), (True, False)])
def test_pairs_equal_single_steps(nh, dims, walls, shifted):
    a = _channel(nh, dims, walls_z=walls, shifted=shifted)
    b = _channel(nh, dims, walls_z=walls, shifted=shifted)
    before = a.launch_count()
    a.step(5)
    if min(dims) >= 16:
        assert a.launch_count() - before == 3, "two pairs and a single step"
    for _ in range(5):
        b.step(1)
    for x, y in zip(_state(a), _state(b)):
        assert np.array_equal(x, y)
    a.step(2)  # a pair that ends a call writes u and rho
    b.step(1)
    b.step(1)
    for x, y in zip(_state(a), _state(b)):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("dt_fd", [2, 3, 12, 17])
@pytest.mark.parametrize("paper_order", [False, True])
def test_pairs_around_fd_updates(nh, dt_fd, paper_order):
    """FD updates after an even and an odd number of steps, direct launches and graphs."""
    a = _channel(nh, (150, 101, 50), dt_fd=dt_fd, paper_order=paper_order)
    b = _channel(nh, (150, 101, 50), dt_fd=dt_fd, paper_order=paper_order)
    n = 3 * dt_fd + 2
    a.step(n)
    for _ in range(n):
        b.step(1)
    for x, y in zip(_state(a), _state(b)):
        assert np.array_equal(x, y)


def test_pair_leaves_the_diagnostics_sums(nh):
    """A call that ends on a pair: folded diagnostics equal the unfolded ones to the summation order."""
    d = []
    for fold in (True, False):
        ch = _channel(nh, (150, 101, 50), dt_fd=4)
        ch.set_diag_fold(fold)
        ch.step(4)
        d.append(ch.diagnostics())
    assert abs(d[0]["mass"] - d[1]["mass"]) <= 2e-6 * abs(d[1]["mass"])
    assert abs(d[0]["energy"] - d[1]["energy"]) <= 2e-6 * abs(d[1]["energy"])
    assert d[0]["max_u"] == pytest.approx(d[1]["max_u"], rel=1e-6) and d[0]["nonfinite"] == 0


def test_batched_pairs_and_channels_in_different_buffers(nh):
    """Batches of uneven channels; channels that reached the same step by pairs and by single steps sit in
    different population buffers and still batch together."""
    dims = [(128, 128, 48), (36, 37, 29), (97, 48, 24)]
    batch = [_channel(nh, d, dt_fd=16) for d in dims]
    alone = [_channel(nh, d, dt_fd=16) for d in dims]
    batch[0].step(4)
    for ch in batch[1:]:
        for _ in range(4):
            ch.step(1)
    nh.batch_step(batch, 38)
    for ch in alone:
        ch.step(42)
    for x, y in zip(batch, alone):
        for p, q in zip(_state(x)[:1] + _state(x)[3:], _state(y)[:1] + _state(y)[3:]):
            assert np.allclose(p, q, rtol=0, atol=1e-6)
    one, two = _channel(nh, dims[0], dt_fd=100), _channel(nh, dims[1], dt_fd=100)
    assert one.N + two.N >= 7.5e5
    nh.batch_step([one, two], 7)
    for ch, d in ((one, dims[0]), (two, dims[1])):
        ref = _channel(nh, d, dt_fd=100)
        for _ in range(7):
            ref.step(1)
        for x, y in zip(_state(ch), _state(ref)):
            assert np.array_equal(x, y)
