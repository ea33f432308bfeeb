"""Batches that mix channels which take their LB steps in pairs (7.5e5 sites or
more) with channels which take them one by one, and batches of paired channels
only, against the channels stepped alone: equal to the last bit.

Pairs and single steps change the population buffer at different rates, so that
after a block the channels of a mixed batch sit in different buffers wherever
the block's length mod 4 is 2 or 3."""
import numpy as np
import pytest

from paper_2503_06610_gb300 import inputs as I

pytestmark = pytest.mark.gpu

LARGE, SMALL = (128, 128, 48), (96, 96, 32)


@pytest.fixture(scope="module")
def nh():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_06610_gb300 import nh as mod
    mod.load_library()
    return mod


def _channel(nh, dims, dt_fd, seed):
    nx, ny, nz = dims
    ch = nh.Channel(dict(nx=nx, ny=ny, nz=nz, walls_z=True, anchoring="homeotropic", shifted=True, tau=0.8,
                         g=(1e-5, 3e-6, 0.0), K=0.005, q0=0.2, W0=0.0, dt_fd=dt_fd, precision="fp32", storage="f32",
                         **I.LESLIE_ALIGN_09))
    ch.set_diag_fold(False)  # the stress kernel with the diagnostics' sums is another kernel
    rng = np.random.Generator(np.random.PCG64(seed))
    ch.set_fields(I.tilted_director(nx, ny, nz, amplitude=0.5, seed=seed),
                  rng.uniform(-0.02, 0.02, size=(3, nx * ny * nz)), 1.0 + rng.uniform(-0.01, 0.01, size=nx * ny * nz))
    return ch


def _equal_alone(nh, batch, dims, dt_fd, steps):
    for k, d in enumerate(dims):
        one = _channel(nh, d, dt_fd, k)
        one.step(steps)
        for x, y in zip(batch[k].get_fields(), one.get_fields()):
            assert np.array_equal(x, y), (k, d)
        assert np.array_equal(batch[k].get_populations(), one.get_populations()), (k, d)


# lengths of all remainders mod 4 that graphs replay (12 and more), and one that is launched directly
@pytest.mark.parametrize("dt_fd", [6, 12, 13, 14, 15, 18])
@pytest.mark.parametrize("at", [0, 2, 3])
@pytest.mark.parametrize("graphs", [True, False])
def test_mixed_batch_equals_single_channels(nh, dt_fd, at, graphs):
    dims = [SMALL] * 3
    dims.insert(at, LARGE)
    batch = [_channel(nh, d, dt_fd, k) for k, d in enumerate(dims)]
    for ch in batch:
        ch.set_graphs(graphs)
    # blocks from every buffer that whole blocks lead to, then from those that a remainder leaves
    calls = [3 * dt_fd, dt_fd + 1, dt_fd - 1, 1, 2 * dt_fd - 1, 2 * dt_fd + 2]
    for steps in calls:
        nh.batch_step(batch, steps)
    _equal_alone(nh, batch, dims, dt_fd, sum(calls))


@pytest.mark.parametrize("dt_fd", [5, 14])
@pytest.mark.parametrize("dims", [[LARGE, (151, 117, 45)], [(131, 97, 60), LARGE, (151, 117, 45)] * 3])
def test_paired_channels_in_one_launch(nh, dt_fd, dims):
    batch = [_channel(nh, d, dt_fd, k) for k, d in enumerate(dims)]
    before = batch[0].launch_count()
    nh.batch_step(batch, 4)
    assert batch[0].launch_count() - before == 2, "two pairs of all channels"
    for steps in (dt_fd - 4, 2 * dt_fd, dt_fd + 3):
        nh.batch_step(batch, steps)
    _equal_alone(nh, batch, dims, dt_fd, 4 * dt_fd + 3)


def test_channels_in_different_buffers(nh):
    """Two steps as a pair and two single ones leave the state in different buffers; the channels still batch."""
    dims = [LARGE, LARGE, SMALL]
    batch = [_channel(nh, d, 12, k) for k, d in enumerate(dims)]
    batch[0].step(2)
    for ch in batch[1:]:
        ch.step(1)
        ch.step(1)
    for steps in (10, 24, 25):
        nh.batch_step(batch, steps)
    _equal_alone(nh, batch, dims, 12, 61)
