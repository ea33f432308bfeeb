"""A batch that is stepped in groups of channels (too large for L2 together)
against its channels stepped alone: every site sees the same operations in the
same order, so all fields are equal to the last bit, at whatever step a call
ends."""
import numpy as np
import pytest

from paper_2503_06610_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _channel(nh, k, dt_fd, **kw):
    nx, ny, nz = [(96, 96, 32), (48, 40, 24), (64, 64, 16), (33, 47, 21)][k % 4]
    p = dict(nx=nx, ny=ny, nz=nz, walls_z=True, anchoring="homeotropic", shifted=True, tau=0.8, g=(1e-5, 3e-6, 0.0),
             K=0.005, q0=0.2, W0=0.0, dt_fd=dt_fd, precision="fp32", storage="f32", **I.LESLIE_ALIGN_09)
    p.update(kw)
    ch = nh.Channel(p)
    rng = np.random.Generator(np.random.PCG64(k))
    ch.set_fields(I.tilted_director(nx, ny, nz, amplitude=0.5, seed=k),
                  rng.uniform(-0.02, 0.02, size=(3, nx * ny * nz)), 1.0 + rng.uniform(-0.01, 0.01, size=nx * ny * nz))
    return ch


# two groups and more; a block too short to be cut; blocks that a call leaves half done
@pytest.mark.parametrize("count,dt_fd,kw", [(9, 5, {}), (24, 16, {}), (10, 1, {}), (18, 6, dict(storage="f16s")),
                                            (6, 4, dict(precision="fp64", storage="f64"))])
def test_groups_equal_single_channels(count, dt_fd, kw):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_06610_gb300 import nh
    batch = [_channel(nh, k, dt_fd, **kw) for k in range(count)]
    for steps in (dt_fd + 3, 1, 2 * dt_fd + 1):
        nh.batch_step(batch, steps)
    for k in range(count):
        one = _channel(nh, k, dt_fd, **kw)
        one.step(3 * dt_fd + 5)
        for x, y in zip(batch[k].get_fields(), one.get_fields()):
            assert np.array_equal(x, y)
        assert np.array_equal(batch[k].get_populations(), one.get_populations())
