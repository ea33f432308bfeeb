"""Read-out of fields into device buffers: any subset of n, u and rho, equal to
the host read-out to the last bit."""
import numpy as np
import pytest

from paper_2503_06610_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(1, 1, 1), (7, 5, 3), (33, 17, 19)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_device_readout_equals_host_readout(dims, precision):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_06610_gb300 import nh
    nx, ny, nz = dims
    N = nx * ny * nz
    ch = nh.Channel(dict(nx=nx, ny=ny, nz=nz, walls_z=False, anchoring="none", tau=0.8, K=0.01, dt_fd=5,
                         precision=precision, **I.LESLIE_ALIGN_09))
    rng = np.random.Generator(np.random.PCG64(2))
    n = rng.normal(size=(3, N))
    ch.set_fields(n / np.linalg.norm(n, axis=0), rng.uniform(-0.02, 0.02, size=(3, N)), 1.0 + rng.uniform(-0.01, 0.01, size=N))
    host = ch.get_fields()
    for pick in range(8):
        out = [torch.full((k * N + 1,), 7.0, dtype=torch.float64, device="cuda") if pick >> i & 1 else None
               for i, k in enumerate((3, 3, 1))]
        nh.nh_get_fields(ch.ctx, *out, on_device=True)
        for o, h in zip(out, host):
            if o is not None:
                o = o.cpu().numpy()
                assert np.array_equal(o[:-1], np.asarray(h).ravel()) and o[-1] == 7.0
