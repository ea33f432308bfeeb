"""Director relaxation: the tiled kernel for a fluid at rest, alone and in
batches (which alternate their buffers), against the per-site kernels."""
import numpy as np
import pytest

from paper_2503_06610_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# tile edges and remainders in x and y, one and few layers, a column longer than a chunk
DIMS = [(64, 32, 16), (33, 17, 9), (31, 9, 70), (70, 65, 3), (16, 12, 1), (7, 5, 33)]


@pytest.fixture(scope="module")
def nh():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_06610_gb300 import nh as mod
    mod.load_library()
    return mod


def _channel(nh, dims, precision, walls, anchoring, seed=1):
    nx, ny, nz = dims
    ch = nh.Channel(dict(nx=nx, ny=ny, nz=nz, walls_z=walls, anchoring=anchoring, shifted=True, tau=0.8, g=(1e-5, 0.0, 0.0),
                         K=0.01, q0=0.3, W0=0.002, dt_fd=3, precision=precision, storage="f64" if precision == "fp64" else "f32",
                         **I.LESLIE_ALIGN_09))
    rng = np.random.Generator(np.random.PCG64(seed))
    ch.set_fields(I.tilted_director(nx, ny, nz, amplitude=0.5, seed=seed),
                  rng.uniform(-0.02, 0.02, size=(3, nx * ny * nz)), np.ones(nx * ny * nz))
    return ch


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("walls,anchoring", [(True, "homeotropic"), (True, "none"), (False, "none")])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_relaxation_equals_per_site_kernels(nh, dims, walls, anchoring, precision):
    # a step rounds a unit director a few times and the flow does not amplify: 4 units in the last place a stage,
    # two stages, at most 8 steps; the LB steps afterwards see forces of that accuracy
    eps = 2.0 ** -53 if precision == "fp64" else 2.0 ** -24
    tol = 4 * 2 * 8 * eps * 2
    ref = _channel(nh, dims, precision, walls, anchoring)
    ref.set_fd_variant(0)
    one = _channel(nh, dims, precision, walls, anchoring)
    batch = [_channel(nh, dims, precision, walls, anchoring, seed) for seed in (1, 2)]
    for steps in (1, 2, 5):
        ref.relax(steps)
        one.relax(steps)
        nh.batch_relax(batch, steps)
        a, b, c = ref.get_fields(), one.get_fields(), batch[0].get_fields()
        assert np.max(np.abs(a[0] - b[0])) <= tol
        assert np.array_equal(b[0], c[0])
        for f in (a, b, c):
            assert np.max(np.abs(f[1])) == 0.0
    # the buffers are where the next step expects them
    for ch in (ref, one, batch[0]):
        ch.step(4)
    a, b, c = ref.get_fields(), one.get_fields(), batch[0].get_fields()
    assert np.max(np.abs(a[0] - b[0])) <= 2 * tol
    assert np.max(np.abs(a[1] - b[1])) <= tol
    assert np.array_equal(b[0], c[0]) and np.array_equal(b[1], c[1])
