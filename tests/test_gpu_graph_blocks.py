"""Blocks replayed from graphs (12 steps and more) against blocks launched
directly: batches, and the block whose last step leaves the diagnostics' sums."""
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


def _channel(nh, dims, dt_fd, seed=1, **kw):
    nx, ny, nz = dims
    p = dict(nx=nx, ny=ny, nz=nz, walls_z=True, anchoring="homeotropic", shifted=True, tau=0.8, g=(1e-5, 3e-6, 0.0),
             K=0.005, q0=0.2, W0=0.0, dt_fd=dt_fd, precision="fp32", storage="f32", **I.LESLIE_ALIGN_09)
    p.update(kw)
    ch = nh.Channel(p)
    rng = np.random.Generator(np.random.PCG64(seed))
    ch.set_fields(I.tilted_director(nx, ny, nz, amplitude=0.5, seed=seed),
                  rng.uniform(-0.02, 0.02, size=(3, nx * ny * nz)), 1.0 + rng.uniform(-0.01, 0.01, size=nx * ny * nz))
    return ch


@pytest.mark.parametrize("dt_fd", [12, 13])
@pytest.mark.parametrize("kw", [{}, dict(storage="bf16s"), dict(precision="fp64", storage="f64")])
def test_batch_with_and_without_graphs(nh, dt_fd, kw):
    dims = [(33, 18, 9), (48, 40, 24), (64, 64, 16)]
    with_, without = ([_channel(nh, d, dt_fd, k, **kw) for k, d in enumerate(dims)] for _ in range(2))
    for ch in without:
        ch.set_graphs(False)
    for steps in (2 * dt_fd + 1, dt_fd - 1, 3 * dt_fd):
        nh.batch_step(with_, steps)
        nh.batch_step(without, steps)
    for a, b in zip(with_, without):
        for x, y in zip(a.get_fields(), b.get_fields()):
            assert np.array_equal(x, y)
        assert np.array_equal(a.get_populations(), b.get_populations())


# single steps, and pairs from 7.5e5 sites; calls of one block replay the graph with the sums from either buffer, longer
# ones end on a block that is launched directly
@pytest.mark.parametrize("dims", [(33, 18, 9), (150, 101, 50)])
@pytest.mark.parametrize("dt_fd", [12, 13, 14, 16])
def test_sums_of_replayed_blocks(nh, dims, dt_fd):
    a, b = _channel(nh, dims, dt_fd), _channel(nh, dims, dt_fd)
    b.set_diag_fold(False)
    for steps in (dt_fd, dt_fd, dt_fd, 2 * dt_fd, dt_fd, 3 * dt_fd, dt_fd + 1, dt_fd - 1, dt_fd):
        a.step(steps)
        b.step(steps)
        p, q = a.diagnostics(), b.diagnostics()
        # FP32 warp sums of 32 values, then FP64: five rounded additions
        for k in ("mass", "energy"):
            assert abs(p[k] - q[k]) <= 2e-6 * abs(q[k]), (steps, k)
        assert p["max_u"] == pytest.approx(q["max_u"], rel=1e-6)
        assert p["nonfinite"] == q["nonfinite"] == 0
