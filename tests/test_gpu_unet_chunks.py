"""Convolution chunks of the warm-start network: one cell alone is cut into
chunks of a plane or two, a batch into chunks of many, whose accumulators go
round the strip several times.  An output's terms are added in the same order
either way, so the forward pass must be equal to the last bit."""
import math

import numpy as np
import pytest

from paper_2503_06610_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,cells", [((64, 64, 32), 8), ((32, 48, 48), 13), ((16, 16, 128), 40), ((32, 80, 16), 20)])
def test_batches_equal_single_cells(dims, cells):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_06610_gb300 import nh
    nx, ny, nz = dims
    dev = torch.device("cuda")
    rng = np.random.default_rng(4)
    flat = I.unet_init_params(4)
    flat[-51:-3] = rng.normal(0, 0.3, size=48)  # a head large enough to move n
    f32 = lambda a: torch.tensor(np.asarray(a), dtype=torch.float32, device=dev)
    params = f32(flat)
    ansatz = f32(np.stack([I.skyrmion_tubes(nx, ny, nz, [(nx / 2 + k % 5, ny / 2)], 5.0) for k in range(cells)]))
    target = f32(np.stack([I.skyrmion_tubes(nx, ny, nz, [(nx / 2 + k % 5, ny / 2)], 3.5 + 0.1 * k) for k in range(cells)]))
    scalars = f32([[2 * math.pi / (12 + k), float(nz), 1e-5 * (k + 1)] for k in range(cells)])

    def run(sl):
        net = nh.UNet(sl.stop - sl.start, *dims)
        net.set_params(params)
        out = torch.empty_like(ansatz[sl])
        grad, loss = torch.zeros_like(params), torch.zeros(1, device=dev)
        net.forward(params, ansatz[sl].contiguous(), scalars[sl].contiguous(), out)
        net.backward(params, ansatz[sl].contiguous(), target[sl].contiguous(), grad, loss)
        torch.cuda.synchronize()
        net.status()
        return out, grad.double(), float(loss)

    out, grad, loss = run(slice(0, cells))
    one = [run(slice(k, k + 1)) for k in range(cells)]
    for k in range(cells):
        assert torch.equal(out[k], one[k][0][0])
    assert abs(loss - np.mean([o[2] for o in one])) <= 1e-5 * loss
    # The mean over the cells.  A cell's gradients are smaller by the batch, which moves their BF16 roundings where it
    # is no power of two: 2^-9 a layer and value, random over the voxels; FP32 sums of a thousand roundings.
    mean = sum(o[1] for o in one) / cells
    tol = 1e-3 if cells & (cells - 1) == 0 else 2e-2
    assert float((grad - mean).norm() / mean.norm()) < tol
