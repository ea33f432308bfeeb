"""The launch shape of a batch's LB steps is the one that was set or tuned."""
import json

import numpy as np
import pytest

from paper_2503_06610_gb300 import inputs as I

pytestmark = pytest.mark.gpu

SHAPES = [(2, 256), (1, 256), (2, 128), (1, 128), (4, 128), (4, 64)]  # sites per thread, threads


@pytest.fixture(scope="module")
def nh():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_06610_gb300 import nh as mod
    mod.load_library()
    return mod


def _channel(nh, dims, storage):
    nx, ny, nz = dims
    ch = nh.Channel(dict(nx=nx, ny=ny, nz=nz, walls_z=True, anchoring="homeotropic", shifted=True, tau=0.8, g=(1e-5, 0.0, 0.0),
                         K=0.005, q0=0.2, W0=0.0, dt_fd=9, precision="fp64" if storage == "f64" else "fp32", storage=storage, **I.LESLIE_ALIGN_09))
    ch.set_fields(I.tilted_director(nx, ny, nz, amplitude=0.5, seed=1))
    return ch


def _launched(nh, batch, steps, path):
    """(launches, shapes) of the batched LB kernel in a call."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]):  # a process's first one may record nothing
        torch.zeros(1, device="cuda").add_(1)
        torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        nh.batch_step(batch, steps)
        torch.cuda.synchronize()
    prof.export_chrome_trace(str(path))
    found = []
    for e in json.loads(path.read_text())["traceEvents"]:
        if e.get("cat") == "kernel" and "lb_batch_kernel" in e["name"]:
            args = e["name"].split("lb_batch_kernel<")[1].split(">")[0].split(",")
            found.append((int(args[4]), int(e["args"]["block"][0])))
    if not found:
        pytest.skip("no kernel records from the profiler")
    return len(found), set(found)


def test_tuned_shape_is_launched_in_groups(nh, tmp_path):
    """1.2 M sites of 164 bytes: three groups."""
    batch = [_channel(nh, (96, 96, 32), "f32") for _ in range(4)]
    batch[0].set_lb_variant(1)
    nh.batch_step(batch, 1)
    chosen = nh.batch_autotune(batch)
    count, shapes = _launched(nh, batch, 8, tmp_path / "t.json")
    assert count == 24
    assert shapes == {SHAPES[chosen]}


def test_shape_that_the_channel_has_already_is_set(nh, tmp_path):
    """Four channels of 2^14 sites take a shape by their joint size; set, the first one's own."""
    batch = [_channel(nh, (32, 32, 16), "f32") for _ in range(4)]
    nh.batch_step(batch, 1)
    assert _launched(nh, batch, 1, tmp_path / "a.json")[1] == {SHAPES[2]}
    batch[0].set_lb_variant(3)
    assert _launched(nh, batch, 1, tmp_path / "b.json")[1] == {SHAPES[3]}


@pytest.mark.parametrize("storage", ["f16s", "bf16s", "f64"])
def test_only_fp32_stores_step_in_groups(nh, tmp_path, storage):
    """Steps that HBM does not bound gain nothing from smaller launches: one for all channels."""
    batch = [_channel(nh, (96, 96, 32), storage) for _ in range(4)]
    nh.batch_step(batch, 1)
    assert _launched(nh, batch, 8, tmp_path / "t.json")[0] == 8
