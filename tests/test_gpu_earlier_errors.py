"""An error that the caller left pending in the CUDA runtime is reported by the next call, from
whichever memory its views come: the call does not clear what it did not cause."""

import ctypes

import pytest
import torch

import synth
from test_gpu_call_routes import _scene

pytestmark = pytest.mark.gpu

W, H = 40, 30


@pytest.mark.parametrize("memory", ["pageable", "pinned", "device"])
def test_a_pending_error_is_reported(gpu_lib, memory):
    from paper_2104_03989_gb300 import binding as B
    from paper_2104_03989_gb300.engine import Context

    rt = ctypes.CDLL("libcudart.so.13")
    raw = torch.from_numpy(synth.sample_views(3, 0, 1, W, H).view("uint8").reshape(1, -1).copy())
    views = {"pageable": raw, "pinned": raw.pin_memory(), "device": raw.cuda()}[memory]
    ctx = Context()
    job = ctx.create_job(_scene(), frozen=True)
    want = ctx.render_reference(job, views, H, W)
    out = torch.empty_like(want)
    torch.cuda.synchronize()
    invalid_device = 101
    assert rt.cudaSetDevice(1 << 20) == invalid_device  # refused on the host; the device stays as it was
    assert rt.cudaPeekAtLastError() == invalid_device
    with pytest.raises(B.AdmsError):
        ctx.render_reference(job, views, H, W, out=out)
    assert rt.cudaGetLastError() == 0
    ctx.render_reference(job, views, H, W, out=out)
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    ctx.close()
