"""A context on a stream of its own beside torch's current one: every call of the autograd front is
ordered after what torch's stream has been given (the caller's writes to the latents, the memory of
the outputs) and torch's stream after the call."""

from types import SimpleNamespace

import pytest
import torch

import synth
from cases import rel_l2, sphere_scene


class _Stream:
    def __init__(self, handle, log):
        self.cuda_stream, self.log = handle, log

    def wait_stream(self, other):
        self.log.append((self.cuda_stream, "waits for", other.cuda_stream))


@pytest.mark.parametrize("call", ["invalidate", "laplacian"])
@pytest.mark.parametrize("own", [True, False])
@pytest.mark.parametrize("recording", [False, True])
def test_calls_are_ordered_with_torchs_stream(monkeypatch, call, own, recording):
    from paper_2104_03989_gb300 import autograd as AG

    log, kept = [], []
    here = _Stream(1, log)
    there = _Stream(2, log) if own else here
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: here)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda d: here.cuda_stream, raising=False)
    monkeypatch.setattr(AG, "_recording", lambda s: recording and s is there, raising=False)
    monkeypatch.setattr(torch.Tensor, "record_stream", lambda t, s: kept.append((t.shape, s.cuda_stream)))
    note = lambda *a: log.append("call")   # noqa: E731
    monkeypatch.setattr(AG, "B", SimpleNamespace(adms_job_invalidate=note, adms_laplacian=note))
    ctx = SimpleNamespace(ctx=None, stream=there)
    if call == "invalidate":
        AG.invalidate(ctx, 0)
    else:
        AG.laplacian(ctx, 0, torch.zeros(5, 3, requires_grad=True))
    # nothing can wait for a stream that is recording, nor for itself
    apart = own and not recording
    assert log == ([(2, "waits for", 1), "call", (1, "waits for", 2)] if apart else ["call"])
    assert kept == ([(torch.Size([]), 2), (torch.Size([5, 3]), 2)] if apart and call == "laplacian" else [])


def _optimize(ctx, steps=4):
    """a caller's own loop: render loss and Laplacian, a late in-place update, the job told of it"""
    from paper_2104_03989_gb300 import autograd as AG

    job = ctx.create_job(sphere_scene(3, 32, 0), loss="l2")
    views = synth.sample_views(1, 0, 2, 64, 48)
    ref = torch.rand(2, 48, 64, 3, generator=torch.Generator().manual_seed(0)).cuda()
    lat = AG.latents(ctx, job)
    torch.cuda.synchronize()
    losses = []
    for _ in range(steps):
        loss = AG.render_loss(ctx, job, views, ref, lat) + 0.1 * AG.laplacian(ctx, job, lat["pos"])
        losses.append(loss.detach() * 1.0)
        grads = torch.autograd.grad(loss, list(lat.values()))
        torch.cuda._sleep(2_000_000)  # about a millisecond
        with torch.no_grad():
            for t, g in zip(lat.values(), grads):
                t -= 0.05 * g / g.abs().max()
        AG.invalidate(ctx, job)
    torch.cuda.synchronize()
    return torch.stack(losses).cpu(), {k: t.detach().cpu().clone() for k, t in lat.items()}


@pytest.mark.gpu
def test_a_loop_on_two_streams_equals_one_on_one(gpu_lib):
    """4 steps with the same float32 arithmetic; the texels' sums differ in order (1e-7 a step, divided by the
    largest): 1e-5 with room."""
    from paper_2104_03989_gb300.engine import Context

    results = []
    for stream in (None, torch.cuda.Stream()):
        ctx = Context(stream=stream)
        results.append(_optimize(ctx))
        ctx.close()
    (la, a), (lb, b) = results
    assert rel_l2(lb, la) < 1e-5 and len(set(la.tolist())) == len(la)
    for k in a:
        assert rel_l2(b[k], a[k]) < 1e-5, k


@pytest.mark.gpu
def test_invalidate_records_into_a_contexts_graph(gpu_lib):
    from paper_2104_03989_gb300 import autograd as AG
    from paper_2104_03989_gb300 import binding as B
    from paper_2104_03989_gb300.engine import Context

    ctx = Context(stream=torch.cuda.Stream())
    job = ctx.create_job(sphere_scene(3, 32, 0), loss="l2")
    views = torch.from_numpy(synth.sample_views(1, 0, 2, 64, 48).view("uint8").reshape(2, -1).copy()).cuda()
    ref = torch.rand(2, 48, 64, 3, generator=torch.Generator().manual_seed(0)).cuda()
    loss = torch.zeros(1, device="cuda")
    ctx.reserve(job, 2, 48, 64)
    pos = ctx.params(job)["pos"]
    torch.cuda.synchronize()
    B.adms_graph_begin(ctx.ctx)
    AG.invalidate(ctx, job)  # torch's current stream is another and records nothing
    B.adms_forward_loss(ctx.ctx, [job], views, [2], [(48, 64)], [ref], loss)
    g = B.adms_graph_end(ctx.ctx)
    B.adms_graph_launch(ctx.ctx, g)
    torch.cuda.synchronize()
    before = float(loss)
    pos *= 1.1
    torch.cuda.synchronize()
    B.adms_graph_launch(ctx.ctx, g)
    torch.cuda.synchronize()
    want = ctx.forward_loss([job], [views], [ref])
    torch.cuda.synchronize()
    assert float(loss) != before and float(loss) == pytest.approx(float(want[0]), rel=1e-6)
    B.adms_graph_destroy(g)
    ctx.close()
