"""The buffers that render_loss's backward hands to the library hold what the library writes, whatever
the shapes of the tensors that the caller passed as latents; torch refuses those that do not fit."""

from types import SimpleNamespace

import pytest
import torch

V, H, W, DH, DW, NB = 7, 4, 8, 2, 4, 3
NEED = {"g_pos": (V, 3), "g_kd": (H, W, 4), "g_disp": (DH, DW), "g_skin_w": (V, NB)}


@pytest.mark.parametrize("pos,kd,disp,w", [
    ((V, 3), (H, W, 4), (DH, DW), (V, NB)),
    ((V - 2, 3), (H, W, 2), (1, 1), (V, 1)),
    ((1, 3), (1,), (DW, DH), (NB, V)),
    ((V * 3,), (H * W, 4), (DH * DW,), (1, V, NB)),
    ((V + 5, 3), (2 * H, W, 4), (DH, DW, 2), (V, NB, 1)),
])
def test_buffers_are_of_the_jobs_sizes(monkeypatch, pos, kd, disp, w):
    from paper_2104_03989_gb300 import autograd as AG

    stream = SimpleNamespace(cuda_stream=0)
    handed = {}
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: stream)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda d: 0, raising=False)
    monkeypatch.setattr(AG, "B", SimpleNamespace(
        adms_job_zero_gradients=lambda *a: None,
        adms_job_sizes=lambda *a: SimpleNamespace(n_verts=V, kd_h=H, kd_w=W, orm_h=1, orm_w=1, nrm_h=1, nrm_w=1, disp_h=DH,
                                                  disp_w=DW, n_bones=NB),
        adms_job_take_gradients=lambda ctx, job, scale, **buf: handed.update(buf)))
    fctx = SimpleNamespace(ctx=SimpleNamespace(ctx=None, stream=stream, backward=lambda *a, **k: None), job=0,
                           names=("pos", "kd", "disp", "w"), shapes=[torch.Size(s) for s in (pos, kd, disp, w)])
    grads = AG._RenderLoss.backward(fctx, torch.ones(()))[5:]
    assert set(handed) == set(NEED)
    for name, shape in NEED.items():
        assert handed[name].numel() == torch.Size(shape).numel() and handed[name].is_contiguous(), name
    assert [tuple(grads[k].shape) for k in (0, 2, 3)] == [NEED["g_pos"], NEED["g_disp"], NEED["g_skin_w"]]
    assert tuple(grads[1].shape) == (kd if torch.Size(kd).numel() == H * W * 4 else NEED["g_kd"])


@pytest.mark.gpu
def test_latents_of_a_wrong_shape_are_refused(gpu_lib):
    import synth
    from cases import sphere_scene
    from paper_2104_03989_gb300 import autograd as AG
    from paper_2104_03989_gb300.engine import Context

    ctx = Context()
    job = ctx.create_job(sphere_scene(3, 32, 0), loss="l2")
    lat = AG.latents(ctx, job)
    views, ref = synth.sample_views(1, 0, 1, 64, 48), torch.rand(1, 48, 64, 3, device="cuda")
    for name, bad in (("pos", lat["pos"].detach()[:5]), ("kd", lat["kd"].detach()[:, :16].contiguous())):
        with pytest.raises(RuntimeError):
            AG.render_loss(ctx, job, views, ref, {**lat, name: bad.requires_grad_(True)}).backward()
    AG.render_loss(ctx, job, views, ref, {**lat, "kd": lat["kd"].detach().view(-1, 4).requires_grad_(True)}).backward()
    torch.cuda.synchronize()
    ctx.close()
