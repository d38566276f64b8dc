"""A backward recorded on its own accumulates once per replay: nothing of it depends on the forward
call having been replayed too. Replays differ in the order of their sums; a texel sums a few dozen
float32 terms (1e-5; a gradient counted twice is off by its whole size)."""

import pytest
import torch

import synth
from cases import rel_l2, sphere_scene

pytestmark = pytest.mark.gpu

W, H = 64, 48


@pytest.mark.parametrize("tess", [0, 1])
def test_replays_of_a_backward_recorded_alone(gpu_lib, tess):
    from paper_2104_03989_gb300 import binding as B
    from paper_2104_03989_gb300.engine import Context

    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = Context(stream=stream)
        job = ctx.create_job(sphere_scene(3, 32, 0, tess), loss="l2")
        views = torch.from_numpy(synth.sample_views(1, 0, 2, W, H).view("uint8").reshape(2, -1).copy()).cuda()
        ref = torch.rand(2, H, W, 3, generator=torch.Generator().manual_seed(0)).cuda()
        ctx.forward_loss([job], [views], [ref])
        ctx.backward([job])
        once = {k: ctx.params(job)[k].clone() for k in ("g_pos", "g_kd_chain")}
        B.adms_job_zero_gradients(ctx.ctx, job)
        ctx.forward_loss([job], [views], [ref])
        torch.cuda.synchronize()
        B.adms_graph_begin(ctx.ctx)
        ctx.backward([job])
        g = B.adms_graph_end(ctx.ctx)
        for n in (1, 2, 3):
            B.adms_graph_launch(ctx.ctx, g)
            torch.cuda.synchronize()
            p = ctx.params(job)
            for k, want in once.items():
                assert rel_l2(p[k].cpu(), n * want.double().cpu()) < 1e-5, (n, k)
        B.adms_graph_destroy(g)
        ctx.close()
