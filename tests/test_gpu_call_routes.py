"""The routes a single-job call takes by the memory and number of its views and by
the size of its image, against one another: views that travel with the launch and
views that are copied give the same bits; a loss finished by the last block of
the AA launch and one finished by a launch of its own differ by the order of the
block sums (compensated, then float64) and two roundings to float32; zeroed
gradients are zero in every word."""

import numpy as np
import pytest
import torch

import synth
from synth.workloads import Scene

pytestmark = pytest.mark.gpu


def _scene(seed=0):
    pos, tri = synth.scenes.icosphere(3)
    uv, tri_uv = synth.scenes.equirect_uv_corners(pos, tri)
    mesh = synth.Mesh(pos, uv, tri, tri_uv)
    rng = np.random.default_rng(seed)
    kd = rng.uniform(0.1, 0.9, (32, 32, 4)).astype(np.float32)
    orm = synth.scenes.constant_texture((1.0, 0.5, 0.2, 0.0))
    return Scene(mesh=mesh, kd=kd, orm=orm, nrm=synth.scenes.constant_texture((0.0, 0.0, 1.0)),
                 optimize=dict(pos=True, kd=True))


def _views(n, W, H):
    return synth.sample_views(3, 0, n, W, H)


@pytest.mark.parametrize("n", [1, 15, 16, 17])
def test_views_give_the_same_image_from_any_memory(gpu_lib, n):
    from paper_2104_03989_gb300.engine import Context

    W, H = 70, 45
    views = _views(n, W, H)
    raw = torch.from_numpy(views.view(np.uint8).reshape(n, -1).copy())
    ctx = Context()
    job = ctx.create_job(_scene(), frozen=True)
    want = ctx.render_reference(job, raw.cuda(), H, W)
    assert want.abs().sum() > 0
    for src in (views, raw, raw.pin_memory()):
        got = ctx.render_reference(job, src, H, W)
        torch.cuda.synchronize()
        assert torch.equal(got, want)
    ctx.close()


@pytest.mark.parametrize("W,H", [(5, 3), (512, 512), (512, 516)])
def test_the_loss_is_the_same_finished_in_either_place(gpu_lib, W, H):
    from paper_2104_03989_gb300 import binding as B
    from paper_2104_03989_gb300.engine import Context

    views = _views(1, W, H)
    ctx = Context()
    jobs = [ctx.create_job(_scene(1)) for _ in range(2)]
    ref = torch.rand((1, H, W, 3), generator=torch.Generator().manual_seed(0)).cuda()
    both = ctx.forward_loss(jobs, [views, views], [ref, ref]).cpu()
    for calls in (1, 2):  # the second call adds to the step's sum
        one = ctx.forward_loss(jobs[:1], [views], [ref]).cpu()
        np.testing.assert_allclose(one.numpy(), both.numpy()[:1], rtol=2.0 ** -22)
        s = ctx.stats(jobs[0])
        assert s["call_loss"] == pytest.approx(float(one[0]), rel=2.0 ** -23)
    ctx.backward(jobs[:1])
    B.adms_job_zero_gradients(ctx.ctx, jobs[0])
    torch.cuda.synchronize()
    p = ctx.params(jobs[0])
    for name in ("g_pos", "g_kd_chain"):
        assert not p[name].any(), name
    ctx.close()

