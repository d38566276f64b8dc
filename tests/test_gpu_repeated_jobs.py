"""An optimizer step whose list names a job twice: the entries' updates one after another (the
schedules first; the second entry meets cleared gradients and the positions' Laplacian term), against
the same two Adam steps in float64. float32 positions of about 1 move by 0.01: 2e-6 is a few
roundings of either; texels likewise. Gradients within a factor 1000 of Adam's eps are left out."""

import numpy as np
import pytest
import torch

import synth
from cases import sphere_scene

pytestmark = pytest.mark.gpu

W, H, LR, LAM = 64, 48, 0.01, 0.3


def _adam2(p, g1, g2):
    """two Adam updates with the bias corrections of the first step"""
    m = v = 0.0
    for g in (g1, g2):
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        p = p - LR * (m / 0.1) / (np.sqrt(v / 0.001) + 1e-8)
    return p


@pytest.mark.parametrize("tex", [8, 64])  # 64: tiled textures, all jobs' in one launch
@pytest.mark.parametrize("order", [(0, 0), (0, 1, 0)])
def test_a_job_named_twice_takes_two_updates_in_turn(gpu_lib, tex, order):
    from paper_2104_03989_gb300 import binding as B
    from paper_2104_03989_gb300.engine import Context

    ctx = Context()
    jobs = [ctx.create_job(sphere_scene(3, tex, s), loss="l2", lr0=LR, lambda0=LAM) for s in range(2)]
    alone = ctx.create_job(sphere_scene(3, tex, 1), loss="l2", lr0=LR, lambda0=LAM)
    views = synth.sample_views(1, 0, 2, W, H)
    ref = torch.rand(2, H, W, 3, generator=torch.Generator().manual_seed(0)).cuda()
    for j in (*jobs, alone):
        ctx.forward_loss([j], [views], [ref])
        ctx.backward([j])
    p = ctx.params(jobs[0])
    before = {k: p[k].double().cpu().numpy() for k in ("pos", "kd", "g_pos")}
    g_kd, lap, g_lap = torch.empty_like(p["kd"]), torch.zeros(1, device="cuda"), torch.empty_like(p["pos"])
    B.adms_job_fold_gradients(ctx.ctx, jobs[0], g_kd=g_kd)
    B.adms_laplacian(ctx.ctx, jobs[0], lap, g_lap)
    torch.cuda.synchronize()
    g_kd, g_lap = g_kd.double().cpu().numpy(), LAM * g_lap.double().cpu().numpy()

    ctx.step([jobs[k] for k in order])
    ctx.step([alone])
    torch.cuda.synchronize()
    p = ctx.params(jobs[0])
    assert p["t"] == 2 and not p["g_pos"].any() and not p["g_kd_chain"].any()
    g1 = before["g_pos"] + g_lap
    big = (np.abs(g1) > 1e-5) & (np.abs(g_lap) > 1e-5)
    assert big.mean() > 0.5
    np.testing.assert_allclose(p["pos"].double().cpu().numpy()[big], _adam2(before["pos"], g1, g_lap)[big], rtol=0, atol=2e-6)
    big = np.abs(g_kd[..., :3]) > 1e-5
    assert big.any()
    want = np.clip(_adam2(before["kd"], g_kd, 0 * g_kd), 0, 1)[..., :3]
    # the range clamp acts after each update: texels near its ends are compared where it cannot have
    inside = big & (np.abs(before["kd"][..., :3] - 0.5) < 0.45)
    np.testing.assert_allclose(p["kd"].double().cpu().numpy()[..., :3][inside], want[inside], rtol=0, atol=2e-6)
    if len(order) == 3:  # the job between the two entries: a step of its own
        a, b = ctx.params(jobs[1]), ctx.params(alone)
        assert a["t"] == b["t"] == 1
        for k in ("pos", "kd", "nrm"):
            torch.testing.assert_close(a[k], b[k], rtol=0, atol=2e-6)
    ctx.close()
