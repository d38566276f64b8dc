"""An optimizer step recorded into a graph takes launches of its own for schedules, positions and
counters (with the flat latents beside the textures) where a direct call fuses them: the same latents
after several steps from the same gradients, for every kind of latent, alone and for several jobs of
one call, with user-given and heuristic lambda. The gradients are given, not rendered, so nothing
depends on the order of a sum; the same float32 operations, each off by half an ulp where the compiler
fuses otherwise: a step of 0.01 is good to 1e-8 of a latent of about 1, its rounding to 6e-8 (1e-6)."""

import dataclasses

import numpy as np
import pytest
import torch

from cases import rel_l2, sphere_scene

pytestmark = pytest.mark.gpu

STEPS = 4
KINDS = {"plain": {}, "small maps": dict(tex=8), "tiled maps": dict(tex=64), "displaced": dict(tess=1),
         "fixed positions": dict(optimize=dict(pos=False, kd=True, orm=True, nrm=True)),
         "positions alone": dict(optimize=dict(pos=True)), "skinned": dict(bones=3)}
GRADS = ("g_pos", "g_kd_chain", "g_orm_chain", "g_nrm_chain", "g_disp", "g_w")


def _job(ctx, seed, tex=32, tess=0, bones=0, optimize=None, lambda0=0.0):
    scene = sphere_scene(3, tex, seed, tess)
    if optimize:
        scene = dataclasses.replace(scene, optimize=optimize)
    job = ctx.create_job(scene, loss="l2", lambda0=lambda0)
    if bones:
        w = np.random.default_rng(seed).uniform(0.1, 1, (len(scene.mesh.pos), bones)).astype(np.float32)
        ctx.skinning(job, w / w.sum(1, keepdims=True), lr_scale=0.3)
        ctx.set_bones(job, np.tile(np.eye(4, dtype=np.float32), (bones, 1, 1)))
    return job


@pytest.mark.parametrize("lambda0", [0.0, 0.2])
@pytest.mark.parametrize("kinds", [(k,) for k in KINDS] + [("plain", "displaced", "fixed positions", "tiled maps")])
def test_a_recorded_step_equals_a_direct_one(gpu_lib, kinds, lambda0):
    from paper_2104_03989_gb300 import binding as B
    from paper_2104_03989_gb300.engine import Context

    states = []
    for recorded in (False, True):
        ctx = Context(stream=torch.cuda.Stream())
        jobs = [_job(ctx, k, lambda0=lambda0, **KINDS[kind]) for k, kind in enumerate(kinds)]
        params = [ctx.params(j) for j in jobs]
        torch.cuda.synchronize()
        if recorded:
            B.adms_graph_begin(ctx.ctx)
            ctx.step(jobs)
            g = B.adms_graph_end(ctx.ctx)
        for step in range(STEPS):
            gen = torch.Generator(device="cuda").manual_seed(step)
            for p in params:
                for k in GRADS:
                    if p.get(k) is not None:
                        p[k].copy_(torch.randn(p[k].shape, generator=gen, device="cuda"))
            torch.cuda.synchronize()
            if recorded:
                B.adms_graph_launch(ctx.ctx, g)
            else:
                ctx.step(jobs)
            torch.cuda.synchronize()
            assert not any(p[k].any() for p in params for k in GRADS if p.get(k) is not None)
        out = []
        for j in jobs:
            p = ctx.params(j)
            assert p["t"] == STEPS
            out.append(({k: p[k].cpu().clone() for k in ("pos", "kd_chain", "orm_chain", "nrm_chain", "disp", "w")
                         if p.get(k) is not None}, ctx.stats(j)))
        states.append(out)
        if recorded:
            B.adms_graph_destroy(g)
        ctx.close()
    for (a, sa), (b, sb) in zip(*states):
        for k in a:
            assert rel_l2(b[k], a[k]) < 1e-6, k
        for k in ("lam", "lr", "laplacian"):
            assert sb[k] == pytest.approx(sa[k], rel=1e-5, abs=1e-12), k
        assert sa["status"] == sb["status"] == 0
