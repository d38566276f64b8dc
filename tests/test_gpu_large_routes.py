"""Routes that only large calls take, at sizes that leave remainders everywhere.

Peeled layers above 2^20 samples each (all layers in one launch, one list of pixels to refine over
layers and views) against the same views one per call (refined where they are shaded): the same
float32 arithmetic, which the compiler may fuse otherwise in the two kernels (1e-5; a pixel refined
with another view's camera or another layer's triangle would be off by its whole colour).

The depth-filtered direct raster in rounds (2^22 triangle-views and more), its tiles looked over by
a small grid (4096 tiles and more), with a last group of the triangles' permutation that is not
full, an odd image and views whose triangles begin inside a group: keys bit for bit."""

import dataclasses

import numpy as np
import pytest
import torch

import synth
from cases import rel_l2
from oracle import visibility as OV
from synth.workloads import Scene

pytestmark = pytest.mark.gpu


def _cloud(n, size, tex, alpha):
    """n quads of half-sides in `size`, noise maps of different sizes"""
    mesh = synth.quad_cloud(n, 3, size=size)
    kd, nrm = synth.noise_textures(tex, seed=1)
    kd[..., 3] = alpha
    return Scene(mesh=mesh, kd=kd, orm=synth.scenes.uniform_orm(tex // 2, 1), nrm=nrm[::2, ::2].copy(),
                 optimize={"pos": True, "kd": True, "orm": True, "nrm": True})


@pytest.mark.parametrize("W,H,layers", [(725, 725, 2), (1027, 513, 3)])
def test_peeled_layers_in_one_launch_equal_one_view_a_call(gpu_lib, W, H, layers):
    from paper_2104_03989_gb300.engine import Context

    assert W * H <= 1 << 20 < 2 * W * H
    views = synth.sample_views(5, 0, 2, W, H)
    ctx = Context()
    job = ctx.create_job(_cloud(400, (0.1, 0.2), 2048, 0.5), frozen=True, layers=layers)
    both = ctx.render_reference(job, views, H, W).cpu().numpy()
    for k in range(2):
        one = ctx.render_reference(job, views[k:k + 1], H, W).cpu().numpy()
        assert np.abs(one).max() > 0.5  # bright enough to be refined
        assert rel_l2(both[k:k + 1], one) < 1e-5, k
    ctx.close()


@pytest.mark.parametrize("quads,W,H,n", [(265003, 533, 517, 8), (700011, 641, 531, 3)])
def test_depth_filtered_rounds_with_remainders(gpu_lib, quads, W, H, n):
    from paper_2104_03989_gb300.engine import Context

    scene = _cloud(quads, (0.005, 0.015), 32, 1.0)
    pos, tri = scene.mesh.pos, scene.mesh.tri_pos
    assert len(tri) % 64 and n * len(tri) >= 1 << 22 and n * ((W + 15) // 16) * ((H + 15) // 16) >= 2 * 2048
    views = synth.sample_views(6, 0, n, W, H)
    want, _ = OV.raster_views(views, pos, tri, W, H)
    ctx = Context()
    job = ctx.create_job(dataclasses.replace(scene, optimize={}), frozen=True, raster_direct_px=256,
                         raster_depth_filter=True)
    ctx.render_reference(job, views, H, W)
    got = ctx.keys(job, (n, H, W)).cpu().numpy().view(np.uint64)
    np.testing.assert_array_equal(got, want)
    assert (want != OV.EMPTY_KEY).any()
    torch.cuda.synchronize()
    ctx.close()


@pytest.mark.parametrize("quads,n,rounds", [(32768, 4, False), (262143, 8, False), (262144, 8, True)])
def test_rounds_are_taken_by_large_clouds_only(gpu_lib, quads, n, rounds):
    """Four rounds and three passes over the tiles' depths in place of one launch. At 2^18 triangle-views the
    rounds took 429 us where one pass takes 222."""
    from paper_2104_03989_gb300 import binding as B
    from paper_2104_03989_gb300.engine import Context

    W = H = 64
    views = synth.sample_views(6, 0, n, W, H)
    launches = []
    for zfilter in (False, True):
        ctx = Context()
        job = ctx.create_job(dataclasses.replace(_cloud(quads, (0.005, 0.015), 32, 1.0), optimize={}), frozen=True,
                             raster_direct_px=256, raster_depth_filter=zfilter)
        ctx.render_reference(job, views, H, W)
        before = B.lib().adms_launch_count()
        ctx.render_reference(job, views, H, W)
        launches.append(B.lib().adms_launch_count() - before)
        torch.cuda.synchronize()
        ctx.close()
    assert launches[1] - launches[0] == (6 if rounds else 0)
