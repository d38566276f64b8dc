"""Maps of equal, partly equal, different and one-texel sizes: each combination has a form of
its own in the shading kernels and their adjoint (all taps shared, those of the last two maps
shared, none, none for a map of one texel). Noise maps against the float64 oracle; maps of
one value, whose size cannot matter, against each other, opaque and in peeled layers."""

import dataclasses

import numpy as np
import pytest
import torch

import synth
from cases import assert_grads_match, fold_mips, oracle_grads, oracle_reference, rel_l2, sphere_scene, unambiguous_inputs

pytestmark = pytest.mark.gpu

W, H = 53, 37
SIZES = [(16, 8, 8), (1, 8, 8), (8, 1, 1), (1, 1, 16), (16, 8, 4), (8, 8, 16), (1, 1, 1)]


def _scene(sizes, seed):
    k, o, n = sizes
    return dataclasses.replace(sphere_scene(4, 8, seed), kd=synth.noise_textures(k, seed=seed)[0],
                               orm=synth.scenes.uniform_orm(o, seed), nrm=synth.noise_textures(n, seed=seed)[1])


def _run(scene, views, refs, loss, **opt):
    """image, loss and gradients (textures folded to level 0) of one forward and backward"""
    from paper_2104_03989_gb300.engine import Context

    ctx = Context()
    job = ctx.create_job(scene, loss=loss, **opt)
    img = torch.zeros((len(views), H, W, 3), device="cuda")
    val = ctx.forward_loss([job], [views], [torch.as_tensor(refs).cuda()], out_img=[img])
    ctx.backward([job])
    torch.cuda.synchronize()
    p = ctx.params(job)
    g = {"pos": p["g_pos"].double().cpu().numpy()}
    for m in ("kd", "orm", "nrm"):
        g[m] = fold_mips(p["g_" + m + "_chain"].cpu(), *p[m].shape[:2], p[m + "_levels"]).numpy()
    out = img.cpu().numpy(), float(val[0]), g
    ctx.close()
    return out


@pytest.mark.parametrize("sizes", SIZES)
def test_noise_maps_match_the_oracle(gpu_lib, sizes):
    views = synth.sample_views(7, 0, 2, W, H)
    refs, _ = oracle_reference(_scene((8, 8, 8), 1), views, H, W)
    scene, refs = unambiguous_inputs(_scene(sizes, 2), views, refs, H, W, "logl1")
    orc = oracle_grads(scene, views, refs, H, W, "logl1")
    img, val, g = _run(scene, views, refs, "logl1")
    assert rel_l2(img, orc["img"]) < 1e-5
    assert val == pytest.approx(orc["loss"], rel=1e-5)
    assert_grads_match(g, orc, str(sizes))


@pytest.mark.parametrize("layers", [0, 2])
@pytest.mark.parametrize("sizes", SIZES)
def test_the_size_of_a_map_of_one_value_does_not_matter(gpu_lib, sizes, layers):
    """Weights of a footprint sum to 1 within a few 2^-24; the gradients' sums over a map have a
    few thousand float32 terms in any order."""
    views = synth.sample_views(7, 0, 2, W, H)
    refs = np.random.default_rng(3).uniform(0, 1, (2, H, W, 3)).astype(np.float32)
    vals = {"kd": (0.6, 0.4, 0.3, 0.7), "orm": (0.2, 0.5, 0.3, 0.0), "nrm": (0.1, 0.2, 0.9, 0.0)}

    def flat(sz):
        maps = {m: np.broadcast_to(np.float32(v), (s, s, 4)).copy() for (m, v), s in zip(vals.items(), sz)}
        return dataclasses.replace(sphere_scene(4, 8, 2), **maps)

    a, b = (_run(flat(sz), views, refs, "l2", layers=layers) for sz in (sizes, (4, 4, 4)))
    assert rel_l2(a[0], b[0]) < 1e-5
    assert a[1] == pytest.approx(b[1], rel=1e-5)
    assert rel_l2(a[2]["pos"], b[2]["pos"]) < 1e-4
    for m in vals:
        ga, gb = (x[2][m].reshape(-1, 4).sum(0, dtype=np.float64) for x in (a, b))
        assert rel_l2(ga, gb) < 1e-4, m
