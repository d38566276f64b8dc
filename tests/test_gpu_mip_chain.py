"""Mip chains and their adjoint at the edges of the tiled path (sides of 32, long
strips, one-texel sides, one level beyond the block that forms the top): the
rebuild bit for bit against the box filter in float32, the fold against float64,
and adms_job_take_gradients against fold, scale and clear as separate calls."""

import numpy as np
import pytest
import torch

import synth
from synth.workloads import Scene

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (2, 1), (1, 64), (16, 16), (32, 32), (32, 64), (64, 2048), (2048, 32), (256, 256), (2048, 2048),
         (4096, 2048)]


def _chain(t):
    """Box-filter chain, float32, the texels of a cell summed row by row."""
    out = [t]
    while max(out[-1].shape[:2]) > 1:
        s = out[-1]
        h, w = s.shape[:2]
        sy, sx = min(h, 2), min(w, 2)
        acc = np.zeros((h // sy, w // sx, 4), np.float32)
        for dy in range(sy):
            for dx in range(sx):
                acc = acc + s[dy::sy, dx::sx]
        out.append(acc * np.float32(1.0 / (sx * sy)))
    return out


@pytest.mark.parametrize("h,w", SIZES)
def test_mip_chain_and_its_adjoint(gpu_lib, h, w):
    from paper_2104_03989_gb300 import stages

    rng = np.random.default_rng(h * 7 + w)
    t = rng.normal(size=(h, w, 4)).astype(np.float32)
    leaf = torch.from_numpy(t).cuda().requires_grad_(True)
    chain = stages.MipChain.apply(leaf)
    want = _chain(t)
    np.testing.assert_array_equal(chain.detach().cpu().numpy(), np.concatenate([x.reshape(-1, 4) for x in want]))
    g = torch.randn(chain.shape, generator=torch.Generator(device="cuda").manual_seed(3), device="cuda")
    got = torch.autograd.grad(chain, leaf, g)[0].cpu().numpy()
    gn, at = g.cpu().numpy().astype(np.float64), 0
    ref, mag = np.zeros((h, w, 4)), np.zeros((h, w, 4))
    for x in want:
        hh, ww = x.shape[:2]
        lv = gn[at:at + hh * ww].reshape(hh, ww, 4) * (hh * ww / (h * w))
        ref += np.repeat(np.repeat(lv, h // hh, 0), w // ww, 1)
        mag += np.repeat(np.repeat(np.abs(lv), h // hh, 0), w // ww, 1)
        at += hh * ww
    # at most 13 additions, each off by half an ulp of a partial sum
    assert (np.abs(got - ref) <= 13 * 2.0 ** -24 * mag).all()


@pytest.mark.parametrize("sizes", [((64, 64), (64, 64), (64, 64)), ((16, 8), (64, 32), (1, 1)), ((128, 32), (2, 2), (64, 1))])
@pytest.mark.parametrize("per_level", [False, True])
def test_taken_gradients_equal_fold_scale_and_clear(gpu_lib, sizes, per_level):
    from paper_2104_03989_gb300 import binding as B
    from paper_2104_03989_gb300.engine import Context

    rng = np.random.default_rng(1)
    mesh = synth.config_small()["cand"].mesh
    tex = [rng.uniform(0.1, 1.0, size=(*s, 4)).astype(np.float32) for s in sizes]
    ctx = Context()
    job = ctx.create_job(Scene(mesh=mesh, kd=tex[0], orm=tex[1], nrm=tex[2],
                               optimize={"pos": True, "kd": True, "orm": True, "nrm": True}),
                         per_level_textures=per_level)
    p = ctx.params(job)
    gen = torch.Generator(device="cuda").manual_seed(5)
    for n in ("g_pos", "g_kd_chain", "g_orm_chain", "g_nrm_chain"):
        p[n].copy_(torch.randn(p[n].shape, generator=gen, device="cuda"))
    scale = torch.tensor(0.37, device="cuda")
    want = {"pos": p["g_pos"] * scale}
    for n in ("kd", "orm", "nrm"):
        buf = torch.empty_like(p["g_" + n])
        B.adms_job_fold_gradients(ctx.ctx, job, **{"g_" + n: buf})
        want[n] = buf * scale
    got = {n: torch.empty_like(w) for n, w in want.items()}
    B.adms_job_take_gradients(ctx.ctx, job, scale, **{"g_" + n: b for n, b in got.items()})
    for n in want:
        assert torch.equal(got[n], want[n]), n
    for n in ("g_pos", "g_kd_chain", "g_orm_chain", "g_nrm_chain"):
        assert not p[n].any(), n
    with pytest.raises(B.AdmsError):  # no displacement map to take from
        B.adms_job_take_gradients(ctx.ctx, job, scale, g_disp=got["pos"])
    ctx.close()
