"""The antialiasing + loss stage on colours that its caller put under the mesh: an empty pixel's
colour counts like any other, in the image, in the loss and in the adjoint.

The image at an empty pixel whose neighbours are empty is its colour. The loss is the sum of the
image's terms: float32 terms and float64 here, each rounded a few times (1e-6). Squared error is
quadratic in the colours, so a central difference of any step is its gradient up to the rounding of
the terms: 2^-23 of the terms that move, up to about 10 beside a lit surface, over steps of 0.25 to
either side is 2e-6, 1e-5 of a slope of 0.2 or more; the sum's 46 bits add less. 1e-4 is asked for."""

import numpy as np
import pytest
import torch

import synth
from cases import sphere_scene

pytestmark = pytest.mark.gpu

W, H = 70, 53


def test_empty_pixels_keep_their_callers_colour(gpu_lib):
    from paper_2104_03989_gb300 import binding as B
    from paper_2104_03989_gb300 import stages as ST

    scene = sphere_scene(3, 16, 1)
    m = scene.mesh
    views = synth.sample_views(2, 0, 2, W, H)
    pipe = ST.Pipeline(m.tri_pos, m.uv, m.tri_uv, m.n_verts, views, H, W)
    pos, kd, orm, nrm = (torch.tensor(a, device="cuda") for a in (m.pos, scene.kd, scene.orm, scene.nrm))
    gen = torch.Generator().manual_seed(0)
    ref = torch.rand(2, H, W, 3, generator=gen).cuda()
    ST.render_loss(pipe, pos, kd, orm, nrm, ref, "l2")
    empty = pipe.keys == -1
    assert empty.any() and not empty.all()
    back = torch.rand(2, H, W, 4, generator=gen).cuda()
    back[..., 3] = 0
    pre = torch.where(empty[..., None], back, pipe.pre).contiguous()
    clip = ST.Setup.apply(pipe, pos)
    scale = 1.0

    def call(p):
        img, loss = torch.zeros(2, H, W, 3, device="cuda"), torch.zeros(1, dtype=torch.float64, device="cuda")
        gprime = pipe.empty(2, H, W, 4)
        B.adms_aa_loss_fwd(pipe.mesh(pos), pipe.views, 2, H, W, clip, pipe.keys, p, ref, ST.LOSS["l2"], scale, img, loss,
                           gprime, pipe.work)
        return img, float(loss), gprime

    img, loss, gprime = call(pre)
    pad = torch.nn.functional.pad(empty.float()[:, None], (1, 1, 1, 1), value=1.0)
    full = torch.nn.functional.avg_pool2d(pad, 3, stride=1)[:, 0] > 0.999  # empty with empty neighbours
    assert full.any()
    torch.testing.assert_close(img[full], pre[..., :3][full], rtol=0, atol=0)
    assert loss == pytest.approx(float(((img.double() - ref.double()) ** 2).sum()), rel=1e-6)

    g_pre, g_clip = pipe.empty(2, H, W, 4), pipe.zeros(2, pipe.V, 4, dtype=torch.float64)
    B.adms_aa_loss_bwd(pipe.mesh(pos), pipe.views, 2, H, W, clip, pipe.keys, pre, gprime,
                       torch.ones(1, device="cuda"), g_pre, g_clip, pipe.work)
    rng = np.random.default_rng(3)
    errs = []
    for group in (full, empty & ~full):
        at = torch.nonzero(group).cpu().numpy()
        for b, y, x in at[rng.choice(len(at), size=min(len(at), 24), replace=False)]:
            c = int(rng.integers(3))
            vals = []
            for s in (0.25, -0.25):
                p = pre.clone()
                p[b, y, x, c] += s
                vals.append(call(p)[1])
            want = (vals[0] - vals[1]) / 0.5
            errs.append(abs(float(g_pre[b, y, x, c]) - want) / max(abs(want), 0.2))
    assert max(errs) < 1e-4
