"""Position gradients of jobs whose maps share no size, two sizes or one texel, opaque and in peeled
layers, against recorded ones: the backward's float32 terms for such maps stay what they are, term
by term. (The oracle cannot tell: both of two ways to fuse the specular adjoint's multiplications are
4e-4 from float64 on scenes like these, and up to 5e-5 from one another.)

PINS: per scene the gradient's norm and its products with four random directions, recorded from the
kernels that take maps of any sizes in one form. A position sums its float32 terms per warp in a
fixed order, then in float64, so repeated runs agree to the last bits of a float32; 1e-6 of the norm
is allowed."""

import dataclasses

import numpy as np
import pytest
import torch

import synth
from cases import sphere_scene

pytestmark = pytest.mark.gpu

W, H, N = 400, 300, 3
PINS = {  # (map sides, layers, seed)
    ((256, 64, 64), 0, 3): (30.62505128, 31.80339819, 28.48193306, -26.61101249, 45.55067557),
    ((256, 64, 64), 2, 6): (11.37225557, -7.586003521, 4.858405271, -13.2278287, -16.04644275),
    ((1, 1, 512), 0, 8): (16.58143726, -19.59241991, -15.02229832, 25.06302308, 4.078313364),
    ((1, 1, 512), 2, 8): (4.112791471, -4.892934762, -3.709537612, 6.290852604, 1.100840663),
    ((1024, 1, 1), 2, 8): (0.4339757956, 0.3449322631, -0.3238551323, 0.1355426664, -0.09393920156),
    ((2048, 512, 1024), 0, 9): (1.189007897, -0.2336684438, 0.2493130381, -2.626281053, -0.1063991516),
    ((1, 256, 256), 0, 8): (9.765669226, 3.253168387, -6.544979431, 19.73409206, -16.79925564),
    ((1, 256, 256), 2, 4): (23.45376896, -27.87011169, -30.7297641, 30.14855138, 6.759909371),
}


def products(sizes, layers, seed):
    from paper_2104_03989_gb300.engine import Context

    k, o, n = sizes
    kd, nrm = synth.noise_textures(k, seed=seed)[0], synth.noise_textures(n, seed=seed)[1]
    kd[..., 3] = 0.5
    scene = dataclasses.replace(sphere_scene(16, 8, seed), kd=kd, orm=synth.scenes.uniform_orm(o, seed), nrm=nrm)
    ctx = Context()
    job = ctx.create_job(scene, loss="l2", layers=layers)
    rng = np.random.default_rng(seed)
    ref = torch.as_tensor(rng.uniform(0, 1, (N, H, W, 3)).astype(np.float32)).cuda()
    ctx.forward_loss([job], [synth.sample_views(seed, 0, N, W, H)], [ref])
    ctx.backward([job])
    torch.cuda.synchronize()
    g = ctx.params(job)["g_pos"].double().cpu().numpy()
    ctx.close()
    return [float(np.linalg.norm(g))] + [float((g * rng.normal(size=g.shape)).sum()) for _ in range(4)]


@pytest.mark.parametrize("case", list(PINS))
def test_gradients_are_the_recorded_ones(gpu_lib, case):
    want = PINS[case]
    got = products(*case)
    err = max(abs(a - b) for a, b in zip(got, want)) / want[0]
    print(case, "%.1e" % err)
    assert err < 1e-6
