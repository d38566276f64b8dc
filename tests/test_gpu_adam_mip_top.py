"""The coarse levels after an optimizer step, on either side of the size at which their block grows: levels
6 and up are the box filter of level 5 bit for bit, the step's gradients are cleared at every level, and
the step is counted, whichever map of the launch is the large one."""

import numpy as np
import pytest
import torch

import synth
from synth.workloads import Scene
from test_gpu_mip_chain import _chain

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [((64, 64), (32, 32), (128, 64)), ((1024, 1024), (256, 64), (1024, 512)),
                                   ((2048, 1024), (1024, 1024), (32, 32)), ((64, 64), (32, 2048), (2048, 2048)),
                                   ((1, 1), (4096, 2048), (64, 64)), ((2048, 512), (16, 16), (1, 1))])
def test_coarse_levels_after_a_step(gpu_lib, sizes):
    from paper_2104_03989_gb300.engine import Context

    rng = np.random.default_rng(2)
    tex = [rng.uniform(0.1, 1.0, size=(*s, 4)).astype(np.float32) for s in sizes]
    ctx = Context()
    job = ctx.create_job(Scene(mesh=synth.config_small()["cand"].mesh, kd=tex[0], orm=tex[1], nrm=tex[2],
                               optimize={"pos": True, "kd": True, "orm": True, "nrm": True}))
    p = ctx.params(job)
    gen = torch.Generator(device="cuda").manual_seed(5)
    names = ("kd", "orm", "nrm")
    for n in names:
        p["g_" + n + "_chain"].copy_(torch.randn(p["g_" + n + "_chain"].shape, generator=gen, device="cuda"))
    before = {n: p[n].clone() for n in names}
    ctx.step([job])
    torch.cuda.synchronize()
    assert ctx.params(job)["t"] == 1
    for n, (h, w) in zip(names, sizes):
        assert not torch.equal(p[n], before[n]), n
        assert not p["g_" + n + "_chain"].any(), n
        dims = [(max(h >> k, 1), max(w >> k, 1)) for k in range(p[n + "_levels"])]
        at = [0, *np.cumsum([a * b for a, b in dims])]
        chain = p[n + "_chain"].cpu().numpy()
        if len(dims) > 6:
            want = _chain(chain[at[5]:at[6]].reshape(*dims[5], 4))
            np.testing.assert_array_equal(chain[at[6]:], np.concatenate([x.reshape(-1, 4) for x in want[1:]]))
    ctx.close()
