"""Peeled keys of deep stacks against the oracle, bit for bit: more triangles per tile than one
staging pass holds, depths in every order the k-buffer's front-to-back classes and its
passing over by a triangle's depth floor meet (equal, two values, both directions, steep triangles
whose floor is far from their fragments, depths outside the view)."""

import numpy as np
import pytest

from oracle import visibility as OV
from test_gpu_raster_sizes import _scene, _view

pytestmark = pytest.mark.gpu

W, H, N = 53, 37, 700


def _stack(order):
    rng = np.random.default_rng(N)
    c = rng.uniform((0, 0), (W, H), (N, 1, 2))
    xy = c + rng.uniform(-45, 45, (N, 3, 2))
    xy[::7] = c[::7] + rng.uniform(-400, 400, (len(c[::7]), 3, 2))  # 64-bit edge functions
    t = np.linspace(0.1, 0.8, N)[:, None]
    z = {"equal": np.full((N, 3), 0.25), "two": np.where(rng.random((N, 1)) < 0.5, 0.25, 0.75) + np.zeros((N, 3)),
         "ascending": t + np.zeros((N, 3)), "descending": t[::-1] + rng.uniform(0, 1e-3, (N, 3)),
         "steep": rng.permuted(np.concatenate([rng.uniform(0, 0.1, (N, 1)), rng.uniform(0.2, 0.9, (N, 2))], 1), axis=1),
         "outside": rng.uniform(-1.5, 2.5, (N, 3))}[order]
    pos = np.stack([xy[..., 0] / (W / 2) - 1, 1 - xy[..., 1] / (H / 2), z], -1).reshape(-1, 3).astype(np.float32)
    return pos, np.arange(3 * N, dtype=np.int32).reshape(-1, 3)


@pytest.mark.parametrize("layers", [1, 2, 8, 16])
@pytest.mark.parametrize("order", ["equal", "two", "ascending", "descending", "steep", "outside"])
def test_peeled_keys_of_deep_stacks(gpu_lib, order, layers):
    from paper_2104_03989_gb300.engine import Context

    pos, tri = _stack(order)
    views = _view(W, H)
    want, _ = OV.raster_views_peeled(views, pos, tri, W, H, layers)
    assert (want[:, -1] != OV.EMPTY_KEY).any()
    ctx = Context()
    job = ctx.create_job(_scene(pos, tri), frozen=True, layers=layers)
    ctx.render_reference(job, views, H, W)
    got = ctx.keys(job, (layers, 2, H, W)).cpu().numpy().view(np.uint64)
    np.testing.assert_array_equal(got, np.swapaxes(want, 0, 1))
    ctx.close()
