"""Visibility keys around the raster's size rules against the oracle, bit for bit:
triangles with snapped extents just below, at and above 96 pixels (int32 and
int64 edge functions), boxes that begin and end at tile borders, triangles that
reach far off screen, one-sample and one-row boxes; binned, rasterized directly
(with and without the key-read filter) and through the k-buffer, with lists that
take the second half of the record buffer."""

import numpy as np
import pytest
import torch

import synth
from oracle import visibility as OV
from synth.workloads import Scene

pytestmark = pytest.mark.gpu


def _screen_soup(W, H, seed):
    """Triangles given by screen positions and depths, as positions under an identity-like view (clip w = 1)."""
    rng = np.random.default_rng(seed)
    tris = []

    def add(pts):
        tris.append([(x, y, z) for (x, y), z in zip(pts, rng.uniform(-0.9, 0.9, 3))])

    for ext in (95.0, 95.99609375, 96.0, 96.00390625, 97.0, 150.0):
        for _ in range(6):
            x, y = rng.uniform(-20, W - 60), rng.uniform(-20, H - 60)
            add([(x, y), (x + ext, y + rng.uniform(0, 90)), (x + rng.uniform(0, 90), y + 80)])
            add([(x, y), (x + rng.uniform(0, 90), y + ext), (x + 70, y + rng.uniform(0, 60))])
    for _ in range(30):  # at tile borders and sample centres, thin and tiny
        x, y = 16.0 * rng.integers(0, W // 16), 16.0 * rng.integers(0, H // 16)
        add([(x, y), (x + 16, y), (x, y + 16)])
        add([(x + 0.5, y + 0.5), (x + 15.5, y + 0.5), (x + 15.5, y + 1.5)])
        add([(x + 7.3, y + 7.2), (x + 8.1, y + 7.9), (x + 7.4, y + 8.2)])
        add([(x, y + 3), (x + 60, y + 3.4), (x + 60, y + 3.9)])
    for _ in range(6):  # far off screen
        add([(-3000.0, rng.uniform(0, H)), (W + 2500.0, rng.uniform(0, H)), (rng.uniform(0, W), 9000.0)])
        add([(rng.uniform(0, W), rng.uniform(0, H)), (-900.0, 20.0), (rng.uniform(0, 60), -700.0)])
    p = np.array(tris, np.float64).reshape(-1, 3)
    pos = np.stack([p[:, 0] / (W / 2) - 1, 1 - p[:, 1] / (H / 2), p[:, 2]], 1).astype(np.float32)
    tri = np.arange(len(pos), dtype=np.int32).reshape(-1, 3)
    return pos, tri[rng.permutation(len(tri))]


def _scene(pos, tri):
    uv = np.random.default_rng(0).uniform(0, 1, (3 * len(tri), 2)).astype(np.float32)
    one = synth.constant_texture((0.5, 0.5, 0.5, 0.5)) if hasattr(synth, "constant_texture") else \
        synth.scenes.constant_texture((0.5, 0.5, 0.5, 0.5))
    return Scene(mesh=synth.Mesh(pos, uv, tri, np.arange(3 * len(tri), dtype=np.int32).reshape(-1, 3)), kd=one, orm=one,
                 nrm=synth.scenes.constant_texture((0.0, 0.0, 1.0)), optimize={})


def _view(W, H):
    v = synth.fixed_view(W, H)
    v[0]["mvp"] = np.eye(4, dtype=np.float32).reshape(-1)
    return np.concatenate([v, v])


@pytest.mark.parametrize("W,H", [(256, 192), (203, 149)])
@pytest.mark.parametrize("direct,zfilter", [(0, False), (64, False), (4096, False), (4096, True)])
def test_keys_match_the_oracle_around_the_size_rules(gpu_lib, W, H, direct, zfilter):
    from paper_2104_03989_gb300.engine import Context

    pos, tri = _screen_soup(W, H, seed=W + direct)
    views = _view(W, H)
    want, _ = OV.raster_views(views, pos, tri, W, H)
    ctx = Context()
    job = ctx.create_job(_scene(pos, tri), frozen=True, raster_direct_px=direct, raster_depth_filter=zfilter)
    ctx.render_reference(job, views, H, W)
    got = ctx.keys(job, (2, H, W)).cpu().numpy().view(np.uint64)
    np.testing.assert_array_equal(got, want)
    assert (want != OV.EMPTY_KEY).mean() > 0.5
    ctx.close()


@pytest.mark.parametrize("layers", [2, 3, 8, 11])
def test_peeled_keys_match_the_oracle_around_the_size_rules(gpu_lib, layers):
    from paper_2104_03989_gb300.engine import Context

    W, H = 203, 149
    pos, tri = _screen_soup(W, H, seed=layers)
    views = _view(W, H)
    want, _ = OV.raster_views_peeled(views, pos, tri, W, H, layers)
    ctx = Context()
    job = ctx.create_job(_scene(pos, tri), frozen=True, layers=layers)
    ctx.render_reference(job, views, H, W)
    got = ctx.keys(job, (layers, 2, H, W)).cpu().numpy().view(np.uint64)
    np.testing.assert_array_equal(got, np.swapaxes(want, 0, 1))
    # lists of about 12 entries per triangle: beyond the 8 of the list buffer itself, none overflows
    assert ctx.stats(job)["tile_overflows"] == 0
    ctx.close()
    torch.cuda.synchronize()
