"""What torch may do with the gradient that arrives at render_loss's backward: keep its graph
(create_graph), batch it (vmap), carry a tangent along. The gradients handed out are the job's
times it, each product rounded once to float32 (2^-23 with the sums' own order)."""

import numpy as np
import pytest
import torch

import synth
from cases import sphere_scene

pytestmark = pytest.mark.gpu

W, H = 64, 48


@pytest.fixture()
def problem(gpu_lib):
    from paper_2104_03989_gb300 import autograd as AG
    from paper_2104_03989_gb300.engine import Context

    ctx = Context()
    job = ctx.create_job(sphere_scene(3, 32, 0), loss="l2")
    lat = AG.latents(ctx, job)
    views = synth.sample_views(1, 0, 2, W, H)
    ref = torch.rand(2, H, W, 3, generator=torch.Generator().manual_seed(0)).cuda()
    loss = lambda: AG.render_loss(ctx, job, views, ref, lat)   # noqa: E731
    base = [g.double() for g in torch.autograd.grad(loss(), list(lat.values()))]
    yield loss, lat, base
    ctx.close()


def test_the_gradients_keep_their_dependence_on_the_incoming_one(problem):
    loss, lat, base = problem
    w = torch.tensor(3.0, device="cuda", requires_grad=True)
    got = torch.autograd.grad(w * loss(), list(lat.values()), create_graph=True)
    for g, b in zip(got, base):
        torch.testing.assert_close(g.double(), 3.0 * b, rtol=1e-5, atol=1e-6 * float(b.abs().max()))
    # d/dw sum (w b)^2 = 2 w sum b^2
    (dw,) = torch.autograd.grad(sum((g.double() ** 2).sum() for g in got) + w, w)
    assert float(dw) == pytest.approx(1.0 + 6.0 * sum(float((b ** 2).sum()) for b in base), rel=1e-5)


@pytest.mark.parametrize("how", ["is_grads_batched", "vmap"])
def test_batched_incoming_gradients(problem, how):
    loss, lat, base = problem
    v, value, leaves = torch.tensor([1.0, -2.0, 0.5], device="cuda"), loss(), list(lat.values())
    if how == "vmap":
        got = torch.func.vmap(lambda x: torch.autograd.grad(value, leaves, x))(v)
    else:
        got = torch.autograd.grad(value, leaves, v, is_grads_batched=True)
    for g, b in zip(got, base):
        assert g.shape == (3, *b.shape)
        for k, s in enumerate((1.0, -2.0, 0.5)):
            torch.testing.assert_close(g[k].double(), s * b, rtol=1e-5, atol=1e-6 * float(b.abs().max()))


def test_a_tangent_of_the_incoming_gradient(problem):
    loss, lat, base = problem
    with torch.autograd.forward_ad.dual_level():
        one = torch.ones((), device="cuda")
        v = torch.autograd.forward_ad.make_dual(one, 3.0 * one)
        got = torch.autograd.grad(loss(), list(lat.values()), v)
        for g, b in zip(got, base):
            g = torch.autograd.forward_ad.unpack_dual(g)
            for x, s in ((g.primal, 1.0), (g.tangent, 3.0)):
                torch.testing.assert_close(x.double(), s * b, rtol=1e-5, atol=1e-6 * float(b.abs().max()))


def test_scaled_gradients_without_a_graph(problem):
    loss, lat, base = problem
    got = torch.autograd.grad(0.25 * loss(), list(lat.values()))
    for g, b in zip(got, base):
        assert not g.requires_grad
        torch.testing.assert_close(g.double(), 0.25 * b, rtol=1e-5, atol=1e-6 * float(b.abs().max()))
