"""torch.autograd.Function front of the render-and-compare step.

`latents(ctx, job)` returns leaf tensors (requires_grad) that alias the job's
library-owned latents: positions (base positions of a tessellated job), the
level 0 of every optimized texture, and the displacement map. Calling
`render_loss(...)` runs adms_forward_loss; its backward runs the hand-written
backward kernels (AA, shading, texel and vertex scatter, tangent frame,
tessellation adjoints) in recompute mode, so nothing the forward rasterized
is read back: keys, pre-AA colours and loss gradients are rebuilt from the
latents and the reference images. `laplacian(...)` wraps Eq. 4's L_delta and
its hand-written gradient. All arithmetic runs in libadms.so.

A job holds one forward's state at a time: call backward before the next
forward of the same job. After changing latents in place (e.g. a torch
optimizer step), call `invalidate(ctx, job)` so mip chains and the vertex
frame are rebuilt.
"""

from __future__ import annotations

import torch

from . import binding as B

TEXTURES = ("kd", "orm", "nrm")
_TAKE = {"pos": "g_pos", "kd": "g_kd", "orm": "g_orm", "nrm": "g_nrm", "disp": "g_disp", "w": "g_skin_w"}


def latents(ctx, job, names=None):
    """{name: leaf tensor aliasing the job's latent, requires_grad=True} for the optimized latents."""
    p = ctx.params(job)
    out = {}
    for name in names or ("pos", "kd", "orm", "nrm", "disp"):
        if name not in p or p[name] is None:
            continue
        if name in TEXTURES and p["g_" + name] is None:
            continue
        if name == "disp" and p.get("g_disp") is None:
            continue
        out[name] = p[name].requires_grad_(True)
    return out


def invalidate(ctx, job):
    here, there = _streams(ctx)
    _order(there, here)  # the caller's writes to the latents
    B.adms_job_invalidate(ctx.ctx, job)
    _order(here, there)


def _recording(stream):
    """Whether a graph is being recorded from the stream (never from the default one)."""
    if stream.cuda_stream == 0:
        return False
    with torch.cuda.stream(stream):
        return torch.cuda.is_current_stream_capturing()


def _streams(ctx):
    """torch's current stream and the context's. Twice the same, so that nothing is ordered, while the context's
    records a graph that torch's has no part in: what is recorded runs when the graph does."""
    there = ctx.stream
    if getattr(there, "cuda_stream", there) == torch._C._cuda_getCurrentRawStream(torch.cuda.current_device()):
        return there, there
    if not hasattr(there, "cuda_stream"):
        there = torch.cuda.ExternalStream(int(there))
    here = torch.cuda.current_stream()
    return (there, there) if _recording(there) and not _recording(here) else (here, there)


def _order(waiting, stream, tensors=()):
    """Order a stream after another's work so far and keep the tensors' memory until the waiting one is through
    with them (nothing to do when both are one stream)."""
    if waiting is not stream:
        waiting.wait_stream(stream)
        for t in tensors:
            t.record_stream(waiting)


def _ordinary(g):
    """Whether an incoming gradient is a plain tensor of values: no graph to keep (create_graph), no forward-mode
    tangent, not batched or wrapped by a function transform (those have no data of their own)."""
    if type(g) is not torch.Tensor or (torch.is_grad_enabled() and g.requires_grad):
        return False
    if torch.autograd.forward_ad._current_level >= 0:
        return False
    try:
        g.data_ptr()
    except RuntimeError:
        return False
    return True


def _gradient_shapes(ctx, job, names, shapes):
    """The shapes of the buffers that the library fills whole: the job's own, whatever tensors the caller passed
    (a texture's may come in another shape of as many texels; torch refuses a gradient that does not fit)."""
    z = B.adms_job_sizes(ctx.ctx, job)
    out = []
    for n, shape in zip(names, shapes):
        if n in TEXTURES:
            own = (getattr(z, n + "_h"), getattr(z, n + "_w"), 4)
            out.append(shape if shape.numel() == own[0] * own[1] * 4 else own)
        else:
            out.append((z.disp_h, z.disp_w) if n == "disp" else (z.n_verts, z.n_bones if n == "w" else 3))
    return out


class _RenderLoss(torch.autograd.Function):
    @staticmethod
    def forward(fctx, ctx, job, views, refs, names, *tensors):
        here, there = _streams(ctx)
        _order(there, here, (refs,))
        loss = torch.empty((), dtype=torch.float32, device="cuda")
        ctx.forward_loss([job], [views], [refs], out_loss=loss)
        _order(here, there)
        fctx.ctx, fctx.job, fctx.names = ctx, job, names
        fctx.shapes = [t.shape for t in tensors]
        return loss

    @staticmethod
    def backward(fctx, g):
        ctx, job = fctx.ctx, fctx.job
        here, there = _streams(ctx)
        grads = [torch.empty(shape, dtype=torch.float32, device=g.device)
                 for shape in _gradient_shapes(ctx, job, fctx.names, fctx.shapes)]
        # an ordinary incoming gradient goes along as the scale of the one pass that hands the job's
        # out; one that torch follows further (a graph, a batch, a tangent) multiplies them in torch
        scale = g.detach().to(torch.float32).contiguous() if _ordinary(g) else None
        _order(there, here, grads if scale is None else (scale, *grads))
        B.adms_job_zero_gradients(ctx.ctx, job)
        ctx.backward([job], recompute_raster=True)
        # folded over the mip chains, the job's buffers left at zero: one pass over each, and
        # nothing for the host to wait for
        B.adms_job_take_gradients(ctx.ctx, job, scale, **{_TAKE[n]: buf for n, buf in zip(fctx.names, grads)})
        _order(here, there)
        if scale is None:
            grads = [buf * g for buf in grads]
        return (None, None, None, None, None, *grads)


def render_loss(ctx, job, views, refs, lat):
    """L_image of one job on one batch of views (Sec. 5.3), differentiable in `lat`."""
    names = tuple(lat.keys())
    return _RenderLoss.apply(ctx, job, views, refs, names, *[lat[n] for n in names])


class _Laplacian(torch.autograd.Function):
    @staticmethod
    def forward(fctx, ctx, job, pos):
        out = torch.empty((), dtype=torch.float32, device=pos.device)
        grad = torch.empty_like(pos)
        here, there = _streams(ctx)
        _order(there, here, (out, grad))
        B.adms_laplacian(ctx.ctx, job, out, grad)
        _order(here, there)
        fctx.save_for_backward(grad)
        return out

    @staticmethod
    def backward(fctx, g):
        (grad,) = fctx.saved_tensors
        return None, None, grad * g


def laplacian(ctx, job, pos):
    """L_delta of Eq. 4 for the job's positions (pos must alias them)."""
    return _Laplacian.apply(ctx, job, pos)
