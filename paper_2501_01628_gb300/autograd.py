"""Differentiable rendering through libvr: a torch.autograd.Function whose
forward is vr_render_frame and whose backward is vr_render_backward (the
adjoint kernels). Argument marshalling only; no pixel or gradient
arithmetic happens in Python.

    r = Renderer(partition=dict(kind="grid", grid=(2, 2, 2)), vmin=0.0, vmax=1.5)
    img = r.render(tf, density, cam)       # tf [n, 4], density [Nz, Ny, Nx]: CUDA float32
    loss = ((img - target) ** 2).mean()
    loss.backward()                         # tf.grad, density.grad

Early termination is off (the adjoint differentiates every lattice sample).
"""
from __future__ import annotations

import torch

from . import vr


class Renderer:
    """One context plus one packed volume, re-packed when the density tensor
    changes (data pointer or version).

    Renders may come from any stream: the context's table, volume and partial images
    serve one render at a time, so a render on another stream than the last one's waits
    (on the device) until that one is done. One host thread at a time."""

    def __init__(self, partition: dict, vmin: float, vmax: float, step_voxels: float = 0.5,
                 device: int | None = None, storage: str = "f32"):
        self.device = torch.cuda.current_device() if device is None else int(device)
        self.ctx = vr.vr_create(self.device)
        self.partition = partition
        self.vmin, self.vmax = float(vmin), float(vmax)
        self.step = float(step_voxels)
        self.storage = storage
        self.vol = None
        self._key = None
        self._shape = None
        self._done = None      # event behind the last render on a stream other than the default one
        self._stream = None    # of the last render (None: no render, or one that is known to be done)
        vr.vr_set_render_params(self.ctx, self.step, 1.0)

    def _enter(self):
        """The current stream, behind the last render if that was on another one. (A
        capture starts with an idle device, and its events mean nothing outside.)"""
        stream = torch.cuda.current_stream()
        if self._stream is not None and stream != self._stream and not torch.cuda.is_current_stream_capturing():
            if self._stream.cuda_stream == 0:
                stream.wait_stream(self._stream)
            else:
                stream.wait_event(self._done)
        return stream

    def _leave(self, stream):
        # the default stream is always there to be waited for; another may be gone by the
        # next render, so an event is left behind on it (6 us of host time)
        if stream.cuda_stream != 0:
            if torch.cuda.is_current_stream_capturing():
                return
            if self._done is None:
                self._done = torch.cuda.Event()
            self._done.record(stream)
        self._stream = stream

    def _bind(self, tf: torch.Tensor, density: torch.Tensor, cam: dict, stream):
        d = density.detach()
        if not (d.is_cuda and d.dtype == torch.float32 and d.is_contiguous()):
            raise ValueError("density must be a contiguous CUDA float32 tensor")
        key = (d.data_ptr(), d._version, tuple(d.shape))
        if self.vol is None or tuple(d.shape) != self._shape:
            if self.vol is not None:
                vr.vr_volume_release(self.vol)
            self.vol = vr.vr_volume_create(self.ctx, d, self.storage, self.partition)
            self._shape = tuple(d.shape)
        elif key != self._key:
            vr.vr_volume_update(self.vol, d)
        self._key = key
        table = tf.detach().contiguous()
        if table.is_cuda and table.dtype == torch.float32 and table.data_ptr() % 16 == 0:
            vr.vr_set_transfer_function_async(self.ctx, table, self.vmin, self.vmax)
            table.record_stream(stream)
        else:
            vr.vr_set_transfer_function(self.ctx, table, self.vmin, self.vmax)
        vr.vr_set_camera(self.ctx, cam)

    def render(self, tf: torch.Tensor, density: torch.Tensor, cam: dict) -> torch.Tensor:
        return _Render.apply(tf, density, self, cam)

    def close(self):
        if self.vol is not None:
            vr.vr_volume_release(self.vol)
            self.vol = None
        if self.ctx is not None:
            vr.vr_destroy(self.ctx)
            self.ctx = None

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass


class _Render(torch.autograd.Function):
    @staticmethod
    def forward(ctx, tf, density, renderer: Renderer, cam: dict):
        stream = renderer._enter()
        try:
            renderer._bind(tf, density, cam, stream)
            out = torch.empty((cam["height"], cam["width"], 4), dtype=torch.float32, device=density.device)
            vr.vr_render_frame(renderer.ctx, renderer.vol, out)
        finally:
            renderer._leave(stream)
        ctx.save_for_backward(tf, density)
        ctx.renderer = renderer
        ctx.cam = cam
        return out

    @staticmethod
    def backward(ctx, grad_out):
        tf, density = ctx.saved_tensors
        r = ctx.renderer
        stream = r._enter()
        try:
            r._bind(tf, density, ctx.cam, stream)
            gtf = torch.zeros_like(tf, dtype=torch.float32)
            gden = torch.zeros_like(density) if ctx.needs_input_grad[1] else None
            vr.vr_render_backward(r.ctx, r.vol, grad_out.contiguous().float(), gtf, gden)
            vr.vr_sync(r.ctx)
        except Exception:
            r._leave(stream)
            raise
        r._stream = None
        return (gtf if ctx.needs_input_grad[0] else None), gden, None, None
