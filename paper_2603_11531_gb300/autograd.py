"""torch.autograd.Function around mgs_render / mgs_render_backward.

Training-style use: Gaussian attributes (N, 24) and, optionally, the MLP
parameters are CUDA tensors that require grad.  Every step of the forward and
backward runs in the library's kernels; this module only moves tensors across
the C-ABI.  The parameters of a step change before the next one, so a step's
scene is borrowed device memory (a copy of the attributes and the MLP packed to
BF16, both from torch's allocator) instead of a loaded scene: uploading the MLP
through the host and allocating and freeing device memory took 1.0 ms of a
step, whatever its size.
"""
from __future__ import annotations

import numpy as np
import torch

from . import (MLP_GRAD_SIZE, Renderer, camera_struct, mgs_borrow_scene, mgs_camera, mgs_load_scene,
               mgs_mlp_blob_bytes, mgs_render_backward, mgs_render_checked, mgs_unload_scene,
               mgs_workspace_captured, render_opts)
from .synth import MLPWeights, f32_to_bf16_bits

_SHAPES = (("w1", (64, 22)), ("b1", (64,)), ("w2", (64, 64)), ("b2", (64,)),
           ("w3", (5, 64)), ("b3", (5,)))
_SIZES = [int(np.prod(shp)) for _, shp in _SHAPES]
# mgs_load_scene stores larger scenes in spatial order, which pays there
_MAX_BORROWED = 1 << 21


def _mlp_from_tensors(ts) -> MLPWeights:
    arr = [t.detach().float().cpu().numpy() for t in ts]
    return MLPWeights(f32_to_bf16_bits(arr[0]), arr[1].astype(np.float32),
                      f32_to_bf16_bits(arr[2]), arr[3].astype(np.float32),
                      f32_to_bf16_bits(arr[4]), arr[5].astype(np.float32))


def _step_scene(renderer, attrs, mlp):
    """The scene of one step and the tensors it borrows."""
    if attrs.ndim == 2 and attrs.shape[0] > _MAX_BORROWED:
        return mgs_load_scene(renderer.ctx, attrs.detach().contiguous(),
                              _mlp_from_tensors(mlp) if mlp else None), ()
    a = attrs.detach().clone(memory_format=torch.contiguous_format)
    params = blob = None
    if mlp:
        params = [t if t.dtype == torch.float32 and t.device == a.device and t.is_contiguous()
                  else t.detach().to(device=a.device, dtype=torch.float32).contiguous() for t in mlp]
        # frozen biases may be columns or rows, as mgs_load_scene takes them
        params = [t if t.ndim == len(shp) else t.detach().reshape(-1) if len(shp) == 1 else t
                  for t, (_, shp) in zip(params, _SHAPES, strict=True)]
        blob = torch.empty(mgs_mlp_blob_bytes(), dtype=torch.uint8, device=a.device)
    return mgs_borrow_scene(renderer.ctx, a, params, blob), (a, blob)


class RenderFn(torch.autograd.Function):
    @staticmethod
    def forward(ctx, renderer, cam, opts, attrs, *mlp):
        scene, ctx.borrowed = _step_scene(renderer, attrs, mlp)
        try:
            cam = cam if isinstance(cam, mgs_camera) else camera_struct(cam)
            H, W = cam.height, cam.width
            rgb = torch.empty((H, W, 3), dtype=torch.float32, device=attrs.device)
            aux = torch.empty((5, H, W), dtype=torch.float32, device=attrs.device)
            mgs_render_checked(renderer.ws, scene, cam, opts, rgb, aux)
        except Exception:
            mgs_unload_scene(scene)
            raise
        ctx.renderer, ctx.cam, ctx.opts, ctx.scene = renderer, cam, opts, scene
        ctx.n_mlp = len(mlp)
        ctx.attrs_shape, ctx.attrs_dtype = attrs.shape, attrs.dtype
        ctx.save_for_backward(aux)
        return rgb

    @staticmethod
    def backward(ctx, g):
        (aux,) = ctx.saved_tensors
        if ctx.scene is None:
            raise ValueError("the scene of this render was released by its first backward")
        dev = aux.device
        d_attrs = torch.empty(ctx.attrs_shape, dtype=torch.float32, device=dev)
        d_mlp = torch.empty(MLP_GRAD_SIZE, dtype=torch.float32, device=dev) if ctx.n_mlp else None
        try:
            mgs_render_backward(ctx.renderer.ws, ctx.scene, ctx.cam, ctx.opts, g.contiguous(), aux,
                                d_attrs, d_mlp)
            # the library frees a loaded scene's memory; and the launch of a graph that
            # holds a render of this renderer cannot be ordered after this pass
            if not ctx.borrowed or mgs_workspace_captured(ctx.renderer.ws):
                torch.cuda.synchronize(dev)
        finally:
            mgs_unload_scene(ctx.scene)
            # the graph may outlive this pass (a program that keeps its losses); the
            # tensors go back to the stream that the pass runs on
            ctx.scene = ctx.borrowed = None
        grads = [None, None, None, d_attrs.to(ctx.attrs_dtype)]
        if ctx.n_mlp:
            grads += [t.view(shp) for t, (_, shp) in zip(d_mlp.split(_SIZES), _SHAPES)]
        return tuple(grads)


def render(renderer: Renderer, attrs: torch.Tensor, cam, mlp: tuple | None = None,
           use_mlp: bool = False, rgb_residual: bool = False, bg=(0.0, 0.0, 0.0)):
    """Differentiable render: returns the (H, W, 3) image; gradients flow to
    `attrs` and, with use_mlp, to the six MLP tensors (w1, b1, w2, b2, w3, b3)."""
    opts = render_opts(use_mlp, rgb_residual, bg)
    if use_mlp:
        if mlp is None or len(mlp) != 6:
            raise ValueError("use_mlp needs the six MLP tensors")
        return RenderFn.apply(renderer, cam, opts, attrs, *mlp)
    return RenderFn.apply(renderer, cam, opts, attrs)
