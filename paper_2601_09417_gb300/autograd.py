"""torch.autograd.Function around the splatting forward/backward of the C ABI.

The forward calls vbm_raster_fwd; the backward calls vbm_raster_bwd, which
reads the per-pixel compositing state the plan saved (the autograd "context"
lives in the plan, so one plan serves one in-flight forward at a time).
"""

import torch

from . import vbm


class SplatRender(torch.autograd.Function):
    """img[V][3][H][W] = render(params[14][stride]) for the views of `plan`."""

    @staticmethod
    def forward(ctx, params, plan, cams_dev, bg=(0.0, 0.0, 0.0), view_begin=0, view_count=None):
        vc = plan.n_views - view_begin if view_count is None else view_count
        # a call over all views writes every pixel; of a part of them, the other views' images are zero
        new = torch.empty if vc == plan.n_views else torch.zeros
        img = new((plan.n_views, 3, plan.height, plan.width), dtype=torch.float32, device=params.device)
        plan.forward(params, cams_dev, img, view_begin=view_begin, view_count=vc, bg=bg)
        ctx.plan, ctx.cams, ctx.bg, ctx.vb, ctx.vc = plan, cams_dev, bg, view_begin, vc
        ctx.save_for_backward(params)
        return img

    @staticmethod
    def backward(ctx, dimg):
        (params,) = ctx.saved_tensors
        # likewise the gradient's columns, where every column belongs to a set that some view sees
        whole = ctx.vc == ctx.plan.n_views and ctx.plan.seen_by_all_views == params.shape[1]
        grad = torch.empty_like(params) if whole else torch.zeros_like(params)
        ctx.plan.backward(params, ctx.cams, dimg.contiguous(), grad, view_begin=ctx.vb, view_count=ctx.vc,
                          bg=ctx.bg)
        return grad, None, None, None, None, None


def render(params, plan, cams_dev, bg=(0.0, 0.0, 0.0), view_begin=0, view_count=None):
    return SplatRender.apply(params, plan, cams_dev, bg, view_begin, view_count)
