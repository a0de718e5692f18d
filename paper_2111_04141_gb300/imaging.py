"""Imaging pipeline around the gridder: dirty images and model visibilities.

The imaging chain of Section 2.3 (Algorithm (convgridding)): gridding, the
inverse FFT of the grid and the correction step, giving the dirty image
(Eq. (ID) of Section 1.7 up to the approximation of the method); and its
adjoint, model image -> visibilities.  Gridding, degridding, the origin
shift and the correction run in libgw's kernels; the FFTs are cuFFT calls
through torch.fft (unnormalised, so the two operators are exact adjoints).

The dirty image is normalised by the sum of the weights of the visibilities
that were gridded (dropped records excluded), so a unit point source
observed by every visibility images to 1 at its pixel.
"""
from __future__ import annotations

from typing import Optional

import torch


def _run(plan, stream, chain, *args) -> torch.Tensor:
    """chain(plan, *args) with every step of it (the library's, the transforms,
    the reductions) on ``stream`` (None: the current one): after the work that
    the current stream holds, which makes the inputs, and before what it gets
    next, which may use the result or the inputs' memory."""
    here = None if stream is None else torch.cuda.current_stream(plan.device)
    if here is None or here.cuda_stream == stream.cuda_stream:
        return chain(plan, *args)
    stream.wait_stream(here)
    try:
        with torch.cuda.stream(stream):
            out = chain(plan, *args)
    finally:
        here.wait_stream(stream)
    out.record_stream(here)
    return out


def dirty_image(plan, uvw, freq, vis, weight: Optional[torch.Tensor] = None,
                normalise: bool = True, stream=None) -> torch.Tensor:
    """[npol, N, N] complex64 dirty image (the real part is the image)."""
    return _run(plan, stream, _dirty_image, uvw, freq, vis, weight, normalise)


def _dirty_image(plan, uvw, freq, vis, weight, normalise):
    g, dropped = plan.grid(uvw, freq, vis, weight=weight, return_dropped=True)
    img = torch.fft.ifft2(g, norm="forward")          # sum_k G_k exp(+j 2 pi k x / N)
    scale, scale_dev = 1.0, None
    if normalise:
        nrow, nchan = uvw.shape[0], freq.shape[0]
        if weight is None:
            scale = 1.0 / max(float(nrow * nchan - dropped), 1e-30)
        else:
            # drops are visibilities whose footprint leaves the grid: their
            # weights are excluded through the index records' valid flags
            raw, _ = plan.index(uvw, freq)
            valid = ((raw[:, 3] >> 16) & 1).to(torch.float32)
            w = weight.reshape(nrow * nchan, -1) * valid[:, None]
            ws = w.sum(0).to(torch.float64).clamp_min(1e-30)     # per polarisation
            scale_dev = (1.0 / ws).to(torch.float32)
    # origin shift, correction and normalisation in one pass
    return plan.finish_image(img, scale=scale, scale_dev=scale_dev)


def model_vis(plan, uvw, freq, image: torch.Tensor, stream=None) -> torch.Tensor:
    """Visibilities [nrow, nchan, npol] of a [npol, N, N] model image: the
    adjoint of the unnormalised dirty image (correct, FFT, shift, degrid)."""
    return _run(plan, stream, _model_vis, uvw, freq, image)


def _model_vis(plan, uvw, freq, image):
    x = image.to(torch.complex64).contiguous().clone()
    plan.correct(x, direction=-1)
    g = torch.fft.fft2(x, norm="backward").contiguous()  # sum_x I_x exp(-j 2 pi k x / N)
    plan.shift(g)
    return plan.degrid(uvw, freq, g)


def dirty_image_wstack(plan, uvw, freq, vis, n_layers: int, w_min: float, w_max: float,
                       normalise: bool = True, stream=None) -> torch.Tensor:
    """Dirty image by w-stacking (Section 1.7.1): a 2-D plan grids every
    visibility onto the grid of its w-layer; each layer grid is inverse
    transformed, re-centred, multiplied by its w-screen
    exp(+j 2 pi w_l (n - 1)) and summed (gw_wstack_combine, which also does
    the re-centring); the sum is corrected once."""
    return _run(plan, stream, _dirty_image_wstack, uvw, freq, vis, n_layers, w_min, w_max,
                normalise)


def _dirty_image_wstack(plan, uvw, freq, vis, n_layers, w_min, w_max, normalise):
    layers, dropped = plan.grid_wstack(uvw, freq, vis, n_layers, w_min, w_max,
                                       return_dropped=True)
    imgs = torch.fft.ifft2(layers, norm="forward")
    del layers
    img = plan.new_grid()
    plan.wstack_combine(imgs, w_min, w_max, img)
    plan.correct(img, direction=+1)
    if normalise:
        img /= max(float(uvw.shape[0] * freq.shape[0] - dropped), 1e-30)
    return img


def dirty_image_hybrid(plan, uvw, freq, vis, sz: int = 15, normalise: bool = True,
                       stream=None) -> torch.Tensor:
    """Dirty image by Hybrid Gridding (Section 2.4, Algorithm (hybrid)) with a
    2-D plan: Gridding Step onto beta N v-rows, column pruning to 2N rows,
    inverse FFT of the 2N x N grid, central N rows corrected."""
    return _run(plan, stream, _dirty_image_hybrid, uvw, freq, vis, sz, normalise)


def _dirty_image_hybrid(plan, uvw, freq, vis, sz, normalise):
    fine, dropped = plan.hybrid_grid(uvw, freq, vis, sz, return_dropped=True)
    pruned = plan.hybrid_prune(sz, fine)
    del fine
    plan.hybrid_shift(pruned)
    raw = torch.fft.ifft2(pruned, norm="forward")
    img = plan.hybrid_image(sz, raw)
    if normalise:
        img /= max(float(uvw.shape[0] * freq.shape[0] - dropped), 1e-30)
    return img
