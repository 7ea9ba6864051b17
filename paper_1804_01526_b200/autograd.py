"""A dense layer and a 3 x 3 convolution whose three GEMMs run in block floating point (Sec. 4.1, Sec. 5.1).

The paper simulates HBFP by redefining PyTorch's linear module with ``autograd.Function``: the
forward product ``Y = X W``, the backward-data product ``dX = dY W^T`` and the backward-weight
product ``dW = X^T dY`` take BFP operands, every other operation (bias, activations, loss, the
optimiser's arithmetic) stays FP32. This module is that wrapper over the library's calls; it holds
no arithmetic of its own, and the passes themselves are autograd nodes in compiled code (``csrc/host.cpp``):

* the weights live in wide storage (16-bit mantissas per tile, ``hbfp_wide_quantize``); the two
  packed narrow views the GEMMs read are the top ``mant_bits`` bits (Sec. 4.2);
* forward and backward-data read those views (``hbfp_gemm_q``), so the backward pass converts no
  weights; activations and gradients are converted by the GEMM call with 1-D blocks along the
  contraction axis; backward-weight is ``hbfp_gemm`` with ``transA = 1``;
* ``apply_update(delta)`` hands the optimiser's FP32 update to ``hbfp_wide_update_value`` and refreshes the
  views in the same launch.

Stochastic rounding draws are keyed by (seed + step, stream id, element index): a layer takes three
consecutive stream ids (X, W, dY) from ``stream_id``.

``HbfpConv3x3`` does the same for a convolution on channels-last activations, on the two operands the
library builds without an FP32 im2col matrix (``hbfp_im2col_packed``, ``hbfp_im2col_packed_t``).
"""
from __future__ import annotations

import torch

from . import binding as hb


class HbfpLinear(torch.nn.Module):
    """``y = x W + b`` with W ``[fin][fout]`` in wide storage; see the module docstring."""

    def __init__(self, fin: int, fout: int, mant_bits: int = 8, tile: int = 24, rounding: int = 1, seed: int = 0,
                 stream_id: int = 0, batch_block: int = 32, bias: bool = True, device="cuda"):
        super().__init__()
        self.fin, self.fout = fin, fout
        self.mant_bits, self.tile, self.rounding, self.seed, self.stream_id = mant_bits, tile, rounding, seed, stream_id
        self.batch_block = batch_block
        self.steps = 0
        w = torch.randn(fin, fout, device=device) * (2.0 / fin) ** 0.5
        self.weight = torch.nn.Parameter(w)
        self.bias = torch.nn.Parameter(torch.zeros(fout, device=device)) if bias else None
        self.wide, self.views = hb.wide_quantize(self.weight.data, self.fmt_weight())
        self._refresh_fp32_copy()

    # ---- formats
    def fmt_weight(self) -> hb.Format:
        return hb.Format(mant_bits=self.mant_bits, block=self.tile, tile=self.tile, rounding=self.rounding,
                         seed=self.seed + self.steps, stream_id=self.stream_id + 1)

    def fmt_act(self, which: int, batch_axis: bool = False) -> hb.Format:
        """Format of X (which = 0) or dY (which = 2); blocks of ``tile`` along a feature axis, of
        ``batch_block`` along the batch axis (backward-weight)."""
        return hb.Format(mant_bits=self.mant_bits, block=self.batch_block if batch_axis else self.tile,
                         rounding=self.rounding, seed=self.seed + self.steps, stream_id=self.stream_id + which)

    # ---- weights
    def _refresh_fp32_copy(self) -> None:
        """The FP32 tensor autograd sees is the value of the wide copy (hbfp_wide_dequantize)."""
        self.weight.data = hb.wide_dequantize(self.wide)

    def apply_update(self, delta: torch.Tensor) -> None:
        """``W <- Q16(float32(W + delta))`` in wide storage, views and the FP32 copy refreshed by the same launch."""
        self.steps += 1
        self.weight.data = hb.wide_update_value(self.wide, delta.contiguous(), self.fmt_weight(), self.views)

    def forward(self, x: torch.Tensor) -> torch.Tensor:
        return hb.host().linear(x, self.weight, self.bias, self.views[0], self.views[1], self.mant_bits, self.tile, self.batch_block,
                                self.rounding, self.seed + self.steps, self.stream_id)


class HbfpConv3x3(torch.nn.Module):
    """3 x 3 convolution, stride 1, one pixel of zero padding, channels-last activations ``[n][h][w][c]``,
    as three BFP GEMMs (Sec. 5.1) without an FP32 im2col matrix: the forward operand is gathered from
    activations converted once per pixel, the backward-weight operand is converted straight from the
    activations, backward-data is the same implicit GEMM on the packed output gradient with the regrouped
    forward weights (a GEMM followed by the FP32 scatter onto the pixels where that does not apply). The weights
    ``[9 c][filters]`` (rows ordered (filter row, filter column, channel)) live in wide storage with
    ``c x c`` tiles, so the K-blocks of weights and activations coincide. Nearest-even rounding."""

    def __init__(self, c: int, fout: int, mant_bits: int = 8, pixel_block: int = 64, device="cuda"):
        super().__init__()
        self.c, self.fout, self.mant_bits, self.pixel_block = c, fout, mant_bits, pixel_block
        self.weight = torch.nn.Parameter(torch.randn(9 * c, fout, device=device) * (2.0 / (9 * c)) ** 0.5)
        self.wide, self.views = hb.wide_quantize(self.weight.data, self.fmt_weight())
        self._refresh_fp32_copy()

    def fmt_weight(self) -> hb.Format:
        return hb.Format(mant_bits=self.mant_bits, block=self.c, tile=self.c)

    def fmt_pixels(self, which: int) -> hb.Format:
        """X (blocks of c channels per pixel) or dY (blocks of c filters per pixel)."""
        return hb.Format(mant_bits=self.mant_bits, block=self.c, stream_id=which)

    def fmt_batch(self, which: int) -> hb.Format:
        """Backward-weight: blocks of ``pixel_block`` consecutive output pixels."""
        return hb.Format(mant_bits=self.mant_bits, block=self.pixel_block, stream_id=which)

    def _refresh_fp32_copy(self) -> None:
        self.weight.data = hb.wide_dequantize(self.wide)

    def apply_update(self, delta: torch.Tensor) -> None:
        self.weight.data = hb.wide_update_value(self.wide, delta.contiguous(), self.fmt_weight(), self.views)

    def forward(self, x: torch.Tensor) -> torch.Tensor:
        return hb.host().conv3x3(x, self.weight, self.views[0], self.views[1], self.mant_bits, self.pixel_block, self.c, self.fout)
