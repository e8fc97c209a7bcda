"""`torch.autograd` front end of the C ABI: a linear layer whose backward pass is
Algorithm 1 (low-rank backpropagation on the selected Walsh-Hadamard bases).

Only the backward pass is the library's: the forward product `y = x W^T + b` is a
plain matrix product and is left to torch (in one call, the bias added in the product's
epilogue, where x, weight and bias are of one type and autocast is off; else as a product
and a sum).  The layer takes the token grid
explicit, x of shape (B, H, W, Cin), or, with `grid=(H, W)`, a token sequence
(B, n + H*W, Cin) whose first n tokens (class tokens) are not part of the grid:
those take exact backpropagation (Eq. 2), and the grid tokens are handed to the
library as a strided view of the sequence, without a copy.  The bias (absent
from the paper's Eq. 1) is optional.
"""
from __future__ import annotations

from typing import Sequence, Tuple

import torch

from . import binding as _b


class LbpLinearFunction:
    """y = x W^T (+ b);  backward: Algorithm 1 on the selected bases.

    With `save_projected` the forward pass keeps x_hat = p(x) (Eq. 3) instead of
    x: r / k^2 of the activation's elements stay alive until the backward pass,
    which then starts at the second step of Algorithm 1.  Called as a
    `torch.autograd.Function` is; forward and backward are native
    (csrc/torch_binding.cpp)."""

    @staticmethod
    def apply(x: torch.Tensor, weight: torch.Tensor, bias, k: int, bases: Sequence[Tuple[int, int]],
              save_projected: bool, grid=None) -> torch.Tensor:
        H, W = (0, 0) if grid is None else (int(grid[0]), int(grid[1]))
        return _b._native().linear(x, weight, bias, int(k), [tuple(p) for p in bases], bool(save_projected), H, W)


class LbpLinear(torch.nn.Module):
    """Linear layer over a (B, H, W, C) token grid with LBP-WHT backward.

    `bases` is an ordered list of 0-based (i, j) sequency pairs, e.g. from
    `lbp_select_bases(k, SEL_L1, m)` (Eq. 8) or `lbp_select_lhe` (Sec. 3.2).
    """

    def __init__(self, in_features: int, out_features: int, k: int,
                 bases: Sequence[Tuple[int, int]], device=None, dtype=None, bias: bool = False,
                 save_projected: bool = False, grid=None):
        super().__init__()
        w = torch.empty((out_features, in_features), device=device, dtype=dtype)
        torch.nn.init.normal_(w, std=in_features ** -0.5)
        self.weight = torch.nn.Parameter(w)
        self.bias = (torch.nn.Parameter(torch.zeros(out_features, device=device, dtype=dtype))
                     if bias else None)
        self.k, self.bases = int(k), [tuple(p) for p in bases]
        self.save_projected = bool(save_projected)
        self.grid = None if grid is None else (int(grid[0]), int(grid[1]))

    def forward(self, x: torch.Tensor) -> torch.Tensor:
        H, W = self.grid or (0, 0)
        return _b._native().linear(x, self.weight, self.bias, self.k, self.bases, self.save_projected, H, W)
