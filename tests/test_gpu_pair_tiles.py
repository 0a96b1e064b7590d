"""The tensor-core product over tiles of a CTA pair (256 rows x 256, 128, 64 or
32 columns) where its geometry changes: a single partial tile, a second row
panel of one row, edges next to a tile boundary, one whole round of the pairs
and the first sizes beyond it (whose left-over tiles are cut into narrower
ones), against an FP64 product.

Bound (as for the other product tests): operand slices of 22 or 11 bits, four
one-sided additions per 64-wide chunk, chunk sums rounded."""
import math

import pytest

from gpu_util import ctx, torch

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]


@pytest.mark.parametrize("nslices", [2, 1])
@pytest.mark.parametrize("n", [1, 31, 65, 129, 257, 500, 769, 1537, 2816, 2817, 3073, 4353])
def test_pair_tiles(n, nslices):
    g = torch.Generator(device="cuda").manual_seed(n)
    Y = torch.randn(n, n, generator=g, device="cuda")
    Y = (Y + Y.T) / (2.0 * math.sqrt(n))
    C = torch.full_like(Y, float("nan"))
    ctx().sym_square(Y, C, nslices=nslices)
    Yd = Y.double()
    rel = (2.0 ** -21 if nslices == 2 else 2.0 ** -10) + 4 * 2.0 ** -23 + math.ceil(n / 64) * 2.0 ** -24
    err = (C.double() - Yd @ Yd).abs()
    assert torch.all(err <= rel * (Yd.abs() @ Yd.abs()) + 1e-30).item()
    assert torch.equal(C, C.T)
