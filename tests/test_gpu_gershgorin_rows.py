"""Row sums of the Gershgorin bounds where the integer summation can go wrong:
rows shorter than a warp's step and next to it, unaligned rows, entries spread
over the whole exponent range, zeros and subnormals, against exact sums.

Bound: n additions of half a place of the row sum (2^-53) and the few operations
after it; a matrix of zeros has bounds of exactly zero."""
import math

import numpy as np
import pytest

import hp_synth
from gpu_util import ctx, torch

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]


def _exact(H):
    lo, hi, big = math.inf, -math.inf, 0.0
    for i, row in enumerate(H):
        s = math.fsum(abs(float(x)) for x in row)
        d = float(H[i, i])
        r = math.fsum([s, -abs(d)])
        lo, hi, big = min(lo, d - r), max(hi, d + r), max(big, s)
    return lo, hi, big


def _matrix(n, kind):
    H = hp_synth.normal(5 + n, n * n).reshape(n, n)
    e = hp_synth.normal(6 + n, n * n).reshape(n, n)
    if kind == "wide":
        H = H * np.exp2(np.clip(np.round(e * 200.0), -900, 900))
    elif kind == "tiny":
        H = H * np.exp2(-1000.0 - np.abs(np.round(e * 20.0)))
    elif kind == "sparse":
        H = np.where(e > 1.5, H, 0.0)
    elif kind == "zero":
        H = np.zeros((n, n))
    return H


@pytest.mark.parametrize("kind", ["plain", "wide", "tiny", "sparse", "zero"])
@pytest.mark.parametrize("n,pad", [(1, 0), (31, 1), (255, 0), (256, 1), (257, 0), (700, 3)])
def test_row_sums(n, pad, kind):
    H = _matrix(n, kind)
    Hd = torch.full((n, n + pad), float("nan"), dtype=torch.float64, device="cuda")
    Hd[:, :n] = torch.from_numpy(H)
    lo, hi, _, bad = ctx().gershgorin(Hd[:, :n])
    rlo, rhi, big = _exact(H)
    assert bad == 0.0
    tol = (n + 4) * (2.0 ** -53 * big + 5e-324)
    assert abs(lo - rlo) <= tol and abs(hi - rhi) <= tol
    if kind == "zero":
        assert lo == 0.0 and hi == 0.0
