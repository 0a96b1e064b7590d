"""The subspace products at the edges of their tiles (a pair's 256 rows, 32 to 256
columns, 64-wide K chunks and slice blocks), with aligned and unaligned operands
and results, against FP64 products.

Bound as for the other tests of these products: 22-bit operand slices, four
one-sided additions per chunk, the chunk sums rounded, and 2^-36 K max|A| max|B|
for entries whose low slice is subnormal in FP16."""
import math

import pytest

from gpu_util import ctx, torch

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]


def _rand(rows, cols, pad, seed):
    """rows x cols inside rows x (cols + pad), the first column left out when pad
    is odd (rows then start off a 16-byte boundary)"""
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn(rows, cols + pad, generator=g, device="cuda", dtype=torch.float64)
    return X[:, pad & 1:(pad & 1) + cols]


def _bound(A, B, chunks):
    rel = 2.0 ** -21 + 4 * 2.0 ** -23 + chunks * 2.0 ** -24
    fl = 2.0 ** -36 * A.abs().max() * B.abs().max() * A.shape[1]
    return rel * (A.abs() @ B.abs().T) + fl


@pytest.mark.parametrize("pad", [0, 3])
@pytest.mark.parametrize("m,n", [(1, 1), (63, 31), (65, 33), (129, 64), (257, 65), (300, 129),
                                 (700, 256), (1000, 257), (5000, 385), (20001, 513)])
def test_project_tiles(m, n, pad):
    P, Y = _rand(m, n, pad, m + n), _rand(m, n, pad, m + n + 1)
    H = torch.full((n, n + pad), 7.0, dtype=torch.float64, device="cuda")
    ctx().project(P, Y, H[:, :n])
    A, B = P.T, Y.T
    err = (H[:, :n] - A @ B.T).abs().triu()
    assert torch.all(err <= _bound(A, B, min(128, math.ceil(m / 64))).triu()).item()
    assert torch.equal(H[:, :n], H[:, :n].T) and torch.all(H[:, n:] == 7.0).item()


@pytest.mark.parametrize("pad", [0, 3])
@pytest.mark.parametrize("m,n", [(1, 1), (63, 31), (65, 33), (256, 64), (257, 65), (513, 129),
                                 (700, 257), (9001, 300), (20001, 513)])
def test_rotate_tiles(m, n, pad):
    P, D = _rand(m, n, pad, m - n), _rand(n, n, 0, n)
    D = (D + D.T) / 2
    O = torch.full((m, n + pad), 5.0, dtype=torch.float64, device="cuda")
    out = O[:, pad & 1:(pad & 1) + n]
    ctx().rotate(P, D, out)
    err = (out - P @ D).abs()
    assert torch.all(err <= _bound(P, D, math.ceil(n / 64))).item()
    out.fill_(5.0)
    assert torch.all(O == 5.0).item()
