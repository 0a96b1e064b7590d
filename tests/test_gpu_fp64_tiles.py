"""The FP64 schedule at sizes around its 16 x 16 tiles and 32-wide K stages,
against the oracle's density matrix.  An FP64 SP2 of about 30 products leaves
||D - D_ref||_F of order 30 n 2^-53 / gap-in-x plus the stop's 2e-10; 1e-8
holds it with a margin at these sizes."""
import numpy as np
import pytest

import hp_synth
import oracle
from gpu_util import ctx, torch

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]


@pytest.mark.parametrize("n", [2, 15, 16, 17, 31, 33, 48, 129, 272])
def test_fp64_schedule_at_tile_edges(n):
    ne = max(1, int(0.75 * n))
    p = hp_synth.gapped(n, ne, (-2.0, -0.1), (0.1, 0.6), 700 + n, tol=1e-10)
    D = np.zeros_like(p.H)
    r = ctx().solve(p.H, ne, tol=1e-10, D=D, precision="fp64")
    ref = oracle.density(p.H, float(ne))
    assert r["status"] == 0
    assert np.linalg.norm(D - ref["D"]) <= 1e-8
    assert np.array_equal(D, D.T)
