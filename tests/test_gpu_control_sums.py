"""The packed sums of the control step where their trees change shape: the sums of
partial tiles behind tr D, the band energy and the idempotency of a solve, with
fewer partials than a warp, one warp's worth, several warps, more than the
block's threads, and (finite temperature) one to several levels of the tree
over the reference tiles, against the trace and energy of the result itself.

Bound: the solve's own tolerances, |tr D - N_e| <= 1e-9 at zero temperature and
the same for the density's trace at finite temperature; |E - tr(Hp D)| <= 1e-12
sum |Hp_ij D_ij|, for at most 2^20 FP64 additions on each side."""
import pytest

import hp_synth
from gpu_util import ctx, torch

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]


@pytest.mark.parametrize("kT", [0.0, 0.02])
@pytest.mark.parametrize("n", [64, 300, 520, 1000])
def test_control_sums(n, kT):
    if kT > 0:
        p = hp_synth.smeared(n, 0.85 * n, kT, -2.0, 1.0, n)
    else:
        p = hp_synth.gapped(n, int(0.6 * n), (-3.0, -0.01), (0.01, 1.0), n)
    H = torch.from_numpy(p.H).cuda()
    D = torch.empty_like(H)
    r = ctx().solve(H, p.ne, kT=kT, D=D)
    assert abs(float(torch.trace(D)) - p.ne) <= 1e-9
    assert abs(r["trace"] - p.ne) <= 1e-9
    assert abs(r["e_band"] - float((H * D).sum())) <= 1e-12 * float((H * D).abs().sum())
