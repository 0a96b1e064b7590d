"""The FP64 schedule's step graph, which takes several products a pass, against the
same steps as plain launches (the profiled solve): whatever the number of steps
is modulo the products of a pass, both take the same steps, so D is bit for bit
the same."""
import pytest

import hp_synth
from gpu_util import ctx, torch

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]


@pytest.mark.parametrize("gap", [0.02, 0.05, 0.1, 0.2, 0.4, 0.8])
def test_graph_takes_the_plain_steps(gap):
    n = 70
    p = hp_synth.gapped(n, 40, (-3.0, -0.5 * gap), (0.5 * gap, 1.0), 61)
    H = torch.from_numpy(p.H).cuda()
    D = [torch.empty_like(H) for _ in range(2)]
    c = ctx()
    r = [c.solve(H, p.ne, D=D[0], precision="fp64")]
    c.profile(True)
    try:
        r.append(c.solve(H, p.ne, D=D[1], precision="fp64"))
    finally:
        c.profile(False)
    assert r[0]["iters"] == r[1]["iters"] and torch.equal(D[0], D[1])
    assert r[0]["trace"] == r[1]["trace"] and r[0]["e_band"] == r[1]["e_band"]
