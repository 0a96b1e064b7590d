"""Tables of problems where the step loop changes its way: more problems than the
schedule table in shared memory holds (256), and batches whose members need
different kernel families in the same step (digit products falling due in
different steps, the FP64 schedule, finite temperature), so that tensor-core
steps wait for the others.  Members at zero temperature are compared with their
constructed density Q f Q^T, members at finite temperature with the same problem
solved alone (with few levels near mu the solve's own placement of mu, not the
table, decides its error: up to 7e-5 at n = 43), within the tolerances of a single
solve, and a second, small batch on the same context follows."""
import math

import numpy as np
import pytest

import hp_synth
from gpu_util import ctx, need_gpu, torch

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]


def _member(n, seed, gap=0.0, kT=0.0, precision="mixed"):
    ne = max(1, int(0.8 * n))
    if kT:
        p = hp_synth.smeared(n, ne, kT, -2.0, 1.0, seed)
    else:
        p = hp_synth.gapped(n, ne, (-3.0, -gap / 2), (gap / 2, 1.0), seed)
    H = torch.from_numpy(p.H).cuda()
    return p, dict(H=H, ne=ne, kT=kT, D=torch.full_like(H, float("nan")), precision=precision,
                   tol=1e-10 if precision == "fp64" else 0.0)


def _check(p, it, r):
    n, ne = p.n, it["ne"]
    assert r["status"] == 0
    if p.kT:
        alone = dict(it, D=torch.empty_like(it["H"]))
        r1 = ctx().solve(**alone)
        ref, e_ref = alone["D"].cpu().numpy(), r1["e_band"]
    else:
        f = (np.arange(n) < ne).astype(float)
        ref, e_ref = (p.Q * f) @ p.Q.T, float(np.sum(f * p.lam))
    D = it["D"].cpu().numpy()
    assert abs(np.trace(D) - ne) <= 1e-9 and abs(r["trace"] - ne) <= 1e-9
    assert np.linalg.norm(D - ref) / math.sqrt(ne) <= 1e-6
    assert abs(r["e_band"] - e_ref) / ne <= 1e-7
    if not p.kT:
        assert np.linalg.norm(D @ D - D) <= 1e-8


def _solve(members):
    rc, res = ctx().solve_batch([it for _, it in members])
    assert rc == 0
    for (p, it), r in zip(members, res):
        _check(p, it, r)


@pytest.mark.parametrize("count", [256, 257, 300])
def test_tables_around_the_shared_schedule(count):
    m = [_member(32 + (7 * k) % 33, 5000 + k, gap=0.1, kT=0.02 if k % 10 == 3 else 0.0) for k in range(count)]
    m[11] = _member(300, 5999, gap=0.05)  # the tiles of a larger one among them
    _solve(m)
    _solve([_member(90, 1, gap=0.1), _member(70, 2, kT=0.02)])


@pytest.mark.parametrize("fp64", [False, True])
def test_families_due_in_different_steps(fp64):
    m = [_member(150 + 40 * k, 6000 + k, gap=0.3 / 3 ** k) for k in range(5)]
    m += [_member(260, 6100, kT=0.01), _member(180, 6101, kT=0.05)]
    if fp64:
        m += [_member(100, 6200, gap=0.1, precision="fp64")]
    _solve(m)


@pytest.mark.parametrize("served", [False, True])
def test_expired_meeting_between_steps(served):
    """The truncated expansion takes Gershgorin bounds, so no certificate launch comes
    before the steps: the meeting that runs out (a word nothing writes, 1 ms) is one
    between two steps, in the step graph's kernel or in a served pass."""
    need_gpu()
    import paper_2301_04642_gb300 as fe
    p = hp_synth.smeared(400, 320, 0.02, -2.0, 1.0, 6300)
    H = torch.from_numpy(p.H).cuda()
    D = [torch.empty_like(H) for _ in range(2)]
    kw = dict(ne=320, kT=0.02, method=fe.FE_METHOD_TRFOE)
    with fe.Context(device=0) as c:
        def solve(D=None):
            return c.wait(c.submit(H, D=D, **kw), timeout_s=60) if served else c.solve(H, D=D, check=False, **kw)

        r0 = solve(D[0])
        c.set_wait(limit_ms=1.0, fail_partner=True)
        r = solve()
        assert r["status"] == r["rc"] == fe.FE_ETIMEOUT
        assert served or "timed out" in c.last_error()
        c.set_wait(limit_ms=2000.0, fail_partner=False)
        r1 = solve(D[1])
    assert r1["status"] == 0 and r1["iters"] == r0["iters"] and torch.equal(D[0], D[1])


@pytest.mark.parametrize("n,kT", [(1300, 0.02), (2000, 0.02), (4200, 0.02), (4200, 0.0)])
def test_control_sums_over_many_tiles(n, kT):
    """More than 32, 64 and 256 reference tiles (41, 72 and 305 of 128 x 256), and more
    product records than the control step has threads (153 tiles of 256 x 256, two
    each), against the trace and energy of the result itself; the sums are of at most
    2^25 terms in chains of at most 2^13, so 1e-12 of the sum of magnitudes holds."""
    make = hp_synth.smeared_reflected if kT else hp_synth.gapped_reflected
    args = (kT, -2.0, 1.0) if kT else ((-3.0, -0.05), (0.05, 1.0))
    p = make(n, int(0.85 * n), *args, n, device="cuda")
    D = torch.empty_like(p.H)
    r = ctx().solve(p.H, p.ne, kT=kT, D=D)
    assert abs(float(torch.trace(D)) - p.ne) <= 1e-9 and abs(r["trace"] - p.ne) <= 1e-9
    assert abs(r["e_band"] - float((p.H * D).sum())) <= 1e-12 * float((p.H * D).abs().sum())
