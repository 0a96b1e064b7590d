"""The memory a call needs: a slot is its matrices, the vectors and one record per
tile, so a context whose budget holds these solves the problem; a projection needs
the slices of both operands and the partial sums.

The sizes are the sum over the buffers, each rounded up to 1 KiB: Hp and D copies,
the two FP64 buffers, FP32 masters, FP16 slices (two per matrix), then the digit
arrays (zero temperature) or the diagonals (finite temperature); 4 n bytes and 16
KiB are allowed for what grows with n alone."""
import pytest

import hp_synth
import oracle
from gpu_util import need_gpu, torch

import numpy as np

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]


def _slot(n, fermi):
    up = lambda x, a: -(-x // a) * a
    k = lambda x: up(x, 1024)
    ldy, lds = up(n, 4), up(n, 8)
    masters, slices = (5, 12) if fermi else (1, 4)
    b = 4 * k(8 * n * n) + masters * k(4 * n * ldy) + slices * k(2 * n * lds) + k(24 * n) + k(32 * n)
    b += k(12 * 6 * up(n, 8)) if fermi else 7 * k(2 * n * lds)
    t = -(-n // 64)
    return b + k(32 * max(608, t * (t + 1) // 2)) + 4 * n + (16 << 10)


@pytest.mark.parametrize("n,kT,precision", [(2048, 0.02, "mixed"), (2900, 0.0, "mixed"), (900, 0.0, "fp64")])
def test_solve_fits_a_budget_of_its_buffers(n, kT, precision):
    need_gpu()
    import paper_2301_04642_gb300 as fe
    if kT:
        p = hp_synth.smeared(n, 0.85 * n, kT, -2.0, 1.0, n, device="cuda")
    else:
        p = hp_synth.gapped(n, int(0.85 * n), (-3.0, -0.05), (0.05, 1.0), n, device="cuda")
    H = p.H if hasattr(p.H, "cuda") else torch.from_numpy(p.H).cuda()
    D = torch.empty_like(H)
    with fe.Context(device=0, hbm_budget_bytes=_slot(n, kT > 0)) as c:
        r = c.solve(H, p.ne, kT=kT, D=D, precision=precision)
    assert r["status"] == 0 and abs(float(torch.trace(D)) - p.ne) <= 1e-9


def test_fp64_schedule_equals_the_oracle_with_more_tiles_than_records():
    """n = 600: 741 tiles of 16 x 16, 608 records in the slot."""
    need_gpu()
    import paper_2301_04642_gb300 as fe
    n, ne = 600, 450
    p = hp_synth.gapped(n, ne, (-2.0, -0.1), (0.1, 0.6), 77, tol=1e-10)
    D = np.zeros_like(p.H)
    with fe.Context(device=0) as c:
        for precision in ("mixed", "fp64", "mixed"):  # the slot is used again
            r = c.solve(p.H, ne, tol=1e-10 if precision == "fp64" else 0.0, D=D, precision=precision)
            assert r["status"] == 0
            if precision == "fp64":
                ref = oracle.density(p.H, float(ne))
                # as for the smaller sizes: 30 products leave 30 n 2^-53 / gap in x, and the stop's 2e-10
                assert np.linalg.norm(D - ref["D"]) <= 1e-8


@pytest.mark.parametrize("m,n", [(4652, 523), (20440, 267), (5843, 521)])
def test_projection_in_a_budget_of_slices_and_sums(m, n):
    """Slices (8 n m) and partial sums of 128 x 192 blocks over the upper triangle; with
    less than its preferred tiles need, the projection takes narrower ones, and the
    result is the same."""
    need_gpu()
    import paper_2301_04642_gb300 as fe
    nk, ti, tj = -(-m // 64), -(-n // 128), -(-n // 192)
    blocks = sum(min(ti, (192 * j + 191) // 128 + 1) for j in range(tj))
    S = max(1, min(max(-(-nk // 128), -(-912 // blocks)), nk // 8))
    S = -(-nk // -(-nk // S))
    lds = -(-m // 8) * 8
    budget = -(-8 * n * lds // 1024) * 1024 + blocks * S * 4 * 128 * 192
    g = torch.Generator(device="cuda").manual_seed(m)
    P, Y = [torch.randn(m, n, generator=g, device="cuda", dtype=torch.float64) for _ in range(2)]
    H = [torch.empty(n, n, device="cuda", dtype=torch.float64) for _ in range(2)]
    for out, b in zip(H, (0, budget)):
        with fe.Context(device=0, hbm_budget_bytes=b) as c:
            c.project(P, Y, out)
    assert torch.equal(H[0], H[1])
    with fe.Context(device=0, hbm_budget_bytes=8 * n * lds) as c, pytest.raises(fe.FeError) as ei:
        c.project(P, Y, H[0])
    assert ei.value.status == fe.FE_ENOMEM


@pytest.mark.parametrize("served", [False, True])
def test_cached_slots_make_way_when_the_device_is_full(served):
    """The budget is taken at fe_create; a program that then allocates most of the
    device leaves room for one slot, whatever sizes came before."""
    need_gpu()
    import paper_2301_04642_gb300 as fe
    probs = [hp_synth.gapped_reflected(n, n // 2, (-3.0, -0.05), (0.05, 1.0), n, device="cuda") for n in (3000, 3100, 3200)]
    with fe.Context(device=0) as c:
        c.solve(probs[0].H, 1500)  # the engines' own buffers
        c.wait(c.submit(probs[0].H, 1500))
        torch.cuda.empty_cache()
        fill = torch.empty(torch.cuda.mem_get_info()[0] - (400 << 20), dtype=torch.uint8, device="cuda")
        for p in probs + probs[:1]:  # 0.52 to 0.59 GB a slot
            if served:
                r = c.wait(c.submit(p.H, p.ne), timeout_s=90)
                assert r["rc"] == 0
            else:
                assert c.solve(p.H, p.ne)["status"] == 0
        del fill
        torch.cuda.empty_cache()
