"""The spectral-bound estimate of a single problem (its own kernel) against the one
for several problems at once: both make the same sums in the same order.

Sizes: a row less and more than a warp's group of 16, a block, a vector beyond
the block's threads, and the largest problem the single-problem kernel takes
and the first it does not.

FP64 problems are certified one at a time, so the bounds of a solve are equal
whether the problem comes alone or in a batch.  The others are certified in one
table, whose tiles (and with them the FP32 sums in ||X_3||_F, relative 2^-20)
depend on what else is in it: with t = 3 + 2.5 ||X_3||_F the widening
cosh(acosh(t) / 8) of a half-width then moves by at most 2^-20 / 4."""
import pytest

from gpu_util import ctx, torch

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]


def _problem(n):
    g = torch.Generator(device="cuda").manual_seed(n)
    A = torch.randn(n, n, generator=g, device="cuda", dtype=torch.float64) * (0.05 / n ** 0.5)
    lam = torch.linspace(-3.0, 1.0, n, device="cuda", dtype=torch.float64)
    lam += torch.where(lam > -1.0, 0.5, -0.5)
    return A + A.T + torch.diag(lam), int((lam < -1.0).sum())


def _bounds(H, ne, **kw):
    one = ctx().solve(H, ne, **kw)
    _, two = ctx().solve_batch([dict(H=H, ne=ne, **kw), dict(H=H, ne=ne, **kw)])
    ev = torch.linalg.eigvalsh(H)
    assert one["eps_min"] <= float(ev[0]) and float(ev[-1]) <= one["eps_max"]
    return one, two


@pytest.mark.parametrize("n", [2, 15, 16, 17, 33, 511, 513])
def test_same_bounds_fp64(n):
    one, two = _bounds(*_problem(n), precision="fp64")
    for r in two:
        assert (r["eps_min"], r["eps_max"]) == (one["eps_min"], one["eps_max"])


@pytest.mark.parametrize("n", [2, 17, 513, 1221, 4864, 4865])
def test_same_bounds_mixed(n):
    one, two = _bounds(*_problem(n))
    tol = 2.0 ** -22 * 0.5 * (one["eps_max"] - one["eps_min"])
    for r in two:
        assert abs(r["eps_min"] - one["eps_min"]) <= tol
        assert abs(r["eps_max"] - one["eps_max"]) <= tol
