"""The FP64 Legendre table under budgets around its size (7.74 GB at nside 512,
lmax 1024): kept whole as soon as it fits, the first orders kept and the others
rebuilt below that; every way gives the same bits."""
import pytest
import torch

from tests.gpu_util import ctx

pytestmark = pytest.mark.gpu
F64 = torch.float64


def _solve(c, kappa, nside, lmax):
    n0 = c.launch_count()
    c.profile(True)
    out = c.poisson_sht(kappa, nside, lmax)
    c.sync()
    built = c.profile_query("k_legendre_build")[0]
    c.profile(False)
    return out, built, c.launch_count() - n0


def test_budget_just_above_the_table_keeps_it():
    c = ctx()
    nside, lmax = 512, 1024
    kappa = torch.randn(12 * nside * nside, dtype=F64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    try:
        c.release_caches()
        ref = _solve(c, kappa, nside, lmax)[0]
        for budget, builds in ((7.8e9, False), (5e9, True), (9e9, False), (0.9e9, True)):
            c.release_caches()
            c.set_table_budget(int(budget))
            for call in range(3):
                out, built, _ = _solve(c, kappa, nside, lmax)
                assert all(torch.equal(out[k], ref[k]) for k in ref), (budget, call)
            assert (built > 0) == builds, (budget, built)
    finally:
        c.set_table_budget(0)
        c.release_caches()


@pytest.mark.parametrize("nside,lmax", [(1, 4), (16, 40), (64, 129)])
def test_small_and_changing_budgets(nside, lmax):
    c = ctx()
    kappa = torch.randn(12 * nside * nside, dtype=F64, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    try:
        c.release_caches()
        ref, _, launches = _solve(c, kappa, nside, lmax)
        for budget in (1, 1 << 17, 1 << 20, 3 << 20, 1 << 18, 6 << 20, 1 << 30):
            c.set_table_budget(budget)
            for call in range(3):
                out = _solve(c, kappa, nside, lmax)[0]
                assert all(torch.equal(out[k], ref[k]) for k in ref), (budget, call)
        c.set_table_budget(0)
        assert _solve(c, kappa, nside, lmax)[1] == 0
    finally:
        c.set_table_budget(0)
        c.release_caches()
