"""The digit-plane Legendre contractions (legendre.cu) at the edges of their
tiles: orders whose rows fill 64-row blocks exactly or by one more, ring
counts below and at a ring block, band limits up to 4 nside, one to eight
columns, values of any magnitude and non-finite ones."""
import pytest
import torch

from oracle import sht, spectra
from tests.gpu_util import ctx, rel_l2

pytestmark = pytest.mark.gpu

# The sums are exact to 2^-61 of max |lambda| max |F|; what remains is the
# FP64 recurrence (a few lmax ulp, up to 4e-14 at lmax 257) and FFT rounding.
TOL = 1e-12


@pytest.mark.parametrize("nside,lmax", [(1, 0), (1, 4), (2, 7), (16, 64), (32, 126), (32, 127), (32, 128), (64, 125),
                                        (64, 129), (128, 253), (128, 257)])
def test_transforms_at_tile_edges(nside, lmax):
    c = ctx()
    g = torch.Generator().manual_seed(nside * 1000 + lmax)
    m = torch.randn(12 * nside * nside, dtype=torch.float64, generator=g)
    alm = c.sht_analysis(m.cuda(), nside, lmax)
    want = sht.analysis(m, nside, lmax)
    assert rel_l2(alm, want) < TOL
    back = c.sht_synthesis(alm, nside, lmax)
    assert rel_l2(back, sht.synthesis(want, nside, lmax)) < TOL


@pytest.mark.parametrize("nside,lmax", [(32, 64), (64, 130)])
def test_eight_columns_match_single_calls(nside, lmax):
    c = ctx()
    g = torch.Generator().manual_seed(7)
    A = torch.eye(2, dtype=torch.float64).reshape(4, 1) + 0.01 * torch.randn(4, 12 * nside * nside, dtype=torch.float64,
                                                                              generator=g)
    got = c.lensing_spectra(A.contiguous().cuda(), nside, lmax)
    g1, g2 = -0.5 * (A[0] - A[3]), -0.5 * (A[1] + A[2])
    E, B = c.eb_analysis(g1.cuda(), g2.cuda(), nside, lmax)
    k = c.sht_analysis((1.0 - 0.5 * (A[0] + A[3])).cuda(), nside, lmax)
    for name, alm in (("E", E), ("B", B), ("kappa", k)):
        assert rel_l2(got[name], c.power_spectrum(alm, lmax)) < TOL, name
    wE, wB = spectra.eb_analysis(g1, g2, nside, lmax)
    assert rel_l2(E, wE) < 1e-11 and rel_l2(B, wB) < 1e-11   # cancelling spin-2 terms: about l times the rounding


def test_power_of_two_scaling_is_exact():
    c = ctx()
    m = torch.randn(12 * 64 * 64, dtype=torch.float64, generator=torch.Generator().manual_seed(3)).cuda()
    ref = c.poisson_sht(m, 64, 128)
    for e in (-700, 700):
        got = c.poisson_sht(m * 2.0 ** e, 64, 128)
        for k in ref:
            assert torch.equal(got[k] * 2.0 ** -e, ref[k]), (e, k)


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_values_are_not_hidden(bad):
    c = ctx()
    m = torch.ones(12 * 32 * 32, dtype=torch.float64, device="cuda")
    m[5000] = bad
    assert bool(c.sht_analysis(m, 32, 64).isnan().all())
    alm = torch.ones(65 * 66 // 2, dtype=torch.complex128, device="cuda")
    alm[40] = bad   # l = 40, m = 0
    assert bool(c.sht_synthesis(alm, 32, 64).isnan().all())
