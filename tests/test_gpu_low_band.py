"""Analyses of one map on both sides of the band limit up to which they are
summed directly (112): limits far below the map's, one ring block and several
chunks of rings, rows at the ends of their blocks."""
import pytest
import torch

from oracle import sht
from tests.gpu_util import ctx, rel_l2

pytestmark = pytest.mark.gpu


# FP64 recurrence and sums over up to 4096 rings, FFT rounding (as the transforms' other tests)
@pytest.mark.parametrize("nside,lmax", [(1, 0), (1, 3), (8, 1), (32, 63), (32, 112), (64, 2), (64, 113), (128, 16),
                                        (128, 111), (256, 33), (512, 10), (1024, 4)])
def test_analysis_matches_oracle(nside, lmax):
    c = ctx()
    m = torch.randn(12 * nside * nside, dtype=torch.float64, generator=torch.Generator().manual_seed(nside + lmax))
    alm = c.sht_analysis(m.cuda(), nside, lmax)
    assert rel_l2(alm, sht.analysis(m, nside, lmax)) < 1e-12


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("pixel", [0, 300, 12 * 128 * 128 - 1])
def test_non_finite_values_are_not_hidden(bad, pixel):
    c = ctx()
    m = torch.ones(12 * 128 * 128, dtype=torch.float64, device="cuda")
    m[pixel] = bad
    assert bool(c.sht_analysis(m, 128, 100).isnan().all())
