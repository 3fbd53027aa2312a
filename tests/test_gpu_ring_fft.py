"""Ring FFTs (ring_fft.cuh): ring lengths on both sides of the 16-point passes
and of the staged polar rings, band limits without and with aliasing, and
output maps that are only 8-byte aligned."""
import pytest
import torch

from oracle import sht
from tests.gpu_util import ctx, rel_l2

pytestmark = pytest.mark.gpu


# FP64 FFT and Legendre rounding: log2(2048) passes of 1e-16 and the recurrence
@pytest.mark.parametrize("nside,lmax", [(4, 16), (16, 63), (32, 20), (64, 256), (128, 100), (256, 300)])
def test_poisson_fields_over_ring_lengths(nside, lmax):
    c = ctx()
    k = torch.randn(12 * nside * nside, dtype=torch.float64, generator=torch.Generator().manual_seed(nside + lmax))
    got = c.poisson_sht(k.cuda(), nside, lmax)
    want = sht.poisson_sht(k, nside, lmax)
    for f in want:
        if f in got:
            assert rel_l2(got[f], want[f]) < 1e-11, f


def test_output_maps_at_odd_addresses():
    c = ctx()
    ns = 64
    npx = 12 * ns * ns
    k = torch.randn(npx, dtype=torch.float64, generator=torch.Generator().manual_seed(5)).cuda()
    names = ("psi", "a_th", "a_ph", "u_tt", "u_pp", "u_tp")
    plan = c.sht_plan([ns], [128], graph=False)
    outs = []
    for shift in (0, 1):
        buf = {f: torch.zeros(npx + 1, dtype=torch.float64, device="cuda")[shift:shift + npx] for f in names}
        plan.execute([k], [buf])
        outs.append(buf)
    c.sync()
    for f in names:
        assert torch.equal(outs[0][f], outs[1][f]), f
    plan.close()
