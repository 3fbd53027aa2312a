"""Smoothing lengths at the limits of the kernel's two forms (sigma up to 2.9
pixels; up to 13 rings and 60 centres of a particle, about 4.2 pixels) and
beyond, also with particles of both kinds in one warp."""
import math

import pytest
import torch

from oracle import healpix as hp, smoothing as sm
from tests.gpu_util import ctx, rel_l2
from workloads import synthetic

pytestmark = pytest.mark.gpu
F64 = torch.float64


def _particles(nside, n):
    z, phi = synthetic.uniform_sphere(n, 5 + nside)
    cap = 1.0 - (torch.arange(20, dtype=F64) / nside) ** 2 / 6.0   # on and between the first rings, both poles
    z = torch.cat([z, cap, -cap])
    return z, torch.cat([phi, torch.linspace(0.0, 6.28, 40, dtype=F64)])


# weights and their sums carry a few ulp each (as in the other smoothing tests)
@pytest.mark.parametrize("nside,sig_pix", [(64, 2.89), (64, 2.91), (64, 3.0), (64, 3.25), (128, 3.75), (64, 4.2), (64, 4.35),
                                           (128, 4.4), (64, 7.0)])
def test_lengths_around_the_limits(nside, sig_pix):
    c = ctx()
    z, phi = _particles(nside, 300)
    sigma = sig_pix * math.sqrt(4 * math.pi / hp.npix(nside))
    got = c.smooth_particles(z.cuda(), phi.cuda(), nside, sigma)
    c.sync()
    assert rel_l2(got, sm.smooth_particles(nside, z, phi, sigma)) < 1e-12
    assert abs(float(got.sum()) - z.numel()) < 1e-9


def test_mixed_lengths_in_a_warp():
    c = ctx()
    nside = 64
    z, phi = _particles(nside, 88)
    sig = torch.linspace(0.2, 6.0, z.numel(), dtype=F64).reshape(2, -1).T.reshape(-1) * math.sqrt(4 * math.pi / hp.npix(nside))
    got = c.smooth_particles(z.cuda(), phi.cuda(), nside, sigma_each=sig.contiguous().cuda())
    c.sync()
    want = torch.zeros(hp.npix(nside), dtype=F64)
    for k in range(z.numel()):
        want += sm.smooth_particles(nside, z[k:k + 1], phi[k:k + 1], float(sig[k]))
    assert rel_l2(got, want) < 1e-12
