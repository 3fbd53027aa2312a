"""The reversed ray step of the galaxy adjoint where its branches change:
deflections on both sides of the series limit |alpha| = 1/32, rays in the
polar blend (above the first ring), rays with no deflection at all."""
import pytest
import torch

from oracle import healpix as hp, rays
from tests.gpu_util import ctx, rel_l2

pytestmark = pytest.mark.gpu
F64 = torch.float64


def _gradients(kappas, nside, lmax, chi, gz, gphi, gchi, weight):
    import paper_1210_3069_gb300 as clc
    c = ctx()
    ko = [k.clone().requires_grad_(True) for k in kappas]
    go = rays.galaxy_shear(ko, nside, lmax, chi, gz, gphi, gchi)
    (go * weight).sum().backward()
    kg = kappas.clone().cuda().requires_grad_(True)
    gg = clc.galaxy_shear(c, kg, nside, lmax, chi, gz.cuda(), gphi.cuda(), gchi.cuda())
    (gg * weight.cuda()).sum().backward()
    c.sync()
    return go.detach(), torch.stack([k.grad for k in ko]), gg.detach(), kg.grad


# FP64 rounding of the chain grows with the tensor's 1 / sin(theta) near a pole
@pytest.mark.parametrize("amp,zlo", [(0.02, -1.0), (2.0, -1.0), (0.02, 0.9995), (2.0, 0.9995)])
def test_gradient_over_deflections_and_at_the_pole(amp, zlo):
    nside, lmax, n = 8, 16, 200
    g = torch.Generator().manual_seed(17)
    kappas = torch.stack([amp * torch.randn(hp.npix(nside), dtype=F64, generator=g) for _ in range(2)])
    gz = zlo + (1.0 - zlo) * torch.rand(n, dtype=F64, generator=g) * 0.9999
    gz[::2] = -gz[::2] if zlo > 0 else gz[::2]
    gphi = 6.2 * torch.rand(n, dtype=F64, generator=g)
    gchi = 101.0 + 198.0 * torch.rand(n, dtype=F64, generator=g)
    w = torch.randn(2, n, dtype=F64, generator=g)
    go, ko, gg, kg = _gradients(kappas, nside, lmax, [100.0, 200.0, 300.0], gz, gphi, gchi, w)
    assert rel_l2(gg, go) < 1e-10
    assert rel_l2(kg, ko) < 1e-9
