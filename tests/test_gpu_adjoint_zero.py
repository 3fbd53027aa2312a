"""Gradient with respect to a plane that deflects nothing: the direction a ray
leaves with depends on the deflection to first order also at zero, and moves
the ray on every later plane."""
import pytest
import torch

from oracle import healpix as hp
from tests.gpu_util import ctx, rel_l2

pytestmark = pytest.mark.gpu
F64 = torch.float64


@pytest.mark.parametrize("zero", [0, 1])
def test_plane_without_deflection(zero):
    import paper_1210_3069_gb300 as clc
    c = ctx()
    nside, lmax, n, chi = 8, 16, 300, [100.0, 200.0, 300.0, 400.0]
    g = torch.Generator().manual_seed(23)
    kappas = 0.5 * torch.randn(3, hp.npix(nside), dtype=F64, generator=g)
    kappas[zero] = 0.0
    gz = 1.9 * torch.rand(n, dtype=F64, generator=g) - 0.95
    args = (gz.cuda(), (6.2 * torch.rand(n, dtype=F64, generator=g)).cuda(),
            (350.0 + 50.0 * torch.rand(n, dtype=F64, generator=g)).cuda())
    w = torch.randn(2, n, dtype=F64, generator=g).cuda()
    d = torch.randn(hp.npix(nside), dtype=F64, generator=g)

    def loss(h):
        k = kappas.clone()
        k[zero] += h * d
        return k.cuda().requires_grad_(True)

    def value(k):
        return (clc.galaxy_shear(c, k, nside, lmax, chi, *args) * w).sum()
    k0, k1 = loss(0.0), loss(1e-9)
    value(k0).backward()
    value(k1).backward()
    c.sync()
    # the gradient is continuous: 1e-9 of the planes' size changes it by about 1e-9
    assert rel_l2(k0.grad, k1.grad) < 1e-7
    # and it is the derivative: central difference, truncation (h over the pixel size)^2 and rounding / h
    h = 1e-5
    with torch.no_grad():
        fd = float(value(loss(h)) - value(loss(-h))) / (2 * h)
    an = float((k0.grad[zero].cpu() * d).sum())
    assert abs(fd - an) <= 1e-6 * max(abs(an), float(torch.linalg.vector_norm(k0.grad[zero]).cpu()))
