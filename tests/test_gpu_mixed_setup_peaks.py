"""Set-up of the mixed-precision patch solver from maps whose neighbouring
pixels differ by orders of magnitude, with every order of the nearer pixel and
ring, and with pixel pairs across longitude zero on either side."""
import pytest
import torch

from oracle import healpix as hp
from tests.gpu_util import ctx

pytestmark = pytest.mark.gpu


# the bound of the set-up's other test: 2^-47 of the potential over the square of the cell size
@pytest.mark.parametrize("nf,ns,nb,ncell", [(8, 8, 1, 16), (32, 4, 2, 32), (64, 64, 4, 32), (128, 32, 8, 32)])
def test_every_pixel_matches_fp64_solver(nf, ns, nb, ncell):
    import paper_1210_3069_gb300 as clc
    c = ctx()
    g = torch.Generator().manual_seed(3 * nf + ncell)
    kappa = torch.exp(3.0 * torch.randn(hp.npix(nf), dtype=torch.float64, generator=g)).sub_(1.0).cuda()
    out = []
    for prec in (clc.FP64, clc.MIXED):
        sol = c.solution(nf, clc.mg_params(ns, 2 * ns, nb, ncell=ncell, nu1=2, nu2=2, fixed_cycles=24, tol=1e-10,
                                           precision=prec))
        out.append(c.poisson_shtmg(kappa, nf, sol, derivatives=True))
        c.sync()
        sol.close()
    for k in ("a_th", "a_ph", "u_tt", "u_pp", "u_tp"):
        ref, got = out[0][k], out[1][k]
        assert float((got - ref).abs().max()) <= 1e-8 * float(ref.abs().max()), k
