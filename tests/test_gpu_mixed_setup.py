"""Set-up of the mixed-precision patch solver where its plan entries change
form: pixel pairs across longitude zero, the polar stencil, coarse and fine
maps against the cells, patches of the smallest sizes."""
import pytest
import torch

from oracle import healpix as hp
from tests.gpu_util import ctx

pytestmark = pytest.mark.gpu


# each field at every pixel against the FP64 solver's, both run to convergence:
# float-float set-up and residual, 2^-47 of the potential over the square of
# the cell size (1 / 400) at the smallest, stays under 1e-8 of the largest value
@pytest.mark.parametrize("nf,ns,nb,ncell", [(16, 4, 1, 16), (16, 16, 4, 16), (64, 8, 2, 64), (64, 32, 4, 32),
                                            (256, 16, 4, 128)])
def test_every_pixel_matches_fp64_solver(nf, ns, nb, ncell):
    import paper_1210_3069_gb300 as clc
    c = ctx()
    g = torch.Generator().manual_seed(nf + ncell)
    kappa = torch.rand(hp.npix(nf), dtype=torch.float64, generator=g).sub_(0.5).cuda()
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
