"""FP64 sums of the orders m = 0, 1 next to the poles at the ends of their
staging: degrees (lmax + 2 for m = 0, one less for m = 1) at multiples of the 32
copied at a time and of the 1024 whose factors are staged, planes that differ."""
import pytest
import torch

from tests.gpu_util import ctx, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[(64, 30), (64, 31), (64, 62)], [(256, 1021), (256, 1022)], [(256, 1023), (64, 32)],
                                   [(256, 1024)] * 3])
def test_polar_rings_match_the_fp64_path(sizes):
    import paper_1210_3069_gb300 as clc
    c = ctx()
    g = torch.Generator().manual_seed(47)
    maps = [torch.randn(12 * n * n, dtype=torch.float64, generator=g).cuda() for n, _ in sizes]
    names = ("psi", "a_th", "a_ph", "u_tt", "u_pp", "u_tp")
    outs = [{k: torch.empty_like(m) for k in names} for m in maps]
    plan = c.sht_plan([n for n, _ in sizes], [l for _, l in sizes], graph=False)
    plan.execute(maps, outs)
    for (n, l), m, o in zip(sizes, maps, outs):
        ref = c.poisson_sht(m, n, l, precision=clc.FP64)
        cap = 2 * 12 * 13   # the first 12 rings and, mirrored, the last
        for k in names:   # the bounds of these sums' other test
            assert rel_l2(o[k], ref[k]) < 1e-5, k
            assert rel_l2(o[k][:cap], ref[k][:cap]) < 3e-5, k
            assert rel_l2(o[k][-cap:], ref[k][-cap:]) < 3e-5, k
    plan.close()
