"""FP64 sums of the orders m = 0, 1 next to the poles (tensor-core batches):
cap sizes that do and do not fill a block's 32 rings, degrees beyond one staged
chunk, several classes; the fields on the polar rings against the FP64 path,
where the orders' Hessian terms cancel."""
import pytest
import torch

from tests.gpu_util import ctx, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[(64, 33)], [(64, 256)], [(128, 511), (64, 128), (128, 511)], [(256, 513)]])
def test_polar_rings_match_the_fp64_path(sizes):
    import paper_1210_3069_gb300 as clc
    c = ctx()
    g = torch.Generator().manual_seed(31)
    maps = [torch.randn(12 * n * n, dtype=torch.float64, generator=g).cuda() for n, _ in sizes]
    names = ("psi", "a_th", "a_ph", "u_tt", "u_pp", "u_tp")
    outs = [{k: torch.empty_like(m) for k in names} for m in maps]
    plan = c.sht_plan([n for n, _ in sizes], [l for _, l in sizes], graph=False)
    plan.execute(maps, outs)
    for (n, l), m, o in zip(sizes, maps, outs):
        ref = c.poisson_sht(m, n, l, precision=clc.FP64)
        cap = 2 * 12 * 13   # the first 12 rings and, mirrored, the last
        for k in names:
            assert rel_l2(o[k], ref[k]) < 1e-5, k            # the mixed path's stated bound
            # on the polar rings alone the uncorrected orders would be off by up to 1 / sin^2 (7e-5 and more)
            assert rel_l2(o[k][:cap], ref[k][:cap]) < 3e-5, k
            assert rel_l2(o[k][-cap:], ref[k][-cap:]) < 3e-5, k
    plan.close()
