"""Pixel indices next to pixel edges: points placed at distances from 0 to 1e-3
pixels of the integers that the index formulas floor, where the fixed-point
and FP32 indices must hand over to the FP64 formulas; counts bit for bit."""
import math

import pytest
import torch

from oracle import binning
from tests.gpu_util import ctx

pytestmark = pytest.mark.gpu
F64 = torch.float64


def _points(nside, n, seed):
    g = torch.Generator().manual_seed(seed)
    off = torch.tensor([0.0, 1e-16, 1e-14, 1e-12, 1e-9, 1e-7, 1e-6, 1e-5, 1e-4, 1e-3], dtype=F64)

    def near(hi):   # integers up to hi, moved by one of the offsets to either side
        k = torch.floor(torch.rand(n, generator=g, dtype=F64) * hi)
        e = off[torch.randint(0, off.numel(), (n,), generator=g)]
        return k + e * torch.where(torch.rand(n, generator=g) < 0.5, -1.0, 1.0)

    # belt: t1 - t2 and t1 + t2 near integers
    a, b = near(5 * nside), near(5 * nside)
    tt, z = (a + b) / (2 * nside) - 0.5, (b - a) / (1.5 * nside)
    keep = (z.abs() <= 2.0 / 3.0) & (tt >= 0) & (tt < 4)
    zs, ps = [z[keep]], [tt[keep] * (math.pi / 2)]
    # caps: tp tmp near an integer, any tmp
    tmp = torch.rand(n, generator=g, dtype=F64) * nside
    tp = (torch.floor(torch.rand(n, generator=g, dtype=F64) * tmp) + near(1.0)) / tmp.clamp(min=1e-9)
    tt = torch.floor(torch.rand(n, generator=g, dtype=F64) * 4) + tp.clamp(0.0, 1.0)
    zc = (1.0 - (tmp / nside) ** 2 / 3.0) * torch.where(torch.rand(n, generator=g) < 0.5, -1.0, 1.0)
    zs.append(zc)
    ps.append((tt * (math.pi / 2)).clamp(0.0, 2 * math.pi))
    return torch.cat(zs), torch.cat(ps)


@pytest.mark.parametrize("nside", [1, 4, 32, 512, 8192])
@pytest.mark.parametrize("nest", [False, True])
def test_points_next_to_pixel_edges(nside, nest):
    import paper_1210_3069_gb300 as clc
    c = ctx()
    z, phi = _points(nside, 200_000, 90 + nside)
    want = binning.bin_counts(nside, z, phi, nest=nest)
    got = c.bin_particles(z.cuda(), phi.cuda(), nside, clc.NEST if nest else clc.RING)
    c.sync()
    assert torch.equal(got.cpu().long(), want)


@pytest.mark.parametrize("shift", [0, 1])
def test_kappa_of_maps_at_any_alignment(shift):
    c = ctx()
    for nside in (64, 128):
        npx = 12 * nside * nside
        counts = torch.randint(0, 6000, (npx + 1,), dtype=torch.int32, generator=torch.Generator().manual_seed(2))
        out = torch.zeros(npx + 1, dtype=F64, device="cuda")[shift:shift + npx]
        c.counts_to_kappa(counts.cuda()[shift:shift + npx], nside, 3.7, 1.3, kappa=out)
        c.sync()
        assert torch.equal(out.cpu(), binning.kappa_from_counts(counts[shift:shift + npx].long(), 3.7, 1.3))
