"""Ray step from lens maps (pure-SHT path): neighbours, bases and projection at
random rays, at pixel centres, at pixel edges and inside the polar rings, and
with the step as the context's first call on a stream that is being captured."""
import pytest
import torch

from oracle import healpix as hp, rays
from tests.gpu_util import ctx

pytestmark = pytest.mark.gpu
F64 = torch.float64
CHI = (100.0, 200.0, 300.0)
KEYS = ("a_th", "a_ph", "u_tt", "u_pp", "u_tp")


def _directions(nside, n, g):
    rt = hp.ring_table(nside)
    th1 = float(torch.atan2(rt["sin_theta"][0], rt["z"][0]))
    z = 2 * torch.rand(n, dtype=F64, generator=g) - 1
    th, ph = torch.acos(z), 6.2831 * torch.rand(n, dtype=F64, generator=g)
    pole = th1 * (0.1 + 1.2 * torch.rand(n, dtype=F64, generator=g))
    pole[::2] = torch.pi - pole[::2]
    th = torch.cat([th, pole, torch.full((8,), 0.5 * th1, dtype=F64)])
    ph = torch.cat([ph, ph.flip(0), 0.25 * torch.pi * torch.arange(8, dtype=F64)])
    v = torch.stack([torch.sin(th) * torch.cos(ph), torch.sin(th) * torch.sin(ph), torch.cos(th)], -1)
    p = torch.randint(0, hp.npix(nside), (n,), generator=g)
    v = torch.cat([v, hp.pix2vec_ring(nside, p)])
    return v / torch.linalg.vector_norm(v, dim=-1, keepdim=True), 0.1 * th1


def _case(nside):
    g = torch.Generator().manual_seed(5 + nside)
    v, th_min = _directions(nside, 500, g)
    f = {k: (1e-2 if k[0] == "a" else 1.0) * (2 * torch.rand(hp.npix(nside), dtype=F64, generator=g) - 1)
         for k in KEYS}
    want = rays.step(rays.init_rays(v, CHI[1]), rays.map_lens(nside, f), *CHI)
    # longitudes in pixels carry their rounding times 4 nside, the bases theirs over sin(theta)
    tol = 64 * 2.2e-16 * (4 * nside + 1.0 / th_min)
    return v, f, want, tol


def _start(c, v):
    M = v.shape[0]
    rs = c.rays(M)
    rs.x.copy_((CHI[1] * v.T).cuda())
    rs.beta.copy_(v.T.cuda())
    eye = torch.tensor([1.0, 0.0, 0.0, 1.0], dtype=F64).reshape(4, 1).expand(4, M)
    rs.A.copy_(eye.cuda())
    rs.Ap.copy_(eye.cuda())
    return rs


def _close(rs, want, tol):
    assert float((rs.x.T.cpu() - want["x"]).abs().max()) <= CHI[2] * tol
    assert float((rs.beta.T.cpu() - want["beta"]).abs().max()) <= tol
    assert float((rs.A.T.cpu() - want["A"].reshape(-1, 4)).abs().max()) <= tol
    assert float((rs.Ap.T.cpu() - want["Ap"].reshape(-1, 4)).abs().max()) <= tol


@pytest.mark.parametrize("nside", [1, 2, 32, 256])
def test_ray_step_from_maps(nside):
    c = ctx()
    v, f, want, tol = _case(nside)
    rs = _start(c, v)
    c.ray_step(rs, *CHI, maps={k: f[k].cuda() for k in KEYS}, nside_maps=nside)
    c.sync()
    _close(rs, want, tol)


def test_first_call_under_capture():
    """The geometry table a first call builds is complete when the call returns,
    not when the captured graph runs; the graph then gives the same step."""
    import paper_1210_3069_gb300 as clc
    nside = 16
    v, f, want, tol = _case(nside)
    maps = {k: f[k].cuda() for k in KEYS}
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        c = clc.Context()
        rs, rs2 = _start(c, v), _start(c, v)
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            c.ray_step(rs, *CHI, maps=maps, nside_maps=nside)
        c.ray_step(rs2, *CHI, maps=maps, nside_maps=nside)
        stream.synchronize()
        _close(rs2, want, tol)
        graph.replay()
        stream.synchronize()
        _close(rs, want, tol)
