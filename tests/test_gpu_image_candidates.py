"""The candidate search of the image finder: galaxies with more candidate
triangles than the list holds, ray lengths far from 1, and rings in reach in
more than one step of a warp (a displacement of many pixels)."""
import pytest
import torch

from oracle import healpix as hp, images as im
from tests.gpu_util import ctx
from workloads import synthetic

pytestmark = pytest.mark.gpu
F64 = torch.float64


def _compare(nside, x, g, K):
    c = ctx()
    A = synthetic.random_jacobians(x.shape[0], 0.1, 3)
    n, tri, img, Ai = c.find_images(nside, x.T.contiguous().cuda(), A.reshape(-1, 4).T.contiguous().cuda(),
                                    g.T.contiguous().cuda(), K)
    c.sync()
    wn, wt, wi, wA = im.find_images(nside, x, A, g, K)
    assert torch.equal(n.cpu().long(), wn) and torch.equal(tri.cpu().T, wt)
    used = wt >= 0
    assert float(torch.linalg.vector_norm(img.cpu().permute(2, 1, 0) - wi, dim=-1)[used].max()) < 1e-13
    return wn


def test_more_candidates_than_the_list_holds():
    # a folded sky: every ray squeezed towards one direction, dozens of triangles over a galaxy
    nside = 8
    c = hp.pix2vec_ring(nside, torch.arange(hp.npix(nside)))
    e = torch.tensor([0.3, -0.2, 0.93], dtype=F64)
    e = e / e.norm()
    x = e + 0.02 * torch.randn(c.shape, dtype=F64, generator=torch.Generator().manual_seed(4))
    g = e + 0.01 * torch.randn(40, 3, dtype=F64, generator=torch.Generator().manual_seed(5))
    wn = _compare(nside, x, g, 8)
    assert int(wn.max()) > 8


@pytest.mark.parametrize("length", [1e-60, 1e-3, 3000.0, 1e80])
def test_any_ray_length(length):
    nside = 16
    x = synthetic.cored_lens_map(hp.pix2vec_ring(nside, torch.arange(hp.npix(nside))),
                                 torch.tensor([0.0, 0.6, 0.8], dtype=F64), 0.15, 0.03)[0]
    z, p = synthetic.uniform_sphere(150, 9)
    _compare(nside, x * length, hp.vec_from_zphi(z, p), 4)


def test_reach_of_many_rings():
    nside = 32
    c = hp.pix2vec_ring(nside, torch.arange(hp.npix(nside)))
    w = torch.tensor(0.9, dtype=F64)
    R = torch.tensor([[1, 0, 0], [0, torch.cos(w), -torch.sin(w)], [0, torch.sin(w), torch.cos(w)]], dtype=F64)
    z, p = synthetic.uniform_sphere(60, 12)
    _compare(nside, c @ R.T, hp.vec_from_zphi(z, p), 2)
