"""Image search where rays end far from their pixels: displacements on both
sides of the reach that is searched by distance (2.5 rad) and next to the
antipode, galaxies at random and exactly on rays, where the owner of a triangle
is as far from the galaxy as the bound allows."""
import pytest
import torch

from oracle import healpix as hp, images as im
from tests.gpu_util import ctx
from workloads import synthetic

pytestmark = pytest.mark.gpu
F64 = torch.float64


@pytest.mark.parametrize("angle", [2.2, 2.45, 2.7, 3.0, 3.12, 3.1415926])
@pytest.mark.parametrize("axis", [0, 2])
def test_far_displacements(angle, axis):
    nside = 16
    w = torch.tensor(-angle, dtype=F64)
    i, j = (axis + 1) % 3, (axis + 2) % 3
    R = torch.eye(3, dtype=F64)
    R[i, i] = R[j, j] = torch.cos(w)
    R[i, j], R[j, i] = -torch.sin(w), torch.sin(w)
    x = hp.pix2vec_ring(nside, torch.arange(hp.npix(nside))) @ R.T
    z, p = synthetic.uniform_sphere(40, 3)
    ring = torch.arange(hp.npix(nside) // 2 - 2 * nside, hp.npix(nside) // 2 + 2 * nside, 3)   # next to the equator
    g = torch.cat([hp.vec_from_zphi(z, p), x[ring], x[:8], x[-8:]])
    c = ctx()
    A = synthetic.random_jacobians(x.shape[0], 0.1, 3)
    n, tri, img, _ = c.find_images(nside, x.T.contiguous().cuda(), A.reshape(-1, 4).T.contiguous().cuda(),
                                   g.T.contiguous().cuda(), 8)
    c.sync()
    wn, wt, wi, _ = im.find_images(nside, x, A, g, 8)
    assert torch.equal(n.cpu().long(), wn) and torch.equal(tri.cpu().T, wt)
    used = wt >= 0
    assert float(torch.linalg.vector_norm(img.cpu().permute(2, 1, 0) - wi, dim=-1)[used].max()) < 1e-13
