"""Library memory that captured work points to: the pointers a captured call
holds are read back from its graph, and must still be live allocations after
calls of another kind on the same context.  Nothing is replayed."""
import ctypes

import pytest
import torch

from oracle import healpix as hp
from tests.gpu_util import ctx

pytestmark = pytest.mark.gpu
F64 = torch.float64
_u = ctypes.c_uint


class _KernelNode(ctypes.Structure):   # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", ctypes.c_void_p), ("grid", _u * 3), ("block", _u * 3), ("smem", _u),
                ("params", ctypes.POINTER(ctypes.c_void_p)), ("extra", ctypes.c_void_p), ("kern", ctypes.c_void_p),
                ("ctx", ctypes.c_void_p)]


def _cuda():
    return ctypes.CDLL("libcuda.so.1")


def _ok(rc):
    assert rc == 0, rc


def _captured(stream, call, node, arg):
    """Pointer argument `arg` of kernel number `node` of the call, captured on the stream."""
    cu, st, g = _cuda(), ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    _ok(cu.cuStreamBeginCapture_v2(st, 2))   # relaxed
    try:
        call()
    finally:
        _ok(cu.cuStreamEndCapture(st, ctypes.byref(g)))
    n = ctypes.c_size_t()
    _ok(cu.cuGraphGetNodes(g, None, ctypes.byref(n)))
    nodes = (ctypes.c_void_p * n.value)()
    _ok(cu.cuGraphGetNodes(g, nodes, ctypes.byref(n)))
    p = _KernelNode()
    _ok(cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(nodes[node]), ctypes.byref(p)))
    ptr = ctypes.c_uint64.from_address(p.params[arg]).value
    _ok(cu.cuGraphDestroy(g))
    assert ptr
    return ptr


def _live(ptr):
    base, size = ctypes.c_uint64(), ctypes.c_size_t()
    return _cuda().cuMemGetAddressRange_v2(ctypes.byref(base), ctypes.byref(size), ctypes.c_uint64(ptr)) == 0


@pytest.fixture()
def own():
    """A context on a stream of its own and that stream."""
    import paper_1210_3069_gb300 as clc
    ctx()   # builds
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        c = clc.Context()
        yield c, stream
        stream.synchronize()
        c.close()


def test_source_table_outlives_image_search(own):
    c, stream = own
    counts = torch.ones(hp.npix(128), dtype=torch.int32, device="cuda")
    kappa = torch.empty(hp.npix(128), dtype=F64, device="cuda")

    def call():
        c.counts_to_kappa(counts, 128, 1.0, 1.0, kappa=kappa)
    c.counts_to_kappa_masked(counts, torch.ones(hp.npix(128), dtype=torch.uint8, device="cuda"), 128, 1.0, kappa=kappa)
    call()
    tab = _captured(stream, call, 0, 2)   # k_kappa_table(nbar, scale, tab)
    x = hp.pix2vec_ring(16, torch.arange(hp.npix(16))).T.contiguous().cuda()
    g = torch.randn(3, 100_000, dtype=F64, device="cuda")
    c.find_images(16, x, None, g, 1, matrices=False)
    stream.synchronize()
    assert _live(tab) and _captured(stream, call, 0, 2) == tab


def test_transform_buffers_outlive_spectra(own):
    c, stream = own
    nside, lmax = 16, 32
    alm = torch.ones((lmax + 1) * (lmax + 2) // 2, dtype=torch.complex128, device="cuda")
    g = torch.ones(2, hp.npix(nside), dtype=F64, device="cuda")

    def synthesis():
        c.sht_synthesis(alm, nside, lmax)

    def shear():
        c.eb_analysis(g[0], g[1], nside, lmax)
    held = []
    for call, arg in ((synthesis, 2), (shear, 4)):   # k_alm_expand(alm, lmax, rhs), k_ring_analysis(.., weight, F, ..)
        call()
        held.append((call, arg, _captured(stream, call, 0, arg)))
    A = torch.eye(2, dtype=F64, device="cuda").reshape(4, 1).expand(4, hp.npix(nside)).contiguous()
    c.lensing_spectra(A, nside, lmax)
    stream.synchronize()
    for call, arg, ptr in held:
        assert _live(ptr) and _captured(stream, call, 0, arg) == ptr


def test_ring_table_outlives_release_caches(own):
    c, stream = own
    z = torch.linspace(-1.0, 1.0, 100, dtype=F64, device="cuda")
    phi = z.abs()
    rho = torch.zeros(hp.npix(32), dtype=F64, device="cuda")

    def smooth():
        c.smooth_particles(z, phi, 32, 0.1, rho=rho)
    rs = c.rays(hp.npix(32))
    c.rays_init_pixels(rs, 32, 2.0)
    maps = {k: torch.zeros(hp.npix(32), dtype=F64, device="cuda") for k in ("a_th", "a_ph", "u_tt", "u_pp", "u_tp")}

    def step():
        c.ray_step(rs, 1.0, 2.0, 3.0, maps=maps, nside_maps=32)
    # k_smooth_particles(z, phi, sig_each, n, nside, sigma, rings, map), k_ray_step(R, V, M, nside_maps, rings, sc)
    held = [_captured(stream, smooth, 0, 6), _captured(stream, step, 0, 4)]
    c.release_caches()
    assert all(_live(p) for p in held)
