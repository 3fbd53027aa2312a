"""Performance cases of the lens-plane library: what users of it have it do,
through its public entry points, over the range of sizes it is used at.

listed() gives the named cases and draw() further ones of the same ranges;
prepare() makes what a program holds before the call (inputs, plans, solver
state), run() is one pass, work() the bytes and operations a pass cannot do
without, and exact() the same result from plain torch in 64 bits, sharing no
code with the library.
"""
import math

import torch

import paper_1210_3069_gb300 as clc

F64 = torch.float64
C128 = torch.complex128
DEV = torch.device("cuda") if torch.cuda.is_available() else torch.device("cpu")

# a shell of 50 Mpc/h at 1025 Mpc/h (the benchmark's plane) and its source scale
CHI_PREV, CHI, CHI_NEXT, SCALE = 975.0, 1025.0, 1075.0, 0.0048
FIELDS = ("a_th", "a_ph", "u_tt", "u_pp", "u_tp")

_CTX = []


def ctx():
    """The program's one library context (it owns scratch, FFT plans and Legendre tables)."""
    if not _CTX:
        _CTX.append(clc.Context(0))
    return _CTX[0]


# ---------------------------------------------------------------------------
# cases

def listed():
    return [
        # a small particle set onto a coarse map and its source: a call bound by latency
        dict(name="source_small", kind="source", nside=64, particles=300_000, nest=False),
        # the particles of a light-cone shell, NEST order (the order of ray bundles)
        dict(name="source_shell", kind="source", nside=2048, particles=20_000_000, nest=True),
        # the single-plane FP64 SHT solve with all lens fields, smallest and at survey resolution
        dict(name="sht_nside64", kind="sht", nside=64, lmax=128),
        dict(name="sht_nside512", kind="sht", nside=512, lmax=1024),
        # batches of planes on the tensor cores: uneven small planes, and one full class
        dict(name="batch_small", kind="batch", nside=128, planes=8, nside2=256, planes2=4),
        dict(name="batch_nside512", kind="batch", nside=512, planes=21, nside2=0, planes2=0),
        # adaptive smoothing of a shell's particles, about one particle per pixel
        dict(name="smooth_shell", kind="smooth", nside=1024, particles=12_000_000, sigma_pix=2.5),
        # the images of a source catalogue on a traced ray grid
        dict(name="images_catalogue", kind="images", nside=512, galaxies=500_000, max_images=4),
        # kappa, E, B and omega spectra of a traced sky
        dict(name="spectra_nside512", kind="spectra", nside=512, lmax=1024),
        # one light-cone plane, the library's main path: bin, SHT+MG in mixed precision, advance every ray
        dict(name="plane_nside1024", kind="plane", nside=1024, particles=12_500_000, nside_bundle=16, ncell=256),
        # the plain FP64 SHT+MG solve with the lens fields at every pixel (the reference the mixed path is held to)
        dict(name="solve_fp64_nside256", kind="solve", nside=256, nside_bundle=8, ncell=128),
        # galaxy shears through a light cone and their gradient with respect to every plane
        dict(name="gradient_nside128", kind="gradient", nside=128, lmax=256, planes=4, galaxies=100_000),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["source", "sht", "sht", "batch", "smooth", "images", "spectra", "plane", "solve", "raytrace",
                       "gradient"])
    if kind == "source":
        return dict(kind=kind, nside=2 ** rng.randint(5, 11), particles=int(_log(rng, 1e4, 2e7)),
                    nest=rng.random() < 0.5)
    if kind == "sht":
        nside = 2 ** rng.randint(4, 9)
        return dict(kind=kind, nside=nside, lmax=rng.randint(nside // 2, 2 * nside))
    if kind == "batch":
        return dict(kind=kind, nside=2 ** rng.randint(6, 8), planes=rng.randint(1, 21), nside2=512,
                    planes2=rng.randint(0, 3))
    if kind == "smooth":
        nside = 2 ** rng.randint(7, 10)
        return dict(kind=kind, nside=nside, particles=int(_log(rng, 1e4, 12.0 * nside * nside)),
                    sigma_pix=rng.uniform(1.0, 4.0))
    if kind == "images":
        return dict(kind=kind, nside=2 ** rng.randint(6, 10), galaxies=int(_log(rng, 3e3, 1e6)),
                    max_images=rng.randint(1, 4))
    if kind == "spectra":
        nside = 2 ** rng.randint(5, 9)
        return dict(kind=kind, nside=nside, lmax=rng.randint(nside // 2, 2 * nside))
    if kind == "plane":
        shape = rng.choice([(128, 4, 128), (128, 2, 256), (256, 4, 256), (512, 8, 256), (512, 16, 128)])
        return dict(kind=kind, nside=shape[0], particles=int(_log(rng, 1e5, 3e6)), nside_bundle=shape[1],
                    ncell=shape[2])
    if kind == "solve":
        shape = rng.choice([(64, 4, 64), (128, 4, 128), (128, 8, 64), (256, 8, 128), (256, 4, 256)])
        return dict(kind=kind, nside=shape[0], nside_bundle=shape[1], ncell=shape[2])
    if kind == "raytrace":
        nside = 2 ** rng.randint(5, 8)
        return dict(kind=kind, nside=nside, lmax=rng.randint(nside, 2 * nside), planes=rng.randint(2, 6))
    nside = 2 ** rng.randint(5, 7)
    return dict(kind=kind, nside=nside, lmax=rng.randint(nside, 2 * nside), planes=rng.randint(1, 4),
                galaxies=int(_log(rng, 1e3, 1e5)))


# ---------------------------------------------------------------------------
# HEALPix (Gorski et al. 2005)

def _rings(nside):
    """z, sin theta, first pixel, pixel count and first longitude of the 4 nside - 1 rings."""
    i = torch.arange(1, 4 * nside, dtype=torch.int64, device=DEV)
    ip = torch.minimum(i, 4 * nside - i)
    cap = ip < nside
    a = ip.to(F64) ** 2 / (3.0 * nside * nside)
    zb = 4.0 / 3.0 - 2.0 * i.to(F64) / (3.0 * nside)
    z = torch.where(cap, torch.where(i < 2 * nside, 1.0 - a, a - 1.0), zb)
    s = torch.where(cap, torch.sqrt(a * (2.0 - a)), torch.sqrt((1 - zb) * (1 + zb)))
    n = torch.where(cap, 4 * ip, torch.full_like(ip, 4 * nside))
    first = torch.cumsum(n, 0) - n
    phi0 = torch.where(cap | ((i - nside) % 2 == 0), math.pi / n.to(F64), torch.zeros_like(z))
    return z, s, first, n, phi0


def _centres(nside):
    """(z, sin theta, phi) of every RING pixel centre."""
    z, s, first, n, phi0 = _rings(nside)
    r = torch.repeat_interleave(torch.arange(z.numel(), device=DEV), n)
    j = torch.arange(12 * nside * nside, device=DEV) - first[r]
    return z[r], s[r], phi0[r] + 2.0 * math.pi * j.to(F64) / n[r].to(F64)


def _vec(z, phi, s=None):
    s = torch.sqrt((1 - z) * (1 + z)) if s is None else s
    return torch.stack([s * torch.cos(phi), s * torch.sin(phi), z], -1)


def _ang2pix(nside, z, phi, nest=False):
    za = z.abs()
    tt = torch.remainder(phi * (2.0 / math.pi), 4.0)
    t1, t2 = nside * (0.5 + tt), nside * z * 0.75
    jp, jm = torch.floor(t1 - t2).long(), torch.floor(t1 + t2).long()
    ntt = torch.floor(tt).long().clamp(max=3)
    tp = tt - ntt
    tmp = nside * torch.sqrt(3.0 * (1.0 - za))
    kp = torch.floor(tp * tmp).long()
    km = torch.floor((1.0 - tp) * tmp).long()
    belt = za <= 2.0 / 3.0
    if not nest:
        ir = nside + 1 + jp - jm
        ip = torch.remainder((jp + jm - nside + (1 - (ir & 1)) + 1) // 2, 4 * nside)
        eq = 2 * nside * (nside - 1) + (ir - 1) * 4 * nside + ip
        ic = kp + km + 1
        q = torch.remainder(torch.floor(tt * ic).long(), 4 * ic)
        cap = torch.where(z > 0, 2 * ic * (ic - 1) + q, 12 * nside * nside - 2 * ic * (ic + 1) + q)
        return torch.where(belt, eq, cap)
    fp, fm = jp // nside, jm // nside
    feq = torch.where(fp == fm, torch.where(fp == 4, fp, fp + 4), torch.where(fp < fm, fp, fm + 8))
    kp, km = kp.clamp(max=nside - 1), km.clamp(max=nside - 1)
    face = torch.where(belt, feq, torch.where(z >= 0, ntt, ntt + 8))
    ix = torch.where(belt, jm % nside, torch.where(z >= 0, nside - km - 1, kp))
    iy = torch.where(belt, nside - jp % nside - 1, torch.where(z >= 0, nside - kp - 1, km))
    p = face * nside * nside
    for b in range(13):
        p = p + (((ix >> b) & 1) << (2 * b)) + (((iy >> b) & 1) << (2 * b + 1))
    return p


# ---------------------------------------------------------------------------
# inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _uniform(n, g):
    return 2.0 * torch.rand(n, generator=g, dtype=F64, device=DEV) - 1.0, \
        2.0 * math.pi * torch.rand(n, generator=g, dtype=F64, device=DEV)


def _waves(m, kmin, kmax, g):
    """Wave vectors of equal variance per octave and phases."""
    k = kmin * (kmax / kmin) ** torch.rand(m, generator=g, dtype=F64, device=DEV)
    kz, kp = _uniform(m, g)
    return k[:, None] * _vec(kz, kp), 2.0 * math.pi * torch.rand(m, generator=g, dtype=F64, device=DEV)


def _particles(n, g):
    """Clustered particles: uniform points moved along the gradient of a random potential."""
    z, phi = _uniform(n, g)
    k, ph = _waves(64, 4.0, 200.0, g)
    amp = 0.6 / (k.norm(dim=1) ** 2 * math.sqrt(32.0))
    zo, po = torch.empty_like(z), torch.empty_like(phi)
    for s in range(0, n, 1 << 20):
        v = _vec(z[s:s + (1 << 20)], phi[s:s + (1 << 20)]).float()
        w = v + torch.sin(v @ k.T.float() + ph.float()) @ (amp[:, None] * k).float()
        w = w.double()
        w = w / w.norm(dim=1, keepdim=True)
        zo[s:s + (1 << 20)] = w[:, 2].clamp(-1.0, 1.0)
        p = torch.atan2(w[:, 1], w[:, 0])
        po[s:s + (1 << 20)] = torch.where(p < 0, p + 2.0 * math.pi, p)
    return zo, po.clamp(max=6.283185307179586)


def _delta(nside, g, kmax=None):
    """A lognormal density contrast at the RING pixel centres."""
    z, s, phi = _centres(nside)
    k, ph = _waves(128, 2.0, kmax or 2.0 * nside, g)
    out = torch.empty_like(z)
    sig2 = math.log(2.0)
    for a in range(0, z.numel(), 1 << 20):
        v = _vec(z[a:a + (1 << 20)], phi[a:a + (1 << 20)], s[a:a + (1 << 20)]).float()
        f = torch.cos(v @ k.T.float() + ph.float()).sum(1).double() * math.sqrt(2.0 * sig2 / 128)
        out[a:a + (1 << 20)] = torch.exp(f - 0.5 * sig2) - 1.0
    return out


def _lensed_sky(nside, g):
    """Source positions x [3, npix] and matrices A [4, npix] of the rays of a traced light cone:
    deflections of some arc minutes from many plane waves, one stronger lens, weak distortions."""
    z, s, phi = _centres(nside)
    n = _vec(z, phi, s)
    k, ph = _waves(48, 3.0, 300.0, g)
    amp = 3e-4 / (k.norm(dim=1) * math.sqrt(24.0))
    d = torch.sin(n @ k.T + ph) @ (amp[:, None] * k)
    zc, pc = _uniform(1, g)
    c = _vec(zc, pc)[0]
    e = c - n * (n @ c)[:, None]
    th = torch.arccos((n @ c).clamp(-1, 1))
    e = e / e.norm(dim=1, keepdim=True).clamp(min=1e-300)
    b = 2e-3 * (torch.sqrt(th * th + 2.5e-5) - 5e-3) / th.clamp(min=1e-9) * ((1 + torch.cos(th)) / 2) ** 2
    x = n + d - n * (n * d).sum(1, keepdim=True) + b[:, None] * e
    x = x / x.norm(dim=1, keepdim=True)
    A = torch.eye(2, dtype=F64, device=DEV).reshape(4, 1) + torch.stack(
        [0.02 * torch.sin(n @ k[i * 8:(i + 1) * 8].T + ph[i * 8:(i + 1) * 8]).sum(1) / 2 for i in range(4)])
    return x.T.contiguous(), A.contiguous()


def _chi(planes):
    """Plane distances (and the source sphere) and source scales of a light cone to z about 1.5."""
    d = 3000.0 / planes
    chi = [(m + 0.5) * d for m in range(planes)] + [planes * d]
    return chi, [0.75 * c * (1.0 + c / 2400.0) * d / 2997.92458 ** 2 * 0.7 for c in chi[:planes]]


def _mg(case, precision):
    nf = case["nside"]
    return clc.mg_params(nf // 4, nf // 2, case["nside_bundle"], ncell=case["ncell"], tol=1e-10, precision=precision)


def _gradient_inputs(case, seed):
    g = _gen(seed)
    chi, scale = _chi(case["planes"])
    ka = torch.stack([sc * _delta(case["nside"], g, kmax=1.0 * case["nside"]) for sc in scale])
    gz, gp = _uniform(case["galaxies"], g)
    gchi = (0.25 + 0.75 * torch.rand(case["galaxies"], generator=g, dtype=F64, device=DEV)) * chi[-1]
    target = 0.02 * torch.randn(2, case["galaxies"], generator=g, dtype=F64, device=DEV)
    return ka, chi, gz, gp, gchi, target


def _raytrace_inputs(case, seed):
    g = _gen(seed)
    chi, scale = _chi(case["planes"])
    return [sc * _delta(case["nside"], g, kmax=1.0 * case["nside"]) for sc in scale], chi


def _solve_input(case, seed):
    return SCALE * _delta(case["nside"], _gen(seed))


def _smooth_inputs(case, seed):
    z, phi = _particles(case["particles"], _gen(seed))
    return z, phi, case["sigma_pix"] * math.sqrt(4.0 * math.pi / (12.0 * case["nside"] ** 2))


def _batch_sizes(case):
    return [(case["nside"], case["planes"]), (case["nside2"], case["planes2"])][:2 if case["planes2"] else 1]


def _batch_maps(case, seed):
    g = _gen(seed)
    return [[_delta(ns, g) for _ in range(p)] for ns, p in _batch_sizes(case)]


# ---------------------------------------------------------------------------
# one pass

def prepare(case, seed):
    kind, c = case["kind"], ctx()
    st = dict(case, ctx=c)
    npx = 12 * case["nside"] ** 2
    if kind in ("source", "plane"):
        st["z"], st["phi"] = _particles(case["particles"], _gen(seed))
        st["counts"] = torch.zeros(npx, dtype=torch.int32, device=DEV)
        st["kappa"] = torch.empty(npx, dtype=F64, device=DEV)
    if kind == "sht":
        st["kappa"] = _delta(case["nside"], _gen(seed))
    if kind == "batch":
        st["maps"] = [m for cls in _batch_maps(case, seed) for m in cls]
        st["out"] = [{f: torch.empty(p, 12 * ns * ns, dtype=F64, device=DEV) for f in ("psi",) + FIELDS}
                     for ns, p in _batch_sizes(case)]
        st["views"] = [{f: t[i] for f, t in o.items()} for o in st["out"] for i in range(o["psi"].shape[0])]
        ns = [n for n, p in _batch_sizes(case) for _ in range(p)]
        st["plan"] = c.sht_plan(ns, [2 * n for n in ns], derivatives=True, graph=True, tune=False)
    if kind == "smooth":
        st["z"], st["phi"], st["sigma"] = _smooth_inputs(case, seed)
    if kind in ("images", "spectra"):
        st["x"], st["A"] = _lensed_sky(case["nside"], _gen(seed))
    if kind == "images":
        st["g"] = _vec(*_uniform(case["galaxies"], _gen(seed + 1))).T.contiguous()
    if kind == "plane":
        st["rays"] = c.rays(npx)
        st["sol"] = c.solution(case["nside"], _mg(case, clc.MIXED))
    if kind == "solve":
        st["kappa"] = _solve_input(case, seed)
        st["sol"] = c.solution(case["nside"], _mg(case, clc.FP64))
    if kind == "raytrace":
        st["kappas"], st["chi"] = _raytrace_inputs(case, seed)
        st["rays"] = c.rays(npx)
    if kind == "gradient":
        st["kappas"], st["chi"], st["gz"], st["gphi"], st["gchi"], st["target"] = _gradient_inputs(case, seed)
    return st


def _source(st, ordering):
    st["counts"].zero_()
    st["ctx"].bin_particles(st["z"], st["phi"], st["nside"], ordering=ordering, counts=st["counts"])
    nbar = st["particles"] / (12 * st["nside"] ** 2)
    return st["ctx"].counts_to_kappa(st["counts"], st["nside"], nbar, SCALE, kappa=st["kappa"])


def run(st):
    c, kind, ns = st["ctx"], st["kind"], st["nside"]
    if kind == "source":
        _source(st, clc.NEST if st["nest"] else clc.RING)
        return {"counts": st["counts"], "kappa": st["kappa"]}
    if kind == "sht":
        return c.poisson_sht(st["kappa"], ns, st["lmax"])
    if kind == "batch":
        st["plan"].execute(st["maps"], st["views"])
        return st["out"]
    if kind == "smooth":
        return c.smooth_particles(st["z"], st["phi"], ns, sigma=st["sigma"])
    if kind == "images":
        return c.find_images(ns, st["x"], st["A"], st["g"], st["max_images"])
    if kind == "spectra":
        return c.lensing_spectra(st["A"], ns, st["lmax"], x=st["x"])
    if kind == "solve":
        return c.poisson_shtmg(st["kappa"], ns, st["sol"], derivatives=True, check=False)
    if kind == "plane":
        kappa = _source(st, clc.RING)
        c.poisson_shtmg(kappa, ns, st["sol"], check=False)
        c.rays_init_pixels(st["rays"], ns, CHI, st["nside_bundle"])
        c.ray_step(st["rays"], CHI_PREV, CHI, CHI_NEXT, sol=st["sol"])
    if kind == "raytrace":
        c.rays_init_pixels(st["rays"], ns, st["chi"][0])
        c.raytrace_planes(clc.SOLVER_SHT, clc.mg_params(ns, st["lmax"], 1), st["kappas"], ns, st["chi"], st["rays"])
    if kind == "gradient":
        k = st["kappas"].clone().requires_grad_(True)
        gam = clc.galaxy_shear(c, k, ns, st["lmax"], st["chi"], st["gz"], st["gphi"], st["gchi"])
        ((gam - st["target"]) ** 2).sum().backward()
        return {"gamma": gam, "grad": k.grad}
    r = st["rays"]
    return {"x": r.x, "beta": r.beta, "A": r.A, "Ap": r.Ap}


def work(case):
    """Each input read and each output written once; operations of the method:
    a Legendre sum is one complex multiply-add (4 flops) per (l, m) and northern ring, a ring FFT 2.5 n log2 n."""
    kind, ns = case["kind"], case["nside"]
    px = 12 * ns * ns

    def leg(ns, lmax):
        return 4.0 * (lmax + 1) * (lmax + 2) / 2 * 2 * ns

    def fft(ns):
        return 12.0 * ns * ns * 2.5 * math.log2(4 * ns)

    if kind == "source":
        return {"bytes": 16 * case["particles"] + 12 * px, "flops": 10 * case["particles"] + 3 * px}
    if kind == "sht":
        return {"bytes": 56 * px, "flops": 4 * leg(ns, case["lmax"]) + 7 * fft(ns)}
    if kind == "batch":
        return {"bytes": sum(56 * 12 * n * n * p for n, p in _batch_sizes(case)),
                "flops": sum(p * (4 * leg(n, 2 * n) + 7 * fft(n)) for n, p in _batch_sizes(case))}
    if kind == "smooth":
        area = math.pi * case["sigma_pix"] ** 2
        return {"bytes": 16 * case["particles"] + 8 * px, "flops": 14 * area * case["particles"]}
    if kind == "images":
        return {"bytes": 56 * px + case["galaxies"] * (24 + 4 + 64 * case["max_images"]),
                "flops": 540 * case["galaxies"]}
    if kind == "spectra":
        return {"bytes": 56 * px + 32 * (case["lmax"] + 1), "flops": 8 * leg(ns, case["lmax"]) + 4 * fft(ns)}
    if kind in ("plane", "solve"):
        cells = 12 * case["nside_bundle"] ** 2 * case["ncell"] ** 2
        sht = 2 * leg(ns // 4, ns // 2) + 2 * fft(ns // 4)
        # ten V-cycles of about 40 operations per fine cell and its coarser levels; the ray step's 530
        if kind == "solve":
            return {"bytes": 48 * px, "flops": sht + 400.0 * cells + 300.0 * px}
        return {"bytes": 16 * case["particles"] + 12 * px + 112 * px, "flops": sht + 400.0 * cells + 530.0 * px}
    if kind == "raytrace":
        return {"bytes": case["planes"] * 8 * px + 112 * px,
                "flops": case["planes"] * (4 * leg(ns, case["lmax"]) + 6 * fft(ns) + 530.0 * px)}
    planes, gal = case["planes"], case["galaxies"]
    return {"bytes": 16 * planes * px + 56 * gal,
            "flops": planes * (3 * (4 * leg(ns, case["lmax"]) + 6 * fft(ns)) + 4.0 * 530 * gal)}


# ---------------------------------------------------------------------------
# the same in plain torch, 64 bits

def _lambda(nside, lmax, m0, m1):
    """lambda_lm(z) [m, l, ring] of m0 <= m < m1, l <= lmax + 1 on all rings, by the recurrence in l on
    mantissas with a power-of-two exponent."""
    z, s, _, _, _ = _rings(nside)
    m = torch.arange(m0, m1, device=DEV)
    mf = m.to(F64)[:, None]
    k = torch.arange(1, m1 + 1, dtype=F64, device=DEV)
    ln = torch.cat([torch.zeros(1, dtype=F64, device=DEV), 0.5 * torch.cumsum(torch.log2((2 * k + 1) / (2 * k)), 0)])
    lg = ln[m][:, None] + 0.5 * math.log2(1.0 / (4.0 * math.pi)) + mf * torch.log2(s)
    e = torch.floor(lg)
    pmm = torch.exp2(lg - e) * torch.where(m % 2 == 1, -1.0, 1.0).to(F64)[:, None]
    out = torch.zeros(m1 - m0, lmax + 2, z.numel(), dtype=F64, device=DEV)
    p1 = torch.zeros_like(pmm)
    p2 = torch.zeros_like(pmm)
    scale = torch.exp2(e.clamp(min=-1000.0))
    for l in range(m0, lmax + 2):
        on = m[:, None] <= l
        a = torch.sqrt((4.0 * l * l - 1.0) / (l * l - mf * mf).clamp(min=1.0))
        b = torch.sqrt(((l - 1.0) ** 2 - mf * mf).clamp(min=0.0) / max(4.0 * (l - 1.0) ** 2 - 1.0, 1.0))
        p0 = torch.where(m[:, None] == l, pmm, a * (z * p1 - b * p2))
        out[:, l] = torch.where(on, p0 * scale, 0.0)
        p2, p1 = p1, torch.where(on, p0, 0.0)
        if l % 8 == 7:
            big = p1.abs() > 2.0 ** 400
            p1 = torch.where(big, p1 * 2.0 ** -400, p1)
            p2 = torch.where(big, p2 * 2.0 ** -400, p2)
            e = torch.where(big, e + 400.0, e)
            scale = torch.exp2(e.clamp(min=-1000.0))
    return out


def _blocks(nside, lmax):
    """(m0, m1, lambda) over blocks of orders of about a gigabyte."""
    step = max(1, int(1e9 / (8.0 * (lmax + 2) * 4 * nside)))
    for m0 in range(0, lmax + 1, step):
        m1 = min(m0 + step, lmax + 1)
        yield m0, m1, _lambda(nside, lmax, m0, m1)


def _ring_analysis(maps, nside, lmax):
    """F [P, m, ring] = weight sum_j map_j e^{-i m phi_j}."""
    _, _, first, n, phi0 = _rings(nside)
    m = torch.arange(lmax + 1, device=DEV)
    cols = []
    for f, k, p0 in zip(first.tolist(), n.tolist(), phi0.tolist()):
        spec = torch.fft.fft(maps[:, f:f + k])
        cols.append(spec[:, m % k] * torch.exp(-1j * p0 * m.to(C128)))
    return torch.stack(cols, -1) * (4.0 * math.pi / (12.0 * nside * nside))


def _ring_synthesis(G, nside, lmax):
    """Map values [P, npix] of Fourier coefficients G [P, m, ring]."""
    _, _, first, n, phi0 = _rings(nside)
    m = torch.arange(lmax + 1, device=DEV)
    two = torch.where(m == 0, 1.0, 2.0).to(F64)
    out = []
    for r, (k, p0) in enumerate(zip(n.tolist(), phi0.tolist())):
        g = G[:, :, r] * (two * torch.exp(1j * p0 * m.to(C128)))
        if lmax + 1 > k:
            g = torch.zeros(G.shape[0], k, dtype=C128, device=DEV).index_add(1, m % k, g)
            out.append(torch.fft.ifft(g).real * k)
        else:
            out.append(torch.fft.ifft(g, n=k).real * k)
    return torch.cat(out, 1)


def _poisson(kappa, nside, lmax, derivs=True):
    """psi and the lens fields [P, npix] of the maps kappa [P, npix]."""
    z, s, _, _, _ = _rings(nside)
    F = _ring_analysis(kappa, nside, lmax)
    l = torch.arange(lmax + 2, dtype=F64, device=DEV)
    inv = torch.where((l > 0) & (l <= lmax), -1.0 / (l * (l + 1)).clamp(min=1.0), torch.zeros_like(l))
    parts = []
    for m0, m1, lam in _blocks(nside, lmax):
        lamc = lam.to(C128)
        klm = torch.einsum("mlr,pmr->pml", lamc, F[:, m0:m1])
        m = torch.arange(m0, m1, dtype=F64, device=DEV)[:, None]
        psi = klm * inv
        if m0 == 0:
            psi = torch.cat([psi[:, :1].real.to(C128), psi[:, 1:]], 1)
        cols = [psi]
        if derivs:
            eps = torch.sqrt((l * l - m * m).clamp(min=0.0) / (4 * l * l - 1).clamp(min=1.0))
            up, dn = torch.zeros_like(psi), torch.zeros_like(psi)
            up[..., 1:] = psi[..., :-1]
            dn[..., :-1] = psi[..., 1:]
            ep = torch.sqrt(((l + 1) ** 2 - m * m).clamp(min=0.0) / (4 * (l + 1) ** 2 - 1))
            cols += [(l - 1) * eps * up - (l + 2) * ep * dn, -l * (l + 1) * psi]
        parts.append(torch.einsum("mlr,qpml->qpmr", lamc, torch.stack(cols)))
    G = torch.cat(parts, 2)
    if not derivs:
        return {"psi": _ring_synthesis(G[0], nside, lmax)}
    mm = torch.arange(lmax + 1, dtype=F64, device=DEV)[:, None]
    g0, g1, g2 = G
    upp = (-mm * mm * g0 + z * g1) / (s * s)
    spec = {"psi": g0, "a_th": -g1 / s, "a_ph": -1j * mm * g0 / s, "u_tt": g2 - upp, "u_pp": upp,
            "u_tp": 1j * mm * (g1 - z * g0) / (s * s)}
    return {k: _ring_synthesis(v, nside, lmax) for k, v in spec.items()}


def _interp(nside, theta, phi):
    """Pixels and weights [..., 8] of the ring-bilinear interpolation."""
    z, s, first, n, phi0 = _rings(nside)
    tr = torch.atan2(s, z)
    nr = tr.numel()
    r = torch.searchsorted(tr, theta.detach().contiguous(), right=True) - 1
    north, south = r < 0, r >= nr - 1
    ra, rb = r.clamp(0, nr - 1), (r + 1).clamp(0, nr - 1)
    gap = torch.where(rb > ra, tr[rb] - tr[ra], torch.ones_like(theta))
    w = torch.where(north, theta / tr[0], torch.where(south, (math.pi - theta) / (math.pi - tr[-1]),
                                                      (theta - tr[ra]) / gap))
    pole = north | south

    def pair(q):
        t = (phi - phi0[q]) * n[q] / (2.0 * math.pi)
        j = torch.floor(t.detach())
        f = t - j
        j = j.long()
        return first[q] + torch.remainder(j, n[q]), first[q] + torch.remainder(j + 1, n[q]), f

    a0, a1, fa = pair(ra)
    b0, b1, fb = pair(rb)
    wa = torch.where(pole, w, 1.0 - w)
    wb = torch.where(pole, torch.zeros_like(w), w)
    wp = torch.where(pole, 0.25 * (1.0 - w), torch.zeros_like(w))
    p0 = torch.where(north, first[0], first[-1])
    return torch.stack([a0, a1, b0, b1, p0, p0 + 1, p0 + 2, p0 + 3], -1), \
        torch.stack([wa * (1 - fa), wa * fa, wb * (1 - fb), wb * fb, wp, wp, wp, wp], -1)


def _angles(v):
    th = torch.atan2(torch.sqrt(v[..., 0] ** 2 + v[..., 1] ** 2), v[..., 2])
    ph = torch.atan2(v[..., 1], v[..., 0])
    return th, torch.where(ph < 0, ph + 2.0 * math.pi, ph)


def _frame(v):
    """theta-hat, phi-hat at unit vectors."""
    rho = torch.sqrt(v[..., 0] ** 2 + v[..., 1] ** 2)
    zero = torch.zeros_like(rho)
    return torch.stack([v[..., 2] * v[..., 0] / rho, v[..., 2] * v[..., 1] / rho, -rho], -1), \
        torch.stack([-v[..., 1] / rho, v[..., 0] / rho, zero], -1)


def _dot(a, b):
    return (a * b).sum(-1)


def _map_lens(fields, nside):
    """The lens fields at unit vectors, interpolated as tangent vectors and tensors."""
    t, q = _frame(_vec(*(lambda z, s, p: (z, p, s))(*_centres(nside))))
    a3 = fields["a_th"][:, None] * t + fields["a_ph"][:, None] * q
    U3 = fields["u_tt"][:, None, None] * t[:, :, None] * t[:, None] + \
        fields["u_pp"][:, None, None] * q[:, :, None] * q[:, None] + \
        fields["u_tp"][:, None, None] * (t[:, :, None] * q[:, None] + q[:, :, None] * t[:, None])

    def at(v):
        ix, w = _interp(nside, *_angles(v))
        a = sum(a3[ix[:, k]] * w[:, k, None] for k in range(8))
        U = sum(U3[ix[:, k]] * w[:, k, None, None] for k in range(8))
        e = _frame(v)
        return [_dot(a, e[0]), _dot(a, e[1])] + \
            [torch.einsum("mi,mij,mj->m", e[i], U, e[j]) for i, j in ((0, 0), (1, 1), (0, 1))]
    return at


def _turn(v, k, w):
    """v rotated about the unit axis k by the angle with (cos, sin) w."""
    return v * w[0][:, None] + torch.cross(k, v, dim=1) * w[1][:, None] + k * (_dot(k, v) * (1 - w[0]))[:, None]


def _carry(A, v0, v1):
    """A [M, 2, 2] parallel transported from v0 to v1."""
    ax = torch.cross(v0, v1, dim=1)
    s = torch.sqrt(_dot(ax, ax).clamp(min=1e-300))
    k = ax / s[:, None]
    e0 = [_turn(e, k, (_dot(v0, v1), s)) for e in _frame(v0)]
    Q = torch.stack([torch.stack([_dot(a, b) for b in e0], -1) for a in _frame(v1)], -2)
    return Q @ A @ Q.transpose(1, 2)


def _step(st, lens, cp, cn, cx):
    """One plane of the ray recursion on (x, beta, A, Ap) with A as [M, 2, 2]."""
    x, be, A, Ap = st
    n = x / x.norm(dim=1, keepdim=True)
    at, ap, utt, upp, utp = lens(n)
    U = torch.stack([torch.stack([utt, utp], -1), torch.stack([utp, upp], -1)], -2)
    c, d = cn / cx * (cx - cp) / (cn - cp), (cx - cn) / cx
    An = (1 - c) * Ap + c * A - d * (U @ A)
    t, q = _frame(n)
    al = at[:, None] * t + ap[:, None] * q
    am = torch.sqrt(_dot(al, al).clamp(min=1e-300))
    be = _turn(be, torch.cross(n, al, dim=1) / am[:, None], (torch.cos(am), torch.sin(am)))
    xb = _dot(x, be)
    dc = (cx - cn) * (cx + cn)
    x1 = x + (dc / (xb + torch.sqrt(xb * xb + dc)))[:, None] * be
    n1 = x1 / x1.norm(dim=1, keepdim=True)
    return x1, be, _carry(An, n, n1), _carry(A, n, n1)


def _start(v, chi):
    eye = torch.eye(2, dtype=F64, device=DEV).expand(v.shape[0], 2, 2)
    return chi * v, v, eye, eye


def _rays_out(st):
    x, be, A, Ap = st
    return {"x": x.T.contiguous(), "beta": be.T.contiguous(), "A": A.reshape(-1, 4).T.contiguous(),
            "Ap": Ap.reshape(-1, 4).T.contiguous()}


def _patch_fields(kappa, nf, nb, n):
    """Lens fields at every RING pixel centre from the patch solves: the SHT potential on the patch edges,
    the discrete Laplacian solved directly (sine transform in phi', tridiagonal in theta'), fourth-order
    differences, bilinear interpolation, rotation to the global basis."""
    ns, lmax = nf // 4, nf // 2
    zf, sf, pf = _centres(nf)
    ks = torch.zeros(12 * ns * ns, dtype=F64, device=DEV).index_add(0, _ang2pix(ns, zf, pf), kappa) / 16.0
    psi = _poisson(ks[None], ns, lmax, derivs=False)["psi"][0]
    h = 4.0 * math.sqrt(math.pi / 3.0) / nb / n
    d = (torch.arange(-1, n + 1, dtype=F64, device=DEV) + 0.5 - n / 2.0) * h
    d[0], d[-1] = -0.5 * n * h, 0.5 * n * h
    th = math.pi / 2 + d
    pv = torch.stack([torch.sin(th)[:, None] * torch.cos(d), torch.sin(th)[:, None] * torch.sin(d),
                      torch.cos(th)[:, None].expand(n + 2, n + 2)], -1)
    t = math.pi / 2 + (torch.arange(n, dtype=F64, device=DEV) + 0.5 - n / 2.0) * h
    si = torch.sin(t)
    aS, aN, b = torch.sin(t + h / 2) / (h * h * si), torch.sin(t - h / 2) / (h * h * si), 1.0 / (h * h * si * si)
    k = torch.arange(1, n + 1, dtype=F64, device=DEV)
    S = torch.sin(math.pi / n * k[:, None] * (torch.arange(n, dtype=F64, device=DEV) + 0.5))
    back = S.T * torch.where(k < n, 2.0 / n, 1.0 / n)
    dia = -(aS + aN)
    dia[0] -= aN[0]
    dia[-1] -= aS[-1]
    dia = dia[:, None] - 4.0 * b[:, None] * torch.sin(math.pi * k / (2 * n)) ** 2
    cp = torch.empty(n, n, dtype=F64, device=DEV)
    den = torch.empty_like(cp)
    for i in range(n):
        den[i] = dia[i] - (aN[i] * cp[i - 1] if i else 0.0)
        cp[i] = aS[i] / den[i]
    D1 = torch.tensor([[-25., 48, -36, 16, -3], [-3, -10, 18, -6, 1], [1, -8, 0, 8, -1]], dtype=F64, device=DEV) / 12
    D2 = torch.tensor([[35., -104, 114, -56, 11], [11, -20, 6, 4, -1], [-1, 16, -30, 16, -1]], dtype=F64,
                      device=DEV) / 12

    def dmat(D, odd):
        M = torch.zeros(n, n, dtype=F64, device=DEV)
        for i in range(n):
            o = min(i, n - 1 - i, 2)
            if i < 2:
                M[i, :5] = D[o]
            elif i > n - 3:
                M[i, n - 5:] = odd * D[o].flip(0)
            else:
                M[i, i - 2:i + 3] = D[2]
        return M

    M1, M2 = dmat(D1, -1.0) / h, dmat(D2, 1.0) / (h * h)
    home = _ang2pix(nb, zf, pf)
    order = torch.argsort(home, stable=True)
    npx, per = zf.numel(), zf.numel() // (12 * nb * nb)
    zb, sb, pb = _centres(nb)
    out = [torch.empty(npx, dtype=F64, device=DEV) for _ in range(5)]
    for b0 in range(0, 12 * nb * nb, 64):
        b1 = min(b0 + 64, 12 * nb * nb)
        zc, sc, pc = zb[b0:b1], sb[b0:b1], pb[b0:b1]
        zero = torch.zeros_like(zc)
        R = torch.stack([torch.stack([sc * torch.cos(pc), sc * torch.sin(pc), zc], -1),
                         torch.stack([-torch.sin(pc), torch.cos(pc), zero], -1),
                         torch.stack([-zc * torch.cos(pc), -zc * torch.sin(pc), sc], -1)], -2)
        tg, pg = _angles(torch.einsum("bji,xyj->bxyi", R, pv))
        ix, w = _interp(ns, tg, pg)
        base = (psi[ix] * w).sum(-1)
        ix, w = _interp(nf, tg[:, 1:-1, 1:-1], pg[:, 1:-1, 1:-1])
        f = (kappa[ix] * w).sum(-1)
        # solve for the correction to the SHT potential: L e = f - L base, zero on the edges
        e = base[:, 1:-1, 1:-1]
        up, dn = base[:, :-2, 1:-1].clone(), base[:, 2:, 1:-1].clone()
        lf, rt = base[:, 1:-1, :-2].clone(), base[:, 1:-1, 2:].clone()
        up[:, 0] = 2 * up[:, 0] - e[:, 0]
        dn[:, -1] = 2 * dn[:, -1] - e[:, -1]
        lf[:, :, 0] = 2 * lf[:, :, 0] - e[:, :, 0]
        rt[:, :, -1] = 2 * rt[:, :, -1] - e[:, :, -1]
        rhs = f - (aS[:, None] * (dn - e) - aN[:, None] * (e - up) + b[:, None] * (lf - 2 * e + rt))
        y = torch.einsum("kj,bij->bik", S, rhs)
        for i in range(n):
            y[:, i] = (y[:, i] - (aN[i] * y[:, i - 1] if i else 0.0)) / den[i]
        for i in range(n - 2, -1, -1):
            y[:, i] -= cp[i] * y[:, i + 1]
        u = e + torch.einsum("jk,bik->bij", back, y)
        up_ = torch.einsum("jk,bik->bij", M1, u)
        part = torch.stack([torch.einsum("ik,bkj->bij", M1, u), up_, torch.einsum("ik,bkj->bij", M2, u),
                            torch.einsum("jk,bik->bij", M2, u), torch.einsum("ik,bkj->bij", M1, up_)], 1)
        pix = order[b0 * per:b1 * per]
        nv = _vec(zf[pix], pf[pix], sf[pix])
        bi = home[pix] - b0
        Rp = R[bi]
        v = torch.einsum("mij,mj->mi", Rp, nv)
        tp, pp = _angles(v)
        pp = torch.where(pp > math.pi, pp - 2 * math.pi, pp)
        xx, yy = (tp - math.pi / 2) / h + n / 2.0 - 0.5, pp / h + n / 2.0 - 0.5
        i0, j0 = torch.floor(xx).clamp(0, n - 2), torch.floor(yy).clamp(0, n - 2)
        fx, fy = (xx - i0)[:, None], (yy - j0)[:, None]
        i0, j0 = i0.long(), j0.long()
        q = (1 - fx) * (1 - fy) * part[bi, :, i0, j0] + fx * (1 - fy) * part[bi, :, i0 + 1, j0] + \
            (1 - fx) * fy * part[bi, :, i0, j0 + 1] + fx * fy * part[bi, :, i0 + 1, j0 + 1]
        s, c = torch.sin(tp), torch.cos(tp)
        al = torch.stack([-q[:, 0], -q[:, 1] / s], -1)
        upp, utp = q[:, 3] / (s * s) + c / s * q[:, 0], q[:, 4] / s - c * q[:, 1] / (s * s)
        U = torch.stack([torch.stack([q[:, 2], utp], -1), torch.stack([utp, upp], -1)], -2)
        local = [torch.einsum("mji,mj->mi", Rp, x) for x in _frame(v)]
        Q = torch.stack([torch.stack([_dot(x, y_) for y_ in local], -1) for x in _frame(nv)], -2)
        al = torch.einsum("mab,mb->ma", Q, al)
        U = Q @ U @ Q.transpose(1, 2)
        for o, val in zip(out, (al[:, 0], al[:, 1], U[:, 0, 0], U[:, 1, 1], U[:, 0, 1])):
            o[pix] = val
    return out


def _smoothed(z, phi, nside, sigma):
    """Unit masses spread over the pixel centres within sigma with weights 1 - (theta / sigma)^2."""
    zr, sr, first, n, phi0 = _rings(nside)
    tr = torch.atan2(sr, zr)
    out = torch.zeros(12 * nside * nside, dtype=F64, device=DEV)
    v = _vec(z, phi)
    th = torch.atan2(torch.sqrt(v[:, 0] ** 2 + v[:, 1] ** 2), v[:, 2])
    h = int(math.ceil(sigma * nside * 1.6)) + 2

    def spread(sel, pix, w, ok):
        w = torch.where(ok, w.clamp(min=0.0), torch.zeros_like(w))
        tot = w.sum(1, keepdim=True)
        none = tot[:, 0] <= 0
        out.index_add_(0, pix.reshape(-1), (w / torch.where(tot > 0, tot, torch.ones_like(tot))).reshape(-1))
        out.index_add_(0, _ang2pix(nside, z[sel][none], phi[sel][none]), torch.ones(int(none.sum()), dtype=F64,
                                                                                      device=DEV))

    def weight(a, b):
        c = torch.linalg.vector_norm(a - b, dim=-1)
        t = 2.0 * torch.asin((0.5 * c).clamp(max=1.0))
        return 1.0 - (t / sigma) ** 2

    reach = min(20 * sigma, math.pi / 2 + 0.01)
    north, south = th < reach, th > math.pi - reach
    polar = north | south
    zc, sc, pc = _centres(nside)
    for cap, side in ((north, 1.0), (south & ~north, -1.0)):
        near = torch.nonzero(side * zc > math.cos(reach + 2 * sigma)).flatten()
        cv = _vec(zc[near], pc[near], sc[near])
        for s in torch.split(torch.nonzero(cap).flatten(), max(1, int(3e7 / max(1, near.numel())))):
            w = weight(v[s][:, None], cv[None])
            if s.numel():
                spread(s, near.expand(s.numel(), -1), w, w > 0)
    rest = torch.nonzero(~polar).flatten()
    dr = torch.arange(-h, h + 1, device=DEV)
    dj = torch.arange(-h - 1, h + 2, device=DEV)
    for s in torch.split(rest, int(1e8 / (dr.numel() * dj.numel()))) if rest.numel() else ():
        r = (torch.searchsorted(tr, th[s].contiguous())[:, None] + dr).clamp(0, tr.numel() - 1)
        dup = torch.zeros_like(r, dtype=torch.bool)
        dup[:, 1:] = r[:, 1:] == r[:, :-1]
        j = torch.floor((phi[s][:, None] - phi0[r]) * n[r] / (2 * math.pi)).long()[..., None] + dj
        ph = phi0[r][..., None] + 2 * math.pi * j.to(F64) / n[r][..., None]
        c = torch.stack([sr[r][..., None] * torch.cos(ph), sr[r][..., None] * torch.sin(ph),
                         zr[r][..., None].expand_as(ph)], -1)
        w = weight(v[s][:, None, None], c)
        pix = first[r][..., None] + torch.remainder(j, n[r][..., None])
        spread(s, pix.reshape(s.numel(), -1), w.reshape(s.numel(), -1),
               ((w > 0) & ~dup[..., None]).reshape(s.numel(), -1))
    return out


def _spectra(x, A, nside, lmax):
    z, s, _, _, _ = _rings(nside)
    zc, sc, pc = _centres(nside)
    v = (x / x.norm(dim=0)).T
    Ai = _carry(A.T.reshape(-1, 2, 2), v, _vec(zc, pc, sc))
    maps = torch.stack([1 - 0.5 * (Ai[:, 0, 0] + Ai[:, 1, 1]), 0.5 * (Ai[:, 0, 1] - Ai[:, 1, 0]),
                        -0.5 * (Ai[:, 0, 0] - Ai[:, 1, 1]), -0.5 * (Ai[:, 0, 1] + Ai[:, 1, 0])])
    F = _ring_analysis(maps, nside, lmax)
    l = torch.arange(lmax + 1, dtype=F64, device=DEV)[:, None]
    norm = torch.sqrt((l + 2) * (l + 1) * l * (l - 1).clamp(min=0.0))[:, 0]
    norm = torch.where(norm > 0, 1.0 / norm.clamp(min=1e-30), torch.zeros_like(norm))
    cl = torch.zeros(4, lmax + 1, dtype=F64, device=DEV)
    for m0, m1, lam in _blocks(nside, lmax):
        m = torch.arange(m0, m1, dtype=F64, device=DEV)[:, None, None]
        scalar = torch.einsum("mlr,pmr->pml", lam[:, :-1].to(C128), F[:2, m0:m1])
        ep = torch.sqrt(((l + 1) ** 2 - m * m).clamp(min=0.0) / (4 * (l + 1) ** 2 - 1))
        e0 = torch.sqrt((l * l - m * m).clamp(min=0.0) / (4 * l * l - 1).clamp(min=1.0))
        low = torch.zeros_like(lam[:, :-1])
        low[:, 1:] = lam[:, :-2]
        dl = (l * ep * lam[:, 1:] - (l + 1) * e0 * low) / s
        a = (-2.0 * z / s * dl - (l * (l + 1) - 2 * m * m / (s * s)) * lam[:, :-1]).to(C128)
        b = (2.0 * m / s * (dl - z / s * lam[:, :-1])).to(C128)
        F1, F2 = F[2, m0:m1], F[3, m0:m1]
        E = (torch.einsum("mlr,mr->ml", a, F1) - 1j * torch.einsum("mlr,mr->ml", b, F2)) * norm
        B = (torch.einsum("mlr,mr->ml", a, F2) + 1j * torch.einsum("mlr,mr->ml", b, F1)) * norm
        keep = torch.where(m[..., 0] <= l[:, 0], torch.where(m[..., 0] == 0, 1.0, 2.0), torch.zeros_like(m[..., 0]))
        for q, alm in enumerate((scalar[0], E, B, scalar[1])):
            cl[q] += (keep * (alm.real ** 2 + alm.imag ** 2)).sum(0)
    cl = cl / (2 * l[:, 0] + 1)
    return dict(zip(("kappa", "E", "B", "omega"), cl))


def _gradient(case, seed):
    ka, chi, gz, gp, gchi, target = _gradient_inputs(case, seed)
    k = ka.clone().requires_grad_(True)
    bins = (torch.searchsorted(torch.tensor(chi, dtype=F64, device=DEV), gchi, right=True) - 1).clamp(
        max=case["planes"] - 1)
    bins = torch.where(gchi < chi[0], torch.full_like(bins, -1), bins)
    st = _start(_vec(gz, gp), chi[0])
    gam = torch.zeros(2, gz.numel(), dtype=F64, device=DEV)
    for m in range(case["planes"]):
        f = {a: b[0] for a, b in _poisson(k[m:m + 1], case["nside"], case["lmax"]).items()}
        st = _step(st, _map_lens(f, case["nside"]), chi[m - 1] if m else 0.0, chi[m], chi[m + 1])
        t = chi[m + 1] / gchi * (gchi - chi[m]) / (chi[m + 1] - chi[m])
        A = (1 - t)[:, None, None] * st[3] + t[:, None, None] * st[2]
        g = torch.stack([-0.5 * (A[:, 0, 0] - A[:, 1, 1]), -0.5 * (A[:, 0, 1] + A[:, 1, 0])])
        gam = gam + torch.where(bins == m, g, torch.zeros_like(g))
    ((gam - target) ** 2).sum().backward()
    return {"gamma": gam.detach(), "grad": k.grad}


def exact(case, seed):
    kind, ns = case["kind"], case["nside"]
    if kind in ("source", "plane"):
        z, phi = _particles(case["particles"], _gen(seed))
        pix = _ang2pix(ns, z, phi, case.get("nest", False))
        counts = torch.bincount(pix, minlength=12 * ns * ns)
        kappa = SCALE * (counts.to(F64) / (case["particles"] / (12 * ns * ns)) - 1.0)
        if kind == "source":
            return {"counts": None, "kappa": kappa}
        L = _patch_fields(kappa, ns, case["nside_bundle"], case["ncell"])
        zc, sc, pc = _centres(ns)
        outs = []
        for s in range(0, zc.numel(), 1 << 21):
            e = slice(s, s + (1 << 21))
            outs.append(_rays_out(_step(_start(_vec(zc[e], pc[e], sc[e]), CHI), lambda n: [f[e] for f in L],
                                        CHI_PREV, CHI, CHI_NEXT)))
        return {k: torch.cat([o[k] for o in outs], 1) for k in outs[0]}
    if kind == "sht":
        return {k: v[0] for k, v in _poisson(_delta(ns, _gen(seed))[None], ns, case["lmax"]).items()}
    if kind == "batch":
        return [_poisson(torch.stack(m), n, 2 * n) for (n, _), m in zip(_batch_sizes(case), _batch_maps(case, seed))]
    if kind == "smooth":
        z, phi, sigma = _smooth_inputs(case, seed)
        return _smoothed(z, phi, ns, sigma)
    if kind == "images":
        return None   # testing every triangle for every galaxy, the plain form, takes far longer than 20 s
    if kind == "spectra":
        x, A = _lensed_sky(ns, _gen(seed))
        return _spectra(x, A, ns, case["lmax"])
    if kind == "solve":
        return dict(zip(FIELDS, _patch_fields(_solve_input(case, seed), ns, case["nside_bundle"], case["ncell"])))
    if kind == "raytrace":
        kappas, chi = _raytrace_inputs(case, seed)
        zc, sc, pc = _centres(ns)
        st = _start(_vec(zc, pc, sc), chi[0])
        for m, k in enumerate(kappas):
            f = {a: b[0] for a, b in _poisson(k[None], ns, case["lmax"]).items()}
            st = _step(st, _map_lens(f, ns), chi[m - 1] if m else 0.0, chi[m], chi[m + 1])
        return _rays_out(st)
    return _gradient(case, seed)
