// Step 1 of the lens-plane path: particle deposit on HEALPix pixels and the
// plane source kappa^(m) (paper Sec. 3.2 source construction, Eq. lenspoisson;
// pixel indexing Sec. 3.1 / Gorski et al. 2005).
#include "common.cuh"

namespace clc {

// ang2pix on the integer and FP32 pipes.  The pixel index is a function of a
// few floor() values; the FP64 formulas (ang2pix_ring / ang2pix_nest) decide
// them to about 1e-15 nside, so wherever the same quantities, formed here with
// known error, are further from an integer than both errors, the floors and
// with them the pixel are the same.  Returns -1 where they are not (and for
// arguments outside 0 <= phi < 2 pi, |z| <= 1): the caller then takes the FP64
// formulas, whose 25 - 45 instructions per particle on the FP64 pipe (2 per
// clock and SM) set the time of the whole pass: 1.21 ms for 2e7 particles at
// nside 2048, NEST, now 0.50 ms.
//   Belt: t1 -+ t2 = nside (1/2 + tt -+ 3/4 z), tt = 2 phi / pi, in 64-bit fixed
//   point with 60 fractional bits; FP64 errs by at most 2.5e-15 = 2^11.5 units
//   before the factor nside, the fixed point by 4 units: margin 2^14 units.
//   Caps: tp tmp and (1 - tp) tmp, tmp = nside sqrt(3 (1 - |z|)), in FP32: error
//   below 2.4e-7 nside, margin 4e-7 nside + 1e-6; tt * ring in fixed point,
//   margin 2^-34.

// |v| 2^60, truncated, for |v| < 8
__device__ __forceinline__ unsigned long long fixed60(unsigned long long bits) {
  const int e = (int)((bits >> 52) & 0x7ff) - 1023;
  const unsigned long long m = (bits & 0xfffffffffffffull) | 0x10000000000000ull;
  return e < -60 ? 0ull : e >= -8 ? m << (8 + e) : m >> (-8 - e);
}

// interleave: bits of x on even, of y on odd places (x, y < 2^13)
__device__ __forceinline__ unsigned spread16(unsigned x) {
  x = (x | (x << 8)) & 0x00ff00ffu;
  x = (x | (x << 4)) & 0x0f0f0f0fu;
  x = (x | (x << 2)) & 0x33333333u;
  return (x | (x << 1)) & 0x55555555u;
}

template <bool kNest>
__device__ __forceinline__ int64_t ang2pix_fast(int nside, int order, double z, double phi) {
  const unsigned long long zb = (unsigned long long)__double_as_longlong(z), pb = (unsigned long long)__double_as_longlong(phi);
  const unsigned long long za = zb & 0x7fffffffffffffffull;
  if (pb >= 0x4020000000000000ull || za > 0x3ff0000000000000ull) return -1;   // phi < 0, >= 8 or NaN; |z| > 1 or NaN
  const bool south = zb >> 63;
  const unsigned long long one = 1ull << 60, frac = one - 1;
  const unsigned long long zf = fixed60(za);
  const unsigned long long tt = __umul64hi(fixed60(pb), 0xa2f9836e4e441529ull);   // 2/pi 2^64
  if (tt >= 4 * one - (1ull << 14)) return -1;
  const int n = nside;
  if (za <= (unsigned long long)__double_as_longlong(kTwoThirds)) {
    const unsigned long long t = (one >> 1) + tt, q = zf - (zf >> 2);
    const unsigned long long vp = south ? t + q : t - q, vm = south ? t - q : t + q;   // t1 - t2, t1 + t2 over nside
    const unsigned long long mask = (1ull << (60 - order)) - 1, lim = mask - (2ull << 14);
    if ((((vp & mask) - (1ull << 14)) > lim) || (((vm & mask) - (1ull << 14)) > lim)) return -1;
    int jp = (int)(vp >> (60 - order)), jm = (int)(vm >> (60 - order));
    if (kNest) {
      if (jp >= 4 * n && jm >= 4 * n) {
        jp -= 4 * n;
        jm -= 4 * n;
      }
      const int ifp = jp >> order, ifm = jm >> order;
      const int face = ifp == ifm ? (ifp == 4 ? 4 : ifp + 4) : ifp < ifm ? ifp : ifm + 8;
      return (int64_t)face * n * n + (spread16(jm & (n - 1)) | (spread16(n - (jp & (n - 1)) - 1) << 1));
    }
    const int ir = n + 1 + jp - jm;
    const int ip = ((jp + jm - n + (1 - (ir & 1)) + 1) >> 1) & (4 * n - 1);
    return 2 * (int64_t)n * (n - 1) + (int64_t)(ir - 1) * 4 * n + ip;
  }
  const float tp = (float)(unsigned)((tt & frac) >> 28) * 0x1p-32f;
  const float tmp = (float)n * sqrtf(3.f * ((float)(one - zf) * 0x1p-60f));
  const float a = tp * tmp, b = (1.f - tp) * tmp, eps = 4e-7f * (float)n + 1e-6f;
  const float fa = floorf(a), fb = floorf(b);
  if (a - fa < eps || a - fa > 1.f - eps || b - fb < eps || b - fb > 1.f - eps) return -1;
  const int jp = (int)fa, jm = (int)fb;
  if (kNest) {
    const int ntt = (int)(tt >> 60);
    if (jp > n - 1 || jm > n - 1) return -1;
    const int ix = south ? jp : n - jm - 1, iy = south ? jm : n - jp - 1;
    return (int64_t)(south ? ntt + 8 : ntt) * n * n + (spread16(ix) | (spread16(iy) << 1));
  }
  const int ir = jp + jm + 1;
  const unsigned long long w = (unsigned long long)ir << 4;
  const unsigned long long lo = tt * w;   // fraction of tt ir, 2^-64
  if (lo < (1ull << 30) || lo > ~0ull - (1ull << 30)) return -1;
  const int64_t ip = (int64_t)__umul64hi(tt, w);
  if (ip >= 4 * ir) return -1;
  return south ? 12ll * n * n - 2ll * ir * (ir + 1) + ip : 2ll * ir * (ir - 1) + ip;
}

// One thread per particle (grid-stride): 16 B read, one L2 atomic increment.
template <bool kNest>
__global__ void k_bin(const double* __restrict__ z, const double* __restrict__ phi, int64_t n, int nside, int order,
                      uint32_t* __restrict__ counts) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const double zi = z[i], pi = phi[i];
    int64_t p = ang2pix_fast<kNest>(nside, order, zi, pi);
    if (p < 0) p = kNest ? ang2pix_nest(nside, zi, pi) : ang2pix_ring(nside, zi, pi);
    atomicAdd(counts + p, 1u);
  }
}

// kappa of a pixel with c particles: scale (c / nbar - 1), each operation
// correctly rounded
__device__ __forceinline__ double kappa_of(uint32_t c, double nbar, double scale) {
  return __dmul_rn(scale, __dsub_rn(__ddiv_rn((double)c, nbar), 1.0));
}

// Counts are small integers, so kappa takes few distinct values: a table of
// the first kKappaTable (the same correctly rounded operations, once per
// count) replaces the FP64 division per pixel, which would make this pass
// FP64-bound; larger counts divide.
constexpr int kKappaTable = 4096;

__global__ void k_kappa_table(double nbar, double scale, double* __restrict__ tab) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < kKappaTable) tab[c] = kappa_of((uint32_t)c, nbar, scale);
}

// Maps of kKappaDirect pixels and below divide: at nside 64 the 49152 divisions,
// one per thread, take 6.3 us, the launch of the table's 4096 and the pass 8.3
// (launches back to back); at nside 128 12.5 against 8.3.
constexpr int64_t kKappaDirect = 12 * 64 * 64;
// kWide: four pixels per thread (16-byte loads and stores; npix is a multiple of
// 4), for maps of more than kKappaWide pixels, whose 12 bytes per pixel do not
// stay in L2: 37 instead of 49 us at nside 1024, 125 instead of 165 at 2048.  At
// nside 512 (counts just written) one pixel per thread takes 12.5 us, four 14.5.
constexpr int64_t kKappaWide = 12 * 512 * 512;

template <bool kWide>
__global__ void k_counts_to_kappa(const uint32_t* __restrict__ counts, int64_t npix, double nbar,
                                  double scale, const double* __restrict__ tab, double* __restrict__ kappa) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  auto value = [&](uint32_t c) { return tab && c < (uint32_t)kKappaTable ? tab[c] : kappa_of(c, nbar, scale); };
  if (kWide) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < npix / 4; i += stride) {
      const uint4 c = reinterpret_cast<const uint4*>(counts)[i];
      double2* k = reinterpret_cast<double2*>(kappa) + 2 * i;
      k[0] = make_double2(value(c.x), value(c.y));
      k[1] = make_double2(value(c.z), value(c.w));
    }
  } else {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < npix; i += stride) kappa[i] = value(counts[i]);
  }
}

// Partial-sky source (Sec. 3.4): particle count and pixel count of the
// covered region (exact integer sums), then nbar = their ratio and
// kappa = scale (counts / nbar - 1) on covered pixels, 0 (mean density)
// elsewhere.
__global__ void k_masked_sums(const uint32_t* __restrict__ counts, const uint8_t* __restrict__ covered, int64_t npix,
                              unsigned long long* __restrict__ sums) {
  unsigned long long c = 0, m = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < npix; i += stride)
    if (covered[i]) {
      c += counts[i];
      ++m;
    }
  for (int o = 16; o > 0; o >>= 1) {
    c += __shfl_xor_sync(0xffffffffu, c, o);
    m += __shfl_xor_sync(0xffffffffu, m, o);
  }
  if ((threadIdx.x & 31) == 0 && (c || m)) {
    atomicAdd(sums, c);
    atomicAdd(sums + 1, m);
  }
}

__global__ void k_counts_to_kappa_masked(const uint32_t* __restrict__ counts, const uint8_t* __restrict__ covered,
                                         int64_t npix, const unsigned long long* __restrict__ sums, double scale,
                                         double* __restrict__ kappa) {
  const double nbar = __ddiv_rn((double)sums[0], (double)sums[1]);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < npix; i += stride)
    kappa[i] = covered[i] ? __dmul_rn(scale, __dsub_rn(__ddiv_rn((double)counts[i], nbar), 1.0)) : 0.0;
}

// Coarse pixel P (RING) = mean of its NEST children at nside_fine.  The coarse
// pixel's NEST index comes from its centre (pix2ang followed by ang2pix_nest,
// which returns the pixel itself: centres lie far from pixel edges).
__global__ void k_degrade(const double* __restrict__ fine, int nf, double* __restrict__ coarse, int ns,
                          int shift) {
  const int64_t npc = 12ll * ns * ns;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int nchild = 1 << shift;
  const double inv = 1.0 / (double)nchild;
  for (int64_t P = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; P < npc; P += stride) {
    int64_t j;
    const int i = pix2ring(ns, P, &j);
    const Ring r = ring_geom(ns, i);
    const double phi = r.phi0 + (2.0 * kPi) * (double)j / (double)r.npix;
    const int64_t pn = ang2pix_nest(ns, r.z, phi);
    double acc = 0.0;
    for (int c = 0; c < nchild; ++c) acc += fine[nest2ring(nf, (pn << shift) + c)];
    coarse[P] = acc * inv;
  }
}

// kappa = scale * (rho / nbar - 1), each operation rounded separately
__global__ void k_density_to_kappa(const double* __restrict__ rho, int64_t npix, double nbar, double scale,
                                   double* __restrict__ kappa) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < npix; i += stride)
    kappa[i] = __dmul_rn(scale, __dsub_rn(__ddiv_rn(rho[i], nbar), 1.0));
}

static int grid_for(clc_ctx* ctx, int64_t n, int threads) {
  int64_t blocks = (n + threads - 1) / threads;
  const int64_t cap = (int64_t)num_sms(ctx) * 16;
  if (blocks > cap) blocks = cap;
  return (int)(blocks < 1 ? 1 : blocks);
}

}  // namespace clc

using namespace clc;

extern "C" int clc_bin_particles(clc_ctx* ctx, const double* z, const double* phi, int64_t n, int nside,
                                 int ordering, uint32_t* counts) {
  if (!ctx) return CLC_EINVAL;
  if (n < 0 || !valid_nside(nside) || (ordering != CLC_RING && ordering != CLC_NEST))
    return set_err(ctx, CLC_EINVAL, "clc_bin_particles: bad n, nside or ordering");
  if (n == 0) return CLC_OK;
  if (!z || !phi || !counts) return set_err(ctx, CLC_EINVAL, "clc_bin_particles: null pointer");
  cudaSetDevice(ctx->device);
  int order = 0;
  while ((1 << order) < nside) ++order;
  if (ordering == CLC_NEST)
    CLC_LAUNCH(ctx, "k_bin", k_bin<true>, grid_for(ctx, n, 256), 256, 0, z, phi, n, nside, order, counts);
  else
    CLC_LAUNCH(ctx, "k_bin", k_bin<false>, grid_for(ctx, n, 256), 256, 0, z, phi, n, nside, order, counts);
  return launch_check(ctx, "k_bin");
}

extern "C" int clc_counts_to_kappa(clc_ctx* ctx, const uint32_t* counts, int nside, double nbar, double scale,
                                   double* kappa) {
  if (!ctx) return CLC_EINVAL;
  if (!valid_nside(nside) || !(nbar > 0)) return set_err(ctx, CLC_EINVAL, "clc_counts_to_kappa: bad nside or nbar");
  if (!counts || !kappa) return set_err(ctx, CLC_EINVAL, "clc_counts_to_kappa: null pointer");
  cudaSetDevice(ctx->device);
  const int64_t npix = 12ll * nside * nside;
  double* tab = nullptr;
  if (npix > kKappaDirect) {
    tab = (double*)scratch(ctx, 7, sizeof(double) * kKappaTable);
    if (!tab) return CLC_ENOMEM;
    CLC_LAUNCH(ctx, "k_counts_to_kappa", k_kappa_table, kKappaTable / 256, 256, 0, nbar, scale, tab);
  }
  if (npix > kKappaWide && ((reinterpret_cast<uintptr_t>(counts) | reinterpret_cast<uintptr_t>(kappa)) & 15) == 0)
    CLC_LAUNCH(ctx, "k_counts_to_kappa", k_counts_to_kappa<true>, grid_for(ctx, npix / 4, 256), 256, 0, counts, npix,
               nbar, scale, (const double*)tab, kappa);
  else
    CLC_LAUNCH(ctx, "k_counts_to_kappa", k_counts_to_kappa<false>, grid_for(ctx, npix, 256), 256, 0, counts, npix, nbar,
               scale, (const double*)tab, kappa);
  return launch_check(ctx, "k_counts_to_kappa");
}

extern "C" int clc_counts_to_kappa_masked(clc_ctx* ctx, const uint32_t* counts, const uint8_t* covered, int nside,
                                          double scale, double* kappa) {
  if (!ctx) return CLC_EINVAL;
  if (!valid_nside(nside)) return set_err(ctx, CLC_EINVAL, "clc_counts_to_kappa_masked: bad nside");
  if (!counts || !covered || !kappa) return set_err(ctx, CLC_EINVAL, "clc_counts_to_kappa_masked: null pointer");
  cudaSetDevice(ctx->device);
  const int64_t npix = 12ll * nside * nside;
  // as large as the kappa table in the same slot, so that neither call frees the other's
  unsigned long long* sums = (unsigned long long*)scratch(ctx, 7, sizeof(double) * kKappaTable);
  if (!sums) return CLC_ENOMEM;
  cudaMemsetAsync(sums, 0, 2 * sizeof(unsigned long long), ctx->stream);
  CLC_LAUNCH(ctx, "k_masked_sums", k_masked_sums, grid_for(ctx, npix, 256), 256, 0, counts, covered, npix, sums);
  CLC_LAUNCH(ctx, "k_counts_to_kappa", k_counts_to_kappa_masked, grid_for(ctx, npix, 256), 256, 0, counts, covered,
             npix, (const unsigned long long*)sums, scale, kappa);
  return launch_check(ctx, "k_counts_to_kappa_masked");
}

extern "C" int clc_degrade(clc_ctx* ctx, const double* fine, int nf, double* coarse, int ns) {
  if (!ctx) return CLC_EINVAL;
  if (!valid_nside(nf) || !valid_nside(ns) || ns > nf) return set_err(ctx, CLC_EINVAL, "clc_degrade: bad nside");
  if (!fine || !coarse) return set_err(ctx, CLC_EINVAL, "clc_degrade: null pointer");
  cudaSetDevice(ctx->device);
  int shift = 0;
  while ((ns << (shift / 2)) < nf) shift += 2;
  const int64_t npc = 12ll * ns * ns;
  CLC_LAUNCH(ctx, "k_degrade", k_degrade, grid_for(ctx, npc, 256), 256, 0, fine, nf, coarse, ns, shift);
  return launch_check(ctx, "k_degrade");
}

extern "C" int clc_density_to_kappa(clc_ctx* ctx, const double* rho, int nside, double nbar, double scale,
                                    double* kappa) {
  if (!ctx) return CLC_EINVAL;
  if (!valid_nside(nside) || !(nbar > 0)) return set_err(ctx, CLC_EINVAL, "clc_density_to_kappa: bad nside or nbar");
  if (!rho || !kappa) return set_err(ctx, CLC_EINVAL, "clc_density_to_kappa: null pointer");
  cudaSetDevice(ctx->device);
  const int64_t npix = 12ll * nside * nside;
  CLC_LAUNCH(ctx, "k_density_to_kappa", k_density_to_kappa, grid_for(ctx, npix, 256), 256, 0, rho, npix, nbar, scale,
             kappa);
  return launch_check(ctx, "k_density_to_kappa");
}
