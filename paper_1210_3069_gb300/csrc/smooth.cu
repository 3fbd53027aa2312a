// Adaptive Epanechnikov smoothing (paper Sec. 3.2): a particle's unit mass goes
// to the RING pixels whose centres lie within angular distance sigma, in
// proportion to 1 - (theta / sigma)^2 (the kernel's normalisation cancels), the
// weights divided by their sum so that the mass is conserved exactly; with no
// centre within sigma the mass goes to the particle's own pixel.
//
// One thread per particle.  On the ring of (z, s) the squared chord to the
// centre at longitude offset dphi is
//   c^2 = (s - sp)^2 + (z - zp)^2 + 4 s sp sin^2(dphi / 2),
// all of it but the last factor per ring, and that a short series in dphi^2.
// The FP64 pipe (2 instructions per clock and SM) sets the time, so FP64 is
// left for the weights alone: ring geometry comes from the context's table, the
// rings and longitudes in reach from FP32 (spans widened by 0.02 pixel; the
// test c^2 < 4 sin^2(sigma / 2) decides).  Unit vectors of every candidate,
// acos, divisions and sincospi per ring in FP64 were about 4000 instructions
// per particle (76.6 ms for 1.2e7 particles, sigma 2.5 pixels, nside 1024); the
// chord is also the more accurate one (no difference of nearby unit vectors).
// The weights wait in shared memory for their sum.
// Now 11.5 ms (FP64 pipe; 18.5 ms with one loop per ring).
#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace clc {

constexpr int kSmoothThreads = 128;

// theta^2 from the chord c^2 of two unit vectors, 4 asin^2(c / 2): the Taylor
// series of asin^2 (through c^6 for c^2 <= 1e-5, through c^14 for c^2 <= 1/400:
// first omitted terms below 1e-17 relative), else directly
__device__ __forceinline__ double theta2_small(double c2) {
  return c2 * fma(c2, fma(c2, 1.0 / 90.0, 1.0 / 12.0), 1.0);
}
__device__ __forceinline__ double theta2_of_chord2(double c2) {
  if (c2 <= 0.0025)
    return c2 * (1.0 + c2 * ((1.0 / 12.0) + c2 * ((1.0 / 90.0) + c2 * ((1.0 / 560.0) + c2 * ((1.0 / 3150.0) +
                                                                                           c2 * (1.0 / 16632.0))))));
  const double t = 2.0 * asin(0.5 * sqrt(c2));
  return t * t;
}

// sin^2 x: series (first omitted term below 1e-17 relative for |x| <= 1/512,
// 1/64 and 1/16), else directly
__device__ __forceinline__ double sin2_of(double x, float span) {
  if (span < 0.0625f) {
    const double y = x * x;
    if (span < 0.00195f) return y * fma(y, fma(y, 2.0 / 45.0, -1.0 / 3.0), 1.0);
    if (span < 0.0156f) return y * fma(y, fma(y, fma(y, -1.0 / 315.0, 2.0 / 45.0), -1.0 / 3.0), 1.0);
    return y * fma(y, fma(y, fma(y, fma(y, fma(y, -2.0 / 467775.0, 2.0 / 14175.0), -1.0 / 315.0), 2.0 / 45.0), -1.0 / 3.0), 1.0);
  }
  const double s = sin(x);
  return s * s;
}

// comparisons of non-negative doubles and signs on the integer pipe
__device__ __forceinline__ bool less_pos(double a, double b) { return __double_as_longlong(a) < __double_as_longlong(b); }
__device__ __forceinline__ bool positive(double a) { return __double_as_longlong(a) > 0; }
// FP32 of a positive double (truncated; 0 below the FP32 range)
__device__ __forceinline__ float narrow_pos(double v) {
  const int hi = __double2hiint(v), e = (hi >> 20) - 896;
  if (e <= 0) return 0.f;
  return e >= 255 ? 3e38f : __uint_as_float(((unsigned)e << 23) | (((unsigned)hi & 0xfffffu) << 3) | ((unsigned)__double2loint(v) >> 29));
}

struct Particle {
  double zp, sp4, sp, pp, c2max, inv_s2;
  float ppf;
  bool tiny;   // c2max <= 1e-5
  int i0, i1;
};

// A ring in reach: c^2 = a + b sin^2 x at x = x0, x0 + pi / npix, ... for the n
// centres from position jl (unwrapped) on; span: largest |x|.
struct RingReach {
  double a, b, x0;
  int jl, n;
  float span;
};

__device__ __forceinline__ double ring_a(const Particle& q, const RingS& R) {
  const double ds = R.r.s - q.sp, dz = R.r.z - q.zp;
  return fma(ds, ds, dz * dz);
}
__device__ __forceinline__ double ring_x0(const Particle& q, const RingS& R, int jl) {
  return fma((double)jl, R.half, 0.5 * (R.r.phi0 - q.pp));
}

__device__ __forceinline__ bool ring_reach(const Particle& q, const RingS& R, RingReach& o) {
  o.a = ring_a(q, R);
  const double rem = q.c2max - o.a;
  if (!positive(rem) || !(__double2hiint(rem) < 0x7ff00000)) return false;   // every centre is at least that far (or NaN)
  const int np = R.r.npix;
  o.b = R.r.s * q.sp4;
  // centres with sin^2(dphi / 2) < rem / b
  o.jl = 0;
  o.n = np;
  o.span = 4.f;
  const float sh2 = narrow_pos(rem) * 1.000001f / narrow_pos(o.b);
  if (sh2 < 1.f) {
    const float inv = (float)np * 0.159154943f, half = R.r.phi0 != 0.0 ? 0.5f : 0.f;
    const float span = asinf(sqrtf(sh2));
    const float base = q.ppf * inv - half, w = 2.f * span * inv * 1.000001f + 0.02f;
    const int lo = (int)ceilf(base - w), hi = (int)floorf(base + w);
    if (hi - lo + 1 < np) {
      o.jl = lo;
      o.n = max(hi - lo + 1, 0);
      o.span = span + 0.07f / (float)np;
    }
  }
  o.x0 = ring_x0(q, R, o.jl);
  return o.n > 0;
}

__device__ __forceinline__ double weight_at(const Particle& q, double a, double b, double x, float span) {
  const double c2 = fma(b, sin2_of(x, span), a);
  if (!less_pos(c2, q.c2max)) return 0.0;
  return fma(-(q.tiny ? theta2_small(c2) : theta2_of_chord2(c2)), q.inv_s2, 1.0);
}

__device__ __forceinline__ int64_t wrapped(const Ring& r, int j) {
  return r.first + (j < 0 ? j + r.npix : j >= r.npix ? j - r.npix : j);
}

// Calls f(ring, position, weight) for every centre in reach, ring by ring.
template <typename F>
__device__ void kernel_pixels(const Particle& q, const RingS* __restrict__ rings, F f) {
  for (int i = q.i0; i <= q.i1; ++i) {
    const RingS R = rings[i - 1];
    RingReach o;
    if (!ring_reach(q, R, o)) continue;
    for (int t = 0; t < o.n; ++t) f(R.r, o.jl + t, weight_at(q, o.a, o.b, fma((double)t, R.half, o.x0), o.span));
  }
}

// The rings of a particle are set up first and its centres then taken in one
// loop over all of them: loops ring by ring run, in every ring, as long as the
// widest of a warp's 32 particles (22 of 32 lanes active).  Particles with more
// rings or centres than the shared arrays hold go ring by ring, twice, and a
// warp with both kinds takes both ways.  Two forms of the arrays, three blocks
// of either on an SM (rings and centres in reach counted at nside 64 and 1024
// over the whole sphere and close to the poles):
//   small: 9 rings, 32 centres, ring terms kept (576 bytes a particle): every
//     particle up to 2.9 pixels (at most 9 and 31; 1 % do not fit at 3.0);
//   large: 13 rings, 60 centres, ring terms formed again (584 bytes): up to
//     4.2 pixels (13 and 60; 10 % do not fit at 4.3).
// With lengths of their own a warp takes the form of its longest.
// 4e6 uniform particles at nside 1024, sigma 1, 2.5, 3, 3.25, 4 and 6 pixels:
// 1.12, 3.94, 7.1, 10.3, 15.1 and 184 ms; with the small form alone 1.12, 3.94,
// 12.2, 102, 52 and 185; with the large one alone 5.4 at 2.5.  Lengths of their
// own, uniform in 1 .. 4 pixels: 28 ms (the small form alone: 71).
constexpr int kMaxRings = 13;

template <int kR, int kC, bool kK>
struct SmoothShared {
  static_assert(kR <= kMaxRings && kC < 256, "rows and packing");
  static constexpr int kRings = kR, kCentres = kC;
  static constexpr bool kKeep = kK;
  // The two forms' columns of a thread are the same addresses (the integers have
  // equally many rows in both), so warps of a block may use different forms.
  int jl[kMaxRings][kSmoothThreads], ring_end[kMaxRings][kSmoothThreads];   // 256 ring + centres up to its end
  double w[kC][kSmoothThreads];
  double a[kK ? kR : 0][kSmoothThreads], b[kK ? kR : 0][kSmoothThreads], x0[kK ? kR : 0][kSmoothThreads];
};
using SmoothSmall = SmoothShared<9, 32, true>;
using SmoothLarge = SmoothShared<kMaxRings, 60, false>;
constexpr double kSmallPixels = 2.9;   // largest sigma of the small form in pixels (square root of their area)

template <typename Sh>
__device__ __forceinline__ void deposit(const Particle& q, double phi_i, int nside, const RingS* __restrict__ rings,
                                        double* __restrict__ map, Sh& S) {
  const int me = threadIdx.x;
  int nr = 0, nc = 0;
  float span = 0.f;
  for (int r = q.i0; r <= q.i1 && nr <= Sh::kRings; ++r) {
    RingReach o;
    if (!ring_reach(q, rings[r - 1], o)) continue;
    if (nr < Sh::kRings && nc + o.n <= Sh::kCentres) {
      nc += o.n;
      if constexpr (Sh::kKeep) {
        S.a[nr][me] = o.a;
        S.b[nr][me] = o.b;
        S.x0[nr][me] = o.x0;
      }
      S.jl[nr][me] = o.jl;
      S.ring_end[nr][me] = r << 8 | nc;
      span = fmaxf(span, o.span);
    } else {
      nr = Sh::kRings;   // does not fit
    }
    ++nr;
  }
  double tot = 0.0;
  if (nr <= Sh::kRings) {
    double a = 0.0, b = 0.0, x = 0.0, h = 0.0;
    int k = 0, end = 0;
    for (int c = 0; c < nc; ++c) {
      if (c == end) {
        const int re = S.ring_end[k][me];
        const RingS& R = rings[(re >> 8) - 1];
        if constexpr (Sh::kKeep) {
          a = S.a[k][me];
          b = S.b[k][me];
          x = S.x0[k][me];
        } else {
          a = ring_a(q, R);
          b = R.r.s * q.sp4;
          x = ring_x0(q, R, S.jl[k][me]);
        }
        h = R.half;
        end = re & 255;
        ++k;
      }
      const double w = weight_at(q, a, b, x, span);
      x += h;
      if (positive(w)) tot += w;
      S.w[c][me] = w;
    }
    if (positive(tot)) {
      const double inv = 1.0 / tot;
      int j = 0;
      Ring r{};
      k = end = 0;
      for (int c = 0; c < nc; ++c, ++j) {
        if (c == end) {
          const int re = S.ring_end[k][me];
          r = rings[(re >> 8) - 1].r;
          j = S.jl[k][me];
          end = re & 255;
          ++k;
        }
        const double w = S.w[c][me];
        if (positive(w)) atomicAdd(map + wrapped(r, j), w * inv);
      }
      return;
    }
  } else {
    kernel_pixels(q, rings, [&](const Ring&, int, double w) {
      if (positive(w)) tot += w;
    });
    if (positive(tot)) {
      const double inv = 1.0 / tot;
      kernel_pixels(q, rings, [&](const Ring& r, int j, double w) {
        if (positive(w)) atomicAdd(map + wrapped(r, j), w * inv);
      });
      return;
    }
  }
  atomicAdd(map + ang2pix_ring(nside, q.zp, phi_i), 1.0);
}

enum { kFormSmall = 0, kFormLarge = 1, kFormWarp = 2 };

template <int kForm>
__global__ void __launch_bounds__(kSmoothThreads) k_smooth_particles(const double* __restrict__ z,
                                                                     const double* __restrict__ phi,
                                                                     const double* __restrict__ sig_each, int64_t n,
                                                                     int nside, double sigma,
                                                                     const RingS* __restrict__ rings,
                                                                     double* __restrict__ map) {
  extern __shared__ __align__(16) unsigned char smem_sm[];
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  double sg = sigma, hs = sin(0.5 * sigma), inv_s2 = 1.0 / (sigma * sigma);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    Particle q;
    q.zp = z[i];
    const double phi_i = phi[i];
    q.pp = phi_i >= 0.0 && phi_i <= 2.0 * kPi ? phi_i : phi_i - 2.0 * kPi * floor(phi_i / (2.0 * kPi));
    if (kForm == kFormWarp) {
      sg = sig_each[i];
      hs = sin(0.5 * sg);
      inv_s2 = 1.0 / (sg * sg);
    }
    q.sp = sqrt((1.0 - q.zp) * (1.0 + q.zp));
    q.sp4 = 4.0 * q.sp;
    q.c2max = 4.0 * hs * hs;
    q.tiny = q.c2max <= 1e-5;
    q.inv_s2 = inv_s2;
    q.ppf = (float)q.pp;
    const float th = atan2f((float)q.sp, (float)q.zp), sf = (float)sg * 1.00001f;
    q.i0 = max(1, (int)ceilf(ring_coord32(nside, fmaxf(0.f, th - sf)) - 0.1f));
    q.i1 = min(4 * nside - 1, (int)floorf(ring_coord32(nside, fminf(3.14159265f, th + sf)) + 0.1f));
    bool large = kForm == kFormLarge;
    if (kForm == kFormWarp)   // (a wrong guess costs time only)
      large = __any_sync(__activemask(), sf * (float)nside > (float)kSmallPixels * 1.02332671f);
    if (large)
      deposit(q, phi_i, nside, rings, map, *reinterpret_cast<SmoothLarge*>(smem_sm));
    else
      deposit(q, phi_i, nside, rings, map, *reinterpret_cast<SmoothSmall*>(smem_sm));
  }
}

}  // namespace clc

using namespace clc;

extern "C" int clc_smooth_particles(clc_ctx* ctx, const double* z, const double* phi, int64_t n, int nside,
                                    double sigma, const double* sigma_each, double* map) {
  if (!ctx) return CLC_EINVAL;
  if (n < 0 || !valid_nside(nside) || nside > 8192 || (!sigma_each && !(sigma > 0.0 && sigma <= 0.5)))
    return set_err(ctx, CLC_EINVAL, "clc_smooth_particles: need n >= 0, nside <= 8192 and 0 < sigma <= 0.5");
  if (n == 0) return CLC_OK;
  if (!z || !phi || !map) return set_err(ctx, CLC_EINVAL, "clc_smooth_particles: null pointer");
  cudaSetDevice(ctx->device);
  int rc;
  const RingS* rings = get_ring_table(ctx, nside, &rc);
  if (rc) return rc;
  const int64_t blocks = std::min<int64_t>((n + kSmoothThreads - 1) / kSmoothThreads, (int64_t)num_sms(ctx) * 32);
  auto launch = [&](auto kern, size_t smem) {
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    CLC_LAUNCH(ctx, "k_smooth_particles", kern, (int)blocks, kSmoothThreads, (int)smem, z, phi, sigma_each, n, nside,
               sigma, rings, map);
  };
  if (sigma_each)
    launch(k_smooth_particles<kFormWarp>, std::max(sizeof(SmoothSmall), sizeof(SmoothLarge)));
  else if (sigma <= kSmallPixels * std::sqrt(kPi / 3.0) / nside)
    launch(k_smooth_particles<kFormSmall>, sizeof(SmoothSmall));
  else
    launch(k_smooth_particles<kFormLarge>, sizeof(SmoothLarge));
  return launch_check(ctx, "k_smooth_particles");
}
