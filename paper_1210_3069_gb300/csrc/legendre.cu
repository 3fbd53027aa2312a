// Legendre step of the SHT (paper Sec. 3.2; the associated-Legendre
// recurrence of Press et al. 2007 Sec. 6.7) with the accuracy of FP64, on the
// tcgen05 tensor cores.
//
// lambda_lm(z_r) is built once per (Nside, lmax) with the three-term
// recurrence in l in FP64, started from lambda_mm = (-1)^m sqrt((2m+1)!! /
// (4 pi (2m)!!)) sin^m(theta) carried as a mantissa and a power-of-two
// exponent (sin^m theta underflows FP64 near the poles at large m).  Analysis
// and synthesis are then per-m matrix products over the northern rings, using
// lambda_lm(-z) = (-1)^(l+m) lambda_lm(z) for the southern mirror rings.
//
// The products are exact integer arithmetic (the error-free splitting of
// Ozaki et al. 2012, "Error-free transformations of matrix multiplication"):
// a table row and a data column are scaled by powers of two to integers of at
// most 62 bits and written as eight signed base-256 digits, small integers
// that FP16 holds exactly.  Digit products are at most 2^14, so an FP32
// accumulator adds the up to 8 digit pairs i + j = g of 128 terms without
// rounding (8 * 128 * 2^14 = 2^24); the sums of each g <= 7 are collected in
// 64-bit integers and rounded once.  Digit pairs with g > 7 are left out: at most
// seven of a term reach 2^-62 of the product of the scales, so a term loses less
// than 2^-59 of it.  The result does not depend on the order of summation.  Rings
// where lambda_lm is small for every l (towards the poles) are scaled up by
// 2^cexp <= 2^24 first.
//   The error is thus relative to the scales, the largest |lambda_lm| 2^cexp of the
// row and the largest |value| 2^-cexp of the column, not to each term: as small as
// that of FP64 sums (2^-53 of the largest term) while the rings (or degrees) of a
// column differ by less than about 2^33 where lambda_lm is small, which sources,
// shears and their coefficients do; a column with larger contrasts keeps fewer
// bits in the sums that its largest values hardly enter.
//
// Eight digits, not seven: the scale is the largest value of a row or column,
// while the FP64 sums this replaces keep every term's own 53 bits.  Near the
// poles the low degrees, whose coefficients are the largest, have tiny
// lambda_lm, and the Hessian multiplies the sum by m^2 / sin^2 theta (up to
// 1.5 nside^2): with seven digits (54 bits) the error of u_pp at nside 512,
// lmax 1024 was 2.2e-12 against 3.1e-14 of plain FP64 sums.
//
// Why digits on the tensor cores: the FP64 pipe does 2 FMA per clock and SM,
// 0.63e12 per second on the chip, and a plane's transforms take 2 FMA per
// table value forward and 6 back; read from HBM as eight FP16 planes (16 bytes,
// 0.42e12 values per second) a value serves up to 16 columns at once, so both
// directions are bound by the table traffic.  At nside 512, lmax 1024 the
// FP64 kernels took 2.2 ms (analysis), 11.8 ms (synthesis of the three sums)
// and 53.4 ms (spin-2 sums of two fields); with them the solve took 19.2 ms and
// the four spectra 63.2, with the digits 7.8 and 7.1 (6.05 and 4.02 with the ring
// FFTs of now).
#include <algorithm>
#include <cmath>

#include "legendre.cuh"
#include "umma.cuh"

namespace clc {

constexpr long long kDigWaitPolls = 1ll << 26;
constexpr int kDigStages = 8;          // digit-plane pairs (16 KB) in flight per CTA
constexpr int kDigFlush = 2;           // blocks of 64 terms per TMEM accumulation
constexpr int kRingScaleMax = 24;      // largest cexp
constexpr int kNonFinite = 0x7fffffff; // column exponent of a column with a NaN or infinity
constexpr size_t kSegBytes = 2ull << 30;   // FP64 recurrence values held at a time while building

// half offset of element (row r, column c < 64) inside a tile of 64-half rows
// in the 128-byte swizzle (8-row groups of 1024 bytes)
__host__ __device__ __forceinline__ uint32_t dig_off(int r, int c) {
  return (uint32_t)((r >> 3) * 512 + (r & 7) * 64 + (((c >> 3) ^ (r & 7)) << 3) + (c & 7));
}

// p * 2^e, exact unless the result is subnormal or zero (one final rounding);
// |p| < 2^410 and e <= 64 here.
__device__ __forceinline__ double scale_pow2(double p, int e) {
  if (e >= -1022) return p * __longlong_as_double((long long)(e + 1023) << 52);
  if (e < -1600) return 0.0;
  return (p * __longlong_as_double((long long)(e + 600 + 1023) << 52)) * 0x1p-600;
}
// the same for any e
__device__ __forceinline__ double times_pow2(double p, int e) {
  if (e >= -1022 && e <= 1023) return p * __longlong_as_double((long long)(e + 1023) << 52);
  return ldexp(p, e);
}

__device__ __forceinline__ int abs_hi(double v) { return __double2hiint(v) & 0x7fffffff; }

// The integer nearest to v 2^e (at most 2^62 in magnitude) as eight signed
// base-256 digits: byte i of it + 0x80..80 is digit i plus 128.  All on the
// integer pipe: scaling and conversion were most of the packing's FP64
// instructions (0.56 ms for eight columns at nside 512, lmax 1024).
__device__ __forceinline__ unsigned long long dig_of(double v, int e) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(v);
  const int ex = (int)(u >> 52) & 0x7ff, sh = ex - 1075 + e;
  const unsigned long long m = (u & 0xfffffffffffffull) | 0x10000000000000ull;
  unsigned long long r = 0;
  if (ex && sh > -64) r = sh >= 0 ? m << sh : (m + (1ull << (-sh - 1))) >> -sh;
  return ((long long)u < 0 ? 0 - r : r) + 0x8080808080808080ull;
}
// digit plane s (0 = most significant) of two values as FP16 integers
__device__ __forceinline__ unsigned dig_pair(unsigned long long y0, unsigned long long y1, int s) {
  const int sh = 8 * (kDigits - 1 - s);
  const unsigned w = 0x64006400u | ((unsigned)(y0 >> sh) & 255u) | (((unsigned)(y1 >> sh) & 255u) << 16);   // 1024 + byte
  const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&w), __half2half2(__ushort_as_half(0x6480)));   // - 1152
  return *reinterpret_cast<const unsigned*>(&d);
}

// ---------------------------------------------------------------------------
// table build

// recurrence coefficients a_lm = sqrt((4l^2 - 1) / (l^2 - m^2)),
// b_lm = sqrt(((l-1)^2 - m^2) / (4 (l-1)^2 - 1)) of the orders ms ..
__global__ void k_legendre_coef(int lt, int ms, double2* __restrict__ ab) {
  const int m = ms + blockIdx.y;
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l > lt || l < m + 2) return;
  const double l2 = (double)l * l, m2 = (double)m * m, k2 = (l - 1.0) * (l - 1.0);
  ab[(size_t)blockIdx.y * (lt + 1) + l] = make_double2(sqrt((4.0 * l * l - 1.0) / (l2 - m2)), sqrt((k2 - m2) / (4.0 * k2 - 1.0)));
}

// lambda_lm of the orders ms .. in FP64, [m][l - m][r], and the ring scales
__global__ void k_legendre_build(int nside, int lmax, int R, const long long* __restrict__ off,
                                 const double* __restrict__ lognorm, const double2* __restrict__ ab,
                                 double* __restrict__ tab, int ms, int8_t* __restrict__ cexp, int ldc) {
  const int m = ms + blockIdx.y;
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= R) return;
  const Ring g = ring_geom(nside, r + 1);
  const double z = g.z;
  const int lt = lmax + 1;  // table band limit
  double* col = tab + off[blockIdx.y];
  const double2* cab = ab + (size_t)blockIdx.y * (lt + 1);
  const double l2 = lognorm[m] + (double)m * log2(g.s);
  int e = (int)floor(l2);
  double p2 = exp2(l2 - (double)e);
  if (m & 1) p2 = -p2;
  double v = scale_pow2(p2, e);
  col[r] = v;
  int top = abs_hi(v);
  if (lt >= m + 1) {
    double p1 = sqrt(2.0 * m + 3.0) * z * p2;
    v = scale_pow2(p1, e);
    col[(size_t)R + r] = v;
    top = max(top, abs_hi(v));
    const double big = 0x1p400, small = 0x1p-400;
    for (int l = m + 2; l <= lt; ++l) {
      const double2 c = cab[l];
      double p0 = c.x * (z * p1 - c.y * p2);
      if (fabs(p0) > big) {
        p0 *= small;
        p1 *= small;
        e += 400;
      }
      v = scale_pow2(p0, e);
      col[(size_t)(l - m) * R + r] = v;
      top = max(top, abs_hi(v));
      p2 = p1;
      p1 = p0;
    }
  }
  // the largest |lambda_lm| of the ring is brought to about 1, by at most 2^kRingScaleMax
  cexp[(size_t)blockIdx.y * ldc + r] = (int8_t)min(max(1023 - (top >> 20), 0), kRingScaleMax);
}

// One warp per row (l, m): the exponent of its largest scaled value and its
// first ring block with a digit.
__global__ void k_dig_rows(int lmax, int R, int ms, const long long* __restrict__ off, const double* __restrict__ tab,
                           const int8_t* __restrict__ cexp, int ldc, const int* __restrict__ gidx,
                           int* __restrict__ rexp, int* __restrict__ rb0) {
  const int ml = blockIdx.y, m = ms + ml;
  const int l = m + blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (l > lmax + 1) return;
  const double* row = tab + off[ml] + (size_t)(l - m) * R;
  const int8_t* c = cexp + (size_t)ml * ldc;
  int top = 0;
  for (int r = lane; r < R; r += 32) {
    const int h = abs_hi(row[r]);
    if (h >= 0x00100000) top = max(top, h + ((int)c[r] << 20));
  }
  top = __reduce_max_sync(0xffffffffu, top);
  const int er = top ? (top >> 20) - 1022 : 0;    // |value| < 2^er
  const int least = (er - 63 + 1023) << 20;       // values below 2^(er - 63) round to zero digits
  int first = R;
  for (int r = lane; r < R; r += 32) {
    const int h = abs_hi(row[r]);
    if (h >= 0x00100000 && h + ((int)c[r] << 20) >= least) {
      first = r;
      break;
    }
  }
  first = __reduce_min_sync(0xffffffffu, first);
  if (lane == 0) {
    const int k = (l - m) >> 1;
    const int b = gidx[2 * ml + ((l - m) & 1)] + (k >> 6);
    rexp[(size_t)b * 64 + (k & 63)] = er;
    atomicMin(rb0 + b, first >> 6);
  }
}

// One CTA per atom: FP64 values to digit planes.
__global__ void __launch_bounds__(256) k_dig_fill(int lmax, int R, int ms, const long long* __restrict__ off,
                                                  const double* __restrict__ tab, const int8_t* __restrict__ cexp,
                                                  int ldc, const int* __restrict__ gidx, const int* __restrict__ grp,
                                                  const int* __restrict__ rexp, const int* __restrict__ rb0,
                                                  __half* const* __restrict__ abase, int blk0) {
  const int blk = blk0 + blockIdx.x, rb = blockIdx.y;
  const int first = rb0[blk];
  if (rb < first) return;
  const int g = grp[blockIdx.x];                  // group within the segment's orders
  const int ml = g >> 1, m = ms + ml;
  const int k0 = (blk - gidx[g]) * 64;
  __half* atom = abase[blk] + (size_t)(rb - first) * kDigits * kAtom;
  for (int u = threadIdx.x; u < 512; u += 256) {
    const int row = u >> 3, ch = u & 7;
    const int l = m + (g & 1) + 2 * (k0 + row);
    const bool ok = l <= lmax + 1;
    const int er = rexp[(size_t)blk * 64 + row];
    const double* src = tab + off[ml] + (size_t)(l - m) * R;
    unsigned long long y[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int r = rb * 64 + ch * 8 + q;
      y[q] = ok && r < R ? dig_of(src[r], (int)cexp[(size_t)ml * ldc + r] + 62 - er) : dig_of(0.0, 0);
    }
#pragma unroll
    for (int s = 0; s < kDigits; ++s)
      *reinterpret_cast<uint4*>(atom + s * kAtom + dig_off(row, ch * 8)) =
          make_uint4(dig_pair(y[0], y[1], s), dig_pair(y[2], y[3], s), dig_pair(y[4], y[5], s), dig_pair(y[6], y[7], s));
  }
}

__global__ void k_ring_factors(int nside, double* __restrict__ fac) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= 2 * nside) return;
  const Ring g = ring_geom(nside, r + 1);
  const double is2 = 1.0 / (g.s * g.s);
  fac[r] = g.z * is2;
  fac[2 * nside + r] = is2;
}

__global__ void k_eps_table(int lmax, int m0, double* __restrict__ eps, double* __restrict__ by_l) {
  const int l = blockIdx.x * blockDim.x + threadIdx.x, m = m0 + blockIdx.y, ld = lmax + 3;
  if (l >= ld) return;
  eps[(size_t)blockIdx.y * ld + l] =
      l > m ? sqrt(((double)l * l - (double)m * m) / (4.0 * l * l - 1.0)) : 0.0;
  if (blockIdx.y == 0) {
    by_l[l] = l > 0 ? -1.0 / ((double)l * (l + 1.0)) : 0.0;
    by_l[ld + l] = l > 1 ? 1.0 / sqrt((l + 2.0) * (l + 1.0) * l * (l - 1.0)) : 0.0;
  }
}

static int row_blocks(int lt, int m, int p) { return m + p <= lt ? ((lt - m - p) / 2 + 1 + 63) / 64 : 0; }

static bool dev_alloc(Buffer& b, size_t bytes) {
  if (b.p && b.bytes >= bytes) return true;
  if (b.p) cudaFree(b.p);
  b.bytes = std::max(bytes, (size_t)16);
  if (cudaMalloc(&b.p, b.bytes) != cudaSuccess) {
    cudaGetLastError();
    b.p = nullptr;
    b.bytes = 0;
    return false;
  }
  return true;
}

int build_legendre_table(clc_ctx* ctx, int nside, int lmax, int m0, int m1, size_t limit, bool stays, LegendreBuild& W,
                         LegendreTable* T) {
  const int lt = lmax + 1, R = 2 * nside, nkb = (R + 63) / 64, ldc = nkb * 64;
  int nm = m1 - m0;
  T->nside = nside;
  T->lmax = lmax;
  T->R = R;
  T->nkb = nkb;
  T->m0 = m0;
  T->m1 = m1;
  T->bytes = 0;
  T->h_gidx.assign(2 * nm + 1, 0);
  for (int g = 0; g < 2 * nm; ++g) T->h_gidx[g + 1] = T->h_gidx[g] + row_blocks(lt, m0 + (g >> 1), g & 1);
  const int nblk = T->h_gidx[2 * nm];
  std::vector<int> h_rb0(nblk, nkb);
  std::vector<__half*> h_abase(nblk, nullptr);
  // log2 of sqrt((2m+1)!! / (4 pi (2m)!!))
  std::vector<double> lognorm(lmax + 1);
  double ln = 0.5 * std::log2(1.0 / (4.0 * kPi));
  for (int m = 0; m <= lmax; ++m) {
    if (m > 0) ln += 0.5 * std::log2((2.0 * m + 1.0) / (2.0 * m));
    lognorm[m] = ln;
  }
  // A segment: orders whose FP64 values fit the build buffer and whose digits
  // (1.6 times those bytes with the usual polar cut) about fill the limit.
  auto order_bytes = [&](int m) { return (size_t)(lt - m + 1) * R * sizeof(double); };
  auto segment_end = [&](int ms) {
    const size_t room = std::min<size_t>(kSegBytes, (limit - std::min(limit, T->bytes)) / 8 * 5);
    size_t acc = order_bytes(ms);
    int me = ms + 1;
    while (me < m1 && acc + order_bytes(me) <= room) acc += order_bytes(me++);
    return me;
  };
  size_t tab_bytes = 0;
  for (int m = m0; m < m1 && tab_bytes < kSegBytes; ++m) tab_bytes += order_bytes(m);
  tab_bytes = std::max(order_bytes(m0), std::min(std::min<size_t>(tab_bytes, kSegBytes), limit / 8 * 5));
  const char* what = "Legendre table allocation failed";
  if (!dev_alloc(T->gidx, sizeof(int) * (2 * nm + 1)) || !dev_alloc(T->rb0, sizeof(int) * nblk) ||
      !dev_alloc(T->abase, sizeof(__half*) * nblk) || !dev_alloc(T->rexp, sizeof(int) * 64 * (size_t)nblk) ||
      !dev_alloc(T->cexp, (size_t)nm * ldc) || !dev_alloc(T->fac, sizeof(double) * 2 * R) ||
      !dev_alloc(T->zero, (size_t)kDigits * kAtom * sizeof(__half)) ||
      !dev_alloc(T->eps, sizeof(double) * (size_t)(nm + 2) * (lmax + 3)) || !dev_alloc(W.tab, tab_bytes) ||
      !dev_alloc(W.ab, sizeof(double2) * (size_t)nm * (lt + 1)) ||
      !dev_alloc(W.ln, sizeof(double) * lognorm.size()) || !dev_alloc(W.off, sizeof(long long) * nm) ||
      !dev_alloc(W.grp, sizeof(int) * nblk))
    return set_err(ctx, CLC_ENOMEM, what);
  if (stays ? !T->atoms.empty() : !T->arena) {
    if (int e = cuda_check(ctx, cudaStreamSynchronize(ctx->stream), "table chunk")) return e;
    T->atoms.clear();
  }
  T->arena = !stays;
  if (!stays && T->atoms.empty()) {
    T->atoms.push_back(std::make_unique<Buffer>());
    if (!dev_alloc(*T->atoms[0], std::min(limit, (size_t)nblk * nkb * kDigits * kAtom * sizeof(__half))))
      return set_err(ctx, CLC_ENOMEM, what);
  }
  cudaStream_t st = ctx->stream;
  cudaMemcpyAsync(T->gidx.p, T->h_gidx.data(), sizeof(int) * (2 * nm + 1), cudaMemcpyHostToDevice, st);
  cudaMemcpyAsync(T->rb0.p, h_rb0.data(), sizeof(int) * nblk, cudaMemcpyHostToDevice, st);
  cudaMemcpyAsync(W.ln.p, lognorm.data(), sizeof(double) * lognorm.size(), cudaMemcpyHostToDevice, st);
  cudaMemsetAsync(T->rexp.p, 0, T->rexp.bytes, st);
  cudaMemsetAsync(T->cexp.p, 0, T->cexp.bytes, st);
  cudaMemsetAsync(T->zero.p, 0, T->zero.bytes, st);
  CLC_LAUNCH(ctx, "k_ring_factors", k_ring_factors, (R + 127) / 128, 128, 0, nside, (double*)T->fac.p);
  int rc;
  for (int ms = m0; ms < T->m1;) {
    int me = segment_end(ms);
    const int n = me - ms, g0 = 2 * (ms - m0), b0 = T->h_gidx[g0];
    int b1 = T->h_gidx[2 * (me - m0)];
    std::vector<long long> off(n);
    long long a = 0;
    for (int m = ms; m < me; ++m) {
      off[m - ms] = a;
      a += (long long)(lt - m + 1) * R;
    }
    std::vector<int> grp(std::max(b1 - b0, 1));
    for (int g = 0; g < 2 * n; ++g)
      for (int b = T->h_gidx[g0 + g]; b < T->h_gidx[g0 + g + 1]; ++b) grp[b - b0] = g;
    cudaMemcpyAsync(W.off.p, off.data(), sizeof(long long) * n, cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(W.grp.p, grp.data(), sizeof(int) * (b1 - b0), cudaMemcpyHostToDevice, st);
    int8_t* cx = (int8_t*)T->cexp.p + (size_t)(ms - m0) * ldc;
    const int* gx = (const int*)T->gidx.p + g0;
    CLC_LAUNCH(ctx, "k_legendre_coef", k_legendre_coef, dim3((lt + 128) / 128, n), 128, 0, lt, ms, (double2*)W.ab.p);
    CLC_LAUNCH(ctx, "k_legendre_build", k_legendre_build, dim3((R + 127) / 128, n), 128, 0, nside, lmax, R,
               (const long long*)W.off.p, (const double*)W.ln.p, (const double2*)W.ab.p, (double*)W.tab.p, ms, cx, ldc);
    CLC_LAUNCH(ctx, "k_dig_rows", k_dig_rows, dim3((lt - ms + 8) / 8, n), 256, 0, lmax, R, ms, (const long long*)W.off.p,
               (const double*)W.tab.p, (const int8_t*)cx, ldc, gx, (int*)T->rexp.p, (int*)T->rb0.p);
    if ((rc = launch_check(ctx, "Legendre table rows"))) return rc;
    cudaMemcpyAsync(h_rb0.data() + b0, (const int*)T->rb0.p + b0, sizeof(int) * (b1 - b0), cudaMemcpyDeviceToHost, st);
    if ((rc = cuda_check(ctx, cudaStreamSynchronize(st), "Legendre table rows"))) return rc;
    // a row block keeps at least the ring blocks of the one before it (lower l);
    // the segment ends with the last order that fits the limit
    size_t bytes = 0;
    for (int m = ms; m < me; ++m) {
      size_t natom = 0;
      for (int g = 2 * (m - m0); g < 2 * (m - m0) + 2; ++g)
        for (int b = T->h_gidx[g]; b < T->h_gidx[g + 1]; ++b) {
          if (b > T->h_gidx[g]) h_rb0[b] = std::min(h_rb0[b], h_rb0[b - 1]);
          natom += nkb - h_rb0[b];
        }
      natom *= kDigits * kAtom * sizeof(__half);
      if (m > m0 && T->bytes + bytes + natom > limit) {
        T->m1 = me = m;
        break;
      }
      bytes += natom;
    }
    if (me == ms) break;
    b1 = T->h_gidx[2 * (me - m0)];
    if (stays) T->atoms.push_back(std::make_unique<Buffer>());
    Buffer& mem = *T->atoms.back();
    const size_t at0 = stays ? 0 : T->bytes;
    if (!dev_alloc(mem, at0 + bytes))   // an arena grows for a first order above the limit only
      return set_err(ctx, CLC_ENOMEM, "Legendre table of " + std::to_string(bytes >> 20) + " MiB does not fit");
    __half* at = (__half*)((uint8_t*)mem.p + at0);
    for (int b = b0; b < b1; ++b) {
      h_abase[b] = at;
      at += (size_t)(nkb - h_rb0[b]) * kDigits * kAtom;
    }
    cudaMemcpyAsync((int*)T->rb0.p + b0, h_rb0.data() + b0, sizeof(int) * (b1 - b0), cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync((__half**)T->abase.p + b0, h_abase.data() + b0, sizeof(__half*) * (b1 - b0), cudaMemcpyHostToDevice,
                    st);
    if (b1 > b0)
      CLC_LAUNCH(ctx, "k_dig_fill", k_dig_fill, dim3(b1 - b0, nkb), 256, 0, lmax, R, ms, (const long long*)W.off.p,
                 (const double*)W.tab.p, (const int8_t*)cx, ldc, gx, (const int*)W.grp.p, (const int*)T->rexp.p,
                 (const int*)T->rb0.p, (__half* const*)T->abase.p, b0);
    // the host arrays of the segment and the build buffers are reused: wait
    if ((rc = launch_check(ctx, "k_dig_fill"))) return rc;
    if ((rc = cuda_check(ctx, cudaStreamSynchronize(st), "Legendre table build"))) return rc;
    T->bytes += bytes;
    ms = me;
    if (!stays && T->bytes > limit / 8 * 7) T->m1 = me;
  }
  nm = T->m1 - m0;
  T->h_gidx.resize(2 * nm + 1);
  CLC_LAUNCH(ctx, "k_eps_table", k_eps_table, dim3((lmax + 130) / 128, nm), 128, 0, lmax, m0, (double*)T->eps.p,
             (double*)T->eps.p + (size_t)nm * (lmax + 3));
  if ((rc = launch_check(ctx, "k_eps_table"))) return rc;
  // work lists.  Analysis: (group, 128-row tile, first ring block); synthesis:
  // (order, 128-ring tile, first row blocks of the two parities).
  std::vector<std::pair<int, int4>> an, sy;
  for (int g = 0; g < 2 * nm; ++g) {
    const int nb = T->h_gidx[g + 1] - T->h_gidx[g];
    for (int t = 0; 2 * t < nb; ++t) {
      const int first = h_rb0[T->h_gidx[g] + std::min(2 * t + 1, nb - 1)];
      an.push_back({nkb - first, make_int4(g, t, first, 0)});
    }
  }
  for (int m = 0; m < nm; ++m)
    for (int t = 0; 2 * t < nkb; ++t) {
      int first[2], len = 0;
      for (int p = 0; p < 2; ++p) {
        const int gb = T->h_gidx[2 * m + p], nb = T->h_gidx[2 * m + p + 1] - gb;
        int b = 0;
        while (b < nb && h_rb0[gb + b] > std::min(2 * t + 1, nkb - 1)) ++b;
        first[p] = b;
        len += nb - b;
      }
      sy.push_back({len, make_int4(m, t, first[0], first[1])});
    }
  auto upload = [&](std::vector<std::pair<int, int4>>& v, Buffer& buf, int* count) -> int {
    std::stable_sort(v.begin(), v.end(), [](const auto& x, const auto& y) { return x.first > y.first; });
    std::vector<int4> it;
    for (auto& x : v) it.push_back(x.second);
    *count = (int)it.size();
    if (!dev_alloc(buf, sizeof(int4) * it.size())) return set_err(ctx, CLC_ENOMEM, what);
    return cuda_check(ctx, cudaMemcpy(buf.p, it.data(), sizeof(int4) * it.size(), cudaMemcpyHostToDevice), "work list");
  };
  if ((rc = upload(an, T->an, &T->n_an))) return rc;
  return upload(sy, T->sy, &T->n_sy);
}

// ---------------------------------------------------------------------------
// data operands: columns of doubles to digit planes.  Block of 64 terms:
// kDigits x kCols rows (digit plane j, column c at row j kCols + c) of 64
// halves; rows of columns not in use are left as they are (they only reach
// accumulator columns that nothing reads).

constexpr int kCols = 16;                          // real columns of a contraction
constexpr int kOpBlock = kDigits * kCols * 64;     // halves of a block

static size_t analysis_op_bytes(int nm, int nkb) { return (size_t)2 * nm * nkb * kOpBlock * sizeof(__half); }
static size_t synthesis_op_bytes(int nblk) { return (size_t)nblk * kOpBlock * sizeof(__half); }

// What a table may take is its budget, or the free memory less the operands, the
// build buffers and 2 GiB; what it does take is known when its rows are (the
// atoms below the polar cut are not stored: 7.74 of at most 9.69 GB at nside 512,
// lmax 1024), so it is built until the limit is reached rather than compared with
// a bound.  When a pass has shown that the whole table exceeds the budget, and
// more than half of it fits, the first orders stay in three quarters of the budget
// and the others are rebuilt in the rest.  Solve with fields at nside 512, lmax
// 1024: 6.1 ms from 7.8 GB on, 12.7 with 7, 15.5 with 4.6, 21.5 with 3 and 23.3
// with 0.5 (compared with the bound and with memory of its own for every range:
// 25.9 with 7.5 and 26.9 with 4.6; the FP64 table before, 4.3 GB, took 19.2 from
// there on and 33.9 with 3); at nside 2048, lmax 4096: 888 ms (1207; 2172).  A
// call on a kept table does not ask for the free memory (10 us of a small one).
int legendre_table_from(clc_ctx* ctx, int nside, int lmax, int m0, LegendreBuild& W,
                        std::shared_ptr<LegendreTable>& own, std::shared_ptr<LegendreTable>* out) {
  const std::pair<int, int> key(nside, lmax);
  const size_t budget = ctx->table_budget;
  const auto known = ctx->leg_bytes.find(key);
  const size_t total = known == ctx->leg_bytes.end() ? 0 : known->second;   // 0: not known yet
  auto it = ctx->leg_tables.find(key);
  size_t held = 0;
  if (it != ctx->leg_tables.end() && !(budget && it->second->bytes > budget)) {
    const LegendreTable& C = *it->second;
    if (m0 >= C.m1) {
      held = C.bytes;
    } else if (C.m1 > lmax || (budget && total > budget)) {
      *out = it->second;
      return CLC_OK;
    } else {   // a part kept under an earlier, smaller budget
      if (int rc = cuda_check(ctx, cudaStreamSynchronize(ctx->stream), "Legendre table")) return rc;
      ctx->leg_tables.erase(it);
      it = ctx->leg_tables.end();
    }
  }
  if (own && own->arena) {   // the next range of a pass
    *out = own;
    return build_legendre_table(ctx, nside, lmax, m0, lmax + 1, own->atoms[0]->bytes, false, W, own.get());
  }
  const bool first = m0 == 0 && it == ctx->leg_tables.end();
  const int nkb = (2 * nside + 63) / 64;
  size_t nblk = 0, build = 0, freeb = 0, totalb = 0;
  for (int m = 0; m <= lmax; ++m) {
    nblk += row_blocks(lmax + 1, m, 0) + row_blocks(lmax + 1, m, 1);
    build += (size_t)(lmax + 2 - m) * 2 * nside * sizeof(double);
  }
  cudaMemGetInfo(&freeb, &totalb);
  if (own)   // a first range that did not take every order: its memory is given back
    for (auto& p : own->atoms) freeb += p->bytes;
  auto grow = [&](int slot, size_t bytes) { return bytes > ctx->scratch[slot].bytes ? bytes : 0; };
  const size_t reserve = (2ull << 30) + std::min(build, kSegBytes) + grow(8, analysis_op_bytes(lmax + 1, nkb)) +
                         grow(9, synthesis_op_bytes((int)nblk));
  const size_t room = freeb > reserve + reserve / 2 ? freeb - reserve : freeb / 4;
  size_t limit = std::min<size_t>(room, 48ull << 30);
  bool stays = false;
  if (first && total <= (budget ? std::min(budget, room) : room)) {
    stays = true;
    limit = budget ? std::min(budget, room) : room;
  } else if (first && budget > total / 2 && budget <= room) {
    stays = true;
    limit = budget - budget / 4;
  } else if (budget) {
    limit = std::min(limit, budget - held);
  }
  if (!own) own = std::make_shared<LegendreTable>();
  if (int rc = build_legendre_table(ctx, nside, lmax, m0, lmax + 1, limit, stays, W, own.get())) return rc;
  *out = own;
  if (first && stays && (own->m1 > lmax || total > limit)) {
    ctx->leg_tables[key] = own;
    own.reset();
  }
  return CLC_OK;
}

// block-wide maxima of four non-negative integers (results in all threads)
__device__ __forceinline__ void block_max4(int v[4], int* sh) {
  const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __syncthreads();   // earlier readers of sh are done
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int x = __reduce_max_sync(0xffffffffu, v[i]);
    if ((threadIdx.x & 31) == 0) sh[4 * warp + i] = x;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    v[i] = sh[i];
    for (int w = 1; w < nw; ++w) v[i] = max(v[i], sh[4 * w + i]);
  }
}

// exponent e of a column with largest absolute high word `hi` (|value| < 2^e)
__device__ __forceinline__ int col_exp(int hi) {
  if (hi >= 0x7ff00000) return kNonFinite;
  return hi ? max(hi >> 20, 1) - 1022 : 0;
}

// high word of |v| scaled by a power of two given as an exponent field (0 for a
// zero or a result below the normal range; infinities and NaN stay)
__device__ __forceinline__ int scaled_hi(double v, int field) {
  const int h = abs_hi(v);
  if (h >= 0x7ff00000) return 0x7ff00000;
  return h < 0x00100000 || h + field < 0x00100000 ? 0 : min(h + field, 0x7fefffff);
}

struct AnaCols {
  const double2* F[8];
  int kind[8];
  int nv;
};

// One CTA per order; column 2 v + re/im of both parities.
__global__ void __launch_bounds__(256) k_dig_pack_analysis(AnaCols a, int nside, int R, int nkb, int ldf, int m0,
                                                           const int8_t* __restrict__ cexp,
                                                           const double* __restrict__ fac, __half* __restrict__ op,
                                                           int* __restrict__ colexp) {
  __shared__ int sh[4 * 8];
  const int ml = blockIdx.x, m = m0 + ml;
  const int8_t* cx = cexp + (size_t)ml * nkb * 64;
  for (int v = blockIdx.y; v < a.nv; v += gridDim.y) {
    const double2* F = a.F[v] + (size_t)m * ldf;
    const int kind = a.kind[v];
    // (even re, even im, odd re, odd im) of ring r
    auto vals = [&](int r, double x[4]) {
      if (r >= R) {
        x[0] = x[1] = x[2] = x[3] = 0.0;
        return;
      }
      const double2 n = F[r];
      double2 s = make_double2(0.0, 0.0);
      if (r + 1 != 2 * nside) s = F[4 * nside - r - 2];
      if (kind == 1) s = make_double2(-s.x, -s.y);
      x[0] = n.x + s.x;
      x[1] = n.y + s.y;
      x[2] = n.x - s.x;
      x[3] = n.y - s.y;
      if (kind) {
        const double w = fac[(size_t)(kind - 1) * R + r];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] *= w;
      }
    };
    int top[4] = {0, 0, 0, 0};
    for (int r = threadIdx.x; r < R; r += 256) {
      double x[4];
      vals(r, x);
      const int c = (int)cx[r] << 20;
#pragma unroll
      for (int i = 0; i < 4; ++i) top[i] = max(top[i], scaled_hi(x[i], -c));
    }
    block_max4(top, sh);
    int ec[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) ec[i] = col_exp(top[i]);
    if (threadIdx.x < 4)
      colexp[(size_t)(2 * ml + (threadIdx.x >> 1)) * kCols + 2 * v + (threadIdx.x & 1)] = ec[threadIdx.x];
    for (int r = 2 * threadIdx.x; r < nkb * 64; r += 512) {
      double x0[4], x1[4];
      vals(r, x0);
      vals(r + 1, x1);
      const int c0 = cx[r], c1 = cx[r + 1];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const bool ok = ec[i] != kNonFinite;
        const unsigned long long y0 = ok ? dig_of(x0[i], 62 - ec[i] - c0) : 0;
        const unsigned long long y1 = ok ? dig_of(x1[i], 62 - ec[i] - c1) : 0;
        __half* dst = op + ((size_t)(2 * ml + (i >> 1)) * nkb + (r >> 6)) * kOpBlock;
#pragma unroll
        for (int s = 0; s < kDigits; ++s)
          *reinterpret_cast<unsigned*>(dst + dig_off(s * kCols + 2 * v + (i & 1), r & 63)) = dig_pair(y0, y1, s);
      }
    }
  }
}

// Right-hand sides of a synthesis: given (rhs, packed with band limit lmax + 1),
// or those of a Poisson solve of the coefficients klm (packed with lmax).
struct SynthRhs {
  const double2* rhs;
  int nq;
  int lq[4];
  const double2* klm;
  const double* eps;    // [m - m0][lmax + 3]
  const double* inv;    // -1 / (l (l + 1))
};

// value of right-hand side q at (l, m), l <= lmax + 1
template <bool kPoisson>
__device__ __forceinline__ double2 synth_rhs(const SynthRhs& s, int q, int lmax, int l, int m, int ml) {
  if (!kPoisson) {
    if (l > s.lq[q]) return make_double2(0.0, 0.0);
    const int lt = lmax + 1;
    return s.rhs[(size_t)q * (alm_idx(lt, lt, lt) + 1) + alm_idx(lt, l, m)];
  }
  auto psi = [&](int ll) -> double2 {
    if (ll < m || ll > lmax) return make_double2(0.0, 0.0);
    const double2 k = s.klm[alm_idx(lmax, ll, m)];
    const double d = s.inv[ll];
    return make_double2(k.x * d, k.y * d);
  };
  if (q == 0) return psi(l);
  if (q == 2) {
    const double2 p = psi(l);
    const double ll1 = -(double)l * (l + 1.0);
    return make_double2(ll1 * p.x, ll1 * p.y);
  }
  const double2 pm = psi(l - 1), pp = psi(l + 1);
  const double* e = s.eps + (size_t)ml * (lmax + 3);
  const double c1 = (l - 1.0) * e[l], c2 = (l + 2.0) * e[l + 1];
  return make_double2(c1 * pm.x - c2 * pp.x, c1 * pm.y - c2 * pp.y);
}

// One CTA per order and right-hand side; column 2 q + re/im of both parities
// (rows l = m + p + 2 k). A Poisson solve's right-hand sides are formed here
// from its coefficients and the table's eps_lm: written out first by a kernel of
// their own they cost two FP64 square roots and divisions per row (94 us at
// nside 512) and a launch. Solve with derivatives, before and after: nside 64
// 151 -> 145 us, nside 512 6117 -> 6076 us.
template <bool kPoisson>
__global__ void __launch_bounds__(256) k_dig_pack_synthesis(SynthRhs s, int lmax, int m0, const int* __restrict__ gidx,
                                                            const int* __restrict__ rexp, __half* __restrict__ op,
                                                            int* __restrict__ colexp) {
  __shared__ int sh[4 * 8];
  const int ml = blockIdx.x, m = m0 + ml, lt = lmax + 1, q = blockIdx.y;
  const int gb[3] = {gidx[2 * ml], gidx[2 * ml + 1], gidx[2 * ml + 2]};
  const int np = max(gb[1] - gb[0], gb[2] - gb[1]) * 32;   // pairs of rows
  // (re, im) of row k of parity p and the row's exponent
  auto val = [&](int p, int k, int& e) -> double2 {
    const int l = m + p + 2 * k;
    e = 0;
    if (l > lt) return make_double2(0.0, 0.0);
    e = rexp[(size_t)gb[p] * 64 + k];
    return synth_rhs<kPoisson>(s, q, lmax, l, m, ml);
  };
  int top[4] = {0, 0, 0, 0};
  for (int k = threadIdx.x; k < 2 * np; k += 256) {
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      int e;
      const double2 v = val(p, k, e);
      top[2 * p] = max(top[2 * p], scaled_hi(v.x, e * 0x100000));
      top[2 * p + 1] = max(top[2 * p + 1], scaled_hi(v.y, e * 0x100000));
    }
  }
  block_max4(top, sh);
  int ec[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) ec[i] = col_exp(top[i]);
  if (threadIdx.x < 4)
    colexp[(size_t)(2 * ml + (threadIdx.x >> 1)) * kCols + 2 * q + (threadIdx.x & 1)] = ec[threadIdx.x];
  for (int t = threadIdx.x; t < np; t += 256) {
    const int k = 2 * t;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      if (k >= (gb[p + 1] - gb[p]) * 64) continue;
      int ea, eb;
      const double2 a = val(p, k, ea), b = val(p, k + 1, eb);
      __half* dst = op + (size_t)(gb[p] + (k >> 6)) * kOpBlock;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int e = ec[2 * p + i];
        const bool ok = e != kNonFinite;
        const unsigned long long y0 = ok ? dig_of(i ? a.y : a.x, 62 - e + ea) : 0;
        const unsigned long long y1 = ok ? dig_of(i ? b.y : b.x, 62 - e + eb) : 0;
#pragma unroll
        for (int j = 0; j < kDigits; ++j)
          *reinterpret_cast<unsigned*>(dst + dig_off(j * kCols + 2 * q + i, k & 63)) = dig_pair(y0, y1, j);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// contractions: persistent, warp-specialised, bulk-copy pipelined
//
// Analysis item (group, 128-row tile): the terms are rings, blocks of 64 from
// the first one with a digit to the equator; A = two atoms (row blocks 2 t and
// 2 t + 1 of the ring block), K-major.  Synthesis item (order, 128-ring tile):
// the terms are rows of parity 0, then of parity 1; A = two atoms (ring blocks
// 2 t and 2 t + 1 of the row block), MN-major.  A block's eight digit planes of
// A (16 KB each) pass through a ring of eight stages; its B operand (all digit
// planes of the data) comes with the first.  Plane i is multiplied by the data
// planes 0 .. 7 - i at once (N = (8 - i) kCols columns) into the accumulator
// columns from i kCols on, so that column block g collects the digit pairs i + j =
// g.  After kDigFlush blocks the four epilogue warps (one row per thread) move
// the sums into 64-bit integers: hi = D0 2^24 + D1 2^16 + D2 2^8 + D3 and lo =
// D4 2^24 + D5 2^16 + D6 2^8 + D7 (the value is hi 2^32 + lo); two accumulators alternate.
// Two data blocks suffice: with eight stages the copy that refills a data
// block is issued after the empty barrier of that block's last plane.
// Warps 0-3: epilogue (TMEM lanes 32w .. 32w + 31), warp 4: bulk copies, warp 5: MMAs.

struct DigArgs {
  const __half* const* abase;
  const int* rb0;
  const int* gidx;
  const __half* zero;
  const __half* op;
  const int* rexp;
  const int* colexp;
  const int8_t* cexp;
  int nside, lmax, R, nkb, m0;
  int nv;             // complex columns
  double2* out[8];    // analysis
  int ltop;           // analysis: highest l, band limit of the packing
  double2* G;         // synthesis
  size_t qstride;
  int ld;
};

template <int N>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t* r);
template <>
__device__ __forceinline__ void tmem_ld<2>(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(taddr));
}
template <>
__device__ __forceinline__ void tmem_ld<8>(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
template <>
__device__ __forceinline__ void tmem_ld<16>(uint32_t taddr, uint32_t* r) {
  tmem_ld<8>(taddr, r);
  tmem_ld<8>(taddr + 8, r + 8);
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// blocks of 64 terms of an item: n[0] of the first, n[1] of the second phase
template <bool kSyn>
__device__ __forceinline__ void dig_counts(const DigArgs& a, int4 w, int n[2]) {
  if (kSyn) {
    n[0] = a.gidx[2 * w.x + 1] - a.gidx[2 * w.x] - w.z;
    n[1] = a.gidx[2 * w.x + 2] - a.gidx[2 * w.x + 1] - w.w;
  } else {
    n[0] = a.nkb - w.z;
    n[1] = 0;
  }
}

template <bool kSyn, int NC>
__global__ void __launch_bounds__(192) k_dig_gemm(DigArgs a, const int4* __restrict__ items, int nitems, int* d_err) {
  constexpr uint32_t kOpBytes = kOpBlock * 2;   // a data block
  constexpr uint32_t kAcc = 128;                // TMEM columns of an accumulator (kDigits kCols)
  extern __shared__ __align__(16) uint8_t smem_g[];
  __shared__ uint64_t full[kDigStages], empty[kDigStages], chunkb[2], freeb[2], drainb;
  __shared__ uint32_t tmem_base;
  __shared__ volatile int abort_flag;
  const uint32_t raw = umma::smem_u32(smem_g);
  uint8_t* base = smem_g + (((raw + 1023u) & ~1023u) - raw);
  uint8_t* opb = base + kDigStages * 16384;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kDigStages; ++s) {
      umma::mbar_init(&full[s], 1);
      umma::mbar_init(&empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      umma::mbar_init(&chunkb[s], 1);
      umma::mbar_init(&freeb[s], 128);
    }
    umma::mbar_init(&drainb, 1);
    abort_flag = 0;
    umma::fence_mbar_init();
  }
  if (warp == 0) umma::tmem_alloc(&tmem_base, 2 * kAcc);
  umma::fence_before_sync();
  __syncthreads();
  umma::fence_after_sync();
  const uint32_t tmem = tmem_base;
  auto fail = [&]() {
    atomicCAS(d_err, 0, kDevTimeout);
    abort_flag = 1;
  };

  if (warp == 4) {
    // ---- producer
    if (lane == 0) {
      uint32_t it = 0, blk = 0;
      int last_it[kDigStages];
      for (int s = 0; s < kDigStages; ++s) last_it[s] = -1;
      for (int item = blockIdx.x; item < nitems && !abort_flag; item += gridDim.x) {
        const int4 w = items[item];
        int n[2];
        dig_counts<kSyn>(a, w, n);
        for (int ph = 0; ph < 2 && !abort_flag; ++ph) {
          // analysis: the two row blocks of the tile
          int i0 = 0, s0 = 0, s1 = a.nkb;
          const __half *b0 = nullptr, *b1 = nullptr;
          if (!kSyn && n[0] > 0) {
            i0 = a.gidx[w.x] + 2 * w.y;
            s0 = a.rb0[i0];
            b0 = a.abase[i0];
            if (i0 + 1 < a.gidx[w.x + 1]) {
              s1 = a.rb0[i0 + 1];
              b1 = a.abase[i0 + 1];
            }
          }
          for (int k = 0; k < n[ph] && !abort_flag; ++k, ++blk) {
            const __half *p0 = a.zero, *p1 = a.zero, *op;
            if (kSyn) {
              const int idx = a.gidx[2 * w.x + ph] + (ph ? w.w : w.z) + k;
              const int first = a.rb0[idx], rb = 2 * w.y;
              const __half* b = a.abase[idx];
              if (rb >= first) p0 = b + (size_t)(rb - first) * kDigits * kAtom;
              if (rb + 1 < a.nkb && rb + 1 >= first) p1 = b + (size_t)(rb + 1 - first) * kDigits * kAtom;
              op = a.op + (size_t)idx * kOpBlock;
            } else {
              const int rb = w.z + k;
              if (rb >= s0) p0 = b0 + (size_t)(rb - s0) * kDigits * kAtom;
              if (rb >= s1) p1 = b1 + (size_t)(rb - s1) * kDigits * kAtom;
              op = a.op + ((size_t)w.x * a.nkb + rb) * kOpBlock;
            }
            for (int d = 0; d < kDigits; ++d, ++it) {
              const int s = (int)(it % kDigStages);
              const uint32_t u = it / kDigStages;
              if (u > 0 && !umma::mbar_wait(&empty[s], (u - 1) & 1u, kDigWaitPolls)) {
                fail();
                break;
              }
              uint8_t* st = base + (size_t)s * 16384;
              umma::mbar_arrive_expect_tx(&full[s], 16384u + (d == 0 ? kOpBytes : 0u));
              umma::bulk_g2s(st, p0 + d * kAtom, 8192u, &full[s]);
              umma::bulk_g2s(st + 8192, p1 + d * kAtom, 8192u, &full[s]);
              if (d == 0) umma::bulk_g2s(opb + (blk & 1u) * kOpBytes, op, kOpBytes, &full[s]);
              last_it[s] = (int)it;
            }
          }
        }
      }
      if (abort_flag)
        for (int s = 0; s < kDigStages; ++s)   // bounded drain of the copies in flight
          if (last_it[s] >= 0) umma::mbar_wait(&full[s], (uint32_t)(last_it[s] / kDigStages) & 1u, kDigWaitPolls);
    }
  } else if (warp == 5) {
    // ---- MMA issuer
    if (lane == 0) {
      uint32_t it = 0, blk = 0, nchunk = 0;
      for (int item = blockIdx.x; item < nitems && !abort_flag; item += gridDim.x) {
        int n[2];
        dig_counts<kSyn>(a, items[item], n);
        for (int ph = 0; ph < 2; ++ph)
          for (int k = 0; k < n[ph] && !abort_flag; ++k, ++blk) {
            const bool first = k % kDigFlush == 0;
            const uint32_t buf = nchunk & 1u;
            if (first && nchunk > 1 && !umma::mbar_wait(&freeb[buf], ((nchunk >> 1) - 1) & 1u, kDigWaitPolls)) {
              fail();   // the epilogue has not released the accumulator
              break;
            }
            const uint32_t sb = umma::smem_u32(opb + (blk & 1u) * kOpBytes);
            for (int d = 0; d < kDigits; ++d, ++it) {
              const int s = (int)(it % kDigStages);
              if (!umma::mbar_wait(&full[s], (it / kDigStages) & 1u, kDigWaitPolls)) {
                fail();
                break;
              }
              umma::fence_after_sync();
              const uint32_t sa = umma::smem_u32(base + (size_t)s * 16384);
              const int N = (kDigits - d) * kCols;
              const uint32_t idesc = kSyn ? umma::idesc_f16_f32_amn(128, N) : umma::idesc_f16_f32(128, N);
              const uint64_t dA = kSyn ? umma::desc_sw128_mn(sa, 8192, 1024) : umma::desc_sw128(sa);
              const uint64_t dB = umma::desc_sw128(sb);
              const uint32_t td = tmem + buf * kAcc + (uint32_t)(d * kCols);
#pragma unroll
              for (int kk = 0; kk < 4; ++kk)
                umma::mma_f16(td, dA + (uint64_t)((kSyn ? kk * 2048 : kk * 32) >> 4), dB + (uint64_t)((kk * 32) >> 4),
                              idesc, (first && d == 0 && kk == 0) ? 0u : 1u);
              umma::commit(&empty[s]);
            }
            if (abort_flag) break;
            if (k % kDigFlush == kDigFlush - 1 || k + 1 == n[ph]) {
              umma::commit(&chunkb[buf]);
              ++nchunk;
            }
          }
      }
      if (abort_flag) {   // bounded wait for the MMAs in flight
        umma::commit(&drainb);
        umma::mbar_wait(&drainb, 0, kDigWaitPolls);
      }
    }
  } else {
    // ---- epilogue warps
    uint32_t nchunk = 0;
    const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16);
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    for (int item = blockIdx.x; item < nitems && !__any_sync(0xffffffffu, abort_flag); item += gridDim.x) {
      const int4 w = items[item];
      int n[2];
      dig_counts<kSyn>(a, w, n);
      double val[kSyn ? 2 : 1][NC];
      bool ok = true;
#pragma unroll
      for (int ph = 0; ph < (kSyn ? 2 : 1); ++ph) {
        long long hi[NC], lo[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) hi[c] = lo[c] = 0;
        for (int k = 0; ok && k < n[ph]; k += kDigFlush, ++nchunk) {
          const uint32_t buf = nchunk & 1u;
          // warp-uniform decision: the TMEM accesses below are whole-warp operations
          const bool got = umma::mbar_wait(&chunkb[buf], (nchunk >> 1) & 1u, kDigWaitPolls);
          if (!__all_sync(0xffffffffu, got)) {
            if (lane == 0) fail();
            ok = false;
            break;
          }
          umma::fence_after_sync();
          uint32_t v[4][NC];
          auto sum4 = [&](int c) {
            return (long long)__float2int_rn(__uint_as_float(v[0][c])) * 16777216 +
                   (long long)__float2int_rn(__uint_as_float(v[1][c])) * 65536 +
                   (long long)__float2int_rn(__uint_as_float(v[2][c])) * 256 + __float2int_rn(__uint_as_float(v[3][c]));
          };
#pragma unroll
          for (int g = 0; g < 4; ++g) tmem_ld<NC>(trow + buf * kAcc + g * kCols, v[g]);
          tmem_wait_ld();
#pragma unroll
          for (int c = 0; c < NC; ++c) hi[c] += sum4(c);
#pragma unroll
          for (int g = 0; g < 4; ++g) tmem_ld<NC>(trow + buf * kAcc + (4 + g) * kCols, v[g]);
          tmem_wait_ld();
          umma::fence_before_sync();
          umma::mbar_arrive(&freeb[buf]);
#pragma unroll
          for (int c = 0; c < NC; ++c) lo[c] += sum4(c);
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) val[ph][c] = fma((double)hi[c], 4294967296.0, (double)lo[c]);
      }
      if (!ok) break;
      __syncwarp();
      if (!kSyn) {
        const int m = a.m0 + (w.x >> 1), k = w.y * 128 + warp * 32 + lane;
        const int l = m + (w.x & 1) + 2 * k;
        if (l <= a.ltop) {
          const int er = a.rexp[(size_t)a.gidx[w.x] * 64 + k] - 68;
          const int* ce = a.colexp + (size_t)w.x * kCols;
          const long long i = alm_idx(a.ltop, l, m);
#pragma unroll
          for (int c = 0; c < NC; c += 2) {
            if (c >= 2 * a.nv) continue;
            const int e0 = ce[c], e1 = ce[c + 1];
            a.out[c >> 1][i] = make_double2(e0 == kNonFinite ? nan : times_pow2(val[0][c], er + e0),
                                            e1 == kNonFinite ? nan : times_pow2(val[0][c + 1], er + e1));
          }
        }
      } else {
        const int m = a.m0 + w.x, r = w.y * 128 + warp * 32 + lane;
        if (r < a.R) {
          const int cr = -68 - (int)a.cexp[(size_t)w.x * a.nkb * 64 + r];
          const int* ce = a.colexp + (size_t)(2 * w.x) * kCols;
#pragma unroll
          for (int c = 0; c < NC; c += 2) {
            if (c >= 2 * a.nv) continue;
            double x[2][2];
#pragma unroll
            for (int p = 0; p < 2; ++p)
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                const int e = ce[p * kCols + c + i];
                x[p][i] = e == kNonFinite ? nan : times_pow2(val[kSyn ? p : 0][c + i], cr + e);
              }
            double2* Gq = a.G + (size_t)(c >> 1) * a.qstride + (size_t)m * a.ld;
            Gq[r] = make_double2(x[0][0] + x[1][0], x[0][1] + x[1][1]);
            if (r + 1 != 2 * a.nside) Gq[4 * a.nside - r - 2] = make_double2(x[0][0] - x[1][0], x[0][1] - x[1][1]);
          }
        }
      }
    }
  }
  umma::fence_before_sync();
  __syncthreads();
  if (warp == 0) umma::tmem_dealloc(tmem, 2 * kAcc);
}

template <bool kSyn, int NC>
static int run_gemm(clc_ctx* ctx, const char* name, const DigArgs& a, const Buffer& items, int n) {
  if (n == 0) return CLC_OK;
  const int smem = 1024 + kDigStages * 16384 + 2 * kOpBlock * 2;
  cudaFuncSetAttribute(k_dig_gemm<kSyn, NC>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  CLC_LAUNCH(ctx, name, (k_dig_gemm<kSyn, NC>), std::min(n, num_sms(ctx)), 192, smem, a, (const int4*)items.p, n,
             ctx->d_err);
  return launch_check(ctx, name);
}

static DigArgs dig_args(const LegendreTable& T, const __half* op, const int* colexp) {
  DigArgs a{};
  a.abase = (const __half* const*)T.abase.p;
  a.rb0 = (const int*)T.rb0.p;
  a.gidx = (const int*)T.gidx.p;
  a.zero = (const __half*)T.zero.p;
  a.op = op;
  a.rexp = (const int*)T.rexp.p;
  a.colexp = colexp;
  a.cexp = (const int8_t*)T.cexp.p;
  a.nside = T.nside;
  a.lmax = T.lmax;
  a.R = T.R;
  a.nkb = T.nkb;
  a.m0 = T.m0;
  return a;
}

// The analysis of one map at low band limits, straight in FP64 on the values the
// digits stand for: a warp per (l, m), its lanes over eight neighbouring rings of
// a row (one 16-byte word per digit plane).  Packing, the contraction's pipeline and
// its walk over the rings take 27 us at nside 128 and 64 at nside 512 however small
// lmax is (the FP64 sums before: 10 and 20 at lmax 16); this way 9.6 and 19.  It is
// FP64 bound (three instructions per value) and grows with lmax^2: it saves 7, 14
// and 20 us at nside 128, 256 and 512 with lmax 100, and loses 5 at the first two
// with lmax 128.  For sht_analysis alone: a_lm are off by 1.5e-16 here (1.9e-16 with
// the FP64 table), where the contraction rounds them once, and a solve, which the
// difference would reach through its synthesis, gains nothing it needs.
constexpr int kRowsLmax = 112;
constexpr int kRowsChunk = 1024;   // rings held at a time

// place of ring t of a chunk: lanes read eight rings each, from different banks
__device__ __forceinline__ int rows_at(int t) { return (t & ~7) | ((t ^ (t >> 3)) & 7); }

__global__ void __launch_bounds__(256) k_legendre_rows(DigArgs a, const double2* __restrict__ Fm, int ldf) {
  __shared__ double2 V[2][kRowsChunk];   // north + (-1)^p south, times 2^(-31 - cexp)
  const int ml = blockIdx.y, m = a.m0 + ml, lane = threadIdx.x & 31;
  const int l = m + blockIdx.x * 8 + (threadIdx.x >> 5), p = (l - m) & 1, row = ((l - m) >> 1) & 63;
  const bool on = l <= a.ltop;
  int first = a.nkb, er = 0;
  const __half* base = nullptr;
  if (on) {
    const int blk = a.gidx[2 * ml + p] + ((l - m) >> 7);
    first = a.rb0[blk];
    base = a.abase[blk];
    er = a.rexp[(size_t)blk * 64 + row];
  }
  const double2* F = Fm + (size_t)m * ldf;
  const int8_t* cx = a.cexp + (size_t)ml * a.nkb * 64;
  double sx = 0.0, sy = 0.0;
  for (int r0 = 0; r0 < a.R; r0 += kRowsChunk) {
    const int n = min(kRowsChunk, a.R - r0);
    __syncthreads();   // the previous chunk is consumed
    for (int t = threadIdx.x; t < n; t += 256) {
      const int r = r0 + t;
      const double2 u = F[r];
      double2 v = make_double2(0.0, 0.0);
      if (r + 1 != 2 * a.nside) v = F[4 * a.nside - r - 2];
      const double w = __longlong_as_double((long long)(1023 - 31 - (int)cx[r]) << 52);
      V[0][rows_at(t)] = make_double2((u.x + v.x) * w, (u.y + v.y) * w);
      V[1][rows_at(t)] = make_double2((u.x - v.x) * w, (u.y - v.y) * w);
    }
    __syncthreads();
    if (!on) continue;
    for (int c = 8 * lane; c < n; c += 256) {
      const int rb = (r0 + c) >> 6;
      unsigned long long y[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) y[q] = rb < first ? 0x8080808080808080ull : 0;
      if (rb >= first) {
        const __half* atom = base + (size_t)(rb - first) * kDigits * kAtom + dig_off(row, c & 63);
#pragma unroll
        for (int s = 0; s < kDigits; ++s) {
          const uint4 d = *reinterpret_cast<const uint4*>(atom + s * kAtom);
          const unsigned w[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
          for (int j = 0; j < 4; ++j) {   // digit + 1152 has digit + 128 as its low byte
            const __half2 h = __hadd2(*reinterpret_cast<const __half2*>(&w[j]), __half2half2(__ushort_as_half(0x6480)));
            const unsigned b = *reinterpret_cast<const unsigned*>(&h);
            y[2 * j] |= (unsigned long long)(b & 255u) << 8 * (kDigits - 1 - s);
            y[2 * j + 1] |= (unsigned long long)((b >> 16) & 255u) << 8 * (kDigits - 1 - s);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (c + q >= n) break;
        const double lam = (double)(long long)(y[q] - 0x8080808080808080ull);
        const double2 v = V[p][rows_at(c + q)];
        sx = fma(lam, v.x, sx);   // (also where lambda is zero: a NaN is not hidden)
        sy = fma(lam, v.y, sy);
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sx += __shfl_xor_sync(0xffffffffu, sx, o);
    sy += __shfl_xor_sync(0xffffffffu, sy, o);
  }
  if (on && lane == 0)
    a.out[0][alm_idx(a.ltop, l, m)] = make_double2(times_pow2(sx, er - 31), times_pow2(sy, er - 31));
}

template <int NC>
static int analysis_cols(clc_ctx* ctx, const LegendreTable& T, const AnaCols& c, int ldf, double2* const* out, int ltop) {
  const int nm = T.m1 - T.m0;
  const size_t ob = analysis_op_bytes(nm, T.nkb);
  __half* op = (__half*)scratch(ctx, 8, ob + sizeof(int) * 2 * nm * kCols);
  if (!op) return CLC_ENOMEM;
  int* colexp = (int*)((uint8_t*)op + ob);
  CLC_LAUNCH(ctx, "k_dig_pack", k_dig_pack_analysis, dim3(nm, c.nv), 256, 0, c, T.nside, T.R, T.nkb, ldf, T.m0,
             (const int8_t*)T.cexp.p, (const double*)T.fac.p, op, colexp);
  if (int rc = launch_check(ctx, "k_dig_pack_analysis")) return rc;
  DigArgs a = dig_args(T, op, colexp);
  a.nv = c.nv;
  for (int v = 0; v < c.nv; ++v) a.out[v] = out[v];
  a.ltop = ltop;
  return run_gemm<false, NC>(ctx, "k_legendre_analysis", a, T.an, T.n_an);
}

int legendre_analysis_map(clc_ctx* ctx, const LegendreTable& T, const double2* F, int ldf, double2* alm) {
  if (T.lmax > kRowsLmax) return legendre_analysis(ctx, T, F, ldf, alm);
  DigArgs a = dig_args(T, nullptr, nullptr);
  a.out[0] = alm;
  a.ltop = T.lmax;
  CLC_LAUNCH(ctx, "k_legendre_analysis", k_legendre_rows, dim3((T.lmax - T.m0) / 8 + 1, T.m1 - T.m0), 256, 0, a, F, ldf);
  return launch_check(ctx, "k_legendre_rows");
}

int legendre_analysis_cols(clc_ctx* ctx, const LegendreTable& T, int nv, const double2* const* F, const int* kind,
                           int ldf, double2* const* out, int ltop) {
  if (ltop < 0) ltop = T.lmax;
  AnaCols c{};
  c.nv = nv;
  for (int v = 0; v < nv; ++v) {
    c.F[v] = F[v];
    c.kind[v] = kind ? kind[v] : 0;
  }
  // the epilogue reads and collects only the columns in use
  if (nv == 1) return analysis_cols<2>(ctx, T, c, ldf, out, ltop);
  if (nv <= 4) return analysis_cols<8>(ctx, T, c, ldf, out, ltop);
  return analysis_cols<16>(ctx, T, c, ldf, out, ltop);
}

template <bool kPoisson>
static int synthesis(clc_ctx* ctx, const LegendreTable& T, const SynthRhs& s, double2* G, int ld) {
  const int nm = T.m1 - T.m0, nblk = T.h_gidx[2 * nm];
  const size_t ob = synthesis_op_bytes(nblk);
  __half* op = (__half*)scratch(ctx, 9, ob + sizeof(int) * 2 * nm * kCols);
  if (!op) return CLC_ENOMEM;
  int* colexp = (int*)((uint8_t*)op + ob);
  CLC_LAUNCH(ctx, "k_dig_pack", k_dig_pack_synthesis<kPoisson>, dim3(nm, s.nq), 256, 0, s, T.lmax, T.m0,
             (const int*)T.gidx.p, (const int*)T.rexp.p, op, colexp);
  if (int rc = launch_check(ctx, "k_dig_pack_synthesis")) return rc;
  DigArgs a = dig_args(T, op, colexp);
  a.nv = s.nq;
  a.G = G;
  a.qstride = (size_t)ld * (T.lmax + 2);
  a.ld = ld;
  return s.nq == 1 ? run_gemm<true, 2>(ctx, "k_legendre_synthesis", a, T.sy, T.n_sy)
                   : run_gemm<true, 8>(ctx, "k_legendre_synthesis", a, T.sy, T.n_sy);
}

int legendre_synthesis(clc_ctx* ctx, const LegendreTable& T, const double2* rhs, int nq, const int* lq, double2* G,
                       int ld) {
  SynthRhs s{};
  s.rhs = rhs;
  s.nq = nq;
  for (int q = 0; q < nq; ++q) s.lq[q] = lq[q];
  return synthesis<false>(ctx, T, s, G, ld);
}

int legendre_synthesis_poisson(clc_ctx* ctx, const LegendreTable& T, const double2* klm, int nq, double2* G, int ld) {
  SynthRhs s{};
  s.nq = nq;
  s.klm = klm;
  s.eps = T.eps_of();
  s.inv = T.by_l();
  return synthesis<true>(ctx, T, s, G, ld);
}

}  // namespace clc
