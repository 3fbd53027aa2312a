// Device side of the ring FFTs (paper Sec. 3.2: FFTs along iso-latitude
// rings), templated on the arithmetic type: FP64 for the FP64 SHT path, FP32
// for the mixed-precision path (whose error budget is set by the FP16 hi + lo
// Legendre contraction, far above FP32 FFT round-off).
//
// A block transforms one ring (synthesis: one output field of one ring) at a
// time with the whole ring in shared memory.  A real ring of n = 4i (polar) or
// 4 Nside (equatorial) samples is handled as a complex sequence of N = n / 2
// points: power-of-two N by an in-place FFT (radix-2 and radix-4 stages, two
// radix-4 stages at a time on 16 points in registers), other N by Bluestein's
// chirp convolution with power-of-two FFTs of M >= 2N - 1 points whose chirp
// and filter spectrum the plan holds.
//
// What bounds it: FP64 rings the FP64 pipe, so the phases e^{i pi k / n} come
// from a table of the plan (four sincospi per thread and field were a third of
// the FP64 instructions) and products with 1 and 0 are not formed; FP32 rings
// the shared-memory passes and barriers, which the 16-point passes halve.  One
// block per (ring, field) instead of one per ring with the six fields in turn:
// the blocks of the longest rings took a quarter of the whole launch each.
// Six fields, FP64: 4.39 -> 3.02 ms at nside 512 (FP64 pipe 55 -> 80 % busy),
// 229 -> 78 us at nside 64, where the serial alias sums of the rings next to
// the poles had set the time; one map, analysis, lmax 1024: 0.73 -> 0.48 ms.  Batch of 21
// planes at nside 512, FP32: 16.5 -> 12.5 ms for the whole solve, bit for bit.
#pragma once

#include "fft.cuh"

namespace clc {

template <typename T>
__device__ __forceinline__ C2<T> cx(T a, T b) {
  C2<T> r;
  r.x = a;
  r.y = b;
  return r;
}
template <typename T>
__device__ __forceinline__ C2<T> operator+(C2<T> a, C2<T> b) { return cx<T>(a.x + b.x, a.y + b.y); }
template <typename T>
__device__ __forceinline__ C2<T> operator-(C2<T> a, C2<T> b) { return cx<T>(a.x - b.x, a.y - b.y); }
// The fused and the rounded product of each component are written out, so that
// the results do not depend on how the compiler contracts the expression at
// each use (a * b and b * a may differ in the last bit of y).
template <typename T>
__device__ __forceinline__ C2<T> operator*(C2<T> a, C2<T> b) {
  return cx<T>(fma(a.x, b.x, -(a.y * b.y)), fma(a.x, b.y, a.y * b.x));
}
template <typename T>
__device__ __forceinline__ C2<T> operator*(C2<T> a, T s) { return cx<T>(a.x * s, a.y * s); }
template <typename T>
__device__ __forceinline__ C2<T> conj(C2<T> a) { return cx<T>(a.x, -a.y); }

__device__ __forceinline__ void sc_pi(double t, double* s, double* c) { sincospi(t, s, c); }
__device__ __forceinline__ void sc_pi(float t, float* s, float* c) { sincospif(t, s, c); }

// e^{i pi t}
template <typename T>
__device__ __forceinline__ C2<T> expi_pi(T t) {
  T s, c;
  sc_pi(t, &s, &c);
  return cx<T>(c, s);
}
// FP32: t reduced to [-1, 1], then the fast sincos intrinsic on pi t
// (absolute error about 2^-21 on [-pi, pi], far inside the mixed path's
// error budget)
template <>
__device__ __forceinline__ C2<float> expi_pi<float>(float t) {
  const float r = fmaf(-2.f, rintf(0.5f * t), t);
  float s, c;
  __sincosf(3.14159265358979f * r, &s, &c);
  return cx<float>(c, s);
}

// e^{i pi q / n} (n = 2N, q >= 0) from the ring's phase table ph[b] = e^{i pi b
// / n}, b <= N / 2; one quarter turn is N steps.
__device__ __forceinline__ C2<double> phase_of(const C2<double>* __restrict__ ph, int N, int q) {
  const int b = q % N, a = (q / N) & 3;
  C2<double> c;
  if (2 * b <= N) {
    c = ph[b];
  } else {             // e^{i pi b / n} = i e^{-i pi (N - b) / n}
    const C2<double> d = ph[N - b];
    c = cx<double>(d.y, d.x);
  }
  if (a & 1) c = cx<double>(-c.y, c.x);
  if (a & 2) c = cx<double>(-c.x, -c.y);
  return c;
}

// Phases of a ring in the arithmetic type: half(q) = e^{i pi q / n}, full(k) =
// e^{-2 pi i k / n} (k <= N).  FP64: the table (its square for full);
// FP32: the fast sincos.
template <typename T>
struct Phase;
template <>
struct Phase<double> {
  const C2<double>* ph;
  int N;
  __device__ __forceinline__ C2<double> half(int q) const { return phase_of(ph, N, q); }
  __device__ __forceinline__ C2<double> full(int k) const {
    const C2<double> c = phase_of(ph, N, k);
    return cx<double>(fma(c.x, c.x, -c.y * c.y), -2.0 * c.x * c.y);
  }
};
template <>
struct Phase<float> {
  int n;
  float a1, a2;   // 1 / n, -2 / n
  __device__ __forceinline__ C2<float> half(int q) const { return expi_pi<float>(a1 * (float)q); }
  __device__ __forceinline__ C2<float> full(int k) const { return expi_pi<float>(a2 * (float)k); }
};
__device__ __forceinline__ void phase_init(Phase<double>& p, const PlanDevT<double>& P, int nside, int i, int n) {
  const int ip = i < 2 * nside ? i : 4 * nside - i;
  p.N = n / 2;
  p.ph = P.phase + phase_offset(ip < nside ? ip : nside);
}
__device__ __forceinline__ void phase_init(Phase<float>& p, const PlanDevT<float>&, int, int, int n) {
  p.n = n;
  p.a1 = 1.0f / (float)n;
  p.a2 = -2.0f / (float)n;
}

// a / b in the arithmetic type (no FP64 division on the FP32 path)
template <typename T>
__device__ __forceinline__ T ratio(int a, int b) { return (T)a / (T)b; }

// padded position of FFT point i in shared memory
template <typename T>
__device__ __forceinline__ int pidx(int i) { return i + (i >> fft_pad_shift<T>()); }

// FP32 -> FP64 by moving the bits (exact for normal floats; zero and
// subnormal floats give zero): keeps the output conversion off the FP64 pipe
__device__ __forceinline__ double to_out(double v) { return v; }
// FP64 map value in the arithmetic type (FP32: rounded on the integer pipe)
template <typename T>
__device__ __forceinline__ T to_in(double v) { return (T)v; }
template <>
__device__ __forceinline__ float to_in<float>(double v) { return d2f_rn(v); }
__device__ __forceinline__ double to_out(float v) { return f2d_exact(v); }

__device__ __forceinline__ int brev(int j, int logM) { return logM == 0 ? 0 : (int)(__brev((unsigned)j) >> (32 - logM)); }
__device__ __forceinline__ bool is_pow2(int v) { return (v & (v - 1)) == 0; }

// Two radix-2 stages (half h, then 2h) on four points at distance h with
// their twiddles w1, w2 (kOne: both 1).
template <typename T, bool kOne>
__device__ __forceinline__ void quad(C2<T>& a0, C2<T>& a1, C2<T>& a2, C2<T>& a3, C2<T> w1, C2<T> w2) {
  C2<T> v = kOne ? a1 : w1 * a1;
  const C2<T> b0 = a0 + v, b1 = a0 - v;
  v = kOne ? a3 : w1 * a3;
  const C2<T> b2 = a2 + v, b3 = a2 - v;
  v = kOne ? b2 : b2 * w2;
  a0 = b0 + v;
  a2 = b0 - v;
  v = kOne ? b3 : b3 * w2;
  v = cx<T>(v.y, -v.x);  // times W_{4h}^h = -i
  a1 = b1 + v;
  a3 = b1 - v;
}

// Radix-4 pass of the stages lg and lg + 1 (kFirst: lg = 1, unit twiddles).
template <typename T, bool kFirst>
__device__ __forceinline__ void pass4(C2<T>* s, int M, int lg, const PlanDevT<T>& P) {
  const int h = 1 << (lg - 1);
  const int sh1 = P.logmmax - lg, sh2 = P.logmmax - lg - 1;
  for (int t = threadIdx.x; t < M / 4; t += blockDim.x) {
    const int p = t & (h - 1);
    const int i0 = ((t >> (lg - 1)) << (lg + 1)) + p;
    const int j0 = pidx<T>(i0), j1 = pidx<T>(i0 + h), j2 = pidx<T>(i0 + 2 * h), j3 = pidx<T>(i0 + 3 * h);
    C2<T> a0 = s[j0], a1 = s[j1], a2 = s[j2], a3 = s[j3];
    C2<T> w1, w2;
    if (!kFirst) {
      w1 = P.tw[p << sh1];
      w2 = P.tw[p << sh2];
    }
    quad<T, kFirst>(a0, a1, a2, a3, w1, w2);
    s[j0] = a0;
    s[j1] = a1;
    s[j2] = a2;
    s[j3] = a3;
  }
  __syncthreads();
}

// The radix-4 passes of the stages lg .. lg + 3 on 16 points in registers.
template <typename T, bool kFirst>
__device__ __forceinline__ void pass16(C2<T>* s, int M, int lg, const PlanDevT<T>& P) {
  const int h = 1 << (lg - 1);
  const int sh = P.logmmax - lg;
  for (int t = threadIdx.x; t < M / 16; t += blockDim.x) {
    const int p = t & (h - 1);
    const int i0 = ((t >> (lg - 1)) << (lg + 3)) + p;
    C2<T> a[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) a[q] = s[pidx<T>(i0 + q * h)];
    {
      C2<T> w1, w2;
      if (!kFirst) {
        w1 = P.tw[p << sh];
        w2 = P.tw[p << (sh - 1)];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) quad<T, kFirst>(a[4 * q], a[4 * q + 1], a[4 * q + 2], a[4 * q + 3], w1, w2);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int pq = p + q * h;
      quad<T, false>(a[q], a[q + 4], a[q + 8], a[q + 12], P.tw[pq << (sh - 2)], P.tw[pq << (sh - 3)]);
    }
#pragma unroll
    for (int q = 0; q < 16; ++q) s[pidx<T>(i0 + q * h)] = a[q];
  }
  __syncthreads();
}

// In-place forward FFT (sign -1) of s[0..2^logM) given in bit-reversed order;
// twiddle W_L^j = tw[j * mmax / L].  padded: the input's second half is zero
// and its places (the odd ones, in bit-reversed order) need not be set.
template <typename T>
__device__ void fft_pow2(C2<T>* s, int logM, const PlanDevT<T>& P, bool padded = false) {
  const int M = 1 << logM;
  int lg = 1;
  if (logM & 1) {
    for (int t = threadIdx.x; t < M / 2; t += blockDim.x) {
      const C2<T> u = s[pidx<T>(2 * t)];
      if (padded) {
        s[pidx<T>(2 * t + 1)] = u;
      } else {
        const C2<T> v = s[pidx<T>(2 * t + 1)];
        s[pidx<T>(2 * t)] = u + v;
        s[pidx<T>(2 * t + 1)] = u - v;
      }
    }
    __syncthreads();
    lg = 2;
  } else if (padded && logM > 0) {
    // the first radix-4 pass with a1 = a3 = 0
    for (int t = threadIdx.x; t < M / 4; t += blockDim.x) {
      const C2<T> a = s[pidx<T>(4 * t)], c = s[pidx<T>(4 * t + 2)];
      const C2<T> v = cx<T>(c.y, -c.x);
      s[pidx<T>(4 * t)] = a + c;
      s[pidx<T>(4 * t + 2)] = a - c;
      s[pidx<T>(4 * t + 1)] = a + v;
      s[pidx<T>(4 * t + 3)] = a - v;
    }
    __syncthreads();
    lg = 3;
  }
  // 16 points per thread where that still fills warps, else 4 (at 64 - 256
  // points half-empty warps made the FP64 solve at nside 64 195 us, not 159)
  const bool wide = logM >= 9;
  if (lg == 1 && lg < logM && !(wide && !(((logM - lg + 1) >> 1) & 1))) {
    pass4<T, true>(s, M, lg, P);
    lg = 3;
  }
  if (wide) {
    if (((logM - lg + 1) >> 1) & 1) {   // an odd number of radix-4 passes is left
      pass4<T, false>(s, M, lg, P);
      lg += 2;
    }
    if (lg == 1) {
      pass16<T, true>(s, M, lg, P);
      lg += 4;
    }
    for (; lg < logM; lg += 4) pass16<T, false>(s, M, lg, P);
  } else {
    for (; lg < logM; lg += 2) pass4<T, false>(s, M, lg, P);
  }
}

// DFT of N points: put every value (dft_put), dft_run, read (dft_get).
template <typename T>
struct Dft {
  C2<T>* s;
  int N, M, logM;
  bool blue;
  const C2<T>* w;   // Bluestein chirp
  const C2<T>* B;   // and filter spectrum
  __device__ __forceinline__ void init(C2<T>* s_, int N_, int ring_class, const PlanDevT<T>& P) {
    s = s_;
    N = N_;
    blue = !is_pow2(N);
    if (!blue) {
      M = N;
      logM = 31 - __clz(N);
    } else {
      const int4 c = P.cls[ring_class];
      M = c.x;
      logM = c.y;
      w = P.chirp + c.z;
      B = P.filter + c.w;
      for (int j = N + threadIdx.x; j < M / 2; j += blockDim.x) s[pidx<T>(brev(j, logM))] = cx<T>(0, 0);
    }
  }
  __device__ __forceinline__ void put(int j, C2<T> v) const {
    s[pidx<T>(brev(j, logM))] = blue ? conj(w[j]) * v : v;
  }
  __device__ __forceinline__ void run(const PlanDevT<T>& P) const {
    __syncthreads();
    fft_pow2<T>(s, logM, P, blue);
    if (!blue) return;
    // filter, conjugate and bit-reverse for the second transform
    for (int k = threadIdx.x; k < M; k += blockDim.x) {
      const int kr = brev(k, logM);
      if (k > kr) continue;
      const C2<T> x = conj(B[k] * s[pidx<T>(k)]);
      if (k < kr) s[pidx<T>(k)] = conj(B[kr] * s[pidx<T>(kr)]);
      s[pidx<T>(kr)] = x;
    }
    __syncthreads();
    fft_pow2<T>(s, logM, P);
  }
  // Z_k, natural order, k < N
  __device__ __forceinline__ C2<T> get(int k) const {
    if (!blue) return s[pidx<T>(k)];
    return conj(w[k]) * (conj(s[pidx<T>(k)]) * ((T)1 / (T)M));
  }
};

__device__ __forceinline__ int ring_class_of(int nside, int i) {
  const int ip = i < 2 * nside ? i : 4 * nside - i;
  return ip < nside ? ip : 0;
}

// F[m * ldf + (i - 1)] = weight * sum_j map_j e^{-i m phi_j} over ring i, m <= lmax.
template <typename T>
__device__ void ring_analysis_ring(const double* __restrict__ map, int nside, int lmax, double weight,
                                   C2<T>* __restrict__ F, int ldf, const PlanDevT<T>& P, int i, C2<T>* s) {
  const Ring r = P.rings[i - 1].r;
  const int n = r.npix, N = n / 2;
  const double* x = map + r.first;
  Dft<T> D;
  D.init(s, N, ring_class_of(nside, i), P);
  for (int j = threadIdx.x; j < N; j += blockDim.x) D.put(j, cx<T>(to_in<T>(x[2 * j]), to_in<T>(x[2 * j + 1])));
  D.run(P);
  if (D.blue) {   // every Z_k is read at least twice
    for (int k = threadIdx.x; k < N; k += blockDim.x) s[pidx<T>(k)] = D.get(k);
    __syncthreads();
  }
  const bool shifted = r.phi0 != 0.0;
  const T w = (T)weight, half = (T)0.5;
  Phase<T> ph;
  phase_init(ph, P, nside, i, n);
  for (int m = threadIdx.x; m <= lmax; m += blockDim.x) {
    const int k = m % n;
    const bool cj = k > N;
    const int kk = cj ? n - k : k;
    const C2<T> Zk = s[pidx<T>(kk == N ? 0 : kk)];
    const C2<T> Zn = conj(s[pidx<T>(kk == 0 ? 0 : N - kk)]);
    const C2<T> A = (Zk + Zn) * half;
    const C2<T> Bv = (Zk - Zn) * half;
    C2<T> tw, sh;   // e^{-2 pi i kk / n}, e^{-i m phi0}
    if constexpr (sizeof(T) == 4) {
      tw = conj(expi_pi<T>(ratio<T>(2 * kk, n)));
      if (shifted) sh = conj(expi_pi<T>(ratio<T>(m % (2 * n), n)));
    } else {
      tw = ph.full(kk);
      if (shifted) sh = conj(ph.half(m % (2 * n)));
    }
    const C2<T> tB = tw * Bv;
    C2<T> X = cx<T>(A.x + tB.y, A.y - tB.x);   // A - i tB
    if (cj) X = conj(X);
    if (shifted) X = cx<T>(fma(-X.y, sh.y, X.x * sh.x), fma(X.y, sh.x, X.x * sh.y));
    F[(size_t)m * ldf + (i - 1)] = X * w;
  }
  __syncthreads();
}

// Legendre sums G_q of one plane: element (m, ring) at m * sm + ring * sr,
// or, with quad set, in groups of four orders per ring:
// ((m / 4) * sm + ring * 4 + m % 4).  P01 (optional, FP32 path): FP64 sums
// of orders m = 0, 1 at P01[q * p01q + m * p01m + ring], used instead of G on
// the ncap rings next to each pole (nring rings in all).
template <typename T>
struct SynthArgsT {
  const C2<T>* G0;
  const C2<T>* G1;
  const C2<T>* G2;
  long long sm, sr;
  int quad;
  const C2<double>* P01;
  long long p01q, p01m;
  int ncap, nring;
  double* out[6];
};

// Fourier coefficient of output field f at order m on one ring from the
// Legendre sums g0 = psi, g1 = sin(t) d_t psi, g2 = kappa_bl (is = 1 / sin t,
// c = cos t).
template <typename S>
__device__ __forceinline__ C2<S> spec_combine(int mode, int f, int m, C2<S> g0, C2<S> g1, C2<S> g2, S is, S is2, S c) {
  if (mode == 0 || f == 0) return g0;
  const S dm = (S)m;
  switch (f) {
    case 1: return cx<S>(-g1.x * is, -g1.y * is);                               // alpha_t
    case 2: return cx<S>(dm * g0.y * is, -dm * g0.x * is);                       // alpha_p = -i m g0 / s
    case 3:                                                                      // u_tt = kappa_bl - u_pp
      return cx<S>(g2.x - (-dm * dm * g0.x + c * g1.x) * is2, g2.y - (-dm * dm * g0.y + c * g1.y) * is2);
    case 4: return cx<S>((-dm * dm * g0.x + c * g1.x) * is2, (-dm * dm * g0.y + c * g1.y) * is2);
    default: {                                                                   // u_tp = i m (g1 - c g0) / s^2
      const C2<S> d = cx<S>(g1.x - c * g0.x, g1.y - c * g0.y);
      return cx<S>(-dm * d.y * is2, dm * d.x * is2);
    }
  }
}

// Ring geometry factors in the arithmetic type and, for the FP64 orders of
// the FP32 path, in FP64.
template <typename T>
struct RingFac {
  T is, is2, c;
  double isd, cd;
};

template <typename T>
__device__ __forceinline__ C2<T> spec_of(const SynthArgsT<T>& a, int mode, int f, int m, int ring0, const RingFac<T>& g) {
  if (a.P01 && m <= 1 && (ring0 < a.ncap || ring0 >= a.nring - a.ncap)) {
    // the polar Hessian terms of m = 0, 1 cancel to O(sin^2 t): combine in FP64
    const C2<double>* P = a.P01 + (size_t)m * a.p01m + ring0;
    const C2<double> z = cx<double>(0.0, 0.0);
    const C2<double> h = spec_combine<double>(mode, f, m, P[0], mode ? P[a.p01q] : z, mode ? P[2 * a.p01q] : z, g.isd,
                                              g.isd * g.isd, g.cd);
    return cx<T>((T)h.x, (T)h.y);
  }
  const size_t idx = a.quad ? (size_t)(m >> 2) * a.sm + (size_t)ring0 * 4 + (m & 3)
                            : (size_t)m * a.sm + (size_t)ring0 * a.sr;
  const C2<T> g0 = a.G0[idx];
  if (mode == 0 || f == 0) return g0;
  const C2<T> g1 = a.G1[idx];
  const C2<T> g2 = f == 3 ? a.G2[idx] : cx<T>(0, 0);
  return spec_combine<T>(mode, f, m, g0, g1, g2, g.is, g.is2, g.c);
}

// Longest ring (pixels) whose coefficients are staged; its FFT takes at most
// 2 kStageRing points of the buffer.
constexpr int kStageRing = 64;

// Real values of output field f of ring i.  s: FFT buffer of buf_len points
// (at least fft_buf_len(plan mmax)).
template <typename T>
__device__ void ring_synthesis_ring(const SynthArgsT<T>& a, int nside, int lmax, int mode, const PlanDevT<T>& P,
                                    int i, int f, C2<T>* s, int buf_len) {
  double* out = a.out[f];
  if (!out) return;
  const RingS rs = P.rings[i - 1];
  const Ring& r = rs.r;
  const int n = r.npix, N = n / 2;
  const int ring0 = i - 1;
  const bool shifted = r.phi0 != 0.0;
  RingFac<T> gf;
  gf.isd = rs.is;
  gf.cd = r.z;
  if constexpr (sizeof(T) == 4) {   // rounded on the integer pipe
    gf.is = d2f_rn(rs.is);
    gf.c = d2f_rn(r.z);
  } else {
    gf.is = rs.is;
    gf.c = r.z;
  }
  gf.is2 = gf.is * gf.is;
  Phase<T> ph;
  phase_init(ph, P, nside, i, n);
  // X_k = c_k [sum_{q>=0} (-1)^q g_{k+qn} + sum_{q>=1} (-1)^q conj(g_{qn-k})]
  // with the half-pixel shift c_k = e^{i pi k / n} (signs and c_k only on
  // shifted rings): the aliases m = k + qn differ from k by q n in phase.
  // The rings next to the poles have hundreds of aliases per k (ring 1: lmax /
  // 4): their coefficients are formed by all threads first (stage), so that the
  // sums do not wait for one load after the other.
  C2<T>* stage = s + 2 * kStageRing;
  const bool staged = n <= kStageRing && lmax >= 4 * n && 2 * kStageRing + lmax + 1 <= buf_len;
  if (staged) {
    for (int m = threadIdx.x; m <= lmax; m += blockDim.x) stage[m] = spec_of<T>(a, mode, f, m, ring0, gf);
    __syncthreads();
  }
  auto coef = [&](int m) -> C2<T> { return staged ? stage[m] : spec_of<T>(a, mode, f, m, ring0, gf); };
  auto spectrum = [&](int k) -> C2<T> {
    C2<T> X = cx<T>(0, 0);
    int q = 0;
    for (int m = k; m <= lmax; m += n, ++q) {
      C2<T> g = coef(m);
      if (m == 0) g.y = (T)0;
      X = (shifted && (q & 1)) ? X - g : X + g;
    }
    q = 1;
    for (int m = (k == 0 ? n : n - k); m <= lmax; m += n, ++q) {
      const C2<T> g = conj(coef(m));
      X = (shifted && (q & 1)) ? X - g : X + g;
    }
    return shifted ? X * ph.half(k) : X;
  };
  // P_k = conj(X_k) + X_{N-k} + i e^{-2 pi i k / n} (conj(X_k) - X_{N-k});
  // the forward DFT of P packs x_{2j} + i x_{2j+1}.  A thread forms P_k and
  // P_{N-k} from the same two spectrum values.
  Dft<T> D;
  D.init(s, N, ring_class_of(nside, i), P);
  auto pack = [&](int k, C2<T> Xk, C2<T> Xn) {
    const C2<T> a1 = conj(Xk);
    const C2<T> t = (a1 - Xn) * ph.full(k);
    D.put(k, cx<T>(a1.x + Xn.x - t.y, a1.y + Xn.y + t.x));
  };
  for (int k = threadIdx.x; 2 * k <= N; k += blockDim.x) {
    const C2<T> Xk = spectrum(k), Xn = spectrum(N - k);
    pack(k, Xk, Xn);
    if (k > 0 && 2 * k < N) pack(N - k, Xn, Xk);
  }
  D.run(P);
  double* x = out + r.first;
  if ((reinterpret_cast<uintptr_t>(x) & 15) == 0) {   // rings start at even pixels: aligned unless the map is not
    for (int j = threadIdx.x; j < N; j += blockDim.x) {
      const C2<T> v = D.get(j);
      *reinterpret_cast<double2*>(x + 2 * j) = make_double2(to_out(v.x), to_out(v.y));
    }
  } else {
    for (int j = threadIdx.x; j < N; j += blockDim.x) {
      const C2<T> v = D.get(j);
      x[2 * j] = to_out(v.x);
      x[2 * j + 1] = to_out(v.y);
    }
  }
  __syncthreads();
}

}  // namespace clc
