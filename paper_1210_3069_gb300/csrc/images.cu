// Grid search for lensed galaxy images (paper Sec. 2.3 and the grid-search
// implementation, Sec. 3.3).  Rays start at the RING pixel centres; the
// triangles joining centres of consecutive rings (every centre closes one
// triangle with its predecessor on its ring and the last centre of the
// neighbouring ring before it in longitude; two cap triangles at each pole)
// map, vertex for vertex, onto the rays' source-sphere positions.  A galaxy
// has one image per source-sphere triangle that contains it (gnomonic
// projection at the galaxy: the three triple products det(g, v_i, v_j) share
// a sign), at the image-sphere point given by the barycentric coordinates of
// that projection; the inverse magnification matrix there comes from the
// ring-bilinear interpolation of the rays' matrices, each parallel
// transported to the image (Appendix B).
//
// Search: a triangle that contains g has its owner (the centre it is listed
// under) within T of g, T the largest distance on the source sphere from an
// owner to the other vertices of its triangles, and that owner's pixel centre
// within D + T, D the largest distance between a ray's source position and
// its pixel centre.  One pass reduces D and T; then one thread per galaxy
// visits the pixel centres within D + T, keeps the owners whose rays lie
// within T and tests their triangles.  The candidate set contains every
// triangle that can contain g, so the result is that of testing all
// triangles.
//
// D, T and the choice of candidates run in FP32 with margins above its rounding
// (2e-6 rad on distances, 6e-6 T on the side of a triangle's edge): they only
// have to keep every triangle that can contain g, and what they keep is decided
// by the exact FP64 products.  An angle from a squared chord (error below 1e-6)
// is off by up to 5e-7 / sin of it, so the margin holds up to D + T = 2.5 rad; beyond,
// where nine tenths of the sphere are in reach anyway, all of it is searched.  All in FP64 (2 instructions per clock and SM)
// the search took 6.91 ms and the bounds 0.84 ms for 5e5 galaxies on the rays
// of nside 512, the pipe 83 % busy.
// Now: FP32 directions 0.02 ms, bounds 0.04 ms, search 0.60 ms (a warp per
// galaxy; bound by scattered reads from L2), exact test, image and matrix 0.79
// ms (FP64 pipe, about 900 instructions per galaxy).
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "sphere.cuh"

namespace clc {

constexpr int kMaxImages = 8;
constexpr double kSearchMargin = 1e-9;   // radians added to D and T in the refusal of too wide searches
constexpr float kMargin32 = 2e-6f;       // radians added to each distance of the FP32 search
constexpr float kReach32 = 2.5f;         // largest D + T searched by distance

// Integer geometry of ring r: first pixel, pixel count n, and h (longitudes
// (2 k + h) pi / n, h = 1 on rings offset by half a pixel).
struct RingI {
  int64_t first;
  int n;
  int h;
};

__device__ __forceinline__ RingI ring_int(int nside, int r) {
  const int64_t ns = nside;
  RingI o;
  if (r < nside) {
    o.n = 4 * r;
    o.first = 2 * (int64_t)r * (r - 1);
    o.h = 1;
  } else if (r > 3 * nside) {
    const int64_t ip = 4 * ns - r;
    o.n = (int)(4 * ip);
    o.first = 12 * ns * ns - 2 * ip * (ip + 1);
    o.h = 1;
  } else {
    o.n = 4 * nside;
    o.first = 2 * ns * (ns - 1) + (int64_t)(r - nside) * 4 * ns;
    o.h = ((r - nside) & 1) == 0 ? 1 : 0;
  }
  return o;
}

// Index on ring b of its last point before point k of ring a in longitude,
// cyclically: the largest j with (2 j + h_b) / n_b < (2 k + h_a) / n_a (two
// rings never share a longitude).
__device__ __forceinline__ int last_before(int k, const RingI& a, const RingI& b) {
  // (2 k + h_a) n_b <= 2^31 at nside 8192: 32-bit unsigned arithmetic
  const unsigned have = (unsigned)(2 * k + a.h) * (unsigned)b.n, need = (unsigned)(b.h * a.n) + 1u;
  return have < need ? b.n - 1 : (int)((have - need) / (2u * (unsigned)a.n));
}

// Vertices, counter-clockwise seen from outside, of triangle 2 p + s (s = 0:
// the strip below p's ring, s = 1: the strip above) for p at position k of
// ring r; false for unused ids.
__device__ __forceinline__ bool tri_vertices_rk(int nside, int64_t p, int r, int k, int s, int64_t v[3]) {
  if (s == 1 && r == 1) {
    if (p == 1) { v[0] = 0; v[1] = 1; v[2] = 2; return true; }
    if (p == 3) { v[0] = 2; v[1] = 3; v[2] = 0; return true; }
    return false;
  }
  if (s == 0 && r == 4 * nside - 1) {
    const int64_t f = 12 * (int64_t)nside * nside - 4;
    if (p == f + 1) { v[0] = f + 2; v[1] = f + 1; v[2] = f; return true; }
    if (p == f + 3) { v[0] = f; v[1] = f + 3; v[2] = f + 2; return true; }
    return false;
  }
  const RingI a = ring_int(nside, r), b = ring_int(nside, s == 0 ? r + 1 : r - 1);
  const int64_t prev = a.first + (k == 0 ? a.n - 1 : k - 1);
  const int64_t q = b.first + last_before(k, a, b);
  v[0] = prev;
  v[1] = s == 0 ? q : p;
  v[2] = s == 0 ? p : q;
  return true;
}

__device__ __forceinline__ bool tri_vertices(int nside, int64_t p, int s, int64_t v[3]) {
  int64_t k;
  const int r = pix2ring(nside, p, &k);
  return tri_vertices_rk(nside, p, r, (int)k, s, v);
}

__device__ __forceinline__ void load3(const double* __restrict__ x, int64_t n, int64_t p, double o[3]) {
  o[0] = x[p];
  o[1] = x[n + p];
  o[2] = x[2 * n + p];
}

// det(g, a, b) = g . (a x b), every product and sum rounded separately in
// this order (the decision must not depend on FMA contraction)
__device__ __forceinline__ double edge_det(const double g[3], const double a[3], const double b[3]) {
  const double c0 = __dsub_rn(__dmul_rn(a[1], b[2]), __dmul_rn(a[2], b[1]));
  const double c1 = __dsub_rn(__dmul_rn(a[2], b[0]), __dmul_rn(a[0], b[2]));
  const double c2 = __dsub_rn(__dmul_rn(a[0], b[1]), __dmul_rn(a[1], b[0]));
  return __dadd_rn(__dadd_rn(__dmul_rn(g[0], c0), __dmul_rn(g[1], c1)), __dmul_rn(g[2], c2));
}

// det(g, x_u, x_v), evaluated on the edge's endpoints in increasing pixel
// order so that the two triangles sharing the edge see opposite values
__device__ __forceinline__ double oriented(const double g[3], int64_t u, const double xu[3], int64_t v,
                                           const double xv[3]) {
  return u < v ? edge_det(g, xu, xv) : -edge_det(g, xv, xu);
}

// Containment of g in the source-sphere triangle v; d[i] = det(g, v_j, v_k)
// for the edge opposite vertex i, gx[i] = g . x_{v_i}.
__device__ __forceinline__ bool contains(const double* __restrict__ x, int64_t n, const double g[3],
                                         const int64_t v[3], double d[3], double gx[3]) {
  double a[3], b[3], c[3];
  load3(x, n, v[0], a);
  load3(x, n, v[1], b);
  load3(x, n, v[2], c);
  d[2] = oriented(g, v[0], a, v[1], b);
  d[0] = oriented(g, v[1], b, v[2], c);
  d[1] = oriented(g, v[2], c, v[0], a);
  gx[0] = dot3(a, g);
  gx[1] = dot3(b, g);
  gx[2] = dot3(c, g);
  const bool pos = d[0] >= 0.0 && d[1] >= 0.0 && d[2] >= 0.0;
  const bool neg = d[0] <= 0.0 && d[1] <= 0.0 && d[2] <= 0.0;
  const bool nz = d[0] != 0.0 || d[1] != 0.0 || d[2] != 0.0;
  return (pos || neg) && nz && gx[0] > 0.0 && gx[1] > 0.0 && gx[2] > 0.0;
}

__device__ __forceinline__ void normalize3(const double a[3], double o[3]) {
  const double is = rsqrt(dot3(a, a));
  o[0] = a[0] * is;
  o[1] = a[1] * is;
  o[2] = a[2] * is;
}

// FP32 unit vector of x (any length, to a few 1e-7; NaN for a non-finite or
// zero x): the exponent of the largest component is taken out on the integer
// pipe, so that the conversion cannot overflow and stays off the FP64 pipe.
__device__ __forceinline__ float narrowed(double v, int emax) {
  const int hi = __double2hiint(v);
  const int e = ((hi >> 20) & 0x7ff) - emax + 127;
  if (e <= 0) return 0.f;
  return __uint_as_float(((unsigned)hi & 0x80000000u) | ((unsigned)e << 23) | (((unsigned)hi & 0xfffffu) << 3) |
                         ((unsigned)__double2loint(v) >> 29));
}

__device__ __forceinline__ void unit32(const double x[3], float o[3]) {
  const int emax = max(max((__double2hiint(x[0]) >> 20) & 0x7ff, (__double2hiint(x[1]) >> 20) & 0x7ff),
                       (__double2hiint(x[2]) >> 20) & 0x7ff);
  if (emax == 0x7ff || emax == 0) {
    o[0] = o[1] = o[2] = __uint_as_float(0x7fc00000u);
    return;
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) o[c] = narrowed(x[c], emax);
  const float is = rsqrtf(o[0] * o[0] + o[1] * o[1] + o[2] * o[2]);
#pragma unroll
  for (int c = 0; c < 3; ++c) o[c] *= is;
}

// FP32 directions of the rays, one 16-byte word each: the search reads scattered
// rays, and three FP64 components in three arrays cost three 32-byte sectors
// and their conversion each time.
__global__ void k_image_units(const double* __restrict__ x, int64_t npx, float4* __restrict__ u) {
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < npx; p += (int64_t)gridDim.x * blockDim.x) {
    double v[3];
    float o[3];
    load3(x, npx, p, v);
    unit32(v, o);
    u[p] = make_float4(o[0], o[1], o[2], 0.f);
  }
}

__device__ __forceinline__ void load_unit32(const float4* __restrict__ u, int64_t p, float o[3]) {
  const float4 v = u[p];
  o[0] = v.x;
  o[1] = v.y;
  o[2] = v.z;
}

__device__ __forceinline__ float chord2f(const float a[3], const float b[3]) {
  const float dx = a[0] - b[0], dy = a[1] - b[1], dz = a[2] - b[2];
  return dx * dx + dy * dy + dz * dz;
}
__device__ __forceinline__ float chord2f_angle(float c2) { return 2.f * asinf(fminf(1.f, 0.5f * sqrtf(c2))); }
__device__ __forceinline__ float angle_chord2f(float a) {
  const float s = sinf(0.5f * a);
  return 4.f * s * s;
}

// cos and sin of the colatitude of ring r
__device__ __forceinline__ void ring_zs32(int nside, int r, float* z, float* s) {
  const bool north = r < nside, south = r > 3 * nside;
  if (north || south) {
    const float f = (float)(north ? r : 4 * nside - r) / (float)nside;
    const float a = f * f * (1.f / 3.f);
    *z = north ? 1.f - a : a - 1.f;
    *s = sqrtf(a * (2.f - a));
  } else {
    *z = (float)(4 * nside - 2 * r) / (float)(3 * nside);
    *s = sqrtf((1.f - *z) * (1.f + *z));
  }
}

// unit vector of the centre of pixel p
__device__ __forceinline__ void centre_vec(int nside, const RingS* __restrict__ rings, int64_t p, double c[3]) {
  int64_t k;
  const Ring g = rings[pix2ring(nside, p, &k) - 1].r;
  double sn, cs;
  sincospi((double)(2 * k + (g.phi0 != 0.0 ? 1 : 0)) / (double)g.npix, &sn, &cs);
  c[0] = g.s * cs;
  c[1] = g.s * sn;
  c[2] = g.z;
}

// bounds[0], bounds[1]: the squared chords of D and T (as the bits of
// non-negative floats, whose integer order is their value order)
__global__ void k_image_bounds(const float4* __restrict__ u, int nside, unsigned* __restrict__ bounds) {
  float dmax = 0.f, tmax = 0.f;
  for (int r = blockIdx.x + 1; r < 4 * nside; r += gridDim.x) {
    const RingI g = ring_int(nside, r);
    float z, s;
    ring_zs32(nside, r, &z, &s);
    const float inv = 1.f / (float)g.n;
    for (int k = blockIdx.y * blockDim.x + threadIdx.x; k < g.n; k += gridDim.y * blockDim.x) {
      const int64_t p = g.first + k;
      float xn[3], yn[3], sn, cs;
      load_unit32(u, p, xn);
      sincospif((float)(2 * k + g.h) * inv, &sn, &cs);
      const float c[3] = {s * cs, s * sn, z};
      dmax = fmaxf(dmax, chord2f(xn, c));
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        int64_t v[3];
        if (!tri_vertices_rk(nside, p, r, k, t, v)) continue;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          if (v[i] == p) continue;
          load_unit32(u, v[i], yn);
          tmax = fmaxf(tmax, chord2f(xn, yn));
        }
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(bounds, __float_as_uint(dmax));
    atomicMax(bounds + 1, __float_as_uint(tmax));
  }
}

// Whether g may lie in the triangle of the unit vectors a, b, c (all FP32,
// relative to g: det(g, a, b) = det(g, a - g, b - g)): false only if two edges
// clearly have g on opposite sides.
__device__ __forceinline__ float side32(const float g[3], const float a[3], const float b[3]) {
  return g[0] * (a[1] * b[2] - a[2] * b[1]) + g[1] * (a[2] * b[0] - a[0] * b[2]) + g[2] * (a[0] * b[1] - a[1] * b[0]);
}
__device__ __forceinline__ bool may_contain(const float g[3], const float a[3], const float b[3], const float c[3],
                                            float tol) {
  const float d0 = side32(g, a, b), d1 = side32(g, b, c), d2 = side32(g, c, a);
  const bool above = d0 > tol || d1 > tol || d2 > tol, below = d0 < -tol || d1 < -tol || d2 < -tol;
  return !(above && below);
}

struct ImageOut {
  int32_t* nimg;
  int64_t* tri;
  double* img;   // [3][max_images][ngal]
  double* A;     // [4][max_images][ngal] or null
};

// What a galaxy's search needs: its FP32 direction, the chord^2 limits of
// owners' rays (c2t) and pixel centres (c2r), the edge tolerance and the rings
// in reach.
struct Search32 {
  float g[3], sp, pp, c2t, c2r, tol;
  int i0, i1;
};

__device__ __forceinline__ bool search_init(int nside, const double g[3], const unsigned* __restrict__ bounds,
                                            Search32& S) {
  unit32(g, S.g);
  if (!(S.g[0] == S.g[0])) return false;
  const float dmax = chord2f_angle(__uint_as_float(bounds[0])), tmax = chord2f_angle(__uint_as_float(bounds[1]));
  const float tm = tmax + kMargin32, R = dmax + tm + kMargin32;
  S.c2t = tm < 1.57f ? angle_chord2f(tm + kMargin32) : 5.f;   // above 4: every point of the sphere
  S.c2r = R < kReach32 ? angle_chord2f(R) : 5.f;
  S.tol = 6e-6f * tm;
  S.sp = sqrtf(S.g[0] * S.g[0] + S.g[1] * S.g[1]);
  const float th = atan2f(S.sp, S.g[2]);
  S.pp = atan2f(S.g[1], S.g[0]);
  if (S.pp < 0.f) S.pp += 6.28318531f;
  // (FP32 rounding of the ring and pixel coordinates is below 0.01 up to nside 8192)
  S.i0 = 1;
  S.i1 = 4 * nside - 1;
  if (R < kReach32) {
    S.i0 = max(S.i0, (int)ceilf(ring_coord32(nside, fmaxf(0.f, th - R)) - 0.1f));
    S.i1 = min(S.i1, (int)floorf(ring_coord32(nside, fminf(3.14159265f, th + R)) + 0.1f));
  }
  return true;
}

// pixel centres of ring i in reach: first position jl (unwrapped) and number
__device__ __forceinline__ int ring_reach(int nside, const Search32& S, int i, const RingI& r, int* jl) {
  float rz, rs;
  ring_zs32(nside, i, &rz, &rs);
  // |c - g|^2 = (rs - sp)^2 + (rz - gz)^2 + 4 rs sp sin^2(dphi / 2) for the ring's centres c
  const float rem = S.c2r - (rs - S.sp) * (rs - S.sp) - (rz - S.g[2]) * (rz - S.g[2]);
  if (rem < 0.f) return 0;
  const float sh2 = rem / (4.f * rs * S.sp);
  *jl = 0;
  if (sh2 < 1.f) {
    const float idphi = (float)r.n * 0.159154943f;
    const float span = 2.f * asinf(sqrtf(sh2)) * idphi, base = S.pp * idphi - 0.5f * (float)r.h;
    const int a = (int)ceilf(base - span - 0.1f), b = (int)floorf(base + span + 0.1f);
    if (b - a + 1 < r.n) {
      *jl = a;
      return max(b - a + 1, 0);
    }
  }
  return r.n;
}

// bit s set: the triangle s of the owner at position j of ring i may contain the galaxy
__device__ __forceinline__ int owner_triangles(const float4* __restrict__ u, int nside, const Search32& S, int i, int j,
                                               int64_t p) {
  float xp[3];
  load_unit32(u, p, xp);
  if (!(chord2f(xp, S.g) <= S.c2t)) return 0;
#pragma unroll
  for (int c = 0; c < 3; ++c) xp[c] -= S.g[c];
  int hit = 0;
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    int64_t v[3];
    if (!tri_vertices_rk(nside, p, i, j, s, v)) continue;
    float y[3][3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      if (v[q] == p) {
#pragma unroll
        for (int c = 0; c < 3; ++c) y[q][c] = xp[c];
      } else {
        load_unit32(u, v[q], y[q]);
#pragma unroll
        for (int c = 0; c < 3; ++c) y[q][c] -= S.g[c];
      }
    }
    if (may_contain(S.g, y[0], y[1], y[2], S.tol)) hit |= 1 << s;
  }
  return hit;
}

// One warp per galaxy: the pixel centres in reach, 32 at a time over rings and
// positions, so that neighbouring lanes read neighbouring rays (one thread per
// galaxy read 32 unrelated places per step and diverged: 1.7 ms of FP32 search).  The
// ids of the triangles that may contain the galaxy go to cand[galaxy][kCand];
// ncand counts them, beyond kCand too.
constexpr int kCand = 6;

__global__ void __launch_bounds__(256) k_search_images(const float4* __restrict__ u, int nside,
                                                       const double* __restrict__ gal, int64_t ngal, int64_t m0,
                                                       int64_t m1, const unsigned* __restrict__ bounds,
                                                       unsigned* __restrict__ cand, int* __restrict__ ncand) {
  const int64_t ml = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), m = m0 + ml;
  const int lane = threadIdx.x & 31;
  if (m >= m1) return;   // whole warps
  double g[3];
  load3(gal, ngal, m, g);
  Search32 S;
  int count = 0;
  if (search_init(nside, g, bounds, S)) {
    for (int ib = S.i0; ib <= S.i1; ib += 32) {
      // lane's ring and the running number of centres up to it
      const int i = ib + lane;
      int jl = 0, n = 0;
      if (i <= S.i1) {
        const RingI r = ring_int(nside, i);
        n = ring_reach(nside, S, i, r, &jl);
      }
      int sum = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, sum, o);
        if (lane >= o) sum += y;
      }
      const int total = __shfl_sync(0xffffffffu, sum, 31);
      for (int t = 0; t < total; t += 32) {
        const int idx = t + lane;
        // the ring of centre idx: the first lane whose running number exceeds it
        int lo = 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
          if (__shfl_sync(0xffffffffu, sum, lo + o - 1) <= idx) lo += o;
        const int before = __shfl_sync(0xffffffffu, sum - n, min(lo, 31)), j0 = __shfl_sync(0xffffffffu, jl, min(lo, 31));
        int hit = 0;
        int64_t p = 0;
        if (idx < total) {
          const int ir = ib + lo;
          const RingI r = ring_int(nside, ir);
          int j = j0 + idx - before;
          j = j < 0 ? j + r.n : j >= r.n ? j - r.n : j;
          p = r.first + j;
          hit = owner_triangles(u, nside, S, ir, j, p);
        }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          const unsigned who = __ballot_sync(0xffffffffu, (hit >> s) & 1);
          if ((hit >> s) & 1) {
            const int at = count + __popc(who & ((1u << lane) - 1u));
            if (at < kCand) cand[ml * kCand + at] = (unsigned)(2 * p + s);
          }
          count += __popc(who);
        }
      }
    }
  }
  if (lane == 0) ncand[ml] = count;
}

// One thread per galaxy: the exact test of its candidates (of every owner in
// reach again if they did not fit the list), the images and their matrices.
__global__ void __launch_bounds__(128) k_find_images(const double* __restrict__ x, const float4* __restrict__ u,
                                                     const double* __restrict__ Ar, int nside, int64_t npx, const RingS* __restrict__ rings,
                                                     const double* __restrict__ gal, int64_t ngal, int64_t m0,
                                                     int64_t m1, const unsigned* __restrict__ bounds,
                                                     const unsigned* __restrict__ cand, const int* __restrict__ ncand,
                                                     int max_images, ImageOut out) {
  const int64_t ml = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, m = m0 + ml;
  if (m >= m1) return;
  double g[3];
  load3(gal, ngal, m, g);
  const double gg = dot3(g, g);
  int64_t found[kMaxImages] = {};
  int nfound = 0, count = 0;
  auto test = [&](int64_t p, int s, int64_t v[3]) {
    double d[3], gx[3];
    if (!contains(x, npx, g, v, d, gx)) return;
    ++count;
    // keep the max_images smallest triangle ids, ascending
    const int64_t id = 2 * p + s;
    int pos = nfound;
    while (pos > 0 && found[pos - 1] > id) --pos;
    if (pos < max_images) {
      const int last = nfound < max_images ? nfound : max_images - 1;
      for (int q = last; q > pos; --q) found[q] = found[q - 1];
      found[pos] = id;
      if (nfound < max_images) ++nfound;
    }
  };
  const int nc = ncand[ml];
  if (gg > 0.0 && isfinite(gg)) {   // otherwise no direction: no image
    if (nc <= kCand) {
      for (int q = 0; q < nc; ++q) {
        const unsigned id = cand[ml * kCand + q];
        int64_t v[3];
        if (tri_vertices(nside, id >> 1, (int)(id & 1), v)) test(id >> 1, (int)(id & 1), v);
      }
    } else {
      Search32 S;
      search_init(nside, g, bounds, S);
      for (int i = S.i0; i <= S.i1; ++i) {
        const RingI r = ring_int(nside, i);
        int jl;
        const int n = ring_reach(nside, S, i, r, &jl);
        for (int t = 0; t < n; ++t) {
          const int j = jl + t < 0 ? jl + t + r.n : jl + t >= r.n ? jl + t - r.n : jl + t;
          const int64_t p = r.first + j;
          const int hit = owner_triangles(u, nside, S, i, j, p);
          for (int s = 0; s < 2; ++s) {
            int64_t v[3];
            if (((hit >> s) & 1) && tri_vertices_rk(nside, p, i, j, s, v)) test(p, s, v);
          }
        }
      }
    }
  }
  out.nimg[m] = count;
  for (int q = 0; q < max_images; ++q) {
    const size_t o = (size_t)q * ngal + m;
    if (q >= nfound) {
      out.tri[o] = -1;
      for (int c = 0; c < 3; ++c) out.img[((size_t)c * max_images + q) * ngal + m] = 0.0;
      if (out.A)
        for (int c = 0; c < 4; ++c) out.A[((size_t)c * max_images + q) * ngal + m] = 0.0;
      continue;
    }
    const int64_t id = found[q];
    int64_t v[3];
    double d[3], gx[3];
    tri_vertices(nside, id >> 1, (int)(id & 1), v);
    contains(x, npx, g, v, d, gx);
    // barycentric coordinates in the gnomonic plane at g; image on the image sphere
    double lam[3], tot = 0.0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      lam[i] = d[i] * gx[i];
      tot += lam[i];
    }
    double w3[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      double c[3];
      centre_vec(nside, rings, v[i], c);
      const double li = lam[i] / tot;
      w3[0] += li * c[0];
      w3[1] += li * c[1];
      w3[2] += li * c[2];
    }
    double ni[3];
    normalize3(w3, ni);
    out.tri[o] = id;
    for (int c = 0; c < 3; ++c) out.img[((size_t)c * max_images + q) * ngal + m] = ni[c];
    if (!out.A) continue;
    // inverse magnification matrix at the image
    const double rho = sqrt(ni[0] * ni[0] + ni[1] * ni[1]);
    double ph = atan2(ni[1], ni[0]);
    if (ph < 0.0) ph += 2.0 * kPi;
    RingInterp w;
    ring_interp(nside, rings, atan2(rho, ni[2]), ph, w);
    double t1[3], p1[3], acc[4] = {0.0, 0.0, 0.0, 0.0};
    tangent_basis(ni, t1, p1);
    for (int k = 0; k < w.n; ++k) {
      if (w.w[k] == 0.0) continue;
      const int64_t pk = w.p[k];
      double xr[3], xn[3], t0[3], p0[3], Ak[4], At[4];
      load3(x, npx, pk, xr);
      normalize3(xr, xn);
      tangent_basis(xn, t0, p0);
      // the transport's plane rotation (without its axis)
      const double wq = dot3(ni, t0) / (1.0 + dot3(xn, ni));
      const double q0 = dot3(t1, t0) - wq * dot3(t1, xn), q1 = dot3(p1, t0) - wq * dot3(p1, xn);
      const double Q[4] = {q0, -q1, q1, q0};
#pragma unroll
      for (int c = 0; c < 4; ++c) Ak[c] = Ar[(size_t)c * npx + pk];
      qaqt(Q, Ak, At);
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[c] += w.w[k] * At[c];
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) out.A[((size_t)c * max_images + q) * ngal + m] = acc[c];
  }
}

}  // namespace clc

using namespace clc;

extern "C" int clc_find_images(clc_ctx* ctx, int nside, const double* x, const double* A, int64_t ngal,
                               const double* g, int max_images, int32_t* nimg, int64_t* tri, double* img,
                               double* A_img) {
  if (!ctx) return CLC_EINVAL;
  if (!valid_nside(nside) || ngal < 0 || max_images < 1 || max_images > kMaxImages)
    return set_err(ctx, CLC_EINVAL, "clc_find_images: bad nside, ngal or max_images (1..8)");
  if (ngal == 0) return CLC_OK;
  if ((A == nullptr) != (A_img == nullptr))
    return set_err(ctx, CLC_EINVAL, "clc_find_images: A and A_img must both be given or both be NULL");
  if (!x || !g || !nimg || !tri || !img)
    return set_err(ctx, CLC_EINVAL, "clc_find_images: null pointer");
  cudaSetDevice(ctx->device);
  const int64_t npx = 12 * (int64_t)nside * nside;
  auto* bounds = (unsigned*)scratch(ctx, 6, 2 * sizeof(unsigned));
  if (!bounds) return CLC_ENOMEM;
  if (cuda_check(ctx, cudaMemsetAsync(bounds, 0, 2 * sizeof(unsigned), ctx->stream), "memset")) return CLC_ECUDA;
  float4* u = (float4*)scratch(ctx, 11, (size_t)npx * sizeof(float4));
  if (!u) return CLC_ENOMEM;
  CLC_LAUNCH(ctx, "k_image_units", k_image_units, (int)std::min<int64_t>((npx + 255) / 256, (int64_t)num_sms(ctx) * 16),
             256, 0, x, npx, u);
  CLC_LAUNCH(ctx, "k_image_bounds", k_image_bounds, dim3(4 * nside - 1, nside >= 1024 ? nside / 512 : 1), 256, 0, u,
             nside, bounds);
  if (int rc = launch_check(ctx, "k_image_bounds")) return rc;
  // the search radius sets the work per galaxy: refuse inputs whose rays
  // moved so far from their pixels that the search would cover a large part
  // of the sphere for many galaxies
  float hb[2];
  if (cuda_check(ctx, cudaMemcpyAsync(hb, bounds, sizeof(hb), cudaMemcpyDeviceToHost, ctx->stream), "bounds copy") ||
      cuda_check(ctx, cudaStreamSynchronize(ctx->stream), "bounds sync"))
    return CLC_ECUDA;
  const double c2d = hb[0], c2t = hb[1];
  if (!std::isfinite(c2d) || !std::isfinite(c2t))
    return set_err(ctx, CLC_EINVAL, "clc_find_images: non-finite ray positions");
  const double dm = 2.0 * std::asin(std::fmin(1.0, 0.5 * std::sqrt(c2d)));
  const double tm = 2.0 * std::asin(std::fmin(1.0, 0.5 * std::sqrt(c2t)));
  const double R = std::fmin(dm + tm + 2 * kSearchMargin, kPi);
  // pixels within R, plus the margin of a few pixels on each ring in range
  const double npxr = 0.5 * (1.0 - std::cos(R)) * (double)npx + 3.0 * (8.0 * R * nside / kPi + 3.0);
  if (npxr * (double)ngal > 5e10)
    return set_err(ctx, CLC_EINVAL, "clc_find_images: rays too far from their pixels for the search (radius " +
                                        std::to_string(R) + " rad)");
  ImageOut out{nimg, tri, img, A_img};
  const int threads = 128;
  const int64_t blocks = (ngal + threads - 1) / threads;
  if (blocks > 0x7fffffff) return set_err(ctx, CLC_EINVAL, "clc_find_images: too many galaxies");
  int rc;
  const RingS* rings = get_ring_table(ctx, nside, &rc);
  if (rc) return rc;
  // candidate lists (28 bytes per galaxy) for up to 2^24 galaxies at a time
  const int64_t part = std::min<int64_t>(ngal, (int64_t)1 << 24);
  auto* cand = (unsigned*)scratch(ctx, 10, (size_t)part * (kCand + 1) * sizeof(unsigned));
  if (!cand) return CLC_ENOMEM;
  int* ncand = (int*)(cand + part * kCand);
  for (int64_t m0 = 0; m0 < ngal; m0 += part) {
    const int64_t m1 = std::min(m0 + part, ngal);
    CLC_LAUNCH(ctx, "k_search_images", k_search_images, (int)((m1 - m0 + 7) / 8), 256, 0, u, nside, g, ngal, m0, m1,
               bounds, cand, ncand);
    CLC_LAUNCH(ctx, "k_find_images", k_find_images, (int)((m1 - m0 + threads - 1) / threads), threads, 0, x, u, A, nside,
               npx, rings, g, ngal, m0, m1, bounds, cand, ncand, max_images, out);
    if ((rc = launch_check(ctx, "k_find_images"))) return rc;
  }
  return CLC_OK;
}
