// Convergence, E/B-mode shear and rotation power spectra of the final
// inverse magnification matrices (paper Sec. 5, Eq. invmagmat).
//
// The shear gamma_1 + i gamma_2 ((theta-hat, phi-hat) basis) is a spin-2
// field.  With eth^2 Y_lm = (A_lm - B_lm) e^{i m phi} and
// eth-bar^2 Y_lm = (A_lm + B_lm) e^{i m phi},
//   A_lm = -2 cot t dlambda_lm - (l(l+1) - 2 m^2 / sin^2 t) lambda_lm,
//   B_lm = (2 m / sin t)(dlambda_lm - cot t lambda_lm),
// the E and B coefficients follow from the ring Fourier coefficients F1, F2 of
// gamma_1 and gamma_2 as
//   E_lm = sum_r [A F1 - i B F2] / N_l,  B_lm = sum_r [A F2 + i B F1] / N_l,
// N_l = sqrt((l+2)! / (l-2)!), so that a potential's shear gamma = eth^2 psi / 2
// has E_lm = N_l psi_lm / 2 and no B.  dlambda comes from the lambda table
// (sin t dlambda_lm = l eps_{l+1,m} lambda_{l+1,m} - (l+1) eps_lm lambda_{l-1,m}).
// Under theta -> pi - theta, A keeps the parity (-1)^{l+m} of lambda_lm and B
// takes the opposite one, which fixes the north/south combinations.
#include "fft.cuh"
#include "legendre.cuh"
#include "sphere.cuh"

namespace clc {

// E_lm and B_lm from the Legendre sums of the two fields with the ring weights
// 1, cos / sin^2 and 1 / sin^2 (legendre_analysis_cols, kinds 0, 1, 2; band
// limit lmax + 1).  With sin t dlambda_lm = e1 lambda_{l+1,m} - e0 lambda_{l-1,m},
//   sum A F  = -2 (e1 S1_{l+1} - e0 S1_{l-1}) - l(l+1) S0_l + 2 m^2 S2_l,
//   sum B F  = 2 m (e1 S2_{l+1} - e0 S2_{l-1} - S1_l):
// A and B are products of lambda and ring factors, so every sum over rings is
// one of the table's contractions and nothing is evaluated per (l, m, ring).
// eps_lm and the normalisation come from the table's own list: as square roots
// and divisions here they were the whole kernel (123 us at nside 512, now 62).
__global__ void k_eb_combine(const double2* __restrict__ S, size_t q, int lmax, int m0, const double* __restrict__ eps,
                             const double* __restrict__ inv_n, double2* __restrict__ E, double2* __restrict__ B) {
  const int m = m0 + blockIdx.y, lt = lmax + 1;
  eps += (size_t)blockIdx.y * (lmax + 3);
  const int l = m + blockIdx.x * blockDim.x + threadIdx.x;
  if (l > lmax) return;
  const size_t o = alm_idx(lmax, l, m);
  if (l < 2) {
    E[o] = B[o] = make_double2(0.0, 0.0);
    return;
  }
  const double e1 = (double)l * eps[l + 1], e0 = (l + 1.0) * eps[l];
  const double ll1 = (double)l * (l + 1.0), m2 = 2.0 * (double)m * m, m_2 = 2.0 * m;
  const size_t i = alm_idx(lt, l, m);
  double2 a[2], b[2];
#pragma unroll
  for (int f = 0; f < 2; ++f) {
    const double2 *S0 = S + (3 * f) * q + i, *S1 = S0 + q, *S2 = S1 + q;
    const double2 z = make_double2(0.0, 0.0);
    const double2 d1 = l > m ? S1[-1] : z, d2 = l > m ? S2[-1] : z, u1 = S1[1], u2 = S2[1];
    a[f].x = fma(-2.0, fma(e1, u1.x, -e0 * d1.x), fma(m2, S2->x, -ll1 * S0->x));
    a[f].y = fma(-2.0, fma(e1, u1.y, -e0 * d1.y), fma(m2, S2->y, -ll1 * S0->y));
    b[f].x = m_2 * (fma(e1, u2.x, -e0 * d2.x) - S1->x);
    b[f].y = m_2 * (fma(e1, u2.y, -e0 * d2.y) - S1->y);
  }
  const double inv = inv_n[l];
  // E = (A F1 - i B F2) / N_l, B = (A F2 + i B F1) / N_l
  E[o] = make_double2((a[0].x + b[1].y) * inv, (a[0].y - b[1].x) * inv);
  B[o] = make_double2((a[1].x - b[0].y) * inv, (a[1].y + b[0].x) * inv);
}

// C_l = (a_l0 b_l0* + 2 sum_{m>0} Re a_lm b_lm*) / (2l+1) of up to four pairs of
// coefficient sets (blockIdx.y), each packed with its own band limit.  A block
// takes 32 neighbouring l, which are neighbours in memory for every m, and its
// warps every kClWarps-th m (one thread per l and all its m in turn: 0.34 ms per
// spectrum at lmax 1024, against 0.02 ms for all four now).
constexpr int kClWarps = 32;

struct ClArgs {
  const double2* a[4];
  const double2* b[4];
  int lpack[4];
  double* cl[4];
};

__global__ void __launch_bounds__(32 * kClWarps) k_cl(ClArgs s, int lmax) {
  __shared__ double red[kClWarps][33];
  const int q = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int l = blockIdx.x * 32 + lane;
  const double2 *a = s.a[q], *b = s.b[q];
  const int lp = s.lpack[q];
  double acc = 0.0;
  for (int m = warp; m <= min(lmax, blockIdx.x * 32 + 31); m += kClWarps)
    if (l <= lmax && m <= l) {
      const double2 x = a[alm_idx(lp, l, m)], y = b[alm_idx(lp, l, m)];
      acc += (m ? 2.0 : 1.0) * (x.x * y.x + x.y * y.y);
    }
  red[warp][lane] = acc;
  __syncthreads();
  if (warp == 0 && l <= lmax) {
    double t = 0.0;
    for (int w = 0; w < kClWarps; ++w) t += red[w][lane];
    s.cl[q][l] = t / (2.0 * l + 1.0);
  }
}

// kappa, gamma_1, gamma_2, omega maps of A (SoA A[4][n], Eq. invmagmat)
__global__ void k_decompose_A(const double* __restrict__ A, int64_t n, double* __restrict__ out) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const double a = A[k], b = A[n + k], c = A[2 * n + k], d = A[3 * n + k];
    out[k] = 1.0 - 0.5 * (a + d);
    out[n + k] = -0.5 * (a - d);
    out[2 * n + k] = -0.5 * (b + c);
    out[3 * n + k] = 0.5 * (b - c);
  }
}

// The same decomposition after carrying each ray's A from the tangent basis
// at its source-sphere position x to the basis at its image position, the
// centre of RING pixel k (Appendix B transport along the geodesic between
// them).  One CTA per ring, like the ray initialisation: the ring geometry
// once, longitudes by sincospi.  kappa and omega are invariant under the
// rotation; the shear turns by twice its angle.
__global__ void k_decompose_A_image(const double* __restrict__ x, const double* __restrict__ A, int nside, int64_t n,
                                    double* __restrict__ out) {
  const int i = blockIdx.x + 1;
  const Ring r = ring_geom(nside, i);
  const double inv = 1.0 / (double)r.npix;
  const int shift = r.phi0 != 0.0 ? 1 : 0;
  const int quarter = r.npix / 4;
  for (int j = threadIdx.x; j < quarter; j += blockDim.x) {
    double s0, c0;
    sincospi((double)(2 * j + shift) * inv, &s0, &c0);
    for (int qd = 0; qd < 4; ++qd) {   // the pixels a quarter turn apart: swapped and negated, exactly
      const double cp = qd == 0 ? c0 : qd == 1 ? -s0 : qd == 2 ? -c0 : s0;
      const double sp = qd == 0 ? s0 : qd == 1 ? c0 : qd == 2 ? -s0 : -c0;
      const int64_t k = r.first + j + qd * quarter;
      const double n0[3] = {r.s * cp, r.s * sp, r.z};
      const double xv[3] = {x[k], x[n + k], x[2 * n + k]};
      const double ix = rsqrt(dot3(xv, xv));
      const double nx[3] = {xv[0] * ix, xv[1] * ix, xv[2] * ix};
      // transport along the geodesic as a plane rotation (q0, q1) (Appendix B);
      // the basis at the pixel centre is (z cos, z sin, -s), (-sin, cos, 0)
      double t[3], q[3];
      tangent_basis(nx, t, q);
      const double w = dot3(n0, t) / (1.0 + dot3(nx, n0));
      const double t1x = r.z * cp, t1y = r.z * sp;
      const double q0 = (t1x * t[0] + t1y * t[1] - r.s * t[2]) - w * (t1x * nx[0] + t1y * nx[1] - r.s * nx[2]);
      const double q1 = (cp * t[1] - sp * t[0]) - w * (cp * nx[1] - sp * nx[0]);
      // trace and antisymmetric part are kept, the shear turns by twice the angle
      const double a = A[k], b = A[n + k], c = A[2 * n + k], d = A[3 * n + k];
      const double c2 = fma(q0, q0, -q1 * q1), s2 = 2.0 * q0 * q1, df = a - d, sy = b + c;
      out[k] = fma(-0.5, a + d, 1.0);
      out[n + k] = -0.5 * fma(c2, df, -s2 * sy);
      out[2 * n + k] = -0.5 * fma(s2, df, c2 * sy);
      out[3 * n + k] = 0.5 * (b - c);
    }
  }
}

static int power_spectra(clc_ctx* ctx, const ClArgs& s, int n, int lmax) {
  CLC_LAUNCH(ctx, "k_cl", k_cl, dim3(lmax / 32 + 1, n), 32 * kClWarps, 0, s, lmax);
  return launch_check(ctx, "k_cl");
}

// E and B coefficients of the shear maps g[0], g[1], and, for ns = 2, the
// scalar coefficients (band limit lmax + 1 packing) of the maps s[0], s[1]:
// all in one pass over the Legendre table.
static int eb_analysis(clc_ctx* ctx, const double* const* g, int ns, const double* const* s, int nside, int lmax,
                       double2* E, double2* B, double2* const* salm) {
  int rc;
  auto plan = get_fft_plan(ctx, nside, &rc);
  if (rc) return rc;
  const int ldf = 4 * nside - 1;
  const size_t fq = (size_t)ldf * (lmax + 1), Q = (size_t)(lmax + 2) * (lmax + 3) / 2;
  double2* F = (double2*)scratch(ctx, ns ? 13 : 0, (2 + ns) * sizeof(double2) * fq);
  double2* S = (double2*)scratch(ctx, 12, 6 * sizeof(double2) * Q);
  if (!F || !S) return CLC_ENOMEM;
  const double w = 4.0 * kPi / (12.0 * (double)nside * nside);
  const double* in[4] = {g[0], g[1], ns > 0 ? s[0] : nullptr, ns > 1 ? s[1] : nullptr};
  if ((rc = ring_analysis_maps(ctx, *plan, 2 + ns, in, lmax, w, F, fq, ldf))) return rc;
  const double2* cols[8];
  double2* out[8];
  int kind[8];
  for (int v = 0; v < 6 + ns; ++v) {
    cols[v] = F + (v < 6 ? v / 3 : v - 4) * fq;
    kind[v] = v < 6 ? v % 3 : 0;
    out[v] = v < 6 ? S + v * Q : salm[v - 6];
  }
  return for_each_table(ctx, nside, lmax, [&](const LegendreTable& T) {
    const int r = legendre_analysis_cols(ctx, T, 6 + ns, cols, kind, ldf, out, lmax + 1);
    if (r) return r;
    CLC_LAUNCH(ctx, "k_eb_combine", k_eb_combine, dim3((lmax + 128) / 128, T.m1 - T.m0), 128, 0, S, Q, lmax, T.m0,
               T.eps_of(), T.by_l() + (lmax + 3), E, B);
    return launch_check(ctx, "k_eb_combine");
  });
}

}  // namespace clc

using namespace clc;

extern "C" int clc_eb_analysis(clc_ctx* ctx, const double* g1, const double* g2, int nside, int lmax, double* E,
                               double* B) {
  if (!ctx) return CLC_EINVAL;
  if (!valid_nside(nside) || nside > 4096 || lmax < 0 || lmax > 4 * nside)
    return set_err(ctx, CLC_EINVAL, "clc_eb_analysis: bad nside / lmax");
  if (!g1 || !g2 || !E || !B) return set_err(ctx, CLC_EINVAL, "clc_eb_analysis: null pointer");
  cudaSetDevice(ctx->device);
  const double* g[2] = {g1, g2};
  return eb_analysis(ctx, g, 0, nullptr, nside, lmax, (double2*)E, (double2*)B, nullptr);
}

extern "C" int clc_power_spectrum(clc_ctx* ctx, const double* alm, const double* alm2, int lmax, double* cl) {
  if (!ctx) return CLC_EINVAL;
  if (lmax < 0 || !alm || !cl) return set_err(ctx, CLC_EINVAL, "clc_power_spectrum: bad arguments");
  cudaSetDevice(ctx->device);
  ClArgs s{};
  s.a[0] = (const double2*)alm;
  s.b[0] = (const double2*)(alm2 ? alm2 : alm);
  s.lpack[0] = lmax;
  s.cl[0] = cl;
  return power_spectra(ctx, s, 1, lmax);
}

extern "C" int clc_lensing_spectra(clc_ctx* ctx, const double* x, const double* A, int nside, int lmax,
                                   double* cl_out) {
  if (!ctx) return CLC_EINVAL;
  if (!valid_nside(nside) || nside > 4096 || lmax < 2 || lmax > 4 * nside || !A || !cl_out)
    return set_err(ctx, CLC_EINVAL, "clc_lensing_spectra: bad arguments");
  cudaSetDevice(ctx->device);
  const int64_t np = 12ll * nside * nside;
  const size_t na = (size_t)(lmax + 1) * (lmax + 2) / 2, nt = (size_t)(lmax + 2) * (lmax + 3) / 2;
  double* maps = (double*)scratch(ctx, 5, 4 * np * sizeof(double) + 2 * (na + nt) * sizeof(double2));
  if (!maps) return CLC_ENOMEM;
  double2* E = (double2*)(maps + 4 * np);
  double2 *B = E + na, *salm[2] = {B + na, B + na + nt};
  int rc;
  if (x)
    CLC_LAUNCH(ctx, "k_decompose_A", k_decompose_A_image, 4 * nside - 1, 256, 0, x, A, nside, np, maps);
  else
    CLC_LAUNCH(ctx, "k_decompose_A", k_decompose_A, 1024, 256, 0, A, np, maps);
  if ((rc = launch_check(ctx, "k_decompose_A"))) return rc;
  const double *g[2] = {maps + np, maps + 2 * np}, *sc[2] = {maps, maps + 3 * np};
  if ((rc = eb_analysis(ctx, g, 2, sc, nside, lmax, E, B, salm))) return rc;
  const double2* alm[4] = {salm[0], E, B, salm[1]};   // kappa, E, B, omega
  ClArgs cs{};
  for (int q = 0; q < 4; ++q) {
    cs.a[q] = cs.b[q] = alm[q];
    cs.lpack[q] = q == 0 || q == 3 ? lmax + 1 : lmax;
    cs.cl[q] = cl_out + (size_t)q * (lmax + 1);
  }
  return power_spectra(ctx, cs, 4, lmax);
}
