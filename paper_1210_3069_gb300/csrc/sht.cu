// SHT entry points and the pure-SHT Poisson solve (paper Sec. 3.2):
// analysis of kappa, psi_lm = -kappa_lm / (l (l + 1)) with the l = 0 term set
// to zero, and synthesis of psi and of its derivatives.  The theta derivative
// is synthesised through the coefficients b_lm of sin(theta) d/dtheta psi,
//   sin t d/dt lambda_lm = l eps_{l+1,m} lambda_{l+1,m} - (l+1) eps_lm lambda_{l-1,m},
//   eps_lm = sqrt((l^2 - m^2) / (4 l^2 - 1)),
// phi derivatives multiply the ring Fourier coefficients by i m, and the
// theta-theta component of the Hessian follows from the Laplacian:
// U_tt = kappa_bl - U_pp with kappa_bl = sum -l(l+1) psi_lm Y_lm.
#include <algorithm>

#include "fft.cuh"
#include "legendre.cuh"

namespace clc {

int poisson_sht_tc(clc_ctx* ctx, const double* const* kappa, int P, int nside, int lmax, double* const* psi,
                   const clc_derivs* out);

// copy alm (band limit lmax) into the lmax + 1 packing, zero at l = lmax + 1
__global__ void k_alm_expand(const double2* __restrict__ alm, int lmax, double2* __restrict__ rhs) {
  const int m = blockIdx.y;
  const int lt = lmax + 1;
  const int l = m + blockIdx.x * blockDim.x + threadIdx.x;
  if (l > lt) return;
  double2 v = make_double2(0.0, 0.0);
  if (l <= lmax) v = alm[alm_idx(lmax, l, m)];
  if (m == 0) v.y = 0.0;
  rhs[alm_idx(lt, l, m)] = v;
}

static int check_sht_args(clc_ctx* ctx, int nside, int lmax, const char* who) {
  if (!valid_nside(nside) || nside > 4096) return set_err(ctx, CLC_EINVAL, std::string(who) + ": bad nside");
  if (lmax < 0 || lmax > 4 * nside) return set_err(ctx, CLC_EINVAL, std::string(who) + ": lmax must be in [0, 4 nside]");
  return CLC_OK;
}

// analysis into a device alm buffer (band limit lmax)
int sht_analysis(clc_ctx* ctx, const double* map, int nside, int lmax, double2* alm) {
  int rc;
  auto plan = get_fft_plan(ctx, nside, &rc);
  if (rc) return rc;
  const int ldf = 4 * nside - 1;
  double2* F = (double2*)scratch(ctx, 0, sizeof(double2) * (size_t)ldf * (lmax + 1));
  if (!F) return CLC_ENOMEM;
  const double w = 4.0 * kPi / (12.0 * (double)nside * nside);
  if ((rc = ring_analysis(ctx, *plan, map, lmax, w, F, ldf))) return rc;
  return for_each_table(ctx, nside, lmax, [&](const LegendreTable& T) { return legendre_analysis_map(ctx, T, F, ldf, alm); });
}

// synthesis of nq right-hand sides (lmax + 1 packing) and the ring FFTs
int sht_synthesis_rhs(clc_ctx* ctx, const double2* rhs, int nq, const int* lq, int nside, int lmax, int mode,
                      double* const out[6]) {
  int rc;
  auto plan = get_fft_plan(ctx, nside, &rc);
  if (rc) return rc;
  const int ld = 4 * nside - 1;
  double2* G = (double2*)scratch(ctx, 3, sizeof(double2) * (size_t)nq * ld * (lmax + 2));
  if (!G) return CLC_ENOMEM;
  if ((rc = for_each_table(ctx, nside, lmax,
                           [&](const LegendreTable& T) { return legendre_synthesis(ctx, T, rhs, nq, lq, G, ld); })))
    return rc;
  return ring_synthesis(ctx, *plan, G, ld, lmax, mode, out);
}

}  // namespace clc

using namespace clc;

extern "C" int clc_set_table_budget(clc_ctx* ctx, size_t bytes) {
  if (!ctx) return CLC_EINVAL;
  ctx->table_budget = bytes;
  return CLC_OK;
}

extern "C" int clc_sht_analysis(clc_ctx* ctx, const double* map, int nside, int lmax, double* alm) {
  if (!ctx) return CLC_EINVAL;
  int rc = check_sht_args(ctx, nside, lmax, "clc_sht_analysis");
  if (rc) return rc;
  if (!map || !alm) return set_err(ctx, CLC_EINVAL, "clc_sht_analysis: null pointer");
  cudaSetDevice(ctx->device);
  return sht_analysis(ctx, map, nside, lmax, (double2*)alm);
}

extern "C" int clc_sht_synthesis(clc_ctx* ctx, const double* alm, int nside, int lmax, double* map) {
  if (!ctx) return CLC_EINVAL;
  int rc = check_sht_args(ctx, nside, lmax, "clc_sht_synthesis");
  if (rc) return rc;
  if (!map || !alm) return set_err(ctx, CLC_EINVAL, "clc_sht_synthesis: null pointer");
  cudaSetDevice(ctx->device);
  const long long Q = alm_idx(lmax + 1, lmax + 1, lmax + 1) + 1;
  double2* rhs = (double2*)scratch(ctx, 2, sizeof(double2) * Q);
  if (!rhs) return CLC_ENOMEM;
  dim3 grid((lmax + 2 + 127) / 128, lmax + 1);
  CLC_LAUNCH(ctx, "k_alm_expand", k_alm_expand, grid, 128, 0, (const double2*)alm, lmax, rhs);
  if ((rc = launch_check(ctx, "k_alm_expand"))) return rc;
  const int lq[1] = {lmax};
  double* out[6] = {map, nullptr, nullptr, nullptr, nullptr, nullptr};
  return sht_synthesis_rhs(ctx, rhs, 1, lq, nside, lmax, 0, out);
}

extern "C" int clc_poisson_sht(clc_ctx* ctx, const double* kappa, int nside, int lmax, int precision, double* psi,
                               const clc_derivs* d) {
  if (!ctx) return CLC_EINVAL;
  int rc = check_sht_args(ctx, nside, lmax, "clc_poisson_sht");
  if (rc) return rc;
  if (!kappa) return set_err(ctx, CLC_EINVAL, "clc_poisson_sht: null kappa");
  if (precision != CLC_FP64 && precision != CLC_MIXED)
    return set_err(ctx, CLC_EINVAL, "clc_poisson_sht: precision must be CLC_FP64 or CLC_MIXED");
  cudaSetDevice(ctx->device);
  const bool derivs = d && (d->a_th || d->a_ph || d->u_tt || d->u_pp || d->u_tp);
  if (!psi && !derivs) return CLC_OK;
  if (precision == CLC_MIXED) return poisson_sht_tc(ctx, &kappa, 1, nside, lmax, &psi, derivs ? d : nullptr);
  double2* klm = (double2*)scratch(ctx, 1, sizeof(double2) * (alm_idx(lmax, lmax, lmax) + 1));
  if (!klm) return CLC_ENOMEM;
  auto plan = get_fft_plan(ctx, nside, &rc);
  if (rc) return rc;
  const int ld = 4 * nside - 1;
  double2* F = (double2*)scratch(ctx, 0, sizeof(double2) * (size_t)ld * (lmax + 1));
  if (!F) return CLC_ENOMEM;
  const int nq = derivs ? 3 : 1;
  double2* G = (double2*)scratch(ctx, 3, sizeof(double2) * (size_t)nq * ld * (lmax + 2));
  if (!G) return CLC_ENOMEM;
  const double w = 4.0 * kPi / (12.0 * (double)nside * nside);
  if ((rc = ring_analysis(ctx, *plan, kappa, lmax, w, F, ld))) return rc;
  // per table (or order range): analysis, then synthesis from the coefficients
  rc = for_each_table(ctx, nside, lmax, [&](const LegendreTable& T) {
    const int r = legendre_analysis(ctx, T, F, ld, klm);
    return r ? r : legendre_synthesis_poisson(ctx, T, klm, nq, G, ld);
  });
  if (rc) return rc;
  if (!derivs) {
    double* out[6] = {psi, nullptr, nullptr, nullptr, nullptr, nullptr};
    return ring_synthesis(ctx, *plan, G, ld, lmax, 0, out);
  }
  double* out[6] = {psi, d->a_th, d->a_ph, d->u_tt, d->u_pp, d->u_tp};
  return ring_synthesis(ctx, *plan, G, ld, lmax, 1, out);
}
