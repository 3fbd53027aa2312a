// Legendre transforms of the HEALPix SHT (paper Sec. 3.2) to FP64 accuracy on
// the tensor cores.
#pragma once

#include <cuda_fp16.h>

#include "common.cuh"

namespace clc {

constexpr int kDigits = 8;      // signed base-256 digits of a table or data value
constexpr int kAtom = 4096;     // halves of one digit plane of a 64 x 64 atom

// lambda_lm(z_r) of the orders m0 <= m < m1 on the R = 2 nside northern rings
// (equator included), l = m .. lmax + 1, as digit planes for the contraction
// kernels of legendre.cu.  Group g = 2 (m - m0) + p holds the rows l = m + p +
// 2 k; 64 rows form a row block, 64 rings a ring block, and the atom of a row
// block and a ring block is kDigits planes of 64 x 64 FP16 integers in the
// 128-byte swizzle.  A row block keeps the atoms of its ring blocks rb0 .. nkb
// - 1 only: towards the pole lambda_lm falls below the last digit.
struct LegendreTable {
  int nside = 0, lmax = 0, R = 0, nkb = 0;
  int m0 = 0, m1 = 0;                            // orders held
  size_t bytes = 0;                              // of the atoms
  std::vector<int> h_gidx;                       // first row block of each group (2 nm + 1)
  Buffer gidx;                                   // the same on the device
  Buffer rb0;                                    // int: first ring block kept, per row block
  Buffer abase;                                  // const __half*: atom of ring block rb0, per row block
  Buffer rexp;                                   // int: row values are below 2^rexp, 64 per row block
  Buffer cexp;                                   // int8: ring r of order m is scaled by 2^cexp, [m - m0][nkb * 64]
  Buffer fac;                                    // double [2][R]: cos / sin^2 and 1 / sin^2 of the rings
  Buffer zero;                                   // an atom of zeros
  // eps_lm = sqrt((l^2 - m^2) / (4 l^2 - 1)) [m - m0][lmax + 3] of l = 0 .. lmax + 2,
  // then by l: -1 / (l (l + 1)) (0 at l = 0) and 1 / sqrt((l+2)(l+1) l (l-1)) (0 below 2)
  Buffer eps;
  const double* eps_of() const { return (const double*)eps.p; }
  const double* by_l() const { return (const double*)eps.p + (size_t)(m1 - m0) * (lmax + 3); }
  std::vector<std::unique_ptr<Buffer>> atoms;    // the atoms, a piece per segment of a table that stays, else one arena
  bool arena = false;
  Buffer an, sy;                                 // work lists of the contractions (int4), longest first
  int n_an = 0, n_sy = 0;
};

// Buffers of a build, kept from one range of orders to the next.
struct LegendreBuild {
  Buffer tab, ab, ln, off, grp;
};
// A table of the orders from m0 on, up to m1 - 1, that fit `limit` bytes of atoms
// (at least one order); T->m1 tells where it ends.  stays: the table may stay,
// fill the limit as far as it goes with memory of its size; otherwise one arena of
// the limit, and an end where the rest would cost another segment.  T may hold an
// earlier range: its buffers are used again.
int build_legendre_table(clc_ctx* ctx, int nside, int lmax, int m0, int m1, size_t limit, bool stays, LegendreBuild& W,
                         LegendreTable* T);
// The table to use for the orders from m0 on: the context's, or one built into
// `own` (made if null).
int legendre_table_from(clc_ctx* ctx, int nside, int lmax, int m0, LegendreBuild& W,
                        std::shared_ptr<LegendreTable>& own, std::shared_ptr<LegendreTable>* T);

// packed index of (l, m) for band limit lmax (m-major)
__host__ __device__ __forceinline__ long long alm_idx(int lmax, int l, int m) {
  return (long long)m * (2 * lmax + 1 - m) / 2 + l;
}

// For v < nv <= 8: out[v][idx(l, m)] = sum_r lambda_lm(r) w_v(r) V_m^{(l+m) % 2}(r)
// from ring Fourier coefficients F[v][m * ldf + ring] (weights already
// applied), for the table's orders and l <= ltop (lmax by default, at most
// lmax + 1), packed with band limit ltop.  V^p is north + (-1)^p south;
// kind[v] (null: all 0) selects the ring weight w: 0: 1; 1: cos / sin^2 (odd
// under the reflection, so V^p is north - (-1)^p south); 2: 1 / sin^2.
int legendre_analysis_cols(clc_ctx* ctx, const LegendreTable& T, int nv, const double2* const* F, const int* kind,
                           int ldf, double2* const* out, int ltop = -1);
inline int legendre_analysis(clc_ctx* ctx, const LegendreTable& T, const double2* F, int ldf, double2* alm,
                             int ltop = -1) {
  return legendre_analysis_cols(ctx, T, 1, &F, nullptr, ldf, &alm, ltop);
}

// The same of one map up to lmax, summed directly at low band limits.
int legendre_analysis_map(clc_ctx* ctx, const LegendreTable& T, const double2* F, int ldf, double2* alm);

// G_q[m][ring] = sum_l lambda_lm(ring) rhs_q[idx'(l, m)] for q < nq <= 4, where
// rhs_q is packed with band limit lmax + 1 (idx' = alm_idx(lmax + 1, l, m)) and
// lq[q] is the highest l used by rhs q.  G_q lives at G + q * ld * (lmax + 2).
int legendre_synthesis(clc_ctx* ctx, const LegendreTable& T, const double2* rhs, int nq, const int* lq,
                       double2* G, int ld);

// The same sums of a Poisson solve straight from the source's coefficients
// klm (band limit lmax): q = 0: psi_lm = -k_lm / (l (l + 1)); with nq = 3 also
// q = 1: b_lm = (l-1) eps_lm psi_{l-1,m} - (l+2) eps_{l+1,m} psi_{l+1,m} (the
// coefficients of sin(theta) d psi / d theta, l <= lmax + 1) and q = 2:
// -l (l + 1) psi_lm.
int legendre_synthesis_poisson(clc_ctx* ctx, const LegendreTable& T, const double2* klm, int nq, double2* G, int ld);

// Run fn on tables covering every order m <= lmax: the context's whole table
// when it fits in device memory (or the context's budget), otherwise tables of
// consecutive order ranges built one after the other in the same memory (the
// recurrence is then recomputed per call).
template <typename Fn>
int for_each_table(clc_ctx* ctx, int nside, int lmax, Fn fn) {
  LegendreBuild W;
  std::shared_ptr<LegendreTable> own;
  size_t bytes = 0;
  for (int m0 = 0; m0 <= lmax;) {
    std::shared_ptr<LegendreTable> T;
    int rc = legendre_table_from(ctx, nside, lmax, m0, W, own, &T);
    if (rc) return rc;
    if ((rc = fn(*T))) return rc;
    m0 = T->m1;
    bytes += T->bytes;
  }
  ctx->leg_bytes[{nside, lmax}] = bytes;
  return own ? cuda_check(ctx, cudaStreamSynchronize(ctx->stream), "table chunk") : CLC_OK;
}

}  // namespace clc
