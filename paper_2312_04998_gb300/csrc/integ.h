// Device-side state of the batched integrator, shared by the fused per-cell
// kernel (cell.cu) and the kernels that work class by class (integrate.cu).
#pragma once

#include "internal.h"

namespace integ {

constexpr int QMAX = 5;  // highest BDF order; the history keeps QMAX + 1 points
// counters[] entries of the compaction (0..3 belong to the attempt loop and
// the adjoint)
constexpr int kCAct = 8;     // slots holding the running cells: [0, counters[kCAct])
constexpr int kCHoles = 9;   // finished cells below the new boundary
constexpr int kCRun = 10;    // running cells above it
constexpr int kCLive = 11;   // running cells counted for the compaction
constexpr int kCounters = 16;
constexpr int kCkpt = SM_CHECKPOINT_EVERY;
enum : int {
  F_NEED_J = 1, F_REJECTED = 2, F_HAS_EPREV = 4, F_NEWTON = 8, F_CONV = 16,
  F_FINAL = 32, F_REFRESH = 64, F_FAILED = 128, F_ATTEMPT = 256
};

struct Dev {
  int n, n_r, nnz_j, mixed, tf32, head;
  int64_t C, ld;
  double rtol, atol, gamma_tol, newton_tol, eta_max, eta_keep, t_end;
  int q_max, max_steps, j_age_max, newton_max, max_conv_fails;
  // per-cell scalars [ld] (tn, alpha: [QMAX+1][ld])
  double *t, *h, *gam, *gam_J, *crate, *dprev, *tn, *alpha;
  int *q, *nh, *n_at_q, *j_age, *flags, *crej, *ccf, *status, *m_it;
  int *steps, *rejects, *conv_fails, *newton_iters, *jac_evals;
  // per-cell vectors [n][ld]; Y is [QMAX+1][n][ld]
  double *Y, *ypred, *y, *psi, *f, *f0, *eprev, *w, *wf;
  int *list, *counters;  // counters[0] = refresh list length, [1] = running cells
  // compaction of the running cells (states that record no steps): cell
  // slots are permuted so that running cells occupy slots [0, counters[kCAct])
  int* slot_cell;        // [ld] slot -> cell of the caller's arrays (and of the packed factors)
  int compact;           // 1: compaction on
  double* kslot;         // [n_r][ld] rate coefficients in slot order (compaction on), else null
  int *holes, *runners;  // [ld] each: the slot pairs of one compaction
  // recording (record > 0): per accepted step m (1-based) at [m-1][ld]; the
  // step history after every kCkpt-th accepted step at checkpoint m / kCkpt
  int record;
  double *log_t, *log_h;
  int* log_q;
  double *ck_Y, *ck_t;   // [K][QMAX+1][n][ld], [K][QMAX+1][ld]
  int* ck_nh;            // [K][ld]
  void* lu;
  int64_t lu_stride;
  int ldm;
  // packed factors read by the substitution (see LUSymbolic): per cell
  // lup_stride values from lup; null when the state keeps dense factors only
  void* lup;
  int64_t lup_stride;
  int lu_cta;   // 1: lu holds one dense working matrix per refresh CTA (not per cell)
  int p_l11, p_u11, p_dinv, p_l21, p_u12, p_d, ldd, n_flev, n_blev;
  const int *u11ptr, *flev_ptr, *flev, *blev_ptr, *blev;
  const int *hop_ptr, *hop_piv;     // head program (see LUSymbolic)
  const int4* hop;
  const int2* hterm;
  int n_hlev;
  const int *perm, *iperm, *lptr, *lidx, *uptr, *uidx, *lrptr, *lridx, *uoff, *lrhead, *lrhoff, *u12off, *lrhk, *srow;
  int n_srow;
  const int2 *jt_slot, *reac;
  const int* sc_ptr;
  const uint32_t* sc_ent;
  const int4* jdesc;     // per Jacobian entry {t0, t1, jrc, row << 16 | col}
  const int* jlong;      // entries with more than kJLong terms
  int n_jlong;
  // coupled temperature (therm = 1, see sm_net_set_thermal): row t_idx of
  // every state vector holds T; k' of the T-dependent reactions is
  // recomputed from it (into kslot) before every right-hand side
  int therm, t_idx, n_cool, bpad;
  double th_heat, th_lam, th_Td, th_zeta;
  const RatePar* rpar;
  const double *th_L, *th_E, *th_dn;   // [n] cooling coefficients, [n] excitation temperatures, [n_r] net particle change
  const int* th_cool;                  // [n_cool] the coolant species
  const double *c_nH, *c_Av, *c_chi;   // [ld] cell conditions, cell order
  double *bz, *bgv, *bs;               // per cell (cell order): z, gamma_J v ([ld][bpad]) and the Schur complement ([ld])
};

__device__ __forceinline__ double& V(double* a, const Dev& d, int s, int64_t c) {
  return a[(int64_t)s * d.ld + c];
}
__device__ __forceinline__ double* Yh(const Dev& d, int i) { return d.Y + (int64_t)i * d.n * d.ld; }

// Weights of the polynomial through (T[i], .), i < m, evaluated at t.
__device__ inline void lagrange(const double* T, int m, double t, double* wts) {
  for (int i = 0; i < m; ++i) {
    double num = 1.0, den = 1.0;
    for (int j = 0; j < m; ++j)
      if (j != i) {
        num *= t - T[j];
        den *= T[i] - T[j];
      }
    wts[i] = num / den;
  }
}

// alpha_i = h l_i'(tau_0) on nodes tau_0 = tnew, tau_i = T[i-1] (i = 1..q).
__device__ inline void bdf_alphas(double tnew, const double* T, int q, double h, double* al) {
  double tau[QMAX + 1];
  tau[0] = tnew;
  for (int i = 1; i <= q; ++i) tau[i] = T[i - 1];
  double s = 0.0;
  for (int i = 1; i <= q; ++i) s += 1.0 / (tau[0] - tau[i]);
  al[0] = h * s;
  for (int i = 1; i <= q; ++i) {
    double num = 1.0, den = 1.0;
    for (int m = 1; m <= q; ++m)
      if (m != i) num *= tau[0] - tau[m];
    for (int m = 0; m <= q; ++m)
      if (m != i) den *= tau[i] - tau[m];
    al[i] = h * num / den;
  }
}

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

}  // namespace integ
