// The fused integrator: one CTA carries one cell through its BDF attempts.
//
// Every cell has its own step size, order and Newton iterations, and nothing
// in an attempt couples cells, so a CTA runs a cell's whole sequence of
// attempts (predict, Jacobian and factorisation when due, Newton rounds, error
// test) in one kernel, with the cell's vectors, reaction rates and working
// panels in shared memory.  Compared with one launch per kernel class over
// all cells, a batch of few cells is no longer bound by launch gaps and by
// the one or two CTAs its 32-cell blocks fill, and a batch of many cells
// keeps FP64 (right-hand side, predictor), FP32 (factorisation) and L2
// (substitution) busy at once, since different cells are in different phases.
//
// Work split inside an attempt (n species, n_r reactions, tail of nt columns):
//   rates, S R    a thread per reaction, then the rows of S in pieces of at
//                 most 32 entries, a piece per lane (CellProg); bound by the
//                 FP64 pipe (2 lanes a clock per SM)
//   Jacobian      an entry per lane over the table of dR/dx in shared memory
//   head          the head program, level by level, in shared memory
//   tail          left-looking by 32-column panels: warp w holds rows
//                 32 w .. 32 w + 31 of the panel in registers (a row per
//                 lane), the finished columns to its left stream from the
//                 packed factors (L2), the 32 x 32 blocks of U of the panel
//                 go round through shared memory.  Every element of the
//                 tail is written once, in its final place.
//   substitution  a warp per 32 rows; the next block's factors are in flight
//                 while the diagonal block's 32-step chain runs
#include "cell.h"
#include <algorithm>

#include "integ.h"

using namespace integ;

namespace {

constexpr int XP = 40;         // row pitch of the 32 x 32 exchange blocks (words): 16-byte rows, few conflicts
constexpr unsigned kFull = 0xffffffffu;

// A cell's scalars while a CTA works on it.
struct CellS {
  double t, h, gam, gam_J, crate, dprev, tnew, err, eta[3];
  double tn[QMAX + 1], alpha[QMAX + 1], wts[QMAX + 1];
  int q, nh, n_at_q, j_age, flags, crej, ccf, status, m_it, steps, rejects, conv_fails, newton_iters, jac_evals;
  int base;      // history point i is scratch slot (base + i) % (QMAX + 1)
  int state, c, best_q;
  int lo, hi;
};
static_assert(sizeof(CellS) <= 512, "shared-memory plan");

struct Args {
  Dev d;
  CellPlan p;
  const int* w;            // index programs (CellProg blob)
  int nb, pitch;
  int n_rsl, n_part, n_rlong, rp_off, rp_ent, rp_dst, row_ptr, row_long;
  int n_jsl, n_jl, jg_off, jg_ent, jg_rc, jg_dst, jg_grp, jl_ptr, jl_ent, jl_rc, jl_dst, jl_grp;
  int n_hlev, hop, hterm, hop_ptr;
  int tg_grp, tg_off, tg_ent, tg_pos;
  int lev_f, lev_b, u12c, n_l21, n_u12;
  int n_vsl, n_vpart, n_vlong, vp_off, vp_ent, vp_dst, vrow_ptr, vrow_long;
  const double* k;
  int64_t ldk;
  double* scratch;
  int *ring, *done;
  int attempts, slice;
  double* timing;
  int timing_kind;
};

// optional cycle counters of the phases (build option SM_PHASE_CLOCKS)
constexpr int kPhaseSlots = 16;
enum { PH_LOAD, PH_PREDICT, PH_RATES, PH_GATHER, PH_SOLVE, PH_FINISH, PH_JAC, PH_HEAD, PH_ASSEMBLE, PH_UPDATE, PH_PANEL };
#ifdef SM_PHASE_CLOCKS
__device__ unsigned long long g_phase_cycles[kPhaseSlots];
#define PHASE_MARK(k)                                                          \
  do {                                                                         \
    if (threadIdx.x == 0) {                                                    \
      const long long ph_now = clock64();                                      \
      atomicAdd(&g_phase_cycles[(k)], (unsigned long long)(ph_now - ph_t));    \
      ph_t = ph_now;                                                           \
    }                                                                          \
  } while (0)
#define PHASE_ARG , long long& ph_t
#define PHASE_PASS , ph_t
#else
#define PHASE_MARK(k) do {} while (0)
#define PHASE_ARG
#define PHASE_PASS
#endif

// ---- packed FP32 arithmetic: two FMAs an instruction -----------------------
typedef unsigned long long f2;
__device__ __forceinline__ f2 pack2(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

__device__ __forceinline__ uint32_t to_tf32(float x) {
  uint32_t u;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(u) : "f"(x));
  return u;
}
__device__ __forceinline__ void split_tf32(float x, uint32_t& hi, uint32_t& lo) {
  hi = to_tf32(x);
  lo = to_tf32(x - __uint_as_float(hi));
}
__device__ __forceinline__ void mma_tf32(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
               "{%0,%1,%2,%3};\n"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ void cp16(void* smem, const void* g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ double flip(double v, int word) {   // v, negated when bit 31 of word is set
  return __hiloint2double(__double2hiint(v) ^ (word & 0x80000000), __double2loint(v));
}

// Sums of the rows cut into pieces: partial sums of the table's entries
// (a piece per lane, two chains), then the pieces of each row in order (rows
// of more than 4 pieces: a warp).  tab[pad slot] must be 0.  All threads.
__device__ __forceinline__ void row_sums(const int* __restrict__ w, int n_sl, int off, int ent, int dst, int row_ptr,
                                         int n_long, int row_long, const double* tab, double* part, double* out,
                                         int n) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int s = warp; s < n_sl; s += nw) {
    const int e0 = __ldg(w + off + s), e1 = __ldg(w + off + s + 1);
    const int* q = w + ent + 32 * e0 + lane;
    const int m = e1 - e0;
    double a0 = 0.0, a1 = 0.0;
    int e = 0;
    for (; e + 4 <= m; e += 4) {
      const int w0 = __ldg(q + 32 * e), w1 = __ldg(q + 32 * e + 32), w2 = __ldg(q + 32 * e + 64), w3 = __ldg(q + 32 * e + 96);
      const double v0 = tab[w0 & 0x7FFFFFFF], v1 = tab[w1 & 0x7FFFFFFF], v2 = tab[w2 & 0x7FFFFFFF],
                   v3 = tab[w3 & 0x7FFFFFFF];
      a0 += flip(v0, w0);
      a1 += flip(v1, w1);
      a0 += flip(v2, w2);
      a1 += flip(v3, w3);
    }
    for (; e < m; ++e) {
      const int w0 = __ldg(q + 32 * e);
      a0 += flip(tab[w0 & 0x7FFFFFFF], w0);
    }
    part[__ldg(w + dst + 32 * s + lane)] = a0 + a1;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const int p0 = __ldg(w + row_ptr + i), p1 = __ldg(w + row_ptr + i + 1);
    if (p1 - p0 > 4) continue;
    double v = 0.0;
    for (int p = p0; p < p1; ++p) v += part[p];
    out[i] = v;
  }
  for (int q = nw - 1 - warp; q < n_long; q += nw) {
    const int i = __ldg(w + row_long + q);
    const int p1 = __ldg(w + row_ptr + i + 1);
    double v = 0.0;
    for (int p = __ldg(w + row_ptr + i) + lane; p < p1; p += 32) v += part[p];
    v = warp_sum(v);
    if (lane == 0) out[i] = v;
  }
}

// Sum over the CTA, valid in warp 0 (all threads must call; one barrier
// inside; `slot` 0..3 keeps independent sums apart).
__device__ __forceinline__ double cta_sum(double v, double* red, int slot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = warp_sum(v);
  if (lane == 0) red[32 * slot + warp] = v;
  __syncthreads();
  if (warp == 0) v = warp_sum(lane < nw ? red[32 * slot + lane] : 0.0);
  return v;
}

// R_j = k'_j prod y into tab (slot n_r = 0), then fs = S R.  Ends with a barrier.
__device__ void cell_rhs(const Args& A, const double* kc, const double* y, double* tab, double* part, double* fs PHASE_ARG) {
  const int n_r = A.d.n_r;
  for (int j = threadIdx.x; j < n_r; j += blockDim.x) {
    const int2 rc = __ldg(A.d.reac + j);
    double v = kc[j] * y[rc.x];
    if (rc.y >= 0) v *= y[rc.y];
    tab[j] = v;
  }
  if (threadIdx.x == 0) tab[n_r] = 0.0;
  __syncthreads();
  PHASE_MARK(PH_RATES);
  row_sums(A.w, A.n_rsl, A.rp_off, A.rp_ent, A.rp_dst, A.row_ptr, A.n_rlong, A.row_long, tab, part, fs, A.d.n);
  __syncthreads();
  PHASE_MARK(PH_GATHER);
}

// ---- coupled temperature ----------------------------------------------------
// k' of the T-dependent reactions (all reactions when init) at temperature T.
__device__ void cell_th_rates(const Args& A, double* kc, double T, double nH, double Av, double chi, bool init) {
  const double lt = log(T * (1.0 / 300.0)), it = 1.0 / T;
  for (int j = threadIdx.x; j < A.d.n_r; j += blockDim.x) {
    const RatePar p = A.d.rpar[j];
    const int cls = (int)p.w;
    if (cls == SM_TWO_BODY || cls == SM_DISS_RECOMB) kc[j] = exp(fma(p.y, lt, p.x) - p.z * it) * nH;
    else if (init) kc[j] = cls == SM_COSMIC_RAY ? p.x * A.d.th_zeta : chi * p.x * exp(-p.z * Av);
  }
  __syncthreads();
}

// Temperature row of fs from y and the chemical rows.  Ends with a barrier.
__device__ void cell_energy(const Args& A, const double* y, double* fs, double nH, double* red) {
  const Dev& d = A.d;
  const int t = d.t_idx;
  const double T = y[t];
  double xt = 0.0, F = 0.0, line = 0.0;
  for (int s = threadIdx.x; s < d.n; s += blockDim.x) {
    if (s == t) continue;
    xt += y[s];
    F += fs[s];
  }
  for (int q = threadIdx.x; q < d.n_cool; q += blockDim.x) {
    const int i = __ldg(d.th_cool + q);
    line = fma(y[i], d.th_L[i] * exp(-d.th_E[i] / T), line);
  }
  xt = cta_sum(xt, red, 0);
  F = cta_sum(F, red, 1);
  line = cta_sum(line, red, 2);
  if (threadIdx.x == 0)
    fs[t] = (d.th_heat - nH * line - d.th_lam * nH * (T - d.th_Td) - 1.5 * T * F) / (1.5 * xt);
  __syncthreads();
}

// ---- substitution -----------------------------------------------------------
__device__ __forceinline__ void load4(const float* p, float (&v)[4]) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
__device__ __forceinline__ void load4(const double* p, double (&v)[4]) {
  const double2 q = *reinterpret_cast<const double2*>(p), r = *reinterpret_cast<const double2*>(p + 2);
  v[0] = q.x; v[1] = q.y; v[2] = r.x; v[3] = r.y;
}

// x := M^-1 x with a cell's packed factors P; x in elimination order, head
// part xh[h], tail part xt (16-byte aligned, 32 nb entries).  tmp holds the
// products of the L21 / U12 entries, which all threads form at once (their
// rows have up to a hundred entries, a chain no single thread should walk).
// Begins and ends with a barrier.
template <class T>
__device__ void cell_solve(const Args& A, const T* P, T* xh, T* xt, T* tmp) {
  constexpr int CH = sizeof(T) == 4 ? 32 : 16;   // columns of a block in registers at a time
  const Dev& d = A.d;
  const int n = d.n, h = d.head, nt = n - h, ldd = d.ldd, nb = A.nb;
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, rb = tid >> 5;
  const T* D = P + d.p_d;
  const int row = 32 * rb + lane;
  __syncthreads();
  // head, forward: a row per thread, level by level, its entries loaded ahead
  constexpr int HE = 4;
  for (int i0 = 0; i0 < h; i0 += nthr) {   // one pass unless the head outgrows the CTA (rows of a pass come first)
    const int i = i0 + tid;
    const bool in = i < h;
    const int p0 = in ? __ldg(d.lrptr + i) : 0, cnt = in ? __ldg(d.lrptr + i + 1) - p0 : 0;
    const int lev = in ? __ldg(A.w + A.lev_f + i) : -1;
    T pv[HE];
    int pi[HE];
#pragma unroll
    for (int e = 0; e < HE; ++e) {
      pv[e] = e < cnt ? P[d.p_l11 + p0 + e] : T(0);
      pi[e] = e < cnt ? __ldg(d.lridx + p0 + e) : 0;
    }
    for (int l = i0 == 0 ? 1 : 0; l < d.n_flev; ++l) {
      if (lev == l) {
        T s = T(0);
#pragma unroll
        for (int e = 0; e < HE; ++e) s += pv[e] * xh[pi[e]];
        for (int e = HE; e < cnt; ++e) s += P[d.p_l11 + p0 + e] * xh[__ldg(d.lridx + p0 + e)];
        xh[i] -= s;
      }
      __syncthreads();
    }
  }
  // L21
#pragma unroll 4
  for (int e = tid; e < A.n_l21; e += nthr) tmp[e] = P[d.p_l21 + e] * xh[__ldg(d.lrhk + e)];
  __syncthreads();
  T xi = T(0);
  if (row < nt) {
    const int e1 = __ldg(d.lrhoff + row + 1);
    T s0 = T(0), s1 = T(0);
    int e = __ldg(d.lrhoff + row);
    for (; e + 4 <= e1; e += 4) {
      s0 += tmp[e];
      s1 += tmp[e + 1];
      s0 += tmp[e + 2];
      s1 += tmp[e + 3];
    }
    for (; e < e1; ++e) s0 += tmp[e];
    xi = xt[row] - (s0 + s1);
  }
  // tail, forward (unit lower triangle)
  for (int K = 0; K < nb; ++K) {
    const int w = min(32, nt - 32 * K);
    const T* col = D + (int64_t)(32 * K) * ldd + row;
    T l[CH];
    const bool use = rb >= K && row < nt;
#pragma unroll
    for (int k = 0; k < CH; ++k) l[k] = use && k < w && (rb > K || k < lane) ? col[(int64_t)k * ldd] : T(0);
    if (rb == K) {
#pragma unroll
      for (int k0 = 0; k0 < 32; k0 += CH) {
        if (k0) {
#pragma unroll
          for (int k = 0; k < CH; ++k) l[k] = use && k0 + k < w && k0 + k < lane ? col[(int64_t)(k0 + k) * ldd] : T(0);
        }
#pragma unroll
        for (int k = 0; k < CH; ++k) {
          const T xk = __shfl_sync(kFull, xi, k0 + k);
          xi -= l[k] * xk;   // l is 0 on and above the diagonal
        }
      }
      xt[row] = row < nt ? xi : T(0);
    }
    __syncthreads();
    if (rb > K && rb < nb) {
#pragma unroll
      for (int k0 = 0; k0 < 32; k0 += CH) {
        if (k0) {
#pragma unroll
          for (int k = 0; k < CH; ++k) l[k] = use ? col[(int64_t)(k0 + k) * ldd] : T(0);
        }
        T a0 = T(0), a1 = T(0);
#pragma unroll
        for (int k = 0; k < CH; k += 4) {
          T xv[4];
          load4(xt + 32 * K + k0 + k, xv);
          a0 += l[k] * xv[0];
          a1 += l[k + 1] * xv[1];
          a0 += l[k + 2] * xv[2];
          a1 += l[k + 3] * xv[3];
        }
        xi -= a0 + a1;
      }
    }
  }
  // tail, backward (inverse pivots on the diagonal)
  for (int K = nb - 1; K >= 0; --K) {
    const int w = min(32, nt - 32 * K);
    const T* col = D + (int64_t)(32 * K) * ldd + row;
    T l[CH];
    const bool use = rb <= K && row < nt;
    constexpr int kTop = 32 - CH;
#pragma unroll
    for (int k = 0; k < CH; ++k)
      l[k] = use && kTop + k < w && (rb < K || kTop + k >= lane) ? col[(int64_t)(kTop + k) * ldd] : T(0);
    if (rb == K) {
#pragma unroll
      for (int k0 = kTop; k0 >= 0; k0 -= CH) {
        if (k0 != kTop) {
#pragma unroll
          for (int k = 0; k < CH; ++k) l[k] = use && k0 + k < w && k0 + k >= lane ? col[(int64_t)(k0 + k) * ldd] : T(0);
        }
#pragma unroll
        for (int k = CH - 1; k >= 0; --k) {
          if (lane == k0 + k) xi *= l[k];
          const T xk = __shfl_sync(kFull, xi, k0 + k);
          if (lane < k0 + k) xi -= l[k] * xk;
        }
      }
      xt[row] = row < nt ? xi : T(0);
    }
    __syncthreads();
    if (rb < K) {
#pragma unroll
      for (int k0 = kTop; k0 >= 0; k0 -= CH) {
        if (k0 != kTop) {
#pragma unroll
          for (int k = 0; k < CH; ++k) l[k] = use && k0 + k < w ? col[(int64_t)(k0 + k) * ldd] : T(0);
        }
        T a0 = T(0), a1 = T(0);
#pragma unroll
        for (int k = 0; k < CH; k += 4) {
          T xv[4];
          load4(xt + 32 * K + k0 + k, xv);
          a0 += l[k] * xv[0];
          a1 += l[k + 1] * xv[1];
          a0 += l[k + 2] * xv[2];
          a1 += l[k + 3] * xv[3];
        }
        xi -= a0 + a1;
      }
    }
  }
  // U12, then the head backward
#pragma unroll 4
  for (int e = tid; e < A.n_u12; e += nthr) tmp[e] = P[d.p_u12 + e] * xt[__ldg(A.w + A.u12c + e)];
  __syncthreads();
  for (int i0 = h > 0 ? (h - 1) / nthr * nthr : -1; i0 >= 0; i0 -= nthr) {
    const int i = i0 + tid;
    const bool in = i < h;
    T xv = T(0);
    int p0 = 0, cnt = 0, u0 = 0, lev = -1;
    T pv[HE], dinv = T(0);
    int pi[HE];
    if (in) {
      p0 = __ldg(d.u11ptr + i);
      cnt = __ldg(d.u11ptr + i + 1) - p0;
      u0 = __ldg(d.uptr + i);
      lev = __ldg(A.w + A.lev_b + i);
      dinv = P[d.p_dinv + i];
    }
#pragma unroll
    for (int e = 0; e < HE; ++e) {
      pv[e] = e < cnt ? P[d.p_u11 + p0 + e] : T(0);
      pi[e] = e < cnt ? __ldg(d.uidx + u0 + e) : 0;
    }
    if (in) {
      const int e1 = __ldg(d.u12off + i + 1);
      T s0 = T(0), s1 = T(0);
      int e = __ldg(d.u12off + i);
      for (; e + 4 <= e1; e += 4) {
        s0 += tmp[e];
        s1 += tmp[e + 1];
        s0 += tmp[e + 2];
        s1 += tmp[e + 3];
      }
      for (; e < e1; ++e) s0 += tmp[e];
      xv = xh[i] - (s0 + s1);
    }
    for (int l = 0; l < d.n_blev; ++l) {
      if (lev == l) {
        T s = T(0);
#pragma unroll
        for (int e = 0; e < HE; ++e)
          if (e < cnt) s += pv[e] * xh[pi[e]];
        for (int e = HE; e < cnt; ++e) s += P[d.p_u11 + p0 + e] * xh[__ldg(d.uidx + u0 + e)];
        xh[i] = (xv - s) * dinv;
      }
      __syncthreads();
    }
  }
  if (h == 0) __syncthreads();
}

// ---- factorisation ----------------------------------------------------------
// Triangular solve of a 32-column block row of the panel: the 32 x 32 block X
// (rows in xk, pitch XP) becomes L_KK^-1 X, L_KK unit lower in ld[k][i].
// One lane per column; pairs of rows share one packed FMA.
__device__ __forceinline__ void trsm_block(float* xk, const float* ld, int lane) {
  f2 x[16];
#pragma unroll
  for (int p = 0; p < 16; ++p) x[p] = pack2(xk[(2 * p) * XP + lane], xk[(2 * p + 1) * XP + lane]);
#pragma unroll
  for (int k = 0; k < 32; ++k) {
    float a, b;
    unpack2(x[k / 2], a, b);
    const float v = -((k & 1) ? b : a);
    if (!(k & 1)) {
      b = fmaf(ld[k * 32 + k + 1], v, b);
      x[k / 2] = pack2(a, b);
    }
    const f2 vv = pack2(v, v);
#pragma unroll
    for (int p = k / 2 + 1; p < 16; ++p) {
      const f2 l = *reinterpret_cast<const f2*>(ld + k * 32 + 2 * p);
      x[p] = fma2(l, vv, x[p]);
    }
  }
#pragma unroll
  for (int p = 0; p < 16; ++p) {
    float a, b;
    unpack2(x[p], a, b);
    xk[(2 * p) * XP + lane] = a;
    xk[(2 * p + 1) * XP + lane] = b;
  }
}
// FP64: 16 columns (c0 ..); lanes 0-15 carry rows 0-15 of a column, lanes
// 16-31 rows 16-31, so every FP64 instruction works for all 32 lanes.
__device__ __forceinline__ void trsm_block16(double* xk, const double* ld, int c0, int lane) {
  const int half = lane >> 4, c = c0 + (lane & 15);
  double x[16];
#pragma unroll
  for (int r = 0; r < 16; ++r) x[r] = xk[(16 * half + r) * XP + c];
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const double v = __shfl_sync(kFull, x[k], lane & 15);
#pragma unroll
    for (int r = 0; r < 16; ++r)
      if (half || r > k) x[r] = fma(-ld[k * 32 + 16 * half + r], v, x[r]);
  }
  if (half) {
#pragma unroll
    for (int k = 0; k < 16; ++k)
#pragma unroll
      for (int r = k + 1; r < 16; ++r) x[r] = fma(-ld[(16 + k) * 32 + 16 + r], x[k], x[r]);
  }
#pragma unroll
  for (int r = 0; r < 16; ++r) xk[(16 * half + r) * XP + c] = x[r];
}

// The head's factors in shared memory (Hv), by dependency levels.
template <class T>
__device__ __forceinline__ void head_program(const Args& A, T* Hv) {
  const int* w = A.w;
  for (int l = 0; l < 2 * A.n_hlev; ++l) {
    const int o1 = __ldg(w + A.hop_ptr + l + 1);
    for (int o = __ldg(w + A.hop_ptr + l) + threadIdx.x; o < o1; o += blockDim.x) {
      const int2 op = __ldg(reinterpret_cast<const int2*>(w + A.hop) + o);
      const int t1 = __ldg(w + A.hop + 2 * o + 3);
      const int dst = op.x & 0xFFFF, piv = (uint32_t)op.x >> 16;
      T v = Hv[dst];
      for (int t = op.y; t < t1; ++t) {
        const uint32_t tm = (uint32_t)__ldg(w + A.hterm + t);
        v -= Hv[tm & 0xFFFF] * Hv[tm >> 16];
      }
      if (!(l & 1)) v = T(1) / v;
      else if (piv != 0xFFFF) v *= Hv[piv];
      Hv[dst] = v;
    }
    __syncthreads();
  }
}

// Panel J of the tail before elimination, in X (column-major, pitch rows):
// its Jacobian entries and the head's Schur complement.  Ends with a barrier.
template <class T>
__device__ __forceinline__ void assemble_panel(const Args& A, int J, T* X, const T* Hv, const T* mbuf) {
  const int* w = A.w;
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nthr >> 5;
  for (int e = tid; e < 32 * A.pitch; e += nthr) X[e] = T(0);
  __syncthreads();
  {
    const int s1 = __ldg(w + A.jg_grp + J + 2);
    for (int e = 32 * __ldg(w + A.jg_grp + J + 1) + tid; e < 32 * s1; e += nthr) {
      const int p = __ldg(w + A.jg_dst + e);
      if (p >= 0) X[p] = mbuf[e];
    }
    const int q1 = __ldg(w + A.jl_grp + J + 2);
    for (int q = __ldg(w + A.jl_grp + J + 1) + tid; q < q1; q += nthr)
      X[__ldg(w + A.jl_dst + q)] = mbuf[32 * A.n_jsl + q];
  }
  __syncthreads();
  const int s1 = __ldg(w + A.tg_grp + J + 1);
  for (int s = __ldg(w + A.tg_grp + J) + warp; s < s1; s += nw) {
    const int e0 = __ldg(w + A.tg_off + s), m = __ldg(w + A.tg_off + s + 1) - e0;
    const int* q = w + A.tg_ent + 32 * e0 + lane;
    const int pos = __ldg(w + A.tg_pos + 32 * s + lane);
    T a = T(0);
    int e = 0;
    for (; e + 4 <= m; e += 4) {
      uint32_t t[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) t[u] = (uint32_t)__ldg(q + 32 * (e + u));
#pragma unroll
      for (int u = 0; u < 4; ++u) a += Hv[t[u] & 0xFFFF] * Hv[t[u] >> 16];
    }
    for (; e < m; ++e) {
      const uint32_t t = (uint32_t)__ldg(q + 32 * e);
      a += Hv[t & 0xFFFF] * Hv[t >> 16];
    }
    if (pos >= 0) X[pos] -= a;
  }
  __syncthreads();
}

// L_KK's columns into ld[k][i] (one warp, 16-byte asynchronous copies).
template <class T>
__device__ __forceinline__ void fetch_diag(const T* D, int ldd, int K, T* ld, int lane) {
  constexpr int PER = 16 / sizeof(T), CPC = 32 / PER;   // chunks per column
#pragma unroll
  for (int u = 0; u < CPC; ++u) {
    const int id = 32 * u + lane, k = id / CPC, i = id % CPC * PER;
    cp16(ld + k * 32 + i, D + (int64_t)(32 * K + k) * ldd + 32 * K + i);
  }
}

// FP32 tail factorisation; TF: the updates on the tensor cores (3xTF32).
template <bool TF>
__device__ void factor_tail(const Args& A, float* D, float* X, float* Xk, float* Ld, const float* Hv, const float* mbuf PHASE_ARG) {
  const int n = A.d.n, nt = n - A.d.head, ldd = A.d.ldd, nb = A.nb, pitch = A.pitch;
  const int lane = threadIdx.x & 31, rb = threadIdx.x >> 5;
  const int row = 32 * rb + lane;
  const bool in = row < nt;
  const int g = lane >> 2, tq = lane & 3;   // fragment coordinates
  for (int J = 0; J < nb; ++J) {
    assemble_panel(A, J, X, Hv, mbuf);
    PHASE_MARK(PH_ASSEMBLE);
    const int w = min(32, nt - 32 * J);
    f2 x[16];             // row `row`, columns in pairs
    float acc[2][4][4];   // TF: the warp's 32 x 32 block as m16n8 fragments
    if (rb < nb) {
      if constexpr (TF) {
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
          for (int nt8 = 0; nt8 < 4; ++nt8)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int r = 32 * rb + mt * 16 + g + (e >> 1) * 8, c = nt8 * 8 + 2 * tq + (e & 1);
              acc[mt][nt8][e] = r < nt ? X[c * pitch + r] : 0.f;
            }
      } else {
#pragma unroll
        for (int p = 0; p < 16; ++p)
          x[p] = in ? pack2(X[2 * p * pitch + row], X[(2 * p + 1) * pitch + row]) : pack2(0.f, 0.f);
      }
    }
    if (J > 0 && rb == 0) fetch_diag(D, ldd, 0, Ld, lane);
    for (int K = 0; K < J; ++K) {
      float* xk = Xk + (K & 1) * 32 * XP;
      float* ld = Ld + (K & 1) * 32 * 32;
      if (rb == K) {
        // this warp's rows are block K: finish their U
        if constexpr (TF) {
#pragma unroll
          for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int nt8 = 0; nt8 < 4; ++nt8)
#pragma unroll
              for (int e = 0; e < 4; ++e)
                xk[(mt * 16 + g + (e >> 1) * 8) * XP + nt8 * 8 + 2 * tq + (e & 1)] = acc[mt][nt8][e];
        } else {
#pragma unroll
          for (int p = 0; p < 16; ++p) *reinterpret_cast<f2*>(xk + lane * XP + 2 * p) = x[p];
        }
        cp_wait();
        __syncwarp();
        trsm_block(xk, ld, lane);
        __syncwarp();
        if (lane < w) {   // column `lane` of the block, 32 consecutive rows
          float* dst = D + (int64_t)(32 * J + lane) * ldd + 32 * K;
#pragma unroll
          for (int r = 0; r < 32; r += 4)
            *reinterpret_cast<float4*>(dst + r) = make_float4(xk[r * XP + lane], xk[(r + 1) * XP + lane],
                                                               xk[(r + 2) * XP + lane], xk[(r + 3) * XP + lane]);
        }
      }
      __syncthreads();
      if (rb == K + 1 && K + 1 < J) fetch_diag(D, ldd, K + 1, Ld + ((K + 1) & 1) * 32 * 32, lane);
      if (rb > K && rb < nb) {
        if constexpr (TF) {
          const float* lcol = D + (int64_t)(32 * K) * ldd + 32 * rb;
#pragma unroll
          for (int k0 = 0; k0 < 32; k0 += 8) {
            uint32_t ah[2][4], al[2][4], bh[4][2], bl[4][2];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const int r = mt * 16 + g + (e & 1) * 8, kk = k0 + tq + (e >> 1) * 4;
                const float v = 32 * rb + r < nt ? -lcol[(int64_t)kk * ldd + r] : 0.f;
                split_tf32(v, ah[mt][e], al[mt][e]);
              }
#pragma unroll
            for (int nt8 = 0; nt8 < 4; ++nt8)
#pragma unroll
              for (int e = 0; e < 2; ++e) split_tf32(xk[(k0 + tq + 4 * e) * XP + nt8 * 8 + g], bh[nt8][e], bl[nt8][e]);
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
              for (int nt8 = 0; nt8 < 4; ++nt8) {
                mma_tf32(acc[mt][nt8], al[mt], bh[nt8]);
                mma_tf32(acc[mt][nt8], ah[mt], bl[nt8]);
                mma_tf32(acc[mt][nt8], ah[mt], bh[nt8]);
              }
          }
        } else {
          const float* lcol = D + (int64_t)(32 * K) * ldd + row;
#pragma unroll
          for (int k0 = 0; k0 < 32; k0 += 16) {
            float l[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) l[k] = in ? -lcol[(int64_t)(k0 + k) * ldd] : 0.f;
#pragma unroll
            for (int k = 0; k < 16; ++k) {
              const f2 ll = pack2(l[k], l[k]);
              const ulonglong2* xr = reinterpret_cast<const ulonglong2*>(xk + (k0 + k) * XP);
#pragma unroll
              for (int c = 0; c < 8; ++c) {
                const ulonglong2 v = xr[c];
                x[2 * c] = fma2(ll, v.x, x[2 * c]);
                x[2 * c + 1] = fma2(ll, v.y, x[2 * c + 1]);
              }
            }
          }
        }
      }
    }
    PHASE_MARK(PH_UPDATE);
    // block J: LU of the diagonal block, then L of the rows below
    float* uj = Xk + (J & 1) * 32 * XP;
    float rv[32];
    if (rb >= J && rb < nb) {
      if constexpr (TF) {
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
          for (int nt8 = 0; nt8 < 4; ++nt8)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int r = 32 * rb + mt * 16 + g + (e >> 1) * 8, c = nt8 * 8 + 2 * tq + (e & 1);
              if (r < nt) X[c * pitch + r] = acc[mt][nt8][e];
            }
        __syncwarp();
#pragma unroll
        for (int b = 0; b < 32; ++b) rv[b] = in ? X[b * pitch + row] : 0.f;
      } else {
#pragma unroll
        for (int p = 0; p < 16; ++p) unpack2(x[p], rv[2 * p], rv[2 * p + 1]);
      }
    }
    if (rb == J) {
      if (lane >= w) {   // rows and columns past the last block's edge: the identity
#pragma unroll
        for (int b = 0; b < 32; ++b) rv[b] = b == lane ? 1.f : 0.f;
      }
#pragma unroll
      for (int kk = 0; kk < 32; ++kk) {
        const float inv = 1.f / __shfl_sync(kFull, rv[kk], kk);
        const float l = rv[kk] * inv;
        const bool below = lane > kk;
        if (below) rv[kk] = l;
#pragma unroll
        for (int b = kk + 1; b < 32; ++b) {
          const float pb = __shfl_sync(kFull, rv[b], kk);
          if (below) rv[b] -= l * pb;
        }
        if (lane == kk) rv[kk] = inv;
      }
#pragma unroll
      for (int b = 0; b < 32; ++b) uj[lane * XP + b] = rv[b];
      float* dst = D + (int64_t)(32 * J) * ldd + row;
#pragma unroll
      for (int b = 0; b < 32; ++b)
        if (in && b < w) dst[(int64_t)b * ldd] = rv[b];
    }
    __syncthreads();
    if (rb > J && rb < nb) {   // then w == 32
#pragma unroll
      for (int kk = 0; kk < 32; ++kk) {
        const float l = rv[kk] * uj[kk * XP + kk];   // inverse pivot
        rv[kk] = l;
#pragma unroll
        for (int b = kk + 1; b < 32; ++b) rv[b] -= l * uj[kk * XP + b];
      }
      float* dst = D + (int64_t)(32 * J) * ldd + row;
#pragma unroll
      for (int b = 0; b < 32; ++b)
        if (in) dst[(int64_t)b * ldd] = rv[b];
    }
    __syncthreads();
    PHASE_MARK(PH_PANEL);
  }
}

// FP64 tail factorisation: two warps per 32 rows, 16 columns each, so that
// the four FP64 pipes of the SM get even shares.
__device__ void factor_tail(const Args& A, double* D, double* X, double* Xk, double* Ld, const double* Hv, const double* mbuf PHASE_ARG) {
  const int n = A.d.n, nt = n - A.d.head, ldd = A.d.ldd, nb = A.nb, pitch = A.pitch;
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  const int cs = wi >= nb, rb = wi < 2 * nb ? wi - cs * nb : nb, c0 = 16 * cs;
  const int row = 32 * rb + lane;
  const bool in = row < nt;
  for (int J = 0; J < nb; ++J) {
    assemble_panel(A, J, X, Hv, mbuf);
    PHASE_MARK(PH_ASSEMBLE);
    const int w = min(32, nt - 32 * J);
    double rv[16];
#pragma unroll
    for (int b = 0; b < 16; ++b) rv[b] = in ? X[(c0 + b) * pitch + row] : 0.0;
    if (J > 0 && rb == 0) fetch_diag(D, ldd, 0, Ld, lane);
    for (int K = 0; K < J; ++K) {
      double* xk = Xk + (K & 1) * 32 * XP;
      double* ld = Ld + (K & 1) * 32 * 32;
      if (rb == K) {
#pragma unroll
        for (int b = 0; b < 16; ++b) xk[lane * XP + c0 + b] = rv[b];
        cp_wait();
        __syncwarp();
        trsm_block16(xk, ld, c0, lane);
        __syncwarp();
#pragma unroll
        for (int b = 0; b < 16; ++b)
          if (c0 + b < w) D[(int64_t)(32 * J + c0 + b) * ldd + row] = xk[lane * XP + c0 + b];
      }
      __syncthreads();
      if (rb == K + 1 && K + 1 < J) fetch_diag(D, ldd, K + 1, Ld + ((K + 1) & 1) * 32 * 32, lane);
      if (rb > K && rb < nb) {
        const double* lcol = D + (int64_t)(32 * K) * ldd + row;
#pragma unroll
        for (int k0 = 0; k0 < 32; k0 += 8) {
          double l[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) l[k] = in ? -lcol[(int64_t)(k0 + k) * ldd] : 0.0;
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const double2* xr = reinterpret_cast<const double2*>(xk + (k0 + k) * XP + c0);
#pragma unroll
            for (int b = 0; b < 8; ++b) {
              const double2 v = xr[b];
              rv[2 * b] = fma(l[k], v.x, rv[2 * b]);
              rv[2 * b + 1] = fma(l[k], v.y, rv[2 * b + 1]);
            }
          }
        }
      }
    }
    PHASE_MARK(PH_UPDATE);
    // block J in four stages: LU of its first 16 columns; L of the rows below
    // there and U12 / LU of the second 16 columns; L of the rows below
    double* uj = Xk + (J & 1) * 32 * XP;
    if (rb == J && lane >= w) {
#pragma unroll
      for (int b = 0; b < 16; ++b) rv[b] = c0 + b == lane ? 1.0 : 0.0;
    }
    auto lu16 = [&](int r0) {   // pivots in lanes r0 .. r0 + 15
#pragma unroll
      for (int kk = 0; kk < 16; ++kk) {
        const double inv = 1.0 / __shfl_sync(kFull, rv[kk], r0 + kk);
        const double l = rv[kk] * inv;
        const bool below = lane > r0 + kk;
        if (below) rv[kk] = l;
#pragma unroll
        for (int b = kk + 1; b < 16; ++b) {
          const double pb = __shfl_sync(kFull, rv[b], r0 + kk);
          if (below) rv[b] -= l * pb;
        }
        if (lane == r0 + kk) rv[kk] = inv;
      }
    };
    auto lrow16 = [&](int r0) {   // l U = a for this thread's row, U at uj rows and columns r0 ..
#pragma unroll
      for (int kk = 0; kk < 16; ++kk) {
        const double l = rv[kk] * uj[(r0 + kk) * XP + r0 + kk];
        rv[kk] = l;
#pragma unroll
        for (int b = kk + 1; b < 16; ++b) rv[b] -= l * uj[(r0 + kk) * XP + r0 + b];
      }
    };
    auto store = [&]() {
#pragma unroll
      for (int b = 0; b < 16; ++b)
        if (in && c0 + b < w) D[(int64_t)(32 * J + c0 + b) * ldd + row] = rv[b];
    };
    if (rb == J && cs == 0) {
      lu16(0);
#pragma unroll
      for (int b = 0; b < 16; ++b) uj[lane * XP + b] = rv[b];
      store();
    }
    __syncthreads();
    if (cs == 0 && rb > J && rb < nb) {
      lrow16(0);
#pragma unroll
      for (int b = 0; b < 16; ++b)
        if (in) X[b * pitch + row] = rv[b];
      store();
    }
    if (rb == J && cs == 1) {
#pragma unroll
      for (int kk = 0; kk < 16; ++kk) {
        const double l = lane > kk ? uj[lane * XP + kk] : 0.0;
#pragma unroll
        for (int b = 0; b < 16; ++b) rv[b] -= l * __shfl_sync(kFull, rv[b], kk);
      }
      lu16(16);
#pragma unroll
      for (int b = 0; b < 16; ++b) uj[lane * XP + 16 + b] = rv[b];
      store();
    }
    __syncthreads();
    if (cs == 1 && rb > J && rb < nb) {
#pragma unroll
      for (int kk = 0; kk < 16; ++kk) {
        const double l = in ? X[kk * pitch + row] : 0.0;
#pragma unroll
        for (int b = 0; b < 16; ++b) rv[b] -= l * uj[kk * XP + 16 + b];
      }
      lrow16(16);
      store();
    }
    __syncthreads();
    PHASE_MARK(PH_PANEL);
  }
}

template <bool TF>
__device__ __forceinline__ void factor(const Args& A, float* D, float* X, float* Xk, float* Ld, const float* Hv, const float* mbuf PHASE_ARG) {
  factor_tail<TF>(A, D, X, Xk, Ld, Hv, mbuf PHASE_PASS);
}
template <bool TF>
__device__ __forceinline__ void factor(const Args& A, double* D, double* X, double* Xk, double* Ld, const double* Hv, const double* mbuf PHASE_ARG) {
  factor_tail(A, D, X, Xk, Ld, Hv, mbuf PHASE_PASS);
}

// The cell being worked on: its shared vectors and global buffers.
template <class T>
struct Cell {
  CellS* S;
  double *red, *yp, *ps, *ws, *wf, *ys, *fs, *tab, *part;
  T *xh, *xt, *tmp;
  double *kc, *hist, *eprev;   // this CTA's global scratch
  T* mbuf;
  T* P;                        // packed factors
  int64_t c, oc;               // slot and cell
  int hn;                      // stride of a history point in scratch
  double nH, Av, chi;
};

// Jacobian at the predicted state, M = I - gamma J and its packed factors.
// y (= predicted state) is restored at the end.
template <class T, bool TF>
__device__ void cell_refresh(const Args& A, Cell<T>& q, unsigned char* sm PHASE_ARG) {
  const Dev& d = A.d;
  const int n = d.n, n_r = d.n_r, tid = threadIdx.x, nthr = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nw = nthr >> 5;
  const int* w = A.w;
  double* dR = reinterpret_cast<double*>(sm + A.p.o_dr);
  float* wsf = reinterpret_cast<float*>(sm + A.p.o_wsf);
  float* wif = reinterpret_cast<float*>(sm + A.p.o_wif);
  const double gamma = q.S->gam;
  // -gamma dR_j/dx for both reactant slots
  for (int j = tid; j < n_r; j += nthr) {
    const int2 rc = __ldg(d.reac + j);
    const double kv = -gamma * q.kc[j];
    dR[2 * j] = rc.y >= 0 ? kv * q.yp[rc.y] : kv;
    dR[2 * j + 1] = rc.y >= 0 ? kv * q.yp[rc.x] : 0.0;
  }
  if (tid == 0) dR[2 * n_r] = 0.0;
  for (int s = tid; s < n; s += nthr) {
    const double wv = q.ws[s];
    q.wf[s] = wv;
    if (d.mixed) {
      wsf[s] = (float)wv;
      wif[s] = (float)(1.0 / wv);
    }
  }
  __syncthreads();
  auto m_value = [&](int rc, double acc) {   // M (W M W^-1 in FP32) at (row species, column species)
    const int i = rc & 0xFFFF, l = (uint32_t)rc >> 16;
    if (i == l) acc += 1.0;
    return sizeof(T) == 4 ? T((float)acc * (wsf[i] * wif[l])) : T(acc);
  };
  for (int s = warp; s < A.n_jsl; s += nw) {
    const int e0 = __ldg(w + A.jg_off + s), m = __ldg(w + A.jg_off + s + 1) - e0;
    const int* p = w + A.jg_ent + 32 * e0 + lane;
    const int rc = __ldg(w + A.jg_rc + 32 * s + lane);
    double a = 0.0;
    if (m > 0) {
      const int w0 = __ldg(p);
      a = flip(dR[w0 & 0x7FFFFFFF], w0);
    }
    int e = 1;
    for (; e + 4 <= m; e += 4) {
      int t[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) t[u] = __ldg(p + 32 * (e + u));
#pragma unroll
      for (int u = 0; u < 4; ++u) a += flip(dR[t[u] & 0x7FFFFFFF], t[u]);
    }
    for (; e < m; ++e) {
      const int w0 = __ldg(p + 32 * e);
      a += flip(dR[w0 & 0x7FFFFFFF], w0);
    }
    q.mbuf[32 * s + lane] = m_value(rc, a);
  }
  for (int s = nw - 1 - warp; s < A.n_jl; s += nw) {   // long entries
    const int e1 = __ldg(w + A.jl_ptr + s + 1);
    double a = 0.0;
    for (int e = __ldg(w + A.jl_ptr + s) + lane; e < e1; e += 32) {
      const int w0 = __ldg(w + A.jl_ent + e);
      a += flip(dR[w0 & 0x7FFFFFFF], w0);
    }
    a = warp_sum(a);
    if (lane == 0) q.mbuf[32 * A.n_jsl + s] = m_value(__ldg(w + A.jl_rc + s), a);
  }
  if (d.therm) {
    // gamma_J sum_j dn_j dR_j/dx_l per species, kept in the border's row
    __syncthreads();
    for (int j = tid; j < n_r; j += nthr) {
      const double dn = -__ldg(d.th_dn + j);
      dR[2 * j] *= dn;
      dR[2 * j + 1] *= dn;
    }
    __syncthreads();
    row_sums(w, A.n_vsl, A.vp_off, A.vp_ent, A.vp_dst, A.vrow_ptr, A.n_vlong, A.vrow_long, dR,
             reinterpret_cast<double*>(sm + A.p.o_vp), d.bgv + q.oc * d.bpad, n);
  }
  __syncthreads();
  PHASE_MARK(PH_JAC);
  T* Hv = reinterpret_cast<T*>(sm + A.p.o_hv);
  for (int e = tid; e <= d.p_d; e += nthr) Hv[e] = T(0);
  __syncthreads();
  {
    const int s1 = __ldg(w + A.jg_grp + 1);
    for (int e = tid; e < 32 * s1; e += nthr) {
      const int p = __ldg(w + A.jg_dst + e);
      if (p >= 0) Hv[p] = q.mbuf[e];
    }
    const int q1 = __ldg(w + A.jl_grp + 1);
    for (int e = tid; e < q1; e += nthr) Hv[__ldg(w + A.jl_dst + e)] = q.mbuf[32 * A.n_jsl + e];
  }
  __syncthreads();
  head_program(A, Hv);
  for (int e = tid; e < d.p_d; e += nthr) q.P[e] = Hv[e];
  PHASE_MARK(PH_HEAD);
  factor<TF>(A, q.P + d.p_d, reinterpret_cast<T*>(sm + A.p.o_x), reinterpret_cast<T*>(sm + A.p.o_xk),
             reinterpret_cast<T*>(sm + A.p.o_ld), Hv, q.mbuf PHASE_PASS);
  for (int s = tid; s < n; s += nthr) q.ys[s] = q.yp[s];
  if (tid == 0) {
    CellS& S = *q.S;
    S.gam_J = gamma;
    S.j_age = 0;
    S.crate = 1.0;
    S.flags &= ~F_NEED_J;
    S.jac_evals += 1;
  }
  __syncthreads();
}

// x := M^-1 b with b given by species in bs (scaled by wf when mixed); the
// solution by species through get(s).
template <class T>
__device__ __forceinline__ T x_get(const Args& A, const Cell<T>& q, int s) {
  const int p = __ldg(A.d.iperm + s);
  return p < A.d.head ? q.xh[p] : q.xt[p - A.d.head];
}
template <class T>
__device__ __forceinline__ void x_put(const Args& A, const Cell<T>& q, int s, double b) {
  if (A.d.mixed) b *= q.wf[s];
  const int p = __ldg(A.d.iperm + s);
  if (p < A.d.head) q.xh[p] = T(b);
  else q.xt[p - A.d.head] = T(b);
}

// Temperature border of a refreshed Newton matrix (T eliminated last): with
// u = dF/dT, v = d f_t/dx and w = d f_t/dT at the predicted state,
// z = M^-1 (-gJ u) and s = 1 - gJ w + gJ v.z; a residual (r, r_T) then has the
// correction (a0 - z b, b), a0 = M^-1 r, b = (r_T + gJ v.a0) / s.
template <class T>
__device__ void cell_border(const Args& A, Cell<T>& q) {
  const Dev& d = A.d;
  const int n = d.n, n_r = d.n_r, t = d.t_idx, tid = threadIdx.x, nthr = blockDim.x;
  const double Tc = q.yp[t], it = 1.0 / Tc;
  double F = 0.0, U = 0.0;
  for (int j = tid; j < n_r; j += nthr) {
    const int2 rc = __ldg(d.reac + j);
    double R = q.kc[j] * q.yp[rc.x];
    if (rc.y >= 0) R *= q.yp[rc.y];
    const RatePar p = d.rpar[j];
    const int cls = (int)p.w;
    const double g = (cls == SM_TWO_BODY || cls == SM_DISS_RECOMB) ? (p.y + p.z * it) * it : 0.0;   // d ln k'/dT
    const double dn = __ldg(d.th_dn + j), Rg = R * g;
    F = fma(dn, R, F);
    U = fma(dn, Rg, U);
    q.tab[j] = Rg;
  }
  if (tid == 0) q.tab[n_r] = 0.0;
  __syncthreads();
  row_sums(A.w, A.n_rsl, A.rp_off, A.rp_ent, A.rp_dst, A.row_ptr, A.n_rlong, A.row_long, q.tab, q.part, q.fs, n);
  F = cta_sum(F, q.red, 0);
  U = cta_sum(U, q.red, 1);
  double xt = 0.0, line = 0.0, dline = 0.0;
  for (int s = tid; s < n; s += nthr)
    if (s != t) xt += q.yp[s];
  for (int e = tid; e < d.n_cool; e += nthr) {
    const int i = __ldg(d.th_cool + e);
    const double cl = d.th_L[i] * exp(-d.th_E[i] * it);
    line = fma(q.yp[i], cl, line);
    dline = fma(q.yp[i] * cl, d.th_E[i] * it * it, dline);
  }
  xt = cta_sum(xt, q.red, 2);
  line = cta_sum(line, q.red, 3);
  __syncthreads();
  dline = cta_sum(dline, q.red, 0);
  const double gJ = q.S->gam_J;
  if (tid == 0) {
    const double i15x = 1.0 / (1.5 * xt);
    const double fT = (d.th_heat - q.nH * line - d.th_lam * q.nH * (Tc - d.th_Td) - 1.5 * Tc * F) * i15x;
    const double w = (-q.nH * dline - d.th_lam * q.nH - 1.5 * F - 1.5 * Tc * U) * i15x;
    q.red[96] = i15x;
    q.red[97] = fT / xt;
    q.red[98] = w;
  }
  for (int s = tid; s < n; s += nthr) x_put(A, q, s, s == t ? 0.0 : -gJ * q.fs[s]);
  cell_solve<T>(A, q.P, q.xh, q.xt, q.tmp);
  const double i15x = q.red[96], fTx = q.red[97], w = q.red[98];
  double* bz = d.bz + q.oc * d.bpad;
  double* bgv = d.bgv + q.oc * d.bpad;
  double vz = 0.0;
  for (int s = tid; s < n; s += nthr) {
    double z = 0.0, gv = 0.0;
    if (s != t) {
      z = (double)x_get(A, q, s);
      if (d.mixed) z /= q.wf[s];
      const double cl = d.th_L[s] > 0.0 ? d.th_L[s] * exp(-d.th_E[s] * it) : 0.0;
      gv = (gJ * (-q.nH * cl) - 1.5 * Tc * bgv[s]) * i15x - gJ * fTx;
    }
    bz[s] = z;
    bgv[s] = gv;
    vz = fma(gv, z, vz);
  }
  vz = cta_sum(vz, q.red, 1);
  if (tid == 0) d.bs[q.oc] = 1.0 - gJ * w + vz;
  for (int s = tid; s < n; s += nthr) q.ys[s] = q.yp[s];
  __syncthreads();
}

// One BDF attempt of the cell; returns false when the cell stopped before it.
template <class T, bool TF>
__device__ bool cell_attempt(const Args& A, Cell<T>& q, unsigned char* sm PHASE_ARG) {
  const Dev& d = A.d;
  CellS& S = *q.S;
  const int n = d.n, tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5;
  long long t0 = 0;
  auto class_begin = [&](int kind) {
    if (A.timing_kind == kind && tid == 0) t0 = clock64();
  };
  auto class_end = [&](int kind) {
    if (A.timing_kind == kind && tid == 0) {
      atomicAdd(A.timing, (double)(clock64() - t0));
      atomicAdd(A.timing + 1, 1.0);
    }
  };
  __syncthreads();   // every thread has taken the last attempt's outcome from S
  // ---- predict
  class_begin(SM_TIME_PREDICT);
  if (warp < 2) {
    // both warps derive the step from the same scalars; warp 0 forms the
    // predictor's weights (a point per lane), warp 1 the BDF coefficients
    int state = 3;
    const double t = S.t;
    double h = S.h;
    const int qq = S.q, nh = S.nh;
    const bool fin = t + h >= d.t_end;
    if (fin) h = d.t_end - t;
    const double tnew = fin ? d.t_end : t + h;
    if (S.steps >= d.max_steps) state = 1;
    else if (tnew == t || !(h > 0.0)) state = 2;
    if (warp == 0) {
      if (state == 3 && nh > 1 && lane <= qq) {
        double num = 1.0, den = 1.0;
        const double ti = S.tn[lane];
        for (int j = 0; j <= qq; ++j)
          if (j != lane) {
            num *= tnew - S.tn[j];
            den *= ti - S.tn[j];
          }
        S.wts[lane] = num / den;
      }
    } else {
      double al = 0.0;
      if (state == 3 && lane >= 1 && lane <= qq) {
        const double ti = S.tn[lane - 1];
        double num = 1.0, den = ti - tnew;
        for (int m = 1; m <= qq; ++m)
          if (m != lane) {
            num *= tnew - S.tn[m - 1];
            den *= ti - S.tn[m - 1];
          }
        al = h * num / den;
      }
      // al_0 = h sum 1 / (tau_0 - tau_i)
      double r = state == 3 && lane >= 1 && lane <= qq ? 1.0 / (tnew - S.tn[lane - 1]) : 0.0;
      double sum = 0.0;
      for (int i = 1; i <= QMAX; ++i) {
        const double v = __shfl_sync(kFull, r, i);
        if (i <= qq) sum += v;
      }
      if (lane == 0) al = h * sum;
      if (lane <= QMAX) S.alpha[lane] = al;
      if (lane == 0) {
        int fl = S.flags & ~(F_CONV | F_FAILED | F_REFRESH | F_FINAL | F_NEWTON | F_ATTEMPT);
        S.state = state;
        if (state == 3) {
          const double gamma = h / al;
          const bool refresh = (fl & F_NEED_J) || S.j_age >= d.j_age_max || fabs(gamma / S.gam_J - 1.0) > d.gamma_tol;
          fl |= F_NEWTON | F_ATTEMPT | (fin ? F_FINAL : 0) | (refresh ? F_REFRESH : 0);
          S.gam = gamma;
          S.tnew = tnew;
          S.err = h;   // the attempt's step; committed after the barrier
          S.m_it = 0;
          S.dprev = 0.0;
        } else {
          S.status = state == 1 ? SM_CELL_MAXSTEPS : SM_CELL_HMIN;
        }
        S.flags = fl;
      }
    }
  }
  __syncthreads();
  if (S.state != 3) return false;
  const double h = S.err, tnew = S.tnew;
  const int qo = S.q, nh = S.nh;
  const bool refresh = (S.flags & F_REFRESH) != 0;
  {
    double wt[QMAX + 1], al[QMAX + 1];
    const double* Yp[QMAX + 1];
    const bool euler = nh == 1;
#pragma unroll
    for (int i = 0; i <= QMAX; ++i) {
      wt[i] = !euler && i <= qo ? S.wts[i] : 0.0;
      al[i] = S.alpha[i];
      int slot = S.base + i;
      if (slot > QMAX) slot -= QMAX + 1;
      Yp[i] = q.hist + (int64_t)slot * q.hn;
    }
    for (int s = tid; s < n; s += nthr) {
      const double y0 = Yp[0][s];
      double yp = euler ? y0 + h * d.f0[(int64_t)s * d.ld + q.c] : wt[0] * y0, pv = 0.0;
#pragma unroll
      for (int i = 1; i <= QMAX; ++i) {
        if (i > qo) break;
        const double yi = i < nh ? Yp[i][s] : 0.0;
        if (!euler) yp += wt[i] * yi;
      }
#pragma unroll
      for (int i = 1; i <= QMAX; ++i) {
        if (i > qo) break;
        pv += al[i] * (i == 1 ? y0 : Yp[i - 1][s]);
      }
      q.yp[s] = yp;
      q.ys[s] = yp;
      q.ps[s] = pv;
      q.ws[s] = 1.0 / (d.rtol * fabs(y0) + d.atol);
    }
  }
  if (tid == 0) S.h = h;
  __syncthreads();
  class_end(SM_TIME_PREDICT);
  PHASE_MARK(PH_PREDICT);
  if (d.therm) cell_th_rates(A, q.kc, q.yp[d.t_idx], q.nH, q.Av, q.chi, false);
  // ---- Jacobian and factors
  if (refresh) {
    class_begin(SM_TIME_REFRESH);
    cell_refresh<T, TF>(A, q, sm PHASE_PASS);
    if (d.therm) cell_border<T>(A, q);
    class_end(SM_TIME_REFRESH);
  }
  // ---- Newton rounds
  const double a0 = S.alpha[0], inv_a0 = 1.0 / a0;
  const double gam = S.gam, gJ = S.gam_J;
  const double scale = gam != gJ ? 2.0 / (1.0 + gam / gJ) : 1.0;
  for (int m = 0; m < d.newton_max; ++m) {
    class_begin(SM_TIME_RHS);
    if (d.therm && m > 0) cell_th_rates(A, q.kc, q.ys[d.t_idx], q.nH, q.Av, q.chi, false);
    cell_rhs(A, q.kc, q.ys, q.tab, q.part, q.fs PHASE_PASS);
    if (d.therm) cell_energy(A, q.ys, q.fs, q.nH, q.red);
    class_end(SM_TIME_RHS);
    class_begin(SM_TIME_SOLVE);
    for (int s = tid; s < n; s += nthr) {
      const double b = -(a0 * q.ys[s] + q.ps[s] - h * q.fs[s]) * inv_a0;
      if (s == d.t_idx) q.red[99] = b;
      x_put(A, q, s, b);
    }
    cell_solve<T>(A, q.P, q.xh, q.xt, q.tmp);
    double bT = 0.0;
    const double* bz = nullptr;
    if (d.therm) {
      const double* bgv = d.bgv + q.oc * d.bpad;
      bz = d.bz + q.oc * d.bpad;
      double dot = 0.0;
      for (int s = tid; s < n; s += nthr) {
        if (s == d.t_idx) continue;
        double a = (double)x_get(A, q, s);
        if (d.mixed) a /= q.wf[s];
        dot = fma(bgv[s], a, dot);
      }
      dot = cta_sum(dot, q.red, 0);
      if (tid == 0) q.red[100] = (q.red[99] + dot) / d.bs[q.oc];
      __syncthreads();
      bT = q.red[100];
    }
    double acc = 0.0;
    for (int s = tid; s < n; s += nthr) {
      double del = (double)x_get(A, q, s);
      if (d.mixed) del /= q.wf[s];
      if (bz) del = s == d.t_idx ? bT : fma(-bz[s], bT, del);
      del *= scale;
      q.ys[s] += del;
      const double v = del * q.ws[s];
      acc += v * v;
    }
    acc = cta_sum(acc, q.red, 1);
    if (tid == 0) {
      const double dn = sqrt(acc / n);
      const int mi = S.m_it;
      double crate = S.crate;
      const double dp = S.dprev;
      bool conv = false, fail = false;
      if (!isfinite(dn)) {
        fail = true;
      } else {
        if (mi > 0) crate = fmax(0.3 * crate, dn / dp);
        if (dn * fmin(1.0, crate) <= d.newton_tol) conv = true;
        else if (mi > 0 && dn > 2.0 * dp) fail = true;
        else if (mi + 1 >= d.newton_max) fail = true;
      }
      S.crate = crate;
      S.dprev = dn;
      S.m_it = mi + 1;
      S.newton_iters += 1;
      if (conv || fail) S.flags = (S.flags & ~F_NEWTON) | (conv ? F_CONV : F_FAILED);
    }
    __syncthreads();
    class_end(SM_TIME_SOLVE);
    PHASE_MARK(PH_SOLVE);
    if (!(S.flags & F_NEWTON)) break;
  }
  // ---- finish: error test, step / order selection, history
  class_begin(SM_TIME_FINISH);
  const bool work = !(S.flags & F_FAILED);
  double acc = 0.0;
  if (work)
    for (int s = tid; s < n; s += nthr) {
      const double v = (q.ys[s] - q.yp[s]) * q.ws[s];
      acc += v * v;
    }
  acc = cta_sum(acc, q.red, 0);
  if (warp == 0) {
    const double err = work ? (nh >= qo + 1 ? h / (tnew - S.tn[qo]) : 1.0 / (qo + 1)) * sqrt(acc / n) : 0.0;
    const bool accepted = work && isfinite(err) && err <= 1.0;
    const int naq = accepted ? S.n_at_q + 1 : 0;
    const bool lo = accepted && naq >= qo + 1 && qo > 1;
    const bool hi = accepted && naq >= qo + 1 && qo < d.q_max && (S.flags & F_HAS_EPREV) && nh + 1 >= qo + 2;
    if (lo && lane < qo) {   // weights of the order q - 1 predictor, a point per lane
      double num = 1.0, den = 1.0;
      const double ti = S.tn[lane];
      for (int j = 0; j < qo; ++j)
        if (j != lane) {
          num *= tnew - S.tn[j];
          den *= ti - S.tn[j];
        }
      S.wts[lane] = num / den;
    }
    if (lane == 0) {
      S.err = err;
      S.state = accepted;
      S.lo = lo;
      S.hi = hi;
    }
  }
  __syncthreads();
  const bool accepted = S.state != 0, lo = S.lo != 0, hi = S.hi != 0;
  double acc_lo = 0.0, acc_hi = 0.0;
  if (lo || hi) {
    for (int s = tid; s < n; s += nthr) {
      const double yv = q.ys[s], wv = q.ws[s];
      if (lo) {
        double p = 0.0;
        for (int i = 0; i < qo; ++i) {
          int slot = S.base + i;
          if (slot > QMAX) slot -= QMAX + 1;
          p += S.wts[i] * q.hist[(int64_t)slot * q.hn + s];
        }
        const double v = (yv - p) * wv;
        acc_lo += v * v;
      }
      if (hi) {
        const double v = ((yv - q.yp[s]) - q.eprev[s]) * wv;
        acc_hi += v * v;
      }
    }
    acc_lo = cta_sum(acc_lo, q.red, 1);
    acc_hi = cta_sum(acc_hi, q.red, 2);
  }
  if (warp == 0 && accepted) {
    // step factors of the three candidate orders, one per lane
    double eta = 0.0;
    if (lane == 0) eta = 0.9 * pow(fmax(S.err, 1e-10), -1.0 / (qo + 1));
    if (lane == 1 && lo) eta = 0.8 * pow(fmax(h / (tnew - S.tn[qo - 1]) * sqrt(acc_lo / n), 1e-10), -1.0 / qo);
    if (lane == 2 && hi) eta = 0.7 * pow(fmax(sqrt(acc_hi / n) / (qo + 2), 1e-10), -1.0 / (qo + 2));
    const double e1 = __shfl_sync(kFull, eta, 1), e2 = __shfl_sync(kFull, eta, 2);
    if (lane == 0) {
      int bq = qo;
      if (lo && e1 > eta) {
        eta = e1;
        bq = qo - 1;
      }
      if (hi && e2 > eta) {
        eta = e2;
        bq = qo + 1;
      }
      S.eta[0] = eta;
      S.best_q = bq;
    }
  }
  __syncthreads();
  const bool keep_e = S.best_q == qo;
  if (accepted) {
    // the newest point takes the slot in front of the ring
    const int slot = S.base == 0 ? QMAX : S.base - 1;
    double* Y0 = q.hist + (int64_t)slot * q.hn;
    for (int s = tid; s < n; s += nthr) {
      const double yv = q.ys[s];
      if (keep_e) q.eprev[s] = yv - q.yp[s];
      Y0[s] = yv;
    }
  }
  __syncthreads();
  if (tid == 0) {
    int fl = S.flags & ~F_ATTEMPT;
    if (fl & F_FAILED) {
      S.conv_fails += 1;
      S.ccf += 1;
      if (S.ccf >= d.max_conv_fails) {
        S.status = SM_CELL_CONV;
      } else {
        if (fl & F_REFRESH) S.h = h * 0.25;
        fl |= F_NEED_J | F_REJECTED;
      }
    } else if (!isfinite(S.err)) {
      S.status = SM_CELL_NAN;
    } else if (!accepted) {
      S.rejects += 1;
      S.crej += 1;
      const double eta = fmax(0.2, 0.9 * pow(S.err, -1.0 / (qo + 1)));
      if (S.crej >= 3 && qo > 1) {
        S.q = 1;
        S.n_at_q = 0;
        fl &= ~F_HAS_EPREV;
      }
      S.h = h * eta;
      fl |= F_REJECTED;
    } else {
      const int nh_new = min(nh + 1, d.q_max + 1);
      for (int i = nh_new - 1; i >= 1; --i) S.tn[i] = S.tn[i - 1];
      S.tn[0] = tnew;
      S.base = S.base == 0 ? QMAX : S.base - 1;
      S.nh = nh_new;
      S.t = tnew;
      S.steps += 1;
      if (d.record && S.steps <= d.record) {
        const int64_t o = (int64_t)(S.steps - 1) * d.ld + q.c;
        d.log_t[o] = tnew;
        d.log_h[o] = h;
        d.log_q[o] = qo;
      }
      S.j_age += 1;
      S.crej = 0;
      S.ccf = 0;
      if (!keep_e) {
        S.q = S.best_q;
        S.n_at_q = 0;
        fl &= ~F_HAS_EPREV;
      } else {
        S.n_at_q += 1;
        fl |= F_HAS_EPREV;
      }
      double eta = fmin(S.eta[0], (fl & F_REJECTED) ? 1.0 : d.eta_max);
      eta = fmax(eta, 0.2);
      if (eta >= 1.0 && eta < d.eta_keep) eta = 1.0;
      S.h = h * eta;
      fl &= ~F_REJECTED;
      if (fl & F_FINAL) S.status = SM_CELL_OK;
    }
    S.flags = fl;
  }
  __syncthreads();
  if (d.record && accepted && S.steps <= d.record && S.steps % kCkpt == 0) {
    // the step history after every kCkpt-th accepted step
    const int kk = S.steps / kCkpt, nhc = S.nh;
    const int64_t vs = (int64_t)n * d.ld;
    double* dst = d.ck_Y + (int64_t)kk * (QMAX + 1) * vs;
    for (int i = 0; i < nhc; ++i) {
      int slot = S.base + i;
      if (slot > QMAX) slot -= QMAX + 1;
      for (int s = tid; s < n; s += nthr) dst[i * vs + (int64_t)s * d.ld + q.c] = q.hist[(int64_t)slot * q.hn + s];
      if (tid == 0) d.ck_t[((int64_t)kk * (QMAX + 1) + i) * d.ld + q.c] = S.tn[i];
    }
    if (tid == 0) d.ck_nh[(int64_t)kk * d.ld + q.c] = nhc;
  }
  class_end(SM_TIME_FINISH);
  PHASE_MARK(PH_FINISH);
  return S.status == SM_CELL_RUNNING;
}

// Shared-memory views and this CTA's global scratch.
template <class T>
__device__ __forceinline__ void cell_views(const Args& A, unsigned char* sm, Cell<T>& q) {
  const CellPlan& p = A.p;
  q.S = reinterpret_cast<CellS*>(sm + p.o_s);
  q.red = reinterpret_cast<double*>(sm + p.o_red);
  q.yp = reinterpret_cast<double*>(sm + p.o_yp);
  q.ps = reinterpret_cast<double*>(sm + p.o_ps);
  q.ws = reinterpret_cast<double*>(sm + p.o_ws);
  q.wf = reinterpret_cast<double*>(sm + p.o_wf);
  q.ys = reinterpret_cast<double*>(sm + p.o_ys);
  q.fs = reinterpret_cast<double*>(sm + p.o_fs);
  q.tab = reinterpret_cast<double*>(sm + p.o_r);
  q.part = reinterpret_cast<double*>(sm + p.o_part);
  q.xh = reinterpret_cast<T*>(sm + p.o_xh);
  q.xt = reinterpret_cast<T*>(sm + p.o_xt);
  q.tmp = reinterpret_cast<T*>(sm + p.o_tmp);
  q.hn = (A.d.n + 31) / 32 * 32;
  q.kc = A.scratch + (int64_t)blockIdx.x * p.scratch;
  q.hist = q.kc + (A.d.n_r + 31) / 32 * 32;
  q.eprev = q.hist + (int64_t)(QMAX + 1) * q.hn;
  q.mbuf = reinterpret_cast<T*>(q.eprev + q.hn);
}

// Rate coefficients of the cell into this CTA's scratch (cell-major).
template <class T>
__device__ __forceinline__ void cell_conditions(const Args& A, Cell<T>& q) {
  const Dev& d = A.d;
  if (d.therm) {
    q.nH = d.c_nH[q.oc];
    q.Av = d.c_Av[q.oc];
    q.chi = d.c_chi[q.oc];
  } else {
    for (int j = threadIdx.x; j < d.n_r; j += blockDim.x) q.kc[j] = A.k[(int64_t)j * A.ldk + q.oc];
  }
}

// The 704-thread bound caps a thread at 88 registers, so that two FP32 CTAs of
// 352 threads (470 species: 11 row blocks) or one FP64 CTA of 704 fill the
// register file of an SM.
template <class T, bool TF>
__global__ void __launch_bounds__(704, 1) cell_kernel(const __grid_constant__ Args A) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int sh_c;
  const Dev& d = A.d;
  const int tid = threadIdx.x, nthr = blockDim.x, n = d.n;
  Cell<T> q;
  cell_views<T>(A, sm, q);
  CellS& S = *q.S;
#ifdef SM_PHASE_CLOCKS
  long long ph_t = clock64();
#endif
  // per-cell scalars: the double rows t .. alpha and the int rows q ..
  // slot_cell of the state are contiguous with stride ld
  constexpr int kD = 6 + 2 * (QMAX + 1);
  for (;;) {
    __syncthreads();
    if (tid == 0) {
      // ring: [0] next entry, [1] entries reserved; an entry holds slot + 1
      // and is 0 between its reservation and its store
      int got = -1;
      volatile int* r = A.ring;
      for (int tries = 0; tries < (1 << 20); ++tries) {   // an entry left behind is its producer's to take
        const int hd = r[0];
        if (hd >= r[1]) break;
        const int v = r[2 + hd];
        if (v == 0) continue;   // its producer is between two instructions
        if (atomicCAS(A.ring, hd, hd + 1) == hd) {
          got = v - 1;
          break;
        }
      }
      __threadfence();
      sh_c = got;
    }
    __syncthreads();
    const int c = sh_c;
    if (c < 0) break;
    if (d.status[c] != SM_CELL_RUNNING) continue;
    __threadfence();
    q.c = c;
    q.oc = d.slot_cell[c];
    q.P = static_cast<T*>(d.lup) + q.oc * d.lup_stride;
    if (tid < kD) {
      const double v = d.t[(int64_t)tid * d.ld + c];
      if (tid == 0) S.t = v;
      else if (tid == 1) S.h = v;
      else if (tid == 2) S.gam = v;
      else if (tid == 3) S.gam_J = v;
      else if (tid == 4) S.crate = v;
      else if (tid == 5) S.dprev = v;
      else if (tid < 6 + QMAX + 1) S.tn[tid - 6] = v;
      else S.alpha[tid - 6 - (QMAX + 1)] = v;
    }
    if (tid == 0) {
      S.q = d.q[c];
      S.nh = d.nh[c];
      S.n_at_q = d.n_at_q[c];
      S.j_age = d.j_age[c];
      S.flags = d.flags[c];
      S.crej = d.crej[c];
      S.ccf = d.ccf[c];
      S.status = SM_CELL_RUNNING;
      S.m_it = d.m_it[c];
      S.steps = d.steps[c];
      S.rejects = d.rejects[c];
      S.conv_fails = d.conv_fails[c];
      S.newton_iters = d.newton_iters[c];
      S.jac_evals = d.jac_evals[c];
      S.base = 0;
      S.best_q = 0;
    }
    cell_conditions<T>(A, q);
    const int nh0 = d.nh[c];
    for (int s = tid; s < n; s += nthr) {
      const int64_t o = (int64_t)s * d.ld + c;
      for (int i = 0; i < nh0; ++i) q.hist[(int64_t)i * q.hn + s] = Yh(d, i)[o];
      q.eprev[s] = d.eprev[o];
      q.wf[s] = d.wf[o];
    }
    __syncthreads();
    if (d.therm) {
      // every coefficient from the current T; the attempt's own passes refresh
      // the T-dependent ones
      cell_th_rates(A, q.kc, q.hist[d.t_idx], q.nH, q.Av, q.chi, true);
    }
    PHASE_MARK(PH_LOAD);
    const int before = A.done[c], todo = min(A.slice, A.attempts - before);
    int made = 0;
    bool run = true;
    while (run && made < todo) {
      run = cell_attempt<T, TF>(A, q, sm PHASE_PASS);
      ++made;
    }
    __syncthreads();
    // back to the state's arrays
    if (tid < kD) {
      double v;
      if (tid == 0) v = S.t;
      else if (tid == 1) v = S.h;
      else if (tid == 2) v = S.gam;
      else if (tid == 3) v = S.gam_J;
      else if (tid == 4) v = S.crate;
      else if (tid == 5) v = S.dprev;
      else if (tid < 6 + QMAX + 1) v = S.tn[tid - 6];
      else v = S.alpha[tid - 6 - (QMAX + 1)];
      d.t[(int64_t)tid * d.ld + c] = v;
    }
    for (int s = tid; s < n; s += nthr) {
      const int64_t o = (int64_t)s * d.ld + c;
      for (int i = 0; i < S.nh; ++i) {
        int slot = S.base + i;
        if (slot > QMAX) slot -= QMAX + 1;
        Yh(d, i)[o] = q.hist[(int64_t)slot * q.hn + s];
      }
      d.eprev[o] = q.eprev[s];
      d.wf[o] = q.wf[s];
    }
    if (tid == 0) {
      d.q[c] = S.q;
      d.nh[c] = S.nh;
      d.n_at_q[c] = S.n_at_q;
      d.j_age[c] = S.j_age;
      d.flags[c] = S.flags;
      d.crej[c] = S.crej;
      d.ccf[c] = S.ccf;
      d.status[c] = S.status;
      d.m_it[c] = S.m_it;
      d.steps[c] = S.steps;
      d.rejects[c] = S.rejects;
      d.conv_fails[c] = S.conv_fails;
      d.newton_iters[c] = S.newton_iters;
      d.jac_evals[c] = S.jac_evals;
      A.done[c] = before + made;
    }
    __threadfence();
    __syncthreads();
    if (tid == 0 && run && before + made < A.attempts) {
      // not done: back to the end of the queue
      const int at = atomicAdd(A.ring + 1, 1);
      __threadfence();
      *(volatile int*)(A.ring + 2 + at) = c + 1;
    }
    PHASE_MARK(PH_LOAD);
  }
}

// Fills the queue with the slots below C and clears the attempt counts.
__global__ void ring_kernel(int64_t C, int* ring, int* done, int64_t total) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) {
    ring[0] = 0;
    ring[1] = (int)C;
  }
  if (i < C) done[i] = 0;
  if (i < total) ring[2 + i] = i < C ? (int)i + 1 : 0;
}

// Start of an integration: validates the inputs of each cell, f0 = f(y0) and
// h0 = min(0.01 / |f0|_wrms, t_end).
template <class T>
__global__ void __launch_bounds__(704, 1) cell_init_kernel(const __grid_constant__ Args A, const double* __restrict__ y,
                                                           int64_t ldu) {
  extern __shared__ __align__(16) unsigned char sm[];
  const Dev& d = A.d;
  const int tid = threadIdx.x, nthr = blockDim.x, n = d.n;
  Cell<T> q;
  cell_views<T>(A, sm, q);
#ifdef SM_PHASE_CLOCKS
  long long ph_t = clock64();
#endif
  for (int64_t c = blockIdx.x; c < d.C; c += gridDim.x) {
    q.c = q.oc = c;
    bool ok = true;
    for (int s = tid; s < n; s += nthr) {
      const double v = y[(int64_t)s * ldu + c];
      q.ys[s] = v;
      Yh(d, 0)[(int64_t)s * d.ld + c] = v;
      ok = ok && isfinite(v);
    }
    cell_conditions<T>(A, q);
    if (!d.therm)
      for (int j = tid; j < d.n_r; j += nthr) ok = ok && isfinite(q.kc[j]);
    __syncthreads();
    if (d.therm)
      ok = ok && q.ys[d.t_idx] > 0.0 && isfinite(q.nH) && q.nH > 0.0 && isfinite(q.Av) && isfinite(q.chi);
    ok = __syncthreads_and(ok);
    if (ok) {
      if (d.therm) cell_th_rates(A, q.kc, q.ys[d.t_idx], q.nH, q.Av, q.chi, true);
      cell_rhs(A, q.kc, q.ys, q.tab, q.part, q.fs PHASE_PASS);
      if (d.therm) cell_energy(A, q.ys, q.fs, q.nH, q.red);
    }
    double acc = 0.0;
    if (ok)
      for (int s = tid; s < n; s += nthr) {
        d.f0[(int64_t)s * d.ld + c] = q.fs[s];
        const double v = q.fs[s] / (d.rtol * fabs(q.ys[s]) + d.atol);
        acc += v * v;
      }
    acc = cta_sum(acc, q.red, 3);
    if (tid == 0) {
      d.slot_cell[c] = (int)c;
      d.status[c] = ok ? SM_CELL_RUNNING : SM_CELL_NAN;
      d.flags[c] = ok ? F_NEED_J : 0;
      d.t[c] = 0.0;
      d.steps[c] = d.rejects[c] = d.conv_fails[c] = d.newton_iters[c] = d.jac_evals[c] = 0;
      d.q[c] = 1;
      d.h[c] = 0.0;
      if (ok) {
        d.h[c] = fmin(0.01 / fmax(sqrt(acc / n), 1e-300), d.t_end);
        d.nh[c] = 1;
        d.tn[c] = 0.0;
        d.n_at_q[c] = 0;
        d.j_age[c] = 0;
        d.gam_J[c] = 1.0;
        d.crate[c] = 1.0;
        d.crej[c] = d.ccf[c] = 0;
        if (d.record) {
          d.ck_t[c] = 0.0;
          d.ck_nh[c] = 1;
        }
      }
    }
    if (d.record && ok)
      for (int s = tid; s < n; s += nthr) d.ck_Y[(int64_t)s * d.ld + c] = q.ys[s];
    __syncthreads();
  }
}

Args make_args(const sm_net* net, const Dev& d, const CellLaunch& L, const double* k, int64_t ldk) {
  const CellProg& p = net->cell;
  Args a{};
  a.d = d;
  a.p = L.plan;
  a.w = p.blob.as<int>();
  a.nb = p.nb; a.pitch = p.pitch;
  a.n_rsl = p.n_rsl; a.n_part = p.n_part; a.n_rlong = p.n_rlong;
  a.rp_off = p.rp_off; a.rp_ent = p.rp_ent; a.rp_dst = p.rp_dst; a.row_ptr = p.row_ptr; a.row_long = p.row_long;
  a.n_jsl = p.n_jsl; a.n_jl = p.n_jl;
  a.jg_off = p.jg_off; a.jg_ent = p.jg_ent; a.jg_rc = p.jg_rc; a.jg_dst = p.jg_dst; a.jg_grp = p.jg_grp;
  a.jl_ptr = p.jl_ptr; a.jl_ent = p.jl_ent; a.jl_rc = p.jl_rc; a.jl_dst = p.jl_dst; a.jl_grp = p.jl_grp;
  a.n_hlev = net->lu.n_hlev; a.hop = p.hop; a.hterm = p.hterm; a.hop_ptr = p.hop_ptr;
  a.tg_grp = p.tg_grp; a.tg_off = p.tg_off; a.tg_ent = p.tg_ent; a.tg_pos = p.tg_pos;
  a.lev_f = p.lev_f; a.lev_b = p.lev_b; a.u12c = p.u12c;
  a.n_l21 = net->lu.lrhoff.back(); a.n_u12 = net->lu.u12off.back();
  a.n_vsl = p.n_vsl; a.n_vpart = p.n_vpart; a.n_vlong = p.n_vlong;
  a.vp_off = p.vp_off; a.vp_ent = p.vp_ent; a.vp_dst = p.vp_dst; a.vrow_ptr = p.vrow_ptr; a.vrow_long = p.vrow_long;
  a.k = k;
  a.ldk = ldk;
  a.scratch = L.scratch;
  a.ring = L.ring;
  a.done = L.done;
  a.timing = L.timing;
  a.timing_kind = L.timing_kind;
  return a;
}

// Attempts a cell makes before it goes back to the end of the queue.  With
// many cells per CTA a cell runs all its attempts at once (its factors stay
// in L2); with few, short turns keep the last wave of cells from leaving
// most of the SMs idle.
int turn(int64_t C, int ctas, int attempts) {
  if (C <= ctas || C >= 8LL * ctas) return attempts;
  return std::max(8, (attempts + 15) / 16);
}

const void* kernel_of(const Dev& d) {
  if (!d.mixed) return (const void*)cell_kernel<double, false>;
  return d.tf32 ? (const void*)cell_kernel<float, true> : (const void*)cell_kernel<float, false>;
}

}  // namespace

sm_status cell_resident(const Dev& d, const CellPlan& plan, int per_sm_cap, int* ctas) {
  *ctas = 0;
  int dev = 0, sms = 0, smem = 0, per = 0;
  SM_TRY_CUDA(cudaGetDevice(&dev));
  SM_TRY_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  SM_TRY_CUDA(cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  const void* init = d.mixed ? (const void*)cell_init_kernel<float> : (const void*)cell_init_kernel<double>;
  // per-kernel caps are shared by every state: always the device's limit
  SM_TRY_CUDA(cudaFuncSetAttribute(kernel_of(d), cudaFuncAttributeMaxDynamicSharedMemorySize, smem - 1024));
  SM_TRY_CUDA(cudaFuncSetAttribute(init, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  SM_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel_of(d), 32 * plan.warps, plan.bytes));
  if (per_sm_cap > 0) per = std::min(per, per_sm_cap);
  *ctas = sms * per;
  return SM_OK;
}

int64_t cell_ring_ints(int64_t C, int ctas, int attempts) {
  const int tn = turn(C, ctas, attempts);
  return 2 + C * ((attempts + tn - 1) / tn);
}

sm_status launch_cell_init(const sm_net* net, const Dev& d, const CellLaunch& L, const double* y, int64_t ldu,
                           const double* k, int64_t ldk, cudaStream_t s) {
  const Args a = make_args(net, d, L, k, ldk);
  const unsigned grid = (unsigned)std::min<int64_t>(d.C, L.ctas);
  if (d.mixed) cell_init_kernel<float><<<grid, 32 * L.plan.warps, L.plan.bytes, s>>>(a, y, ldu);
  else cell_init_kernel<double><<<grid, 32 * L.plan.warps, L.plan.bytes, s>>>(a, y, ldu);
  SM_TRY_CUDA(cudaGetLastError());
  return SM_OK;
}

sm_status launch_cell_attempts(const sm_net* net, const Dev& d, const CellLaunch& L, const double* k, int64_t ldk,
                               int attempts, cudaStream_t s) {
  Args a = make_args(net, d, L, k, ldk);
  a.attempts = attempts;
  a.slice = turn(d.C, L.ctas, attempts);
  const int64_t total = cell_ring_ints(d.C, L.ctas, attempts) - 2;
  ring_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(d.C, L.ring, L.done, total);
  SM_TRY_CUDA(cudaGetLastError());
  const unsigned grid = (unsigned)std::min<int64_t>(d.C, L.ctas);
  const int threads = 32 * L.plan.warps;
  if (!d.mixed) cell_kernel<double, false><<<grid, threads, L.plan.bytes, s>>>(a);
  else if (d.tf32) cell_kernel<float, true><<<grid, threads, L.plan.bytes, s>>>(a);
  else cell_kernel<float, false><<<grid, threads, L.plan.bytes, s>>>(a);
  SM_TRY_CUDA(cudaGetLastError());
  return SM_OK;
}

extern "C" sm_status sm_phase_cycles(int32_t device, double* h_out, int32_t reset) {
#ifdef SM_PHASE_CLOCKS
  if (!h_out || device < 0) return SM_EINVAL;
  int prev = -1;
  if (cudaGetDevice(&prev) != cudaSuccess || cudaSetDevice(device) != cudaSuccess) return SM_ECUDA;
  unsigned long long v[kPhaseSlots];
  SM_TRY_CUDA(cudaMemcpyFromSymbol(v, g_phase_cycles, sizeof(v)));
  for (int i = 0; i < kPhaseSlots; ++i) h_out[i] = (double)v[i];
  if (reset) {
    const unsigned long long z[kPhaseSlots] = {0};
    SM_TRY_CUDA(cudaMemcpyToSymbol(g_phase_cycles, z, sizeof(z)));
  }
  cudaSetDevice(prev);
  return SM_OK;
#else
  (void)device;
  (void)h_out;
  (void)reset;
  return SM_ENOTSUP;
#endif
}
