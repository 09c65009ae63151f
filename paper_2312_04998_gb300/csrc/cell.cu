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
//   rates, S R    a thread per reaction, then the rows of S in chains, a chain
//                 per lane (CellProg); bound by the FP64 pipe (2 lanes a clock
//                 per SM)
//   Jacobian      an entry per lane over the table of dR/dx in shared memory
//   head          the head program, level by level, in shared memory
//   tail          right-looking by 32-column panels, its 32 x 32 blocks as
//                 register tiles of one warp each (see factor_tail)
//   substitution  a warp per 32 rows; the next block's factors are in flight
//                 while the diagonal block's 32-step chain runs
// Every sum that a step depends on is formed in the order of the class-by-class
// kernels (integrate.cu), which serve large batches and the networks that do not
// fit: the two take the same steps to the last bit (with the 16-cell gather).
//
// Cycles per cell on one SM, 470 species, 6000 reactions, FP32 factors: rates
// 15 k, S R 29 k and substitution 118 k per Newton iteration; predict 14 k,
// finish 26 k per attempt; Jacobian 69 k, head 54 k, assembly 197 k, panels
// 171 k, trailing updates 428 k per factorisation.  (One launch per kernel class:
// 2.28 M per factorisation.)  4096 cells, first 1e-3 yr: 1203 -> 723 ms; 128 cells
// of a slab, 1e3 yr: 562 -> 57 ms; one cell of 32 species, 1e6 yr: 17.0 -> 4.9 ms.
#include "cell.h"
#include <algorithm>
#include <type_traits>

#include "integ.h"

using namespace integ;

namespace {

constexpr int XP = 36;         // row pitch of the 32 x 32 exchange blocks (words): 16-byte rows, few conflicts
constexpr unsigned kFull = 0xffffffffu;

// A cell's scalars while a CTA works on it.
struct CellS {
  double t, h, gam, gam_J, crate, dprev, tnew, err, eta, inv_a0, scale;
  double tn[QMAX + 1], alpha[QMAX + 1], wts[QMAX + 1], wlo[QMAX + 1];
  int q, nh, n_at_q, j_age, flags, crej, ccf, status, m_it, steps, rejects, conv_fails, newton_iters, jac_evals;
  int base;      // history point i is scratch slot (base + i) % (QMAX + 1)
  int state, best_q;
  int hn;                         // stride of a history point in scratch
  long long c, oc;                // slot and cell
  double *kc, *hist, *eprev;      // this CTA's global scratch: k', history ring, last error vector
  void *mbuf, *P;                 // Jacobian values in program order (scratch); the cell's packed factors
  double nH, Av, chi;             // conditions (coupled temperature)
  long long t0, ph_t;             // clocks of the timed class and the last phase mark
};
static_assert(sizeof(CellS) <= kCellScalars, "shared-memory plan");

struct Args {
  Dev d;
  CellPlan p;
  const int* w;            // index programs (CellProg blob)
  int nb, pitch, n_slot, rx, iperm;
  int rp_deal, rp_ent, rp_dst, row, row_more;
  int n_jsl, n_jl, n_jw, jg_off, jg_ent, jg_rc, jg_dst, jg_grp, jl_off, jl_ent, jl_rc, jd_grp, jd_ent;
  int n_hlev, hop, hterm, hop_ptr;
  int tg_grp, tg_ent;
  int lev_f, lev_b, hx;
  int vp_deal, vp_ent, vp_dst, vrow, vrow_more;
  const double* k;
  int64_t ldk;
  double* scratch;
  int *ring, *done;
  int attempts, slice;
  double* timing;
  int timing_kind;
};

static_assert(sizeof(Args) <= kCellArgs, "shared-memory plan");

// The launch's arguments are copied to the front of the CTA's shared memory,
// where the phases take them and the vectors from: kept in registers, the many
// addresses made the inner loops spill, each spill a trip to L2 next to 200 KB
// of shared memory.  (The phases are inlined for the same reason: a call saves
// registers to memory.)
extern __shared__ __align__(16) unsigned char sm[];
__device__ __forceinline__ const Args& args() { return *reinterpret_cast<const Args*>(sm); }
__device__ __forceinline__ CellS& scalars() { return *reinterpret_cast<CellS*>(sm + kCellArgs); }
template <class V> __device__ __forceinline__ V* at(int offset) { return reinterpret_cast<V*>(sm + offset); }

// optional cycle counters of the phases (build option SM_PHASE_CLOCKS)
constexpr int kPhaseSlots = 16;
enum { PH_LOAD, PH_PREDICT, PH_RATES, PH_GATHER, PH_SOLVE, PH_FINISH, PH_JAC, PH_HEAD, PH_ASSEMBLE, PH_UPDATE, PH_PANEL };
#ifdef SM_PHASE_CLOCKS
__device__ unsigned long long g_phase_cycles[kPhaseSlots];
#define PHASE_MARK(k)                                                                 \
  do {                                                                                \
    if (threadIdx.x == 0) {                                                           \
      const long long ph_now = clock64();                                             \
      atomicAdd(&g_phase_cycles[(k)], (unsigned long long)(ph_now - scalars().ph_t)); \
      scalars().ph_t = ph_now;                                                        \
    }                                                                                 \
  } while (0)
#else
#define PHASE_MARK(k) do {} while (0)
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
// A plain load that stays where it is written: left to itself the compiler
// forms the addresses of a whole block of strided loads first, and spills.
__device__ __forceinline__ float ld_here(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ double ld_here(const double* p) {
  double v;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The coefficient of an index word.
__device__ __forceinline__ double coef(int word) { return __hiloint2double(word & 0xFFFF0000, 0); }

// Sums of rows cut into chains (see Chains in cell_prog.cpp): a chain per lane,
// slices of 32 chains per warp, dealt so that the schedulers' FP64 units (a warp's
// FMA holds one for 64 cycles) have equal work.  tab[pad slot] must be 0.  All
// threads.
__device__ __forceinline__ void row_sums(const int* __restrict__ w, int deal, int ent, int dst, int row, int more,
                                         const double* tab, double* part, double* out, int n) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int rw = (int)threadIdx.x < n ? __ldg(w + row + threadIdx.x) : 0;
  const int2 own = __ldg(reinterpret_cast<const int2*>(w + deal) + warp);
  const int4* meta = reinterpret_cast<const int4*>(w + deal);
  int4 mt = own.x < own.y ? __ldg(meta + own.x) : make_int4(0, 0, 0, 0);
  for (int i = own.x; i < own.y; ++i) {
    const int* q = w + ent + 32 * mt.x + lane;
    const int m = mt.y, to = __ldg(w + dst + 32 * mt.z + lane);
    int t[4], nx[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) t[u] = u < m ? __ldg(q + 32 * u) : 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) nx[u] = 4 + u < m ? __ldg(q + 32 * (4 + u)) : 0;
    if (i + 1 < own.y) mt = __ldg(meta + i + 1);
    double a = 0.0;
    int e = 4;
    for (; e <= m; e += 4) {
      int n2[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) n2[u] = e + 4 + u < m ? __ldg(q + 32 * (e + 4 + u)) : 0;
#pragma unroll
      for (int u = 0; u < 4; ++u) a = fma(coef(t[u]), tab[t[u] & 0xFFFF], a);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        t[u] = nx[u];
        nx[u] = n2[u];
      }
    }
    // (an FP64 instruction that is predicated off holds the unit all the same,
    // and short branches become predicates: the rest as a loop)
#pragma unroll 1
    for (e -= 4; e < m; ++e) {
      a = fma(coef(t[0]), tab[t[0] & 0xFFFF], a);
      t[0] = t[1];
      t[1] = t[2];
    }
    part[to] = a;
  }
  __syncthreads();
  auto of = [&](int word) {
    const double* p = part + (word & 0xFFFF);
    return word < 0 ? (p[0] + p[1]) + (p[2] + p[3]) : p[0];
  };
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    if (i >= (int)blockDim.x) rw = __ldg(w + row + i);
    double v = of(rw);
    const int x = (rw & 0x7FFFFFFF) >> 16;
    if (x)
      for (int q = x - 1;; ++q) {
        const int word = __ldg(w + more + q);
        v += of(word);
        if (word & (1 << 30)) break;
      }
    out[i] = v;
  }
}

// Sums over the CTA are formed as by 512 threads whatever the CTA's size, so
// that a cell's result does not depend on the batch that it is part of: the
// term of index i belongs to virtual thread i mod 512, each warp of those is
// summed by shuffles, the warps in order.
constexpr int kVirt = 512, RS = kVirt / 32;

// Partial sums of f(i), i < n, into reduction slot `slot`; all threads.
template <class F>
__device__ __forceinline__ void sum_parts(int slot, int n, F f) {
  double* red = at<double>(kCellRed) + RS * slot;
  const int top = min(kVirt, (n + 31) / 32 * 32);
  for (int v = threadIdx.x; v < top; v += blockDim.x) {
    double a = 0.0;
    for (int i = v; i < n; i += kVirt) a += f(i);
    a = warp_sum(a);
    if ((v & 31) == 0) red[v >> 5] = a;
  }
}
// Their sum, by one warp after a barrier; the result in every lane.
__device__ __forceinline__ double sum_total(int slot, int n) {
  const int lane = threadIdx.x & 31, parts = min(RS, (n + 31) / 32);
  return warp_sum(lane < parts ? at<double>(kCellRed)[RS * slot + lane] : 0.0);
}

// R_j = k'_j prod y (slot n_r of the table = 0), then fs = S R at state y.
// Ends with a barrier.
__device__ __forceinline__ void cell_rhs() {
  const Args& A = args();
  const int n_r = A.d.n_r;
  const int2* rx = reinterpret_cast<const int2*>(A.w + A.rx);
  const double* kc = scalars().kc;
  const double* y = at<double>(A.p.o_ys);
  double* tab = at<double>(A.p.o_r);
#pragma unroll 4
  for (int j = threadIdx.x; j < n_r; j += blockDim.x) {
    const int ab = __ldg(rx + j).x;
    double v = kc[j] * y[ab & 0xFFFF];
    const int b = (uint32_t)ab >> 16;
    if (b != 0xFFFF) v *= y[b];
    tab[j] = v;
  }
  if (threadIdx.x == 0) tab[n_r] = 0.0;
  __syncthreads();
  PHASE_MARK(PH_RATES);
  row_sums(A.w, A.rp_deal, A.rp_ent, A.rp_dst, A.row, A.row_more, tab, at<double>(A.p.o_part),
           at<double>(A.p.o_fs), A.d.n);
  __syncthreads();
  PHASE_MARK(PH_GATHER);
}

// ---- coupled temperature ----------------------------------------------------
// k' of the T-dependent reactions (all reactions when init) at temperature T.
__device__ __forceinline__ void cell_th_rates(double T, bool init) {
  const Args& A = args();
  const CellS& S = scalars();
  double* kc = S.kc;
  const double nH = S.nH, lt = log(T * (1.0 / 300.0)), it = 1.0 / T;
  const RatePar* par = A.d.rpar;
  for (int j = threadIdx.x; j < A.d.n_r; j += blockDim.x) {
    const RatePar p = par[j];
    const int cls = (int)p.w;
    if (cls == SM_TWO_BODY || cls == SM_DISS_RECOMB) kc[j] = exp(fma(p.y, lt, p.x) - p.z * it) * nH;
    else if (init) kc[j] = cls == SM_COSMIC_RAY ? p.x * A.d.th_zeta : S.chi * p.x * exp(-p.z * S.Av);
  }
  __syncthreads();
}

// Temperature row of fs from y and the chemical rows.  Ends with a barrier.
__device__ __forceinline__ void cell_energy() {
  const Args& A = args();
  const Dev& d = A.d;
  const double* y = at<double>(A.p.o_ys);
  double* fs = at<double>(A.p.o_fs);
  const int t = d.t_idx;
  const double T = y[t], nH = scalars().nH;
  const int n = d.n;
  sum_parts(0, n, [&](int i) { return i == t ? 0.0 : y[i]; });
  sum_parts(1, n, [&](int i) { return i == t ? 0.0 : fs[i]; });
  __syncthreads();
  if (threadIdx.x < 32) {
    const double xt = sum_total(0, n), F = sum_total(1, n);
    double line = 0.0;   // in order
    for (int q0 = 0; q0 < d.n_cool; q0 += 32) {
      double v = 0.0, yv = 0.0;
      if (q0 + (int)threadIdx.x < d.n_cool) {
        const int i = __ldg(d.th_cool + q0 + threadIdx.x);
        v = d.th_L[i] * exp(-d.th_E[i] / T);
        yv = y[i];
      }
      for (int q = 0; q < min(32, d.n_cool - q0); ++q) line = fma(__shfl_sync(kFull, yv, q), __shfl_sync(kFull, v, q), line);
    }
    if (threadIdx.x == 0)
      fs[t] = (d.th_heat - nH * line - d.th_lam * nH * (T - d.th_Td) - 1.5 * T * F) / (1.5 * xt);
  }
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
__device__ __forceinline__ void store4(float* p, const float (&v)[4]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void store4(double* p, const double (&v)[4]) {
  *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
  *reinterpret_cast<double2*>(p + 2) = make_double2(v[2], v[3]);
}

// Before a substitution, asynchronously into shared memory: the head's packed
// factors (hd) and the tail's diagonal blocks (dg: [nb][32 columns][32 rows]),
// which the dependent chains read.
template <class T>
__device__ __forceinline__ void solve_prefetch() {
  constexpr int PER = 16 / sizeof(T), CPC = 32 / PER;
  const Args& A = args();
  const Dev& d = A.d;
  const T* P = static_cast<const T*>(scalars().P);
  T* hd = at<T>(A.p.o_hd);
  T* dg = at<T>(A.p.o_dg);
  const int nt = d.n - d.head, p_d = d.p_d, nthr = blockDim.x;
  const int64_t ldd = d.ldd;
  for (int e = threadIdx.x * PER; e < p_d; e += nthr * PER) cp16(hd + e, P + e);
  for (int q = threadIdx.x; q < nt * CPC; q += nthr) {   // q: (column, chunk of its block's rows)
    const int c = q / CPC, i = q % CPC * PER;
    cp16(dg + c * 32 + i, P + p_d + c * ldd + (c & ~31) + i);
  }
}

// Diagonal blocks (a row per lane), column by column: one shuffle and one FMA
// a step, the factors' loads ahead of the chain.
template <class T>
__device__ __forceinline__ T diag_forward(T xi, const T* dg, int lane, int w) {
#pragma unroll 8
  for (int k = 0; k < 32; ++k) {
    const T l = lane > k ? dg[k * 32 + lane] : T(0);
    const T xk = __shfl_sync(kFull, xi, k);
    if (k < w) xi -= l * xk;   // (past w: padding)
  }
  return xi;
}
template <class T>
__device__ __forceinline__ T diag_backward(T xi, const T* dg, int lane, int w) {
  // a product, a shuffle and an FMA a step: every lane forms its own entry's
  // product with its inverse pivot, the shuffle takes lane k's; a finished
  // lane's result is kept aside, what it computes after that is not used
  const T inv = lane < w ? dg[lane * 32 + lane] : T(0);
  T out = T(0);
  if (lane >= w) xi = T(0);   // (past w: padding)
#pragma unroll 8
  for (int k = 31; k >= 0; --k) {
    const T u = lane < k && k < w ? dg[k * 32 + lane] : T(0);
    const T t = xi * inv;
    const T xk = __shfl_sync(kFull, t, k);
    out = lane == k ? t : out;
    xi -= u * xk;
  }
  return out;
}

// One row block of the tail in a warp's registers: its entry per lane and the
// 32 columns in flight.
template <class T>
struct RowBlock {
  T x, ln[32];
  // From the first of w columns at p; with fewer than 32 the last one again,
  // for entries of x that are 0.  (Rows past the tail's end are padding: their
  // lanes compute on it and are not read.)
  __device__ __forceinline__ void load(const T* p, int64_t ldd, int w) {
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      ln[k] = ld_here(p);
      if (k + 1 < w) p += ldd;
    }
  }
  __device__ __forceinline__ void apply(const T* xk) {
    T a = T(0);
#pragma unroll
    for (int k = 0; k < 32; k += 4) {
      T v[4];
      load4(xk + k, v);
#pragma unroll
      for (int u = 0; u < 4; ++u) a += ln[k + u] * v[u];
    }
    x -= a;
  }
};

// x := M^-1 x with the cell's packed factors; x in elimination order, head part
// xh[h], tail part xt (16-byte aligned, 32 nb entries), after solve_prefetch.
// In the tail warp i carries row block i,
// its next 32 columns in flight; as soon as a block's columns are applied its
// warp solves the next diagonal block.  (Row blocks past the CTA's warps are
// worked on in place, by warp i mod nw, without loads ahead.)
// Begins and ends with a barrier.
template <class T>
__device__ __forceinline__ void cell_solve() {
  const Args& A = args();
  const Dev& d = A.d;
  T* xh = at<T>(A.p.o_xh);
  T* xt = at<T>(A.p.o_xt);
  T* hd = at<T>(A.p.o_hd);
  const T* dg = at<T>(A.p.o_dg);
  const int n = d.n, h = d.head, nt = n - h, nb = A.nb;
  const int64_t ldd = d.ldd;
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, nw = nthr >> 5;
  const int ra = tid >> 5;   // this warp's row block
  const T* D = static_cast<const T*>(scalars().P) + d.p_d;
  const bool ina = 32 * ra + lane < nt;
  RowBlock<T> a;
  if (ra > 0 && ra < nb) a.load(D + 32 * ra + lane, ldd, 32);
  cp_wait();
  __syncthreads();
  // a row of head factors against x: entries [e0, e1) of the packed head, hx
  // their index in x
  const uint16_t* hx = at<uint16_t>(A.p.o_hx);
  auto row_dot = [&](int e0, int e1, const T* x) {
    T v = T(0);
#pragma unroll 4
    for (int e = e0; e < e1; ++e) v += hd[e] * x[hx[e]];
    return v;
  };
  // head, forward: a row per thread, level by level
  for (int i0 = 0; i0 < h; i0 += nthr) {   // one pass unless the head outgrows the CTA (rows of a pass come first)
    const int i = i0 + tid;
    const bool inh = i < h;
    const int p0 = inh ? __ldg(d.lrptr + i) : 0, p1 = inh ? __ldg(d.lrptr + i + 1) : 0;
    const int lev = inh ? __ldg(A.w + A.lev_f + i) : -1;
    for (int l = i0 == 0 ? 1 : 0; l < d.n_flev; ++l) {
      if (lev == l) xh[i] -= row_dot(d.p_l11 + p0, d.p_l11 + p1, xh);
      __syncthreads();
    }
  }
  if (h == 0) __syncthreads();
  auto l21_row = [&](int row) {
    return xt[row] - row_dot(d.p_l21 + __ldg(d.lrhoff + row), d.p_l21 + __ldg(d.lrhoff + row + 1), xh);
  };
  a.x = ina ? l21_row(32 * ra + lane) : T(0);
  for (int r = ra + nw; r < nb; r += nw)
    if (32 * r + lane < nt) xt[32 * r + lane] = l21_row(32 * r + lane);
  // block column K applied to row block r in place
  auto far = [&](int r, int K, int w) {
    const T* p = D + (32 * K) * ldd + 32 * r + lane;
    T v = T(0);
#pragma unroll 8
    for (int k = 0; k < w; ++k) v += p[k * ldd] * xt[32 * K + k];
    if (32 * r + lane < nt) xt[32 * r + lane] -= v;
  };
  auto far_solve = [&](int r, bool forward) {
    const int w = min(32, nt - 32 * r);
    const T v = xt[32 * r + lane];
    const T x = forward ? diag_forward(v, dg + r * 1024, lane, w) : diag_backward(v, dg + r * 1024, lane, w);
    xt[32 * r + lane] = lane < w ? x : T(0);
  };
  // tail, forward (unit lower triangle)
  for (int K = -1; K < nb - 1; ++K) {
    if (K >= 0) {
      __syncthreads();
      if (K < ra && ra < nb) {
        a.apply(xt + 32 * K);
        if (K + 1 < ra) a.load(D + (32 * (K + 1)) * ldd + 32 * ra + lane, ldd, 32);
      }
      for (int r = ra + nw; r < nb; r += nw)
        if (r > K) far(r, K, 32);
    }
    if (K + 1 == ra) {
      a.x = diag_forward(a.x, dg + ra * 1024, lane, min(32, nt - 32 * ra));
      xt[32 * ra + lane] = ina ? a.x : T(0);
      if (ra < nb - 1) a.load(D + (32 * (nb - 1)) * ldd + 32 * ra + lane, ldd, nt - 32 * (nb - 1));   // the way back's first
    } else if (K + 1 >= nw && (K + 1) % nw == ra) {
      __syncwarp();
      far_solve(K + 1, true);
    }
  }
  __syncthreads();
  // tail, backward (inverse pivots on the diagonal)
  auto col = [&](int K) { return D + (32 * K) * ldd + 32 * ra + lane; };
  for (int K = nb; K > 0; --K) {
    if (K < nb) {
      __syncthreads();
      if (K > ra) {
        a.apply(xt + 32 * K);
        if (K - 1 > ra) a.load(col(K - 1), ldd, 32);
      }
      for (int r = ra + nw; r < K; r += nw) far(r, K, min(32, nt - 32 * K));
    }
    if (K - 1 == ra) {
      a.x = diag_backward(a.x, dg + ra * 1024, lane, min(32, nt - 32 * ra));
      xt[32 * ra + lane] = ina ? a.x : T(0);
    } else if (K - 1 >= nw && (K - 1) % nw == ra) {
      __syncwarp();
      far_solve(K - 1, false);
    }
  }
  __syncthreads();
  // U12, then the head backward
  for (int i0 = h > 0 ? (h - 1) / nthr * nthr : -1; i0 >= 0; i0 -= nthr) {
    const int i = i0 + tid;
    const bool inh = i < h;
    T xv = T(0);
    int e0 = 0, e1 = 0, lev = -1;
    if (inh) {
      e0 = d.p_u11 + __ldg(d.u11ptr + i);
      e1 = d.p_u11 + __ldg(d.u11ptr + i + 1);
      lev = __ldg(A.w + A.lev_b + i);
      xv = xh[i] - row_dot(d.p_u12 + __ldg(d.u12off + i), d.p_u12 + __ldg(d.u12off + i + 1), xt);
    }
    for (int l = 0; l < d.n_blev; ++l) {
      if (lev == l) xh[i] = (xv - row_dot(e0, e1, xh)) * hd[d.p_dinv + i];
      __syncthreads();
    }
  }
  if (h == 0) __syncthreads();
}

// ---- factorisation ----------------------------------------------------------
// The triangular kernels of 32 x 32 blocks hold one row (or column) of 32
// entries per lane and run eight of them at a time in rolled loops, the
// remaining ones rotated to the front of the register array: unrolled over all
// 32 each would be straight-line code executed once per panel.  `more(g)`
// says whether the entries 8 g .. 8 g + 7 past the current eight exist.

// LU of the diagonal block in uj (by rows, pitch XP), a row per lane, pivot rows
// by shuffles: U and the inverse pivots back to uj, L by columns into
// lj[k][i]; the first w columns to D (dst: this lane's row).
template <class T>
__device__ __forceinline__ void lu_block(T* uj, T* lj, T* dst, int64_t ldd, int w, int lane) {
  T c[32];   // row `lane` of the block (in uj); the identity past w
#pragma unroll
  for (int j = 0; j < 32; ++j) c[j] = j == lane ? T(1) : T(0);
  if (lane < w) {
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (j < w) c[j] = uj[lane * XP + j];
  }
  __syncwarp();
#pragma unroll 1
  for (int b0 = 0; b0 < 32; b0 += 8) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const T inv = T(1) / __shfl_sync(kFull, c[k], b0 + k);
      const T l = lane > b0 + k ? c[k] * inv : T(0);
#pragma unroll
      for (int j = k + 1; j < 8; ++j) c[j] -= l * __shfl_sync(kFull, c[j], b0 + k);
#pragma unroll
      for (int g = 8; g < 32; g += 8)
        if (b0 + g < 32) {
#pragma unroll
          for (int j = g; j < g + 8; ++j) c[j] -= l * __shfl_sync(kFull, c[j], b0 + k);
        }
      if (lane > b0 + k) c[k] = l;
      if (lane == b0 + k) c[k] = inv;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      uj[lane * XP + b0 + k] = c[k];
      lj[(b0 + k) * 32 + lane] = c[k];
      if (lane < w && b0 + k < w) dst[(b0 + k) * ldd] = c[k];
    }
#pragma unroll
    for (int j = 0; j < 24; ++j) c[j] = c[j + 8];
  }
}

// The same in FP64 for a block that no other work of the CTA can hide (the first
// one; all of a tail of up to 32): its columns dealt to four warps, one per
// scheduler.  The FMAs of 32 columns hold one scheduler's FP64 unit for 32 k cycles,
// and with the 32 reciprocals one warp took 73 k, four take 37 k; the elements'
// operations and their order are the same.  (In FP32 one warp is faster than 32
// barriers: 14 k.)  All threads; begins with the block in uj (warp 0's) and ends
// without a barrier.
template <class T>
__device__ __forceinline__ void lu_block_all(T* uj, T* lj, T* lbuf, T* dst, int64_t ldd, int w, int lane, int warp) {
  constexpr int NW = 4, NC = 32 / NW;   // warp v has columns v, v + NW, ..
  __syncthreads();
  T c[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    const int j = NW * q + warp;
    c[q] = warp < NW && lane < w && j < w ? uj[lane * XP + j] : j == lane ? T(1) : T(0);
  }
  __syncthreads();   // (read by all before columns go back)
#pragma unroll
  for (int kk = 0; kk < NC; ++kk) {
#pragma unroll 1
    for (int v = 0; v < NW; ++v) {
      const int k = NW * kk + v;
      T* lk = lbuf + 32 * (k & 1);
      if (warp == v) {
        const T inv = T(1) / __shfl_sync(kFull, c[kk], k);
        const T l = lane > k ? c[kk] * inv : T(0);
        lk[lane] = l;
        if (lane > k) c[kk] = l;
        if (lane == k) c[kk] = inv;
      }
      __syncthreads();
      if (warp < NW) {
        const T l = lk[lane];
        if (warp > v) c[kk] -= l * __shfl_sync(kFull, c[kk], k);
#pragma unroll
        for (int q = kk + 1; q < NC; ++q) c[q] -= l * __shfl_sync(kFull, c[q], k);
      }
    }
  }
  if (warp < NW) {
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      const int j = NW * q + warp;
      uj[lane * XP + j] = c[q];
      lj[j * 32 + lane] = c[q];
      if (lane < w && j < w) dst[j * ldd] = c[q];
    }
  }
}

// c := c U^-1 for a row c (U by rows at tri, inverse pivots on its diagonal),
// or c := L^-1 c for a column c (UNIT; L by columns at tri); pitch TP.  out(i,
// v): entry i's eight results from i on.
template <class T, bool UNIT, int TP, class Out>
__device__ __forceinline__ void tri_solve(T (&c)[32], const T* tri, Out out) {
#pragma unroll 1
  for (int b0 = 0; b0 < 32; b0 += 8) {
    const T* t = tri + b0 * TP + b0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      T r[8];
#pragma unroll
      for (int g = 0; g < 8; g += 4) {
        T q[4];
        load4(t + k * TP + g, q);
#pragma unroll
        for (int u = 0; u < 4; ++u) r[g + u] = q[u];
      }
      if (!UNIT) c[k] *= r[k];
#pragma unroll
      for (int j = k + 1; j < 8; ++j) c[j] -= c[k] * r[j];
#pragma unroll
      for (int g = 8; g < 32; g += 4)
        if (b0 + g < 32) {
          T q[4];
          load4(t + k * TP + g, q);
#pragma unroll
          for (int u = 0; u < 4; ++u) c[g + u] -= c[k] * q[u];
        }
    }
    out(b0, c);
#pragma unroll
    for (int j = 0; j < 24; ++j) c[j] = c[j + 8];
  }
}

// 32 x 32 blocks of the trailing update in a warp's registers as 4 x 8 tiles:
// lane (ty, tx) = (lane / 4, lane % 4) has rows 4 ty .. 4 ty + 3 and columns
// 8 tx .. 8 tx + 7.  A column of the left operand and a row of the right one
// then cost three 16-byte shared-memory reads per 32 FP32 FMAs (a row per lane
// needs eight, which bound the update at half the FMA rate); FP32 FMAs in
// pairs.  mul: C -= L X with L [k][LP] and X [k][UP].
template <class T, bool TF> struct Tile;

template <> struct Tile<float, false> {
  static constexpr int LP = 32, UP = 32, CW = 32;   // pitches, columns
  f2 x[4][4];
  __device__ __forceinline__ void load(const float* D, int64_t ldd, int cols, int lane) {   // D: the block's corner
    const float* p = D + (8 * (lane & 3)) * ldd + 4 * (lane >> 2);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float a[4] = {0.f, 0.f, 0.f, 0.f}, b[4] = {0.f, 0.f, 0.f, 0.f};
      if (8 * (lane & 3) + 2 * q < cols) load4(p + (2 * q) * ldd, a);
      if (8 * (lane & 3) + 2 * q + 1 < cols) load4(p + (2 * q + 1) * ldd, b);
#pragma unroll
      for (int i = 0; i < 4; ++i) x[i][q] = pack2(a[i], b[i]);
    }
  }
  __device__ __forceinline__ void store(float* D, int64_t ldd, int cols, int lane) const {
    float* p = D + (8 * (lane & 3)) * ldd + 4 * (lane >> 2);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) unpack2(x[i][q], a[i], b[i]);
      if (8 * (lane & 3) + 2 * q < cols) store4(p + (2 * q) * ldd, a);
      if (8 * (lane & 3) + 2 * q + 1 < cols) store4(p + (2 * q + 1) * ldd, b);
    }
  }
  __device__ __forceinline__ void to_rows(float* X, int lane) const {   // row-major, pitch XP
    float* p = X + 4 * (lane >> 2) * XP + 8 * (lane & 3);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      *reinterpret_cast<ulonglong2*>(p + i * XP) = make_ulonglong2(x[i][0], x[i][1]);
      *reinterpret_cast<ulonglong2*>(p + i * XP + 4) = make_ulonglong2(x[i][2], x[i][3]);
    }
  }
  __device__ __forceinline__ void mul(const float* L, const float* X, int lane) {
    const float* lp = L + 4 * (lane >> 2);
    const float* xp = X + 8 * (lane & 3);
#pragma unroll 4
    for (int k = 0; k < 32; ++k) {
      float l[4];
      load4(lp + LP * k, l);
      const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(xp + UP * k);
      const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(xp + UP * k + 4);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const f2 a = pack2(-l[i], -l[i]);
        x[i][0] = fma2(a, v.x, x[i][0]);
        x[i][1] = fma2(a, v.y, x[i][1]);
        x[i][2] = fma2(a, u.x, x[i][2]);
        x[i][3] = fma2(a, u.y, x[i][3]);
      }
    }
  }
};

// FP64: half a block, 32 x 16, as 4 x 4 tiles.
template <> struct Tile<double, false> {
  static constexpr int LP = 32, UP = 32, CW = 16;
  double x[4][4];
  __device__ __forceinline__ void load(const double* D, int64_t ldd, int cols, int lane) {
    const double* p = D + (4 * (lane & 3)) * ldd + 4 * (lane >> 2);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      double a[4] = {0.0, 0.0, 0.0, 0.0};
      if (4 * (lane & 3) + q < cols) load4(p + q * ldd, a);
#pragma unroll
      for (int i = 0; i < 4; ++i) x[i][q] = a[i];
    }
  }
  __device__ __forceinline__ void store(double* D, int64_t ldd, int cols, int lane) const {
    double* p = D + (4 * (lane & 3)) * ldd + 4 * (lane >> 2);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double a[4] = {x[0][q], x[1][q], x[2][q], x[3][q]};
      if (4 * (lane & 3) + q < cols) store4(p + q * ldd, a);
    }
  }
  __device__ __forceinline__ void to_rows(double* X, int lane) const {
    double* p = X + 4 * (lane >> 2) * XP + 4 * (lane & 3);
#pragma unroll
    for (int i = 0; i < 4; ++i) store4(p + i * XP, x[i]);
  }
  __device__ __forceinline__ void mul(const double* L, const double* X, int lane) {
    const double* lp = L + 4 * (lane >> 2);
    const double* xp = X + 4 * (lane & 3);
#pragma unroll 4
    for (int k = 0; k < 32; ++k) {
      double l[4], v[4];
      load4(lp + LP * k, l);
      load4(xp + UP * k, v);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) x[i][q] = fma(-l[i], v[q], x[i][q]);
    }
  }
};

// The same block as mma.m16n8k8 fragments: each operand x = hi + lo with hi =
// tf32(x), lo = tf32(x - hi), products hi hi + hi lo + lo hi, FP32 sums.
template <> struct Tile<float, true> {
  static constexpr int LP = 36, UP = 36, CW = 32;   // (fragment reads of four rows at a time)
  float c[2][4][4];
  template <class F> __device__ __forceinline__ void each(int lane, F f) {
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int e = 0; e < 4; ++e) f(mt * 16 + (lane >> 2) + (e >> 1) * 8, q * 8 + 2 * (lane & 3) + (e & 1), c[mt][q][e]);
  }
  __device__ __forceinline__ void load(const float* D, int64_t ldd, int cols, int lane) {
    each(lane, [&](int i, int j, float& v) { v = j < cols ? D[j * ldd + i] : 0.f; });
  }
  __device__ __forceinline__ void store(float* D, int64_t ldd, int cols, int lane) {
    each(lane, [&](int i, int j, float& v) {
      if (j < cols) D[j * ldd + i] = v;
    });
  }
  __device__ __forceinline__ void to_rows(float* X, int lane) {
    each(lane, [&](int i, int j, float& v) { X[i * XP + j] = v; });
  }
  __device__ __forceinline__ void mul(const float* L, const float* X, int lane) {
    const int g = lane >> 2, t = lane & 3;
#pragma unroll 1
    for (int k0 = 0; k0 < 32; k0 += 8) {
      uint32_t ah[2][4], al[2][4], bh[4][2], bl[4][2];
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int e = 0; e < 4; ++e)
          split_tf32(-L[(k0 + t + (e >> 1) * 4) * LP + mt * 16 + g + (e & 1) * 8], ah[mt][e], al[mt][e]);
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int e = 0; e < 2; ++e) split_tf32(X[(k0 + t + 4 * e) * UP + q * 8 + g], bh[q][e], bl[q][e]);
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          mma_tf32(c[mt][q], al[mt], bh[q]);
          mma_tf32(c[mt][q], ah[mt], bl[q]);
          mma_tf32(c[mt][q], ah[mt], bh[q]);
        }
    }
  }
};

// The head's factors in shared memory (Hv), by dependency levels; each
// thread's first op of the next level is loaded ahead of the barrier.
template <class T>
__device__ __forceinline__ void head_program() {
  const Args& A = args();
  T* Hv = at<T>(A.p.o_hv);
  const int* w = A.w;
  const int4* ops = reinterpret_cast<const int4*>(w + A.hop);
  const int tid = threadIdx.x, nthr = blockDim.x, parts = 2 * A.n_hlev;
  int o0 = 0, o1 = parts > 0 ? __ldg(w + A.hop_ptr + 1) : 0;
  int4 first = tid < o1 ? __ldg(ops + tid) : make_int4(0, 0, 0, 0);
  for (int l = 0; l < parts; ++l) {
    const int o2 = l + 1 < parts ? __ldg(w + A.hop_ptr + l + 2) : o1;
    auto run = [&](const int4& op) {
      const int dst = op.x & 0xFFFF, piv = (uint32_t)op.x >> 16;
      T v = Hv[dst];
      for (int t = op.y; t < op.z; t += 4) {
        uint32_t tm[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) tm[u] = t + u < op.z ? (uint32_t)__ldg(w + A.hterm + t + u) : 0u;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (t + u < op.z) v -= Hv[tm[u] & 0xFFFF] * Hv[tm[u] >> 16];
      }
      if (!(l & 1)) v = T(1) / v;
      else if (piv != 0xFFFF) v *= Hv[piv];
      Hv[dst] = v;
    };
    int o = o0 + tid;
    if (o < o1) run(first);
    for (o += nthr; o < o1; o += 4 * nthr) {
      int4 op[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (o + u * nthr < o1) op[u] = __ldg(ops + o + u * nthr);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (o + u * nthr < o1) run(op[u]);
    }
    o0 = o1;
    o1 = o2;
    if (o0 + tid < o1) first = __ldg(ops + o0 + tid);
    __syncthreads();
  }
}

// The tail before elimination (Jacobian entries and the head's Schur
// complement) into its place in the packed factors.  A warp forms kGroup
// columns at a time in its own shared tile, so that the warps' loads overlap
// and no barrier separates the steps.
template <class T>
__device__ __forceinline__ void assemble_tail() {
  const Args& A = args();
  const int* w = A.w;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, pitch = A.pitch;
  const int nt = A.d.n - A.d.head, groups = (nt + kGroup - 1) / kGroup, nwa = A.p.asm_warps;
  const int64_t ldd = A.d.ldd;
  T* X = at<T>(A.p.o_x) + warp * A.p.asm_tile;
  const T* Hv = at<T>(A.p.o_hv);
  const T* mbuf = static_cast<const T*>(scalars().mbuf);
  T* D = static_cast<T*>(scalars().P) + A.d.p_d;
  if (warp >= nwa) return;
  for (int G = warp; G < groups; G += nwa) {
    for (int e = lane * (16 / (int)sizeof(T)); e < A.p.asm_tile; e += 32 * (16 / (int)sizeof(T)))
      *reinterpret_cast<float4*>(X + e) = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncwarp();
    {
      const int* gp = w + A.jg_grp + G + 1;
      const int e1 = 32 * __ldg(gp + 1), l0 = __ldg(w + A.jd_grp + G + 1), l1 = __ldg(w + A.jd_grp + G + 2);
#pragma unroll 4
      for (int e = 32 * __ldg(gp) + lane; e < e1; e += 32) {
        const int p = __ldg(w + A.jg_dst + e);
        const T v = mbuf[e];
        if (p >= 0) X[p] = v;
      }
      for (int q = l0 + lane; q < l1; q += 32) {   // long entries: {position, index}
        const int2 t = __ldg(reinterpret_cast<const int2*>(w + A.jd_ent) + q);
        X[t.x] = mbuf[32 * A.n_jsl + t.y];
      }
    }
    __syncwarp();
    // the group's targets: a stream of rows of words, per slice {position |
    // terms << 16}, then the terms; kRows rows in flight ahead of their use
    {
      constexpr int kRows = 12;
      const int r1 = __ldg(w + A.tg_grp + G + 1);
      int r = __ldg(w + A.tg_grp + G);
      const int* q = w + A.tg_ent + lane;
      uint32_t t[kRows];
#pragma unroll
      for (int u = 0; u < kRows; ++u) t[u] = r + u < r1 ? (uint32_t)__ldg(q + 32 * (r + u)) : 0xFFFFu;
      T a = T(0);
      uint32_t pos = 0xFFFFu;
      int left = 0;
      for (; r < r1 + 1; r += kRows) {   // (one row more: the last slice's result)
        uint32_t nx[kRows];
#pragma unroll
        for (int u = 0; u < kRows; ++u) nx[u] = r + kRows + u < r1 ? (uint32_t)__ldg(q + 32 * (r + kRows + u)) : 0xFFFFu;
#pragma unroll
        for (int u = 0; u < kRows; ++u) {
          if (left > 0) {
            a += Hv[t[u] & 0xFFFF] * Hv[t[u] >> 16];
            --left;
          } else {
            if (pos != 0xFFFFu) X[pos] -= a;
            pos = t[u] & 0xFFFF;
            left = (int)(t[u] >> 16);
            a = T(0);
          }
        }
#pragma unroll
        for (int u = 0; u < kRows; ++u) t[u] = nx[u];
      }
      if (pos != 0xFFFFu && left == 0) X[pos] -= a;
    }
    __syncwarp();
#pragma unroll
    for (int c = 0; c < kGroup; ++c)
      if (kGroup * G + c < nt) {
        T* col = D + (kGroup * G + c) * ldd;
#pragma unroll 4
        for (int r = lane; r < nt; r += 32) col[r] = X[c * pitch + r];
      }
    __syncwarp();
  }
}

// LU of the tail, right-looking by 32-column panels on the packed factors (in
// L2): per panel the rows below the diagonal block and the block row right of
// it are solved block by block, every warp a block at a time, and kept in
// shared memory for the trailing update, whose blocks the warps take in turn.
// The block that holds the next panel's diagonal comes first and is factorised
// at once by the warp that updated it, while the others go on.  Against a
// left-looking form (a chain of a product and a triangular solve per pair of
// blocks: 55 links for 11 block columns against 11 here) this reads and writes
// the trailing blocks, 3 MB of L2 traffic per 349-column tail.
struct TailView {
  int nt, nb, lane, warp, nw;
  int64_t ldd;
  __device__ __forceinline__ TailView() {
    const Args& A = args();
    nt = A.d.n - A.d.head;
    nb = A.nb;
    ldd = A.d.ldd;
    lane = threadIdx.x & 31;
    warp = threadIdx.x >> 5;
    nw = blockDim.x >> 5;
  }
  template <class T> __device__ __forceinline__ T* block(int r, int j) const {
    return static_cast<T*>(scalars().P) + args().d.p_d + (32 * j) * ldd + 32 * r;
  }
  __device__ __forceinline__ int width(int j) const { return min(32, nt - 32 * j); }
};

// L of the blocks below the diagonal block J and U of the blocks right of it.
template <class T, bool TF>
__device__ __forceinline__ void solve_panel(int J) {
  constexpr int LP = Tile<T, TF>::LP, UP = Tile<T, TF>::UP;
  const Args& A = args();
  const TailView v;
  const int64_t ldd = v.ldd;
  const int lane = v.lane, m = v.nb - 1 - J;   // block rows below, block columns to the right
  for (int q = v.warp; q < 2 * m; q += v.nw) {
    T c[32];
    if (q < m) {   // rows of block (J + 1 + q, J), a row per lane
      const int r = J + 1 + q;
      T* p = v.block<T>(r, J) + lane;
      {   // (rows past the tail's end are padding)
        const T* s = p;
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          c[j] = ld_here(s);
          s += ldd;
        }
      }
      T* o = at<T>(A.p.o_lp) + (r - 1) * 32 * LP + lane;
      tri_solve<T, false, XP>(c, at<T>(A.p.o_uj), [&](int, const T(&x)[32]) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          *o = x[k];
          *p = x[k];
          o += LP;
          p += ldd;
        }
      });
    } else {   // columns of block (J, j), a column per lane
      const int j = J + 1 + q - m;
      const bool in = lane < v.width(j);
      T* p = v.block<T>(J, j) + (in ? lane : 0) * ldd;   // (lanes past the last column: not stored)
#pragma unroll
      for (int i = 0; i < 32; i += 4) {
        T x[4];
        load4(p + i, x);
#pragma unroll
        for (int u = 0; u < 4; ++u) c[i + u] = x[u];
      }
      T* o = at<T>(A.p.o_up) + (j - 1) * 32 * UP + lane;
      tri_solve<T, true, 32>(c, at<T>(A.p.o_lj), [&](int b0, const T(&x)[32]) {
        const T lo[4] = {x[0], x[1], x[2], x[3]}, hi[4] = {x[4], x[5], x[6], x[7]};
        if (in) {
          store4(p + b0, lo);
          store4(p + b0 + 4, hi);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) o[(b0 + k) * UP] = x[k];
      });
    }
  }
}

template <class T, bool TF>
__device__ __forceinline__ void factor_tail() {
  using Tl = Tile<T, TF>;
  constexpr int LP = Tl::LP, UP = Tl::UP, CW = Tl::CW, HB = 32 / CW;
  const Args& A = args();
  const TailView v;
  const int lane = v.lane, nb = v.nb;
  int* next = at<int>(A.p.o_next);
  auto take = [&]() {
    int t = 0;
    if (lane == 0) t = atomicAdd(next, 1);
    return __shfl_sync(kFull, t, 0);
  };
  for (int J = -1; J + 1 < nb; ++J) {
    const int m = nb - 1 - J;
    const T* Lp = at<T>(A.p.o_lp) + J * 32 * LP;   // of block row J + 1
    const T* Up = at<T>(A.p.o_up) + J * 32 * UP;
    if (J >= 0) {
      __syncthreads();
      if (threadIdx.x == 0) *next = HB;   // (the first block is warp 0's)
      solve_panel<T, TF>(J);
      __syncthreads();
      PHASE_MARK(PH_PANEL);
    }
    if (v.warp == 0) {
      // the next diagonal block: updated, and factorised at once
      T *uj = at<T>(A.p.o_uj), *D = v.block<T>(J + 1, J + 1);
      const int w = v.width(J + 1);
#pragma unroll 1
      for (int h = 0; h < HB; ++h) {
        Tl x;
        x.load(D + (CW * h) * v.ldd, v.ldd, w - CW * h, lane);
        if (J >= 0) x.mul(Lp, Up + CW * h, lane);
        x.to_rows(uj + CW * h, lane);
      }
      __syncwarp();
      if (sizeof(T) == 4 || J >= 0) lu_block(uj, at<T>(A.p.o_lj), D + lane, v.ldd, w, lane);
    }
    if (J < 0) {
      if constexpr (sizeof(T) == 8) lu_block_all(at<T>(A.p.o_uj), at<T>(A.p.o_lj), at<T>(A.p.o_lbuf), v.block<T>(0, 0) + lane, v.ldd,
                                                 v.width(0), lane, v.warp);
      PHASE_MARK(PH_PANEL);
      continue;
    }
    // the other trailing blocks in turn, by columns
    const int mm = m * m * HB;
    auto corner = [&](int t) { return v.block<T>(J + 1 + t / HB % m, J + 1 + t / HB / m) + (CW * (t % HB)) * v.ldd; };
    auto cols = [&](int t) { return v.width(J + 1 + t / HB / m) - CW * (t % HB); };
    int t = take();
    Tl x;
    if (t < mm) x.load(corner(t), v.ldd, cols(t), lane);
    while (t < mm) {
      const T *lp = Lp + (t / HB % m) * 32 * LP, *up = Up + (t / HB / m) * 32 * UP + CW * (t % HB);
      if constexpr (sizeof(T) == 4) {
        const int u = take();
        Tl y;   // the next block is on its way while this one is worked on
        if (u < mm) y.load(corner(u), v.ldd, cols(u), lane);
        x.mul(lp, up, lane);
        x.store(corner(t), v.ldd, cols(t), lane);
        x = y;
        t = u;
      } else {   // (a block's FP64 products take a hundred times its loads)
        x.mul(lp, up, lane);
        x.store(corner(t), v.ldd, cols(t), lane);
        t = take();
        if (t < mm) x.load(corner(t), v.ldd, cols(t), lane);
      }
    }
    PHASE_MARK(PH_UPDATE);
  }
  __syncthreads();
}

// Jacobian at the predicted state, M = I - gamma J and its packed factors.
// y (= predicted state) is restored at the end.

// First the Jacobian: -gamma dR_j/dx in a shared table, then M's entries in
// program order into mbuf (global scratch).
template <class T>
__device__ __forceinline__ void cell_jacobian() {
  const Args& A = args();
  const Dev& d = A.d;
  const CellS& S = scalars();
  const int n = d.n, n_r = d.n_r, tid = threadIdx.x, nthr = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nw = nthr >> 5;
  const int* w = A.w;
  double* dR = at<double>(A.p.o_dr);
  float* wsf = at<float>(A.p.o_wsf);
  float* wif = at<float>(A.p.o_wif);
  const double* yp = at<double>(A.p.o_yp);
  const double* kc = S.kc;
  T* mbuf = static_cast<T*>(S.mbuf);
  const double gamma = S.gam;
  // dR_j/dx for every reactant
  const int2* rx = reinterpret_cast<const int2*>(w + A.rx);
#pragma unroll 4
  for (int j = tid; j < n_r; j += nthr) {
    const int2 r = __ldg(rx + j);
    const double kv = kc[j];
    const int b = (uint32_t)r.x >> 16;
    dR[r.y] = b != 0xFFFF ? kv * yp[b] : kv;
    if (b != 0xFFFF) dR[r.y + 1] = kv * yp[r.x & 0xFFFF];
  }
  if (tid == 0) dR[A.n_slot] = 0.0;
  if constexpr (sizeof(T) == 4) {
    const double* ws = at<double>(A.p.o_ws);
    double *wf = at<double>(A.p.o_wf), *wi = at<double>(A.p.o_wi);
    for (int s = tid; s < n; s += nthr) {
      const double wv = ws[s], iv = 1.0 / wv;
      wf[s] = wv;
      wi[s] = iv;
      wsf[s] = (float)wv;
      wif[s] = (float)iv;
    }
  }
  __syncthreads();
  auto m_value = [&](int rc, double acc) {   // M (W M W^-1 in FP32) at (row species, column species)
    const int i = rc & 0xFFFF, l = (uint32_t)rc >> 16;
    const double m = fma(-gamma, acc, i == l ? 1.0 : 0.0);
    if constexpr (sizeof(T) == 4) return T((float)m * (wsf[i] * wif[l]));
    else return T(m);
  };
  // entries of at most kJShort words, four slices at a time, all their index
  // words in flight at once
  {
    const int4* off = reinterpret_cast<const int4*>(w + A.jg_off);
    const int* p = w + A.jg_ent + lane;
    int s = 4 * warp;
    int4 m0 = make_int4(0, 0, 0, 0), m1 = m0;
    if (s < A.n_jsl) {
      m0 = __ldg(off + s / 2);
      m1 = __ldg(off + s / 2 + 1);
    }
    for (; s < A.n_jsl; s += 4 * nw) {
      const int of[4] = {m0.x, m0.z, m1.x, m1.z}, len[4] = {m0.y, m0.w, m1.y, m1.w};
      int rc[4], t[kJShort][4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        rc[u] = __ldg(w + A.jg_rc + 32 * (s + u) + lane);
#pragma unroll
        for (int e = 0; e < kJShort; ++e) t[e][u] = e < len[u] ? __ldg(p + 32 * (of[u] + e)) : A.n_slot;
      }
      if (s + 4 * nw < A.n_jsl) {
        m0 = __ldg(off + (s + 4 * nw) / 2);
        m1 = __ldg(off + (s + 4 * nw) / 2 + 1);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        // the first word's coefficient is +-1; most slices end there
        const double v = dR[t[0][u] & 0xFFFF];
        double a = __hiloint2double(__double2hiint(v) ^ (t[0][u] & 0x80000000), __double2loint(v));
        if (len[u] > 1) {
          double x[kJShort];
#pragma unroll
          for (int e = 1; e < kJShort; ++e) x[e] = dR[t[e][u] & 0xFFFF];
#pragma unroll
          for (int e = 1; e < kJShort; ++e)
            asm volatile("fma.rn.f64 %0, %1, %2, %0;" : "+d"(a) : "d"(coef(t[e][u])), "d"(x[e]));   // (not ahead of the branch)
        }
        if (len[u] > 0) mbuf[32 * (s + u) + lane] = m_value(rc[u], a);
      }
    }
  }
  // the entries of more words: a chain per lane, of up to kJLong words of an
  // entry or of every 32nd word of a longer one
  {
    const int2* off = reinterpret_cast<const int2*>(w + A.jl_off);
    for (int s = nw - 1 - warp; s < A.n_jl; s += nw) {
      const int2 mt = __ldg(off + s);
      const int* q = w + A.jl_ent + 32 * mt.x + lane;
      const int m = mt.y, rc = __ldg(w + A.jl_rc + 32 * s + lane);
      int t[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) t[u] = u < m ? __ldg(q + 32 * u) : 0;
      double a = 0.0;
      int e = 4;
      for (; e <= m; e += 4) {
        int nx[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) nx[u] = e + u < m ? __ldg(q + 32 * (e + u)) : 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) a = fma(coef(t[u]), dR[t[u] & 0xFFFF], a);
#pragma unroll
        for (int u = 0; u < 4; ++u) t[u] = nx[u];
      }
#pragma unroll 1
      for (e -= 4; e < m; ++e) {
        a = fma(coef(t[0]), dR[t[0] & 0xFFFF], a);
        t[0] = t[1];
        t[1] = t[2];
      }
      if (s < A.n_jw) a = warp_sum(a);
      mbuf[32 * (A.n_jsl + s) + lane] = m_value(rc, a);
    }
  }
  if (d.therm) {
    // sum_j dn_j dR_j/dx_l per species, kept in the border's row
    __syncthreads();
    for (int j = tid; j < n_r; j += nthr) {
      const double dn = __ldg(d.th_dn + j);
      const int2 r = __ldg(rx + j);
      dR[r.y] *= dn;
      if ((uint32_t)r.x >> 16 != 0xFFFF) dR[r.y + 1] *= dn;
    }
    __syncthreads();
    row_sums(w, A.vp_deal, A.vp_ent, A.vp_dst, A.vrow, A.vrow_more, dR, at<double>(A.p.o_vp),
             d.bgv + S.oc * d.bpad, n);
  }
  __syncthreads();
  PHASE_MARK(PH_JAC);
}

// The head's entries of M into shared memory, their factors, and those out.
template <class T>
__device__ __forceinline__ void cell_head() {
  const Args& A = args();
  const int tid = threadIdx.x, nthr = blockDim.x, p_d = A.d.p_d;
  const int* w = A.w;
  T* Hv = at<T>(A.p.o_hv);
  const T* mbuf = static_cast<const T*>(scalars().mbuf);
  for (int e = tid; e <= p_d; e += nthr) Hv[e] = T(0);
  __syncthreads();
  {
    const int s1 = __ldg(w + A.jg_grp + 1);
#pragma unroll 4
    for (int e = tid; e < 32 * s1; e += nthr) {
      const int p = __ldg(w + A.jg_dst + e);
      const T v = mbuf[e];
      if (p >= 0) Hv[p] = v;
    }
    const int q1 = __ldg(w + A.jd_grp + 1);
    for (int e = tid; e < q1; e += nthr) {
      const int2 t = __ldg(reinterpret_cast<const int2*>(w + A.jd_ent) + e);
      Hv[t.x] = mbuf[32 * A.n_jsl + t.y];
    }
  }
  __syncthreads();
  head_program<T>();
  T* P = static_cast<T*>(scalars().P);
  for (int e = tid; e < p_d; e += nthr) P[e] = Hv[e];
  PHASE_MARK(PH_HEAD);
}

template <class T, bool TF>
__device__ __forceinline__ void cell_refresh() {
  cell_jacobian<T>();
  cell_head<T>();
  assemble_tail<T>();
  __syncthreads();
  PHASE_MARK(PH_ASSEMBLE);
  factor_tail<T, TF>();
  const Args& A = args();
  for (int s = threadIdx.x; s < A.d.n; s += blockDim.x) at<double>(A.p.o_ys)[s] = at<double>(A.p.o_yp)[s];
  if (threadIdx.x == 0) {
    CellS& S = scalars();
    S.gam_J = S.gam;
    S.j_age = 0;
    S.crate = 1.0;
    S.flags &= ~F_NEED_J;
    S.jac_evals += 1;
  }
  __syncthreads();
}

// The substitution's vector by species: x_put scales the right-hand side by
// the factorisation's weights (FP32), x_get undoes it.
template <class T>
__device__ __forceinline__ double x_get(const Args& A, int s) {
  const int p = at<uint16_t>(A.p.o_ip)[s];
  const double v = (double)(p < A.d.head ? at<T>(A.p.o_xh)[p] : at<T>(A.p.o_xt)[p - A.d.head]);
  if constexpr (sizeof(T) == 4) {
    // v / w: from the rounded reciprocal, corrected by the quotient's residual
    const double w = at<double>(A.p.o_wf)[s], iw = at<double>(A.p.o_wi)[s], q = v * iw;
    return fma(fma(-q, w, v), iw, q);
  } else {
    return v;
  }
}
template <class T>
__device__ __forceinline__ void x_put(const Args& A, int s, double b) {
  if constexpr (sizeof(T) == 4) b *= at<double>(A.p.o_wf)[s];
  const int p = at<uint16_t>(A.p.o_ip)[s];
  if (p < A.d.head) at<T>(A.p.o_xh)[p] = T(b);
  else at<T>(A.p.o_xt)[p - A.d.head] = T(b);
}

// Temperature border of a refreshed Newton matrix (T eliminated last): with
// u = dF/dT, v = d f_t/dx and w = d f_t/dT at the predicted state,
// z = M^-1 (-gJ u) and s = 1 - gJ w + gJ v.z; a residual (r, r_T) then has the
// correction (a0 - z b, b), a0 = M^-1 r, b = (r_T + gJ v.a0) / s.
template <class T>
__device__ __forceinline__ void cell_border() {
  const Args& A = args();
  const Dev& d = A.d;
  const CellS& S = scalars();
  const double* yp = at<double>(A.p.o_yp);
  const double* fs = at<double>(A.p.o_fs);
  double* tab = at<double>(A.p.o_r);
  double* red = at<double>(kCellRed);
  const double nH = S.nH;
  const int n = d.n, n_r = d.n_r, t = d.t_idx, tid = threadIdx.x, nthr = blockDim.x;
  const double Tc = yp[t], it = 1.0 / Tc;
  // R_j, and R_j d ln k'_j/dT into the table
  auto rate = [&](int j) {
    const int ab = __ldg(A.w + A.rx + 2 * j);
    double R = S.kc[j] * yp[ab & 0xFFFF];
    if ((uint32_t)ab >> 16 != 0xFFFF) R *= yp[(uint32_t)ab >> 16];
    return R;
  };
  for (int j = tid; j < n_r; j += nthr) {
    const RatePar p = d.rpar[j];
    const int cls = (int)p.w;
    tab[j] = cls == SM_TWO_BODY || cls == SM_DISS_RECOMB ? rate(j) * ((p.y + p.z * it) * it) : 0.0;
  }
  if (tid == 0) tab[n_r] = 0.0;
  __syncthreads();
  row_sums(A.w, A.rp_deal, A.rp_ent, A.rp_dst, A.row, A.row_more, tab, at<double>(A.p.o_part),
           at<double>(A.p.o_fs), n);
  sum_parts(0, n_r, [&](int j) { return __ldg(d.th_dn + j) * rate(j); });
  sum_parts(1, n_r, [&](int j) { return __ldg(d.th_dn + j) * tab[j]; });
  sum_parts(2, n, [&](int i) { return i == t ? 0.0 : yp[i]; });
  sum_parts(3, d.n_cool, [&](int q) {
    const int i = __ldg(d.th_cool + q);
    return yp[i] * (d.th_L[i] * exp(-d.th_E[i] * it));
  });
  sum_parts(4, d.n_cool, [&](int q) {
    const int i = __ldg(d.th_cool + q);
    return yp[i] * (d.th_L[i] * exp(-d.th_E[i] * it)) * (d.th_E[i] * it * it);
  });
  __syncthreads();
  const double gJ = S.gam_J;
  if (tid < 32) {
    const double F = sum_total(0, n_r), U = sum_total(1, n_r), xt = sum_total(2, n), line = sum_total(3, d.n_cool),
                 dline = sum_total(4, d.n_cool);
    const double i15x = 1.0 / (1.5 * xt);
    const double fT = (d.th_heat - nH * line - d.th_lam * nH * (Tc - d.th_Td) - 1.5 * Tc * F) * i15x;
    const double w = (-nH * dline - d.th_lam * nH - 1.5 * F - 1.5 * Tc * U) * i15x;
    red[kRedX] = i15x;
    red[kRedX + 1] = fT / xt;
    red[kRedX + 2] = w;
  }
  solve_prefetch<T>();
  for (int s = tid; s < n; s += nthr) x_put<T>(A, s, s == t ? 0.0 : -gJ * fs[s]);
  cell_solve<T>();
  const double i15x = red[kRedX], fTx = red[kRedX + 1], w = red[kRedX + 2];
  double* bz = d.bz + S.oc * d.bpad;
  double* bgv = d.bgv + S.oc * d.bpad;
  sum_parts(0, n, [&](int s) {
    double z = 0.0, gv = 0.0;
    if (s != t) {
      z = x_get<T>(A, s);
      const double cl = d.th_L[s] > 0.0 ? d.th_L[s] * exp(-d.th_E[s] * it) : 0.0;
      gv = (-nH * cl - 1.5 * Tc * bgv[s]) * i15x - fTx;
    }
    bz[s] = z;
    bgv[s] = gJ * gv;
    return gv * z;
  });
  __syncthreads();
  if (tid < 32) {
    const double vz = sum_total(0, n);
    if (tid == 0) d.bs[S.oc] = 1.0 - gJ * w + gJ * vz;
  }
  for (int s = tid; s < n; s += nthr) at<double>(A.p.o_ys)[s] = yp[s];
  __syncthreads();
}

// The clock cycles of the timed class (sm_opts.timing_kind), by thread 0.
__device__ __forceinline__ void class_begin(int kind) {
  if (args().timing_kind == kind && threadIdx.x == 0) scalars().t0 = clock64();
}
__device__ __forceinline__ void class_end(int kind) {
  if (args().timing_kind == kind && threadIdx.x == 0) {
    atomicAdd(args().timing, (double)(clock64() - scalars().t0));
    atomicAdd(args().timing + 1, 1.0);
  }
}

__device__ __forceinline__ void cell_predict() {
  const Args& A = args();
  const Dev& d = A.d;
  CellS& S = scalars();
  const int n = d.n, tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5;
  __syncthreads();   // every thread has taken the last attempt's outcome from S
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
      // lanes 0..q: the predictor on q + 1 points; lanes 16..: the order
      // q - 1 predictor on q points, which the error test may rate
      const int i = lane & 15, np = lane < 16 ? qq + 1 : qq;
      if (state == 3 && nh > 1 && i < np) {
        double num = 1.0, den = 1.0;
        const double ti = S.tn[i];
        for (int j = 0; j < np; ++j)
          if (j != i) {
            num *= tnew - S.tn[j];
            den *= ti - S.tn[j];
          }
        (lane < 16 ? S.wts : S.wlo)[i] = num / den;
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
  if (S.state != 3) return;
  const double h = S.err;
  const int qo = S.q, nh = S.nh;
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
      Yp[i] = S.hist + (int64_t)slot * S.hn;
    }
    for (int s = tid; s < n; s += nthr) {
      const double y0 = Yp[0][s];
      double yp = euler ? y0 + h * d.f0[(int64_t)s * d.ld + S.c] : wt[0] * y0, pv = 0.0;
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
      at<double>(A.p.o_yp)[s] = yp;
      at<double>(A.p.o_ys)[s] = yp;
      at<double>(A.p.o_ps)[s] = pv;
      at<double>(A.p.o_ws)[s] = 1.0 / (d.rtol * fabs(y0) + d.atol);
    }
  }
  if (tid == 0) S.h = h;
  __syncthreads();
  class_end(SM_TIME_PREDICT);
  PHASE_MARK(PH_PREDICT);
}

// One Newton round after the right-hand side: FP64 residual, substitution,
// update, convergence test.
template <class T>
__device__ __forceinline__ void cell_newton() {
  const Args& A = args();
  const Dev& d = A.d;
  CellS& S = scalars();
  const int n = d.n, tid = threadIdx.x, nthr = blockDim.x;
  double* ys = at<double>(A.p.o_ys);
  double* red = at<double>(kCellRed);
  class_begin(SM_TIME_SOLVE);
  solve_prefetch<T>();   // in place of the rates, which are done with
  {
    const double* ps = at<double>(A.p.o_ps);
    const double* fs = at<double>(A.p.o_fs);
    const double a0 = S.alpha[0], inv_a0 = S.inv_a0, h = S.h;
    for (int s = tid; s < n; s += nthr) {
      const double b = -(a0 * ys[s] + ps[s] - h * fs[s]) * inv_a0;
      if (s == d.t_idx) red[kRedX + 3] = b;
      x_put<T>(A, s, b);
    }
  }
  cell_solve<T>();
  double bT = 0.0;
  const double* bz = nullptr;
  if (d.therm) {
    const double* bgv = d.bgv + S.oc * d.bpad;
    bz = d.bz + S.oc * d.bpad;
    sum_parts(0, n, [&](int s) { return s == d.t_idx ? 0.0 : bgv[s] * x_get<T>(A, s); });
    __syncthreads();
    if (tid < 32) {
      const double dot = sum_total(0, n);
      if (tid == 0) red[kRedX + 4] = (red[kRedX + 3] + dot) / d.bs[S.oc];
    }
    __syncthreads();
    bT = red[kRedX + 4];
  }
  const double scale = S.scale;
  const double* ws = at<double>(A.p.o_ws);
  sum_parts(1, n, [&](int s) {
    double del = x_get<T>(A, s);
    if (bz) del = s == d.t_idx ? bT : fma(-bz[s], bT, del);
    del *= scale;
    ys[s] += del;
    const double v = del * ws[s];
    return v * v;
  });
  __syncthreads();
  double acc = 0.0;
  if (tid < 32) acc = sum_total(1, n);
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
}

// Error test, step / order selection, history.
__device__ __forceinline__ void cell_finish() {
  const Args& A = args();
  const Dev& d = A.d;
  CellS& S = scalars();
  const int n = d.n, tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const double* ys = at<double>(A.p.o_ys);
  const double* yp = at<double>(A.p.o_yp);
  const double* ws = at<double>(A.p.o_ws);
  const double h = S.h, tnew = S.tnew;
  const int qo = S.q, nh = S.nh;
  class_begin(SM_TIME_FINISH);
  // the error and the neighbouring orders' estimates in one pass (the latter
  // count only if the step is accepted); one pow call serves the three step
  // factors, an order per lane
  const bool work = !(S.flags & F_FAILED);
  const bool due = work && S.n_at_q + 1 >= qo + 1;
  const bool lo = due && qo > 1;
  const bool hi = due && qo < d.q_max && (S.flags & F_HAS_EPREV) && nh + 1 >= qo + 2;
  double* nv = at<double>(A.p.o_nv);
  const int N = A.p.nv;
  if (work)
    for (int s = tid; s < n; s += nthr) {
      const double y = ys[s], dy = y - yp[s], wv = ws[s];
      nv[s] = dy * wv;
      if (lo) {
        double p = 0.0;
        for (int i = 0; i < qo; ++i) {
          int slot = S.base + i;
          if (slot > QMAX) slot -= QMAX + 1;
          p += S.wlo[i] * S.hist[(int64_t)slot * S.hn + s];
        }
        nv[N + s] = (y - p) * wv;
      }
      if (hi) nv[2 * N + s] = (dy - S.eprev[s]) * wv;
    }
  __syncthreads();
  if (warp == 0) {
    // eight lanes a norm, each every eighth term, then the eight in order: the
    // order of the class-by-class finish kernel (the step that follows depends
    // on the last bit)
    const int g = lane >> 3;
    double sq = 0.0;
    if (g == 0 ? work : g == 1 ? lo : g == 2 ? hi : false) {
      const double* p = nv + g * N;
#pragma unroll 8
      for (int s = lane & 7; s < n; s += 8) sq = fma(p[s], p[s], sq);
    }
    double tot = __shfl_sync(kFull, sq, 8 * g);
#pragma unroll
    for (int i = 1; i < 8; ++i) tot += __shfl_sync(kFull, sq, 8 * g + i);
    const double acc = __shfl_sync(kFull, tot, 0), acc_lo = __shfl_sync(kFull, tot, 8), acc_hi = __shfl_sync(kFull, tot, 16);
    const double err = work ? (nh >= qo + 1 ? h / (tnew - S.tn[qo]) : 1.0 / (qo + 1)) * sqrt(acc / n) : 0.0;
    const bool accepted = work && isfinite(err) && err <= 1.0;
    double base = err, ord = qo + 1, fac = 0.9;
    if (lane == 1 && lo) {
      base = h / (tnew - S.tn[qo - 1]) * sqrt(acc_lo / n);
      ord = qo;
      fac = 0.8;
    }
    if (lane == 2 && hi) {
      base = sqrt(acc_hi / n) / (qo + 2);
      ord = qo + 2;
      fac = 0.7;
    }
    // accepted: bounded below (a zero error must not stop the step's growth)
    double eta = 0.0;
    if (work && isfinite(err)) eta = fac * pow(accepted ? fmax(base, 1e-10) : base, -1.0 / ord);
    const double e1 = __shfl_sync(kFull, eta, 1), e2 = __shfl_sync(kFull, eta, 2);
    if (lane == 0) {
      int bq = qo;
      if (accepted && lo && e1 > eta) {
        eta = e1;
        bq = qo - 1;
      }
      if (accepted && hi && e2 > eta) {
        eta = e2;
        bq = qo + 1;
      }
      S.eta = eta;
      S.best_q = bq;
      S.err = err;
      S.state = accepted;
    }
  }
  __syncthreads();
  const bool accepted = S.state != 0, keep_e = S.best_q == qo;
  if (accepted) {
    // the newest point takes the slot in front of the ring
    const int slot = S.base == 0 ? QMAX : S.base - 1;
    double* Y0 = S.hist + (int64_t)slot * S.hn;
    for (int s = tid; s < n; s += nthr) {
      const double yv = ys[s];
      if (keep_e) S.eprev[s] = yv - yp[s];
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
      const double eta = fmax(0.2, S.eta);
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
        const int64_t o = (int64_t)(S.steps - 1) * d.ld + S.c;
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
      double eta = fmin(S.eta, (fl & F_REJECTED) ? 1.0 : d.eta_max);
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
      for (int s = tid; s < n; s += nthr) dst[i * vs + (int64_t)s * d.ld + S.c] = S.hist[(int64_t)slot * S.hn + s];
      if (tid == 0) d.ck_t[((int64_t)kk * (QMAX + 1) + i) * d.ld + S.c] = S.tn[i];
    }
    if (tid == 0) d.ck_nh[(int64_t)kk * d.ld + S.c] = nhc;
  }
  class_end(SM_TIME_FINISH);
  PHASE_MARK(PH_FINISH);
}

// One BDF attempt of the cell; returns false when the cell stopped before or
// in it.
template <class T, bool TF>
__device__ __forceinline__ bool cell_attempt() {
  const Args& A = args();
  const Dev& d = A.d;
  CellS& S = scalars();
  cell_predict();
  if (S.state != 3) return false;
  if (d.therm) cell_th_rates(at<double>(A.p.o_yp)[d.t_idx], false);
  if (S.flags & F_REFRESH) {
    class_begin(SM_TIME_REFRESH);
    cell_refresh<T, TF>();
    if (d.therm) cell_border<T>();
    class_end(SM_TIME_REFRESH);
  }
  if (threadIdx.x == 0) {
    const double gam = S.gam, gJ = S.gam_J;
    S.inv_a0 = 1.0 / S.alpha[0];
    S.scale = gam != gJ ? 2.0 / (1.0 + gam / gJ) : 1.0;
  }
  for (int m = 0; m < d.newton_max; ++m) {
    class_begin(SM_TIME_RHS);
    if (d.therm && m > 0) cell_th_rates(at<double>(A.p.o_ys)[d.t_idx], false);
    cell_rhs();
    if (d.therm) cell_energy();
    class_end(SM_TIME_RHS);
    cell_newton<T>();
    if (!(S.flags & F_NEWTON)) break;
  }
  cell_finish();
  return S.status == SM_CELL_RUNNING;
}

// Copies the launch's arguments to shared memory and sets up this CTA's global
// scratch.  Ends with a barrier.
template <class T>
__device__ __forceinline__ void cell_begin(const Args& from) {
  const uint32_t* src = reinterpret_cast<const uint32_t*>(&from);
  for (int i = threadIdx.x; i < (int)(sizeof(Args) / 4); i += blockDim.x) reinterpret_cast<uint32_t*>(sm)[i] = src[i];
  __syncthreads();
  const Args& A = args();
  uint16_t* ip = at<uint16_t>(A.p.o_ip);
  for (int s = threadIdx.x; s < A.d.n; s += blockDim.x) ip[s] = (uint16_t)__ldg(A.w + A.iperm + s);
  uint16_t* hx = at<uint16_t>(A.p.o_hx);
  for (int e = threadIdx.x; e < A.d.p_d; e += blockDim.x) hx[e] = (uint16_t)__ldg(A.w + A.hx + e);
  if (threadIdx.x == 0) {
    CellS& S = scalars();
    S.hn = (A.d.n + 31) / 32 * 32;
    S.kc = A.scratch + (int64_t)blockIdx.x * A.p.scratch;
    S.hist = S.kc + (A.d.n_r + 31) / 32 * 32;
    S.eprev = S.hist + (int64_t)(QMAX + 1) * S.hn;
    S.mbuf = S.eprev + S.hn;
#ifdef SM_PHASE_CLOCKS
    S.ph_t = clock64();
#endif
  }
  __syncthreads();
}

// Rate coefficients of cell oc into this CTA's scratch (cell-major), or the
// cell's conditions with a coupled temperature (to S, by thread 0).
__device__ __forceinline__ void cell_conditions(int64_t oc) {
  const Args& A = args();
  const Dev& d = A.d;
  CellS& S = scalars();
  if (d.therm) {
    if (threadIdx.x == 0) {
      S.nH = d.c_nH[oc];
      S.Av = d.c_Av[oc];
      S.chi = d.c_chi[oc];
    }
  } else {
    double* kc = S.kc;
    const double* k = A.k + oc;
    const int64_t ldk = A.ldk;
#pragma unroll 8
    for (int j = threadIdx.x; j < d.n_r; j += blockDim.x) kc[j] = k[(int64_t)j * ldk];
  }
}

// 12 warps at 168 registers: the register tiles of the tail and a row block with
// its next 32 columns need about that many, and a 349-column tail has 11 blocks.
// (16 warps at 128 registers spilled in every inner loop; two CTAs an SM do not
// fit the shared memory of a 470-species cell.)
template <class T, bool TF>
__global__ void __launch_bounds__(kMaxCellThreads, 1) cell_kernel(const __grid_constant__ Args from) {
  __shared__ int sh_c;
  cell_begin<T>(from);
  const Args& A = args();
  const Dev& d = A.d;
  const int tid = threadIdx.x, nthr = blockDim.x, n = d.n;
  CellS& S = scalars();
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
    const int64_t oc = d.slot_cell[c];
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
      S.c = c;
      S.oc = oc;
      S.P = static_cast<T*>(d.lup) + oc * d.lup_stride;
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
    cell_conditions(oc);
    const int nh0 = d.nh[c];
    for (int s = tid; s < n; s += nthr) {
      const int64_t o = (int64_t)s * d.ld + c;
      for (int i = 0; i < nh0; ++i) S.hist[(int64_t)i * S.hn + s] = Yh(d, i)[o];
      S.eprev[s] = d.eprev[o];
      if constexpr (sizeof(T) == 4) {
        const double wv = d.wf[o];
        at<double>(A.p.o_wf)[s] = wv;
        at<double>(A.p.o_wi)[s] = 1.0 / wv;   // (meaningless, and unused, before the first factorisation)
      }
    }
    __syncthreads();
    if (d.therm) {
      // every coefficient from the current T; the attempt's own passes refresh
      // the T-dependent ones
      cell_th_rates(S.hist[d.t_idx], true);
    }
    PHASE_MARK(PH_LOAD);
    const int before = A.done[c], todo = min(A.slice, A.attempts - before);
    int made = 0;
    bool run = true;
    while (run && made < todo) {
      run = cell_attempt<T, TF>();
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
        Yh(d, i)[o] = S.hist[(int64_t)slot * S.hn + s];
      }
      d.eprev[o] = S.eprev[s];
      if constexpr (sizeof(T) == 4) d.wf[o] = at<double>(A.p.o_wf)[s];
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
__global__ void __launch_bounds__(kMaxCellThreads, 1) cell_init_kernel(const __grid_constant__ Args from, const double* __restrict__ y,
                                                           int64_t ldu) {
  cell_begin<T>(from);
  const Args& A = args();
  const Dev& d = A.d;
  const CellS& S = scalars();
  const int tid = threadIdx.x, nthr = blockDim.x, n = d.n;
  double* ys = at<double>(A.p.o_ys);
  const double* fs = at<double>(A.p.o_fs);
  for (int64_t c = blockIdx.x; c < d.C; c += gridDim.x) {
    bool ok = true;
    for (int s = tid; s < n; s += nthr) {
      const double v = y[(int64_t)s * ldu + c];
      ys[s] = v;
      Yh(d, 0)[(int64_t)s * d.ld + c] = v;
      ok = ok && isfinite(v);
    }
    cell_conditions(c);
    if (!d.therm)
      for (int j = tid; j < d.n_r; j += nthr) ok = ok && isfinite(S.kc[j]);
    __syncthreads();
    if (d.therm) ok = ok && ys[d.t_idx] > 0.0 && isfinite(S.nH) && S.nH > 0.0 && isfinite(S.Av) && isfinite(S.chi);
    ok = __syncthreads_and(ok);
    if (ok) {
      if (d.therm) cell_th_rates(ys[d.t_idx], true);
      cell_rhs();
      if (d.therm) cell_energy();
    }
    double* nv = at<double>(A.p.o_nv);
    if (ok)
      for (int s = tid; s < n; s += nthr) {
        d.f0[(int64_t)s * d.ld + c] = fs[s];
        nv[s] = fs[s] / (d.rtol * fabs(ys[s]) + d.atol);
      }
    __syncthreads();
    double acc = 0.0;
    if (ok && tid == 0)   // in order, as the class-by-class path
#pragma unroll 8
      for (int s = 0; s < n; ++s) acc = fma(nv[s], nv[s], acc);
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
      for (int s = tid; s < n; s += nthr) d.ck_Y[(int64_t)s * d.ld + c] = ys[s];
    __syncthreads();
  }
}

// The CTA shape of a batch: wide CTAs (12 warps) where every cell has an SM of
// its own, narrow ones (4 warps, two and more per SM) for more cells of networks
// whose tails have at most four blocks, which give 12 warps nothing to do.
const CellShape& shape(const CellLaunch& L, int64_t C) { return C > L.sms && L.narrow.ctas > 0 ? L.narrow : L.wide; }

Args make_args(const sm_net* net, const Dev& d, const CellLaunch& L, const double* k, int64_t ldk) {
  const CellProg& p = net->cell;
  Args a{};
  a.d = d;
  a.p = shape(L, d.C).plan;
  a.w = p.blob.as<int>();
  a.nb = p.nb; a.pitch = p.pitch; a.n_slot = p.n_slot; a.rx = p.rx; a.iperm = p.iperm;
  const int narrow = a.p.warps < kMaxCellThreads / 32;
  a.rp_deal = p.rp_deal[narrow]; a.rp_ent = p.rp_ent; a.rp_dst = p.rp_dst; a.row = p.row; a.row_more = p.row_more;
  a.n_jsl = p.n_jsl; a.n_jl = p.n_jl;
  a.jg_off = p.jg_off; a.jg_ent = p.jg_ent; a.jg_rc = p.jg_rc; a.jg_dst = p.jg_dst; a.jg_grp = p.jg_grp;
  a.n_jw = p.n_jw; a.jl_off = p.jl_off; a.jl_ent = p.jl_ent;
  a.jl_rc = p.jl_rc; a.jd_grp = p.jd_grp; a.jd_ent = p.jd_ent;
  a.n_hlev = net->lu.n_hlev; a.hop = p.hop; a.hterm = p.hterm; a.hop_ptr = p.hop_ptr;
  a.tg_grp = p.tg_grp; a.tg_ent = p.tg_ent;
  a.lev_f = p.lev_f; a.lev_b = p.lev_b; a.hx = p.hx;
  a.vp_deal = p.vp_deal[narrow]; a.vp_ent = p.vp_ent; a.vp_dst = p.vp_dst; a.vrow = p.vrow; a.vrow_more = p.vrow_more;
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

sm_status cell_shapes(const sm_net* net, const Dev& d, bool thermal, int per_sm_cap, CellLaunch* L) {
  L->wide = L->narrow = CellShape{};
  int smem = 0;
  SM_TRY_CUDA(cudaDeviceGetAttribute(&L->sms, cudaDevAttrMultiProcessorCount, net->device));
  SM_TRY_CUDA(cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, net->device));
  const void* init = d.mixed ? (const void*)cell_init_kernel<float> : (const void*)cell_init_kernel<double>;
  const size_t esz = d.mixed ? 4 : 8;
  // per-kernel caps are shared by every state: always the device's limit
  // (less the kernel's own static shared memory)
  const int top = smem - 1024;
  SM_TRY_CUDA(cudaFuncSetAttribute(kernel_of(d), cudaFuncAttributeMaxDynamicSharedMemorySize, top));
  SM_TRY_CUDA(cudaFuncSetAttribute(init, cudaFuncAttributeMaxDynamicSharedMemorySize, top));
  auto resident = [&](int warps, CellShape* s) -> sm_status {
    s->plan = cell_plan(net, esz, d.tf32 != 0, thermal, warps, (size_t)std::max(top, 0));
    if (!s->plan.ok) return SM_OK;
    int per = 0;
    SM_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel_of(d), 32 * warps, s->plan.bytes));
    if (per_sm_cap > 0) per = std::min(per, per_sm_cap);
    s->ctas = L->sms * per;
    return SM_OK;
  };
  sm_status r = resident(kMaxCellThreads / 32, &L->wide);
  if (r != SM_OK) return r;
  // a tail of few blocks has no work for more than four warps
  if (net->cell.nb <= 4 && (r = resident(4, &L->narrow)) != SM_OK) return r;
  if (L->narrow.ctas < 2 * L->sms) L->narrow.ctas = 0;   // alone on an SM the wide one is faster
  return SM_OK;
}

int64_t cell_ring_ints(const CellLaunch& L, int64_t C, int attempts) {
  const int tn = turn(C, shape(L, C).ctas, attempts);
  return 2 + C * ((attempts + tn - 1) / tn);
}

sm_status launch_cell_init(const sm_net* net, const Dev& d, const CellLaunch& L, const double* y, int64_t ldu,
                           const double* k, int64_t ldk, cudaStream_t s) {
  const Args a = make_args(net, d, L, k, ldk);
  const CellShape& q = shape(L, d.C);
  const unsigned grid = (unsigned)std::min<int64_t>(d.C, q.ctas);
  if (d.mixed) cell_init_kernel<float><<<grid, 32 * q.plan.warps, q.plan.bytes, s>>>(a, y, ldu);
  else cell_init_kernel<double><<<grid, 32 * q.plan.warps, q.plan.bytes, s>>>(a, y, ldu);
  SM_TRY_CUDA(cudaGetLastError());
  return SM_OK;
}

sm_status launch_cell_attempts(const sm_net* net, const Dev& d, const CellLaunch& L, const double* k, int64_t ldk,
                               int attempts, cudaStream_t s) {
  Args a = make_args(net, d, L, k, ldk);
  a.attempts = attempts;
  const CellShape& q = shape(L, d.C);
  a.slice = turn(d.C, q.ctas, attempts);
  const int64_t total = cell_ring_ints(L, d.C, attempts) - 2;
  ring_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(d.C, L.ring, L.done, total);
  SM_TRY_CUDA(cudaGetLastError());
  const unsigned grid = (unsigned)std::min<int64_t>(d.C, q.ctas);
  const int threads = 32 * q.plan.warps;
  if (!d.mixed) cell_kernel<double, false><<<grid, threads, q.plan.bytes, s>>>(a);
  else if (d.tf32) cell_kernel<float, true><<<grid, threads, q.plan.bytes, s>>>(a);
  else cell_kernel<float, false><<<grid, threads, q.plan.bytes, s>>>(a);
  SM_TRY_CUDA(cudaGetLastError());
  return SM_OK;
}

extern "C" sm_status sm_cell_phase_cycles(int32_t device, double* h_out, int32_t reset) {
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
