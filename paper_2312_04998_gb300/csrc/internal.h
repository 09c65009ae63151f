// Internal structures of the stoichiometry-matrix library (not part of the ABI).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "stoich.h"

// Jacobian entries with more terms than this are gathered by a whole warp.
constexpr int kJLong = 32;

// Device status word bits written by kernels (never trap).
enum : int32_t {
  DEV_ERR_NONE = 0,
  DEV_ERR_BOUNDS = 1,   // an index check failed; the access was skipped
  DEV_ERR_TIMEOUT = 2,  // a bounded wait ran out
};

#define SM_TRY_CUDA(expr)                                      \
  do {                                                         \
    cudaError_t _e = (expr);                                   \
    if (_e != cudaSuccess) {                                   \
      sm_set_last_cuda_error(_e, #expr);                       \
      return (_e == cudaErrorMemoryAllocation) ? SM_ENOMEM : SM_ECUDA; \
    }                                                          \
  } while (0)

void sm_set_last_cuda_error(cudaError_t e, const char* what);

// Rate-law parameters of one reaction: (log alpha for two-body classes,
// alpha otherwise; beta; gamma; class as a double).
struct __align__(32) RatePar {
  double x, y, z, w;
};

// A device allocation owned by a handle.
struct DevArray {
  void* p = nullptr;
  size_t bytes = 0;
  sm_status upload(const void* h, size_t n);
  sm_status ensure(size_t n);  // grow (no copy) to at least n bytes
  void release();
  template <class T> T* as() const { return static_cast<T*>(p); }
};

// Traversal format as uploaded: see the sm_net_export documentation.
struct Format {
  int32_t fmt = SM_FMT_CRS, order = SM_ORDER_NONE, C = 1, sigma = 1;
  std::vector<int32_t> ptr, idx, idx2, len;
  int32_t longest = 0;                    // SELL: the largest of len
  std::vector<double> val;
  // Device-only companion indices: CRS row ids, CCS column ids, COO column
  // per nonzero, SELL row ids (-1 = padding row).
  std::vector<int32_t> aux;
  // Packed device entries: column (or row) in the low 24 bits, signed
  // coefficient in the high 8 bits.
  std::vector<uint32_t> packed;
  // CRS partitions: per chunk the first nonzero, for 32 chunks (chunk_nz,
  // the default 16-cell gather) and for 64 / 16 chunks (the 8- and 32-cell
  // gathers of the integrator), n_chunks + 1 entries each.
  std::vector<int32_t> chunk_nz, chunk_nz64, chunk_nz16;
  DevArray d_ptr, d_packed, d_aux, d_chunk, d_chunk64, d_chunk16;
};

// Symbolic LU of the Newton matrix M = I - gamma J (no pivoting).
struct LUSymbolic {
  int32_t n = 0, ld = 0, head = 0;
  std::vector<int32_t> perm, iperm;       // perm[p] = species at position p
  std::vector<int32_t> lptr, lidx;        // per pivot: rows below it (positions)
  std::vector<int32_t> uptr, uidx;        // per pivot: columns right of it
  std::vector<int32_t> lrptr, lridx;      // per row: columns of L left of the diagonal
  std::vector<int32_t> jrc;               // per J pattern entry: (row position << 16) | column position
  std::vector<int32_t> lrhead;            // per tail row: entries of its L row in head columns
  std::vector<int32_t> lrhoff;            // exclusive prefix sum of lrhead (n - head + 1 entries)
  std::vector<int32_t> u12off;            // per head row: start of its tail-column U entries, packed
  std::vector<int32_t> lrhk;              // head column of each L21 entry in compact row order
  std::vector<int32_t> srow;              // tail rows with L21 entries, longest first
  std::vector<int32_t> uoff;              // per head row k: [n_panels + 1] offsets into its U list where
                                          // the tail columns of each 32-wide panel start
  // Packed factor layout read by the substitution (per cell, values only,
  // in the precision of the factors), segment offsets in elements:
  //   [p_l11, +lrptr[head])   L11: head rows' L entries, order of lrptr/lridx
  //   [p_u11, +u11ptr[head])  U11: head rows' U entries in head columns
  //   [p_dinv, +head)         inverse pivots of the head
  //   [p_l21, +lrhoff[nt])    L21: tail rows' L entries in head columns
  //   [p_u12, +u12off[head])  U12: head rows' U entries in tail columns
  //   [p_d, +nt * ldd)        the dense tail block, column-major (L below the
  //                           diagonal, U above, inverse pivots on it)
  int32_t p_l11 = 0, p_u11 = 0, p_dinv = 0, p_l21 = 0, p_u12 = 0, p_d = 0, ldd = 0;
  int64_t p_size = 0;
  std::vector<int32_t> u11ptr;            // per head row: start of its U11 entries (head + 1)
  std::vector<int32_t> flev_ptr, flev;    // head rows grouped by forward-substitution level
  std::vector<int32_t> blev_ptr, blev;    // head rows grouped by backward-substitution level
  // Head program of the refresh: the sparse head's factors (L11, U11, inverse
  // pivots, L21, U12) computed in the packed layout, level by level.  Pivot k
  // depends on the pivots m < k with l_km or u_mk nonzero; all pivots of one
  // level are independent.  Per level l, ops [hop_ptr[2l], hop_ptr[2l+1]) are
  // the level's pivots, [hop_ptr[2l+1], hop_ptr[2l+2]) its U-row and L-column
  // entries.  An op is {packed index written, offset in the dense working
  // matrix read, first term, end of terms}; its value is
  //   a - sum over its terms (x, y) of H[x] * H[y]
  // (H = the packed head values), inverted for a pivot, times H[hop_piv]
  // (the inverse pivot) for an L entry (hop_piv = -1 otherwise).
  std::vector<int32_t> hop_ptr, hop, hop_piv, hterm;   // hop: 4 ints per op, hterm: 2 per term
  int32_t n_hlev = 0;
  int64_t nnz = 0, flops = 0;
  DevArray d_u11ptr, d_flev_ptr, d_flev, d_blev_ptr, d_blev, d_hop_ptr, d_hop, d_hop_piv, d_hterm;
  DevArray d_lptr, d_lidx, d_uptr, d_uidx, d_lrptr, d_lridx, d_perm, d_iperm, d_uoff, d_lrhead, d_lrhoff, d_u12off, d_lrhk, d_srow;
};

// Words of the index programs: table slot (16 bits) | the upper half of the
// double c << 16, for c of at most five significant bits; any other c goes in
// parts.
inline int32_t coef_word(int32_t slot, int c) {
  const double v = c;
  uint64_t u;
  std::memcpy(&u, &v, sizeof u);
  return (int32_t)((uint32_t)slot | (uint32_t)(u >> 48) << 16);
}
template <class F> void for_coef_parts(int c, F f) {
  while (c != 0) {
    const int part = c >= -31 && c <= 31 ? c : c / 32 * 32;
    f(part);
    c -= part;
  }
}

constexpr int kJShort = 4;   // (see CellProg)

// Index programs of one network for the fused integrator (cell.cu), packed
// into one device blob of 32-bit words (offsets below in words).  "Sliced"
// lists hold work items in slices of 32 (one item per lane), sorted by length
// inside a group and padded to the slice's longest; slice s has the pair
// {first row, rows} at off + 2 s, and entry e of lane l lies at
// 32 * (first row + e) + l, so a warp reads its index words in 128-byte lines.
struct CellProg {
  bool ok = false;               // false: the network is outside the programs' index ranges
  int32_t nb = 0;                // 32-wide blocks of the dense tail
  int32_t pitch = 0;             // rows of one tail column in shared memory (odd)
  int32_t n_slot = 0;            // derivative slots: one per reactant
  int32_t rx = 0;                // per reaction {reactants a | b << 16 (0xFFFF: none), first derivative slot}
  int32_t iperm = 0;             // per species: position in elimination order
  // right-hand side: rows of S in chains (see cell_prog.cpp); entry = reaction |
  // upper half of the double coefficient << 16 (pads read slot n_r = 0)
  // (dealt to the warps of a wide and of a narrow CTA)
  int32_t n_chain = 0, rp_deal[2] = {0, 0};
  int32_t rp_ent = 0, rp_dst = 0, row = 0, row_more = 0;
  // Jacobian: entries of at most kJShort words in slices by destination group
  // (0 = head, 1 + G = the tail's columns kGroup G .. of the assembly); entry
  // word = derivative slot | upper half of the double coefficient << 16, pads
  // read slot n_slot = 0.  Of the other entries ("long") those of more than
  // kJLong words have a slice each (the first n_jw, word e in lane e mod 32).
  // jd: by group {destination, 32 x slice + lane of the long entry}.
  int32_t n_jsl = 0, n_jl = 0, n_jw = 0;
  int32_t jg_off = 0, jg_ent = 0, jg_rc = 0, jg_dst = 0, jg_grp = 0;
  int32_t jl_off = 0, jl_ent = 0, jl_rc = 0, jd_grp = 0, jd_ent = 0;
  // head program (see LUSymbolic): per op {dst | pivot << 16, first term, end
  // of terms, 0}; term = x | y << 16
  int32_t hop = 0, hterm = 0, hop_ptr = 0;
  // head's Schur complement on the tail: targets by column group, in slices of
  // 32 sorted by length: a row of {position | terms << 16} (0xFFFF: no target),
  // then the rows of terms (L21 index | U12 index << 16, pads read slot p_d =
  // 0), in pivot order; tg_grp: first row of each group
  int32_t tg_grp = 0, tg_ent = 0;
  // substitution: levels of the head rows; per packed head entry the index in x
  // (L11, U11, L21: head part, U12: tail part) that it multiplies
  int32_t lev_f = 0, lev_b = 0, hx = 0;
  // column sums of dn_j dR_j/dx_l (coupled temperature): derivative slots of
  // each species in chains like the right-hand side
  int32_t n_vchain = 0, vp_deal[2] = {0, 0};
  int32_t vp_ent = 0, vp_dst = 0, vrow = 0, vrow_more = 0;
  std::vector<int32_t> h;
  DevArray blob;
};

// Program of the Jacobian kernel (kern_jac.cu): per group (a CTA's columns) a
// run of passes {slots, segments}; slot = product {reaction, partner or -1};
// segment = an entry's terms in the pass's products (coef_word each).
struct JacProg {
  std::vector<int32_t> group, pass, slot, seg, term;
  int32_t slots = 0;   // most products of a pass
  DevArray blob;       // pass, seg, term, slot, group
};

struct sm_net {
  int device = 0;
  int32_t n_s = 0, n_r = 0, n_elem = 0;
  std::vector<int32_t> comp, reac, prod;
  std::vector<int8_t> cls;
  std::vector<double> alpha, beta, gamma;
  std::vector<int32_t> order;  // reactants per reaction
  // S in column-compressed form, original order, rows ascending.
  std::vector<int32_t> s_colptr, s_row;
  std::vector<int8_t> s_coef;
  // Row orders and column orders for SM_ORDER_NONE / NNZ / RCM.
  std::vector<int32_t> row_order[3], col_order[3];
  Format cur;
  // The integrator's masked CRS gather: CRS in each row order (NONE, NNZ,
  // RCM; built on first use and kept for the network's life, so that a
  // captured graph never refers to released arrays), the selected order and
  // the cells per CTA of the gather (8, 16 or 32), chosen by sm_net_autotune.
  Format integ_fmt[3];
  int32_t integ_order = SM_ORDER_NONE, integ_kc = 16;
  // Jacobian pattern (CRS, species order) and contribution list per entry:
  // term = coef * k'[j] * (partner >= 0 ? y[partner] : 1).
  std::vector<int32_t> jp_ptr, jp_col, jt_ptr, jt_rx, jt_partner;
  std::vector<int8_t> jt_coef;
  LUSymbolic lu;
  CellProg cell;
  // Device copies used by the kernels.
  DevArray d_reac;        // int2 per reaction: reactant indices (-1 = none)
  DevArray d_rate;        // RatePar per reaction: (log alpha | alpha, beta, gamma, class)
  DevArray d_ratefix, d_ratetab;           // the same for the fixed-point exponential (see kern_rates.cu)
  DevArray d_jt_slot;                      // (reaction | coef << 24, reactant slot) per term
  std::vector<int32_t> jlong;              // Jacobian entries with more than kJLong terms
  DevArray d_jdesc, d_jlong;               // per entry {t0, t1, jrc, row << 16 | col}; long entries
  DevArray d_sc_ptr, d_sc_ent;             // S by columns: pointers and (species | coef << 24)
  JacProg jac;
  DevArray d_status;      // int32 device status word
  DevArray d_scratch;     // reaction-rate scratch for rhs_eval
  sm_net_info info{};
  // Coupled temperature (sm_net_set_thermal; states copy it at creation):
  // slot th_t holds T (-1: off), line-cooling coefficients and excitation
  // temperatures per species, and the constant parameters.
  int32_t th_t = -1;
  double th_heat = 0.0, th_lam = 0.0, th_Td = 0.0, th_zeta = 0.0;
  std::vector<double> th_L, th_E;
};

// Host-side builders (net_build.cpp).
sm_status net_build_host(const sm_net_desc* d, sm_net* net);
sm_status net_upload(sm_net* net);
sm_status net_select_format(sm_net* net, int32_t fmt, int32_t order, int32_t C, int32_t sigma);
sm_status build_format(const sm_net* net, int32_t fmt, int32_t order, int32_t C, int32_t sigma,
                       Format* out);
// Builds (once) the integrator's CRS format in row order `order`.
sm_status integ_format(sm_net* net, int32_t order);

// Kernel launchers (one per .cu file).
struct __align__(32) RateFix {   // a reaction's rate for the fixed-point exponential; OTHER: from its RatePar
  enum { OTHER, TWO_BODY, PHOTO };
  double beta = 0.0, gamma = 0.0;
  long long la = 0;   // log2 alpha
  long long kind = OTHER;
};
std::vector<double> rate_table();
std::vector<RateFix> rate_fixed(const sm_net* net, const std::vector<double>& table);
sm_status launch_rates(const sm_net* net, int64_t C, const double* T, const double* nH,
                       const double* Av, const double* chi, double zeta, double* k, int64_t ld, cudaStream_t s);
sm_status launch_rhs(const sm_net* net, int64_t C, const double* k, const double* y,
                     double* f, int64_t ld, double* scratch, int64_t ld_scratch, cudaStream_t s);
// Masked CRS right-hand side for the integrator: cells whose mask word has
// `bit` set are evaluated; whole thread blocks without such a cell exit, and
// with cact (device, may be null) so do blocks of cells at or past *cact.
sm_status launch_rhs_masked(const sm_net* net, int64_t C, const double* k, int64_t ldk,
                            const double* y, double* f, int64_t ld, double* scratch, int64_t ldr,
                            const int* mask, int bit, const int* cact, cudaStream_t s);
// Per-device set-up of the right-hand-side kernels (constant tables); called
// when a network is uploaded.
sm_status rhs_prepare_device(int device);
JacProg build_jac_prog(const sm_net* net);
sm_status launch_jac(const sm_net* net, int64_t C, const double* k, const double* y,
                     double* J, int64_t ld, cudaStream_t s);

inline bool ld_ok(int64_t C, int64_t ld) { return C >= 0 && ld >= C && ld % 32 == 0; }
