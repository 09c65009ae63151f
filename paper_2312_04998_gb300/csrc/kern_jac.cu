// Jacobian values J = S dR/dx on the static pattern, cells as the fast axis.
//
// J_il = sum over reactions j with S_ij != 0 and species l among their
// reactants of S_ij dR_j/dx_l, where dR_j/dx_l = k'_j times the other
// reactant's abundance (2 k'_j x_l for a squared reactant, k'_j for a one-body
// reaction).
//
// The bound is FP64 arithmetic (a warp's instruction holds its scheduler's FP64
// unit for 64 cycles).  Walking the entries row by row, a product and an FMA per
// term with each term's loads waiting for its index word, 4096 cells of 470
// species took 1455 us.  Every term of column l uses one of the products
// k'_j x_other of l's reactions, about 4.5 terms each, and 3 of 4 entries have a
// single term of coefficient +-1.  So a CTA takes the columns (all rows) of a
// run of species for 32 cells: it forms their products once, in shared memory,
// and the entries are sums of those: a sign flip for the first term, an addition
// for every further one.  An entry's terms are added in the order of its list,
// as before, so the values are unchanged to the last bit: 332 us, of which FP64
// arithmetic (10 k products, 21 k sums a cell) takes 200 and storing J 90.
#include <algorithm>

#include "internal.h"

namespace {

constexpr int kWarps = 8;
constexpr int kSlots = 192;      // products held at a time (48 KB: four CTAs an SM)
constexpr int kCarry = 1 << 30;  // segment goes on from the value stored by an earlier pass

__device__ __forceinline__ double coef(int word) { return __hiloint2double(word & 0xFFFF0000, 0); }
__device__ __forceinline__ double flip(double v, int word) {   // v, negated when bit 31 of word is set
  return __hiloint2double(__double2hiint(v) ^ (word & 0x80000000), __double2loint(v));
}
// a + the n terms at q.  (An FP64 instruction that is predicated off holds the
// unit all the same, and the compiler predicates short branches: fours without
// a condition, then a loop.)
__device__ __forceinline__ double add_terms(double a, const double* t, const int* __restrict__ q, int n) {
#pragma unroll 1
  for (; n >= 4; n -= 4, q += 4) {
    const int4 w = __ldg(reinterpret_cast<const int4*>(q));
    const double v0 = t[(w.x & 0xFFFF) * 32], v1 = t[(w.y & 0xFFFF) * 32], v2 = t[(w.z & 0xFFFF) * 32],
                 v3 = t[(w.w & 0xFFFF) * 32];
    a = fma(coef(w.x), v0, a);
    a = fma(coef(w.y), v1, a);
    a = fma(coef(w.z), v2, a);
    a = fma(coef(w.w), v3, a);
  }
#pragma unroll 1
  for (; n > 0; --n, ++q) {
    const int w = __ldg(q);
    a = fma(coef(w), t[(w & 0xFFFF) * 32], a);
  }
  return a;
}

__global__ void __launch_bounds__(32 * kWarps, 4)
jac_kernel(int64_t C, const int* __restrict__ group, const int4* __restrict__ pass, const int2* __restrict__ slot,
           const int4* __restrict__ seg, const int* __restrict__ term, const double* __restrict__ k,
           const double* __restrict__ y, double* __restrict__ J, int64_t ld) {
  extern __shared__ double tab[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t c0 = (int64_t)blockIdx.x * 32 + lane, c = min(c0, C - 1);   // (lanes past the end: no stores)
  const bool live = c0 < C;
  const int p1 = __ldg(group + blockIdx.y + 1);
  for (int p = __ldg(group + blockIdx.y); p < p1; ++p) {
    const int4 ps = __ldg(pass + 2 * p);   // slots [x, y), plain segments [z, w)
    const int end = __ldg(&pass[2 * p + 1].x);   // other segments [w, end)
    constexpr int U = 8;
    for (int s = ps.x + warp; s < ps.y; s += U * kWarps) {
      int2 w[U];
      double kv[U], yv[U];
#pragma unroll
      for (int u = 0; u < U; ++u) w[u] = __ldg(slot + min(s + u * kWarps, ps.y - 1));
#pragma unroll
      for (int u = 0; u < U; ++u) {
        kv[u] = k[(int64_t)w[u].x * ld + c];
        yv[u] = w[u].y >= 0 ? y[(int64_t)w[u].y * ld + c] : 0.0;
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (s + u * kWarps < ps.y) {
          if (w[u].y >= 0) kv[u] *= yv[u];
          tab[(s + u * kWarps - ps.x) * 32 + lane] = kv[u];
        }
    }
    __syncthreads();
    const double* t = tab + lane;
    // segments: {entry | kCarry, further terms, their words, first term's word};
    // plain ones begin with a term of coefficient +-1
    constexpr int G = 4;
    for (int g = ps.z + warp; g < ps.w; g += G * kWarps) {
      int4 sg[G];
#pragma unroll
      for (int u = 0; u < G; ++u) sg[u] = __ldg(seg + min(g + u * kWarps, ps.w - 1));
#pragma unroll
      for (int u = 0; u < G; ++u) {
        if (g + u * kWarps >= ps.w) break;
        double a = flip(t[(sg[u].w & 0xFFFF) * 32], sg[u].w);
        a = add_terms(a, t, term + sg[u].z, sg[u].y);
        if (live) J[(int64_t)sg[u].x * ld + c] = a;
      }
    }
    for (int g = ps.w + warp; g < end; g += kWarps) {   // any terms, added to what an earlier pass stored (kCarry) or to 0
      const int4 s = __ldg(seg + g);
      double* dst = J + (int64_t)(s.x & (kCarry - 1)) * ld + c;
      const double a = add_terms(s.x & kCarry ? *dst : 0.0, t, term + s.z, s.y);
      if (live) *dst = a;
    }
    if (p + 1 < p1) __syncthreads();
  }
}

}  // namespace

JacProg build_jac_prog(const sm_net* net) {
  JacProg P;
  const int32_t n = net->n_s;
  std::vector<std::vector<int32_t>> col(n);   // entries of each column
  std::vector<int64_t> terms(n, 0);
  for (int32_t i = 0; i < n; ++i)
    for (int32_t e = net->jp_ptr[i]; e < net->jp_ptr[i + 1]; ++e) {
      const int32_t l = net->jp_col[e];
      col[l].push_back(e);
      terms[l] += std::max(net->jt_ptr[e + 1] - net->jt_ptr[e], 1);
    }
  // each column's products, by reaction
  std::vector<std::vector<int32_t>> rx(n);   // indices into jt (one term per product)
  std::vector<int32_t> seen(net->n_r, -1), local(net->n_r, 0);
  int64_t work = 0;
  for (int32_t l = 0; l < n; ++l) {
    for (int32_t e : col[l])
      for (int32_t t = net->jt_ptr[e]; t < net->jt_ptr[e + 1]; ++t)
        if (seen[net->jt_rx[t]] != l) {
          seen[net->jt_rx[t]] = l;
          rx[l].push_back(t);
        }
    std::sort(rx[l].begin(), rx[l].end(), [&](int32_t a, int32_t b) { return net->jt_rx[a] < net->jt_rx[b]; });
    work += terms[l] + (int64_t)rx[l].size();
  }
  // groups of whole columns of about 1/64 of the work; the rows of a long column
  // are dealt to several groups, each forming its products again, while those
  // stay less than half as many as the group's terms
  const int64_t goal = std::max<int64_t>(work / 64, 48);
  struct Group {
    std::vector<int32_t> cols;
    int32_t part = 0, parts = 1;
    int64_t work = 0, slots = 0;
  };
  std::vector<Group> groups;
  std::vector<int32_t> order(n);
  for (int32_t l = 0; l < n; ++l) order[l] = l;
  auto cost = [&](int32_t l) { return terms[l] + (int64_t)rx[l].size(); };
  std::stable_sort(order.begin(), order.end(), [&](int32_t a, int32_t b) { return cost(a) > cost(b); });
  for (int32_t l : order) {
    const int64_t sl = (int64_t)rx[l].size();
    const int64_t parts = std::max<int64_t>(1, std::min((cost(l) + goal - 1) / goal, terms[l] / std::max<int64_t>(2 * sl, 1)));
    if (parts > 1 || cost(l) >= goal || sl > kSlots || groups.empty() || groups.back().parts > 1 ||
        groups.back().work + cost(l) > goal + goal / 4 || groups.back().slots + sl > kSlots) {
      for (int32_t q = 0; q < parts; ++q) {
        Group g;
        g.cols = {l};
        g.part = q;
        g.parts = (int32_t)parts;
        g.work = terms[l] / parts + sl;
        g.slots = sl;
        groups.push_back(g);
      }
    } else {
      groups.back().cols.push_back(l);
      groups.back().work += cost(l);
      groups.back().slots += sl;
    }
  }
  std::stable_sort(groups.begin(), groups.end(), [](const Group& a, const Group& b) { return a.work > b.work; });
  P.group.push_back(0);
  std::vector<std::vector<int32_t>> have;   // a group's segments by pass, 4 words each
  std::vector<int32_t> ts, words, o;
  for (const Group& g : groups) {
    // passes: runs of at most kSlots products (several columns only if all fit)
    size_t total = 0;
    for (int32_t l : g.cols) total += rx[l].size();
    const size_t passes = std::max<size_t>(1, (total + kSlots - 1) / kSlots);
    have.resize(std::max(have.size(), passes));
    for (auto& v : have) v.clear();
    size_t base = 0;
    for (int32_t l : g.cols) {
      for (size_t q = 0; q < rx[l].size(); ++q) {
        const int32_t t = rx[l][q];
        local[net->jt_rx[t]] = (int32_t)(base + q);
        P.slot.push_back(net->jt_rx[t]);
        P.slot.push_back(net->jt_partner[t]);
      }
      base += rx[l].size();
      int32_t row = 0;
      for (int32_t e : col[l]) {
        if (row++ % g.parts != g.part) continue;
        // its terms by product (the order of the list, which goes by reaction)
        ts.clear();
        for (int32_t t = net->jt_ptr[e]; t < net->jt_ptr[e + 1]; ++t) ts.push_back(t);
        auto at = [&](int32_t t) { return local[net->jt_rx[t]]; };
        auto before = [&](int32_t a, int32_t b) { return at(a) < at(b); };
        if (!std::is_sorted(ts.begin(), ts.end(), before)) std::stable_sort(ts.begin(), ts.end(), before);
        size_t i = 0;
        do {   // one segment per pass that has terms of it (an entry without terms: one, empty)
          const size_t p = ts.empty() ? 0 : at(ts[i]) / kSlots, i0 = i;
          while (i < ts.size() && (size_t)at(ts[i]) < (p + 1) * kSlots) ++i;
          words.clear();
          for (size_t q = i0; q < i; ++q)
            for_coef_parts(net->jt_coef[ts[q]], [&](int c) { words.push_back(coef_word(at(ts[q]) - (int32_t)(p * kSlots), c)); });
          const bool plain = i0 == 0 && !words.empty() && (words[0] & 0x7FFF0000) == 0x3FF00000;
          have[p].insert(have[p].end(), {e | (i0 > 0 ? kCarry : 0), (int32_t)words.size() - (plain ? 1 : 0),
                                         (int32_t)P.term.size(), plain ? words[0] : 0});
          P.term.insert(P.term.end(), words.begin() + (plain ? 1 : 0), words.end());
          while (P.term.size() % 4) P.term.push_back(0);
        } while (i < ts.size());
      }
    }
    const int32_t s0 = (int32_t)(P.slot.size() / 2 - total);
    for (size_t p = 0; p < passes; ++p) {
      const size_t m = have[p].size() / 4;
      o.resize(m);
      for (size_t i = 0; i < m; ++i) o[i] = (int32_t)i;
      const int32_t* hp = have[p].data();
      std::stable_sort(o.begin(), o.end(), [&](int32_t a, int32_t b) {
        const bool pa = hp[4 * a + 3] != 0, pb = hp[4 * b + 3] != 0;
        return pa != pb ? pa : hp[4 * a + 1] > hp[4 * b + 1];
      });
      int32_t plain = 0;
      for (size_t i = 0; i < m; ++i) plain += hp[4 * i + 3] != 0;
      const int32_t z = (int32_t)(P.seg.size() / 4);
      P.pass.insert(P.pass.end(), {s0 + (int32_t)(p * kSlots), s0 + (int32_t)std::min(total, (p + 1) * kSlots), z, z + plain,
                                   z + (int32_t)m, 0, 0, 0});
      for (int32_t i : o) P.seg.insert(P.seg.end(), hp + 4 * i, hp + 4 * i + 4);
      P.slots = std::max(P.slots, std::min<int32_t>(kSlots, (int32_t)(total - p * kSlots)));
    }
    P.group.push_back((int32_t)(P.pass.size() / 8));
  }
  return P;
}

sm_status launch_jac(const sm_net* net, int64_t C, const double* k, const double* y, double* J,
                     int64_t ld, cudaStream_t s) {
  if (C == 0) return SM_OK;
  const JacProg& P = net->jac;
  const int* pass = P.blob.as<int>();
  const int* seg = pass + P.pass.size();
  const int* term = seg + P.seg.size();
  const int* slot = term + P.term.size();
  dim3 grid((unsigned)((C + 31) / 32), (unsigned)(P.group.size() - 1));
  jac_kernel<<<grid, 32 * kWarps, sizeof(double) * 32 * std::max(P.slots, 1), s>>>(
      C, slot + P.slot.size(), reinterpret_cast<const int4*>(pass), reinterpret_cast<const int2*>(slot),
      reinterpret_cast<const int4*>(seg), term, k, y, J, ld);
  SM_TRY_CUDA(cudaGetLastError());
  return SM_OK;
}
