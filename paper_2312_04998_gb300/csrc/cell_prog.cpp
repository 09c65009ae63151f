// Index programs of the fused per-cell integrator (see cell.h), built once per
// network on the host.
#include <algorithm>
#include <numeric>

#include "cell.h"

namespace {

struct Sliced {
  std::vector<int32_t> off, ent;   // off: {first row, rows} per slice, rows of 32 words
  int32_t slices() const { return (int32_t)off.size() / 2; }
};

// Appends the items (lists of words) named by `order` as slices of 32 lanes,
// their lengths rounded up to a multiple of `mult`.
void add_slices(const std::vector<std::vector<int32_t>>& items, const std::vector<int32_t>& order, int32_t pad,
                size_t mult, Sliced* s) {
  for (size_t b = 0; b < order.size(); b += 32) {
    size_t len = 0;
    for (size_t l = b; l < std::min(order.size(), b + 32); ++l) len = std::max(len, items[order[l]].size());
    len = (len + mult - 1) / mult * mult;
    const size_t base = s->ent.size();
    s->ent.resize(base + 32 * len, pad);
    for (size_t l = b; l < std::min(order.size(), b + 32); ++l)
      for (size_t e = 0; e < items[order[l]].size(); ++e) s->ent[base + 32 * e + (l - b)] = items[order[l]][e];
    s->off.push_back((int32_t)(base / 32));
    s->off.push_back((int32_t)len);
  }
}
// Empty slices up to a multiple of 4.
void fill_slices(Sliced* s) {
  while (s->slices() % 4) {
    s->off.push_back((int32_t)(s->ent.size() / 32));
    s->off.push_back(0);
  }
}

std::vector<int32_t> by_length(const std::vector<std::vector<int32_t>>& items, int32_t lo, int32_t hi) {
  std::vector<int32_t> o(hi - lo);
  std::iota(o.begin(), o.end(), lo);
  std::stable_sort(o.begin(), o.end(), [&](int32_t a, int32_t b) { return items[a].size() > items[b].size(); });
  return o;
}

// Rows of words cut into chains.  A row is summed as the CRS gather sums it:
// the nonzeros of the matrix in kChunks equal chunks; of a row's part in a
// chunk the entries 0, 4, 8 .., 1, 5, .. and so on are four sums (what is left
// past the last four goes to the first), added as (0 + 1) + (2 + 3); then the
// parts in order.  So a cell's results do not depend on whether its right-hand
// side comes from here or from the gather, to the last bit, and a longest chain
// is an eighth of a hub row.
struct Chains {
  Sliced s;
  // row: first chain | four chains << 31 | (first further part + 1) << 16;
  // more: the further parts, a word each (the last one's bit 30 set)
  std::vector<int32_t> dst, row, more;
  int32_t n_chain = 0;
  bool ok = true;

  // The slices dealt to the nw warps of a CTA: {first, end} of each warp's, then
  // per slice {first row, rows, slice, 0}.  Longest first, each to the scheduler
  // (warp mod 4) with the fewest rows so far and there to the warp with the
  // fewest: dealt in turns, the longest chain shared its scheduler's FP64 unit with
  // two more warps' slices and finished last.
  std::vector<int32_t> deal(int32_t nw) const {
    std::vector<std::vector<int32_t>> mine(nw);
    std::vector<int64_t> load(nw, 0), unit(4, 0);
    for (int32_t k = 0; k < s.slices(); ++k) {   // (slices come longest first)
      const int32_t u = (int32_t)(std::min_element(unit.begin(), unit.end()) - unit.begin());
      int32_t w = u;
      for (int32_t v = u; v < nw; v += 4)
        if (load[v] < load[w]) w = v;
      mine[w].push_back(k);
      load[w] += s.off[2 * k + 1];
      unit[u] += s.off[2 * k + 1];
    }
    std::vector<int32_t> out, list;
    for (int32_t w = 0; w < nw; ++w) {
      out.push_back((int32_t)(2 * nw + list.size()) / 4);
      for (int32_t k : mine[w]) list.insert(list.end(), {s.off[2 * k], s.off[2 * k + 1], k, 0});
      out.push_back((int32_t)(2 * nw + list.size()) / 4);
    }
    out.insert(out.end(), list.begin(), list.end());
    return out;
  }
};
constexpr size_t kChunks = 32;
constexpr int32_t kWide = kMaxCellThreads / 32, kNarrow = 4;   // warps of the two CTA shapes
static_assert(kWide % 4 == 0, "deal: whole schedulers, 16-byte lists");


Chains cut_rows(const std::vector<std::vector<int32_t>>& rows, int32_t pad) {
  size_t words = 0, z = 0, ch = 0;
  for (auto& r : rows) words += r.size();
  Chains p;
  std::vector<std::vector<int32_t>> items;
  for (const auto& r : rows) {
    std::vector<int32_t> parts;
    for (size_t b = 0; b < r.size() || parts.empty();) {
      while (ch + 1 < kChunks && z + b >= words * (ch + 1) / kChunks) ++ch;   // the chunk that holds entry z + b
      const size_t e = ch + 1 < kChunks ? std::min(r.size(), words * (ch + 1) / kChunks - z) : r.size();
      const size_t m = (e - b) / 4 * 4, first = items.size();
      items.resize(first + (m > 0 ? 4 : 1));
      for (size_t q = b; q < e; ++q) items[first + (q - b < m ? (q - b) % 4 : 0)].push_back(r[q]);
      parts.push_back((int32_t)first | (m > 0 ? (int32_t)0x80000000 : 0));
      b = std::max(e, b + 1);
    }
    z += r.size();
    if (parts.size() > 1) parts[0] |= (int32_t)(p.more.size() + 1) << 16;
    p.row.push_back(parts[0]);
    p.more.insert(p.more.end(), parts.begin() + 1, parts.end());
    if (parts.size() > 1) p.more.back() |= 1 << 30;
  }
  p.n_chain = (int32_t)items.size();
  p.ok = items.size() < 65535 && p.more.size() < 16383;
  const std::vector<int32_t> order = by_length(items, 0, p.n_chain);
  add_slices(items, order, pad, 1, &p.s);
  p.dst = order;
  p.dst.resize((size_t)p.s.slices() * 32, p.n_chain);   // pad lanes write one slot past the chains
  return p;
}

}  // namespace

void build_cell_prog(const sm_net* net, CellProg* out) {
  CellProg p;
  const LUSymbolic& lu = net->lu;
  const int32_t n = net->n_s, n_r = net->n_r, h = lu.head, nt = n - h;
  p.nb = (nt + 31) / 32;
  p.pitch = nt | 1;
  if (n >= 65535 || n_r >= 32000 || lu.p_d >= 65535 || (int64_t)kGroup * p.pitch >= 65535 || h >= 32768) {
    *out = std::move(p);
    return;
  }
  auto put = [&](const std::vector<int32_t>& v) {
    const int32_t o = (int32_t)p.h.size();
    p.h.insert(p.h.end(), v.begin(), v.end());
    p.h.resize((p.h.size() + 31) / 32 * 32, 0);   // every list starts on a 128-byte line
    return o;
  };
  bool fits = true;
  std::vector<int32_t> slot(n_r);   // first derivative slot of each reaction
  {
    std::vector<int32_t> rx;
    for (int32_t j = 0; j < n_r; ++j) {
      const int32_t a = net->reac[2 * j], b = net->reac[2 * j + 1];
      slot[j] = p.n_slot;
      p.n_slot += b >= 0 ? 2 : 1;
      rx.push_back((int32_t)((uint32_t)a | (uint32_t)(b >= 0 ? b : 0xFFFF) << 16));
      rx.push_back(slot[j]);
    }
    p.rx = put(rx);
    p.iperm = put(lu.iperm);
  }
  // right-hand side
  {
    std::vector<std::vector<int32_t>> rows(n);
    for (int32_t j = 0; j < n_r; ++j)
      for (int32_t q = net->s_colptr[j]; q < net->s_colptr[j + 1]; ++q)
        for_coef_parts(net->s_coef[q], [&](int c) { rows[net->s_row[q]].push_back(coef_word(j, c)); });
    const Chains r = cut_rows(rows, coef_word(n_r, 1));
    p.n_chain = r.n_chain;
    p.rp_deal[0] = put(r.deal(kWide));
    p.rp_deal[1] = put(r.deal(kNarrow));
    p.rp_ent = put(r.s.ent);
    p.rp_dst = put(r.dst);
    p.row = put(r.row);
    p.row_more = put(r.more);
    fits = fits && r.ok;
  }
  // reactant incidences
  {
    std::vector<std::vector<int32_t>> rows(n);
    for (int32_t j = 0; j < n_r; ++j) {
      const int32_t a = net->reac[2 * j], b = net->reac[2 * j + 1];
      rows[a].push_back(coef_word(slot[j], 1));
      if (b >= 0) rows[b].push_back(coef_word(slot[j] + 1, 1));
    }
    const Chains r = cut_rows(rows, coef_word(p.n_slot, 1));
    p.n_vchain = r.n_chain;
    p.vp_deal[0] = put(r.deal(kWide));
    p.vp_deal[1] = put(r.deal(kNarrow));
    p.vp_ent = put(r.s.ent);
    p.vp_dst = put(r.dst);
    p.vrow = put(r.row);
    p.vrow_more = put(r.more);
    fits = fits && r.ok;
  }
  // packed index of the head's factors (as in the head program of LUSymbolic)
  std::vector<int32_t> hpos((size_t)n * n, -1);   // (row, column) in elimination order -> packed head index
  {
    const int32_t np1 = p.nb + 1;
    for (int32_t i = 0; i < n; ++i)
      for (int32_t q = lu.lrptr[i]; q < lu.lrptr[i + 1]; ++q) {
        const int32_t k = lu.lridx[q];
        if (i < h) hpos[(size_t)i * n + k] = lu.p_l11 + q;
        else if (k < h) hpos[(size_t)i * n + k] = lu.p_l21 + lu.lrhoff[i - h] + (q - lu.lrptr[i]);
      }
    for (int32_t k = 0; k < h; ++k) {
      hpos[(size_t)k * n + k] = lu.p_dinv + k;
      const int32_t q12 = lu.uoff[(size_t)k * np1];
      for (int32_t q = lu.uptr[k]; q < lu.uptr[k + 1]; ++q) {
        const int32_t j = lu.uidx[q];
        hpos[(size_t)k * n + j] = j < h ? lu.p_u11 + lu.u11ptr[k] + (q - lu.uptr[k]) : lu.p_u12 + lu.u12off[k] + (q - q12);
      }
    }
  }
  auto tail_pos = [&](int32_t i, int32_t j) { return ((j - h) % kGroup) * p.pitch + (i - h); };
  // Jacobian entries by destination group
  {
    const int32_t ng = 1 + (nt + kGroup - 1) / kGroup;
    std::vector<std::vector<int32_t>> items(net->jp_col.size());
    std::vector<int32_t> rc(items.size()), dst(items.size()), grp(items.size());
    for (int32_t i = 0; i < n; ++i)
      for (int32_t e = net->jp_ptr[i]; e < net->jp_ptr[i + 1]; ++e) {
        const int32_t l = net->jp_col[e], pi = lu.iperm[i], pl = lu.iperm[l];
        for (int32_t t = net->jt_ptr[e]; t < net->jt_ptr[e + 1]; ++t) {
          const int32_t j = net->jt_rx[t], cf = net->jt_coef[t];
          const int32_t w = slot[j] + (net->reac[2 * j] == l ? 0 : 1);
          if (items[e].empty() && cf != 1 && cf != -1) items[e].push_back(coef_word(p.n_slot, 1));   // (see cell_jacobian)
          for_coef_parts(cf, [&](int c) { items[e].push_back(coef_word(w, c)); });
        }
        if (items[e].empty()) items[e].push_back(coef_word(p.n_slot, 1));
        rc[e] = i | (l << 16);
        const bool tail = pi >= h && pl >= h;
        grp[e] = tail ? 1 + (pl - h) / kGroup : 0;
        dst[e] = tail ? tail_pos(pi, pl) : hpos[(size_t)pi * n + pl];
      }
    std::vector<std::vector<int32_t>> in(ng);
    std::vector<int32_t> lng;
    for (size_t e = 0; e < items.size(); ++e)
      if (items[e].size() > (size_t)kJShort) lng.push_back((int32_t)e);
      else in[grp[e]].push_back((int32_t)e);
    Sliced s;
    std::vector<int32_t> g(1, 0), sd, sr;
    for (int32_t q = 0; q < ng; ++q) {
      std::stable_sort(in[q].begin(), in[q].end(),
                       [&](int32_t a, int32_t b) { return items[a].size() > items[b].size(); });
      add_slices(items, in[q], coef_word(p.n_slot, 1), 1, &s);
      for (int32_t e : in[q]) {
        sr.push_back(rc[e]);
        sd.push_back(dst[e]);
      }
      sr.resize((size_t)s.slices() * 32, 0);
      sd.resize((size_t)s.slices() * 32, -1);
      g.push_back(s.slices());
    }
    fill_slices(&s);
    sr.resize((size_t)s.slices() * 32, 0);
    sd.resize((size_t)s.slices() * 32, -1);
    // long entries, longest first: a slice each while they have more than kJLong
    // words (dealt to the lanes in turn), else a slice of 32
    std::stable_sort(lng.begin(), lng.end(), [&](int32_t a, int32_t b) { return items[a].size() > items[b].size(); });
    Sliced ls;
    std::vector<int32_t> lr, at(lng.size()), dg(1, 0), de;
    size_t t = 0;
    for (; t < lng.size() && items[lng[t]].size() > (size_t)kJLong; ++t) {
      const std::vector<int32_t>& it = items[lng[t]];
      std::vector<std::vector<int32_t>> lanes(32);
      std::vector<int32_t> all(32);
      std::iota(all.begin(), all.end(), 0);
      for (size_t e = 0; e < it.size(); ++e) lanes[e % 32].push_back(it[e]);
      at[t] = 32 * ls.slices();
      add_slices(lanes, all, coef_word(p.n_slot, 1), 1, &ls);
      lr.resize((size_t)32 * ls.slices(), 0);
      lr[at[t]] = rc[lng[t]];
    }
    p.n_jw = ls.slices();
    for (; t < lng.size(); t += 32) {
      const size_t m = std::min<size_t>(32, lng.size() - t);
      const int32_t base = 32 * ls.slices();
      add_slices(items, std::vector<int32_t>(lng.begin() + t, lng.begin() + t + m), coef_word(p.n_slot, 1), 1, &ls);
      lr.resize((size_t)32 * ls.slices(), 0);
      for (size_t l = 0; l < m; ++l) {
        at[t + l] = base + (int32_t)l;
        lr[base + l] = rc[lng[t + l]];
      }
    }
    std::vector<std::vector<int32_t>> by(ng);
    for (size_t l = 0; l < lng.size(); ++l) by[grp[lng[l]]].insert(by[grp[lng[l]]].end(), {dst[lng[l]], at[l]});
    for (const auto& v : by) {
      de.insert(de.end(), v.begin(), v.end());
      dg.push_back((int32_t)de.size() / 2);
    }
    p.n_jsl = s.slices();
    p.n_jl = ls.slices();
    p.jg_off = put(s.off);
    p.jg_ent = put(s.ent);
    p.jg_rc = put(sr);
    p.jg_dst = put(sd);
    p.jg_grp = put(g);
    p.jl_off = put(ls.off);
    p.jl_ent = put(ls.ent);
    p.jl_rc = put(lr);
    p.jd_grp = put(dg);
    p.jd_ent = put(de);
  }
  // head program, terms packed
  {
    std::vector<int32_t> op, tm;
    const size_t nops = lu.hop_piv.size();
    for (size_t o = 0; o < nops; ++o) {
      op.push_back(lu.hop[4 * o] | (lu.hop_piv[o] >= 0 ? lu.hop_piv[o] << 16 : (int32_t)0xFFFF0000));
      op.push_back(lu.hop[4 * o + 2]);
      op.push_back(lu.hop[4 * o + 3]);
      op.push_back(0);
    }
    for (size_t t = 0; t < lu.hterm.size(); t += 2) tm.push_back(lu.hterm[t] | (lu.hterm[t + 1] << 16));
    p.hop = put(op);
    p.hterm = put(tm);
    p.hop_ptr = put(lu.hop_ptr);
  }
  // Schur targets by panel
  {
    // every target's terms, in pivot order (counted, then filled)
    std::vector<int32_t> at((size_t)nt * nt + 1, 0), term;
    auto each = [&](auto f) {
      for (int32_t k = 0; k < h; ++k)
        for (int32_t a = lu.lptr[k]; a < lu.lptr[k + 1]; ++a) {
          const int32_t i = lu.lidx[a];
          if (i < h) continue;
          const int32_t l = hpos[(size_t)i * n + k];
          for (int32_t b = lu.uptr[k]; b < lu.uptr[k + 1]; ++b)
            if (lu.uidx[b] >= h) f((size_t)(lu.uidx[b] - h) * nt + (i - h), l, k, lu.uidx[b]);
        }
    };
    each([&](size_t q, int32_t, int32_t, int32_t) { ++at[q + 1]; });
    for (size_t q = 0; q < (size_t)nt * nt; ++q) at[q + 1] += at[q];
    term.resize(at[(size_t)nt * nt]);
    std::vector<int32_t> fill(at.begin(), at.end() - 1);
    each([&](size_t q, int32_t l, int32_t k, int32_t j) { term[fill[q]++] = l | (hpos[(size_t)k * n + j] << 16); });
    std::vector<int32_t> g(1, 0), ent, o;
    const int32_t pad = lu.p_d | (lu.p_d << 16);
    auto size = [&](int32_t q) { return at[q + 1] - at[q]; };
    for (int32_t J = 0; J * kGroup < nt; ++J) {
      o.clear();
      for (int32_t q = kGroup * J * nt; q < std::min(kGroup * (J + 1), nt) * nt; ++q)
        if (size(q) > 0) o.push_back(q);
      std::stable_sort(o.begin(), o.end(), [&](int32_t x, int32_t y) { return size(x) > size(y); });
      for (size_t b = 0; b < o.size(); b += 32) {
        const int32_t len = size(o[b]);
        const size_t base = ent.size();
        ent.resize(base + 32 * ((size_t)len + 1), pad);
        for (size_t l = 0; l < 32; ++l) {
          const bool in = b + l < o.size();
          const int32_t q = in ? o[b + l] : 0;
          ent[base + l] = (in ? tail_pos(h + q % nt, h + q / nt) : 0xFFFF) | (len << 16);
          for (int32_t e = 0; in && e < size(q); ++e) ent[base + 32 * ((size_t)e + 1) + l] = term[at[q] + e];
        }
      }
      g.push_back((int32_t)(ent.size() / 32));
    }
    p.tg_grp = put(g);
    p.tg_ent = put(ent);
  }
  // levels of the head rows and columns of U12
  {
    std::vector<int32_t> lf(h, 0), lb(h, 0), hx(lu.p_d, 0);
    for (size_t l = 0; l + 1 < lu.flev_ptr.size(); ++l)
      for (int32_t q = lu.flev_ptr[l]; q < lu.flev_ptr[l + 1]; ++q) lf[lu.flev[q]] = (int32_t)l;
    for (size_t l = 0; l + 1 < lu.blev_ptr.size(); ++l)
      for (int32_t q = lu.blev_ptr[l]; q < lu.blev_ptr[l + 1]; ++q) lb[lu.blev[q]] = (int32_t)l;
    for (int32_t i = 0; i < h; ++i)
      for (int32_t q = lu.lrptr[i]; q < lu.lrptr[i + 1]; ++q) hx[lu.p_l11 + q] = lu.lridx[q];
    for (size_t q = 0; q < lu.lrhk.size(); ++q) hx[lu.p_l21 + q] = lu.lrhk[q];
    for (int32_t k = 0; k < h; ++k) {
      const int32_t u0 = lu.uptr[k], q12 = lu.uoff[(size_t)k * (p.nb + 1)];
      for (int32_t q = u0; q < q12; ++q) hx[lu.p_u11 + lu.u11ptr[k] + (q - u0)] = lu.uidx[q];
      for (int32_t q = q12; q < lu.uptr[k + 1]; ++q) hx[lu.p_u12 + lu.u12off[k] + (q - q12)] = lu.uidx[q] - h;
    }
    p.lev_f = put(lf);
    p.lev_b = put(lb);
    p.hx = put(hx);
  }
  p.ok = fits;
  *out = std::move(p);
}

CellPlan cell_plan(const sm_net* net, size_t esz, bool tf, bool thermal, int warps, size_t smem_max) {
  CellPlan c;
  const CellProg& p = net->cell;
  const LUSymbolic& lu = net->lu;
  const int n = net->n_s, n_r = net->n_r, h = lu.head;
  c.warps = warps;
  if (!p.ok) return c;
  auto up = [](size_t v) { return (int)((v + 15) / 16 * 16); };
  c.nv = (n + 1) / 2 * 2;
  size_t o = kCellFixed;
  auto take = [&](size_t bytes) {
    const int at = (int)o;
    o = up(o + bytes);
    return at;
  };
  const size_t vec = sizeof(double) * c.nv;
  c.o_ip = take(sizeof(uint16_t) * n);
  c.o_hx = take(sizeof(uint16_t) * lu.p_d);
  c.o_yp = take(vec);
  c.o_ps = take(vec);
  c.o_ws = take(vec);
  c.o_wf = take(esz == 4 ? vec : 0);
  c.o_wi = take(esz == 4 ? vec : 0);
  c.o_u = (int)o;
  size_t top = o;
  auto phase = [&]() { top = std::max(top, o); o = c.o_u; };
  // Newton rounds: the right-hand side's tables, then (in their place) the
  // substitution's vectors
  c.o_ys = take(vec);
  c.o_fs = take(vec);
  const size_t o_b = o;
  c.o_r = take(sizeof(double) * (n_r + 1));
  c.o_part = take(sizeof(double) * (std::max(p.n_chain, thermal ? p.n_vchain : 0) + 1));
  top = std::max(top, o);
  o = o_b;
  c.o_xh = take(esz * std::max(h, 1));
  c.o_xt = take(esz * 32 * p.nb);
  c.o_hd = take(esz * std::max(lu.p_d, 1));
  c.o_dg = take(esz * 1024 * p.nb);
  top = std::max(top, o);
  o = o_b;
  c.o_nv = take(3 * vec);   // the error test's terms
  phase();
  // Jacobian gather (vpart of the coupled temperature follows the table)
  c.o_dr = take(sizeof(double) * ((size_t)p.n_slot + 1));
  c.o_wsf = take(esz == 4 ? sizeof(float) * n : 0);
  c.o_wif = take(esz == 4 ? sizeof(float) * n : 0);
  c.o_vp = take(thermal ? sizeof(double) * (p.n_vchain + 1) : 0);
  phase();
  c.o_hv = take(esz * (lu.p_d + 1));
  {
    // assembly tiles: one per warp as far as they fit
    c.asm_tile = (int)(up(esz * kGroup * p.pitch) / esz);
    const size_t left = smem_max > o ? smem_max - o : 0;
    c.asm_warps = std::min<int>(warps, (int)(left / (esz * c.asm_tile)));
    c.o_x = take(esz * c.asm_tile * std::max(c.asm_warps, 1));
  }
  phase();
  c.o_lp = take(esz * 32 * (tf ? 36 : 32) * std::max(p.nb - 1, 1));
  c.o_up = take(esz * 32 * (tf ? 36 : 32) * std::max(p.nb - 1, 1));
  c.o_uj = take(esz * (32 * 36 + 32));   // (reads past the last row's end stay inside)
  c.o_lj = take(esz * (32 * 32 + 32));
  c.o_lbuf = take(esz * 64);
  c.o_next = take(16);
  phase();
  c.bytes = top;
  c.ok = top <= smem_max && c.asm_warps > 0;
  const size_t mb = esz * 32 * ((size_t)p.n_jsl + p.n_jl);
  c.scratch = (int64_t)((n_r + 31) / 32 * 32 + (QMAX_HIST + 1) * (int64_t)((n + 31) / 32 * 32) + (mb + 7) / 8 + 32) / 32 * 32;
  return c;
}
