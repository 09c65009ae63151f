// Index programs of the fused per-cell integrator (see cell.h), built once per
// network on the host.
#include <algorithm>
#include <numeric>

#include "cell.h"

namespace {

struct Sliced {
  std::vector<int32_t> off, ent;   // off in rows of 32 words
  int32_t slices() const { return (int32_t)off.size() - 1; }
  Sliced() : off(1, 0) {}
};

// Appends the items (lists of words) named by `order` as slices of 32 lanes.
void add_slices(const std::vector<std::vector<int32_t>>& items, const std::vector<int32_t>& order, int32_t pad,
                Sliced* s) {
  for (size_t b = 0; b < order.size(); b += 32) {
    size_t len = 0;
    for (size_t l = b; l < std::min(order.size(), b + 32); ++l) len = std::max(len, items[order[l]].size());
    const size_t base = s->ent.size();
    s->ent.resize(base + 32 * len, pad);
    for (size_t l = b; l < std::min(order.size(), b + 32); ++l)
      for (size_t e = 0; e < items[order[l]].size(); ++e) s->ent[base + 32 * e + (l - b)] = items[order[l]][e];
    s->off.push_back(s->off.back() + (int32_t)len);
  }
}

std::vector<int32_t> by_length(const std::vector<std::vector<int32_t>>& items, int32_t lo, int32_t hi) {
  std::vector<int32_t> o(hi - lo);
  std::iota(o.begin(), o.end(), lo);
  std::stable_sort(o.begin(), o.end(), [&](int32_t a, int32_t b) { return items[a].size() > items[b].size(); });
  return o;
}

// Rows of words cut into pieces; piece results land row-contiguously.
struct Pieces {
  Sliced s;
  std::vector<int32_t> dst, row_ptr, lng;
  int32_t n_part = 0;
};
constexpr int kLongRow = 4;   // rows of more pieces are summed by a warp

Pieces cut_rows(const std::vector<std::vector<int32_t>>& rows, int32_t pad) {
  size_t words = 0;
  for (auto& r : rows) words += r.size();
  // about 24 slices of pieces where the rows are long enough, so that every
  // warp of a CTA has one or two; pieces of 4 to 32 entries
  const size_t len = std::min<size_t>(32, std::max<size_t>(4, (words + 767) / 768));
  Pieces p;
  std::vector<std::vector<int32_t>> items;
  p.row_ptr.push_back(0);
  for (size_t i = 0; i < rows.size(); ++i) {
    const size_t n = rows[i].size(), np = (n + len - 1) / len;
    for (size_t q = 0; q < np; ++q)
      items.emplace_back(rows[i].begin() + n * q / np, rows[i].begin() + n * (q + 1) / np);
    p.row_ptr.push_back((int32_t)items.size());
    if (np > kLongRow) p.lng.push_back((int32_t)i);
  }
  p.n_part = (int32_t)items.size();
  const std::vector<int32_t> order = by_length(items, 0, p.n_part);
  add_slices(items, order, pad, &p.s);
  p.dst = order;
  p.dst.resize((size_t)p.s.slices() * 32, p.n_part);   // pad lanes write one slot past the pieces
  return p;
}

}  // namespace

void build_cell_prog(const sm_net* net, CellProg* out) {
  CellProg p;
  const LUSymbolic& lu = net->lu;
  const int32_t n = net->n_s, n_r = net->n_r, h = lu.head, nt = n - h;
  p.nb = (nt + 31) / 32;
  p.pitch = nt | 1;
  if (n >= 65535 || lu.p_d >= 65535 || (int64_t)32 * p.pitch >= 65536) {
    *out = std::move(p);
    return;
  }
  auto put = [&](const std::vector<int32_t>& v) {
    const int32_t o = (int32_t)p.h.size();
    p.h.insert(p.h.end(), v.begin(), v.end());
    p.h.resize((p.h.size() + 31) / 32 * 32, 0);   // every list starts on a 128-byte line
    return o;
  };
  const int32_t kSign = (int32_t)0x80000000;
  // right-hand side
  {
    std::vector<std::vector<int32_t>> rows(n);
    for (int32_t j = 0; j < n_r; ++j)
      for (int32_t q = net->s_colptr[j]; q < net->s_colptr[j + 1]; ++q)
        for (int c = std::abs((int)net->s_coef[q]); c > 0; --c)
          rows[net->s_row[q]].push_back(j | (net->s_coef[q] < 0 ? kSign : 0));
    const Pieces r = cut_rows(rows, n_r);
    p.n_rsl = r.s.slices();
    p.n_part = r.n_part;
    p.n_rlong = (int32_t)r.lng.size();
    p.rp_off = put(r.s.off);
    p.rp_ent = put(r.s.ent);
    p.rp_dst = put(r.dst);
    p.row_ptr = put(r.row_ptr);
    p.row_long = put(r.lng);
  }
  // reactant incidences
  {
    std::vector<std::vector<int32_t>> rows(n);
    for (int32_t j = 0; j < n_r; ++j) {
      const int32_t a = net->reac[2 * j], b = net->reac[2 * j + 1];
      rows[a].push_back(2 * j);
      if (b >= 0) rows[b].push_back(2 * j + 1);
    }
    const Pieces r = cut_rows(rows, 2 * n_r);
    p.n_vsl = r.s.slices();
    p.n_vpart = r.n_part;
    p.n_vlong = (int32_t)r.lng.size();
    p.vp_off = put(r.s.off);
    p.vp_ent = put(r.s.ent);
    p.vp_dst = put(r.dst);
    p.vrow_ptr = put(r.row_ptr);
    p.vrow_long = put(r.lng);
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
  auto tail_pos = [&](int32_t i, int32_t j) { return ((j - h) % 32) * p.pitch + (i - h); };
  // Jacobian entries by destination group
  {
    const int32_t ng = 1 + p.nb;
    std::vector<std::vector<int32_t>> items(net->jp_col.size());
    std::vector<int32_t> rc(items.size()), dst(items.size()), grp(items.size());
    for (int32_t i = 0; i < n; ++i)
      for (int32_t e = net->jp_ptr[i]; e < net->jp_ptr[i + 1]; ++e) {
        const int32_t l = net->jp_col[e], pi = lu.iperm[i], pl = lu.iperm[l];
        for (int32_t t = net->jt_ptr[e]; t < net->jt_ptr[e + 1]; ++t) {
          const int32_t j = net->jt_rx[t], cf = net->jt_coef[t];
          const int32_t w = 2 * j + (net->reac[2 * j] == l ? 0 : 1);
          for (int c = std::abs(cf); c > 0; --c) items[e].push_back(w | (cf < 0 ? kSign : 0));
        }
        rc[e] = i | (l << 16);
        const bool tail = pi >= h && pl >= h;
        grp[e] = tail ? 1 + (pl - h) / 32 : 0;
        dst[e] = tail ? tail_pos(pi, pl) : hpos[(size_t)pi * n + pl];
      }
    std::vector<std::vector<int32_t>> in(ng), lng(ng);
    for (size_t e = 0; e < items.size(); ++e)
      (items[e].size() > (size_t)kJLong ? lng : in)[grp[e]].push_back((int32_t)e);
    Sliced s;
    std::vector<int32_t> g(1, 0), src, sd, sr, lp(1, 0), le, lr, ld, lg(1, 0);
    for (int32_t q = 0; q < ng; ++q) {
      std::stable_sort(in[q].begin(), in[q].end(),
                       [&](int32_t a, int32_t b) { return items[a].size() > items[b].size(); });
      add_slices(items, in[q], 2 * n_r, &s);
      for (int32_t e : in[q]) {
        sr.push_back(rc[e]);
        sd.push_back(dst[e]);
      }
      sr.resize((size_t)s.slices() * 32, 0);
      sd.resize((size_t)s.slices() * 32, -1);
      g.push_back(s.slices());
      for (int32_t e : lng[q]) {
        le.insert(le.end(), items[e].begin(), items[e].end());
        lp.push_back((int32_t)le.size());
        lr.push_back(rc[e]);
        ld.push_back(dst[e]);
      }
      lg.push_back((int32_t)ld.size());
    }
    p.n_jsl = s.slices();
    p.n_jl = (int32_t)ld.size();
    p.jg_off = put(s.off);
    p.jg_ent = put(s.ent);
    p.jg_rc = put(sr);
    p.jg_dst = put(sd);
    p.jg_grp = put(g);
    p.jl_ptr = put(lp);
    p.jl_ent = put(le);
    p.jl_rc = put(lr);
    p.jl_dst = put(ld);
    p.jl_grp = put(lg);
  }
  // head program, terms packed
  {
    std::vector<int32_t> op, tm;
    const size_t nops = lu.hop_piv.size();
    for (size_t o = 0; o < nops; ++o) {
      op.push_back(lu.hop[4 * o] | (lu.hop_piv[o] >= 0 ? lu.hop_piv[o] << 16 : (int32_t)0xFFFF0000));
      op.push_back(lu.hop[4 * o + 2]);
    }
    op.push_back(0);
    op.push_back((int32_t)lu.hterm.size() / 2);
    for (size_t t = 0; t < lu.hterm.size(); t += 2) tm.push_back(lu.hterm[t] | (lu.hterm[t + 1] << 16));
    p.hop = put(op);
    p.hterm = put(tm);
    p.hop_ptr = put(lu.hop_ptr);
  }
  // Schur targets by panel
  {
    std::vector<std::vector<int32_t>> tgt((size_t)nt * nt);
    for (int32_t k = 0; k < h; ++k)
      for (int32_t a = lu.lptr[k]; a < lu.lptr[k + 1]; ++a) {
        const int32_t i = lu.lidx[a];
        if (i < h) continue;
        for (int32_t b = lu.uptr[k]; b < lu.uptr[k + 1]; ++b) {
          const int32_t j = lu.uidx[b];
          if (j >= h)
            tgt[(size_t)(j - h) * nt + (i - h)].push_back(hpos[(size_t)i * n + k] | (hpos[(size_t)k * n + j] << 16));
        }
      }
    Sliced s;
    std::vector<int32_t> g(1, 0), pos;
    for (int32_t J = 0; J < p.nb; ++J) {
      const int32_t lo = 32 * J * nt, hi = std::min(32 * (J + 1), nt) * nt;
      std::vector<int32_t> o = by_length(tgt, lo, hi);
      while (!o.empty() && tgt[o.back()].empty()) o.pop_back();
      add_slices(tgt, o, lu.p_d | (lu.p_d << 16), &s);
      for (int32_t q : o) pos.push_back(tail_pos(h + q % nt, h + q / nt));
      pos.resize((size_t)s.slices() * 32, -1);
      g.push_back(s.slices());
    }
    p.n_tsl = s.slices();
    p.tg_grp = put(g);
    p.tg_off = put(s.off);
    p.tg_ent = put(s.ent);
    p.tg_pos = put(pos);
  }
  // levels of the head rows and columns of U12
  {
    std::vector<int32_t> lf(h, 0), lb(h, 0), uc;
    for (size_t l = 0; l + 1 < lu.flev_ptr.size(); ++l)
      for (int32_t q = lu.flev_ptr[l]; q < lu.flev_ptr[l + 1]; ++q) lf[lu.flev[q]] = (int32_t)l;
    for (size_t l = 0; l + 1 < lu.blev_ptr.size(); ++l)
      for (int32_t q = lu.blev_ptr[l]; q < lu.blev_ptr[l + 1]; ++q) lb[lu.blev[q]] = (int32_t)l;
    for (int32_t k = 0; k < h; ++k)
      for (int32_t q = lu.uoff[(size_t)k * (p.nb + 1)]; q < lu.uptr[k + 1]; ++q) uc.push_back(lu.uidx[q] - h);
    p.lev_f = put(lf);
    p.lev_b = put(lb);
    p.u12c = put(uc);
  }
  p.ok = true;
  *out = std::move(p);
}

CellPlan cell_plan(const sm_net* net, size_t esz, bool thermal, size_t smem_max) {
  CellPlan c;
  const CellProg& p = net->cell;
  const LUSymbolic& lu = net->lu;
  const int n = net->n_s, n_r = net->n_r, h = lu.head;
  // FP64 blocks of 32 rows are shared by two warps (16 columns each)
  const int lw = p.nb * (esz == 8 ? 2 : 1);
  c.warps = std::max(8, lw);
  if (!p.ok || c.warps > 22) return c;   // 22 warps x 88 registers a thread fill the register file
  auto up = [](size_t v) { return (int)((v + 15) / 16 * 16); };
  c.nv = (n + 1) / 2 * 2;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const int at = (int)o;
    o = up(o + bytes);
    return at;
  };
  const size_t vec = sizeof(double) * c.nv;
  c.o_red = take(sizeof(double) * 4 * 32);
  c.o_s = take(512);
  c.o_yp = take(vec);
  c.o_ps = take(vec);
  c.o_ws = take(vec);
  c.o_wf = take(vec);
  c.o_u = (int)o;
  size_t top = o;
  auto phase = [&]() { top = std::max(top, o); o = c.o_u; };
  // Newton rounds: the right-hand side's tables, then (in their place) the
  // substitution's vectors
  c.o_ys = take(vec);
  c.o_fs = take(vec);
  const size_t o_b = o;
  c.o_r = take(sizeof(double) * (n_r + 1));
  c.o_part = take(sizeof(double) * (std::max(p.n_part, thermal ? p.n_vpart : 0) + 1));
  top = std::max(top, o);
  o = o_b;
  c.o_xh = take(esz * std::max(h, 1));
  c.o_xt = take(esz * 32 * p.nb);
  c.o_tmp = take(esz * std::max<size_t>(1, std::max(lu.lrhoff.back(), lu.u12off.back())));
  phase();
  // Jacobian gather (vpart of the coupled temperature follows the table)
  c.o_dr = take(sizeof(double) * (2 * (size_t)n_r + 1));
  c.o_wsf = take(sizeof(float) * n);
  c.o_wif = take(sizeof(float) * n);
  c.o_vp = take(thermal ? sizeof(double) * (p.n_vpart + 1) : 0);
  phase();
  c.o_hv = take(esz * (lu.p_d + 1));
  c.o_x = take(esz * 32 * p.pitch);
  c.o_xk = take(esz * 2 * 32 * 40);
  c.o_ld = take(esz * 2 * 32 * 32);
  phase();
  c.bytes = top;
  c.ok = top <= smem_max;
  const size_t mb = esz * ((size_t)p.n_jsl * 32 + p.n_jl);
  c.scratch = (int64_t)((n_r + 31) / 32 * 32 + (QMAX_HIST + 1) * (int64_t)((n + 31) / 32 * 32) + (mb + 7) / 8 + 32) / 32 * 32;
  return c;
}
