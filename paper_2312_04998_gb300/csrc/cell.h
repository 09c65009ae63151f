// The fused per-cell integrator: index programs (host), shared-memory plan and
// launch interface of cell.cu.
#pragma once

#include "internal.h"

namespace integ { struct Dev; }

void build_cell_prog(const sm_net* net, CellProg* p);

// Start of every CTA's shared memory: the launch's arguments, the cell's
// scalars, the reduction slots (5 of 16 doubles) and 8 doubles more (kRedX).
constexpr int kCellArgs = 1440, kCellScalars = 464, kRedX = 5 * 16;
constexpr int kCellRed = kCellArgs + kCellScalars, kCellFixed = kCellRed + (kRedX + 8) * 8;
constexpr int kGroup = 4;               // tail columns a warp assembles at a time
constexpr int kMaxCellThreads = 384;

// Shared-memory plan of the fused kernel (byte offsets) for one precision.
struct CellPlan {
  bool ok = false;
  int warps = 0, nv = 0;
  int o_ip, o_hx, o_yp, o_ps, o_ws, o_wf, o_wi, o_u;   // o_u: start of the phase-shared area
  int o_nv;                                            // error test
  int o_ys, o_fs, o_r, o_part, o_xh, o_xt, o_hd, o_dg;   // Newton rounds
  int o_dr, o_wsf, o_wif, o_vp;                     // Jacobian gather
  int o_hv, o_x, asm_tile, asm_warps;               // head, assembly (tile size in elements, warps with one)
  int o_lp, o_up, o_uj, o_lj, o_lbuf, o_next;        // tail
  size_t bytes = 0;
  int64_t scratch = 0;   // doubles of global scratch per CTA
};

// Plan for a network in FP64 (esz 8) or FP32 (esz 4) factors,
// with CTAs of `warps` warps; tf: tensor-core updates.
CellPlan cell_plan(const sm_net* net, size_t esz, bool tf, bool thermal, int warps, size_t smem_max);

constexpr int QMAX_HIST = 6;   // history points of a cell

// One CTA shape and the CTAs of it that fit the device at once.
struct CellShape {
  CellPlan plan;
  int ctas = 0;
};

struct CellLaunch {
  CellShape wide, narrow;
  int sms = 0;
  double* scratch = nullptr; // plan.scratch doubles per CTA
  int* ring = nullptr;       // work queue: [0] head, [1] tail, [2..] cells + 1
  int* done = nullptr;       // [ld] attempts made by each cell in this launch
  double* timing = nullptr;  // device: [0] cycles in the timed class, [1] its passes
  int timing_kind = 0;
  int max_ctas() const { return wide.ctas > narrow.ctas ? wide.ctas : narrow.ctas; }
};

// The CTA shapes for a state (no shape has CTAs: the network does not fit).
sm_status cell_shapes(const sm_net* net, const integ::Dev& d, bool thermal, int per_sm_cap, CellLaunch* L);
// f0, h0 and the start values of every cell from the caller's y (and k).
sm_status launch_cell_init(const sm_net* net, const integ::Dev& d, const CellLaunch& L, const double* y, int64_t ldu,
                           const double* k, int64_t ldk, cudaStream_t s);
// Up to `attempts` BDF attempts of every running cell; the ring must hold
// cell_ring_ints.
int64_t cell_ring_ints(const CellLaunch& L, int64_t C, int attempts);
sm_status launch_cell_attempts(const sm_net* net, const integ::Dev& d, const CellLaunch& L, const double* k,
                               int64_t ldk, int attempts, cudaStream_t s);
