// The fused per-cell integrator: index programs (host), shared-memory plan and
// launch interface of cell.cu.
#pragma once

#include "internal.h"

namespace integ { struct Dev; }

void build_cell_prog(const sm_net* net, CellProg* p);

// Shared-memory plan of the fused kernel (byte offsets) for one precision.
struct CellPlan {
  bool ok = false;
  int warps = 0, nv = 0;
  int o_red, o_s, o_yp, o_ps, o_ws, o_wf, o_u;      // o_u: start of the phase-shared area
  int o_ys, o_fs, o_r, o_part, o_xh, o_xt, o_tmp;   // Newton rounds
  int o_dr, o_wsf, o_wif, o_vp;                     // Jacobian gather
  int o_hv, o_x, o_xk, o_ld;                        // factorisation
  size_t bytes = 0;
  int64_t scratch = 0;   // doubles of global scratch per CTA
};

// Plan for a network in FP64 (esz 8) or FP32 (esz 4) factors.
CellPlan cell_plan(const sm_net* net, size_t esz, bool thermal, size_t smem_max);

constexpr int QMAX_HIST = 6;   // history points of a cell

struct CellLaunch {
  CellPlan plan;
  int ctas = 0;              // resident CTAs
  double* scratch = nullptr; // ctas * plan.scratch doubles
  int* ring = nullptr;       // work queue: [0] head, [1] tail, [2..] cells + 1
  int* done = nullptr;       // [ld] attempts made by each cell in this launch
  double* timing = nullptr;  // device: [0] cycles in the timed class, [1] its passes
  int timing_kind = 0;
};

// CTAs of the fused kernel that fit the device at once (0: none).
sm_status cell_resident(const integ::Dev& d, const CellPlan& plan, int per_sm_cap, int* ctas);
// f0, h0 and the start values of every cell from the caller's y (and k).
sm_status launch_cell_init(const sm_net* net, const integ::Dev& d, const CellLaunch& L, const double* y, int64_t ldu,
                           const double* k, int64_t ldk, cudaStream_t s);
// Up to `attempts` BDF attempts of every running cell; *ring_ints is the
// size the ring must have.  Returns the number of kernels launched in *launched.
int64_t cell_ring_ints(int64_t C, int ctas, int attempts);
sm_status launch_cell_attempts(const sm_net* net, const integ::Dev& d, const CellLaunch& L, const double* k,
                               int64_t ldk, int attempts, cudaStream_t s);
