// Right-hand side f = S R(x) (Eq. 7), batched with cells as the fast axis.
//
// Four traversals of S, the GPU counterparts of the paper's Listings 1-4:
//  * CRS  (Listing 3): rows gathered; the nonzeros of S are cut into equal
//    chunks (a warp or half-warp each) so the long hub rows (H: ~2000
//    nonzeros) are shared; rows split across chunks are summed in chunk order
//    through shared memory, so results are deterministic.
//  * COO  (Listing 1): each nonzero adds coef * R_col into f_row (two indirect
//    indices, FP64 atomics in L2).
//  * CCS  (Listing 2): each reaction's rate is formed once in registers and
//    scattered to its (at most six) species (FP64 atomics in L2).
//  * SELL-C-sigma (Listing 4): one thread per (cell, row of a slice) walks
//    the slice column-major, pads included.
// In every traversal a lane owns one cell: index loads are warp-uniform
// broadcasts and abundance / rate loads are 128-byte coalesced rows.
#include <algorithm>
#include <atomic>
#include <mutex>
#include <type_traits>

#include "internal.h"

namespace {

__constant__ double c_coef[256];  // (double)(int8_t)i : coefficient decode table
constexpr int kCells = 16;        // cells per CTA (half a warp)
constexpr int kChunks = 32;       // CRS nonzero chunks per CTA (two per warp)
constexpr int kRThreads = 128;
constexpr int kRChunk = 64;

__device__ __forceinline__ double neg_if(double v, bool neg) {
  return neg ? __longlong_as_double(__double_as_longlong(v) ^ (1ll << 63)) : v;
}

// R_j = k'_j * x_a * x_b, multiplied left to right.
__global__ void __launch_bounds__(kRThreads)
reaction_rate_kernel(int n_r, int64_t C, const int2* __restrict__ reac, const double* __restrict__ k,
                     int64_t ldk, const double* __restrict__ y, int64_t ldy, double* __restrict__ r,
                     int64_t ldr, int chunk, const int* __restrict__ mask, int bit, const int* __restrict__ cact) {
  if (cact && (int64_t)blockIdx.x * kRThreads >= *cact) return;   // no running cell in this block
  const int64_t c = (int64_t)blockIdx.x * kRThreads + threadIdx.x;
  const bool act = c < C && (!mask || (mask[c] & bit));
  if (mask && !__syncthreads_or(act)) return;
  if (!act) return;
  const int j1 = min(n_r, (int)(blockIdx.y + 1) * chunk);
#pragma unroll 4
  for (int j = blockIdx.y * chunk; j < j1; ++j) {
    const int2 a = __ldg(reac + j);
    double v = k[(int64_t)j * ldk + c] * y[(int64_t)a.x * ldy + c];
    if (a.y >= 0) v *= y[(int64_t)a.y * ldy + c];
    r[(int64_t)j * ldr + c] = v;
  }
}

// Reactions per thread of that kernel: kRChunk, fewer where that leaves less
// than 16 warps per SM (37 cells of 180 reactions: the kernel's latency is one
// round of loads, not 16).
int rate_chunk(int64_t n_r, int64_t C) {
  constexpr int kSms = 152;
  const int64_t fit = n_r * ((C + 31) / 32) / (16 * kSms);
  return (int)std::min<int64_t>(kRChunk, std::max<int64_t>(4, fit));
}

// Whether the SELL kernel reads ahead.  A row of the longest slice is a chain of
// L entries, the batch's entries (pads included) fill the device's threads
// `rounds` times for as long; ahead / not, over 32, 120 and 470 species, slice
// heights 8 to 32 and 37 to 65,536 cells: 0.26 to 0.89 at up to 0.8 rounds, 0.92
// to 1.01 at 1.3 to 2.1, 0.99 to 1.11 from 2.4 on.
bool sell_ahead(const Format& F, int64_t C) {
  constexpr double kThreads = 152 * 2048.0;
  const double rounds = (double)F.packed.size() * (double)C / (kThreads * std::max(F.longest, 1));
  return rounds < 2.25;
}

// sum over entries [b, e) of coef * r[col]: four independent partial sums, U
// entries' loads in flight (index words, then rates: the gather waits for
// memory, not for the FP64 unit).  Eight for a warp per chunk; the half-warps of
// the masked gather are no faster with them (4096 cells: 431 us, 426 with four).
template <int U>
__device__ __forceinline__ double dot_range(const uint32_t* __restrict__ ent, int b, int e,
                                            const double* __restrict__ r, int64_t ldr, int64_t c) {
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  int p = b;
  auto run = [&](auto n) {
    constexpr int N = decltype(n)::value;
    for (; p + N - 1 < e; p += N) {
      uint32_t w[N];
      double v[N];
#pragma unroll
      for (int u = 0; u < N; ++u) w[u] = __ldg(ent + p + u);
#pragma unroll
      for (int u = 0; u < N; ++u) v[u] = r[(int64_t)(w[u] & 0xFFFFFFu) * ldr + c];
#pragma unroll
      for (int u = 0; u < N; ++u) s[u % 4] = fma(c_coef[w[u] >> 24], v[u], s[u % 4]);
    }
  };
  if constexpr (U == 8) run(std::integral_constant<int, 8>());
  run(std::integral_constant<int, 4>());
  for (; p < e; ++p) {
    const uint32_t w0 = __ldg(ent + p);
    s[0] = fma(c_coef[w0 >> 24], r[(int64_t)(w0 & 0xFFFFFFu) * ldr + c], s[0]);
  }
  return (s[0] + s[1]) + (s[2] + s[3]);
}

// CRS gather of KC cells per block (cells as the fast axis) with KCH nonzero
// chunks of about equal size, KC x KCH = 512 threads; a warp covers 32 / KC
// chunks.  Rows split across chunks are summed in chunk order through shared
// memory, so results do not depend on scheduling.
template <int KC, int KCH>
__global__ void __launch_bounds__(KC * KCH)
rhs_crs_kernel(int n_s, int64_t C, const int* __restrict__ row_ptr, const uint32_t* __restrict__ ent,
               const int* __restrict__ row_id, const int4* __restrict__ chunk,
               const double* __restrict__ r, int64_t ldr, double* __restrict__ f, int64_t ld,
               const int* __restrict__ mask, int bit, const int* __restrict__ cact) {
  static_assert(KC * KCH == kCells * kChunks && 32 % KC == 0, "block shape");
  if (cact && (int64_t)blockIdx.x * KC >= *cact) return;      // no running cell in this block
  __shared__ double part[KCH][2][KC];
  __shared__ int carry_row[KCH];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ch = warp * (32 / KC) + lane / KC, cl = lane % KC;
  const int64_t c0 = (int64_t)blockIdx.x * KC + cl;
  const bool live = c0 < C && (!mask || (mask[c0] & bit));
  if (mask && !__syncthreads_or(live)) return;
  const int64_t c = live ? c0 : 0;  // dead lanes read cell 0 and store nothing
  // per chunk {end, row that it goes on with (-1: none), first and end of the
  // rows that begin in it}; its first nonzero is the end of the chunk before
  const int4 ci = __ldg(chunk + ch);
  const int z0 = ch > 0 ? __ldg(&chunk[ch - 1].x) : 0, z1 = ci.x, rc = ci.y;
  const double carry = rc >= 0 ? dot_range<4>(ent, z0, min(__ldg(row_ptr + rc + 1), z1), r, ldr, c) : 0.0;
  // -2 marks an empty chunk (possible when nnz < KCH): fix-ups skip it
  if (cl == 0) carry_row[ch] = z0 == z1 ? -2 : rc;
  part[ch][0][cl] = carry;
  const int r_first = ci.z, r_end = ci.w;
  double tail = 0.0;
  int tail_row = -1;
  // (Reading the next row's end and place ahead, as the cluster kernel does, is
  // slower here, where an SM has 48 warps to cover these loads: right-hand sides
  // of 32,768 cells' first 3e-4 yr 0.83 s with it, 0.70 s without.)
  for (int row = r_first; row < r_end; ++row) {
    const int b = __ldg(row_ptr + row), e = __ldg(row_ptr + row + 1);
    const double s = dot_range<4>(ent, b, min(e, z1), r, ldr, c);
    if (e <= z1) {
      if (live) f[(int64_t)__ldg(row_id + row) * ld + c] = s;
    } else {
      tail = s;
      tail_row = row;
    }
  }
  part[ch][1][cl] = tail;
  __syncthreads();
  if (tail_row >= 0) {
    double tot = part[ch][1][cl];
    for (int w = ch + 1; w < KCH; ++w) {
      if (carry_row[w] == -2) continue;
      if (carry_row[w] != tail_row) break;
      tot += part[w][0][cl];
    }
    if (live) f[(int64_t)__ldg(row_id + tail_row) * ld + c] = tot;
  }
}

// The same sums for every cell (rhs_eval): a warp per chunk and 32 cells, the 32
// chunks of a group over a cluster of eight CTAs, which pass the parts of split
// rows through distributed shared memory.  With 16 cells per chunk the two
// halves of a warp walked rows of different lengths in turns; and a CTA of all
// chunks left 4096 cells as 256 CTAs, 2 on some SMs and 1 on others (1024 small
// ones: 7 or 6).  470 species, rates and gather, L2 flushed, one CTA per 16 cells
// / this: 199 / 112 us for 33 cells, 218 / 137 for 1024, 435 / 346 for 4096, 834 /
// 610 for 8192; the smaller networks tried (120, 32 species) gain at every size
// too.  4096 cells: FP64 arithmetic takes 255 us.
constexpr int kClChunks = 4, kCl = kChunks / kClChunks;

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t remote(const void* p, int rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}

__global__ void __cluster_dims__(kCl, 1, 1) __launch_bounds__(32 * kClChunks)
rhs_crs_cluster_kernel(int64_t C, const int* __restrict__ row_ptr, const uint32_t* __restrict__ ent,
                       const int* __restrict__ row_id, const int4* __restrict__ chunk, const double* __restrict__ r,
                       int64_t ldr, double* __restrict__ f, int64_t ld) {
  __shared__ double part[kClChunks][32];   // the part of the row that the chunk goes on with
  __shared__ int carry_row[kClChunks];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ch = (blockIdx.x % kCl) * kClChunks + warp;
  const int64_t c0 = (int64_t)(blockIdx.x / kCl) * 32 + lane;
  const bool live = c0 < C;
  const int64_t c = live ? c0 : 0;  // dead lanes read cell 0 and store nothing
  const int4 ci = __ldg(chunk + ch);
  const int z0 = ch > 0 ? __ldg(&chunk[ch - 1].x) : 0, z1 = ci.x, rc = ci.y;
  part[warp][lane] = rc >= 0 ? dot_range<8>(ent, z0, min(__ldg(row_ptr + rc + 1), z1), r, ldr, c) : 0.0;
  if (lane == 0) carry_row[warp] = z0 == z1 ? -2 : rc;   // -2: empty chunk
  double tail = 0.0;
  int tail_row = -1, tail_id = 0;
  int b = ci.z < ci.w ? __ldg(row_ptr + ci.z) : 0, e = ci.z < ci.w ? __ldg(row_ptr + ci.z + 1) : 0;
  int id = ci.z < ci.w ? __ldg(row_id + ci.z) : 0;
  for (int row = ci.z; row < ci.w; ++row) {   // (the next row's end and place are read ahead)
    const bool more = row + 1 < ci.w;
    const int e2 = more ? __ldg(row_ptr + row + 2) : 0, id2 = more ? __ldg(row_id + row + 1) : 0;
    const double s = dot_range<8>(ent, b, min(e, z1), r, ldr, c);
    if (e <= z1) {
      if (live) f[(int64_t)id * ld + c] = s;
    } else {
      tail = s;
      tail_row = row;
      tail_id = id;
    }
    b = e;
    e = e2;
    id = id2;
  }
  cluster_sync();
  if (tail_row >= 0) {
    for (int w = ch + 1; w < kChunks; ++w) {
      int from;
      double v;
      asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(from) : "r"(remote(&carry_row[w % kClChunks], w / kClChunks)));
      if (from == -2) continue;
      if (from != tail_row) break;
      asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(remote(&part[w % kClChunks][lane], w / kClChunks)));
      tail += v;
    }
    if (live) f[(int64_t)tail_id * ld + c] = tail;
  }
  cluster_sync();   // the parts stay until everyone has read them
}

// COO: nonzeros in column-major order; ent = row | coef, col[] = reaction.
__global__ void __launch_bounds__(kRThreads)
rhs_coo_kernel(int nnz, int64_t C, const uint32_t* __restrict__ ent, const int* __restrict__ col,
               const double* __restrict__ r, int64_t ldr, double* __restrict__ f, int64_t ld) {
  const int64_t c = (int64_t)blockIdx.x * kRThreads + threadIdx.x;
  if (c >= C) return;
  const int p1 = min(nnz, (int)(blockIdx.y + 1) * kRChunk);
  for (int p = blockIdx.y * kRChunk; p < p1; ++p) {
    const uint32_t w = __ldg(ent + p);
    const int cf = (int)(int8_t)(w >> 24);
    double v = r[(int64_t)__ldg(col + p) * ldr + c];
    if (cf != 1 && cf != -1) v *= (double)(cf < 0 ? -cf : cf);
    atomicAdd(f + (int64_t)(w & 0xFFFFFFu) * ld + c, neg_if(v, cf < 0));
  }
}

// CCS: per reaction, R formed in registers then scattered to its species.
__global__ void __launch_bounds__(kRThreads)
rhs_ccs_kernel(int n_r, int64_t C, const int* __restrict__ col_ptr, const uint32_t* __restrict__ ent,
               const int* __restrict__ col_id, const int2* __restrict__ reac,
               const double* __restrict__ k, const double* __restrict__ y, double* __restrict__ f,
               int64_t ld) {
  const int64_t c = (int64_t)blockIdx.x * kRThreads + threadIdx.x;
  if (c >= C) return;
  const int q1 = min(n_r, (int)(blockIdx.y + 1) * kRChunk);
  for (int q = blockIdx.y * kRChunk; q < q1; ++q) {
    const int j = __ldg(col_id + q);
    const int2 a = __ldg(reac + j);
    double v = k[(int64_t)j * ld + c] * y[(int64_t)a.x * ld + c];
    if (a.y >= 0) v *= y[(int64_t)a.y * ld + c];
    const int pe = __ldg(col_ptr + q + 1);
    for (int p = __ldg(col_ptr + q); p < pe; ++p) {
      const uint32_t w = __ldg(ent + p);
      const int cf = (int)(int8_t)(w >> 24);
      double u = v;
      if (cf != 1 && cf != -1) u *= (double)(cf < 0 ? -cf : cf);
      atomicAdd(f + (int64_t)(w & 0xFFFFFFu) * ld + c, neg_if(u, cf < 0));
    }
  }
}

// SELL-C-sigma: block = kCells cells x C slice rows, one slice per blockIdx.y.
// Bound by the chain of the longest row while a batch is small: 1501 cells of 470
// species took 727 us with each entry's loads waiting for the one before, 285 us
// with them ahead (kAhead).  That takes 72 registers; once there are entries
// enough to keep an SM's 2048 threads busy, the plain loop with its 32 is the
// faster one (see sell_ahead).
template <bool kAhead>
__global__ void rhs_sell_kernel(int64_t C, int slice_h, const int* __restrict__ slice_ptr,
                                const uint32_t* __restrict__ ent, const int* __restrict__ row_id,
                                const double* __restrict__ r, int64_t ldr, double* __restrict__ f,
                                int64_t ld) {
  const int cl = threadIdx.x, rr = threadIdx.y, s = blockIdx.y;
  const int64_t c = (int64_t)blockIdx.x * kCells + cl;
  if (c >= C) return;
  const int i = __ldg(row_id + (int64_t)s * slice_h + rr);
  const int b = __ldg(slice_ptr + s);
  const int L = (__ldg(slice_ptr + s + 1) - b) / slice_h;
  double acc = 0.0;
  const uint32_t* q = ent + b + rr;
  auto entry = [&](int k) {
    const uint32_t w = __ldg(q + k * slice_h);
    acc = fma(c_coef[w >> 24], r[(int64_t)(w & 0xFFFFFFu) * ldr + c], acc);
  };
  if constexpr (kAhead) {
    // a row is one chain of FMAs (2000 in the hub rows): while eight entries are
    // added, the rates of the next eight and the index words of those after are
    // on their way
    constexpr int U = 8;
    auto words = [&](int k, uint32_t (&w)[U]) {
#pragma unroll
      for (int u = 0; u < U; ++u) w[u] = k + U <= L ? __ldg(q + (k + u) * slice_h) : 0;
    };
    auto rates = [&](int k, const uint32_t (&w)[U], double (&v)[U]) {
#pragma unroll
      for (int u = 0; u < U; ++u) v[u] = k + U <= L ? r[(int64_t)(w[u] & 0xFFFFFFu) * ldr + c] : 0.0;
    };
    uint32_t w0[U], w1[U];
    double v0[U];
    words(0, w0);
    words(U, w1);
    rates(0, w0, v0);
    int k = 0;
    for (; k + U <= L; k += U) {
      uint32_t w2[U];
      double v1[U];
      rates(k + U, w1, v1);
      words(k + 2 * U, w2);
#pragma unroll
      for (int u = 0; u < U; ++u) acc = fma(c_coef[w0[u] >> 24], v0[u], acc);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        w0[u] = w1[u];
        w1[u] = w2[u];
        v0[u] = v1[u];
      }
    }
#pragma unroll 1
    for (; k < L; ++k) entry(k);
  } else {
    for (int k = 0; k < L; ++k) entry(k);
  }
  if (i >= 0) f[(int64_t)i * ld + c] = acc;
}

constexpr int kMaxDevices = 64;
std::atomic<bool> g_coef_ready[kMaxDevices];
std::mutex g_coef_mu;

}  // namespace

// Loads the coefficient decode table into `device`'s constant memory (the
// device must be current).  Called once per device when a network is built,
// so that the right-hand-side launches never issue this synchronous copy;
// thread-safe.
sm_status rhs_prepare_device(int device) {
  if (device < 0 || device >= kMaxDevices) return SM_EINVAL;
  if (g_coef_ready[device].load(std::memory_order_acquire)) return SM_OK;
  std::lock_guard<std::mutex> lock(g_coef_mu);
  if (g_coef_ready[device].load(std::memory_order_relaxed)) return SM_OK;
  double t[256];
  for (int i = 0; i < 256; ++i) t[i] = (double)(int8_t)i;
  SM_TRY_CUDA(cudaMemcpyToSymbol(c_coef, t, sizeof(t)));
  g_coef_ready[device].store(true, std::memory_order_release);
  return SM_OK;
}

namespace {

sm_status ensure_coef_table(int device) {
  if (device >= 0 && device < kMaxDevices && g_coef_ready[device].load(std::memory_order_acquire))
    return SM_OK;
  return rhs_prepare_device(device);
}

}  // namespace

sm_status launch_rhs(const sm_net* net, int64_t C, const double* k, const double* y, double* f,
                     int64_t ld, double* scratch, int64_t ldr, cudaStream_t s) {
  if (C == 0) return SM_OK;
  sm_status st = ensure_coef_table(net->device);
  if (st != SM_OK) return st;
  const Format& F = net->cur;
  const unsigned groups_r = (unsigned)((C + kRThreads - 1) / kRThreads);
  if (F.fmt == SM_FMT_CCS) {
    SM_TRY_CUDA(cudaMemsetAsync(f, 0, sizeof(double) * (size_t)net->n_s * ld, s));
    dim3 grid(groups_r, (unsigned)((net->n_r + kRChunk - 1) / kRChunk));
    rhs_ccs_kernel<<<grid, kRThreads, 0, s>>>(net->n_r, C, F.d_ptr.as<int>(), F.d_packed.as<uint32_t>(),
                                              F.d_aux.as<int>(), net->d_reac.as<int2>(), k, y, f, ld);
    SM_TRY_CUDA(cudaGetLastError());
    return SM_OK;
  }
  {
    const int chunk = rate_chunk(net->n_r, C);
    dim3 grid(groups_r, (unsigned)((net->n_r + chunk - 1) / chunk));
    reaction_rate_kernel<<<grid, kRThreads, 0, s>>>(net->n_r, C, net->d_reac.as<int2>(), k, ld, y, ld,
                                                    scratch, ldr, chunk, nullptr, 0, nullptr);
    SM_TRY_CUDA(cudaGetLastError());
  }
  const unsigned groups = (unsigned)((C + kCells - 1) / kCells);
  if (F.fmt == SM_FMT_CRS) {
    if ((int)F.chunk_nz.size() != kChunks + 1) return SM_EINVAL;
    rhs_crs_cluster_kernel<<<(unsigned)((C + 31) / 32) * kCl, 32 * kClChunks, 0, s>>>(
        C, F.d_ptr.as<int>(), F.d_packed.as<uint32_t>(), F.d_aux.as<int>(), F.d_chunk.as<int4>(), scratch, ldr, f, ld);
  } else if (F.fmt == SM_FMT_COO) {
    SM_TRY_CUDA(cudaMemsetAsync(f, 0, sizeof(double) * (size_t)net->n_s * ld, s));
    const int nnz = (int)F.idx.size();
    dim3 grid(groups_r, (unsigned)((nnz + kRChunk - 1) / kRChunk));
    rhs_coo_kernel<<<grid, kRThreads, 0, s>>>(nnz, C, F.d_packed.as<uint32_t>(), F.d_aux.as<int>(),
                                              scratch, ldr, f, ld);
  } else {
    dim3 block(kCells, F.C);
    dim3 grid(groups, (unsigned)F.len.size());
    const auto kernel = sell_ahead(F, C) ? rhs_sell_kernel<true> : rhs_sell_kernel<false>;
    kernel<<<grid, block, 0, s>>>(C, F.C, F.d_ptr.as<int>(), F.d_packed.as<uint32_t>(), F.d_aux.as<int>(), scratch, ldr,
                                  f, ld);
  }
  SM_TRY_CUDA(cudaGetLastError());
  return SM_OK;
}

sm_status launch_rhs_masked(const sm_net* net, int64_t C, const double* k, int64_t ldk,
                            const double* y, double* f, int64_t ld, double* scratch, int64_t ldr,
                            const int* mask, int bit, const int* cact, cudaStream_t s) {
  if (C == 0) return SM_OK;
  sm_status st = ensure_coef_table(net->device);
  if (st != SM_OK) return st;
  const Format& F = net->integ_fmt[net->integ_order];
  if (F.packed.empty()) return SM_EINVAL;
  const int chunk = rate_chunk(net->n_r, C);
  dim3 grid((unsigned)((C + kRThreads - 1) / kRThreads), (unsigned)((net->n_r + chunk - 1) / chunk));
  reaction_rate_kernel<<<grid, kRThreads, 0, s>>>(net->n_r, C, net->d_reac.as<int2>(), k, ldk, y, ld,
                                                  scratch, ldr, chunk, mask, bit, cact);
  SM_TRY_CUDA(cudaGetLastError());
  const int kc = net->integ_kc;
  const unsigned nb = (unsigned)((C + kc - 1) / kc);
  if (kc == 8) {
    rhs_crs_kernel<8, 64><<<nb, kCells * kChunks, 0, s>>>(net->n_s, C, F.d_ptr.as<int>(),
        F.d_packed.as<uint32_t>(), F.d_aux.as<int>(), F.d_chunk64.as<int4>(), scratch, ldr, f, ld, mask, bit, cact);
  } else if (kc == 32) {
    rhs_crs_kernel<32, 16><<<nb, kCells * kChunks, 0, s>>>(net->n_s, C, F.d_ptr.as<int>(),
        F.d_packed.as<uint32_t>(), F.d_aux.as<int>(), F.d_chunk16.as<int4>(), scratch, ldr, f, ld, mask, bit, cact);
  } else {
    rhs_crs_kernel<16, 32><<<nb, kCells * kChunks, 0, s>>>(net->n_s, C, F.d_ptr.as<int>(),
        F.d_packed.as<uint32_t>(), F.d_aux.as<int>(), F.d_chunk.as<int4>(), scratch, ldr, f, ld, mask, bit, cact);
  }
  SM_TRY_CUDA(cudaGetLastError());
  return SM_OK;
}
