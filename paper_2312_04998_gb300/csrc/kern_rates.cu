// Rate coefficients k'[n_r][ld], cells as the fast axis.
//
// The paper precomputes the coefficients outside the stiff solver, once per
// hydro step (Section 3).  k' = alpha (T/300)^beta exp(-gamma/T) n_H is an
// exponential per (reaction, cell), and an FP64 instruction of a warp holds its
// scheduler's FP64 unit for 64 cycles: with a library exp (about 17 of them)
// 98 M coefficients took 2.97 ms, all of it FP64 arithmetic, against 0.12 ms
// for storing them.  So the exponential is mostly integer arithmetic here:
//   log2 k' = beta log2(T/300) - gamma log2(e)/T  (FP64, two instructions at
//   most) + log2 alpha + log2 n_H (fixed point, prepared per reaction and cell)
// as a 64-bit fixed-point number of units 1/4096; its integer part picks
// 2^(i/4096) from a table in shared memory and the binary exponent, the
// fraction's 2^f - 1 < 1.7e-4 is a cubic in integers (remainder below 4e-17),
// put below the leading 1 of a double, and one FP64 product ends it.  The
// rounding of log alpha and n_H, which a sum in FP64 would add at the
// magnitude of the whole exponent, does not arise: 16,384 cells x 6000 reactions
// 2964 -> 881 us, error against 64-bit references 1.8e-15 -> 2.5e-16.
//
// A lane has one cell, a warp a run of reactions (long enough to pay for the
// cell's logarithms, short enough to fill the SMs); reaction parameters are
// warp-uniform broadcasts.
#include <cmath>
#include <cstring>

#include "internal.h"

namespace {

constexpr int kUnits = 4096;      // table entries per octave
constexpr int kFrac = 41;         // fraction bits of the fixed-point numbers (units 1 / kUnits)
constexpr double kLog2e = 1.4426950408889634074;
constexpr int kRatesWarps = 8;
constexpr int kSms = 152;

// log2(v) in units 1 / kUnits, fixed point, given v = 2^e m, 1 <= m < 2, and a
// table entry i close to m: log2 m = i / kUnits + log2(1 + z), z = m / t - 1
// (m - t is exact).  |z| < 5e-4: five terms of the series.
__host__ __device__ inline long long log2_fixed(int e, double m, int i, double t) {
  const double z = (m - t) / t;
  const double p = z * (1.0 + z * (-0.5 + z * (1.0 / 3.0 + z * (-0.25 + z * 0.2))));
  return ((long long)(e * kUnits + i) << kFrac) + (long long)(p * (kUnits * kLog2e) * (double)(1ll << kFrac));
}
constexpr int kMaxLog = 120;      // |log2| of the fixed-point factors: sums stay inside 64 bits

__device__ __forceinline__ bool cell_fixed(double v, const double* tab, long long* out) {
  const int hi = __double2hiint(v);
  const int e = (hi >> 20) - 1023;   // (a negative v: far out of range)
  if (hi < 0 || e < -kMaxLog || e >= kMaxLog) return false;
  const double m = __hiloint2double((hi & 0xFFFFF) | 0x3FF00000, __double2loint(v));
  const int i = min(max((int)(log2f((float)m) * kUnits), 0), kUnits - 1);
  *out = log2_fixed(e, m, i, tab[i]);
  return true;
}

// 2^((x + add) / kUnits), add in fixed point; false where x is out of range or
// the result is not a normal number.
__device__ __forceinline__ bool exp2_fixed(double x, long long add, const double* tab, double* out) {
  const int hi = __double2hiint(x), e = (hi >> 20) & 0x7FF;
  // |x| = M 2^(e - 1075); x 2^kFrac = (M << 10) >> (1044 - e), |x| < 2^21
  unsigned long long M = ((unsigned long long)((hi & 0xFFFFF) | 0x100000) << 32) | (unsigned)__double2loint(x);
  const int sh = min(1044 - e, 63);
  long long F = (long long)((M << 10) >> (sh & 63));
  if (hi < 0) F = -F;
  F += add;
  const int n = (int)(F >> kFrac);
  const unsigned long long g = __umul64hi((unsigned long long)F << (64 - kFrac), 0xB17217F7D1CF79ABull);   // ln 2
  // 2^f - 1 in units 2^-76: g + g^2 / 2 + g^3 / 6
  const unsigned u = (unsigned)(g >> 32);
  const unsigned long long u2 = (unsigned long long)u * u;
  const unsigned u3 = __umulhi((unsigned)(u2 >> 32), u);
  const unsigned long long p = (g + (u2 >> 13) + (((unsigned long long)u3 * 43691u) >> 10) + (1u << 23)) >> 24;
  const int E = n >> 12;
  const double b = __hiloint2double((int)(((unsigned)(0x3FF + E) << 20) + (unsigned)(p >> 32)), (int)(unsigned)p);
  *out = tab[n & (kUnits - 1)] * b;
  return e <= 1023 + 20 && (unsigned)(E + 1020) <= 2040u;
}

__global__ void __launch_bounds__(32 * kRatesWarps)
rates_kernel(int n_r, int64_t C, int chunk, const RatePar* __restrict__ par, const RateFix* __restrict__ fix,
             const double* __restrict__ table, const double* __restrict__ T, const double* __restrict__ nH,
             const double* __restrict__ Av, const double* __restrict__ chi, double zeta, double* __restrict__ k,
             int64_t ld) {
  __shared__ double tab[kUnits];
  for (int i = threadIdx.x; i < kUnits; i += blockDim.x) tab[i] = table[i];
  __syncthreads();
  const int64_t c = (int64_t)blockIdx.x * 32 + (threadIdx.x & 31);
  if (c >= C) return;
  const int j0 = (blockIdx.y * kRatesWarps + (threadIdx.x >> 5)) * chunk;
  const int j1 = min(n_r, j0 + chunk);
  if (j0 >= j1) return;
  const double t = T[c], n = nH[c], av = Av[c];
  const double fuv = chi ? chi[c] : 1.0;   // FUV field on the photorates
  const double lt = log(t * (1.0 / 300.0));
  const double it = 1.0 / t;
  constexpr double K = kUnits * kLog2e;
  const double ltu = lt * K, itu = -K / t, avu = -K * av;
  long long ln = 0, lc = 0;
  const bool okn = isfinite(ltu) && isfinite(itu) && cell_fixed(n, tab, &ln);
  const bool okc = isfinite(avu) && (!chi || cell_fixed(fuv, tab, &lc));
  double* out = k + (int64_t)j0 * ld + c;
  for (int j = j0; j < j1; ++j, out += ld) {
    const RateFix f = fix[j];
    double v;
    bool ok = false;
    if (f.kind == RateFix::TWO_BODY) {
      const double x = f.gamma != 0.0 ? fma(f.gamma, itu, f.beta * ltu) : f.beta != 0.0 ? f.beta * ltu : 0.0;
      ok = exp2_fixed(x, f.la + ln, tab, &v) && okn;
    } else if (f.kind == RateFix::PHOTO) {
      ok = exp2_fixed(f.gamma != 0.0 ? f.gamma * avu : 0.0, f.la + lc, tab, &v) && okc;
    }
    if (!ok) {   // cosmic rays, and whatever the fixed-point form does not cover
      const RatePar p = par[j];  // (log alpha | alpha, beta, gamma, class)
      const int cls = (int)p.w;
      if (cls == SM_TWO_BODY || cls == SM_DISS_RECOMB) v = exp(fma(p.y, lt, p.x) - p.z * it) * n;
      else if (cls == SM_COSMIC_RAY) v = p.x * zeta;
      else v = fuv * p.x * exp(-p.z * av);
    }
    *out = v;
  }
}

}  // namespace

std::vector<double> rate_table() {
  std::vector<double> t(kUnits);
  for (int i = 0; i < kUnits; ++i) t[i] = std::exp2(i / (double)kUnits);
  return t;
}

std::vector<RateFix> rate_fixed(const sm_net* net, const std::vector<double>& table) {
  std::vector<RateFix> v(net->n_r);
  for (int32_t j = 0; j < net->n_r; ++j) {
    RateFix& f = v[j];
    f.beta = net->beta[j];
    f.gamma = net->gamma[j];
    const int c = net->cls[j];
    int e = 0;
    const double a = net->alpha[j], m = 2.0 * std::frexp(a, &e);   // a = m 2^(e - 1)
    const bool pos = a > 0.0 && std::isfinite(a) && std::abs(e) < kMaxLog;
    f.kind = !pos || c == SM_COSMIC_RAY                  ? RateFix::OTHER
             : c == SM_TWO_BODY || c == SM_DISS_RECOMB ? RateFix::TWO_BODY
                                                         : RateFix::PHOTO;
    if (f.kind == RateFix::OTHER) continue;
    const int i = std::min(std::max((int)(std::log2(m) * kUnits), 0), kUnits - 1);
    f.la = log2_fixed(e - 1, m, i, table[i]);
  }
  return v;
}

sm_status launch_rates(const sm_net* net, int64_t C, const double* T, const double* nH,
                       const double* Av, const double* chi, double zeta, double* k, int64_t ld, cudaStream_t s) {
  if (C == 0) return SM_OK;
  const int64_t groups = (C + 31) / 32;
  // two rounds of 32 warps per SM; a warp's cell set-up costs about as much as
  // 20 coefficients
  const int chunk = (int)std::min<int64_t>(512, std::max<int64_t>(16, groups * net->n_r / (2 * 32 * kSms)));
  dim3 grid((unsigned)groups, (unsigned)((net->n_r + chunk * kRatesWarps - 1) / (chunk * kRatesWarps)));
  rates_kernel<<<grid, 32 * kRatesWarps, 0, s>>>(net->n_r, C, chunk, net->d_rate.as<RatePar>(),
                                                 net->d_ratefix.as<RateFix>(), net->d_ratetab.as<double>(), T, nH, Av,
                                                 chi, zeta, k, ld);
  SM_TRY_CUDA(cudaGetLastError());
  return SM_OK;
}
