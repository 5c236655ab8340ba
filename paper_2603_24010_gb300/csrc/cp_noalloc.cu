// cp_noalloc.cu -- an allocation-free variant of the ion push.
//
// Some callers cannot call cudaMalloc: a simulation step embedded in a
// real-time control loop or a host process that must not grow device
// memory after start-up, or code that runs while another component owns the
// allocator.  For them cp_push_ions_noalloc pushes one FP32 ion population
// through one step (gather, kick, drift, absorption, ion-induced secondary
// emission, deposit) using only buffers the caller passes in.  What the
// context path keeps in memory of its own stays in those too: the impacts of
// a CTA are listed in its shared memory, their velocities in the ions' u
// until their electrons are drawn, and the tallies are the caller's counts.
// So calls share nothing: each waits for its own stream alone.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>

#include "cp_common.cuh"

namespace cpk_na {

using cpk::floor_split;
using cpk::frac16;
using cpk::kTagSee;
using cpk::philox4x64_10;
using cpk::u01;
using cpk::U64x4;

constexpr int kThreads = 1024;
constexpr int kMaxCells = 4096;          // shared-memory grid limit
constexpr int64_t kMaxIons = 1 << 19;    // ions of one call
constexpr int kMostCta = 8191;           // ions of one CTA (13-bit places in its list of impacts)
constexpr int kAhead = 4;                // ions per thread requested together

// The caller's six counts while the kernel runs: the first four as they are
// returned, then the electrons asked for so far and the CTAs that are done.
enum { kAbs0 = 0, kAbs1 = 1, kEmit0 = 2, kEmit1 = 3, kSeCount = 4, kDone = 5, kCounts = 6 };

struct Params {
  int N;
  float kap;         // kick factor (half or full) in cells/step^2 per V/m
  double dx, dt, m_i, e, m_e;
  double see_scale, gamma_coef, gamma_max, E_ref_eV, see_vth;
  uint64_t seed;
  int64_t step;
};

__device__ __forceinline__ unsigned lane() { return threadIdx.x & 31u; }

// v units of charge on node k of the caller's grid (end nodes doubled)
__device__ __forceinline__ void add_node(long long* G, int N, int k, long long v) {
  if (v == 0) return;
  if (k == 0 || k == N) v <<= 1;
  atomicAdd(reinterpret_cast<unsigned long long*>(&G[k]), static_cast<unsigned long long>(v));
}

// The grid and the counts start at zero.
__global__ void __launch_bounds__(256) k_clear(long long* __restrict__ G, int nodes, unsigned long long* __restrict__ counts) {
  const int k = blockIdx.x * 256 + threadIdx.x;
  if (k < nodes) G[k] = 0;
  if (k < kCounts) counts[k] = 0ULL;
}

// The whole call in one kernel (and a clear), one CTA per SM at most: each CTA
// pushes a contiguous range of the ions (gather, kick, drift, absorption,
// deposit into 32-bit node sums), then turns the ions it saw absorbed into
// electrons (the context path's arithmetic and draws), and the last CTA out
// completes the counts.
//
// Bound: latency (a call moves 12 MB at most): the ions are requested before
// the field table is formed, and one table per SM is formed at all because the
// conversion from FP64 runs at two values a cycle.  Call at 524288 ions and 4096
// cells: 52.9 -> 39.6 us, with the host's wait for the counts (three kernels,
// two memsets and 64-bit shared atomics before; 39.0 with a list of impacts in
// memory that all calls share and take turns for).
// counts: [0] absorbed at x = 0, [1] at x = d, [2] emitted at x = 0, [3] at x =
// d, [4] electrons written (at most se_cap), [5] convection count at x = 0.
__global__ void __launch_bounds__(kThreads, 1)
k_push_ions(Params p, const double* __restrict__ E, float* __restrict__ xi, float* __restrict__ u,
            const uint32_t* __restrict__ id, int64_t n, long long* __restrict__ G, float* __restrict__ se_xi,
            float* __restrict__ se_u, int64_t se_cap, unsigned long long* __restrict__ counts) {
  extern __shared__ unsigned int smem_na[];
  __shared__ unsigned int s_abs_n, s_abs[2], s_emit[2], s_round[2];
  const int N = p.N, tid = static_cast<int>(threadIdx.x);
  unsigned int* nd = smem_na;                                 // the ions' node sums (at most 2^13 ions a CTA)
  unsigned int* ne = nd + (N + 1);                            // a round's electrons'
  float* tab = reinterpret_cast<float*>(ne + (N + 1));        // E_{k-1/2}, ends repeated
  const int64_t lo = n * blockIdx.x / gridDim.x, hi = n * (blockIdx.x + 1) / gridDim.x;
  uint16_t* hit = reinterpret_cast<uint16_t*>(tab + (N + 2));  // this CTA's impacts: place from lo on | electrode << 13
  float x[kAhead], v[kAhead];
  auto fetch = [&](int64_t k0) {
#pragma unroll
    for (int c = 0; c < kAhead; ++c) {
      const int64_t k = k0 + tid + c * kThreads;
      x[c] = (k < hi) ? xi[k] : -1.0f;
      v[c] = (k < hi) ? u[k] : 0.0f;
    }
  };
  fetch(lo);
  for (int k = tid; k <= N + 1; k += kThreads) {
    tab[k] = static_cast<float>(E[k == 0 ? 0 : (k <= N ? k - 1 : N - 1)]);
    if (k <= N) nd[k] = ne[k] = 0u;
  }
  if (tid == 0) {
    s_abs_n = 0u;
    s_abs[0] = s_abs[1] = s_emit[0] = s_emit[1] = 0u;
  }
  __syncthreads();
  const float Nr = static_cast<float>(N);
  for (int64_t k0 = lo; k0 < hi; k0 += kAhead * kThreads) {
    if (k0 > lo) fetch(k0);
#pragma unroll
    for (int c = 0; c < kAhead; ++c) {
      if (!(x[c] > 0.f && x[c] < Nr)) continue;
      const int64_t k = k0 + tid + c * kThreads;
      float t;
      const int j = floor_split(x[c] - 0.5f, &t);
      const float e0 = tab[j + 1];
      const float un = fmaf(p.kap, fmaf(t, tab[j + 2] - e0, e0), v[c]);
      const float xn = x[c] + un;
      if (!(xn > 0.f && xn < Nr)) {
        const int el = (xn <= 0.f) ? 0 : 1;
        atomicAdd(&s_abs[el], 1u);
        hit[atomicAdd(&s_abs_n, 1u)] = static_cast<uint16_t>(static_cast<int>(k - lo) | el << 13);  // every ion fits
        xi[k] = -1.f;
        u[k] = un;  // until its electrons are drawn
      } else {
        xi[k] = xn;
        u[k] = un;
        float f;
        const int i = floor_split(xn, &f);
        const unsigned int w1 = frac16(f);
        atomicAdd(&nd[i], 65536u - w1);
        atomicAdd(&nd[i + 1], w1);
      }
    }
  }
  __syncthreads();
  for (int k = tid; k <= N; k += kThreads) add_node(G, N, k, nd[k]);
  // secondary emission, an impact per thread and round; a round's electrons
  // (at most 1024 x 15, below 2^32 in a node sum) go through node sums of
  // their own where they are many
  const int na = static_cast<int>(s_abs_n);
  const double pi = 3.14159265358979323846;
  for (int r0 = 0; r0 < na; r0 += kThreads) {
    const bool act = r0 + tid < na;
    int nse = 0;
    uint32_t ion = 0;
    int el = 0;
    unsigned int* const electrons = &s_round[r0 / kThreads & 1];
    if (tid == 0) *electrons = 0u;
    __syncthreads();
    if (act) {
      const int h = hit[r0 + tid];
      const int64_t k = lo + (h & 0x1FFF);
      el = h >> 13;
      ion = id[k];
      const double vi = __ddiv_rn(__dmul_rn(static_cast<double>(u[k]), p.dx), p.dt);
      u[k] = 0.f;
      const double Eev = __ddiv_rn(__dmul_rn(__dmul_rn(__dmul_rn(0.5, p.m_i), vi), vi), p.e);
      double g = __dmul_rn(__dmul_rn(p.see_scale, p.gamma_coef), __dsqrt_rn(__ddiv_rn(Eev, p.E_ref_eV)));
      if (g > p.gamma_max) g = p.gamma_max;
      if (!(g > 0.0)) g = 0.0;
      const U64x4 w = philox4x64_10(ion, static_cast<uint64_t>(p.step), 0, 0, p.seed, kTagSee);
      const double fl = floor(g);
      nse = static_cast<int>(fl) + ((u01(w.w[0]) < __dsub_rn(g, fl)) ? 1 : 0);
      if (nse) atomicAdd(&s_emit[el], static_cast<unsigned int>(nse));
    }
    const int incl = cpk::warp_incl_scan(nse);
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    unsigned long long base = 0;
    if (lane() == 31 && total) {
      base = atomicAdd(&counts[kSeCount], static_cast<unsigned long long>(total));
      atomicAdd(electrons, static_cast<unsigned int>(total));
    }
    __syncthreads();
    const bool few = *electrons <= 64u;
    base = __shfl_sync(0xffffffffu, base, 31);
    for (int j = 0; j < nse; ++j) {
      const U64x4 wv = philox4x64_10(ion, static_cast<uint64_t>(p.step), static_cast<uint64_t>(1 + j), 0, p.seed, kTagSee);
      const double ua = u01(wv.w[0]), ub = u01(wv.w[1]), frac = u01(wv.w[2]);
      const double z = sqrt(-2.0 * log(ua)) * cos(2.0 * pi * ub);
      const double use = p.see_vth * fabs(z) * p.dt / p.dx;
      const double xd = (el == 0) ? __dmul_rn(use, frac) : __dsub_rn(static_cast<double>(N), __dmul_rn(use, frac));
      const float xr = cpk::nudge_inside<float>(xd, N);
      const unsigned long long slot = base + static_cast<unsigned long long>(incl - nse + j);
      if (slot < static_cast<unsigned long long>(se_cap)) {
        se_xi[slot] = xr;
        se_u[slot] = static_cast<float>(el == 0 ? use : -use);
        float f;
        const int i = floor_split(xr, &f);
        const unsigned int w1 = frac16(f);
        if (few) {
          add_node(G, N, i, static_cast<long long>(w1) - 65536);
          add_node(G, N, i + 1, -static_cast<long long>(w1));
        } else {
          atomicAdd(&ne[i], 65536u - w1);
          atomicAdd(&ne[i + 1], w1);
        }
      }
    }
    if (few) continue;
    __syncthreads();
    for (int k = tid; k <= N; k += kThreads) {
      add_node(G, N, k, -static_cast<long long>(ne[k]));
      ne[k] = 0u;
    }
  }
  __syncthreads();
  if (tid == 0) {
    if (s_abs[0]) atomicAdd(&counts[kAbs0], static_cast<unsigned long long>(s_abs[0]));
    if (s_abs[1]) atomicAdd(&counts[kAbs1], static_cast<unsigned long long>(s_abs[1]));
    if (s_emit[0]) atomicAdd(&counts[kEmit0], static_cast<unsigned long long>(s_emit[0]));
    if (s_emit[1]) atomicAdd(&counts[kEmit1], static_cast<unsigned long long>(s_emit[1]));
    __threadfence();
    if (atomicAdd(&counts[kDone], 1ULL) == gridDim.x - 1) {
      __threadfence();
      const unsigned long long se = __ldcg(&counts[kSeCount]), cap = static_cast<unsigned long long>(se_cap);
      counts[4] = se < cap ? se : cap;
      counts[5] = __ldcg(&counts[kAbs0]) + __ldcg(&counts[kEmit0]);
    }
  }
}

constexpr size_t push_smem(int N) { return 12 * static_cast<size_t>(N + 2) + sizeof(uint16_t) * (kMostCta + 1); }

// The push kernel's shared-memory limit, set once per device.
std::mutex g_mu;
bool g_ready[64] = {};

int configure(int dev) {
  if (dev < 0 || dev >= 64) return CP_ERR_ARG;
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_ready[dev]) {
    if (cudaFuncSetAttribute(k_push_ions, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(push_smem(kMaxCells))) != cudaSuccess) {
      cudaGetLastError();
      return CP_ERR_CUDA;
    }
    g_ready[dev] = true;
  }
  return CP_OK;
}

}  // namespace cpk_na

extern "C" int cp_push_ions_noalloc(const cp_gap* gap, const cp_see_beam* see, double dt, uint64_t seed,
                                    int64_t step, int32_t half_kick, const double* E, float* xi,
                                    float* u, const uint32_t* id, int64_t n, int64_t* G, float* se_xi,
                                    float* se_u, int64_t se_cap, int64_t* counts, void* stream) {
  using namespace cpk_na;
  if (!gap || !see || !E || !G || !counts || n < 0 || (n > 0 && (!xi || !u || !id)) || se_cap < 0 ||
      (se_cap > 0 && (!se_xi || !se_u)) || !(dt > 0) || !(gap->d > 0) || !(gap->m_i > 0) ||
      !(gap->e > 0) || !(gap->m_e > 0) || step < 0)
    return CP_ERR_ARG;
  // the SEE law as cp_create accepts it: a bounded mean yield keeps the
  // per-impact draw loop and the warp scan of counts small, and a finite,
  // non-negative emission temperature keeps the emitted positions finite
  if (!(see->gamma_max >= 0.0 && see->gamma_max <= 14.0) || !(see->scale >= 0.0) ||
      !std::isfinite(see->scale) || !(see->gamma_coef >= 0.0) || !std::isfinite(see->gamma_coef) ||
      !(see->T_emit_eV >= 0.0) || !std::isfinite(see->T_emit_eV) || !(see->E_ref_eV >= 0.0) ||
      !std::isfinite(see->E_ref_eV) || see->count_law != CP_SEE_COUNT_BERNOULLI ||
      see->energy_law != CP_SEE_ENERGY_MAXWELL)
    return CP_ERR_ARG;
  if (gap->n_cells < 2 || gap->n_cells > kMaxCells) return CP_ERR_ARG;  // shared-memory grid limit
  if (n > kMaxIons) return CP_ERR_CAPACITY;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return CP_ERR_CUDA;
  const int rc = configure(dev);
  if (rc != CP_OK) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int N = gap->n_cells;
  Params p;
  p.N = N;
  p.dx = gap->d / N;
  p.dt = dt;
  p.m_i = gap->m_i;
  p.e = gap->e;
  p.m_e = gap->m_e;
  const double kappa = gap->e * dt * dt / (gap->m_i * p.dx);
  p.kap = static_cast<float>(half_kick ? 0.5 * kappa : kappa);
  p.see_scale = see->scale;
  p.gamma_coef = see->gamma_coef;
  p.gamma_max = see->gamma_max;
  p.E_ref_eV = see->E_ref_eV > 0 ? see->E_ref_eV : 1000.0;
  p.see_vth = std::sqrt(gap->e * see->T_emit_eV / gap->m_e);
  p.seed = seed;
  p.step = step;
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return CP_ERR_CUDA;
  // at least 512 ions a CTA (each forms the field table and flushes a grid),
  // at most 8191 (its 32-bit node sums stay below 2^29)
  const int64_t want = std::max<int64_t>((n + 511) / 512, 1);
  const int grid = static_cast<int>(std::max<int64_t>(std::min<int64_t>(want, sms), (n + kMostCta - 1) / kMostCta));
  long long* Gl = reinterpret_cast<long long*>(G);
  unsigned long long* tally = reinterpret_cast<unsigned long long*>(counts);
  k_clear<<<(N + 256) / 256, 256, 0, st>>>(Gl, N + 1, tally);
  k_push_ions<<<grid, kThreads, push_smem(N), st>>>(p, E, xi, u, id, n, Gl, se_xi, se_u, se_cap, tally);
  if (cudaGetLastError() != cudaSuccess) return CP_ERR_CUDA;
  // the counts back for the status: the electrons asked for may exceed se_cap
  int64_t c[kCounts];
  if (cudaMemcpyAsync(c, counts, sizeof(c), cudaMemcpyDefault, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return CP_ERR_CUDA;
  return c[kEmit0] + c[kEmit1] > se_cap ? CP_ERR_CAPACITY : CP_OK;
}
