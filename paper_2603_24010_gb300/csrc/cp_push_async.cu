// cp_push_async.cu -- the FP32 particle push with per-thread asynchronous
// copies.
//
// Same step as k_push (gather, kick, drift, absorption, SEE, beam, fixed-
// point deposit; Sec. 2.2.2, 2.3, 2.4.1, App. C, App. E.2), with the HBM
// stream kept deeper in flight: every thread owns a ring of three 32-byte
// slots in shared memory (x and u of its four particles of a tile) filled by
// cp.async copies, so two tiles are always on their way while the third is
// processed, without holding registers for them and without block-wide
// synchronisation (each thread waits only for its own copy groups).  To make
// room for the ring at two CTAs per SM, the field table keeps only the
// half-grid values, padded by a copy of each end value (the slope is
// recomputed from neighbours exactly as the solve forms it, and is zero past
// either end), and the deposit uses one 32-bit sum per node.

#include "cp_common.cuh"
#include "cp_mlp.cuh"

namespace cpk {

constexpr int kAStages = 3;  // slots per thread: two tiles in flight, one processed

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// 16-byte global -> shared copy, cached in L2 only
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// fold the node sums into the int64 grid (end nodes doubled) and clear them
__device__ __forceinline__ void fold_nodes(unsigned int* nd, long long* Gs, int N, long long sign) {
  for (int k = threadIdx.x; k <= N; k += kThreads) {
    long long a = nd[k];
    if (a) {
      nd[k] = 0u;
      if (k == 0 || k == N) a <<= 1;
      Gs[k] += sign * a;
    }
  }
}

// CIC deposit of one particle into the node sums: node i gets 2^16 - W1,
// node i+1 W1, with i = floor(x) and W1 = floor(2^16 (x - i)).  x 2^16 is
// exact (power-of-two scaling) and below 2^32 (the N + 1 node sums and the
// field table take 8 B per cell of shared memory, so N < 2^16), so one
// truncating conversion gives i in its high and W1 in its low 16 bits.
__device__ __forceinline__ void deposit_nodes(unsigned int* nd, float x) {
  const unsigned int F = __float2uint_rz(x * 65536.0f);
  const unsigned int i = F >> 16;
  const unsigned int w1 = F & 0xFFFFu;
  atomicAdd(&nd[i], 65536u - w1);
  atomicAdd(&nd[i + 1], w1);
}

// gather from the padded field table Et[k] = E_{k-1/2} (k = 1..N), Et[0] =
// E_{1/2}, Et[N+1] = E_{N-1/2}: the pair (E_{j+1/2}, slope) of the pair table
// is formed here with the same FP32 subtraction, and the repeated end values
// give the constant extension (slope +0) for j = -1 and j = N-1
__device__ __forceinline__ float gather_tab(const float* Et, float x) {
  const float s = x - 0.5f;
  const float jf = floorf(s);
  const int j = static_cast<int>(jf);
  const float t = s - jf;
  const float e0 = Et[j + 1];
  return fmaf(t, Et[j + 2] - e0, e0);
}

constexpr size_t kRingBytes = static_cast<size_t>(kAStages) * kThreads * 32;
constexpr int kTailRound = kThreads / 4;  // absorbed-ion records per round of the push's tail
// the tail keeps the beam's node sums (N + 1 <= 11390 words) and the first
// electrons' draws (2 kTailRound doubles) in the ring
static_assert(4 * 11392 + 16 * kTailRound <= kRingBytes, "tail scratch lives in the ring");
static_assert(2 * kTailRound <= kThreads && kTailRound % 32 == 0, "tail roles are whole warps");
static_assert(sizeof(PredScratch) <= kRingBytes, "predictor scratch lives in the ring");
static_assert(kThreads >= kHid * 8, "the network takes 8 lanes per neuron");

// The learned weak-coupling predictor for the level the previous solve
// committed (its row from that level's diagnostics), run by the push's extra
// CTA (all its threads), with the network read from global memory (L2).
// Its J_hat is for the level this push starts.
__device__ __noinline__ void predictor_in_push(DevState* S, const PredNet* net, double C,
                                               PredScratch* sp) {
  __shared__ PredLevel L;
  const int pos0 = ldcg(&S->feat_pos);
  double v_old = 0.0;
  if (threadIdx.x < kPredIn - kPredFeat)
    v_old = ldcg(&S->feat[(pos0 + 1 + static_cast<int>(threadIdx.x) / kPredFeat) & (kPredWindow - 1)]
                        [threadIdx.x % kPredFeat]);
  if (threadIdx.x == 0) {
    L.Qconv = ldcg(&S->cur.Q_conv);
    L.phi0 = ldcg(&S->cur.V_gap);
    L.phi0_prev = ldcg(&S->pv_phi0);
    L.Qsurf = ldcg(&S->cur.Q_surf);
    L.Qsurf_prev = ldcg(&S->pv_Qsurf);
    L.Qn = ldcg(&S->cur.Q_circ);
    L.Q1 = ldcg(&S->Qh[1]);
    L.emitted = static_cast<double>(ldcg(&S->cur.emitted[0]));
    L.ion_eV = ldcg(&S->cur.ion_energy_eV);
    L.had_pred = ldcg(&S->pred_ready);
    L.J_pred = ldcg(&S->J_pred);
    L.err_avg = ldcg(&S->err_avg);
    L.J_avg = ldcg(&S->J_avg);
    L.n_eval = ldcg(&S->n_eval);
    L.pos = pos0;
    L.n_feat = ldcg(&S->n_feat);
  }
  __syncthreads();
  pred_level<kThreads>(net, C, S, &L, v_old, sp);
}

size_t push_async_smem_bytes(int N) {
  return kRingBytes + align16(sizeof(long long) * (N + 1)) + align16(sizeof(unsigned int) * (N + 1)) +
         align16(sizeof(float) * (N + 2));
}

__global__ void __launch_bounds__(kThreads, kCtasPerSm) k_push_async(Bufs B, int do_push) {
  const DevParams* __restrict__ P = B.P;
  DevState* S = B.S;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_abs_n;
  __shared__ int s_flag[2];  // [0] stopped, [1] overflow
  __shared__ unsigned long long s_cnt[2][kSpecies];
  __shared__ unsigned long long s_emit[2];
  __shared__ long long s_conv, s_energy;
  __shared__ unsigned int s_cfl;

  // Set-up that needs nothing of the previous kernel runs before the wait for
  // it: the parameters are written once, and the shared grid sums are this
  // CTA's own.
  const int N = P->N;
  float4* ring = reinterpret_cast<float4*>(smem);  // [stage][x | u][thread]
  long long* Gs = reinterpret_cast<long long*>(smem + kRingBytes);
  unsigned int* nd = reinterpret_cast<unsigned int*>(smem + kRingBytes + align16(sizeof(long long) * (N + 1)));
  float* Et = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(nd) + align16(sizeof(unsigned int) * (N + 1)));
  for (int k = threadIdx.x; k <= N; k += kThreads) {
    Gs[k] = 0;
    nd[k] = 0u;
  }
  if (threadIdx.x == 0) {
    s_flag[1] = 0;
    s_abs_n = 0;
    s_conv = 0;
    s_energy = 0;
    s_cfl = 0u;
    s_emit[0] = s_emit[1] = 0ULL;
  }
  if (threadIdx.x < 2 * kSpecies) s_cnt[threadIdx.x / kSpecies][threadIdx.x % kSpecies] = 0ULL;

  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  if (threadIdx.x == 0) s_flag[0] = (ldcg(&S->status) != 0);
  // the field table of the solve just finished: eight loads per thread in
  // flight together (one L2 round trip for N <= 4095)
  const float2* Epair = reinterpret_cast<const float2*>(B.Epair);
  for (int k0 = threadIdx.x; k0 <= N; k0 += 8 * kThreads) {
    float e[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int k = k0 + q * kThreads;
      e[q] = (k <= N) ? Epair[k].x : 0.0f;  // pair 0 repeats E_{1/2}
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int k = k0 + q * kThreads;
      if (k <= N) {
        Et[k] = e[q];
        if (k == N) Et[N + 1] = e[q];
      }
    }
  }
  __syncthreads();
  if (s_flag[0]) return;
  const int64_t step = S->level;
  // With a network installed the launch has one CTA more, which runs the
  // learned predictor for the level the previous solve committed (levels
  // >= 1).  Scheduled last, it takes the first slot a pushing CTA frees, so
  // the network runs beside the other CTAs' ends.
  const bool pred_cta = (B.net != nullptr && B.net_in_push);
  const unsigned int G = gridDim.x - (pred_cta ? 1u : 0u);  // pushing CTAs
  if (blockIdx.x == G) {
    if (do_push && step >= 1) predictor_in_push(S, B.net, P->C, reinterpret_cast<PredScratch*>(smem));
    return;
  }

  const bool half = (S->pushed == 0);
  const float Nr = static_cast<float>(N);
  const int cap = P->abs_cap;
  AbsRec* my_abs = B.abs + static_cast<size_t>(blockIdx.x) * cap;
  unsigned int cfl = 0u;
  float4* my_slot = ring + threadIdx.x;  // x at + stage * 2 kThreads, u kThreads further

  for (int s = 0; s < kSpecies; ++s) {
    float* __restrict__ xs = reinterpret_cast<float*>(S->xi[s]);
    float* __restrict__ us = reinterpret_cast<float*>(S->u[s]);
    const int64_t n = S->n_proc[s];  // multiple of 4
    if (n == 0) continue;  // the same for every thread of the CTA
    const int64_t ntiles = (n + kTile - 1) / kTile;
    const int mine = (ntiles > blockIdx.x) ? static_cast<int>((ntiles - blockIdx.x + G - 1) / G) : 0;
    const long long sign = (s == CP_IONS) ? 1LL : -1LL;
    const float kap = P->kap_f[half ? 0 : 1][s];
    const uint32_t* ids = S->id;
    unsigned int a0 = 0u, a1 = 0u;
    int since = 0;
    const int64_t stride = static_cast<int64_t>(G) * kTile;
    const int64_t base0 = static_cast<int64_t>(blockIdx.x) * kTile + static_cast<int64_t>(threadIdx.x) * kPerThread;
    int64_t b_next = base0;  // first particle of this thread's next tile to fetch
    int st_next = 0;         // its ring slot
    auto issue = [&](bool go) {  // this thread's four particles of its next tile
      float4* slot = my_slot + st_next * (kThreads * 2);
      if (go && b_next < n) {
        cp_async16(slot, xs + b_next);
        if (do_push) cp_async16(slot + kThreads, us + b_next);
      }
      cp_async_commit();
      b_next += stride;
      st_next = (st_next == kAStages - 1) ? 0 : st_next + 1;
    };
    issue(0 < mine);
    issue(1 < mine);
    int64_t base = base0;  // first particle of this thread's tile j
    int st = 0;            // its ring slot
    for (int j = 0; j < mine; ++j, base += stride, st = (st == kAStages - 1) ? 0 : st + 1) {
      issue(j + 2 < mine);
      cp_async_wait<2>();  // this thread's copies of tile j have landed
      const bool valid = base < n;  // the last tile's tail lanes hold no particles
      const float4* slot = my_slot + st * (kThreads * 2);
      if (do_push && valid) {
        const float4 xa = slot[0];
        const float4 ua = slot[kThreads];
        float xv[4] = {xa.x, xa.y, xa.z, xa.w};
        float uv[4] = {ua.x, ua.y, ua.z, ua.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          bool dep = false;
          if (xv[q] > 0.0f && xv[q] < Nr) {  // live (dead slots hold -1)
            const float E = gather_tab(Et, xv[q]);
            const float un = fmaf(kap, E, uv[q]);
            const float xn = xv[q] + un;
            cfl = max(cfl, __float_as_uint(fabsf(un)));
            if (!(xn > 0.0f && xn < Nr)) {  // absorbed (a non-finite value counts at x = d)
              const int el = (xn <= 0.0f) ? 0 : 1;
              if (el) ++a1; else ++a0;
              if (s == CP_IONS) {
                const int slot_i = atomicAdd(&s_abs_n, 1);
                if (slot_i < cap) {
                  AbsRec r;
                  r.id = ids[base + q];
                  r.electrode = static_cast<uint32_t>(el);
                  r.u = static_cast<double>(un);
                  my_abs[slot_i] = r;
                }
              }
              xv[q] = -1.0f;
              uv[q] = 0.0f;
            } else {
              dep = true;
              xv[q] = xn;
              uv[q] = un;
            }
          }
          if (dep) deposit_nodes(nd, xv[q]);
        }
        store4(xs + base, xv);
        store4(us + base, uv);
      } else if (!do_push && valid) {
        const float4 xa = slot[0];
        const float xv[4] = {xa.x, xa.y, xa.z, xa.w};
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (xv[q] > 0.0f && xv[q] < Nr) deposit_nodes(nd, xv[q]);
      }
      if (++since == kFlushTiles) {  // bounds every 32-bit node sum below 2^32
        __syncthreads();
        fold_nodes(nd, Gs, N, sign);
        __syncthreads();
        since = 0;
      }
    }
    cp_async_wait<0>();
    __syncthreads();
    fold_nodes(nd, Gs, N, sign);
    __syncthreads();
    a0 = warp_sum_u(a0);
    a1 = warp_sum_u(a1);
    if (lane_id() == 0) {
      if (a0) atomicAdd(&s_cnt[0][s], static_cast<unsigned long long>(a0));
      if (a1) atomicAdd(&s_cnt[1][s], static_cast<unsigned long long>(a1));
    }
  }
  cfl = warp_max_u(cfl);
  if (lane_id() == 0 && cfl) atomicMax(&s_cfl, cfl);
  // This CTA's share [kb0, kb1) of the step's beam ions.  They carry the
  // other sign than emitted electrons, so they deposit into node sums of
  // their own, in the ring (idle now: every copy was waited for).
  const int Bn = do_push ? P->beam_per_step : 0;
  const int nbc = (Bn + static_cast<int>(G) - 1) / static_cast<int>(G);
  const int kb0 = min(Bn, static_cast<int>(blockIdx.x) * nbc);
  const int kb1 = min(Bn, kb0 + nbc);
  unsigned int* ndb = reinterpret_cast<unsigned int*>(smem);
  double* s_v0 = reinterpret_cast<double*>(smem + align16(sizeof(unsigned int) * (N + 1)));
  double* s_f0 = s_v0 + kTailRound;
  if (kb1 > kb0)
    for (int k = threadIdx.x; k <= N; k += kThreads) ndb[k] = 0u;
  __syncthreads();
  if (do_push) {
    // --- secondary emission from the ions this CTA saw absorbed, and the beam.
    // Per round of kTailRound records, three FP64 chains run in different
    // warps: the SE counts (threads [0, kTailRound), from the bottom), the
    // beam ions (the same threads, from the top) and the first emitted
    // electron's draws of each record (threads [kTailRound, 2 kTailRound)).
    const int n_abs = s_abs_n;
    if (n_abs > cap && threadIdx.x == 0) s_flag[1] = 1;
    const int na = min(n_abs, cap);
    const int nb = kb1 - kb0;
    const double dx = P->dx, dt = P->dt;
    const int rounds = max((na + kTailRound - 1) / kTailRound, (nb + kTailRound - 1) / kTailRound);
    const int64_t ion_base = S->n_proc[CP_IONS];  // == n_alloc at the push's start
    const bool counter = threadIdx.x < kTailRound;  // warp-uniform roles
    const bool drawer = !counter && threadIdx.x < 2 * kTailRound;
    for (int rd = 0; rd < rounds; ++rd) {
      const int t = static_cast<int>(threadIdx.x) % kTailRound;
      const int r = rd * kTailRound + t;
      if (drawer && r < na) {  // the first electron's speed and fraction of the step
        double f0;
        s_v0[t] = see_speed(P, my_abs[r].id, step, 0, &f0);
        s_f0[t] = f0;
      }
      const bool act = counter && r < na;
      int nse = 0;
      AbsRec rec;
      rec.id = 0; rec.electrode = 0; rec.u = 0.0;
      if (act) {
        rec = my_abs[r];
        const double v = __ddiv_rn(__dmul_rn(rec.u, dx), dt);
        const double Eev = __ddiv_rn(__dmul_rn(__dmul_rn(__dmul_rn(0.5, P->m_i), v), v), P->e);
        nse = see_count(P, Eev, rec.id, step);
        if (rec.electrode == 0) {
          atomicAdd(reinterpret_cast<unsigned long long*>(&s_energy),
                    static_cast<unsigned long long>(__double2ll_rn(Eev * 256.0)));
          atomicAdd(reinterpret_cast<unsigned long long*>(&s_conv),
                    static_cast<unsigned long long>(static_cast<long long>(nse)));
        }
        if (nse) atomicAdd(&s_emit[rec.electrode], static_cast<unsigned long long>(nse));
      }
      // beam ion kk: entry position N - |u_b| frac, speed -|u_b|, in slot
      // n_proc + kk (ions are appended by the beam alone, so the slots are
      // known without a shared counter; n_alloc grows by Bn at the end)
      const int kk = kb0 + rd * kTailRound + (kTailRound - 1 - t);
      if (counter) {
        if (kk < kb1) {
          const U64x4 wv = philox4x64_10(static_cast<uint64_t>(kk), static_cast<uint64_t>(step), 0,
                                         0, P->seed, kTagBeam);
          const double frac = u01(wv.w[0]);
          const double ub = beam_speed_fp32(P, u01(wv.w[1]));
          const float xr = nudge_inside<float>(__dsub_rn(static_cast<double>(N), __dmul_rn(ub, frac)), N);
          const unsigned long long slot = static_cast<unsigned long long>(ion_base + kk);
          if (slot < static_cast<unsigned long long>(P->cap[CP_IONS])) {
            reinterpret_cast<float*>(S->xi[CP_IONS])[slot] = xr;
            reinterpret_cast<float*>(S->u[CP_IONS])[slot] = static_cast<float>(-ub);
            S->id[slot] = S->beam_id_base + static_cast<uint32_t>(step * Bn + kk);
            deposit_nodes(ndb, xr);
          } else {
            s_flag[1] = 1;
          }
        }
      }
      __syncthreads();  // the first electrons' draws are in shared memory
      if (counter) {
        const int incl = warp_incl_scan(nse);
        const int tot = __shfl_sync(0xffffffffu, incl, 31);
        unsigned long long wbase = 0ULL;
        if (lane_id() == 31 && tot > 0)
          wbase = atomicAdd(reinterpret_cast<unsigned long long*>(&S->n_alloc[CP_SECONDARIES]),
                            static_cast<unsigned long long>(tot));
        wbase = __shfl_sync(0xffffffffu, wbase, 31);
        if (act && nse > 0) {
          float* xs = reinterpret_cast<float*>(S->xi[CP_SECONDARIES]);
          float* us = reinterpret_cast<float*>(S->u[CP_SECONDARIES]);
          for (int j = 0; j < nse; ++j) {
            double frac, vse;
            if (j == 0) {
              vse = s_v0[t];
              frac = s_f0[t];
            } else {
              vse = see_speed(P, rec.id, step, j, &frac);
            }
            const double use = vse * dt / dx;
            const double xd = (rec.electrode == 0) ? __dmul_rn(use, frac) : __dsub_rn(static_cast<double>(N), __dmul_rn(use, frac));
            const float xr = nudge_inside<float>(xd, N);
            const float ur = static_cast<float>(rec.electrode == 0 ? use : -use);
            const unsigned long long slot = wbase + static_cast<unsigned long long>(incl - nse + j);
            if (slot < static_cast<unsigned long long>(P->cap[CP_SECONDARIES])) {
              xs[slot] = xr;
              us[slot] = ur;
              deposit_nodes(nd, xr);
            } else {
              s_flag[1] = 1;
            }
          }
        }
      }
      // per round at most kTailRound x 64 electrons and kTailRound beam ions
      // per node sum: below 2^32 with a fold between rounds
      __syncthreads();
      if (rd + 1 < rounds) {
        if (na > 0) fold_nodes(nd, Gs, N, -1LL);
        if (nb > 0) fold_nodes(ndb, Gs, N, 1LL);
        __syncthreads();
      }
    }
    if (na > 0) fold_nodes(nd, Gs, N, -1LL);
    if (nb > 0) fold_nodes(ndb, Gs, N, 1LL);
  }
  __syncthreads();

  // --- add this CTA's grid and tallies into the global ones ------------------
  for (int kq = threadIdx.x; kq <= N; kq += kThreads) {
    const long long g = Gs[kq];
    if (g != 0)
      atomicAdd(reinterpret_cast<unsigned long long*>(&B.G[kq]), static_cast<unsigned long long>(g));
  }
  if (threadIdx.x == 0 && do_push) {
    for (int e = 0; e < 2; ++e)
      for (int s = 0; s < kSpecies; ++s)
        if (s_cnt[e][s]) atomicAdd(&S->absorbed[e][s], s_cnt[e][s]);
    if (s_emit[0]) atomicAdd(&S->emitted[0], s_emit[0]);
    if (s_emit[1]) atomicAdd(&S->emitted[1], s_emit[1]);
    const long long conv = static_cast<long long>(s_cnt[0][CP_IONS]) -
                           static_cast<long long>(s_cnt[0][CP_ELECTRONS]) -
                           static_cast<long long>(s_cnt[0][CP_SECONDARIES]) + s_conv;
    if (conv) atomicAdd(reinterpret_cast<unsigned long long*>(&S->conv_count),
                        static_cast<unsigned long long>(conv));
    if (s_energy) atomicAdd(reinterpret_cast<unsigned long long*>(&S->ion_energy_q),
                            static_cast<unsigned long long>(s_energy));
    if (s_cfl) atomicMax(&S->max_cfl_bits, s_cfl);
    if (blockIdx.x == 0 && P->beam_per_step > 0) {
      atomicAdd(&S->injected, static_cast<unsigned long long>(P->beam_per_step));
      atomicAdd(reinterpret_cast<unsigned long long*>(&S->n_alloc[CP_IONS]),
                static_cast<unsigned long long>(P->beam_per_step));
    }
    if (s_flag[1]) atomicCAS(&S->status, 0, CP_ERR_CAPACITY);
  }
}

cudaError_t push_async_configure(size_t smem) {
  return cudaFuncSetAttribute(k_push_async, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(smem));
}

cudaError_t push_async_occupancy(size_t smem, int* blocks_per_sm) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_push_async, kThreads, smem);
}

cudaError_t push_async_launch(const Bufs& B, int grid, size_t smem, cudaStream_t st, int do_push) {
  cudaLaunchConfig_t cfg = {};
  // one CTA more runs the learned predictor when the push carries it
  cfg.gridDim = dim3(grid + ((B.net != nullptr && B.net_in_push) ? 1 : 0), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_push_async, B, do_push);
}

}  // namespace cpk
