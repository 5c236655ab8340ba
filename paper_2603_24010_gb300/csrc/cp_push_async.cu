// cp_push_async.cu -- the particle push of a single gap, with per-thread
// asynchronous copies.
//
// One time step (arXiv 2603.24010) is two launches, this push and the cluster
// solve of cp_solve.cu.  k_push streams every particle once: CIC gather of
// E^n from a shared-memory table (App. C), leapfrog kick and drift (Sec.
// 2.2.2), absorption at the electrodes (Sec. 2.4.1), the CIC deposit of
// rho^{n+1} in fixed point (2^16 units per macroparticle charge, boundary
// nodes doubled as in App. E.2), secondary emission from the absorbed ions
// (Sec. 2.3, Algorithm see_sampling_1d; Philox4x64-10 draws keyed by (seed,
// step, ion id)) and the step's beam ions.
//
// What bounds it: at 1e7 particles and more the HBM stream and the shared-
// memory pipe (two table reads and two node-sum atomics per particle at
// random cells); below that a fixed latency, which is why everything the
// previous solve does not write is done before the wait for it:
//
// * every thread owns a ring of shared-memory slots (x and u of its four
//   particles of a tile) filled by cp.async copies, so the next tiles are on
//   their way while one is processed, without registers held for them and
//   without block-wide waits.  The first tiles are requested before the wait
//   (the solve changes no particle but the up to three padding slots behind
//   a species' last one, and the last vector is read directly; a push behind
//   anything else than a solve starts when that has completed, push_launch);
// * the beam ions are drawn before the wait (their draws need the level
//   alone, which the previous push left in B.next_step);
// * one flat list of tiles over the three species, so that small species
//   share the CTAs;
// * one signed 32-bit sum per node for both signs of charge, folded into an
//   int64 sum only when 31 tiles' worth may be in it (fewer: never);
// * the tail's FP64 chains (emission counts, and the first electron's draws)
//   run in half of the warps while the others add the CTA's grid into the
//   global one; an impact's further electrons are spread over the lanes.
//   The chains start from shared memory (records and parameters), divide by
//   reciprocals, fetch the electrons' slots beside a barrier, and few
//   electrons go straight to the global grid (the tail of a CTA with impacts
//   took 6-8 us; step at 3e5 particles 19.4 -> 18.3 us, at 3e7 with impacts
//   in every CTA 102.1 -> 98.3).
// * after the wait one warp of a CTA reads what the solve left (level, flags,
//   slots in use): read by every warp of 304 CTAs, those few lines took longer
//   than the field table (1 us of a step at 3e5 particles).
//
// FP64 particles: an SM issues 2 FP64 operations a cycle, so comparisons,
// floors and conversions are done on the integer pipe (8 FP64 operations a
// particle instead of 15), and a tile is 1024 particles, so that small
// populations reach every SM.
//
// Graph-timed step before -> after (GB300): FP64, 256 cells, 1.4e5 particles
// 38.6 -> 18.3 us; FP64 Tesla gap 40.9 -> 21.8; FP32, 4096 cells, 3.3e5
// particles 22.9 -> 16.3, 1e6 (1531 cells) 17.5 -> 14.8, 1.5e7 59.3 -> 46.6,
// 3.1e7 (impacts every step) 118 -> 98.3.

#include <cstddef>

#include "cp_common.cuh"
#include "cp_mlp.cuh"
#include "cp_push.cuh"

namespace cpk {

// A thread's ring: three slots of one 16-byte vector of x and one of u (four
// FP32 or two FP64 particles), at [stage][x | u][thread].
constexpr int kStages = 3;
constexpr size_t kRingBytes = static_cast<size_t>(kStages) * kThreads * 32;
template <typename real>
struct Vec {
  static constexpr int kN = 16 / sizeof(real);     // particles per thread and tile
  static constexpr int kTileN = kThreads * kN;     // particles per tile
};

constexpr int kTailRound = kThreads / 4;  // absorbed-ion records per round of the push's tail
// the tail keeps the emitted electrons' node sums (N + 1 <= 11390 words) and
// the first electrons' draws (2 kTailRound doubles) in the ring
static_assert(4 * 11392 + 16 * kTailRound <= kRingBytes, "tail scratch lives in the ring");
static_assert(kThreads == 4 * kTailRound && kTailRound % 32 == 0, "tail roles are whole warps");
static_assert(sizeof(PredScratch) <= kRingBytes, "predictor scratch lives in the ring");
static_assert(kThreads >= kHid * 8, "the network takes 8 lanes per neuron");

// Node sums hold the sum of +w (ions) and -w (electrons) modulo 2^32.  A tile
// adds at most 2^27 to a node, so after `pos` ion and `neg` electron tiles
// the sum lies in [-neg 2^27, pos 2^27], which 32 bits tell apart while pos +
// neg <= 31.
__device__ __forceinline__ long long node_value(unsigned int v, int neg) {
  const unsigned int off = static_cast<unsigned int>(neg) << 27;
  return static_cast<long long>(v + off) - static_cast<long long>(off);
}

// fold the node sums into the int64 grid and clear them (the first fold of a
// launch writes the grid)
__device__ __forceinline__ void fold_nodes(unsigned int* nd, long long* Gs, int N, int neg, bool first) {
  for (int k = threadIdx.x; k <= N; k += kThreads) {
    const long long a = node_value(nd[k], neg);
    nd[k] = 0u;
    Gs[k] = first ? a : Gs[k] + a;
  }
}

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


template <typename real>
static size_t push_smem(int N) {
  return kRingBytes + align16(sizeof(long long) * (N + 1)) + align16(sizeof(unsigned int) * (N + 1)) +
         align16(sizeof(real) * (N + 2));
}

// What the tail needs of the parameters, in shared memory (the first touch of
// a global parameter costs an L2 round trip on the tail's chain), with the
// reciprocals of its divisors.
struct SeeConst {
  double see_scale, gamma_coef, gamma_max, E_ref_eV, see_vth, see_ln_mu, see_ln_sigma, e, m_e, m_i, dx, dt;
  double r_E_ref, r_e, r_dx, r_dt;
  uint64_t seed;
  int32_t see_count_law, see_energy_law;
};

__device__ __forceinline__ double over_E_ref(const SeeConst* c, double E) { return div_by(E, c->E_ref_eV, c->r_E_ref); }

constexpr unsigned int kFewElectrons = 32;  // emitted by a CTA straight into the global grid
constexpr int kRecShared = 28;  // absorbed-ion records kept in shared memory (the others in global)

// Static shared memory of a push: a multiple of 128 bytes, since the dynamic
// part follows it and the ring wants whole aligned sectors (behind 944 bytes,
// which split every 32-byte sector of the copies in two, the step at 3e7
// particles took 110 us instead of 97).
template <typename real>
struct alignas(128) PushShared {
  int abs_n, over;
  unsigned int cnt[2][kSpecies];
  unsigned int emit[2];
  long long conv, energy;
  unsigned int cfl;
  real* xi[kSpecies];
  real* u[kSpecies];
  long long n[kSpecies];     // slots in use
  int tile[kSpecies + 1];    // first tile of each species in the flat list
  int64_t step;
  int stop, half, moved;
  SeeConst see;
  AbsRec rec[kRecShared];
};

// The push of one CTA.  PUSH: the step's push; else the deposit of the loaded
// particles (level 0).  The list and the level are read before the wait, where
// a CTA that starts late (other kernels on the device held its place) may find
// them already moved on by CTAs of this very push that have finished.  What
// the solve left is compared after the wait: on a difference nothing has been
// done, the result is false, and the CTA begins again with LATE, from what
// the solve left.
template <typename real, bool PUSH, bool LATE>
__device__ __forceinline__ bool push_cta(const Bufs& B, PushShared<real>& sh, unsigned char* smem, int G) {
  using V = Vec<real>;
  const DevParams* __restrict__ P = B.P;
  DevState* S = B.S;
  int &s_abs_n = sh.abs_n, &s_over = sh.over;
  auto& s_cnt = sh.cnt;
  auto& s_emit = sh.emit;
  long long &s_conv = sh.conv, &s_energy = sh.energy;
  unsigned int& s_cfl = sh.cfl;
  auto& s_xi = sh.xi;
  auto& s_u = sh.u;
  auto& s_n = sh.n;
  auto& s_tile = sh.tile;
  SeeConst& C = sh.see;
  auto& s_rec = sh.rec;

  if (LATE) __syncthreads();  // the first attempt's readings are done
  const int tid = static_cast<int>(threadIdx.x);
  const int N = P->N;
  long long* Gs = reinterpret_cast<long long*>(smem + kRingBytes);
  unsigned int* nd = reinterpret_cast<unsigned int*>(smem + kRingBytes + align16(sizeof(long long) * (N + 1)));
  real* Et = reinterpret_cast<real*>(reinterpret_cast<unsigned char*>(nd) + align16(sizeof(unsigned int) * (N + 1)));
  const int cta = static_cast<int>(blockIdx.x);
  // --- before the previous solve has finished --------------------------------
  for (int k = tid; k <= N; k += kThreads) nd[k] = 0u;
  if (tid == 0) {
    s_abs_n = 0;
    s_over = 0;
    s_conv = 0;
    s_energy = 0;
    s_cfl = 0u;
    s_emit[0] = s_emit[1] = 0u;
  }
  if (tid < 2 * kSpecies) s_cnt[tid / kSpecies][tid % kSpecies] = 0u;
  if (tid < 32) {  // the flat tile list
    long long n = 0;
    if (tid < kSpecies) {
      s_xi[tid] = static_cast<real*>(ldcg(&S->xi[tid]));
      s_u[tid] = static_cast<real*>(ldcg(&S->u[tid]));
      // the solve rounds n_alloc up to a multiple of 4, this reads it before or after
      n = LATE ? static_cast<long long>(ldcg(&S->n_proc[tid]))
               : min(static_cast<long long>((ldcg(&S->n_alloc[tid]) + 3) & ~int64_t(3)), static_cast<long long>(P->cap[tid]));
      s_n[tid] = n;
    }
    int t = static_cast<int>((n + V::kTileN - 1) / V::kTileN);
    t = warp_incl_scan(t);
    if (tid < kSpecies) s_tile[tid + 1] = t;
    if (tid == 0) s_tile[0] = 0;
    if (tid == kSpecies) sh.step = LATE ? ldcg(&S->level) : ldcg(B.next_step);
  }
  if (PUSH && tid == kThreads - 32) {
    C.see_scale = P->see_scale; C.gamma_coef = P->gamma_coef; C.gamma_max = P->gamma_max;
    C.E_ref_eV = P->E_ref_eV; C.see_vth = P->see_vth; C.see_ln_mu = P->see_ln_mu; C.see_ln_sigma = P->see_ln_sigma;
    C.e = P->e; C.m_e = P->m_e; C.m_i = P->m_i; C.dx = P->dx; C.dt = P->dt;
    C.r_E_ref = 1.0 / P->E_ref_eV; C.r_e = 1.0 / P->e; C.r_dx = 1.0 / P->dx; C.r_dt = 1.0 / P->dt;
    C.seed = P->seed;
    C.see_count_law = P->see_count_law; C.see_energy_law = P->see_energy_law;
  }
  uint32_t* const ids = static_cast<uint32_t*>(ldcg(reinterpret_cast<void* const*>(&S->id)));
  const uint32_t id_base = S->beam_id_base;
  // this CTA's share [kb0, kb1) of the step's beam ions, one per thread of
  // the first round
  const int Bn = PUSH ? P->beam_per_step : 0;
  const int nbc = (Bn + G - 1) / G;
  const int kb0 = min(Bn, cta * nbc), kb1 = min(Bn, kb0 + nbc);
  __syncthreads();
  const int64_t step = sh.step;  // the level this push starts from (one thread's reading for the whole CTA)
  auto draw_beam = [&](int kk, real* x, real* u) {
    const U64x4 wv = philox4x64_10(static_cast<uint64_t>(kk), static_cast<uint64_t>(step), 0, 0, P->seed, kTagBeam);
    const double frac = u01(wv.w[0]);
    const double ub = beam_speed<real>(P, u01(wv.w[1]));
    *x = nudge_inside<real>(__dsub_rn(static_cast<double>(N), __dmul_rn(ub, frac)), N);
    *u = static_cast<real>(-ub);
  };
  // This CTA's tiles cta, cta + G, ... of the flat list, species by species:
  // `left` tiles of species `s`, the next at x, u (this thread's particles);
  // the species' last four, at x_end, are not copied.
  struct Cursor {
    real *x, *u, *x_end;
    int s, left;
  };
  auto enter = [&](Cursor& c) {  // the next species in which this CTA has tiles, from c.s on
    for (; c.s < kSpecies; ++c.s) {
      const int t0 = s_tile[c.s], t1 = s_tile[c.s + 1];
      const int first = cta + ((max(t0 - cta, 0) + G - 1) / G) * G;  // this CTA's first tile at or behind t0
      c.left = (first < t1) ? (t1 - first + G - 1) / G : 0;
      if (c.left > 0) {
        const long long b = static_cast<long long>(first - t0) * V::kTileN + tid * V::kN;
        c.x = s_xi[c.s] + b;
        c.u = s_u[c.s] + b;
        c.x_end = s_xi[c.s] + s_n[c.s] - 4;
        return;
      }
    }
  };
  const long long stride = static_cast<long long>(G) * V::kTileN;
  float4* slots = reinterpret_cast<float4*>(smem) + tid;
  Cursor nxt;  // the next tile to request
  nxt.s = 0;
  nxt.left = 0;
  enter(nxt);
  const bool any = nxt.left > 0;  // this CTA has tiles
  int st_next = 0;
  auto issue = [&]() {
    if (nxt.left > 0) {
      if (nxt.x < nxt.x_end) {
        float4* d = slots + st_next * (2 * kThreads);
        cp_async16(d, nxt.x);
        if (PUSH) cp_async16(d + kThreads, nxt.u);
      }
      nxt.x += stride;
      nxt.u += stride;
      if (--nxt.left == 0) {
        ++nxt.s;
        enter(nxt);
      }
    }
    cp_async_commit();
    st_next = (st_next == kStages - 1) ? 0 : st_next + 1;
  };
#pragma unroll
  for (int j = 0; j < kStages - 1; ++j) issue();
  // this thread's beam ion of the first round
  real bx = real(0), bu = real(0);
  if (kb0 + tid < kb1) draw_beam(kb0 + tid, &bx, &bu);

  if (!LATE) {
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
  }
  // what the solve left, by one warp of the CTA (read by all, the line serves
  // thousands of warps at once)
  if (tid < 32) {
    static_assert(offsetof(DevState, pushed) == offsetof(DevState, level) + 8 &&
                      offsetof(DevState, status) == offsetof(DevState, level) + 12,
                  "level | pushed, status");
    long long w = 0;  // lane 0: level, 1: pushed and status, 2-4: slots in use
    if (tid < 2) w = ldcg(reinterpret_cast<const long long*>(&S->level) + tid);
    else if (tid < 2 + kSpecies) w = ldcg(&S->n_proc[tid - 2]);
    const bool differs = !LATE && ((tid == 0 && w != step) || (tid >= 2 && tid < 2 + kSpecies && w != s_n[tid - 2]));
    const unsigned int moved = __ballot_sync(0xffffffffu, differs);
    if (tid == 1) {
      sh.half = (static_cast<int>(w) == 0);
      sh.stop = static_cast<int>(w >> 32);
      sh.moved = (moved != 0u);
    }
  }
  if (PUSH && any) load_table<real, kThreads>(Et, B.Etab, N);  // of the solve just finished
  __syncthreads();
  if (sh.stop || sh.moved) {
    cp_async_wait<0>();
    return sh.stop != 0;
  }
  const bool half = sh.half;
  // the beam: slots behind the ions in use (ions are appended by the beam
  // alone, so the slots are known without a shared counter)
  bool folded = false;
  int pos = 0, neg = 0;  // tiles' worth of each sign in the node sums
  for (int k0 = kb0, round = 0; k0 < kb1; k0 += kThreads, ++round) {
    if (round % V::kN == 0 && ++pos > kFlushTiles) {  // (beams of millions a step)
      __syncthreads();
      fold_nodes(nd, Gs, N, 0, !folded);
      __syncthreads();
      folded = true;
      pos = 1;
    }
    const int kk = k0 + tid;
    if (kk >= kb1) continue;
    if (round > 0) draw_beam(kk, &bx, &bu);
    const long long slot = s_n[CP_IONS] + kk;
    if (slot < P->cap[CP_IONS]) {
      s_xi[CP_IONS][slot] = bx;
      s_u[CP_IONS][slot] = bu;
      ids[slot] = id_base + static_cast<uint32_t>(step * Bn + kk);
      deposit_nodes(nd, fix_pos(bx), 1);
    } else {
      s_over = 1;
    }
  }

  const real Nr = static_cast<real>(N);
  const int cap = P->abs_cap;
  AbsRec* my_abs = B.abs + static_cast<size_t>(cta) * cap;
  typename Bits<real>::type cfl = 0;
  int st = 0;  // ring slot of this thread's tile
  Cursor cur;
  cur.s = 0;
  cur.left = 0;
  for (enter(cur); cur.s < kSpecies; ++cur.s, enter(cur)) {
    const int sign = (cur.s == CP_IONS) ? 1 : -1;
    const real kap = kick<real>(P, half, cur.s);
    for (; cur.left > 0; --cur.left, cur.x += stride, cur.u += stride, st = (st == kStages - 1) ? 0 : st + 1) {
      issue();
      if (pos + neg == kFlushTiles) {  // bounds every node sum to 32 bits
        __syncthreads();
        fold_nodes(nd, Gs, N, neg, !folded);
        __syncthreads();
        folded = true;
        pos = neg = 0;
      }
      if (sign > 0) ++pos; else ++neg;
      cp_async_wait<kStages - 1>();  // this thread's copies of the tile have landed
      real xv[V::kN], uv[V::kN];
      if (cur.x < cur.x_end) {
        const float4* d = slots + st * (2 * kThreads);
        get_vec(d, xv);
        if (PUSH) get_vec(d + kThreads, uv);
      } else if (cur.x < cur.x_end + 4) {  // the species' last four: the padding among them was set after the copies began
#pragma unroll
        for (int q = 0; q < V::kN; ++q) {
          xv[q] = __ldcg(cur.x + q);
          uv[q] = __ldcg(cur.u + q);
        }
      } else {
        continue;  // the last tile's tail lanes hold no particles
      }
      if (PUSH) {
#pragma unroll
        for (int q = 0; q < V::kN; ++q) {
          bool dep = false;
          if (inside(xv[q], Nr)) {  // live (dead slots hold -1)
            const real E = gather_tab(Et, xv[q]);
            const real un = fma(kap, E, uv[q]);
            const real xn = xv[q] + un;
            max_abs(cfl, un);
            if (!inside(xn, Nr)) {  // absorbed (a non-finite value counts at x = d)
              const int el = (xn <= real(0)) ? 0 : 1;
              atomicAdd(&s_cnt[el][cur.s], 1u);
              if (sign > 0) {
                const int slot_i = atomicAdd(&s_abs_n, 1);
                if (slot_i < cap) {
                  AbsRec r;
                  r.id = ids[cur.x + q - s_xi[CP_IONS]];
                  r.electrode = static_cast<uint32_t>(el);
                  r.u = static_cast<double>(un);
                  if (slot_i < kRecShared) s_rec[slot_i] = r;
                  else my_abs[slot_i] = r;
                }
              }
              xv[q] = real(-1);
              uv[q] = real(0);
            } else {
              dep = true;
              xv[q] = xn;
              uv[q] = un;
            }
          }
          if (dep) deposit_nodes(nd, fix_pos(xv[q]), sign);
        }
        put_vec(cur.x, xv);
        put_vec(cur.u, uv);
      } else {
#pragma unroll
        for (int q = 0; q < V::kN; ++q)
          if (inside(xv[q], Nr)) deposit_nodes(nd, fix_pos(xv[q]), sign);
      }
    }
  }
  cp_async_wait<0>();
  const unsigned int cflf = warp_max_u(float_bits(cfl));
  if (lane_id() == 0 && cflf) atomicMax(&s_cfl, cflf);
  __syncthreads();

  // --- the CTA's grid into the global one; secondary emission ------------------
  // With impacts, per round of kTailRound records: the emission counts
  // (threads [0, kTailRound)), the first emitted electron's draws of each
  // record (threads [kTailRound, 2 kTailRound)), and, beside the first round's
  // chains, the grid (the other half of the CTA).
  const int na = PUSH ? min(s_abs_n, cap) : 0;
  if (PUSH && tid == 0 && s_abs_n > cap) s_over = 1;
  auto flush = [&](int first, int threads) {
    for (int k = first; k <= N; k += threads)
      add_global(B.G, k, N, node_value(nd[k], neg) + (folded ? Gs[k] : 0LL));
  };
  if (na == 0) {
    flush(tid, kThreads);
  } else {
    unsigned int* ndb = reinterpret_cast<unsigned int*>(smem);  // the emitted electrons' node sums
    double* s_v0 = reinterpret_cast<double*>(smem + align16(sizeof(unsigned int) * (N + 1)));
    double* s_f0 = s_v0 + kTailRound;
    const int rounds = (na + kTailRound - 1) / kTailRound;
    const bool counter = tid < kTailRound, drawer = !counter && tid < 2 * kTailRound;  // warp-uniform roles
    for (int rd = 0; rd < rounds; ++rd) {
      const int t = tid % kTailRound;
      const int r = rd * kTailRound + t;
      const bool act = counter && r < na;
      int nse = 0, incl = 0;
      unsigned long long wbase = 0ULL;
      AbsRec rec;
      rec.id = 0; rec.electrode = 0; rec.u = 0.0;
      if (tid < 2 * kTailRound && r < na) rec = (r < kRecShared) ? s_rec[r] : my_abs[r];
      if (tid >= kThreads / 2) {
        for (int k = tid - kThreads / 2; k <= N; k += kThreads / 2) ndb[k] = 0u;
        if (rd == 0) flush(tid - kThreads / 2, kThreads / 2);
      }
      if (drawer && r < na) {  // the first electron's speed and fraction of the step
        double f0;
        s_v0[t] = see_speed(&C, rec.id, step, 0, &f0);
        s_f0[t] = f0;
      }
      if (counter) {
        if (act) {
          const double v = div_by(__dmul_rn(rec.u, C.dx), C.dt, C.r_dt);
          const double Eev = div_by(__dmul_rn(__dmul_rn(__dmul_rn(0.5, C.m_i), v), v), C.e, C.r_e);
          nse = see_count(&C, Eev, rec.id, step);
          if (rec.electrode == 0) {
            atomicAdd(reinterpret_cast<unsigned long long*>(&s_energy),
                      static_cast<unsigned long long>(__double2ll_rn(Eev * 256.0)));
            atomicAdd(reinterpret_cast<unsigned long long*>(&s_conv),
                      static_cast<unsigned long long>(static_cast<long long>(nse)));
          }
          if (nse) atomicAdd(&s_emit[rec.electrode], static_cast<unsigned int>(nse));
        }
        incl = warp_incl_scan(nse);
        if (lane_id() == 31 && incl > 0)  // the warp's slots, on their way beside the barrier
          wbase = atomicAdd(reinterpret_cast<unsigned long long*>(&S->n_alloc[CP_SECONDARIES]),
                            static_cast<unsigned long long>(incl));
      }
      __syncthreads();  // the first electrons' draws are in shared memory, ndb is clear
      // a few electrons go straight into the global grid, more through node
      // sums of the CTA's own
      const bool few = rounds == 1 && s_emit[0] + s_emit[1] <= kFewElectrons;
      if (counter) {
        // electron j of the impact (id, el): its place and speed, then its slot
        auto emit = [&](uint32_t el, int place, bool go, double vse, double frac) {
          real xr = real(0), ur = real(0);
          if (go) {
            const double use = div_by(vse * C.dt, C.dx, C.r_dx);
            const double xd = (el == 0) ? __dmul_rn(use, frac) : __dsub_rn(static_cast<double>(N), __dmul_rn(use, frac));
            xr = nudge_inside<real>(xd, N);
            ur = static_cast<real>(el == 0 ? use : -use);
          }
          const unsigned long long slot = __shfl_sync(0xffffffffu, wbase, 31) + static_cast<unsigned long long>(place);
          if (!go) return;
          if (slot >= static_cast<unsigned long long>(P->cap[CP_SECONDARIES])) {
            s_over = 1;
            return;
          }
          s_xi[CP_SECONDARIES][slot] = xr;
          s_u[CP_SECONDARIES][slot] = ur;
          const unsigned int F = fix_pos(xr);
          if (few) {
            const long long w1 = F & 0xFFFFu;
            add_global(B.G, F >> 16, N, w1 - 65536);
            add_global(B.G, (F >> 16) + 1, N, -w1);
          } else {
            deposit_nodes(ndb, F, 1);
          }
        };
        if (__any_sync(0xffffffffu, nse > 0)) emit(rec.electrode, incl - nse, nse > 0, s_v0[t], s_f0[t]);
        // the impacts' further electrons, one per lane and pass (a chain of
        // FP64 functions each)
        const int more = max(nse - 1, 0);
        const int inclm = warp_incl_scan(more);
        const int totm = __shfl_sync(0xffffffffu, inclm, 31);
        for (int e0 = 0; e0 < totm; e0 += 32) {
          const int e = e0 + static_cast<int>(lane_id());
          int src = 0;  // first lane whose inclusive count exceeds e
#pragma unroll
          for (int o = 16; o > 0; o >>= 1)
            if (__shfl_sync(0xffffffffu, inclm, src + o - 1) <= e) src += o;
          src = min(src, 31);
          const uint32_t id = __shfl_sync(0xffffffffu, rec.id, src);
          const uint32_t el = __shfl_sync(0xffffffffu, rec.electrode, src);
          const int j = 1 + e - __shfl_sync(0xffffffffu, inclm - more, src);
          const int first = __shfl_sync(0xffffffffu, incl - nse, src);
          double frac = 0.0, vse = 0.0;
          if (e < totm) vse = see_speed(&C, id, step, j, &frac);
          emit(el, first + j, e < totm, vse, frac);
        }
      }
      if (few) break;
      __syncthreads();  // at most kTailRound x 64 electrons per round: below 2^32
      for (int k = tid; k <= N; k += kThreads) add_global(B.G, k, N, -static_cast<long long>(ndb[k]));
      if (rd + 1 < rounds) __syncthreads();
    }
    __syncthreads();
  }
  if (tid == 0 && PUSH) {
    for (int e = 0; e < 2; ++e)
      for (int s = 0; s < kSpecies; ++s)
        if (s_cnt[e][s]) atomicAdd(&S->absorbed[e][s], static_cast<unsigned long long>(s_cnt[e][s]));
    if (s_emit[0]) atomicAdd(&S->emitted[0], static_cast<unsigned long long>(s_emit[0]));
    if (s_emit[1]) atomicAdd(&S->emitted[1], static_cast<unsigned long long>(s_emit[1]));
    const long long conv = static_cast<long long>(s_cnt[0][CP_IONS]) -
                           static_cast<long long>(s_cnt[0][CP_ELECTRONS]) -
                           static_cast<long long>(s_cnt[0][CP_SECONDARIES]) + s_conv;
    if (conv) atomicAdd(reinterpret_cast<unsigned long long*>(&S->conv_count),
                        static_cast<unsigned long long>(conv));
    if (s_energy) atomicAdd(reinterpret_cast<unsigned long long*>(&S->ion_energy_q),
                            static_cast<unsigned long long>(s_energy));
    if (s_cfl) atomicMax(&S->max_cfl_bits, s_cfl);
    if (cta == 0) {
      if (Bn > 0) {
        atomicAdd(&S->injected, static_cast<unsigned long long>(Bn));
        atomicAdd(reinterpret_cast<unsigned long long*>(&S->n_alloc[CP_IONS]), static_cast<unsigned long long>(Bn));
      }
      *B.next_step = step + 1;
    }
    if (s_over) atomicCAS(&S->status, 0, CP_ERR_CAPACITY);
  }
  return true;
}

template <typename real, bool PUSH>
__device__ __noinline__ void push_cta_late(const Bufs& B, PushShared<real>& sh, unsigned char* smem, int G) {
  push_cta<real, PUSH, true>(B, sh, smem, G);
}

template <typename real, bool PUSH>
__global__ void __launch_bounds__(kThreads, kCtasPerSm) k_push(const __grid_constant__ Bufs B) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ PushShared<real> sh;
  // With a network installed the launch has one CTA more, which runs the
  // learned predictor for the level the previous solve committed (levels
  // >= 1).  Scheduled last, it takes the first slot a pushing CTA frees, so
  // the network runs beside the other CTAs' ends.
  const bool pred_cta = (B.net != nullptr && B.net_in_push);
  const int G = static_cast<int>(gridDim.x) - (pred_cta ? 1 : 0);  // pushing CTAs
  if (static_cast<int>(blockIdx.x) == G) {
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
    if (ldcg(&B.S->status) != 0) return;
    if (PUSH && ldcg(&B.S->level) >= 1) predictor_in_push(B.S, B.net, B.P->C, reinterpret_cast<PredScratch*>(smem));
    return;
  }
  if (!push_cta<real, PUSH, false>(B, sh, smem, G)) push_cta_late<real, PUSH>(B, sh, smem, G);
}

// ---------------------------------------------------------------------------
// Host-side launchers (internal C++ interface used by cp_api.cu)
// ---------------------------------------------------------------------------
static const void* push_fn(int precision, int do_push) {
  if (precision == CP_FP32)
    return do_push ? reinterpret_cast<const void*>(k_push<float, true>)
                   : reinterpret_cast<const void*>(k_push<float, false>);
  return do_push ? reinterpret_cast<const void*>(k_push<double, true>)
                 : reinterpret_cast<const void*>(k_push<double, false>);
}

size_t push_smem_bytes(int N, int precision) {
  return precision == CP_FP32 ? push_smem<float>(N) : push_smem<double>(N);
}

// Shared memory by which cp_create accepts a gap (the documented limits of
// 11,390 cells with FP32 and 7,231 with FP64 particles): the FP64 push
// itself takes less.
size_t push_smem_limit_bytes(int N, int precision) {
  if (precision == CP_FP32) return push_smem<float>(N);
  return align16(sizeof(long long) * (N + 1)) + align16(sizeof(unsigned int) * 2 * N) + 2 * sizeof(double) * (N + 1);
}

// Every context sharing a kernel may ask for another size, so the kernels'
// limit is the largest the device allows.
cudaError_t push_configure(int precision) {
  int dev = 0, most = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  for (int do_push = 0; do_push < 2 && e == cudaSuccess; ++do_push) {
    cudaFuncAttributes at;
    e = cudaFuncGetAttributes(&at, push_fn(precision, do_push));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(push_fn(precision, do_push), cudaFuncAttributeMaxDynamicSharedMemorySize,
                               most - static_cast<int>(at.sharedSizeBytes));
  }
  return e;
}

cudaError_t push_occupancy(int precision, size_t smem, int* blocks_per_sm) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, push_fn(precision, 1), kThreads, smem);
}

// Push and solve are launched with programmatic dependent launch: each may
// be scheduled while its predecessor finishes and waits in
// cudaGridDependencySynchronize() until that grid has completed.  A push reads
// particles, store pointers and slot counts ahead of that wait, which is sound
// behind a solve alone: the solve let it start only after its own wait for the
// push that wrote them.  behind_solve = false (behind a removal, a graph or
// nothing) leaves the attribute out, and the push starts when everything
// before it has completed.
cudaError_t push_launch(int precision, const Bufs& B, int grid, size_t smem, cudaStream_t st, int do_push,
                        bool behind_solve) {
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
  cfg.numAttrs = behind_solve ? 1 : 0;
  void* args[] = {const_cast<Bufs*>(&B)};
  return cudaLaunchKernelExC(&cfg, push_fn(precision, do_push), args);
}

}  // namespace cpk
