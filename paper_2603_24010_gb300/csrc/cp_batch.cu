// cp_batch.cu -- the ensemble path: many independent gap instances advanced
// by one persistent launch per stage.
//
// k_push_ens: the particle tiles of every (instance, species) pair form one
//   flat work list (instance-major, then species, then tile); each CTA takes
//   one contiguous share of it, so it meets only a few instances and loads
//   each instance's gather table and flushes each instance's deposit grid
//   once per step.  Per tile the arithmetic is that of the single-instance
//   push (cp_push.cuh: same gather, kick, drift, absorption test and
//   fixed-point deposit), so an instance advanced in the ensemble follows
//   exactly the trajectory it follows alone.  Secondary emission and the beam
//   are handled after the tiles: emitted electrons and beam ions are deposited
//   with int64 global atomics straight into their instance's grid.
// k_compact_ens / k_swap_ens: removal of absorbed particles over the same
//   flat list, then one thread per instance swaps the buffers.
// The solve of every instance (a cluster of 1, 2 or 4 CTAs) is
// k_solve_ens in cp_solve.cu.
#include <algorithm>

#include "cp_common.cuh"
#include "cp_push.cuh"

namespace cpk {

// Absorbed ion of the ensemble push: instance and electrode packed.
struct AbsRecE {
  uint32_t id;
  uint32_t inst_el;  // instance * 2 + electrode
  double u;
};

constexpr int kEnsMaxEntries = 3 * 2048;  // (instance, species) pairs: at most 2048 instances

// The fixed-point CIC deposit of one particle, added straight into an int64
// global grid.
template <typename real>
__device__ __forceinline__ void deposit_global(long long* G, int N, real x, int sign) {
  const unsigned int F = fix_pos(x);
  const long long w1 = F & 0xFFFFu;
  add_global(G, F >> 16, N, sign * (65536LL - w1));
  add_global(G, (F >> 16) + 1, N, sign * w1);
}

// Exclusive prefix of the tile counts of every (instance, species) pair into
// off[0..n] (off[n] = total).  STOPPED: with the entries of stopped instances
// (else 0): every CTA of a push must see the same list, also one that starts
// after another has stopped an instance.
template <int THREADS, bool STOPPED>
__device__ void tile_offsets(const Bufs* __restrict__ Ball, int E, int tile, int* off, int* wsum) {
  const int n = 3 * E;
  const int per = (n + THREADS - 1) / THREADS;
  const int j0 = min(static_cast<int>(threadIdx.x) * per, n), j1 = min(j0 + per, n);
  int loc = 0;
  for (int j = j0; j < j1; ++j) {
    const DevState* S = Ball[j / 3].S;
    const long long np = (STOPPED || ldcg(&S->status) == 0) ? ldcg(&S->n_proc[j % 3]) : 0LL;
    const int t = static_cast<int>((np + tile - 1) / tile);
    off[j] = t;
    loc += t;
  }
  // block exclusive scan of the per-thread sums
  int incl = loc;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (static_cast<int>(lane_id()) >= o) incl += y;
  }
  const int w = threadIdx.x >> 5;
  if (lane_id() == 31) wsum[w] = incl;
  __syncthreads();
  int wbase = 0;
  for (int q = 0; q < w; ++q) wbase += wsum[q];
  int run = wbase + incl - loc;
  for (int j = j0; j < j1; ++j) {
    const int t = off[j];
    off[j] = run;
    run += t;
  }
  if (threadIdx.x == THREADS - 1) off[n] = wbase + incl;
  __syncthreads();
}

// a thread's particles from global memory
__device__ __forceinline__ void ld_vec(const float* p, float (&v)[4]) {
  const float4 a = __ldcs(reinterpret_cast<const float4*>(p));
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}
__device__ __forceinline__ void ld_vec(const double* p, double (&v)[2]) {
  const double2 a = __ldcs(reinterpret_cast<const double2*>(p));
  v[0] = a.x; v[1] = a.y;
}

// --- the push ------------------------------------------------------------------
constexpr int kEnsSegs = 8;    // segments of a CTA's share listed at a time

template <typename real, int THREADS>
struct EnsTile {
  static constexpr int kN = 16 / sizeof(real);  // particles per thread
  static constexpr int kTileN = THREADS * kN;
  static constexpr int kLog = (kTileN == 4096) ? 12 : (kTileN == 2048) ? 11 : (kTileN == 1024) ? 10 : 9;
  static_assert(kTileN == 1 << kLog, "tile sizes are powers of two");
  // a tile adds at most 2^kShift to a node; 32 bits tell the signed sums of
  // this many tiles apart
  static constexpr int kShift = 16 + kLog;
  static constexpr int kMost = (1 << (32 - kShift)) - 1;
};

// Tiles [t0, t1) of one (instance, species).
template <typename real>
struct EnsSeg {
  real *x, *u;
  const uint32_t* ids;
  long long n;  // slots
  real kap;
  int inst, s, t0, t1;
};

template <typename real, int THREADS>
struct alignas(128) EnsShared {
  EnsSeg<real> seg[kEnsSegs];
  unsigned int cnt[2][kSpecies];
  long long u_next;
  int nseg, abs_n;
  unsigned int cfl;
  int wsum[THREADS / 32];
};

constexpr int ens_min_ctas(int threads, size_t es) { return threads == 256 ? 3 : (threads == 512 && es == 4) ? 2 : 1; }

// One launch pushes every instance.  Each CTA takes one contiguous share of
// the flat (instance, species, tile) list and keeps the field table and the
// node sums of one instance at a time.
//
// What bounds it: the HBM stream of the particles, and close behind it the
// shared-memory pipe (two table reads and two node-sum atomics per particle at
// random cells).  A thread requests its next four particles before it works on
// the present ones, running on across the segments of the share; they wait in
// registers, since a ring of asynchronous copies puts a third more traffic on
// the shared-memory pipe (230 us without the tail instead of 217).  One signed
// 32-bit sum per node and a table of E alone take 16 bytes of shared memory a
// cell.  The end of a CTA is latency: impacts and their electrons one per
// lane, the beams dealt over all CTAs, in slots that need no counter.
//
// 160 gaps of 260 to 3985 cells, 7.0e7 particles: push 231 -> 222 us, step in
// a graph 268 -> 264 (with the removal's interleaving 209 and 239).
template <typename real, int THREADS>
__global__ void __launch_bounds__(THREADS, ens_min_ctas(THREADS, sizeof(real)))
k_push_ens(const Bufs* __restrict__ Ball, int E, int n_max, int beam_chunks,
           AbsRecE* __restrict__ abs_all, int abs_cap) {
  using V = EnsTile<real, THREADS>;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ EnsShared<real, THREADS> sh;
  const int tid = static_cast<int>(threadIdx.x);
  long long* Gs = reinterpret_cast<long long*>(smem);
  unsigned int* nd = reinterpret_cast<unsigned int*>(smem + align16(sizeof(long long) * (n_max + 1)));
  real* Et = reinterpret_cast<real*>(reinterpret_cast<unsigned char*>(nd) + align16(sizeof(unsigned int) * (n_max + 1)));
  int* off = reinterpret_cast<int*>(reinterpret_cast<unsigned char*>(Et) + align16(sizeof(real) * (n_max + 2)));
  for (int k = tid; k <= n_max; k += THREADS) nd[k] = 0u;
  if (tid == 0) {
    sh.abs_n = 0;
    sh.cfl = 0u;
  }
  if (tid < 2 * kSpecies) sh.cnt[tid / kSpecies][tid % kSpecies] = 0u;

  cudaGridDependencySynchronize();  // the previous solves (or removal) have completed
  cudaTriggerProgrammaticLaunchCompletion();
  AbsRecE* my_abs = abs_all + static_cast<size_t>(blockIdx.x) * abs_cap;

  int cur = -1, N = 0;  // the instance whose table and sums are in shared memory
  real Nr = real(0);
  bool folded = false;
  int pos = 0, neg = 0;  // tiles of each sign in the node sums
  typename Bits<real>::type cfl = 0;
  auto node_value = [&](unsigned int v) {
    const unsigned int o = static_cast<unsigned int>(neg) << V::kShift;
    return static_cast<long long>(v + o) - static_cast<long long>(o);
  };
  // the current instance's grid and tallies into global memory
  auto flush = [&]() {
    const unsigned int c = warp_max_u(float_bits(cfl));
    if (lane_id() == 0 && c) atomicMax(&sh.cfl, c);
    cfl = 0;
    __syncthreads();
    long long* G = Ball[cur].G;
    for (int k = tid; k <= N; k += THREADS) {
      add_global(G, k, N, node_value(nd[k]) + (folded ? Gs[k] : 0LL));
      nd[k] = 0u;
    }
    if (tid == 0) {
      DevState* S = Ball[cur].S;
      for (int e = 0; e < 2; ++e)
        for (int s = 0; s < kSpecies; ++s)
          if (sh.cnt[e][s]) atomicAdd(&S->absorbed[e][s], static_cast<unsigned long long>(sh.cnt[e][s]));
      const long long conv = static_cast<long long>(sh.cnt[0][CP_IONS]) -
                             static_cast<long long>(sh.cnt[0][CP_ELECTRONS]) -
                             static_cast<long long>(sh.cnt[0][CP_SECONDARIES]);
      if (conv) atomicAdd(reinterpret_cast<unsigned long long*>(&S->conv_count),
                          static_cast<unsigned long long>(conv));
      if (sh.cfl) atomicMax(&S->max_cfl_bits, sh.cfl);
      sh.cfl = 0u;
      for (int e = 0; e < 2; ++e)
        for (int s = 0; s < kSpecies; ++s) sh.cnt[e][s] = 0u;
    }
    folded = false;
    pos = neg = 0;
  };

  // Fetch cursor over the listed segments: `left` more tiles of segment q,
  // the next at x, u for this thread, whose particles end at x_end.
  struct Cursor {
    const real *x, *u, *x_end;
    int q, left;
  };
  const int nthr = tid * V::kN;
  tile_offsets<THREADS, true>(Ball, E, V::kTileN, off, sh.wsum);
  const long long U = off[3 * E], u1 = U * (blockIdx.x + 1) / gridDim.x;
  for (long long u0 = U * blockIdx.x / gridDim.x, u_next; u0 < u1; u0 = u_next) {
    if (tid == 0) {  // the next segments of [u0, u1)
      int lo = 0, hi = 3 * E;  // the entry holding tile u0: off[j] <= u0 < off[j+1]
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= u0) lo = mid;
        else hi = mid;
      }
      int q = 0;
      long long u = u0;
      for (int j = lo; u < u1 && q < kEnsSegs; ++j) {
        const int end = static_cast<int>(min(u1, static_cast<long long>(off[j + 1])));
        if (end <= u) continue;  // no tiles
        sh.seg[q].inst = j / 3;
        sh.seg[q].s = j % 3;
        sh.seg[q].t0 = static_cast<int>(u - off[j]);
        sh.seg[q].t1 = end - off[j];
        u = end;
        ++q;
      }
      sh.nseg = q;
      sh.u_next = u;
    }
    __syncthreads();
    if (tid < sh.nseg) {
      EnsSeg<real>& g = sh.seg[tid];
      const Bufs& B = Ball[g.inst];
      DevState* S = B.S;
      g.x = static_cast<real*>(ldcg(&S->xi[g.s]));
      g.u = static_cast<real*>(ldcg(&S->u[g.s]));
      g.ids = static_cast<const uint32_t*>(ldcg(reinterpret_cast<void* const*>(&S->id)));
      g.n = ldcg(&S->n_proc[g.s]);
      g.kap = kick<real>(B.P, ldcg(&S->pushed) == 0, g.s);
      if (ldcg(&S->status) != 0) g.t1 = g.t0;  // stopped
    }
    __syncthreads();
    const int nseg = sh.nseg;
    u_next = sh.u_next;
    Cursor nxt;
    auto enter = [&](int q) {
      nxt.left = 0;
      for (; q < nseg; ++q) {
        const EnsSeg<real>& g = sh.seg[q];
        if (g.t1 > g.t0) {
          const long long b = static_cast<long long>(g.t0) * V::kTileN + nthr;
          nxt.x = g.x + b;
          nxt.u = g.u + b;
          nxt.x_end = g.x + g.n;
          nxt.left = g.t1 - g.t0;
          break;
        }
      }
      nxt.q = q;
    };
    real xq[V::kN], uq[V::kN];
    auto fetch = [&]() {
      if (nxt.left > 0) {
        if (nxt.x < nxt.x_end) {
          ld_vec(nxt.x, xq);
          ld_vec(nxt.u, uq);
        }
        nxt.x += V::kTileN;
        nxt.u += V::kTileN;
        if (--nxt.left == 0) enter(nxt.q + 1);
      }
    };
#pragma unroll
    for (int c = 0; c < V::kN; ++c) xq[c] = uq[c] = real(0);
    enter(0);
    fetch();

    for (int q = 0; q < nseg; ++q) {
      const EnsSeg<real>& g = sh.seg[q];
      if (g.t1 == g.t0) continue;
      if (g.inst != cur) {
        if (cur >= 0) flush();
        cur = g.inst;
        const Bufs& B = Ball[cur];
        N = B.P->N;
        Nr = static_cast<real>(N);
        const real* Etab = static_cast<const real*>(B.Etab);
        for (int k = tid; k < N + 2; k += THREADS) Et[k] = __ldcg(&Etab[k]);
        __syncthreads();
      }
      const int s = g.s, sign = (s == CP_IONS) ? 1 : -1;
      const real kap = g.kap;
      const long long b = static_cast<long long>(g.t0) * V::kTileN + nthr;
      real* x = g.x + b;
      real* u = g.u + b;
      const real* const x_end = g.x + g.n;
      for (int left = g.t1 - g.t0; left > 0; --left, x += V::kTileN, u += V::kTileN) {
        real xv[V::kN], uv[V::kN];
#pragma unroll
        for (int c = 0; c < V::kN; ++c) {
          xv[c] = xq[c];
          uv[c] = uq[c];
        }
        fetch();
        if (pos + neg == V::kMost) {  // bounds every node sum to 32 bits
          __syncthreads();
          for (int k = tid; k <= N; k += THREADS) {
            const long long a = node_value(nd[k]);
            nd[k] = 0u;
            Gs[k] = folded ? Gs[k] + a : a;
          }
          __syncthreads();
          folded = true;
          pos = neg = 0;
        }
        if (sign > 0) ++pos; else ++neg;
        if (x >= x_end) continue;
#pragma unroll
        for (int c = 0; c < V::kN; ++c) {
          bool dep = false;
          if (inside(xv[c], Nr)) {  // live (dead slots hold -1)
            const real un = fma(kap, gather_tab(Et, xv[c]), uv[c]);
            const real xn = xv[c] + un;
            max_abs(cfl, un);
            if (!inside(xn, Nr)) {  // absorbed (a non-finite value counts at x = d)
              const int el = (xn <= real(0)) ? 0 : 1;
              atomicAdd(&sh.cnt[el][s], 1u);
              if (sign > 0) {
                const int slot = atomicAdd(&sh.abs_n, 1);
                if (slot < abs_cap) {
                  AbsRecE r;
                  r.id = g.ids[x + c - g.x];
                  r.inst_el = static_cast<uint32_t>(2 * cur + el);
                  r.u = static_cast<double>(un);
                  my_abs[slot] = r;
                } else {
                  atomicCAS(&Ball[cur].S->status, 0, CP_ERR_CAPACITY);
                }
              }
              xv[c] = real(-1);
              uv[c] = real(0);
            } else {
              dep = true;
              xv[c] = xn;
              uv[c] = un;
            }
          }
          if (dep) deposit_nodes(nd, fix_pos(xv[c]), sign);
        }
        put_vec(x, xv);
        put_vec(u, uv);
      }
    }
    __syncthreads();  // the listed segments are done
  }
  __syncthreads();
  if (cur >= 0) flush();

  // --- secondary emission from the ions this CTA saw absorbed ---------------
  // one record per lane (a warp's FP64 operation takes the pipe equally long
  // for any number of lanes): the counts, then the electrons one per lane
  const int na = min(sh.abs_n, abs_cap);
  const int lane = tid & 31;
  for (int r0 = tid - lane; r0 < na; r0 += THREADS) {
    const int r = r0 + lane;
    int nse = 0;
    unsigned long long wb = 0ULL;
    AbsRecE rec;
    rec.id = 0; rec.inst_el = 0; rec.u = 0.0;
    if (r < na) {
      rec = my_abs[r];
      const int el = static_cast<int>(rec.inst_el & 1u);
      const Bufs& B = Ball[rec.inst_el >> 1];
      const DevParams* Pi = B.P;
      DevState* Si = B.S;
      const double v = __ddiv_rn(__dmul_rn(rec.u, Pi->dx), Pi->dt);
      const double Eev = __ddiv_rn(__dmul_rn(__dmul_rn(__dmul_rn(0.5, Pi->m_i), v), v), Pi->e);
      nse = see_count(Pi, Eev, rec.id, ldcg(&Si->level));
      if (el == 0) {
        atomicAdd(reinterpret_cast<unsigned long long*>(&Si->ion_energy_q),
                  static_cast<unsigned long long>(__double2ll_rn(Eev * 256.0)));
        if (nse) atomicAdd(reinterpret_cast<unsigned long long*>(&Si->conv_count),
                           static_cast<unsigned long long>(static_cast<long long>(nse)));
      }
      if (nse) {
        atomicAdd(&Si->emitted[el], static_cast<unsigned long long>(nse));
        wb = atomicAdd(reinterpret_cast<unsigned long long*>(&Si->n_alloc[CP_SECONDARIES]),
                       static_cast<unsigned long long>(nse));
      }
    }
    const int incl = warp_incl_scan(nse);
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    for (int e0 = 0; e0 < total; e0 += 32) {
      const int e = e0 + lane;
      int src = 0;  // the record of electron e: the first lane whose count exceeds e
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
        if (__shfl_sync(0xffffffffu, incl, src + o - 1) <= e) src += o;
      src = min(src, 31);
      const uint32_t id = __shfl_sync(0xffffffffu, rec.id, src);
      const uint32_t ie = __shfl_sync(0xffffffffu, rec.inst_el, src);
      const int jn = e - __shfl_sync(0xffffffffu, incl - nse, src);
      const unsigned long long slot = __shfl_sync(0xffffffffu, wb, src) + static_cast<unsigned long long>(jn);
      if (e >= total) continue;
      const Bufs& B = Ball[ie >> 1];
      const DevParams* Pi = B.P;
      DevState* Si = B.S;
      const bool left = (ie & 1u) == 0u;
      const int Ni = Pi->N;
      double frac;
      const double vse = see_speed(Pi, id, ldcg(&Si->level), jn, &frac);
      const double use = vse * Pi->dt / Pi->dx;
      const double xd = left ? __dmul_rn(use, frac) : __dsub_rn(static_cast<double>(Ni), __dmul_rn(use, frac));
      const real xr = nudge_inside<real>(xd, Ni);
      if (slot < static_cast<unsigned long long>(Pi->cap[CP_SECONDARIES])) {
        static_cast<real*>(Si->xi[CP_SECONDARIES])[slot] = xr;
        static_cast<real*>(Si->u[CP_SECONDARIES])[slot] = static_cast<real>(left ? use : -use);
        deposit_global<real>(B.G, Ni, xr, -1);
      } else {
        atomicCAS(&Si->status, 0, CP_ERR_CAPACITY);
      }
    }
  }

  // --- the beams: THREADS ions of one instance at a time ----------------------
  // Ions are appended by the beam alone, behind the slots in use.
  for (long long item = blockIdx.x; item < static_cast<long long>(E) * beam_chunks; item += gridDim.x) {
    const int inst = static_cast<int>(item / beam_chunks);
    const int k0 = static_cast<int>(item - static_cast<long long>(inst) * beam_chunks) * THREADS;  // below the largest beam
    const Bufs& B = Ball[inst];
    const DevParams* Pi = B.P;
    DevState* Si = B.S;
    const int Bn = Pi->beam_per_step, k = k0 + tid;
    if (Bn <= k0 || ldcg(&Si->status) != 0) continue;
    if (k < Bn) {
      const int64_t step = ldcg(&Si->level);
      const int Ni = Pi->N;
      const U64x4 wv = philox4x64_10(static_cast<uint64_t>(k), static_cast<uint64_t>(step), 0, 0, Pi->seed, kTagBeam);
      const double frac = u01(wv.w[0]);
      const double ub = beam_speed<real>(Pi, u01(wv.w[1]));
      const real xr = nudge_inside<real>(__dsub_rn(static_cast<double>(Ni), __dmul_rn(ub, frac)), Ni);
      const int64_t slot = ldcg(&Si->n_proc[CP_IONS]) + k;
      if (slot < Pi->cap[CP_IONS]) {
        static_cast<real*>(Si->xi[CP_IONS])[slot] = xr;
        static_cast<real*>(Si->u[CP_IONS])[slot] = static_cast<real>(-ub);
        Si->id[slot] = Si->beam_id_base + static_cast<uint32_t>(step * Bn + k);
        deposit_global<real>(B.G, Ni, xr, 1);
      } else {
        atomicCAS(&Si->status, 0, CP_ERR_CAPACITY);
      }
    }
    if (k == 0) {
      atomicAdd(&Si->injected, static_cast<unsigned long long>(Bn));
      atomicAdd(reinterpret_cast<unsigned long long*>(&Si->n_alloc[CP_IONS]), static_cast<unsigned long long>(Bn));
    }
  }
}

// ---------------------------------------------------------------------------
// Removal of absorbed particles over the flat (instance, species, tile) list
// ---------------------------------------------------------------------------
template <typename real>
__global__ void __launch_bounds__(kThreads, sizeof(real) == 4 ? 3 : 1) k_compact_ens(const Bufs* __restrict__ Ball, int E) {
  constexpr int TILE = kThreads * kPerThread;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int wsum[kThreads / 32];
  PackShared<real>& sh = *reinterpret_cast<PackShared<real>*>(smem);
  int* off = reinterpret_cast<int*>(smem + align16(sizeof(PackShared<real>)));
  tile_offsets<kThreads, false>(Ball, E, TILE, off, wsum);
  const long long U = off[3 * E];
  // each CTA takes one contiguous share of the tiles
  const long long u1 = U * (blockIdx.x + 1) / gridDim.x;
  long long u = U * blockIdx.x / gridDim.x;
  int j = 0, hi = 3 * E;  // the entry holding tile u: off[j] <= u < off[j+1]
  while (hi - j > 1) {
    const int mid = (j + hi) >> 1;
    if (off[mid] <= u) j = mid;
    else hi = mid;
  }
  for (; u < u1; ++j) {
    const long long end = min(u1, static_cast<long long>(off[j + 1]));
    if (end <= u) continue;  // no tiles
    DevState* S = Ball[j / 3].S;
    const int s = j % 3;
    const real* xs = static_cast<const real*>(S->xi[s]);
    const real* us = static_cast<const real*>(S->u[s]);
    const uint32_t* is = s == CP_IONS ? S->id : nullptr;
    real* xd = static_cast<real*>(S->xi_alt[s]);
    real* ud = static_cast<real*>(S->u_alt[s]);
    uint32_t* id_d = S->id_alt;
    const int64_t n = S->n_proc[s], chunks = off[j + 1] - off[j];
    for (int64_t t = u - off[j]; t < end - off[j]; ++t)
      pack_block<real>(sh, xs, us, is, n, chunks, t, xd, ud, id_d, &S->compact_n[s]);
    u = end;
  }
}

// One thread per instance: pad the packed stores to whole vectors and swap.
template <typename real>
__global__ void k_swap_ens(const Bufs* __restrict__ Ball, int E) {
  const int inst = blockIdx.x * blockDim.x + threadIdx.x;
  if (inst >= E) return;
  DevState* S = Ball[inst].S;
  if (S->status != 0) return;
  for (int s = 0; s < kSpecies; ++s) {
    const long long cnt = static_cast<long long>(S->compact_n[s]);
    const long long c4 = (cnt + 3) & ~3LL;
    real* xd = reinterpret_cast<real*>(S->xi_alt[s]);
    real* ud = reinterpret_cast<real*>(S->u_alt[s]);
    for (long long k = cnt; k < c4; ++k) {
      xd[k] = real(-1);
      ud[k] = real(0);
    }
    void* t0 = S->xi[s];
    S->xi[s] = S->xi_alt[s];
    S->xi_alt[s] = t0;
    void* t1 = S->u[s];
    S->u[s] = S->u_alt[s];
    S->u_alt[s] = t1;
    S->n_alloc[s] = c4;
    S->n_proc[s] = c4;
    S->compact_n[s] = 0ULL;
  }
  uint32_t* t2 = S->id;
  S->id = S->id_alt;
  S->id_alt = t2;
}

// ---------------------------------------------------------------------------
// Host-side launchers
// ---------------------------------------------------------------------------
size_t push_ens_smem_bytes(int n_max, int precision, int E) {
  const size_t es = (precision == CP_FP32) ? 4 : 8;
  return align16(sizeof(long long) * (n_max + 1)) + align16(sizeof(unsigned int) * (n_max + 1)) +
         align16(es * (n_max + 2)) + align16(sizeof(int) * (3 * E + 1));
}

int ens_max_instances() { return kEnsMaxEntries / 3; }

template <typename real, int T>
static const void* push_ens_fn() {
  return reinterpret_cast<const void*>(k_push_ens<real, T>);
}

static const void* push_ens_kernel(int precision, int threads) {
  if (precision == CP_FP32) {
    if (threads == 256) return push_ens_fn<float, 256>();
    if (threads == 1024) return push_ens_fn<float, 1024>();
    return push_ens_fn<float, 512>();
  }
  if (threads == 256) return push_ens_fn<double, 256>();
  if (threads == 1024) return push_ens_fn<double, 1024>();
  return push_ens_fn<double, 512>();
}

// Resident CTAs per SM of the ensemble push for a block size (0: not
// launchable).  The kernels' shared-memory limit is the largest the device
// allows: ensembles of other sizes share them.
cudaError_t push_ens_occupancy(int precision, int threads, size_t smem, int* per_sm) {
  const void* fn = push_ens_kernel(precision, threads);
  int dev = 0, most = 0;
  cudaFuncAttributes at;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&at, fn);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, most - static_cast<int>(at.sharedSizeBytes));
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, fn, threads, smem);
}

cudaError_t push_ens_launch(int precision, int threads, int grid, size_t smem, const Bufs* Ball,
                            int E, int n_max, int beam_max, void* abs, int abs_cap, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int chunks = beam_max / threads + (beam_max % threads != 0 ? 1 : 0);  // of the largest beam
  void* args[] = {&Ball, &E, &n_max, &chunks, &abs, &abs_cap};
  return cudaLaunchKernelExC(&cfg, push_ens_kernel(precision, threads), args);
}

size_t abs_rec_ens_bytes() { return sizeof(AbsRecE); }

__global__ void k_status_ens(const Bufs* __restrict__ Ball, int E, int* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < E) out[i] = Ball[i].S->status;
}

cudaError_t status_ens_launch(const Bufs* Ball, int E, int* out, cudaStream_t st) {
  k_status_ens<<<(E + 127) / 128, 128, 0, st>>>(Ball, E, out);
  return cudaGetLastError();
}

static size_t compact_ens_smem(int precision, int E) {
  return align16(precision == CP_FP32 ? sizeof(PackShared<float>) : sizeof(PackShared<double>)) + sizeof(int) * (3 * E + 1);
}

// The removal's shared-memory limit: the largest number of instances'.
cudaError_t compact_ens_configure(int precision) {
  const void* fn = precision == CP_FP32 ? reinterpret_cast<const void*>(k_compact_ens<float>)
                                        : reinterpret_cast<const void*>(k_compact_ens<double>);
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(compact_ens_smem(precision, ens_max_instances())));
}

cudaError_t compact_ens_launch(int precision, const Bufs* Ball, int E, int grid, cudaStream_t st) {
  const size_t smem = compact_ens_smem(precision, E);
  if (precision == CP_FP32) k_compact_ens<float><<<grid, kThreads, smem, st>>>(Ball, E);
  else k_compact_ens<double><<<grid, kThreads, smem, st>>>(Ball, E);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (precision == CP_FP32) k_swap_ens<float><<<(E + 127) / 128, 128, 0, st>>>(Ball, E);
  else k_swap_ens<double><<<(E + 127) / 128, 128, 0, st>>>(Ball, E);
  return cudaGetLastError();
}

}  // namespace cpk
