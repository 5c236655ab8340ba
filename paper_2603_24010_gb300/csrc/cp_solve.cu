// cp_solve.cu -- the coupled field/circuit solve of a new time level.
//
// k_solve (one thread-block cluster of 1 to 16 CTAs) solves the level: the
//   bordered tridiagonal system of App. B with the circuit row of Sec. 2.4.2
//   (strict, Eq. Poisson_BC2) or Sec. 2.4.3 (weak, Eq. Poisson_BC3) is
//   factorised into two bidiagonal scans whose charge sums are exact integers
//   (one associative scan gives the int64 prefix of the charge grid and the
//   prefix of that); FP64 enters only at the final scaling, so the solve is
//   direct and its backward error is checked over every row and the circuit
//   row, with FP64 iterative refinement if it exceeds the requested tolerance.
//   Chunk totals and residual maxima are pushed into every rank's shared
//   memory (st.async on a transaction barrier).
#include <algorithm>
#include <cstddef>

#include "cp_common.cuh"
#include "cp_mlp.cuh"

namespace cpk {
// ---------------------------------------------------------------------------
// Scans and reductions for the cluster solve
// ---------------------------------------------------------------------------
__device__ __forceinline__ long long shfl_up_t(long long v, int o) {
  return __shfl_up_sync(0xffffffffu, v, o);
}
__device__ __forceinline__ double shfl_up_t(double v, int o) {
  return __shfl_up_sync(0xffffffffu, v, o);
}
__device__ __forceinline__ __int128 shfl_up_t(__int128 v, int o) {
  const unsigned long long lo = static_cast<unsigned long long>(v);
  const unsigned long long hi = static_cast<unsigned long long>(static_cast<unsigned __int128>(v) >> 64);
  const unsigned long long l2 = __shfl_up_sync(0xffffffffu, lo, o);
  const unsigned long long h2 = __shfl_up_sync(0xffffffffu, hi, o);
  return static_cast<__int128>((static_cast<unsigned __int128>(h2) << 64) | l2);
}

// Sign-magnitude conversion: both 64-bit halves of |v| are non-negative, so
// hi 2^64 + lo has no cancellation (error below 1 ulp of |v|).
__device__ __forceinline__ double i128_to_double(__int128 v) {
  const bool neg = v < 0;
  const unsigned __int128 m = neg ? static_cast<unsigned __int128>(-v) : static_cast<unsigned __int128>(v);
  const unsigned long long hi = static_cast<unsigned long long>(m >> 64);
  const unsigned long long lo = static_cast<unsigned long long>(m);
  const double d = fma(static_cast<double>(hi), 18446744073709551616.0, static_cast<double>(lo));
  return neg ? -d : d;
}

// In-place inclusive scan of a[idx(m)], m = 0..n-1 (idx = m, or n-1-m for a
// suffix scan), contiguous runs per thread; returns the CTA total.
template <typename T>
__device__ T cta_scan(T* a, int n, bool reverse, T* wsum) {
  const int per = (n + kSolveThreads - 1) / kSolveThreads;
  const int lo = min(static_cast<int>(threadIdx.x) * per, n);
  const int hi = min(lo + per, n);
  T s = T(0);
  for (int m = lo; m < hi; ++m) s += a[reverse ? n - 1 - m : m];
  T incl = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T y = shfl_up_t(incl, o);
    if (static_cast<int>(lane_id()) >= o) incl += y;
  }
  const int w = threadIdx.x >> 5;
  __syncthreads();
  if (lane_id() == 31) wsum[w] = incl;
  __syncthreads();
  if (threadIdx.x < 32) {
    T t = (threadIdx.x < kSolveThreads / 32) ? wsum[threadIdx.x] : T(0);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const T y = shfl_up_t(t, o);
      if (static_cast<int>(threadIdx.x) >= o) t += y;
    }
    wsum[threadIdx.x] = t;
  }
  __syncthreads();
  T run = (w > 0 ? wsum[w - 1] : T(0)) + (incl - s);
  for (int m = lo; m < hi; ++m) {
    const int k = reverse ? n - 1 - m : m;
    run += a[k];
    a[k] = run;
  }
  const T total = wsum[kSolveThreads / 32 - 1];
  __syncthreads();
  return total;
}

__device__ double cta_sum(double v, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5;
  __syncthreads();
  if (lane_id() == 0) red[w] = v;
  __syncthreads();
  double t = 0.0;
  for (int k = 0; k < kSolveThreads / 32; ++k) t += red[k];
  __syncthreads();
  return t;
}

// Exclusive prefix (in rank order, or reverse rank order) and total over the
// cluster of one value per CTA, through distributed shared memory.
template <typename T>
__device__ void cluster_prefix(T mine, T* slot, bool reverse, T* excl, T* total) {
  cg::cluster_group cl = cg::this_cluster();
  if (threadIdx.x == 0) *slot = mine;
  cl.sync();
  const unsigned me = cl.block_rank();
  const unsigned nr = cl.num_blocks();
  T acc = T(0), tot = T(0);
  for (unsigned r = 0; r < nr; ++r) {
    const T v = *cl.map_shared_rank(slot, r);
    if (reverse ? (r > me) : (r < me)) acc += v;
    tot += v;
  }
  *excl = acc;
  *total = tot;
  cl.sync();
}

// FP64 direct solve of the same tridiagonal system for an arbitrary right-hand
// side (used by the refinement sweeps): on entry v[k] = b_{lo+k}, b0 = b_0;
// on exit v[k] = x_{lo+k}.  D_i = D_0 - sum_{j=1..i} b_j, D_0 = b_0 - gam x_0,
// x_0 (1 + N gam) = N b_0 - sum_i sum_{j=1..i} b_j, x_i = sum_{k>=i} D_k.
__device__ void cluster_tri_solve_f64(double* v, int lo, int m, int N, double b0, double gam,
                                      double* wsum, double* slot, double* sc) {
  if (lo == 0 && threadIdx.x == 0 && m > 0) v[0] = 0.0;
  __syncthreads();
  double off, tot;
  const double t1 = cta_scan(v, m, false, wsum);
  cluster_prefix(t1, slot, false, &off, &tot);
  double part = 0.0;
  for (int k = threadIdx.x; k < m; k += kSolveThreads) {
    v[k] += off;  // B_i
    part += v[k];
  }
  const double Tl = cta_sum(part, wsum);
  double o2, T;
  cluster_prefix(Tl, slot, false, &o2, &T);
  if (threadIdx.x == 0) {
    const double x0 = (static_cast<double>(N) * b0 - T) / (1.0 + static_cast<double>(N) * gam);
    sc[0] = b0 - gam * x0;
  }
  __syncthreads();
  const double D0 = sc[0];
  for (int k = threadIdx.x; k < m; k += kSolveThreads) v[k] = D0 - v[k];
  __syncthreads();
  const double t3 = cta_scan(v, m, true, wsum);  // suffix sums within the chunk
  double o3, T3;
  cluster_prefix(t3, slot, true, &o3, &T3);  // sums of the chunks after this one
  for (int k = threadIdx.x; k < m; k += kSolveThreads) v[k] += o3;
  __syncthreads();
}

// ---------------------------------------------------------------------------
// The solve of one level by the CTAs of one cluster.
//
// Bound: latency.  A level is a chain of short dependent stages (grid loads,
// scan, exchange, potential of node 0, rows, residual, exchange, decision),
// so what counts is the number of stages and what each waits for:
//
// * roles: warps 0-7 own the rows; warp 8 reads the circuit state, forms the
//   circuit row while the others scan, and exchanges the totals and the
//   residual maxima with the other ranks; warp 9 commits the level while the
//   rows are evaluated and checked (the commit needs phi_0 only; the backward
//   error is filled in last);
// * the exchanges are one-way: every rank pushes its values into every
//   rank's shared memory with st.async and waits on its own transaction
//   barrier (no cluster barrier and no remote load on the path), and a rank
//   may leave once everything addressed to it has arrived;
// * what the predecessor does not write (parameters, barrier set-up) is read
//   and done before the wait for it;
// * outputs are written before the backward error is known, and again in the
//   rare case that it calls for a refinement.
//
// Rows per thread: chunk / 256, and the cluster has one CTA per 256 rows up
// to 16.  FP64 is what a row costs (about a dozen operations at 2 per cycle
// and SM), so more rows per SM cost more than the exchange saves.
// Measured (GB300, event-bracketed launch; an empty kernel reads 4-5 us): 11.6
// us at 256 cells and 12.4 us at 4096, against 18.4 us for one 16-CTA cluster
// of 512 threads with cluster barriers, remote loads and a commit at the end.
// Graph-timed step: 22.9 against 30.4 us (4096 cells, 3.3e5 FP32 particles),
// 17.5 against 24.5 us (1531 cells, 1e6), 118 against 125 us (4096, 3.1e7).
// ---------------------------------------------------------------------------
constexpr int kRowWarps = kRowThreads / 32;
constexpr int kCircuitWarp = kRowWarps;     // warp 8
constexpr int kCommitWarp = kRowWarps + 1;  // warp 9
static_assert(kSolveThreads == kRowThreads + 64, "two more warps than rows");

// a b as a 128-bit integer from one 64 x 64 -> 128 product
__device__ __forceinline__ __int128 mul_wide(long long a, long long b) {
  const unsigned long long lo = static_cast<unsigned long long>(a) * static_cast<unsigned long long>(b);
  const long long hi = __mul64hi(a, b);
  return static_cast<__int128>((static_cast<unsigned __int128>(static_cast<unsigned long long>(hi)) << 64) | lo);
}

// The accumulator of the prefix of prefixes: int64 when the stores cannot
// hold enough charge to overflow it (|sum| <= 2^16 macroparticles N < 2^62),
// else int128.
template <typename Acc>
__device__ __forceinline__ Acc len_times(int len, long long s1);
template <>
__device__ __forceinline__ long long len_times<long long>(int len, long long s1) {
  return static_cast<long long>(len) * s1;
}
template <>
__device__ __forceinline__ __int128 len_times<__int128>(int len, long long s1) {
  return mul_wide(len, s1);
}
// exactly rounded |v| with v's sign; the two forms agree where both apply
__device__ __forceinline__ double acc_to_double(long long v) { return static_cast<double>(v); }
__device__ __forceinline__ double acc_to_double(__int128 v) { return i128_to_double(v); }

// Scan segment of the charge grid: s1 = sum of G_i, s2 = sum over the
// segment of the inclusive prefix of G within it.  "a then b" with len_b
// rows in b: (a1 + b1, a2 + b2 + len_b a1).
template <typename Acc>
struct alignas(16) Seg {
  Acc s2;
  long long s1;
};

template <typename Acc>
__device__ __forceinline__ Seg<Acc> seg_then(const Seg<Acc>& a, const Seg<Acc>& b, int len_b) {
  Seg<Acc> r;
  r.s1 = a.s1 + b.s1;
  r.s2 = a.s2 + b.s2 + len_times<Acc>(len_b, a.s1);
  return r;
}

template <typename Acc>
__device__ __forceinline__ Seg<Acc> shfl_up_seg(const Seg<Acc>& v, int o) {
  Seg<Acc> r;
  r.s1 = shfl_up_t(v.s1, o);
  r.s2 = shfl_up_t(v.s2, o);
  return r;
}

// |x| as the bit pattern of a non-negative double: such patterns order like
// the values, so maxima can be taken on the integer pipe (GB300's FP64 pipe
// is narrow).
__device__ __forceinline__ unsigned long long abs_bits(double x) {
  return static_cast<unsigned long long>(__double_as_longlong(x)) & 0x7FFFFFFFFFFFFFFFULL;
}

// Warp maximum of 64-bit patterns: the high words first, then the low words
// of the lanes that hold the largest high word (two hardware reductions).
__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long v) {
  const unsigned int hi = static_cast<unsigned int>(v >> 32);
  const unsigned int mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned int ml = __reduce_max_sync(0xffffffffu, hi == mh ? static_cast<unsigned int>(v) : 0u);
  return (static_cast<unsigned long long>(mh) << 32) | ml;
}

struct alignas(16) MaxSlot {
  unsigned long long rmax, xmax, bmax;  // bit patterns of non-negative doubles (bmax: integer)
  unsigned long long lost;              // the rank's wait for the totals ran out
};

// Dynamic shared memory of one rank's rows: G, phi, E, b and r.
__host__ __device__ constexpr size_t solve_rows_bytes(int chunk) {
  return align16(8 * static_cast<size_t>(chunk)) + align16(4 * 8 * static_cast<size_t>(chunk));
}

// --- one-way exchange between the ranks of a cluster ------------------------
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ uint32_t remote_addr(const void* p, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr(p)), "r"(rank));
  return r;
}
// 16 bytes into another rank's shared memory, counted on its barrier
__device__ __forceinline__ void push16(uint32_t dst, unsigned long long a, unsigned long long b, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(dst),
               "l"(a), "l"(b), "r"(bar)
               : "memory");
}
// Polls of an exchange's barrier before a rank gives up (which: 0 the totals,
// 1 the maxima).  A test builds the library with limits that run out.
constexpr int kMostPolls = 1 << 20;
#ifndef CP_EXCHANGE_POLLS
#define CP_EXCHANGE_POLLS(which) kMostPolls
#endif
// Wait for the barrier's first phase; false when the limit of polls is
// reached (a rank that never sent: cannot happen unless one failed).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, int limit) {
  for (int i = 0; i < limit; ++i) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_addr(bar))
        : "memory");
    if (done) return true;
  }
  return false;
}

// Circuit charge, surface charge and current of a solved level from the
// circuit scalars of the solve (sc: [2] g, [3] K or Q^n, [6] Q_conv, [7]
// sigma_{n-1}, [8] Q^{n-1}, [9] Q^{n-2}) and the level's phi_0.  strict: a
// circuit whose charge follows Q^n = K - g phi_0^n (series RLC or Tesla).
__device__ __forceinline__ void level_charges(const DevParams* P, const double* sc, bool strict,
                                              double phi0, double* Qn, double* sigma_n, double* I) {
  const double Qconv = sc[6], sigma_prev = sc[7], Q1 = sc[8], Q2 = sc[9];
  if (strict) {
    *Qn = sc[3] - sc[2] * phi0;                             // Eqs. Q4_phi_relation, K_def
    *sigma_n = sigma_prev + (Qconv + *Qn - Q1) * P->inv_A;  // Eq. sigma_update
    *I = (3.0 * *Qn - 4.0 * Q1 + Q2) * P->inv_2dt;
  } else if (P->circuit != CP_CIRCUIT_OPEN) {
    *Qn = sc[3];                                            // weak: the circuit's loop charge
    *sigma_n = sigma_prev + (Qconv + *Qn - Q1) * P->inv_A;  // Eq. top_plate_charge
    *I = (3.0 * *Qn - 4.0 * Q1 + Q2) * P->inv_2dt;
  } else {
    *Qn = Q1;
    *sigma_n = sigma_prev + Qconv * P->inv_A;
    *I = 0.0;
  }
}

// The installed network is copied into shared memory while the solve runs
// (asynchronous copies, waited for only when the network runs).
__device__ __forceinline__ void prefetch_net(const PredNet* net, PredNet* s_net) {
  const char* src = reinterpret_cast<const char*>(net);
  char* dst = reinterpret_cast<char*>(s_net);
  for (size_t o = 16 * static_cast<size_t>(threadIdx.x); o < kPredNetBytes; o += 16 * kSolveThreads)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst + o)), "l"(src + o) : "memory");
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// The words of the device state that a solve reads, as one block: from
// `level` up to the compaction counters.
constexpr int kStateWord0 = offsetof(DevState, level) / 8;
constexpr int kStateWords = (offsetof(DevState, compact_n) - offsetof(DevState, level)) / 8;
static_assert(offsetof(DevState, level) % 8 == 0 && offsetof(DevState, compact_n) % 8 == 0, "whole words");

// Predictor step on one CTA (all threads), for the paths that keep it in the
// solve: the level's row from the solve's scalars, then the shared predictor
// level (check, ring append, network on the copy in shared memory, s_net).
// `st` is the copy of the device state as the solve found it.
__device__ __noinline__ void predictor_update(const DevParams* P, DevState* S, const DevState* st,
                                              const PredNet* s_net, const double* sc, bool strict_c,
                                              double phi0) {
  __shared__ PredScratch sp;
  __shared__ PredLevel L;
  const int pos0 = st->feat_pos;
  if (threadIdx.x == 0) {
    double Qn, sigma_n, I;
    level_charges(P, sc, strict_c, phi0, &Qn, &sigma_n, &I);
    L.Qconv = sc[6];
    L.phi0 = phi0;
    L.phi0_prev = sc[32];
    L.Qsurf = __dmul_rn(sigma_n, P->area);
    L.Qsurf_prev = __dmul_rn(sc[7], P->area);
    L.Qn = Qn;
    L.Q1 = sc[8];
    L.emitted = static_cast<double>(st->emitted[0]);
    L.ion_eV = static_cast<double>(st->ion_energy_q) / 256.0;
    L.had_pred = st->pred_ready;
    L.J_pred = st->J_pred;
    L.err_avg = st->err_avg;
    L.J_avg = st->J_avg;
    L.n_eval = st->n_eval;
    L.pos = pos0;
    L.n_feat = st->n_feat;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");  // this thread's copies of the network
  __syncthreads();
  // the 7 older rows of the window (ring slots pos+1..pos+7, oldest first)
  double v_old = 0.0;
  if (threadIdx.x < kPredIn - kPredFeat)
    v_old = st->feat[(pos0 + 1 + static_cast<int>(threadIdx.x) / kPredFeat) & (kPredWindow - 1)]
                    [threadIdx.x % kPredFeat];
  pred_level<kRowThreads>(s_net, P->C, S, &L, v_old, &sp);
}

// What the commit writes for a level whose electrode potential is phi0 (one
// warp; every value comes from the shared copies, so a second call after a
// refinement writes the same fields again).
// (The pointers are passed one by one: a reference to the kernel's parameter
// block would force a copy of it into local memory for the whole solve.)
__device__ __noinline__ int commit_level(DevState* S, cp_diag* hist, int64_t hist_rows, const double* vs,
                                         const DevParams* P, const DevState* st, const double* sc, int do_push,
                                         int mode, bool strict_c, double phi0, double eta) {
  const int lane = static_cast<int>(lane_id());
  const int64_t level = st->level + (do_push ? 1 : 0);
  const double Q1 = sc[8], Q2 = sc[9], Q3 = sc[10];
  double Qn, sigma_n, I;
  level_charges(P, sc, strict_c, phi0, &Qn, &sigma_n, &I);
  int status = 0;
  if (!isfinite(phi0) || !isfinite(sigma_n) || !isfinite(Qn)) status = CP_ERR_NONFINITE;
  if (lane == 0) {
    const double dt = P->dt, A = P->area;
    const bool on = do_push != 0;
    cp_diag d;
    d.step = level;
    d.t = static_cast<double>(level) * dt;
    d.V_gap = phi0;
    d.I_circ = I;
    d.Q_surf = sigma_n * A;
    d.Q_conv = sc[6];
    d.Q_circ = Qn;
    d.V_source = sc[4];
    d.residual = eta;
    d.ion_energy_eV = on ? static_cast<double>(st->ion_energy_q) / 256.0 : 0.0;
    d.max_cfl = on ? static_cast<double>(__uint_as_float(st->max_cfl_bits)) : 0.0;
    d.J_hat = sc[15];
    for (int s = 0; s < kSpecies; ++s) {
      d.n_live[s] = st->n_live[s];
      for (int e = 0; e < 2; ++e) {
        d.absorbed[e][s] = on ? static_cast<int64_t>(st->absorbed[e][s]) : 0;
        d.n_live[s] -= d.absorbed[e][s];
      }
    }
    d.emitted[0] = on ? static_cast<int64_t>(st->emitted[0]) : 0;
    d.emitted[1] = on ? static_cast<int64_t>(st->emitted[1]) : 0;
    d.injected = on ? static_cast<int64_t>(st->injected) : 0;
    d.n_live[1] += d.injected;
    d.n_live[2] += d.emitted[0] + d.emitted[1];
    d.conv_count = on ? st->conv_count : 0;
    S->cur = d;
    if (level < hist_rows) hist[level] = d;
    for (int s = 0; s < kSpecies; ++s) S->n_live[s] = d.n_live[s];
    S->pv_phi0 = sc[32];  // the predictor's previous level (phi_0, Q_surf)
    S->pv_Qsurf = sc[7] * A;
    S->sigma = sigma_n;
    S->phi0_last = phi0;
    S->Qh[3] = Q3;
    S->Qh[2] = Q2;
    S->Qh[1] = Q1;
    S->Qh[0] = Qn;
    // source and BDF2 history of the next level (off the next solve's critical path)
    S->nxt_Vs = (level + 1 < hist_rows + 1) ? vs[level + 1] : 0.0;
    S->nxt_hist = P->L4dt2 * (24.0 * Qn - 22.0 * Q1 + 8.0 * Q2 - Q3) + P->R2dt * (4.0 * Qn - Q1);
    S->level = level;
    if (do_push) S->pushed = 1;
  }
  // the push's tallies start the next step at zero
  if (lane < 2 * kSpecies) S->absorbed[lane / kSpecies][lane % kSpecies] = 0ULL;
  if (lane == 8) S->emitted[0] = S->emitted[1] = 0ULL;
  if (lane == 9) {
    S->injected = 0ULL;
    S->conv_count = 0;
    S->ion_energy_q = 0;
    S->max_cfl_bits = 0u;
  }
  if (P->circuit == CP_CIRCUIT_TESLA && do_push) {  // the five loop charges
    double q = 0.0;
    if (lane < 5) {
      q = (mode == 0) ? sc[40 + lane] - phi0 * P->t_ws[lane] : sc[40 + lane] + sc[36] * P->t_ww[lane];
      for (int k = 3; k > 0; --k) S->Qt[k][lane] = st->Qt[k - 1][lane];
      S->Qt[0][lane] = q;
    }
    if (!__all_sync(0xffffffffu, isfinite(q))) status = CP_ERR_NONFINITE;
  }
  return status;
}

// A rank is lost when one of its waits ran out, or when another rank says with
// its maxima that its first did.  It commits and refines nothing (the status is
// CP_ERR_TIMEOUT) and leaves behind two cluster barriers: at the first every
// rank has sent all it sends or has left, at the second those about to refine
// have read the flags, and have left as well.  What is addressed to it must
// have arrived before it may leave.
__device__ __noinline__ void leave_lost(uint64_t* bars) {
  cg::cluster_group cl = cg::this_cluster();
  cl.sync();
  cl.sync();
  mbar_wait(&bars[0], kMostPolls);
  mbar_wait(&bars[1], kMostPolls);
  asm volatile("cp.async.wait_all;" ::: "memory");  // the network's copies
}

// Before a refinement: whether any rank is lost (all ranks that are not call
// this: they have the same backward error).
__device__ __noinline__ bool any_lost(int* lost) {
  cg::cluster_group cl = cg::this_cluster();
  cl.sync();
  int n = 0;
  for (unsigned r = 0; r < cl.num_blocks(); ++r) n += *cl.map_shared_rank(lost, r);
  cl.sync();
  return n != 0;
}

// Everything the refinement needs of the solve (rare path).
struct Refine {
  double *ph, *Ee, *bb, *rr;
  double *sc, *wd, *slotd, *edge;  // edge[2]: this rank's first and last potential
  unsigned long long (*wu)[32];
  MaxSlot* slot;
  double* s_eta;
  int lo, hi, m, N;
  double gam, inv_dx, tol;
  bool strict_rlc;
};

// The normwise backward error of the solved rows and of the circuit row.
__device__ __forceinline__ double backward_error(const DevParams* P, const double* sc, bool strict_rlc, double gam,
                                                 double rmd, double xmd, double bmd, double p0) {
  const double nA = fmax(fabs(1.0 + gam) + 1.0, 4.0);
  const double den = nA * xmd + bmd;
  double e = den > 0.0 ? rmd / den : 0.0;
  if (strict_rlc) {  // the circuit row with the potential of row 0
    const double Qn = sc[3] - sc[2] * p0;
    const double kvl = P->a21 * Qn - (sc[4] + sc[5]) + p0;
    const double kden = P->a21 * fabs(Qn) + fabs(sc[4] + sc[5]) + fabs(p0);
    if (kden > 0.0) e = fmax(e, fabs(kvl) / kden);
  }
  return e;
}

__device__ __forceinline__ double row_residual(const double* ph, double b, int k, int i, int m, double gam,
                                               double prev_phi, double next_phi) {
  const double xp = (k + 1 < m) ? ph[k + 1] : next_phi;
  if (i == 0) return (1.0 + gam) * ph[k] - xp - b;
  const double xq = (k > 0) ? ph[k - 1] : prev_phi;
  return (xq - 2.0 * ph[k] + xp) - b;
}

// At most three sweeps x -= A^{-1} r in FP64, until the backward error is
// within tol; all threads of the cluster.  Returns the last backward error;
// *phi0 is the refined potential of node 0.
__device__ __noinline__ double refine(const Refine& R, const DevParams* P, double prev_phi, double next_phi,
                                      double* phi0) {
  cg::cluster_group cl = cg::this_cluster();
  const int rank = static_cast<int>(cl.block_rank()), nr = static_cast<int>(cl.num_blocks());
  const int m = R.m, lo = R.lo, hi = R.hi, N = R.N;
  double eta = 0.0;
  for (int sweep = 1; sweep <= 3; ++sweep) {
    for (int k = threadIdx.x; k < m; k += kSolveThreads)
      R.rr[k] = row_residual(R.ph, R.bb[k], k, lo + k, m, R.gam, prev_phi, next_phi);
    __syncthreads();
    if (rank == 0 && threadIdx.x == 0) R.sc[14] = R.rr[0];
    cl.sync();
    const double r0all = cl.map_shared_rank(&R.sc[14], 0)[0];
    cluster_tri_solve_f64(R.rr, lo, m, N, r0all, R.gam, R.wd, R.slotd, R.sc + 16);
    for (int k = threadIdx.x; k < m; k += kSolveThreads) R.ph[k] -= R.rr[k];
    __syncthreads();
    if (threadIdx.x == 0 && m > 0) {
      R.edge[0] = R.ph[0];
      R.edge[1] = R.ph[m - 1];
    }
    cl.sync();
    next_phi = (hi < N) ? cl.map_shared_rank(R.edge, rank + 1)[0] : 0.0;
    prev_phi = (lo > 0) ? cl.map_shared_rank(R.edge, rank - 1)[1] : 0.0;
    *phi0 = cl.map_shared_rank(R.edge, 0)[0];
    for (int k = threadIdx.x; k < m; k += kSolveThreads)
      R.Ee[k] = (R.ph[k] - ((k + 1 < m) ? R.ph[k + 1] : next_phi)) * R.inv_dx;
    // backward error over the cluster
    unsigned long long rm = 0ULL, xm = 0ULL, bm = 0ULL;
    for (int k = threadIdx.x; k < m; k += kSolveThreads) {
      rm = max(rm, abs_bits(row_residual(R.ph, R.bb[k], k, lo + k, m, R.gam, prev_phi, next_phi)));
      xm = max(xm, abs_bits(R.ph[k]));
      bm = max(bm, abs_bits(R.bb[k]));
    }
    rm = warp_max_u64(rm);
    xm = warp_max_u64(xm);
    bm = warp_max_u64(bm);
    if (lane_id() == 0) {
      R.wu[0][threadIdx.x >> 5] = rm;
      R.wu[1][threadIdx.x >> 5] = xm;
      R.wu[2][threadIdx.x >> 5] = bm;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      MaxSlot q = {0ULL, 0ULL, 0ULL, 0ULL};
      for (int w = 0; w < kSolveThreads / 32; ++w) {
        q.rmax = max(q.rmax, R.wu[0][w]);
        q.xmax = max(q.xmax, R.wu[1][w]);
        q.bmax = max(q.bmax, R.wu[2][w]);
      }
      *R.slot = q;
    }
    cl.sync();
    if (threadIdx.x == 0) {
      unsigned long long a = 0ULL, b = 0ULL, c = 0ULL;
      for (int r = 0; r < nr; ++r) {
        const MaxSlot* q = cl.map_shared_rank(R.slot, r);
        a = max(a, q->rmax);
        b = max(b, q->xmax);
        c = max(c, q->bmax);
      }
      *R.s_eta = backward_error(P, R.sc, R.strict_rlc, R.gam, __longlong_as_double(static_cast<long long>(a)),
                                __longlong_as_double(static_cast<long long>(b)),
                                __longlong_as_double(static_cast<long long>(c)), *phi0);
    }
    cl.sync();  // remote reads done; the error is in every rank's shared memory
    eta = *R.s_eta;
    if (!(eta > R.tol)) break;
  }
  return eta;
}

template <typename real, typename Acc>
__device__ __forceinline__ void solve_body(const Bufs& B, int do_push, int mode, double tol) {
  cg::cluster_group cl = cg::this_cluster();
  const int rank = static_cast<int>(cl.block_rank());
  const int nr = static_cast<int>(cl.num_blocks());
  DevState* S = B.S;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ DevParams sP;                                  // the gap's parameters
  __shared__ __align__(16) unsigned long long s_st[sizeof(DevState) / 8];  // the state before the solve
  __shared__ Seg<Acc> wseg[kRowWarps];
  __shared__ Seg<Acc> slotA[kSolveCtasMax];                 // every rank's totals, pushed here
  __shared__ MaxSlot slotC[kSolveCtasMax];                  // every rank's maxima, pushed here
  __shared__ __align__(8) uint64_t bars[2];
  __shared__ Seg<Acc> s_off;                                // everything before this rank's rows
  __shared__ Acc s_U;
  __shared__ unsigned long long wu[3][32];
  __shared__ double wd[32];
  __shared__ double sc[48];
  __shared__ double s_edge[2];
  __shared__ double slotd, s_eta;
  __shared__ int s_lost;                                    // an exchange of this rank was not completed

  const int tid = static_cast<int>(threadIdx.x), lane = tid & 31, warp = tid >> 5;
  const DevParams* P = &sP;
  const DevState* st = reinterpret_cast<const DevState*>(s_st);
  // --- before the push has finished: parameters and barriers ----------------
  {
    static_assert(sizeof(DevParams) % 8 == 0, "whole words");
    const unsigned long long* src = reinterpret_cast<const unsigned long long*>(B.P);
    unsigned long long* dst = reinterpret_cast<unsigned long long*>(&sP);
    for (int k = tid; k < static_cast<int>(sizeof(DevParams) / 8); k += kSolveThreads) dst[k] = src[k];
  }
  if (tid == 0) s_lost = 0;
  if (nr > 1) {
    if (tid == 0) {
      mbar_init(&bars[0]);
      mbar_init(&bars[1]);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      mbar_expect(&bars[0], static_cast<uint32_t>(nr * sizeof(Seg<Acc>)));
      mbar_expect(&bars[1], static_cast<uint32_t>(nr * sizeof(MaxSlot)));
    }
    cl.sync();  // every rank's barriers are ready before anyone pushes
  } else {
    __syncthreads();
  }
  const int N = P->N;
  const int chunk = (N + nr - 1) / nr;
  const int lo = min(rank * chunk, N);
  const int hi = min(lo + chunk, N);
  const int m = hi - lo;
  const int per = (chunk + kRowThreads - 1) / kRowThreads;  // rows per row thread
  long long* Gv = reinterpret_cast<long long*>(smem);       // G_i of this rank's rows
  double* ph = reinterpret_cast<double*>(smem + align16(8 * chunk));
  double* Ee = ph + chunk;
  double* bb = Ee + chunk;
  double* rr = bb + chunk;                                  // refinement; else the fields in `real`
  real* ef = reinterpret_cast<real*>(rr);
  const bool last_rows = (hi == N && m > 0);                // this rank owns row N-1 (and node N)
  const bool runs_net = (B.net != nullptr && !B.net_in_push && do_push && rank == (nr > 1 ? 1 : 0));
  PredNet* s_net = reinterpret_cast<PredNet*>(smem + solve_rows_bytes(chunk));

  cudaGridDependencySynchronize();  // the push that deposited G has completed
  cudaTriggerProgrammaticLaunchCompletion();
  const int stop = ldcg(&S->status);
  long long G0 = 0;
  if (warp < kRowWarps) {
    for (int k = tid; k < m; k += kRowThreads) Gv[k] = ldcg(&B.G[lo + k]);
  } else if (warp == kCircuitWarp) {
    G0 = ldcg(&B.G[0]);
    const unsigned long long* src = reinterpret_cast<const unsigned long long*>(S);
    for (int k = lane; k < kStateWords; k += 32) s_st[kStateWord0 + k] = ldcg(&src[kStateWord0 + k]);
    __syncwarp();
  }
  if (stop) return;  // the status cannot change before every rank has read it: all ranks agree
  if (runs_net) prefetch_net(B.net, s_net);
  if (per > 1) __syncthreads();

  Seg<Acc> mine, wexcl;
  mine.s1 = 0;
  mine.s2 = 0;
  wexcl = mine;
  const int r0 = min(tid * per, m), r1 = (warp < kRowWarps) ? min(r0 + per, m) : r0;
  unsigned long long bm = 0ULL;
  if (warp < kRowWarps) {
    // --- scan: this thread's rows, then the warp ---------------------------
    for (int q = 0; q < per; ++q) {  // rows past the chunk's end hold no charge
      const int k = tid * per + q;
      if (k < m) {
        const long long g = Gv[k];
        B.Glast[lo + k] = g;
        if (k > 0) B.G[lo + k] = 0;  // a chunk's first row (and G_0) is cleared after the last exchange
        if (lo + k > 0) {            // S'_i = sum_{j=1..i} G_j leaves G_0 out
          mine.s1 += g;
          bm = max(bm, static_cast<unsigned long long>(llabs(g)));
        }
      }
      mine.s2 += mine.s1;
    }
    Seg<Acc> incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const Seg<Acc> y = shfl_up_seg(incl, o);
      if (lane >= o) incl = seg_then(y, incl, o * per);
    }
    wexcl = shfl_up_seg(incl, 1);
    if (lane == 0) {
      wexcl.s1 = 0;
      wexcl.s2 = 0;
    }
    if (lane == 31) wseg[warp] = incl;
  } else if (warp == kCircuitWarp) {
    // circuit row, first part (every rank evaluates the same scalars): the
    // source, the BDF2 history, the circuit solve and the x = 0 row's
    // right-hand side need no scan.
    // Tesla circuit: the new level's loop charges for phi_0 = 0 from the 20
    // history values (one per lane, warp sums)
    double tq[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    if (P->circuit == CP_CIRCUIT_TESLA && do_push) {
      const double h = (lane < 20) ? st->Qt[lane / 5][lane % 5] : 0.0;  // levels n-1..n-4
      const double(*Pm)[20] = (mode == 0) ? P->t_Ps : P->t_Pw;
#pragma unroll
      for (int i = 0; i < 5; ++i) {
        double v = (lane < 20) ? Pm[i][lane] * h : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        tq[i] = v;
      }
    }
    if (lane == 0) {
      const double qw = P->e * P->weight;
      const long long conv = do_push ? st->conv_count : 0LL;
      const double Q1 = st->Qh[0], Q2 = st->Qh[1], Q3 = st->Qh[2];
      // source and BDF2 history of the new level: precomputed by the previous
      // solve except for the first solve of a run
      double Vs, hist;
      if (do_push) {
        Vs = st->nxt_Vs;
        hist = st->nxt_hist;
      } else {
        Vs = B.vs[st->level];
        const double Q4 = st->Qh[3];
        hist = P->L4dt2 * (24.0 * Q1 - 22.0 * Q2 + 8.0 * Q3 - Q4) + P->R2dt * (4.0 * Q1 - Q2);
      }
      const double phi0_prev = st->phi0_last;
      // learned weak scheme: the network's prediction of the plasma's change
      // of C phi_0 over this step, used while its tracked error is within bound
      double J_used = 0.0;
      if (B.net != nullptr && mode == 2) {
        if (B.net_in_push) J_used = st->J_eff;  // the push formed the usable prediction
        else if (st->pred_ready && st->n_eval >= kPredMinEval && st->err_avg <= B.net->bound * st->J_avg)
          J_used = st->J_pred;
      }
      double g = 0.0, Qpart = Q1, gam = 0.0, inv_den = 1.0;
      if (P->circuit == CP_CIRCUIT_SERIES_RLC) {
        if (mode == 0) {  // strict: Q^n = K - g phi_0^n (Eqs. Q4_phi_relation, K_def)
          g = P->g_strict;
          Qpart = g * (Vs + hist);
          gam = P->gam_strict;
          inv_den = P->inv_den_strict;
        } else {
          // weak (Sec. 2.4.3): the circuit alone, its load capacitor starting
          // from phi_0^{n-1}: a21 Q - hist + phi_0^{n-1} + (Q - Q^{n-1} + J)/C = V_s
          Qpart = (Vs + hist + (Q1 - J_used) * P->inv_C - phi0_prev) * P->g_weak;
        }
      } else if (P->circuit == CP_CIRCUIT_TESLA) {
        // Q1 here is the load capacitor's loop charge Q4^{n-1}
        if (!do_push) {  // level 0: the circuit as it rests before t = 0
          Qpart = Q1;
        } else if (mode == 0) {  // strict: Q4^n = K - [T'^{-1}]_44 phi_0^n
          g = P->t_ws[3];
          Qpart = tq[3];
          gam = P->gam_tesla;
          inv_den = P->inv_den_tesla;
        } else {  // weak: loop 4's capacitor voltage phi_0^{n-1} + (Q4 - Q4^{n-1} + J)/C3
          const double s = (Q1 - J_used) * P->inv_C - phi0_prev;
          Qpart = tq[3] + s * P->t_ww[3];
          sc[36] = s;
        }
        for (int i = 0; i < 5; ++i) sc[40 + i] = tq[i];
      }
      const double Qconv = static_cast<double>(conv) * qw;
      const double sigma_prev = st->sigma;
      // x = 0 row: Eq. Poisson_BC2 (strict) / Eq. Poisson_BC3 (weak), with
      // rho_0 dx^2 / (2 eps0) = alpha G_0 / 2 (G_0 is even: boundary doubling)
      const double b0 = P->dx_eps0 * (sigma_prev + (Qconv + Qpart - Q1) * P->inv_A) +
                        P->alpha * static_cast<double>(G0 / 2);
      sc[0] = b0; sc[1] = gam; sc[2] = g; sc[3] = Qpart; sc[4] = Vs; sc[5] = hist;
      sc[6] = Qconv; sc[7] = sigma_prev; sc[8] = Q1; sc[9] = Q2; sc[10] = Q3;
      sc[15] = J_used;
      sc[32] = phi0_prev;
      sc[35] = inv_den;
    }
  } else if (rank == nr - 1 && lane < kSpecies) {
    // the next push processes the slots in use, rounded up to whole vectors;
    // the padding slots are made dead here
    const int s = lane;
    long long na = static_cast<long long>(ldcg(&S->n_alloc[s]));
    if (na > P->cap[s]) na = P->cap[s];
    const long long na4 = (na + 3) & ~3LL;
    real* xs = reinterpret_cast<real*>(ldcg(&S->xi[s]));
    real* us = reinterpret_cast<real*>(ldcg(&S->u[s]));
    for (long long k = na; k < na4; ++k) {
      xs[k] = real(-1);
      us[k] = real(0);
    }
    S->n_alloc[s] = na4;
    S->n_proc[s] = na4;
  }
  if (last_rows && tid == kSolveThreads - 1) {
    B.Glast[N] = ldcg(&B.G[N]);
    B.G[N] = 0;
  }
  __syncthreads();

  // --- the ranks' totals, and the electrode potential ------------------------
  Seg<Acc> bexcl;  // everything of this CTA before this warp
  bexcl.s1 = 0;
  bexcl.s2 = 0;
  if (warp < kRowWarps) {
    for (int q = 0; q < warp; ++q) bexcl = seg_then(bexcl, wseg[q], 32 * per);
  } else if (warp == kCircuitWarp) {
    Seg<Acc> tot = wseg[0];
#pragma unroll
    for (int q = 1; q < kRowWarps; ++q) tot = seg_then(tot, wseg[q], 32 * per);
    // the rows past the chunk's end each added the chunk's total once more
    tot.s2 -= len_times<Acc>(kRowThreads * per - m, tot.s1);
    Seg<Acc> v = tot;
    if (nr > 1) {
      if (lane < nr) {
        const uint32_t dst = remote_addr(&slotA[rank], lane), bar = remote_addr(&bars[0], lane);
        if constexpr (sizeof(Acc) == 8) {
          push16(dst, static_cast<unsigned long long>(tot.s2), static_cast<unsigned long long>(tot.s1), bar);
        } else {
          push16(dst, static_cast<unsigned long long>(tot.s2),
                 static_cast<unsigned long long>(static_cast<unsigned __int128>(tot.s2) >> 64), bar);
          push16(dst + 16, static_cast<unsigned long long>(tot.s1), 0ULL, bar);
        }
      }
      if (__any_sync(0xffffffffu, !mbar_wait(&bars[0], CP_EXCHANGE_POLLS(0))) && lane == 0) {
        s_lost = 1;
        atomicCAS(&S->status, 0, CP_ERR_TIMEOUT);
      }
      v.s1 = 0;
      v.s2 = 0;
      if (lane < nr) v = slotA[lane];
    } else if (lane > 0) {
      v.s1 = 0;
      v.s2 = 0;
    }
    // inclusive scan over the ranks; rank r holds rows_of(r) rows
    int len = max(0, min(chunk, N - lane * chunk));
    if (lane >= nr) len = 0;
    Seg<Acc> ci = v;
#pragma unroll
    for (int o = 1; o < kSolveCtasMax; o <<= 1) {
      const Seg<Acc> y = shfl_up_seg(ci, o);
      const int ly = __shfl_up_sync(0xffffffffu, len, o);
      if (lane >= o) {
        ci = seg_then(y, ci, len);
        len += ly;
      }
    }
    Seg<Acc> ce = shfl_up_seg(ci, 1);
    if (lane == 0) {
      ce.s1 = 0;
      ce.s2 = 0;
    }
    if (lane == rank) s_off = ce;  // everything before this rank
    if (lane == nr - 1) {
      const Acc U = ci.s2;
      const double b0 = sc[0], gam = sc[1], inv_den = sc[35];
      const double phi0 = (static_cast<double>(N) * b0 + P->alpha * acc_to_double(U)) * inv_den;
      const double D0 = b0 - gam * phi0;  // D_0 = x_0 - x_1
      s_U = U;
      sc[11] = D0;
      sc[24] = D0 * P->inv_dx;        // E_0
      sc[25] = P->alpha * P->inv_dx;  // dE_i / dS'_i
    }
    mine = ci;  // kept for the edges: lane `rank` holds everything up to this rank's end
  }
  __syncthreads();
  const double b0 = sc[0], gam = sc[1], D0 = sc[11];
  const double alpha = P->alpha, inv_dx = P->inv_dx;
  const double E0 = sc[24], Ea = sc[25];
  const Acc U = s_U;
  const bool strict_rlc = (P->circuit == CP_CIRCUIT_SERIES_RLC && mode == 0);
  // the level's charge follows Q^n = K - g phi_0^n (g = 0 at a Tesla level 0)
  const bool strict_c = (P->circuit != CP_CIRCUIT_OPEN) && (mode == 0 || (P->circuit == CP_CIRCUIT_TESLA && !do_push));
  // D_i = D_0 + alpha S'_i;  x_i = (N - i) D_0 + alpha (U - P_i);  E_i = D_i / dx
  if (warp < kRowWarps) {
    // everything before this thread's rows: rank, then warp, then lane
    const Seg<Acc> off = seg_then(seg_then(s_off, bexcl, 32 * per * warp), wexcl, lane * per);
    long long Sr = off.s1;  // S'_i, running
    Acc Pex = off.s2;       // P_i = sum_{k<i} S'_k (exclusive)
    for (int k = r0; k < r1; ++k) {
      const int i = lo + k;
      const long long g = (i == 0) ? 0LL : Gv[k];
      Sr += g;
      const double x = fma(static_cast<double>(N - i), D0, alpha * acc_to_double(U - Pex));
      const double e = fma(Ea, static_cast<double>(Sr), E0);
      ph[k] = x;
      Ee[k] = e;
      ef[k] = static_cast<real>(e);
      bb[k] = (i == 0) ? b0 : -alpha * static_cast<double>(g);
      Pex += Sr;
    }
  } else if (warp == kCircuitWarp) {
    // The neighbouring chunks' edge values follow from the exact prefixes with
    // the same arithmetic their owners use, so no exchange is needed:
    // x_{lo-1} needs P_{lo-1} = P_lo - S'_{lo-1}; x_hi needs P_hi.
    Seg<Acc> no;  // everything up to and including this rank's rows
    if (lane == rank) slotA[rank] = mine;
    __syncwarp();
    no = slotA[rank];
    const Seg<Acc> ro = s_off;
    const int i = (lane == 0) ? lo - 1 : (lane == 1) ? hi : 0;  // lanes 0-2: x_{lo-1}, x_hi, x_0
    const Acc Pi = (lane == 0) ? ro.s2 - static_cast<Acc>(ro.s1) : (lane == 1) ? no.s2 : Acc(0);
    const double x = fma(static_cast<double>(N - i), D0, alpha * acc_to_double(U - Pi));
    if (lane == 0) sc[26] = (lo > 0) ? x : 0.0;
    if (lane == 1) sc[27] = (hi < N) ? x : 0.0;
    if (lane == 2) sc[29] = x;
  }
  __syncthreads();
  const double prev_phi = sc[26], next_phi = sc[27], phi0 = sc[29];
  double phi0_fin = phi0;
  int status = 0;  // of the committed values (commit warp of rank 0)
  real* Etab = static_cast<real*>(B.Etab);
  if (warp < kRowWarps) {
    // outputs
    unsigned long long rm = 0ULL, xm = 0ULL;
    for (int k = tid; k < (s_lost ? 0 : m); k += kRowThreads) {
      const int i = lo + k;
      const double x = ph[k];
      const double ri = row_residual(ph, bb[k], k, i, m, gam, prev_phi, next_phi);
      rm = max(rm, abs_bits(ri));
      xm = max(xm, abs_bits(x));
      B.E64[i] = Ee[k];
      B.phi[i] = x;
      const real e0 = ef[k];
      Etab[i + 1] = e0;
      if (i == 0) Etab[0] = e0;
      if (i == N - 1) Etab[N + 1] = e0;
    }
    rm = warp_max_u64(rm);
    xm = warp_max_u64(xm);
    bm = warp_max_u64(bm);
    if (lane == 0) {
      wu[0][warp] = rm;
      wu[1][warp] = xm;
      wu[2][warp] = bm;
    }
  } else if (warp == kCommitWarp) {
    if (last_rows && lane == 31) B.phi[N] = 0.0;
    if (rank == 0 && !s_lost)
      status = commit_level(S, B.hist, B.hist_rows, B.vs, P, st, sc, do_push, mode, strict_c, phi0, 0.0);
  }
  if (warp != kCommitWarp)  // the commit goes on beside the error's exchange
    asm volatile("bar.sync 1, %0;" ::"n"(kRowThreads + 32) : "memory");
  // --- backward error over the cluster ----------------------------------------
  if (warp == kCircuitWarp) {
    MaxSlot q;
    q.rmax = warp_max_u64(lane < kRowWarps ? wu[0][lane] : 0ULL);
    q.xmax = warp_max_u64(lane < kRowWarps ? wu[1][lane] : 0ULL);
    q.bmax = warp_max_u64(lane < kRowWarps ? wu[2][lane] : 0ULL);
    if (nr > 1) {
      if (lane < nr) {
        const uint32_t dst = remote_addr(&slotC[rank], lane), bar = remote_addr(&bars[1], lane);
        push16(dst, q.rmax, q.xmax, bar);
        push16(dst + 16, q.bmax, s_lost ? 1ULL : 0ULL, bar);
      }
      const bool out = __any_sync(0xffffffffu, !mbar_wait(&bars[1], CP_EXCHANGE_POLLS(1)));
      const bool told = __any_sync(0xffffffffu, lane < nr && slotC[lane].lost != 0ULL);
      if (lane == 0 && (out || told)) s_lost = 1;
      if (lane == 0 && out) atomicCAS(&S->status, 0, CP_ERR_TIMEOUT);
      q.rmax = warp_max_u64(lane < nr ? slotC[lane].rmax : 0ULL);
      q.xmax = warp_max_u64(lane < nr ? slotC[lane].xmax : 0ULL);
      q.bmax = warp_max_u64(lane < nr ? slotC[lane].bmax : 0ULL);
    }
    if (lane == 0) {
      // max |b_i| = max(alpha max |G_i| over rows >= 1, |b_0|)
      const double bmd = fmax(alpha * static_cast<double>(q.bmax), fabs(b0));
      s_eta = backward_error(P, sc, strict_rlc, gam, __longlong_as_double(static_cast<long long>(q.rmax)),
                             __longlong_as_double(static_cast<long long>(q.xmax)), bmd, phi0);
      if (m > 0) B.G[lo] = 0;  // every rank has read it
    }
  }
  __syncthreads();
  if (s_lost) {
    leave_lost(bars);
    return;
  }
  double eta = s_eta;
  if (eta > tol) {  // the same on every rank that is not lost
    if (nr > 1 && any_lost(&s_lost)) return;
    Refine R;
    R.ph = ph; R.Ee = Ee; R.bb = bb; R.rr = rr;
    R.sc = sc; R.wd = wd; R.slotd = &slotd; R.edge = s_edge;
    R.wu = wu; R.slot = &slotC[0]; R.s_eta = &s_eta;
    R.lo = lo; R.hi = hi; R.m = m; R.N = N;
    R.gam = gam; R.inv_dx = inv_dx; R.tol = tol;
    R.strict_rlc = strict_rlc;
    eta = refine(R, P, prev_phi, next_phi, &phi0_fin);
    for (int k = tid; k < m; k += kSolveThreads) {
      const int i = lo + k;
      B.E64[i] = Ee[k];
      B.phi[i] = ph[k];
      const real e0 = static_cast<real>(Ee[k]);
      Etab[i + 1] = e0;
      if (i == 0) Etab[0] = e0;
      if (i == N - 1) Etab[N + 1] = e0;
    }
    if (rank == 0 && warp == kCommitWarp)
      status = commit_level(S, B.hist, B.hist_rows, B.vs, P, st, sc, do_push, mode, strict_c, phi0_fin, eta);
  }
  if (rank == 0 && tid == 32 * kCommitWarp) {
    const int64_t level = st->level + (do_push ? 1 : 0);
    S->cur.residual = eta;
    if (level < B.hist_rows) B.hist[level].residual = eta;
    if (status == 0 && eta > tol) status = CP_ERR_RESIDUAL;
    if (status != 0) atomicCAS(&S->status, 0, status);
  }
  if (runs_net) predictor_update(P, S, st, s_net, sc, strict_c, phi0_fin);
}

// Registers: one CTA per SM here, 168 a thread without spills (96 is the
// compiler's own choice: graph step at 1531 cells and 1e6 particles 15.24 us
// instead of 15.09, at 4096 cells and 3.3e5 16.2 instead of 15.95); the
// ensemble's clusters share the SMs, two CTAs each (step of 160 instances 238.5
// us, 247.6 with one CTA per SM).
template <typename real, typename Acc>
__global__ void __launch_bounds__(kSolveThreads, 1) k_solve(Bufs B, int do_push, int mode, double tol) {
  solve_body<real, Acc>(B, do_push, mode, tol);
}

// Ensemble: cluster i solves instance i.
template <typename real, typename Acc>
__global__ void __launch_bounds__(kSolveThreads, 2)
k_solve_ens(const Bufs* __restrict__ Ball, int do_push, int mode, double tol) {
  const Bufs B = Ball[blockIdx.x / cg::this_cluster().num_blocks()];
  solve_body<real, Acc>(B, do_push, mode, tol);
}

// ---------------------------------------------------------------------------
// Host-side launchers
// ---------------------------------------------------------------------------
static const void* solve_fn(int precision, bool wide) {
  if (precision == CP_FP32)
    return wide ? reinterpret_cast<const void*>(k_solve<float, __int128>)
                : reinterpret_cast<const void*>(k_solve<float, long long>);
  return wide ? reinterpret_cast<const void*>(k_solve<double, __int128>)
              : reinterpret_cast<const void*>(k_solve<double, long long>);
}

static const void* solve_ens_fn(int precision, bool wide) {
  if (precision == CP_FP32)
    return wide ? reinterpret_cast<const void*>(k_solve_ens<float, __int128>)
                : reinterpret_cast<const void*>(k_solve_ens<float, long long>);
  return wide ? reinterpret_cast<const void*>(k_solve_ens<double, __int128>)
              : reinterpret_cast<const void*>(k_solve_ens<double, long long>);
}

// Whether the prefix of prefixes of a gap of N cells whose stores hold
// cap[] macroparticles needs 128 bits (per_particle: charge units of one).
bool solve_wide(int N, const int64_t cap[kSpecies], double per_particle) {
  const double most = static_cast<double>(std::max(cap[CP_IONS], cap[CP_ELECTRONS] + cap[CP_SECONDARIES]));
  const double rows = static_cast<double>(N) + kSolveCtasMax * kRowThreads;  // padding rows included
  return !(per_particle * most * rows < 4.611686018427387904e18);            // 2^62
}

// Every context sharing a kernel may ask for another size, so each kernel's
// limit is the largest the device allows.
static cudaError_t allow_all_smem(const void* fn) {
  int dev = 0, most = 0;
  cudaFuncAttributes at;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&at, fn);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              most - static_cast<int>(at.sharedSizeBytes));
}

cudaError_t solve_configure(int precision, bool wide) { return allow_all_smem(solve_fn(precision, wide)); }
cudaError_t solve_ens_configure(int precision, bool wide) {
  return allow_all_smem(solve_ens_fn(precision, wide));
}

size_t solve_smem_bytes(int N, int ctas, bool net) {
  return solve_rows_bytes((N + ctas - 1) / ctas) + (net ? kPredNetBytes : 0);
}

// CTAs of a solve of N rows: one per 256 rows, at most 16 (where the device
// runs non-portable clusters, else 8).
cudaError_t solve_cluster_size(int precision, bool wide, int N, int* ctas) {
  int want = 1;
  while (want < kSolveCtasMax && want * kRowThreads < N) want *= 2;
  *ctas = std::min(want, kSolveCtas);
  if (want <= kSolveCtas) return cudaSuccess;
  const void* fn = solve_fn(precision, wide);
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
    cudaGetLastError();
    return cudaSuccess;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(want, 1, 1);
  cfg.blockDim = dim3(kSolveThreads, 1, 1);
  cfg.dynamicSmemBytes = solve_smem_bytes(N, want, true);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = want;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg) == cudaSuccess && clusters >= 1) *ctas = want;
  cudaGetLastError();
  return cudaSuccess;
}

// CTAs per instance of an ensemble's solve.  One CTA per instance leaves the
// FP64 work of the few largest gaps on one SM each, more CTAs cost the
// exchange: 4 while the clusters fit the device in about two waves, then 2,
// then 1.
int solve_ens_cluster_size(int n_max, int E, int sms) {
  int nr = 1;
  while (nr < 4 && nr * kRowThreads < n_max && 2 * nr * E <= 8 * sms) nr *= 2;
  return nr;
}

static cudaLaunchConfig_t solve_config(int grid, int ctas, size_t smem, cudaStream_t st, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3(kSolveThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = ctas;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cfg;
}

cudaError_t solve_ens_launch(int precision, bool wide, const Bufs* Ball, int n_inst, int ctas, size_t smem,
                             cudaStream_t st, int do_push, int mode, double tol) {
  cudaLaunchAttribute attr[2];
  const cudaLaunchConfig_t cfg = solve_config(n_inst * ctas, ctas, smem, st, attr);
  void* args[] = {&Ball, &do_push, &mode, &tol};
  return cudaLaunchKernelExC(&cfg, solve_ens_fn(precision, wide), args);
}

cudaError_t solve_launch(int precision, bool wide, const Bufs& B, int ctas, size_t smem, cudaStream_t st,
                         int do_push, int mode, double tol) {
  cudaLaunchAttribute attr[2];
  const cudaLaunchConfig_t cfg = solve_config(ctas, ctas, smem, st, attr);
  void* args[] = {const_cast<Bufs*>(&B), &do_push, &mode, &tol};
  return cudaLaunchKernelExC(&cfg, solve_fn(precision, wide), args);
}

}  // namespace cpk
