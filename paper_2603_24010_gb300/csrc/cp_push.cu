// cp_push.cu -- the removal of absorbed particles and small set-up kernels of
// the 1D gap (its push is cp_push_async.cu, its solve cp_solve.cu).
//
// k_compact packs the live particles of every species into the spare
//   buffers every few steps (dead slots are skipped by the push until then).
#include "cp_push.cuh"

namespace cpk {
// ---------------------------------------------------------------------------
// Removal of absorbed particles: live slots are packed into the spare buffers
// (interleaved, see pack_block) and the buffers are swapped by the last CTA.
// Physics does not depend on particle order.
// ---------------------------------------------------------------------------
template <typename real>
__global__ void __launch_bounds__(kThreads) k_compact(Bufs B) {
  DevState* S = B.S;
  __shared__ PackShared<real> sh;
  __shared__ unsigned int s_ticket;
  __shared__ int s_stop;
  if (threadIdx.x == 0) s_stop = (ldcg(&S->status) != 0);
  __syncthreads();
  if (s_stop) return;
  for (int s = 0; s < kSpecies; ++s) {
    const real* xs = reinterpret_cast<const real*>(S->xi[s]);
    const real* us = reinterpret_cast<const real*>(S->u[s]);
    real* xd = reinterpret_cast<real*>(S->xi_alt[s]);
    real* ud = reinterpret_cast<real*>(S->u_alt[s]);
    const int64_t n = S->n_proc[s], chunks = pack_chunks(n);
    for (int64_t t = blockIdx.x; t < chunks; t += gridDim.x)
      pack_block<real>(sh, xs, us, s == CP_IONS ? S->id : nullptr, n, chunks, t, xd, ud, S->id_alt, &S->compact_n[s]);
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_ticket = atomicAdd(&S->compact_done, 1u);
  __syncthreads();
  if (s_ticket != gridDim.x - 1) return;
  __threadfence();
  if (threadIdx.x < kSpecies) {
    const int s = threadIdx.x;
    const long long cnt = static_cast<long long>(ldcg(&S->compact_n[s]));
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
  if (threadIdx.x == 0) {
    uint32_t* t2 = S->id;
    S->id = S->id_alt;
    S->id_alt = t2;
    S->compact_done = 0u;
  }
}

// polarity V_s(t_n) for n = 0..rows-1, once at set-up (the source of Sec. 2.1)
__global__ void k_source_table(const DevParams* P, double* vs, int64_t rows) {
  for (int64_t n = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; n < rows;
       n += static_cast<int64_t>(gridDim.x) * blockDim.x)
    vs[n] = P->polarity * source_voltage(P, static_cast<double>(n) * P->dt);
}

cudaError_t source_table_launch(const DevParams* P, double* vs, int64_t rows, cudaStream_t st) {
  const int grid = static_cast<int>((rows + 255) / 256 < 1024 ? (rows + 255) / 256 : 1024);
  k_source_table<<<grid, 256, 0, st>>>(P, vs, rows);
  return cudaGetLastError();
}

// Initial plasma: n co-located electron/ion pairs at temperature T (the
// paper's runs start from a loaded plasma, Sec. 3.1).  Pair k draws
// Philox4x64-10 counter (k, 0, 0, 0) under key (seed, load tag): xi = N u0
// (uniform in the gap), and the Box-Muller pair of u1, u2 gives the two
// velocities, z_e th_e and z_i th_i (th = sqrt(e T / m) dt / dx, a 1D
// Maxwellian).  Positions are rounded to the store's precision and kept
// inside (0, N); ion ids are k.
template <typename real>
__global__ void k_load_pairs(real* xe, real* ue, real* xo, real* uo, uint32_t* id, int64_t n, int N,
                             double th_e, double th_i, uint64_t seed) {
  const double pi = 3.14159265358979323846;
  for (int64_t k = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; k < n;
       k += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const U64x4 w = philox4x64_10(static_cast<uint64_t>(k), 0, 0, 0, seed, kTagLoad);
    const real x = nudge_inside<real>(__dmul_rn(static_cast<double>(N), u01(w.w[0])), N);
    const double r = sqrt(-2.0 * log(u01(w.w[1])));
    const double a = __dmul_rn(2.0 * pi, u01(w.w[2]));
    xe[k] = x;
    xo[k] = x;
    ue[k] = static_cast<real>(__dmul_rn(th_e, __dmul_rn(r, cos(a))));
    uo[k] = static_cast<real>(__dmul_rn(th_i, __dmul_rn(r, sin(a))));
    id[k] = static_cast<uint32_t>(k);
  }
}

cudaError_t load_pairs_launch(int precision, void* xe, void* ue, void* xo, void* uo, uint32_t* id,
                              int64_t n, int N, double th_e, double th_i, uint64_t seed, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int grid = static_cast<int>((n + 255) / 256 < 8192 ? (n + 255) / 256 : 8192);
  if (precision == CP_FP32)
    k_load_pairs<float><<<grid, 256, 0, st>>>(static_cast<float*>(xe), static_cast<float*>(ue),
                                              static_cast<float*>(xo), static_cast<float*>(uo), id, n, N,
                                              th_e, th_i, seed);
  else
    k_load_pairs<double><<<grid, 256, 0, st>>>(static_cast<double*>(xe), static_cast<double*>(ue),
                                               static_cast<double*>(xo), static_cast<double*>(uo), id, n,
                                               N, th_e, th_i, seed);
  return cudaGetLastError();
}

template <typename real>
__global__ void k_fill(real* p, int64_t n, real v) {
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    p[i] = v;
}

// ---------------------------------------------------------------------------
// Host-side launchers (internal C++ interface used by cp_api.cu)
// ---------------------------------------------------------------------------
cudaError_t compact_launch(int precision, const Bufs& B, int grid, cudaStream_t st) {
  if (precision == CP_FP32)
    k_compact<float><<<grid, kThreads, 0, st>>>(B);
  else
    k_compact<double><<<grid, kThreads, 0, st>>>(B);
  return cudaGetLastError();
}

cudaError_t fill_launch(int precision, void* p, int64_t n, double v, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int grid = static_cast<int>((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096);
  if (precision == CP_FP32)
    k_fill<float><<<grid, 256, 0, st>>>(reinterpret_cast<float*>(p), n, static_cast<float>(v));
  else
    k_fill<double><<<grid, 256, 0, st>>>(reinterpret_cast<double*>(p), n, v);
  return cudaGetLastError();
}

}  // namespace cpk
