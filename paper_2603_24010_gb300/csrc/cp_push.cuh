// cp_push.cuh -- what the particle pushes of the single gap (cp_push_async.cu)
// and of the ensemble (cp_batch.cu) share: asynchronous copies of particle
// vectors, the gather from a shared-memory field table and the fixed-point
// deposit into 32-bit node sums.
#pragma once

#include "cp_common.cuh"

namespace cpk {

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

// a thread's particles: from a ring slot, from and to global memory
__device__ __forceinline__ void get_vec(const float4* d, float (&v)[4]) {
  const float4 a = *d;
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}
__device__ __forceinline__ void get_vec(const float4* d, double (&v)[2]) {
  const double2 a = *reinterpret_cast<const double2*>(d);
  v[0] = a.x; v[1] = a.y;
}
__device__ __forceinline__ void put_vec(float* p, const float (&v)[4]) { store4(p, v); }
__device__ __forceinline__ void put_vec(double* p, const double (&v)[2]) {
  __stcs(reinterpret_cast<double2*>(p), make_double2(v[0], v[1]));
}

// 0 < x < N.  FP64: on the bit patterns, which order like the values (GB300's
// FP64 pipe takes 16 cycles for a warp's comparison).
__device__ __forceinline__ bool inside(float x, float N) { return x > 0.0f && x < N; }
__device__ __forceinline__ bool inside(double x, double N) {
  return static_cast<unsigned long long>(__double_as_longlong(x)) - 1ULL <
         static_cast<unsigned long long>(__double_as_longlong(N)) - 1ULL;
}

// running maximum of |u| as a bit pattern, and its FP32 value's bits
__device__ __forceinline__ void max_abs(unsigned int& m, float u) { m = max(m, __float_as_uint(fabsf(u))); }
__device__ __forceinline__ void max_abs(unsigned long long& m, double u) {
  m = max(m, static_cast<unsigned long long>(__double_as_longlong(u)) & 0x7FFFFFFFFFFFFFFFULL);
}
__device__ __forceinline__ unsigned int float_bits(unsigned int m) { return m; }
__device__ __forceinline__ unsigned int float_bits(unsigned long long m) {
  return __float_as_uint(static_cast<float>(__longlong_as_double(static_cast<long long>(m))));
}
template <typename real>
struct Bits;
template <>
struct Bits<float> {
  using type = unsigned int;
};
template <>
struct Bits<double> {
  using type = unsigned long long;
};

template <typename real>
__device__ __forceinline__ real kick(const DevParams* P, bool half, int s) {
  if constexpr (sizeof(real) == 4) return P->kap_f[half ? 0 : 1][s];
  else return P->kap_d[half ? 0 : 1][s];
}

// v units of charge on node k of an int64 grid (end nodes doubled)
__device__ __forceinline__ void add_global(long long* G, int k, int N, long long v) {
  if (v == 0) return;
  if (k == 0 || k == N) v <<= 1;
  atomicAdd(reinterpret_cast<unsigned long long*>(&G[k]), static_cast<unsigned long long>(v));
}

// Fixed-point position of a particle inside the gap: cell i in the high and
// W1 = floor(2^16 (x - i)) in the low 16 bits.  x 2^16 is exact (power-of-two
// scaling) and below 2^32 (N < 2^16), so one truncating conversion gives both.
__device__ __forceinline__ unsigned int fix_pos(float x) {
  float f;
  const int i = floor_split(x, &f);
  return (static_cast<unsigned int>(i) << 16) | frac16(f);
}
// FP64: the mantissa shifted down (the integer pipe; 0 < x < 2^16)
__device__ __forceinline__ unsigned int fix_pos(double x) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
  const int sh = 1023 + 36 - static_cast<int>(b >> 52);  // 52 - 16 - exponent, at least 21
  return static_cast<unsigned int>(((b & 0xFFFFFFFFFFFFFULL) | 0x10000000000000ULL) >> min(sh, 63));
}

// j = floor(x - 1/2) and t = (x - 1/2) - j of a position inside the gap
__device__ __forceinline__ int half_cell(float x, float* t) {
  return floor_split(x - 0.5f, t);
}
// FP64: j = floor((floor(2 x) - 1) / 2) from the mantissa, and as a double
// from the bits of 2^52 + 2^51 + j (two additions instead of a floor and two
// conversions on the FP64 pipe)
__device__ __forceinline__ int half_cell(double x, double* t) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
  const int sh = 1023 + 51 - static_cast<int>(b >> 52);  // 52 - 1 - exponent, at least 36
  const int h = static_cast<int>(((b & 0xFFFFFFFFFFFFFULL) | 0x10000000000000ULL) >> min(sh, 63));
  const int j = (h - 1) >> 1;
  const double jf = __longlong_as_double(0x4338000000000000LL + j) - 6755399441055744.0;
  *t = (x - 0.5) - jf;
  return j;
}

// CIC deposit into the node sums: node i gets sign (2^16 - W1), node i+1
// sign W1 (sign +1 or -1).
__device__ __forceinline__ void deposit_nodes(unsigned int* nd, unsigned int F, int sign) {
  const unsigned int i = F >> 16;
  const unsigned int w1 = (F & 0xFFFFu) * static_cast<unsigned int>(sign);
  atomicAdd(&nd[i], 65536u * static_cast<unsigned int>(sign) - w1);
  atomicAdd(&nd[i + 1], w1);
}

// The field table of a level into shared memory (N + 2 values, whole 16-byte
// vectors): three vectors per thread in flight together (a fourth costs the
// push's loop registers), one L2 round trip for N <= 6142 FP32 cells at 512
// threads.  A table of E alone instead of pairs: a step at 4096 cells and 3.3e5
// particles 16.7 -> 16.3 us.
template <typename real, int THREADS>
__device__ __forceinline__ void load_table(real* Et, const void* Etab, int N) {
  const int nv = (static_cast<int>(sizeof(real)) * (N + 2) + 15) / 16;
  const float4* src = static_cast<const float4*>(Etab);
  float4* dst = reinterpret_cast<float4*>(Et);
  for (int k0 = threadIdx.x; k0 < nv; k0 += 3 * THREADS) {
    float4 e[3];
#pragma unroll
    for (int q = 0; q < 3; ++q)
      if (k0 + q * THREADS < nv) e[q] = __ldcg(src + k0 + q * THREADS);
#pragma unroll
    for (int q = 0; q < 3; ++q)
      if (k0 + q * THREADS < nv) dst[k0 + q * THREADS] = e[q];
  }
}

// gather from the padded field table Et[k] = E_{k-1/2} (k = 1..N), Et[0] =
// E_{1/2}, Et[N+1] = E_{N-1/2}: the pair (E_{j+1/2}, slope) of the pair table
// is formed here with the same subtraction, and the repeated end values give
// the constant extension (slope +0) for j = -1 and j = N-1
template <typename real>
__device__ __forceinline__ real gather_tab(const real* Et, real x) {
  real t;
  const int j = half_cell(x, &t);
  const real e0 = Et[j + 1];
  return fma(t, Et[j + 2] - e0, e0);
}

// Entry speed [cells/step] of a beam ion from its second draw: in FP32 the
// FP32 pushes' form, in FP64 the definition's order of operations.
template <typename real>
__device__ __forceinline__ double beam_speed(const DevParams* P, double u) {
  if constexpr (sizeof(real) == 4) {
    return beam_speed_fp32(P, u);
  } else {
    const double Eb = (P->beam_mode == 0)
                          ? P->beam_E_eV
                          : __dadd_rn(P->beam_Emin_eV, __dmul_rn(__dsub_rn(P->beam_Emax_eV, P->beam_Emin_eV), u));
    const double v = sqrt(2.0 * Eb * P->e / P->m_i);
    return v * P->dt / P->dx;
  }
}

// --- removal of absorbed particles ------------------------------------------------
// A block packs up to 2048 slots of a store at a time into the spare buffers:
// warp w takes chunk `t` of 128 slots of region w (the store cut in 16 regions of
// `region` slots), and the live ones leave interleaved, one of each warp in turn.
//
// The interleaving is for the pushes that follow.  Ions of one step's beam lie in
// consecutive slots and, with one energy, in the same one or two cells, where a
// warp's node-sum atomics go to the same addresses; dealt out, neighbouring lanes
// hold ions of 16 distant regions.  Impacts spread over the CTAs likewise.  The
// outputs go through shared memory and leave as whole runs.
// Bound: the HBM stream.  3.1e7 particles of one beam energy: removal 330 -> 155
// us, step in a graph 109 -> 98.6; 1.5e7: 148 -> 77, 51.2 -> 47.3; an ensemble of
// 7.0e7: 530 -> 370, 264 -> 242 (packed warp by warp in place before, with an
// atomic per warp and four partial stores).
constexpr int kPackWarps = kThreads / 32;
constexpr int kPackChunk = 32 * kPerThread;
template <typename real>
struct PackShared {
  static constexpr int kSlots = kThreads * kPerThread;
  real x[kSlots + kSlots / 32], u[kSlots + kSlots / 32];
  uint32_t id[kSlots + kSlots / 32];
  int before[kPackChunk];         // live slots of all warps with a rank below r
  unsigned int longer[kPackChunk];  // warps with more than r live slots
  int count[kPackWarps];
  unsigned long long base;
};

// slots per region of n, and chunks per region
__host__ __device__ inline int64_t pack_chunks(int64_t n) {
  return (n + static_cast<int64_t>(kPackWarps) * kPackChunk - 1) / (static_cast<int64_t>(kPackWarps) * kPackChunk);
}

template <typename real>
__device__ __forceinline__ void pack_block(PackShared<real>& sh, const real* __restrict__ xs, const real* __restrict__ us,
                                           const uint32_t* __restrict__ is, int64_t n, int64_t chunks, int64_t t,
                                           real* __restrict__ xd, real* __restrict__ ud, uint32_t* __restrict__ id_d,
                                           unsigned long long* packed) {
  const int tid = static_cast<int>(threadIdx.x), w = tid >> 5;
  const int64_t base = (w * chunks + t) * kPackChunk + static_cast<int64_t>(lane_id()) * kPerThread;
  real xv[kPerThread], uv[kPerThread];
  uint32_t iv[kPerThread] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int q = 0; q < kPerThread; ++q) {
    xv[q] = real(-1);
    uv[q] = real(0);
  }
  if (base < n) {
    load4(xs + base, xv);
    load4(us + base, uv);
    if (is) {
      const uint4 a = __ldcs(reinterpret_cast<const uint4*>(is + base));
      iv[0] = a.x; iv[1] = a.y; iv[2] = a.z; iv[3] = a.w;
    }
  }
  int c = 0;
#pragma unroll
  for (int q = 0; q < kPerThread; ++q) c += (xv[q] > real(0)) ? 1 : 0;
  const int incl = warp_incl_scan(c);
  if (lane_id() == 31) sh.count[w] = incl;
  __syncthreads();  // also: the block before has left the buffers
  if (tid < kPackChunk) {
    int b = 0;
    unsigned int m = 0u;
#pragma unroll
    for (int q = 0; q < kPackWarps; ++q) {
      const int cq = sh.count[q];
      b += min(cq, tid);
      m |= (cq > tid ? 1u : 0u) << q;
    }
    sh.before[tid] = b;
    sh.longer[tid] = m;
  } else if (tid == kThreads - 1) {
    int total = 0;
#pragma unroll
    for (int q = 0; q < kPackWarps; ++q) total += sh.count[q];
    sh.base = total ? atomicAdd(packed, static_cast<unsigned long long>(total)) : 0ULL;
  }
  __syncthreads();
  int r = incl - c;
#pragma unroll
  for (int q = 0; q < kPerThread; ++q) {
    if (xv[q] > real(0)) {
      const int o = sh.before[r] + __popc(sh.longer[r] & ((1u << w) - 1u));
      ++r;
      const int k = o + (o >> 5);
      sh.x[k] = xv[q];
      sh.u[k] = uv[q];
      if (is) sh.id[k] = iv[q];
    }
  }
  int total = 0;
#pragma unroll
  for (int q = 0; q < kPackWarps; ++q) total += sh.count[q];
  const unsigned long long o0 = sh.base;
  __syncthreads();
  for (int o = tid; o < total; o += kThreads) {
    const int k = o + (o >> 5);
    xd[o0 + o] = sh.x[k];
    ud[o0 + o] = sh.u[k];
    if (is) id_d[o0 + o] = sh.id[k];
  }
}

}  // namespace cpk
