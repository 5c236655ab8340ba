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

}  // namespace cpk
