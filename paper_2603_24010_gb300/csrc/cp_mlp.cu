// cp_mlp.cu -- the weak-coupling predictor network: packing of an installed
// network, training samples from the diagnostics history, and the training
// kernels (initialisation, scales, forward, loss + gradient, Adam).
//
// The network (40 -> 64 -> 64 -> 64 -> 2, GELU) trains in FP32, which the
// tensor cores do not offer (their FP32 input form keeps 10 mantissa bits).
// The batch kernel runs on the FP32 pipe with the network in shared memory,
// up to 64 samples per tile and per-CTA gradient sums kept in registers; a
// second kernel adds the per-CTA partial sums in a fixed order, so the
// gradient is bit-reproducible.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "cp_mlp.cuh"

namespace cpk {

// Parameter offsets in the FP32 master array (W[out][in] row-major).
constexpr int kOffW1 = 0;
constexpr int kOffB1 = kOffW1 + kHid * kPredIn;  // 2560
constexpr int kOffW2 = kOffB1 + kHid;            // 2624
constexpr int kOffB2 = kOffW2 + kHid * kHid;     // 6720
constexpr int kOffW3 = kOffB2 + kHid;            // 6784
constexpr int kOffB3 = kOffW3 + kHid * kHid;     // 10880
constexpr int kOffW4 = kOffB3 + kHid;            // 10944
constexpr int kOffB4 = kOffW4 + kPredOut * kHid; // 11072
constexpr int kNParam = kOffB4 + kPredOut;       // 11074
static_assert(kNParam == CP_MLP_NPARAM, "parameter layout");

constexpr int kTrainThreads = 256;
constexpr int kTileS = 64;         // most samples per tile
constexpr int kTrainMaxCtas = 256; // rows of the partial-sum scratch
constexpr int kWorkRow = kNParam + 1;  // per-CTA gradient + loss

__device__ __forceinline__ float bf16_round(float w) {
  return __bfloat162float(__float2bfloat16_rn(w));
}
__device__ __forceinline__ uint16_t bf16_bits(float w) {
  return __bfloat16_as_ushort(__float2bfloat16_rn(w));
}

// ---------------------------------------------------------------------------
// Installed network: BF16 weight bits and FP32 biases.
// ---------------------------------------------------------------------------
__global__ void k_pack_predictor(const float* __restrict__ p, PredNet* net) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < kNParam; i += gridDim.x * blockDim.x) {
    const float w = p[i];
    if (i < kOffB1) net->W1[i - kOffW1] = bf16_bits(w);
    else if (i < kOffW2) net->b1[i - kOffB1] = w;
    else if (i < kOffB2) net->W2[i - kOffW2] = bf16_bits(w);
    else if (i < kOffW3) net->b2[i - kOffB2] = w;
    else if (i < kOffB3) net->W3[i - kOffW3] = bf16_bits(w);
    else if (i < kOffW4) net->b3[i - kOffB3] = w;
    else if (i < kOffB4) net->W4[i - kOffW4] = bf16_bits(w);
    else net->b4[i - kOffB4] = w;
  }
}

// ---------------------------------------------------------------------------
// Training samples from the history rows (one thread per sample).
// ---------------------------------------------------------------------------
__global__ void k_samples(const DevParams* __restrict__ P, const cp_diag* __restrict__ h,
                          int64_t first, int64_t n, float* __restrict__ X, float* __restrict__ Y) {
  const int64_t k = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const int64_t L = first + k;  // newest level of the window
  float* x = X + k * kPredIn;
  for (int j = 0; j < kPredWindow; ++j) {
    const int64_t m = L - (kPredWindow - 1) + j;
    const cp_diag& r = h[m];
    const cp_diag& q = h[m - 1];
    x[j * kPredFeat + 0] = static_cast<float>(r.Q_conv);
    x[j * kPredFeat + 1] = static_cast<float>(r.V_gap - q.V_gap);
    x[j * kPredFeat + 2] = static_cast<float>(r.Q_surf - q.Q_surf);
    x[j * kPredFeat + 3] = static_cast<float>(static_cast<double>(r.emitted[0]));
    x[j * kPredFeat + 4] = static_cast<float>(r.ion_energy_eV);
  }
  const cp_diag& a = h[L + 1];
  const cp_diag& b = h[L];
  const double J = P->C * (a.V_gap - b.V_gap) - (a.Q_circ - b.Q_circ);
  Y[2 * k + 0] = static_cast<float>(a.Q_conv);
  Y[2 * k + 1] = static_cast<float>(J);
}

// ---------------------------------------------------------------------------
// Initialisation: He-uniform weights from Philox draws, zero biases.
// ---------------------------------------------------------------------------
__global__ void k_mlp_init(float* __restrict__ p, uint64_t seed) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < kNParam; i += gridDim.x * blockDim.x) {
    int fan_in = 0;
    if (i < kOffB1) fan_in = kPredIn;
    else if (i >= kOffW2 && i < kOffB2) fan_in = kHid;
    else if (i >= kOffW3 && i < kOffB3) fan_in = kHid;
    else if (i >= kOffW4 && i < kOffB4) fan_in = kHid;
    if (fan_in == 0) {
      p[i] = 0.0f;
      continue;
    }
    const U64x4 r = philox4x64_10(static_cast<uint64_t>(i), 0, 0, 0, seed, kTagInit);
    const double u = u01(r.w[0]);
    p[i] = static_cast<float>((2.0 * u - 1.0) * sqrt(6.0 / fan_in));
  }
}

// ---------------------------------------------------------------------------
// Scales: root mean squares of the five features and two targets (one
// block, fixed summation order).
// ---------------------------------------------------------------------------
__device__ double g_scale_sums[kPredFeat + kPredOut];

__global__ void __launch_bounds__(1024) k_mlp_scales(const float* __restrict__ X,
                                                     const float* __restrict__ Y, int64_t n) {
  __shared__ double part[kPredFeat + kPredOut][32];
  double acc[kPredFeat + kPredOut];
  for (int f = 0; f < kPredFeat + kPredOut; ++f) acc[f] = 0.0;
  for (int64_t i = threadIdx.x; i < n * kPredIn; i += blockDim.x) {
    const double v = X[i];
    acc[(i % kPredIn) % kPredFeat] += v * v;
  }
  for (int64_t i = threadIdx.x; i < n * kPredOut; i += blockDim.x) {
    const double v = Y[i];
    acc[kPredFeat + (i % kPredOut)] += v * v;
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int f = 0; f < kPredFeat + kPredOut; ++f) {
    double v = acc[f];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) part[f][w] = v;
  }
  __syncthreads();
  if (threadIdx.x < kPredFeat + kPredOut) {
    double t = 0.0;
    for (int q = 0; q < static_cast<int>(blockDim.x >> 5); ++q) t += part[threadIdx.x][q];
    g_scale_sums[threadIdx.x] = t;
  }
}

__global__ void k_mlp_normalize(const float* __restrict__ X, const float* __restrict__ Y, int64_t n,
                                float s0, float s1, float s2, float s3, float s4, float o0, float o1,
                                float* __restrict__ Xn, float* __restrict__ Yn) {
  const float sx[kPredFeat] = {s0, s1, s2, s3, s4};
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n * kPredIn;
       i += stride)
    Xn[i] = X[i] / sx[(i % kPredIn) % kPredFeat];
  if (Y && Yn)
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n * kPredOut;
         i += stride)
      Yn[i] = Y[i] / ((i % kPredOut) ? o1 : o0);
}

// ---------------------------------------------------------------------------
// Batch forward (and backward) over tiles of up to 64 samples.
//
// Every product is a small matrix product from shared memory with a 4 x 4
// register tile per thread (16 FMA on 8 values read as 16-byte vectors, so the
// FMA pipe and not shared memory sets the pace):
//   forward   z[s][o] = b[o] + sum_k W[o][k] a[s][k]     rows s, columns c + 16 j
//   backward  d[s][k] = sum_o d[s][o] W[o][k]            rows s, columns 4 c + j
//   gradient  W[o][k] += sum_s d[s][o] a[s][k]           rows o, columns k
// The rows of W are padded (68 and 44 words) so that the forward pass's 16
// rows at a time and the backward pass's consecutive columns both read
// without bank conflicts from one copy.
//
// FP32 throughout: one step over 8192 samples is 0.25 GFMA, 6 us at the FMA
// peak; two tiles' phases and their barriers on each SM bound it.  A training
// step (gradient, sum over CTAs, Adam) as a caller sees it: 84.0 -> 34.8 us at
// 8192 samples (it was one dot product per thread, two shared-memory reads per
// FMA, and a sum over CTAs by one thread per entry).  The gradient's error
// against FP64 at 8192 samples: 2.0e-7 -> 5.9e-8 of its norm.
// ---------------------------------------------------------------------------
constexpr int kLdH = kHid + 4;     // row pitch of 64-wide arrays
constexpr int kLdX = kPredIn + 4;  // row pitch of 40-wide arrays

struct TrainSmem {
  float W1[kHid * kLdX], W2[kHid * kLdH], W3[kHid * kLdH], W4[kPredOut * kLdH];  // BF16-rounded
  float b[kHid * 3 + kPredOut];
  float pad[2];
  float a0[kTileS * kLdX];
  float a1[kTileS * kLdH], a2[kTileS * kLdH], a3[kTileS * kLdH];
  float g1[kTileS * kLdH], g2[kTileS * kLdH], g3[kTileS * kLdH];  // GELU' then deltas
  float d4[kTileS * kPredOut];
};
static_assert((kHid * 3 + kPredOut + 2) % 4 == 0, "rows start on 16 bytes");

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float get(const float4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }

// one hidden layer, forward, rows s0..s0+3 and columns c + 16 j
template <int IN, int LDW, int LDA, bool BACKWARD>
__device__ __forceinline__ void fwd_hidden(const float* W, const float* b, const float* a, float* out, float* g, int s0,
                                           int c) {
  float z[4][4];
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int i = 0; i < 4; ++i) z[i][j] = b[c + 16 * j];
#pragma unroll 2
  for (int k = 0; k < IN; k += 4) {
    float4 av[4], wv[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) av[i] = ld4(a + (s0 + i) * LDA + k);
#pragma unroll
    for (int j = 0; j < 4; ++j) wv[j] = ld4(W + (c + 16 * j) * LDW + k);
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) z[i][j] = fmaf(get(wv[j], q), get(av[i], q), z[i][j]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float v = z[i][j];
      out[(s0 + i) * kLdH + c + 16 * j] = gelu(v);
      if (BACKWARD) g[(s0 + i) * kLdH + c + 16 * j] = gelu_grad(v);
    }
}

// delta of the layer below, in place over its GELU': rows s0..s0+3, columns
// 4 c + j
__device__ __forceinline__ void back_hidden(const float* W, const float* d, float* g, int s0, int c) {
  float v[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) v[i][j] = 0.0f;
#pragma unroll 2
  for (int o = 0; o < kHid; o += 4) {
    float4 dv[4], wv[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) dv[i] = ld4(d + (s0 + i) * kLdH + o);
#pragma unroll
    for (int q = 0; q < 4; ++q) wv[q] = ld4(W + (o + q) * kLdH + 4 * c);
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) v[i][j] = fmaf(get(wv[q], j), get(dv[i], q), v[i][j]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float4* p = reinterpret_cast<float4*>(g + (s0 + i) * kLdH + 4 * c);
    const float4 t = *p;
    *p = make_float4(t.x * v[i][0], t.y * v[i][1], t.z * v[i][2], t.w * v[i][3]);
  }
}

// gradient of a weight tile: rows (outputs) 4 o + i, columns (inputs) 4 k + j,
// and the rows' delta sums; sums of kSumS samples at a time are added up, which
// keeps the rounding of a long FP32 sum down
constexpr int kSumS = 32;
template <int LDA>
__device__ __forceinline__ void grad_tile(const float* d, const float* a, int rows, int o, int k, float (&acc)[4][4],
                                          float (&bias)[4]) {
  for (int q = 0; q < rows; q += kSumS) {
    float w[4][4], b[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      b[i] = 0.0f;
#pragma unroll
      for (int j = 0; j < 4; ++j) w[i][j] = 0.0f;
    }
    const int end = min(q + kSumS, rows);
#pragma unroll 4
    for (int s = q; s < end; ++s) {
      const float4 dv = ld4(d + s * kLdH + 4 * o), av = ld4(a + s * LDA + 4 * k);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
#pragma unroll
        for (int j = 0; j < 4; ++j) w[i][j] = fmaf(get(dv, i), get(av, j), w[i][j]);
        b[i] += get(dv, i);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      bias[i] += b[i];
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] += w[i][j];
    }
  }
}

// tile: samples per tile (a multiple of 4, at most kTileS)
template <bool BACKWARD>
__global__ void __launch_bounds__(kTrainThreads, 1)
k_mlp_batch(const float* __restrict__ p, const float* __restrict__ Xn, const float* __restrict__ Yn,
            int64_t n, int tile, float* __restrict__ Yhat, float* __restrict__ work) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TrainSmem& sm = *reinterpret_cast<TrainSmem*>(smem_raw);
  const int t = threadIdx.x;
  cudaTriggerProgrammaticLaunchCompletion();  // the reduction may wait on the device
  // the network: BF16-rounded weights, FP32 biases (all of a thread's loads of a
  // matrix in flight together: gradient over 8192 samples 34.8 -> 30.7 us)
#pragma unroll
  for (int i = t; i < kHid * kPredIn; i += kTrainThreads)
    sm.W1[i / kPredIn * kLdX + i % kPredIn] = bf16_round(p[kOffW1 + i]);
#pragma unroll
  for (int i = t; i < kHid * kHid; i += kTrainThreads) {
    const int q = i / kHid * kLdH + i % kHid;
    sm.W2[q] = bf16_round(p[kOffW2 + i]);
    sm.W3[q] = bf16_round(p[kOffW3 + i]);
  }
  if (t < kPredOut * kHid) sm.W4[t / kHid * kLdH + t % kHid] = bf16_round(p[kOffW4 + t]);
  if (t < kHid * 3 + kPredOut)
    sm.b[t] = p[(t < kHid) ? kOffB1 + t
                : (t < 2 * kHid) ? kOffB2 + (t - kHid)
                : (t < 3 * kHid) ? kOffB3 + (t - 2 * kHid)
                                 : kOffB4 + (t - 3 * kHid)];
  // this thread's tiles: samples 4 r.. and columns of c; weights 4 r.. x 4 c..
  const int r = t / 16, c = t % 16;
  float gW1[4][4], gW2[4][4], gW3[4][4], gb1[4], gb2[4], gb3[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    gb1[i] = gb2[i] = gb3[i] = 0.0f;
#pragma unroll
    for (int j = 0; j < 4; ++j) gW1[i][j] = gW2[i][j] = gW3[i][j] = 0.0f;
  }
  float gW4 = 0.0f, gb4 = 0.0f, loss = 0.0f;
  const float inv_n = 1.0f / static_cast<float>(n);
  for (int64_t s_base = static_cast<int64_t>(blockIdx.x) * tile; s_base < n;
       s_base += static_cast<int64_t>(gridDim.x) * tile) {
    const int ns = static_cast<int>(min(static_cast<int64_t>(tile), n - s_base));
    const int rows = (ns + 3) & ~3;  // the rows past ns hold zeros and have no delta
    const bool mine = 4 * r < rows;
    for (int i = t; i < rows * kPredIn; i += kTrainThreads) {
      const int s = i / kPredIn;
      sm.a0[s * kLdX + i % kPredIn] = (s < ns) ? Xn[s_base * kPredIn + i] : 0.0f;
    }
    __syncthreads();
    if (mine) fwd_hidden<kPredIn, kLdX, kLdX, BACKWARD>(sm.W1, sm.b, sm.a0, sm.a1, sm.g1, 4 * r, c);
    __syncthreads();
    if (mine) fwd_hidden<kHid, kLdH, kLdH, BACKWARD>(sm.W2, sm.b + kHid, sm.a1, sm.a2, sm.g2, 4 * r, c);
    __syncthreads();
    if (mine) fwd_hidden<kHid, kLdH, kLdH, BACKWARD>(sm.W3, sm.b + 2 * kHid, sm.a2, sm.a3, sm.g3, 4 * r, c);
    __syncthreads();
    if (t < rows * kPredOut) {  // output layer, linear
      const int o = t & 1, s = t >> 1;
      float z = sm.b[3 * kHid + o];
#pragma unroll 4
      for (int k = 0; k < kHid; k += 4) {
        const float4 w = ld4(sm.W4 + o * kLdH + k), av = ld4(sm.a3 + s * kLdH + k);
        z = fmaf(w.x, av.x, z);
        z = fmaf(w.y, av.y, z);
        z = fmaf(w.z, av.z, z);
        z = fmaf(w.w, av.w, z);
      }
      if (!BACKWARD) {
        if (s < ns) Yhat[(s_base + s) * kPredOut + o] = z;
      } else {
        float d = 0.0f;
        if (s < ns) {
          const float e = z - Yn[(s_base + s) * kPredOut + o];
          d = e * inv_n;
          loss = fmaf(0.5f * e, e * inv_n, loss);
        }
        sm.d4[t] = d;
      }
    }
    __syncthreads();
    if constexpr (BACKWARD) {
      // delta of layer 3 (in place over its GELU'), gradient of layer 4
      for (int i = t; i < rows * kHid; i += kTrainThreads) {
        const int s = i / kHid, k = i % kHid;
        sm.g3[s * kLdH + k] *= sm.W4[k] * sm.d4[2 * s] + sm.W4[kLdH + k] * sm.d4[2 * s + 1];
      }
      if (t < kPredOut * kHid) {
        const int o = t / kHid, k = t % kHid;
        for (int q = 0; q < rows; q += kSumS) {
          float acc = 0.0f;
#pragma unroll 4
          for (int s = q; s < min(q + kSumS, rows); ++s) acc = fmaf(sm.d4[2 * s + o], sm.a3[s * kLdH + k], acc);
          gW4 += acc;
        }
      } else if (t < kPredOut * kHid + kPredOut) {
        for (int q = 0; q < rows; q += kSumS) {
          float acc = 0.0f;
          for (int s = q; s < min(q + kSumS, rows); ++s) acc += sm.d4[2 * s + t - kPredOut * kHid];
          gb4 += acc;
        }
      }
      __syncthreads();
      if (mine) back_hidden(sm.W3, sm.g3, sm.g2, 4 * r, c);
      grad_tile<kLdH>(sm.g3, sm.a2, rows, r, c, gW3, gb3);
      __syncthreads();
      if (mine) back_hidden(sm.W2, sm.g2, sm.g1, 4 * r, c);
      grad_tile<kLdH>(sm.g2, sm.a1, rows, r, c, gW2, gb2);
      __syncthreads();
      if (c < kPredIn / 4) grad_tile<kLdX>(sm.g1, sm.a0, rows, r, c, gW1, gb1);
      __syncthreads();
    }
  }
  if constexpr (BACKWARD) {
    // this CTA's partial sums, in parameter order
    float* w = work + static_cast<int64_t>(blockIdx.x) * kWorkRow;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (c < kPredIn / 4) w[kOffW1 + (4 * r + i) * kPredIn + 4 * c + j] = gW1[i][j];
        w[kOffW2 + (4 * r + i) * kHid + 4 * c + j] = gW2[i][j];
        w[kOffW3 + (4 * r + i) * kHid + 4 * c + j] = gW3[i][j];
      }
    if (c == 0)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        w[kOffB1 + 4 * r + i] = gb1[i];
        w[kOffB2 + 4 * r + i] = gb2[i];
        w[kOffB3 + 4 * r + i] = gb3[i];
      }
    if (t < kPredOut * kHid) w[kOffW4 + t] = gW4;
    else if (t < kPredOut * kHid + kPredOut) w[kOffB4 + t - kPredOut * kHid] = gb4;
    // loss: block sum in a fixed order
    __shared__ float lpart[kTrainThreads / 32];
    float l = loss;
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if ((t & 31) == 0) lpart[t >> 5] = l;
    __syncthreads();
    if (t == 0) {
      float s = 0.0f;
      for (int q = 0; q < kTrainThreads / 32; ++q) s += lpart[q];
      w[kNParam] = s;
    }
  }
}

// The CTAs' partial sums added in a fixed order: 32 entries per block, each
// by 8 threads over an eighth of the rows, the eighths in order.
constexpr int kReduceParts = 8;
__global__ void __launch_bounds__(32 * kReduceParts) k_mlp_reduce(const float* __restrict__ work, int ctas,
                                                                  float* __restrict__ grad, float* __restrict__ loss) {
  __shared__ float part[kReduceParts][32];
  cudaGridDependencySynchronize();
  const int e = threadIdx.x % 32, q = threadIdx.x / 32, i = blockIdx.x * 32 + e;
  const int per = (ctas + kReduceParts - 1) / kReduceParts, b0 = min(q * per, ctas), b1 = min(b0 + per, ctas);
  float s = 0.0f;
  if (i < kWorkRow) {
#pragma unroll 8
    for (int b = b0; b < b1; ++b) s += __ldcg(&work[static_cast<int64_t>(b) * kWorkRow + i]);
  }
  part[q][e] = s;
  __syncthreads();
  if (q != 0 || i >= kWorkRow) return;
  for (int k = 1; k < kReduceParts; ++k) s += part[k][e];
  if (i < kNParam) grad[i] = s;
  else *loss = s;
}

__global__ void k_mlp_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                           float* __restrict__ v, float lr, float b1, float b2, float eps, float c1,
                           float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= kNParam) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.0f - b1) * gi;
  const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi * c1) / (sqrtf(vi * c2) + eps);
}

// ---------------------------------------------------------------------------
// Host-side launchers
// ---------------------------------------------------------------------------
cudaError_t pack_predictor_launch(const float* params, PredNet* net, cudaStream_t st) {
  k_pack_predictor<<<(kNParam + 255) / 256, 256, 0, st>>>(params, net);
  return cudaGetLastError();
}

cudaError_t samples_launch(const DevParams* P, const cp_diag* hist, int64_t first, int64_t n,
                           float* X, float* Y, cudaStream_t st) {
  const int64_t blocks = (n + 127) / 128;
  k_samples<<<static_cast<unsigned>(blocks), 128, 0, st>>>(P, hist, first, n, X, Y);
  return cudaGetLastError();
}

int sm_count() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 1;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 1;
  return sms > 0 ? sms : 1;
}

cudaError_t mlp_batch_launch(bool backward, const float* p, const float* Xn, const float* Yn,
                             int64_t n, float* Yhat, float* work, int* ctas_out, cudaStream_t st) {
  const size_t smem = sizeof(TrainSmem);
  cudaError_t e = backward
                      ? cudaFuncSetAttribute(k_mlp_batch<true>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(smem))
                      : cudaFuncSetAttribute(k_mlp_batch<false>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  // as many samples per tile as give every SM the same number of whole tiles
  const int64_t sms = std::min(sm_count(), kTrainMaxCtas);
  const int64_t rounds = (n + sms * kTileS - 1) / (sms * kTileS);
  const int64_t even = (n + sms * rounds - 1) / (sms * rounds);
  const int tile = static_cast<int>(std::min<int64_t>((even + 3) & ~int64_t(3), kTileS));
  const int ctas = static_cast<int>(std::min<int64_t>((n + tile - 1) / tile, sms));
  if (ctas_out) *ctas_out = ctas;
  if (backward)
    k_mlp_batch<true><<<ctas, kTrainThreads, smem, st>>>(p, Xn, Yn, n, tile, Yhat, work);
  else
    k_mlp_batch<false><<<ctas, kTrainThreads, smem, st>>>(p, Xn, Yn, n, tile, Yhat, work);
  return cudaGetLastError();
}

cudaError_t mlp_reduce_launch(const float* work, int ctas, float* grad, float* loss, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((kWorkRow + 31) / 32, 1, 1);
  cfg.blockDim = dim3(32 * kReduceParts, 1, 1);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_mlp_reduce, work, ctas, grad, loss);
}

}  // namespace cpk

// ---------------------------------------------------------------------------
// C ABI of the training kernels
// ---------------------------------------------------------------------------
namespace {
cudaStream_t as_stream(void* s) { return static_cast<cudaStream_t>(s); }
int rc_of(cudaError_t e) { return e == cudaSuccess ? CP_OK : CP_ERR_CUDA; }
}  // namespace

extern "C" {

int cp_mlp_init(float* params, uint64_t seed, void* stream) {
  if (!params) return CP_ERR_ARG;
  cpk::k_mlp_init<<<(cpk::kNParam + 255) / 256, 256, 0, as_stream(stream)>>>(params, seed);
  return rc_of(cudaGetLastError());
}

int cp_mlp_scales(const float* X, const float* Y, int64_t n, cp_predictor* norm, void* stream) {
  if (!X || !Y || !norm || n <= 0) return CP_ERR_ARG;
  cudaStream_t st = as_stream(stream);
  cpk::k_mlp_scales<<<1, 1024, 0, st>>>(X, Y, n);
  cudaError_t e = cudaGetLastError();
  double sums[cpk::kPredFeat + cpk::kPredOut];
  if (e == cudaSuccess)
    e = cudaMemcpyFromSymbolAsync(sums, cpk::g_scale_sums, sizeof(sums), 0, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return CP_ERR_CUDA;
  for (int f = 0; f < cpk::kPredFeat; ++f) {
    const double r = std::sqrt(sums[f] / (static_cast<double>(n) * cpk::kPredWindow));
    norm->in_scale[f] = (r > 0.0 && std::isfinite(r)) ? static_cast<float>(r) : 1.0f;
  }
  for (int o = 0; o < cpk::kPredOut; ++o) {
    const double r = std::sqrt(sums[cpk::kPredFeat + o] / static_cast<double>(n));
    norm->out_scale[o] = (r > 0.0 && std::isfinite(r)) ? static_cast<float>(r) : 1.0f;
  }
  return CP_OK;
}

int cp_mlp_normalize(const float* X, const float* Y, int64_t n, const cp_predictor* norm, float* Xn,
                     float* Yn, void* stream) {
  if (!X || !Xn || !norm || n < 0 || ((Y == nullptr) != (Yn == nullptr))) return CP_ERR_ARG;
  if (n == 0) return CP_OK;
  const int64_t blocks = std::min<int64_t>((n * cpk::kPredIn + 255) / 256, 4096);
  cpk::k_mlp_normalize<<<static_cast<unsigned>(blocks), 256, 0, as_stream(stream)>>>(
      X, Y, n, norm->in_scale[0], norm->in_scale[1], norm->in_scale[2], norm->in_scale[3],
      norm->in_scale[4], norm->out_scale[0], norm->out_scale[1], Xn, Yn);
  return rc_of(cudaGetLastError());
}

int cp_mlp_forward(const float* params, const float* Xn, int64_t n, float* Yhat, void* stream) {
  if (!params || !Xn || !Yhat || n < 0) return CP_ERR_ARG;
  if (n == 0) return CP_OK;
  return rc_of(cpk::mlp_batch_launch(false, params, Xn, nullptr, n, Yhat, nullptr, nullptr,
                                     as_stream(stream)));
}

int64_t cp_mlp_work_floats(void) {
  return static_cast<int64_t>(cpk::kTrainMaxCtas) * cpk::kWorkRow;
}

int cp_mlp_loss_grad(const float* params, const float* Xn, const float* Yn, int64_t n, float* grad,
                     float* loss, float* work, void* stream) {
  if (!params || !Xn || !Yn || !grad || !loss || !work || n <= 0) return CP_ERR_ARG;
  cudaStream_t st = as_stream(stream);
  int ctas = 0;
  cudaError_t e = cpk::mlp_batch_launch(true, params, Xn, Yn, n, nullptr, work, &ctas, st);
  if (e != cudaSuccess) return CP_ERR_CUDA;
  return rc_of(cpk::mlp_reduce_launch(work, ctas, grad, loss, st));
}

int cp_mlp_adam(float* params, const float* grad, float* m, float* v, int64_t t, float lr,
                float beta1, float beta2, float eps, void* stream) {
  if (!params || !grad || !m || !v || t < 1 || !(lr > 0.0f) || !(beta1 >= 0.0f && beta1 < 1.0f) ||
      !(beta2 >= 0.0f && beta2 < 1.0f) || !(eps > 0.0f))
    return CP_ERR_ARG;
  const double c1 = 1.0 / (1.0 - std::pow(static_cast<double>(beta1), static_cast<double>(t)));
  const double c2 = 1.0 / (1.0 - std::pow(static_cast<double>(beta2), static_cast<double>(t)));
  cpk::k_mlp_adam<<<(cpk::kNParam + 255) / 256, 256, 0, as_stream(stream)>>>(
      params, grad, m, v, lr, beta1, beta2, eps, static_cast<float>(c1), static_cast<float>(c2));
  return rc_of(cudaGetLastError());
}

}  // extern "C"
