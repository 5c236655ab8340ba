// cp_gap2d.cu -- the 2D planar gap: x normal to the electrodes, y periodic.
//
// The cycle of the 1D gap (arXiv 2603.24010) in two dimensions, arranged for
// the GB300:
//
// * Particle store: structure of arrays per species (x, u in the 1D state's
//   buffers, y, w here), kept sorted by 32 x 32-cell tiles (counting sort
//   every `sort_every` steps, which also drops absorbed particles); each
//   tile's segment starts on a 16-byte boundary.
// * k2_push: a persistent grid takes work items of up to 32768 particles of
//   one tile from an atomic queue; the item's field window (the tile plus 4
//   cells of halo, E_x and E_y, each node paired with its neighbour in y)
//   is staged in shared memory, and its charge goes into five exact 32-bit
//   sums per cell (count, sum of wx1, sum of wy1, high and low parts of the
//   sum of wx1 wy1), from which the flush forms every node's int64 charge.
//   Particles that left their window since the sort (and the unsorted tail
//   of emitted electrons and beam ions) gather from and deposit into global
//   memory directly, with the same arithmetic.
// * Solve: each row of the grid is summed exactly (the int64 column sums are
//   the 1D coupled problem of Sec. 2.4.2/2.4.3, solved by the 1D cluster
//   solve, circuit and history included) and Fourier-transformed in y
//   (FFT, FP32); every transverse mode k != 0 solves its tridiagonal system
//   in x with phi = 0 on both electrodes (Thomas as two scans, one warp per
//   mode, beside the mean's solve); the inverse transform and the 1D field
//   give E_x = E_0(x) + dE_x and E_y on the staggered grid.
#include <cuda_runtime.h>

#include <algorithm>

#include "cp_common.cuh"
#include "cp_gap2d.cuh"

namespace cpk {

// ---------------------------------------------------------------------------
// Gather and deposit helpers (global coordinates; the window only changes
// where the values are read from or added to)
// ---------------------------------------------------------------------------
struct Stencil2 {
  int i, i1, j, j1;   // E_x: x half-grid indices, y node indices
  float t, v;
  int a, a1, jj, jj1; // E_y: x node indices, y half-grid indices
  float fx, vy;
};

__device__ __forceinline__ int wrapi(int j, int N) { return j < 0 ? j + N : (j >= N ? j - N : j); }

__device__ __forceinline__ Stencil2 stencil2(const Dev2D& D, float x, float y) {
  Stencil2 st;
  const float s = x - 0.5f;
  float sf = floorf(s);
  int i = static_cast<int>(sf);
  float t = s - sf;
  if (s < 0.0f) {
    i = 0;
    t = 0.0f;
  } else if (i >= D.Nx - 1) {
    i = D.Nx - 1;
    t = 0.0f;
  }
  st.i = i;
  st.i1 = min(i + 1, D.Nx - 1);
  st.t = t;
  const float yf = floorf(y);
  st.j = wrapi(static_cast<int>(yf), D.Ny);
  st.j1 = wrapi(st.j + 1, D.Ny);
  st.v = y - yf;
  const float xf = floorf(x);
  st.a = static_cast<int>(xf);
  st.a1 = st.a + 1;
  st.fx = x - xf;
  const float sy = y - 0.5f;
  const float syf = floorf(sy);
  st.jj = wrapi(static_cast<int>(syf), D.Ny);
  st.jj1 = wrapi(st.jj + 1, D.Ny);
  st.vy = sy - syf;
  return st;
}

__device__ __forceinline__ float bilin(float f00, float f10, float f01, float f11, float a, float b) {
  return (1.0f - b) * ((1.0f - a) * f00 + a * f10) + b * ((1.0f - a) * f01 + a * f11);
}

// window index of a 2x2 stencil's origin node (gx, gy) when the whole
// stencil lies in the window (origin at most kW2-2 from the window's edge);
// -1 otherwise
__device__ __forceinline__ int win_rel(int gx, int gy, int ox, int oy, int Ny) {
  const int lx = gx - ox;
  int ly = gy - oy;
  if (ly < 0) ly += Ny;
  else if (ly >= Ny) ly -= Ny;
  if (static_cast<unsigned>(lx) > static_cast<unsigned>(kW2 - 2) ||
      static_cast<unsigned>(ly) > static_cast<unsigned>(kW2 - 2))
    return -1;
  return lx * kW2 + ly;
}

// fixed-point bilinear weights floor(frac 2^16) per axis: the corner
// products sum to 2^32 per macroparticle (x - floor(x) and the power-of-two
// scaling are exact, so the truncation decides alone)
__device__ __forceinline__ void deposit_weights(float x, float y, int Ny, int* i, int* j, int* j1,
                                                unsigned long long* w00, unsigned long long* w10,
                                                unsigned long long* w01, unsigned long long* w11) {
  const float xf = floorf(x), yf = floorf(y);
  *i = static_cast<int>(xf);
  *j = static_cast<int>(yf);
  *j1 = wrapi(*j + 1, Ny);
  const unsigned int wx1 = __float2uint_rz((x - xf) * 65536.0f);
  const unsigned int wy1 = __float2uint_rz((y - yf) * 65536.0f);
  const unsigned int wx0 = 65536u - wx1, wy0 = 65536u - wy1;
  *w00 = static_cast<unsigned long long>(wx0) * wy0;
  *w10 = static_cast<unsigned long long>(wx1) * wy0;
  *w01 = static_cast<unsigned long long>(wx0) * wy1;
  *w11 = static_cast<unsigned long long>(wx1) * wy1;
}

// cell (i, j) of a particle and its per-axis weights wx1 = floor(frac(x) 2^16),
// wy1 = floor(frac(y) 2^16), as deposit_weights forms them
__device__ __forceinline__ void cell_weights(float x, float y, int* i, int* j, unsigned int* wx1,
                                             unsigned int* wy1) {
  const float xf = floorf(x), yf = floorf(y);
  *i = static_cast<int>(xf);
  *j = static_cast<int>(yf);
  *wx1 = __float2uint_rz((x - xf) * 65536.0f);
  *wy1 = __float2uint_rz((y - yf) * 65536.0f);
}

__device__ __forceinline__ void atomic_add_i64(long long* p, long long v) {
  atomicAdd(reinterpret_cast<unsigned long long*>(p), static_cast<unsigned long long>(v));
}

__device__ __forceinline__ void deposit2_global(const Dev2D& D, float x, float y, long long sign) {
  int i, j, j1;
  unsigned long long w00, w10, w01, w11;
  deposit_weights(x, y, D.Ny, &i, &j, &j1, &w00, &w10, &w01, &w11);
  const long long di = (i == 0) ? 2 : 1, di1 = (i + 1 == D.Nx) ? 2 : 1;
  long long* G = D.G2;
  const long long r0 = static_cast<long long>(i) * D.Ny, r1 = static_cast<long long>(i + 1) * D.Ny;
  if (w00) atomic_add_i64(&G[r0 + j], sign * di * static_cast<long long>(w00));
  if (w10) atomic_add_i64(&G[r1 + j], sign * di1 * static_cast<long long>(w10));
  if (w01) atomic_add_i64(&G[r0 + j1], sign * di * static_cast<long long>(w01));
  if (w11) atomic_add_i64(&G[r1 + j1], sign * di1 * static_cast<long long>(w11));
}

// ---------------------------------------------------------------------------
// k2_push
// ---------------------------------------------------------------------------
// Field and deposit window of one CTA.  The field window holds each node's
// value and that of the next node in y (one 8-byte load per stencil column).
// The deposit window, by cell (indexed like its lower corner node): the
// particle count n, the sums x, y of the per-axis weights wx1, wy1 and the
// high bits and low 16 bits of the sum of wx1 wy1 (< 2^32 each).  The four
// corner weights of a particle are linear in these (A = 2^16):
// w00 = A^2 - A wx1 - A wy1 + wx1 wy1, w10 = A wx1 - wx1 wy1,
// w01 = A wy1 - wx1 wy1, w11 = wx1 wy1; the flush forms each node's exact
// int64 sum from its four cells.  An item of at most 32768 particles keeps
// every 32-bit sum below 2^31.
constexpr int kWin2 = kW2 * kW2;
__device__ __forceinline__ void get2(const float* p, float (&v)[2]) {
  const float2 t = __ldcs(reinterpret_cast<const float2*>(p));
  v[0] = t.x; v[1] = t.y;
}
__device__ __forceinline__ void put2(float* p, const float (&v)[2]) {
  __stcs(reinterpret_cast<float2*>(p), make_float2(v[0], v[1]));
}
struct Window2 {
  float2 Ex[kWin2], Ey[kWin2];
  unsigned int n[kWin2], x[kWin2], y[kWin2], hi[kWin2], lo[kWin2];
};

__device__ __forceinline__ void deposit_window(Window2& W, int d, unsigned int wx1, unsigned int wy1) {
  const unsigned int xy = wx1 * wy1;  // < 2^32
  atomicAdd(&W.n[d], 1u);
  atomicAdd(&W.x[d], wx1);
  atomicAdd(&W.y[d], wy1);
  atomicAdd(&W.hi[d], xy >> 16);
  atomicAdd(&W.lo[d], xy & 0xFFFFu);
}

// The work item in hand and the CTA's tallies.
struct Item2 {
  float *xs, *us, *ys, *ws;
  const uint32_t* ids;
  AbsRec2* abs;
  float kx, ky;
  int s, ox, oy, win, abs_cap;
  int abs_n, over;
  unsigned int cfl;
  unsigned int cnt[2][kSpecies];
};

// The general path of one live particle (slot p, values before the step):
// gather and deposit in the window where the stencils fit, else in global
// memory; absorption.  Out of line: few particles take it, and inlined it
// costs the others registers.
__device__ __noinline__ void push_general(const Dev2D& D, Item2& T, Window2& W, long long p, float x, float y, float u,
                                          float w) {
  const int Ny = D.Ny, ox = T.ox, oy = T.oy;
  const bool win = T.win != 0;
  const Stencil2 st = stencil2(D, x, y);
  float ex, ey;
  // window origins of the two 2x2 stencils (the window is contiguous in y, so
  // the corners sit at +1 row / +1 column of their origin)
  const int le = win_rel(st.i, st.j, ox, oy, Ny), lf = win_rel(st.a, st.jj, ox, oy, Ny);
  if (win && le >= 0 && lf >= 0) {
    const int e00 = le, e10 = le + (st.i1 - st.i) * kW2;
    const int f00 = lf, f10 = lf + kW2;
    const float2 cx0 = W.Ex[e00], cx1 = W.Ex[e10], cy0 = W.Ey[f00], cy1 = W.Ey[f10];
    ex = bilin(cx0.x, cx1.x, cx0.y, cx1.y, st.t, st.v);
    ey = bilin(cy0.x, cy1.x, cy0.y, cy1.y, st.fx, st.vy);
  } else {
    const float* Ex = D.Ex;
    const float* Ey = D.Ey;
    const long long ri = static_cast<long long>(st.i) * Ny, ri1 = static_cast<long long>(st.i1) * Ny;
    const long long ra = static_cast<long long>(st.a) * Ny, ra1 = static_cast<long long>(st.a1) * Ny;
    ex = bilin(__ldg(&Ex[ri + st.j]), __ldg(&Ex[ri1 + st.j]), __ldg(&Ex[ri + st.j1]), __ldg(&Ex[ri1 + st.j1]), st.t,
               st.v);
    ey = bilin(__ldg(&Ey[ra + st.jj]), __ldg(&Ey[ra1 + st.jj]), __ldg(&Ey[ra + st.jj1]), __ldg(&Ey[ra1 + st.jj1]),
               st.fx, st.vy);
  }
  const float un = fmaf(T.kx, ex, u);
  const float wn = fmaf(T.ky, ey, w);
  const float xn = x + un;
  float yn = y + wn;
  if (yn < 0.0f) yn += D.Nyf;
  if (yn >= D.Nyf) yn -= D.Nyf;
  if (!(yn >= 0.0f && yn < D.Nyf)) {  // more than one period in a step (or not finite)
    yn -= D.Nyf * floorf(yn / D.Nyf);
    if (!(yn >= 0.0f && yn < D.Nyf)) yn = 0.0f;
  }
  atomicMax(&T.cfl, __float_as_uint(fmaxf(fabsf(un), fabsf(wn))));
  if (!(xn > 0.0f && xn < D.Nxf)) {  // absorbed
    const int el = (xn <= 0.0f) ? 0 : 1;
    atomicAdd(&T.cnt[el][T.s], 1u);
    if (T.s == CP_IONS) {
      const int slot = atomicAdd(&T.abs_n, 1);
      if (slot < T.abs_cap) {
        AbsRec2 r;
        r.id = T.ids[p];
        r.el = static_cast<uint32_t>(el);
        r.u = un;
        r.w = wn;
        r.eta = yn;
        r.pad = 0.0f;
        T.abs[slot] = r;
      } else {
        T.over = 1;
      }
    }
    T.xs[p] = -1.0f;
    T.us[p] = 0.0f;
    T.ys[p] = 0.0f;
    T.ws[p] = 0.0f;
    return;
  }
  T.xs[p] = xn;
  T.us[p] = un;
  T.ys[p] = yn;
  T.ws[p] = wn;
  int i, j;
  unsigned int wx1, wy1;
  cell_weights(xn, yn, &i, &j, &wx1, &wy1);
  const int d00 = win ? win_rel(i, j, ox, oy, Ny) : -1;
  if (d00 >= 0) deposit_window(W, d00, wx1, wy1);
  else deposit2_global(D, xn, yn, T.s == CP_IONS ? 1LL : -1LL);
}

// What bounds it: instruction issue and, for grids whose tiles hold few
// particles, the staging and flush of each item's window.  Floors come from
// one addition rounded down instead of floor and conversion instructions (a
// quarter of the issue rate), window indices from masks, range checks are two
// compares, two particles per thread are processed while the next two are on
// their way, and what few particles need is out of line.  Push at 1024 x 1024
// cells, 2e7 particles: 226 -> 176 us; at 96 x 128, 3e5: 42.4 -> 21.8 us
// (items sized by the store, the beam's draws as items of their own).
__global__ void __launch_bounds__(kThreads2, 2)
k2_push(const DevParams* __restrict__ P, DevState* S, const Dev2D* __restrict__ Dp,
        const __grid_constant__ Dev2D Dc, int* __restrict__ item_ctr, AbsRec2* __restrict__ abs_all,
        int abs_cap) {
  extern __shared__ __align__(16) unsigned char smem2[];
  Window2& W = *reinterpret_cast<Window2*>(smem2);
  __shared__ Item2 T;
  __shared__ int s_items[2 * kSpecies + 1];  // item offsets: sorted / tail per species
  __shared__ int s_stop;
  __shared__ unsigned long long s_emit[2];
  __shared__ long long s_conv, s_energy;

  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  // the fields fixed at creation come from the launch parameters; the sort
  // swaps the y, w buffers and sets n_sorted on the device, so those are read
  // from the device copy
  const Dev2D& D = Dc;
  // beam ions per work item: about two items per CTA, whole warps
  const int nbeam = min(kThreads2, (P->beam_per_step / (2 * static_cast<int>(gridDim.x)) + 32) & ~31);
  if (threadIdx.x == 0) {
    s_stop = (ldcg(&S->status) != 0);
    T.abs_n = 0;
    T.over = 0;
    T.cfl = 0u;
    T.abs = abs_all + static_cast<size_t>(blockIdx.x) * abs_cap;
    T.abs_cap = abs_cap;
    T.ids = S->id;
    s_conv = 0;
    s_energy = 0;
    s_emit[0] = s_emit[1] = 0ULL;
    int acc = (P->beam_per_step + nbeam - 1) / nbeam;  // the beam's items come first
    for (int s = 0; s < kSpecies; ++s) {
      s_items[2 * s] = acc;
      acc += D.wi_off[s * (D.T + 1) + D.T];
      s_items[2 * s + 1] = acc;
      const long long tail = S->n_proc[s] - Dp->n_sorted[s];
      acc += static_cast<int>((tail + kPass2 - 1) / kPass2);
    }
    s_items[2 * kSpecies] = acc;
  }
  if (threadIdx.x < 2 * kSpecies) T.cnt[threadIdx.x / kSpecies][threadIdx.x % kSpecies] = 0u;
  __syncthreads();
  if (s_stop) return;
  const bool half = (S->pushed == 0);
  const int64_t step = S->level;
  const int Ny = D.Ny;
  unsigned int cfl = 0u;

  const int n_items = s_items[2 * kSpecies];
  // Work items are taken from a queue (one atomic ticket per item): items
  // differ in size (whole and partial tiles, the unsorted tails), and a
  // fixed round-robin deal left CTAs idle while others finished theirs.
  // The last CTA out resets the queue for the next launch.
  __shared__ int s_item[2];
  if (threadIdx.x == 0) s_item[0] = atomicAdd(&item_ctr[0], 1);
  for (int turn = 0;; turn ^= 1) {
    __syncthreads();  // the ticket is there, and every thread has read the one before it
    const int item = s_item[turn];
    if (item >= n_items) break;
    if (threadIdx.x == 0) s_item[turn ^ 1] = atomicAdd(&item_ctr[0], 1);  // the next item's, in its shadow
    if (item < s_items[0]) {
      // Beam ions entering at x = d with a Gaussian transverse profile, one
      // per thread.  Their draws are FP64 chains (2 operations a cycle and SM,
      // about 5 us), so they are items of their own, spread over the CTAs.
      // Their slots lie behind the ions in use: the beam alone appends ions.
      const int Bn = P->beam_per_step, k = item * nbeam + static_cast<int>(threadIdx.x);
      if (static_cast<int>(threadIdx.x) < nbeam && k < Bn) {
        const double pi = 3.14159265358979323846;
        const U64x4 wv = philox4x64_10(static_cast<uint64_t>(k), static_cast<uint64_t>(step), 0, 0, P->seed, kTagBeam);
        const double frac = u01(wv.w[0]);
        const double Eb = (P->beam_mode == 0)
                              ? P->beam_E_eV
                              : __dadd_rn(P->beam_Emin_eV, __dmul_rn(__dsub_rn(P->beam_Emax_eV, P->beam_Emin_eV), u01(wv.w[1])));
        const double ub = sqrt(2.0 * Eb * P->e / P->m_i) * P->dt / P->dx;
        const double z = sqrt(-2.0 * log(u01(wv.w[2]))) * cos(2.0 * pi * u01(wv.w[3]));
        double yc = D.beam_yc + D.beam_sigma * z;
        yc -= static_cast<double>(Ny) * floor(yc / static_cast<double>(Ny));
        float yr = static_cast<float>(yc);
        if (!(yr < D.Nyf)) yr = 0.0f;
        const float xr = nudge_inside<float>(__dsub_rn(static_cast<double>(D.Nx), __dmul_rn(ub, frac)), D.Nx);
        const long long slot = S->n_proc[CP_IONS] + k;
        if (slot < P->cap[CP_IONS]) {
          static_cast<float*>(S->xi[CP_IONS])[slot] = xr;
          static_cast<float*>(S->u[CP_IONS])[slot] = static_cast<float>(-ub);
          static_cast<float*>(Dp->y[CP_IONS])[slot] = yr;
          static_cast<float*>(Dp->w[CP_IONS])[slot] = 0.0f;
          S->id[slot] = S->beam_id_base + static_cast<uint32_t>(step * Bn + k);
          deposit2_global(D, xr, yr, 1LL);
        } else {
          T.over = 1;
        }
      }
      continue;
    }
    int s = 0;
    while (item >= s_items[2 * s + 2]) ++s;
    const bool tail = item >= s_items[2 * s + 1];
    long long p0, p1;
    int ox = 0, oy = 0;
    bool win = false;
    if (!tail) {
      const int k = item - s_items[2 * s];
      const int* wo = D.wi_off + s * (D.T + 1);
      int lo = 0, hi = D.T;  // tile with wo[t] <= k < wo[t+1]
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (wo[mid] <= k) lo = mid;
        else hi = mid;
      }
      const int t = lo;
      const int* ts = D.tile_start + s * (D.T + 1);
      const int chunk = Dp->chunk[s];
      p0 = ts[t] + static_cast<long long>(k - wo[t]) * chunk;
      p1 = min(static_cast<long long>(ts[t + 1]), p0 + chunk);
      ox = (t / D.nty) * kT2 - kH2 - 1;
      oy = (t % D.nty) * kT2 - kH2 - 1;
      win = D.use_win != 0;
      // stage the field window, all of a thread's loads in flight; zero the
      // deposit window
      constexpr int kNodes = (kW2 * kW2 + kThreads2 - 1) / kThreads2;
      float e[kNodes][4];
#pragma unroll
      for (int c = 0; c < kNodes; ++c) {
        const int q = threadIdx.x + c * kThreads2;
        const int gx = ox + q / kW2;
        const int gy = (oy + q % kW2) & (Ny - 1), gy1 = (gy + 1) & (Ny - 1);
        const long long r = static_cast<long long>(gx) * Ny;
        const bool ix = win && q < kW2 * kW2 && gx >= 0 && gx < D.Nx, iy = win && q < kW2 * kW2 && gx >= 0 && gx <= D.Nx;
        e[c][0] = ix ? __ldcg(&D.Ex[r + gy]) : 0.0f;
        e[c][1] = ix ? __ldcg(&D.Ex[r + gy1]) : 0.0f;
        e[c][2] = iy ? __ldcg(&D.Ey[r + gy]) : 0.0f;
        e[c][3] = iy ? __ldcg(&D.Ey[r + gy1]) : 0.0f;
      }
#pragma unroll
      for (int c = 0; c < kNodes; ++c) {
        const int q = threadIdx.x + c * kThreads2;
        if (q < kW2 * kW2) {
          W.Ex[q] = make_float2(e[c][0], e[c][1]);
          W.Ey[q] = make_float2(e[c][2], e[c][3]);
          W.n[q] = W.x[q] = W.y[q] = W.hi[q] = W.lo[q] = 0u;
        }
      }
    } else {
      const int k = item - s_items[2 * s + 1];
      p0 = Dp->n_sorted[s] + static_cast<long long>(k) * kPass2;
      p1 = min(static_cast<long long>(S->n_proc[s]), p0 + kPass2);
    }
    float* xs = reinterpret_cast<float*>(S->xi[s]);
    float* us = reinterpret_cast<float*>(S->u[s]);
    float* ys = reinterpret_cast<float*>(Dp->y[s]);
    float* ws = reinterpret_cast<float*>(Dp->w[s]);
    const float kx = D.kx[half ? 0 : 1][s], ky = D.ky[half ? 0 : 1][s];
    // half-grid columns (window coordinates) of the fast path: both of a
    // stencil's columns inside the gap and the window
    const int ymask = Ny - 1;
    const int lo_h = max(0, -ox);
    const int hi_h = min(D.Nx - 2 - ox, kW2 - 3);
    if (hi_h < lo_h) win = false;  // (no cell of the tile has one)
    const unsigned int n_h = static_cast<unsigned int>(hi_h - lo_h);
    if (threadIdx.x == 0) {
      T.xs = xs; T.us = us; T.ys = ys; T.ws = ws;
      T.kx = kx; T.ky = ky;
      T.s = s; T.ox = ox; T.oy = oy; T.win = win;
    }
    __syncthreads();
    // the next pass's particles are requested before this pass's are processed
    const long long base0 = p0 + static_cast<long long>(threadIdx.x) * kPer2;
    constexpr long long kStep = kThreads2 * kPer2;
    float nx[kPer2], nu[kPer2], ny[kPer2], nw[kPer2];
    auto fetch = [&](long long b) {
      get2(xs + b, nx);
      get2(us + b, nu);
      get2(ys + b, ny);
      get2(ws + b, nw);
    };
    if (base0 < p1) fetch(base0);
    for (long long base = base0; base < p1; base += kStep) {
      float xv[kPer2], uv[kPer2], yv[kPer2], wv[kPer2];
#pragma unroll
      for (int q = 0; q < kPer2; ++q) {
        xv[q] = nx[q];
        uv[q] = nu[q];
        yv[q] = ny[q];
        wv[q] = nw[q];
      }
      if (base + kStep < p1) fetch(base + kStep);
      // Fast path, without divergent branches: a live particle whose
      // stencils lie in the window and off the electrodes' half cells, that
      // stays inside the gap and whose deposit lands in the window (the
      // common case).  Every other live particle is flagged and takes the
      // general path below, on its unchanged values, with the same
      // arithmetic.
      unsigned int slow = 0u;
#pragma unroll
      for (int q = 0; q < kPer2; ++q) {
        const float x = xv[q], y = yv[q];
        const bool alive = (x > 0.0f && x < D.Nxf);
        if (!win) {
          if (alive) slow |= 1u << q;
          continue;
        }
        float fx, fy, tx, ty;  // fractions on the nodes and on the half grid
        const int i = floor_split(x, &fx) - ox, ih = floor_split(x - 0.5f, &tx) - ox;
        const int j = (floor_split(y, &fy) - oy) & ymask, jh = (floor_split(y - 0.5f, &ty) - oy) & ymask;
        // ih in [lo_h, lo_h + n_h] puts i = ih or ih + 1 into the window too, and
        // jh <= kW2 - 3 does so for j = jh or jh + 1
        const bool gw = alive && static_cast<unsigned>(ih - lo_h) <= n_h && jh <= kW2 - 3;
        const int e0 = gw ? ih * kW2 + j : 0, f0 = gw ? i * kW2 + jh : 0;
        const float2 cx0 = W.Ex[e0], cx1 = W.Ex[e0 + kW2], cy0 = W.Ey[f0], cy1 = W.Ey[f0 + kW2];
        const float ex = bilin(cx0.x, cx1.x, cx0.y, cx1.y, tx, fy);
        const float ey = bilin(cy0.x, cy1.x, cy0.y, cy1.y, fx, ty);
        const float un = fmaf(kx, ex, uv[q]);
        const float wn = fmaf(ky, ey, wv[q]);
        const float xn = x + un;
        float yn = y + wn;
        if (yn < 0.0f) yn += D.Nyf;
        if (yn >= D.Nyf) yn -= D.Nyf;
        const bool inside = (xn > 0.0f && xn < D.Nxf) && (yn >= 0.0f && yn < D.Nyf);
        const int di = floor_split(xn, &fx) - ox;
        const int dj = (floor_split(yn, &fy) - oy) & ymask;
        const bool good = gw && inside && static_cast<unsigned>(di) <= kW2 - 2 && dj <= kW2 - 2;
        if (good) {
          deposit_window(W, di * kW2 + dj, frac16(fx), frac16(fy));
          cfl = max(cfl, __float_as_uint(fmaxf(fabsf(un), fabsf(wn))));
          xv[q] = xn;
          uv[q] = un;
          yv[q] = yn;
          wv[q] = wn;
        } else if (alive) {
          slow |= 1u << q;
        }
      }
      put2(xs + base, xv);
      put2(us + base, uv);
      put2(ys + base, yv);
      put2(ws + base, wv);
      if (slow) {  // rewrites the flagged particles' slots
#pragma unroll
        for (int q = 0; q < kPer2; ++q)
          if ((slow >> q) & 1u) push_general(D, T, W, base + q, xv[q], yv[q], uv[q], wv[q]);
      }
    }
    if (win) {  // flush the deposit window into the int64 grid
      __syncthreads();
      for (int q = threadIdx.x; q < kW2 * kW2; q += kThreads2) {
        const int p = q / kW2, r = q % kW2;
        constexpr long long A = 65536;
        auto sxy = [&](int c) { return (static_cast<long long>(W.hi[c]) << 16) + static_cast<long long>(W.lo[c]); };
        // w00 of cell (p, r), w10 of (p-1, r), w01 of (p, r-1), w11 of (p-1, r-1)
        long long v = A * A * static_cast<long long>(W.n[q]) - A * static_cast<long long>(W.x[q]) -
                      A * static_cast<long long>(W.y[q]) + sxy(q);
        if (p > 0) v += A * static_cast<long long>(W.x[q - kW2]) - sxy(q - kW2);
        if (r > 0) v += A * static_cast<long long>(W.y[q - 1]) - sxy(q - 1);
        if (p > 0 && r > 0) v += sxy(q - kW2 - 1);
        if (v == 0) continue;
        const int gx = ox + q / kW2;
        const int gy = wrapi(oy + q % kW2, Ny);
        const long long dbl = (gx == 0 || gx == D.Nx) ? 2 : 1;
        atomic_add_i64(&D.G2[static_cast<long long>(gx) * Ny + gy], s == CP_IONS ? dbl * v : -dbl * v);
      }
      __syncthreads();
    }
  }
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(&item_ctr[1], 1) == static_cast<int>(gridDim.x) - 1) {  // every CTA has left the queue
      item_ctr[0] = 0;
      item_ctr[1] = 0;
      __threadfence();
    }
  }
  cfl = warp_max_u(cfl);
  if (lane_id() == 0 && cfl) atomicMax(&T.cfl, cfl);
  __syncthreads();

  // --- secondary emission from the ions this CTA saw absorbed ---------------
  const int na = min(T.abs_n, abs_cap);
  const double dx = P->dx, dt = P->dt, dy = D.dy;
  for (int r = threadIdx.x; r < na; r += kThreads2) {
    const AbsRec2 rec = T.abs[r];
    const double vx = static_cast<double>(rec.u) * dx / dt;
    const double vy = static_cast<double>(rec.w) * dy / dt;
    const double Eev = 0.5 * P->m_i * (vx * vx + vy * vy) / P->e;
    const int nse = see_count(P, Eev, rec.id, step);
    const int el = static_cast<int>(rec.el);
    if (el == 0) {
      atomicAdd(reinterpret_cast<unsigned long long*>(&s_energy),
                static_cast<unsigned long long>(__double2ll_rn(Eev * 256.0)));
      if (nse) atomicAdd(reinterpret_cast<unsigned long long*>(&s_conv),
                         static_cast<unsigned long long>(static_cast<long long>(nse)));
    }
    if (nse == 0) continue;
    atomicAdd(&s_emit[el], static_cast<unsigned long long>(nse));
    const unsigned long long wb =
        atomicAdd(reinterpret_cast<unsigned long long*>(&S->n_alloc[CP_SECONDARIES]),
                  static_cast<unsigned long long>(nse));
    float* xs = reinterpret_cast<float*>(S->xi[CP_SECONDARIES]);
    float* us = reinterpret_cast<float*>(S->u[CP_SECONDARIES]);
    float* ys = reinterpret_cast<float*>(Dp->y[CP_SECONDARIES]);
    float* ws = reinterpret_cast<float*>(Dp->w[CP_SECONDARIES]);
    for (int jn = 0; jn < nse; ++jn) {
      double frac;
      const double use = see_speed(P, rec.id, step, jn, &frac) * dt / dx;
      const double xd = (el == 0) ? __dmul_rn(use, frac) : __dsub_rn(static_cast<double>(D.Nx), __dmul_rn(use, frac));
      const float xr = nudge_inside<float>(xd, D.Nx);
      const unsigned long long slot = wb + static_cast<unsigned long long>(jn);
      if (slot < static_cast<unsigned long long>(P->cap[CP_SECONDARIES])) {
        xs[slot] = xr;
        us[slot] = static_cast<float>(el == 0 ? use : -use);
        ys[slot] = rec.eta;
        ws[slot] = 0.0f;
        deposit2_global(D, xr, rec.eta, -1LL);
      } else {
        T.over = 1;
      }
    }
  }

  __syncthreads();
  if (threadIdx.x == 0) {
    for (int e = 0; e < 2; ++e)
      for (int s = 0; s < kSpecies; ++s)
        if (T.cnt[e][s]) atomicAdd(&S->absorbed[e][s], static_cast<unsigned long long>(T.cnt[e][s]));
    if (s_emit[0]) atomicAdd(&S->emitted[0], s_emit[0]);
    if (s_emit[1]) atomicAdd(&S->emitted[1], s_emit[1]);
    const long long conv = static_cast<long long>(T.cnt[0][CP_IONS]) -
                           static_cast<long long>(T.cnt[0][CP_ELECTRONS]) -
                           static_cast<long long>(T.cnt[0][CP_SECONDARIES]) + s_conv;
    if (conv) atomic_add_i64(&S->conv_count, conv);
    if (s_energy) atomic_add_i64(&S->ion_energy_q, s_energy);
    if (T.cfl) atomicMax(&S->max_cfl_bits, T.cfl);
    if (blockIdx.x == 0 && P->beam_per_step > 0) {
      atomicAdd(&S->injected, static_cast<unsigned long long>(P->beam_per_step));
      atomicAdd(reinterpret_cast<unsigned long long*>(&S->n_alloc[CP_IONS]),
                static_cast<unsigned long long>(P->beam_per_step));
    }
    if (T.over) atomicCAS(&S->status, 0, CP_ERR_CAPACITY);
  }
}

// Level 0: deposit every live particle of one species (global atomics).
__global__ void k2_deposit0(const DevState* S, const Dev2D* Dp, int s) {
  const Dev2D& D = *Dp;
  const float* xs = reinterpret_cast<const float*>(S->xi[s]);
  const float* ys = reinterpret_cast<const float*>(D.y[s]);
  const long long n = S->n_proc[s];
  const long long sign = (s == CP_IONS) ? 1LL : -1LL;
  for (long long k = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; k < n;
       k += static_cast<long long>(gridDim.x) * blockDim.x) {
    const float x = xs[k];
    if (x > 0.0f && x < D.Nxf) deposit2_global(D, x, ys[k], sign);
  }
}

// ---------------------------------------------------------------------------
// Counting sort by tile (drops dead slots; tile segments padded to 4)
// ---------------------------------------------------------------------------
__device__ __forceinline__ int tile_of(const Dev2D& D, float x, float y) {
  const int tx = min(static_cast<int>(x) / kT2, D.ntx - 1);
  const int ty = min(static_cast<int>(y) / kT2, D.nty - 1);
  return tx * D.nty + ty;
}

// Counting sort in three passes, each block owning one contiguous range of
// slots: per-block tile histograms, then (one block) the tile segments and
// every block's base in each tile, then the scatter with shared-memory
// cursors -- no global atomics on the per-tile cursors.
__device__ __forceinline__ void block_range(long long n, long long* b0, long long* b1) {
  *b0 = n * blockIdx.x / gridDim.x;
  *b1 = n * (blockIdx.x + 1) / gridDim.x;
}

// exclusive prefix of v over the block's threads (blockDim a multiple of 32)
__device__ __forceinline__ int block_excl_scan(int v, int* wsum) {
  const int incl = warp_incl_scan(v);
  if (lane_id() == 31) wsum[threadIdx.x >> 5] = incl;
  __syncthreads();
  int base = 0;
  for (int q = 0; q < static_cast<int>(threadIdx.x >> 5); ++q) base += wsum[q];
  return base + incl - v;
}

__global__ void k2_hist(const DevState* S, Dev2D* Dp) {
  extern __shared__ int hist[];
  const int s = blockIdx.y;
  const Dev2D& D = *Dp;
  for (int t = threadIdx.x; t < D.T; t += blockDim.x) hist[t] = 0;
  __syncthreads();
  const float* xs = reinterpret_cast<const float*>(S->xi[s]);
  const float* ys = reinterpret_cast<const float*>(D.y[s]);
  long long b0, b1;
  block_range(S->n_proc[s], &b0, &b1);
  // warp-uniform trips; each run of consecutive lanes in one tile (sorted
  // data: most of a warp) is counted by one shared-memory atomic
  constexpr int U = 4;
  const long long step = static_cast<long long>(blockDim.x) * U;
  for (long long k0 = b0 + (threadIdx.x & ~31u); k0 < b1; k0 += step) {
    float x[U], y[U];
#pragma unroll
    for (int c = 0; c < U; ++c) {
      const long long k = k0 + static_cast<long long>(c) * blockDim.x + lane_id();
      const bool in = k < b1;
      x[c] = in ? xs[k] : -1.0f;
      y[c] = in ? ys[k] : 0.0f;
    }
#pragma unroll
    for (int c = 0; c < U; ++c) {
      const int t = (x[c] > 0.0f && x[c] < D.Nxf) ? tile_of(D, x[c], y[c]) : -1;
      const int tp = __shfl_up_sync(0xffffffffu, t, 1);
      const bool start = (lane_id() == 0) || (t != tp);
      const unsigned starts = __ballot_sync(0xffffffffu, start);
      const unsigned later = starts & ~((2u << lane_id()) - 1u);
      const int next = later ? __ffs(later) - 1 : 32;
      if (start && t >= 0) atomicAdd(&hist[t], next - static_cast<int>(lane_id()));
    }
  }
  __syncthreads();
  const int G = gridDim.x;  // layout [tile][block]: each tile's counts contiguous
  for (int t = threadIdx.x; t < D.T; t += blockDim.x) D.bhist[(static_cast<long long>(s) * D.T + t) * G + blockIdx.x] = hist[t];
}

// one block per species: tile segment starts (padded to 4) and the dead
// padding in the destination
__global__ void k2_scan(DevState* S, Dev2D* Dp) {
  Dev2D& D = *Dp;
  __shared__ int wsum[32];
  const int s = blockIdx.x, T = D.T;
  const int* cnt = D.tile_cnt + s * T;
  int* ts = D.tile_start + s * (T + 1);
  const int per = (T + blockDim.x - 1) / blockDim.x;
  const int t0 = min(static_cast<int>(threadIdx.x) * per, T), t1 = min(t0 + per, T);
  int a = 0;
  for (int t = t0; t < t1; ++t) a += (cnt[t] + 3) & ~3;
  int ra = block_excl_scan(a, wsum);
  float* xd = reinterpret_cast<float*>(S->xi_alt[s]);
  float* ud = reinterpret_cast<float*>(S->u_alt[s]);
  const long long cap = D.cap[s];
  for (int t = t0; t < t1; ++t) {
    ts[t] = ra;
    const int c = cnt[t], c4 = (c + 3) & ~3;
    for (int k = c; k < c4; ++k) {  // dead padding slots
      if (ra + k < cap) {
        xd[ra + k] = -1.0f;
        ud[ra + k] = 0.0f;
      }
    }
    ra += c4;
  }
  if (threadIdx.x == blockDim.x - 1) ts[T] = ra;
}

// one block per tile: exclusive scan of the per-block counts over the blocks
// (each block's offset within the tile) and the tile's total
__global__ void k2_tilescan(Dev2D* Dp, int G) {
  Dev2D& D = *Dp;
  __shared__ int wsum[32];
  const int t = blockIdx.x, s = blockIdx.y, T = D.T;
  const int per = (G + blockDim.x - 1) / blockDim.x;
  const int b0 = min(static_cast<int>(threadIdx.x) * per, G), b1 = min(b0 + per, G);
  int* col = D.bhist + (static_cast<long long>(s) * T + t) * G;
  int loc = 0;
  for (int b = b0; b < b1; ++b) loc += col[b];
  int run = block_excl_scan(loc, wsum);
  for (int b = b0; b < b1; ++b) {
    const int c = col[b];
    col[b] = run;
    run += c;
  }
  if (threadIdx.x == blockDim.x - 1) D.tile_cnt[s * T + t] = run;
}

__global__ void __launch_bounds__(512, 2) k2_scatter(const DevState* S, Dev2D* Dp) {
  extern __shared__ int cur[];
  const Dev2D& D = *Dp;
  const int s = blockIdx.y;
  for (int t = threadIdx.x; t < D.T; t += blockDim.x)  // this block's first slot in each tile
    cur[t] = D.tile_start[s * (D.T + 1) + t] + D.bhist[(static_cast<long long>(s) * D.T + t) * gridDim.x + blockIdx.x];
  __syncthreads();
  const float* xs = reinterpret_cast<const float*>(S->xi[s]);
  const float* us = reinterpret_cast<const float*>(S->u[s]);
  const float* ys = reinterpret_cast<const float*>(D.y[s]);
  const float* ws = reinterpret_cast<const float*>(D.w[s]);
  float* xd = reinterpret_cast<float*>(S->xi_alt[s]);
  float* ud = reinterpret_cast<float*>(S->u_alt[s]);
  float* yd = reinterpret_cast<float*>(D.y_alt[s]);
  float* wd = reinterpret_cast<float*>(D.w_alt[s]);
  const uint32_t* is = S->id;
  uint32_t* id_d = S->id_alt;
  const bool ions = (s == CP_IONS);
  long long b0, b1;
  block_range(S->n_proc[s], &b0, &b1);
  constexpr int U = 2;  // warp chunks whose loads are issued together
  const long long step = static_cast<long long>(blockDim.x) * U;
  for (long long k0 = b0 + (threadIdx.x & ~31u); k0 < b1; k0 += step) {
    float x[U], y[U], u[U], w[U];
    uint32_t id[U];
#pragma unroll
    for (int c = 0; c < U; ++c) {  // every load first: one memory round trip per U chunks
      const long long k = k0 + static_cast<long long>(c) * blockDim.x + lane_id();
      const bool in = k < b1;
      x[c] = in ? xs[k] : -1.0f;
      y[c] = in ? ys[k] : 0.0f;
      u[c] = in ? us[k] : 0.0f;
      w[c] = in ? ws[k] : 0.0f;
      id[c] = (in && ions) ? is[k] : 0u;
    }
#pragma unroll
    for (int c = 0; c < U; ++c) {
      const int t = (x[c] > 0.0f && x[c] < D.Nxf) ? tile_of(D, x[c], y[c]) : -1;
      // runs of consecutive lanes in one tile: the run's first lane reserves
      // its length, every lane takes the slot of its place in the run
      const int tp = __shfl_up_sync(0xffffffffu, t, 1);
      const bool start = (lane_id() == 0) || (t != tp);
      const unsigned starts = __ballot_sync(0xffffffffu, start);
      const unsigned later = starts & ~((2u << lane_id()) - 1u);  // run starts after this lane
      const int next = later ? __ffs(later) - 1 : 32;
      const int rs = 31 - __clz(starts & ((2u << lane_id()) - 1u));  // this lane's run start
      int base = 0;
      if (start && t >= 0) base = atomicAdd(&cur[t], next - static_cast<int>(lane_id()));
      base = __shfl_sync(0xffffffffu, base, rs);
      if (t < 0) continue;
      const long long o = static_cast<long long>(base) + (static_cast<int>(lane_id()) - rs);
      if (o >= D.cap[s]) continue;  // the sorted store would not fit (reported by k2_finish)
      xd[o] = x[c];
      ud[o] = u[c];
      yd[o] = y[c];
      wd[o] = w[c];
      if (ions) id_d[o] = id[c];
    }
  }
}

// One block per species: the push's work items and the sorted buffers swapped
// in.  An item holds at most `chunk` particles of one tile: about two items
// for each of the push's G CTAs, so that small stores reach every SM, in
// whole passes of a CTA, and at most kChunk2 (the deposit window's sums).
__global__ void k2_finish(DevState* S, Dev2D* Dp, int G) {
  Dev2D& D = *Dp;
  __shared__ int wsum[32];
  const int s = blockIdx.x, T = D.T;
  const int* cnt = D.tile_cnt + s * T;
  int* wo = D.wi_off + s * (T + 1);
  const long long n = D.tile_start[s * (T + 1) + T];
  const long long want = (n / (2 * G) + kPass2 - 1) / kPass2;
  const int chunk = kPass2 * static_cast<int>(max(1LL, min(want, static_cast<long long>(kChunk2 / kPass2))));
  const int per = (T + blockDim.x - 1) / blockDim.x;
  const int t0 = min(static_cast<int>(threadIdx.x) * per, T), t1 = min(t0 + per, T);
  int a = 0;
  for (int t = t0; t < t1; ++t) a += (cnt[t] + chunk - 1) / chunk;
  int run = block_excl_scan(a, wsum);
  for (int t = t0; t < t1; ++t) {
    wo[t] = run;
    run += (cnt[t] + chunk - 1) / chunk;
  }
  if (threadIdx.x == blockDim.x - 1) wo[T] = run;
  if (threadIdx.x != 0) return;
  D.chunk[s] = chunk;
  void* t;
  t = S->xi[s]; S->xi[s] = S->xi_alt[s]; S->xi_alt[s] = t;
  t = S->u[s]; S->u[s] = S->u_alt[s]; S->u_alt[s] = t;
  t = D.y[s]; D.y[s] = D.y_alt[s]; D.y_alt[s] = t;
  t = D.w[s]; D.w[s] = D.w_alt[s]; D.w_alt[s] = t;
  if (s == CP_IONS) {
    uint32_t* ti = S->id;
    S->id = S->id_alt;
    S->id_alt = ti;
  }
  long long m = D.tile_start[s * (T + 1) + T];
  if (m > D.cap[s]) {
    m = D.cap[s] & ~3LL;
    atomicCAS(&S->status, 0, CP_ERR_CAPACITY);
  }
  D.n_sorted[s] = m;
  S->n_alloc[s] = m;
  S->n_proc[s] = m;
}

// ---------------------------------------------------------------------------
// Transverse transforms
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// Step's solve (row sums and transforms, modes, fields) at 1024 x 1024 cells:
// 113 -> 56 us launched one after the other, about 42 us in the graph (one
// launch fewer, modes beside the mean's solve).
//
// FFT of n = 2^log points (n >= 8), sign -1 forward (twiddles tw[k] =
// exp(-2 pi i k/n)), +1 inverse (conjugates): radix-2 decimation in time, its
// butterflies taken three stages at a time on eight values in registers, so
// that the points pass through shared memory every third stage only.
// Stage `half` joins (p, p + half) with twiddle (p mod half) n / (2 half).
//
// Thread t of n/8 starts with the points t + q n/8 (q = 0..7), which are the
// eight neighbours 8 b + r of the bit-reversed order, b = rev(t), r = rev3(q).

__device__ __forceinline__ int fft_pad(int i) { return i + (i >> 5); }  // spreads strides over the banks
__host__ __device__ constexpr int fft_words(int n) { return n + (n >> 5); }

__device__ __forceinline__ void butterfly(float2& a, float2& b, float2 w, bool inverse) {
  if (inverse) w.y = -w.y;
  const float2 u = a, v = cmul(b, w);
  a = make_float2(u.x + v.x, u.y + v.y);
  b = make_float2(u.x - v.x, u.y - v.y);
}

// STAGES stages from `half` on of the points v[r] = [.. + r half + pos]
template <int STAGES>
__device__ __forceinline__ void fft_stages(float2 (&v)[1 << STAGES], const float2* __restrict__ tw, int n, int half,
                                           int pos, bool inverse) {
#pragma unroll
  for (int g = 0; g < STAGES; ++g) {
    const int stride = n / (2 * half) >> g;
#pragma unroll
    for (int r = 0; r < (1 << STAGES); ++r) {
      if (r & (1 << g)) continue;
      const int k = (r & ((1 << g) - 1)) * half + pos;
      butterfly(v[r], v[r | (1 << g)], tw[k * stride], inverse);
    }
  }
}

// one pass of STAGES stages through shared memory
template <int STAGES>
__device__ __forceinline__ void fft_pass(float2* buf, const float2* __restrict__ tw, int n, int half, bool inverse) {
  constexpr int R = 1 << STAGES;
  for (int b = threadIdx.x; b < n / R; b += blockDim.x) {
    const int pos = b & (half - 1), base = (b - pos) * R + pos;
    float2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = buf[fft_pad(base + r * half)];
    fft_stages<STAGES>(v, tw, n, half, pos, inverse);
#pragma unroll
    for (int r = 0; r < R; ++r) buf[fft_pad(base + r * half)] = v[r];
  }
}

// The transform of the points load(c, q, j), j = t + q n/8 with t = tid + c
// kFftThreads (c < ROUNDS: 1 up to n = 1024, else 4), by all threads of the
// CTA; the result is in buf (fft_pad order) after the last barrier.
constexpr int kFftThreads = 128;

template <int ROUNDS, typename Load>
__device__ __forceinline__ void fft(float2* buf, const float2* __restrict__ tw, int n, int logn, bool inverse,
                                    Load load) {
#pragma unroll
  for (int c = 0; c < ROUNDS; ++c) {
    const int t = static_cast<int>(threadIdx.x) + c * kFftThreads;
    if (t < n / 8) {
      float2 v[8];
      // rev3(q) of q = 0..7
      v[0] = load(c, 0, t);
      v[4] = load(c, 1, t + n / 8);
      v[2] = load(c, 2, t + 2 * (n / 8));
      v[6] = load(c, 3, t + 3 * (n / 8));
      v[1] = load(c, 4, t + 4 * (n / 8));
      v[5] = load(c, 5, t + 5 * (n / 8));
      v[3] = load(c, 6, t + 6 * (n / 8));
      v[7] = load(c, 7, t + 7 * (n / 8));
      fft_stages<3>(v, tw, n, 1, 0, inverse);
      const int b = (logn > 3) ? static_cast<int>(__brev(static_cast<unsigned>(t)) >> (35 - logn)) : 0;
#pragma unroll
      for (int r = 0; r < 8; ++r) buf[fft_pad(8 * b + r)] = v[r];
    }
  }
  __syncthreads();
  int half = 8, left = logn - 3;
  for (; left >= 3; left -= 3, half *= 8) {
    fft_pass<3>(buf, tw, n, half, inverse);
    __syncthreads();
  }
  if (left == 2) fft_pass<2>(buf, tw, n, half, inverse);
  if (left == 1) fft_pass<1>(buf, tw, n, half, inverse);
  if (left) __syncthreads();
}

// Row i: exact row sum into the 1D grid, copy and clear, spectrum of the
// fluctuation (rows 1..Nx-1).  The row's charges stay in registers from the
// sum to the transform's first stages.
template <int ROUNDS>
__global__ void __launch_bounds__(kFftThreads) k2_fwd(const __grid_constant__ Dev2D D, long long* G1) {
  extern __shared__ float2 buf[];
  __shared__ long long wsum[kFftThreads / 32];
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  const int i = blockIdx.x;
  const int Ny = D.Ny, n8 = Ny / 8;
  long long* row = D.G2 + static_cast<long long>(i) * Ny;
  long long* last = D.G2last + static_cast<long long>(i) * Ny;
  long long g[ROUNDS][8];
  long long acc = 0;
#pragma unroll
  for (int c = 0; c < ROUNDS; ++c) {
    const int t = static_cast<int>(threadIdx.x) + c * kFftThreads;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      g[c][q] = (t < n8) ? __ldcg(&row[t + q * n8]) : 0;
      acc += g[c][q];
    }
  }
#pragma unroll
  for (int c = 0; c < ROUNDS; ++c) {
    const int t = static_cast<int>(threadIdx.x) + c * kFftThreads;
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (t < n8) {
        last[t + q * n8] = g[c][q];
        row[t + q * n8] = 0;
      }
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane_id() == 0) wsum[threadIdx.x >> 5] = acc;
  __syncthreads();
  long long tot = 0;
#pragma unroll
  for (int q = 0; q < kFftThreads / 32; ++q) tot += wsum[q];
  if (threadIdx.x == 0) G1[i] = tot;
  if (i == 0 || i == D.Nx) return;
  const double mean = static_cast<double>(tot) / static_cast<double>(Ny);
  fft<ROUNDS>(buf, D.tw, Ny, D.logNy, false, [&](int c, int q, int) {
    return make_float2(static_cast<float>((static_cast<double>(g[c][q]) - mean) * D.rho_scale), 0.0f);
  });
  float2* R = D.R + static_cast<long long>(i) * (Ny / 2 + 1);
  for (int k = threadIdx.x; k <= Ny / 2; k += kFftThreads) R[k] = buf[fft_pad(k)];
}

// One warp per mode k = 1..Ny/2: Thomas over i = 1..Nx-1 with phi = 0 at
// both ends for  Phi_{i-1} - (2 + kappa_k) Phi_i + Phi_{i+1} = -dx^2 R_i / eps0.
// The elimination factors depend on (i, k) only and are tabulated once
// (k2_tables).  Both substitutions are first-order linear recurrences,
// d_i = a_i d_{i-1} + b_i (a_i = -inv_i, b_i = c inv_i R_i) forward and
// x_i = -c'_i x_{i+1} + d_i backward; each lane composes the affine map of
// its segment of rows, a warp scan of the maps gives every segment its
// incoming value, and the lanes then apply their segments.
struct Aff {
  float a;
  float2 b;
};

__device__ __forceinline__ Aff aff_then(Aff f, Aff g) {  // g after f
  Aff h;
  h.a = g.a * f.a;
  h.b = make_float2(fmaf(g.a, f.b.x, g.b.x), fmaf(g.a, f.b.y, g.b.y));
  return h;
}

__device__ __forceinline__ Aff aff_shfl_up(Aff f, int o) {
  Aff r;
  r.a = __shfl_up_sync(0xffffffffu, f.a, o);
  r.b.x = __shfl_up_sync(0xffffffffu, f.b.x, o);
  r.b.y = __shfl_up_sync(0xffffffffu, f.b.y, o);
  return r;
}

constexpr int kModesCta = 4;  // modes (warps) per CTA; 2 above 2048 rows (shared memory)

// A mode's rows in shared memory, row i (from 0) at i + i/32: the lanes of a
// warp, each in its own segment of rows, mostly hit different banks.
__host__ __device__ constexpr int modes_at(int i) { return i + (i >> 5); }
__host__ __device__ constexpr int modes_rows(int n) { return modes_at(n) + 1; }

// W modes per CTA, one warp each; the CTA fetches the modes' rows together
// (neighbouring modes are neighbours in memory), eight loads per thread in
// flight, and the four sweeps run in shared memory.
template <int W>
__global__ void __launch_bounds__(32 * W) k2_modes(const __grid_constant__ Dev2D D, float c_rhs) {
  extern __shared__ float2 buf[];
  const int k0 = 1 + blockIdx.x * W;
  const int M = D.Ny / 2 + 1;
  const int nk = min(W, M - k0);
  const int lane = static_cast<int>(lane_id()), w = static_cast<int>(threadIdx.x) >> 5;
  const int n = D.Nx - 1;  // rows 1..n
  const int seg = (n + 31) / 32, S = modes_rows(n);
  float* tin = reinterpret_cast<float*>(buf + W * S);
  float* tcp = tin + W * S;
  const int m = static_cast<int>(threadIdx.x) % W;   // this thread's mode, and rows i0, i0 + 32, ...
  const int i0 = static_cast<int>(threadIdx.x) / W;
  const int mine = (m < nk) ? n : 0;
  const long long g0 = static_cast<long long>(1) * M + k0 + m;
  // the elimination factors do not change: fetched before the spectra are ready
  for (int j = i0; j < mine; j += 32 * 8) {
    float a[8], b[8];
#pragma unroll
    for (int c = 0; c < 8; ++c)
      if (j + 32 * c < mine) {
        a[c] = __ldg(&D.tinv[g0 + static_cast<long long>(j + 32 * c) * M]);
        b[c] = __ldg(&D.cp[g0 + static_cast<long long>(j + 32 * c) * M]);
      }
#pragma unroll
    for (int c = 0; c < 8; ++c)
      if (j + 32 * c < mine) {
        tin[m * S + modes_at(j + 32 * c)] = a[c];
        tcp[m * S + modes_at(j + 32 * c)] = b[c];
      }
  }
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  for (int j = i0; j < mine; j += 32 * 8) {
    float2 a[8];
#pragma unroll
    for (int c = 0; c < 8; ++c)
      if (j + 32 * c < mine) a[c] = __ldcg(&D.R[g0 + static_cast<long long>(j + 32 * c) * M]);
#pragma unroll
    for (int c = 0; c < 8; ++c)
      if (j + 32 * c < mine) buf[m * S + modes_at(j + 32 * c)] = a[c];
  }
  __syncthreads();
  if (w < nk) {
    const int r0 = min(n, lane * seg), r1 = min(n, r0 + seg);  // this lane's rows
    float2* r = buf + w * S;
    const float* inv = tin + w * S;
    const float* cp = tcp + w * S;
    // forward: compose this segment's map
    Aff f;
    f.a = 1.0f;
    f.b = make_float2(0.0f, 0.0f);
#pragma unroll 4
    for (int i = r0; i < r1; ++i) {
      const int q = modes_at(i);
      const float iv = inv[q];
      const float2 rr = r[q];
      Aff g;
      g.a = -iv;
      g.b = make_float2(c_rhs * iv * rr.x, c_rhs * iv * rr.y);
      f = aff_then(f, g);
    }
    // exclusive scan over the lanes: the map from d_0 = 0 to this segment's start
    Aff incl = f;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const Aff y = aff_shfl_up(incl, o);
      if (lane >= o) incl = aff_then(y, incl);
    }
    const Aff ex = aff_shfl_up(incl, 1);
    float2 d = (lane == 0) ? make_float2(0.0f, 0.0f) : ex.b;
    // forward: apply
#pragma unroll 4
    for (int i = r0; i < r1; ++i) {
      const int q = modes_at(i);
      const float iv = inv[q];
      const float2 rr = r[q];
      const float a = -iv;
      d = make_float2(fmaf(a, d.x, c_rhs * iv * rr.x), fmaf(a, d.y, c_rhs * iv * rr.y));
      r[q] = d;
    }
    // backward: x_i = -c'_i x_{i+1} + d_i, segments from the last row down
    Aff g;
    g.a = 1.0f;
    g.b = make_float2(0.0f, 0.0f);
#pragma unroll 4
    for (int i = r1 - 1; i >= r0; --i) {
      const int q = modes_at(i);
      Aff h;
      h.a = -cp[q];
      h.b = r[q];
      g = aff_then(g, h);
    }
    // reverse exclusive scan (lane 31 holds the last rows)
    Aff incl2 = g;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      Aff y;
      y.a = __shfl_down_sync(0xffffffffu, incl2.a, o);
      y.b.x = __shfl_down_sync(0xffffffffu, incl2.b.x, o);
      y.b.y = __shfl_down_sync(0xffffffffu, incl2.b.y, o);
      if (lane + o < 32) incl2 = aff_then(y, incl2);
    }
    const float bx = __shfl_down_sync(0xffffffffu, incl2.b.x, 1);
    const float by = __shfl_down_sync(0xffffffffu, incl2.b.y, 1);
    float2 x = (lane == 31) ? make_float2(0.0f, 0.0f) : make_float2(bx, by);
#pragma unroll 4
    for (int i = r1 - 1; i >= r0; --i) {
      const int q = modes_at(i);
      const float2 dd = r[q];
      const float cc = cp[q];
      x = make_float2(fmaf(-cc, x.x, dd.x), fmaf(-cc, x.y, dd.y));
      r[q] = x;
    }
  }
  __syncthreads();
  for (int i = i0; i < mine; i += 32) D.R[g0 + static_cast<long long>(i) * M] = buf[m * S + modes_at(i)];
}

// Row i: inverse transform of the mode solution and the fields,
//   E_x = E_0(x) + (phit_ij - phit_i+1,j)/dx, E_y = (phit_ij - phit_i,j+1)/dy
// (phit = 0 on both electrodes).  Row i + 1 is transformed here as well rather
// than fetched from its owner.
template <int ROUNDS>
__global__ void __launch_bounds__(kFftThreads) k2_fields(const __grid_constant__ Dev2D D,
                                                         const double* __restrict__ E64) {
  extern __shared__ float2 buf[];
  const int Ny = D.Ny, Nx = D.Nx, M = Ny / 2 + 1;
  const int i = blockIdx.x;
  float* p = reinterpret_cast<float*>(buf + fft_words(Ny));  // rows i and i + 1
  const float inv_n = 1.0f / static_cast<float>(Ny);
  for (int c = 0; c < 2; ++c) {
    if (i + c > 0 && i + c < Nx) {
      const float2* R = D.R + static_cast<long long>(i + c) * M;
      fft<ROUNDS>(buf, D.tw, Ny, D.logNy, true, [&](int, int, int k) {
        float2 v = make_float2(0.0f, 0.0f);
        if (k > 0) {
          const float2 q = __ldcg(&R[k < M ? k : Ny - k]);
          v = make_float2(q.x, k < M ? q.y : -q.y);
          if (k == Ny / 2) v.y = 0.0f;
        }
        return v;
      });
      for (int j = threadIdx.x; j < Ny; j += kFftThreads) p[c * Ny + j] = buf[fft_pad(j)].x * inv_n;
    } else {
      for (int j = threadIdx.x; j < Ny; j += kFftThreads) p[c * Ny + j] = 0.0f;
    }
    __syncthreads();
  }
  const long long r = static_cast<long long>(i) * Ny;
  const float E0 = (i < Nx) ? static_cast<float>(E64[i]) : 0.0f;
  for (int j = threadIdx.x; j < Ny; j += kFftThreads) {
    const float v = p[j];
    const int j1 = (j + 1 == Ny) ? 0 : j + 1;
    D.phit[r + j] = v;
    D.Ey[r + j] = (v - p[j1]) * D.inv_dy;
    if (i < Nx) D.Ex[r + j] = E0 + (v - p[Ny + j]) * D.inv_dx;
  }
}

__global__ void k2_tables(Dev2D* Dp, double r2) {
  Dev2D& D = *Dp;
  const int Ny = D.Ny, M = Ny / 2 + 1;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < M; k += gridDim.x * blockDim.x) {
    double sn, cs;
    sincospi(2.0 * k / Ny, &sn, &cs);
    const double kap = r2 * (2.0 - 2.0 * cs);
    D.kappa[k] = static_cast<float>(kap);
    if (k < Ny / 2) D.tw[k] = make_float2(static_cast<float>(cs), static_cast<float>(-sn));
    // Thomas elimination of mode k: inv_i = 1/(b - c'_{i-1}), c'_i = inv_i (last row 0)
    const double bk = -(2.0 + kap);
    double cprev = 0.0;
    for (int i = 1; i < D.Nx; ++i) {
      const double iv = 1.0 / (bk - cprev);
      const double c = (i + 1 < D.Nx) ? iv : 0.0;
      D.tinv[static_cast<long long>(i) * M + k] = static_cast<float>(iv);
      D.cp[static_cast<long long>(i) * M + k] = static_cast<float>(c);
      cprev = c;
    }
  }
}

// ---------------------------------------------------------------------------
// Host-side launchers
// ---------------------------------------------------------------------------
constexpr size_t kCwinBytes = sizeof(Window2);

cudaError_t push2_occupancy(int* per_sm) {
  const cudaError_t e = cudaFuncSetAttribute(k2_push, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(kCwinBytes));
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, k2_push, kThreads2, kCwinBytes);
}

cudaError_t push2_launch(const DevParams* P, DevState* S, void* D, const void* D_host, void* abs,
                         int abs_cap, int grid, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3(kThreads2, 1, 1);
  cfg.dynamicSmemBytes = kCwinBytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k2_push, P, S, static_cast<const Dev2D*>(D),
                            *static_cast<const Dev2D*>(D_host), static_cast<Dev2D*>(D)->item_ctr,
                            static_cast<AbsRec2*>(abs), abs_cap);
}

cudaError_t sort2_launch(DevState* S, void* D, int T, int sms, cudaStream_t st) {
  Dev2D* Dp = static_cast<Dev2D*>(D);
  const size_t hs = sizeof(int) * T;
  const int G = 2 * sms;  // must match the blocks the per-block histograms were sized for
  k2_hist<<<dim3(G, kSpecies), 512, hs, st>>>(S, Dp);
  k2_tilescan<<<dim3(T, kSpecies), 128, 0, st>>>(Dp, G);
  k2_scan<<<kSpecies, 1024, 0, st>>>(S, Dp);
  k2_scatter<<<dim3(G, kSpecies), 512, hs, st>>>(S, Dp);
  k2_finish<<<kSpecies, 1024, 0, st>>>(S, Dp, G);
  return cudaGetLastError();
}

static cudaLaunchConfig_t pdl_config(int grid, int threads, size_t smem, cudaStream_t st,
                                     cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

static int modes_per_cta(int Nx) { return Nx > 2048 ? kModesCta / 2 : kModesCta; }

static size_t modes_smem(int Nx) {
  return (sizeof(float2) + 2 * sizeof(float)) * modes_per_cta(Nx) * modes_rows(Nx - 1);
}

static size_t fields_smem(int Ny) { return sizeof(float2) * fft_words(Ny) + 2 * sizeof(float) * Ny; }

// The kernels' shared-memory limits (the largest any grid needs: contexts
// share the kernels).
cudaError_t solve2_configure() {
  const int most = static_cast<int>(sizeof(int)) * (4096 / kT2) * (4096 / kT2);  // the sort's tile counters
  cudaError_t es = cudaFuncSetAttribute(k2_hist, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (es == cudaSuccess) es = cudaFuncSetAttribute(k2_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (es != cudaSuccess) return es;
  cudaError_t e = cudaFuncSetAttribute(k2_modes<kModesCta>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(modes_smem(2048)));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k2_modes<kModesCta / 2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(modes_smem(4096)));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k2_fields<4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(fields_smem(4096)));
}

cudaError_t solve2_fwd_launch(const void* D_host, long long* G1, int Nx, int Ny, cudaStream_t st) {
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = pdl_config(Nx + 1, kFftThreads, sizeof(float2) * fft_words(Ny), st, attr);
  const Dev2D& D = *static_cast<const Dev2D*>(D_host);
  return Ny <= 8 * kFftThreads ? cudaLaunchKernelEx(&cfg, k2_fwd<1>, D, G1) : cudaLaunchKernelEx(&cfg, k2_fwd<4>, D, G1);
}

cudaError_t solve2_modes_launch(const void* D_host, int Nx, int Ny, float c_rhs, cudaStream_t st) {
  const int W = modes_per_cta(Nx), M = Ny / 2;
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = pdl_config((M + W - 1) / W, 32 * W, modes_smem(Nx), st, attr);
  const Dev2D& D = *static_cast<const Dev2D*>(D_host);
  return W == kModesCta ? cudaLaunchKernelEx(&cfg, k2_modes<kModesCta>, D, c_rhs)
                        : cudaLaunchKernelEx(&cfg, k2_modes<kModesCta / 2>, D, c_rhs);
}

// One row per CTA: it transforms its successor's too, and the many small CTAs
// hide each other's latency (step at 1024 x 1024 cells: 252.6 us, two rows
// 251.5, three 255.5; at 96 x 128: 37.5, two rows 39.0).
cudaError_t solve2_fields_launch(const void* D_host, int Nx, int Ny, const double* E64, cudaStream_t st) {
  const Dev2D& D = *static_cast<const Dev2D*>(D_host);
  if (Ny <= 8 * kFftThreads) k2_fields<1><<<Nx + 1, kFftThreads, fields_smem(Ny), st>>>(D, E64);
  else k2_fields<4><<<Nx + 1, kFftThreads, fields_smem(Ny), st>>>(D, E64);
  return cudaGetLastError();
}

cudaError_t deposit2_level0_launch(DevState* S, const void* D, int sms, cudaStream_t st) {
  for (int s = 0; s < kSpecies; ++s)
    k2_deposit0<<<2 * sms, 512, 0, st>>>(S, static_cast<const Dev2D*>(D), s);
  return cudaGetLastError();
}

cudaError_t tables2_launch(void* D, int Ny, double r2, cudaStream_t st) {
  k2_tables<<<(Ny / 2 + 128) / 128, 128, 0, st>>>(static_cast<Dev2D*>(D), r2);
  return cudaGetLastError();
}

}  // namespace cpk
