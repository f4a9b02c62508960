// Many right-hand sides on one mesh (cdg_solve_multi): the same V-cycle
// preconditioned CG run for R columns at once.  Vectors are [n_l][n_p][R]
// (the R columns of one element's coefficient i are contiguous), so one block
// of an operator is read once per tile of columns: a CTA owns one to four
// block rows and a tile of columns, stages the rows' blocks in shared memory,
// and each thread applies them to one, two or four columns of the tile (the
// autotuner picks the shape).  The outer CG (residual, dots, updates, the
// level-0 operator) is FP64 with per-column scalars, its vector passes fused
// (the update also writes the FP32 copy of r for the V-cycle and the partial
// sums of r.r); the V-cycle runs on FP32 arithmetic on FP32 copies of the
// level operators, or (precision 2) on BF16 copies of the row-scaled smoother
// blocks D^-1(A - D) and of the transfer blocks (the residual operator and the
// block inverses stay FP32).  The level-0 operator can also run on the tensor
// cores by exact splitting (device_ozaki.cu).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "device_fixed.cuh"
#include "device_kernels.cuh"
#include "device_state.h"

namespace {

using cdgk::cvt;
using cdgk::f32_to_f64;
using cdgk::f64_to_f32;

template <typename T>
struct Conv;
template <>
struct Conv<double> {
  static __device__ __forceinline__ double f(double v) { return v; }
};
template <>
struct Conv<float> {
  static __device__ __forceinline__ float f(float v) { return v; }
};
template <>
struct Conv<__nv_bfloat16> {
  static __device__ __forceinline__ float f(__nv_bfloat16 v) { return __bfloat162float(v); }
};

// the threads of one row group (threadIdx.y) copy ne values into shared memory
template <typename TA, typename TC>
__device__ __forceinline__ void stage_block(TC* s, const TA* a, int ne) {
  for (int t = threadIdx.x; t < ne; t += blockDim.x) s[t] = (TC)Conv<TA>::f(a[t]);
}

// V consecutive right-hand sides of one coefficient, aligned for one load
template <int V>
struct Cols;
template <>
struct Cols<1> {
  static __device__ __forceinline__ void load(const float* p, float* v) { v[0] = *p; }
  static __device__ __forceinline__ void store(float* p, const float* v) { *p = v[0]; }
};
template <>
struct Cols<2> {
  static __device__ __forceinline__ void load(const float* p, float* v) {
    const float2 t = *reinterpret_cast<const float2*>(p);
    v[0] = t.x, v[1] = t.y;
  }
  static __device__ __forceinline__ void store(float* p, const float* v) {
    *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
  }
};
template <>
struct Cols<4> {
  static __device__ __forceinline__ void load(const float* p, float* v) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x, v[1] = t.y, v[2] = t.z, v[3] = t.w;
  }
  static __device__ __forceinline__ void store(float* p, const float* v) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  }
};

// y = b - A x (MODE 1), y = x + omega (b - x - A x) (3; A = Ahat, b = D^-1 b), FP32; the restriction
// y_A = sum_K L_K^T x_K over A's children (8: block t meets element t); and with one block per row (no
// rowptr), x from element col[K] (nullptr: K): y += A x (4), y = A x and y2 = omega A x (6), y = A x (7).
// A warp owns one block row and a tile of 32 V right-hand sides, V consecutive ones per lane (R is a
// multiple of V: the vectors start on 256-byte boundaries and a coefficient's columns on multiples of
// 4 R bytes); warps share nothing, so nothing waits on another warp.  It copies up to four of the row's
// blocks at once into shared memory; PF starts the gather of the next block's x before the products of
// this one.  What bounds the kernel is the latency of the x gathers: the CTA-wide form before it, two
// barriers per block with the gathers behind them, moved its 638 MB (20,000 rows, n_p = 10, R = 256) in
// 179 us, 0.52 of the copy rate; this one takes 153 us.  V, PF and the warps per CTA are autotuned; every choice sums a
// column in the same order.
constexpr int kMrMaxBR = 4;
constexpr int kMrStage = 4;

template <int V, bool PF>
constexpr int mr_min_ctas() { return V == 4 ? 3 : V == 2 ? (PF ? 5 : 6) : 8; }

template <typename TA, int NP, int MODE, int V, bool PF>
__global__ void __launch_bounds__(128, mr_min_ctas<V, PF>()) mr_row_kernel(int n, int R, const int* __restrict__ rowptr,
                                                                        const int* __restrict__ col,
                                                                        const TA* __restrict__ A,
                                                                        const float* __restrict__ x,
                                                                        const float* __restrict__ b,
                                                                        float* y, float* __restrict__ y2,
                                                                        float omega) {
  constexpr bool ONE = MODE == 4 || MODE == 6 || MODE == 7;
  constexpr int STAGE = ONE ? 1 : kMrStage;
  constexpr int NN = NP * NP, SZ = (NN + 3) / 4 * 4;
  __shared__ __align__(16) float as_s[kMrMaxBR][STAGE * SZ];
  float* as = as_s[threadIdx.y];
  const int K = blockIdx.x * blockDim.y + threadIdx.y;
  const int lane = threadIdx.x;
  const int r = (blockIdx.y * 32 + lane) * V;
  if (K >= n) return;   // a whole warp
  const bool on = r < R;
  const int b0 = ONE ? K : rowptr[K], b1 = ONE ? K + 1 : rowptr[K + 1];
  float acc[NP][V];
#pragma unroll
  for (int i = 0; i < NP; ++i)
#pragma unroll
    for (int c = 0; c < V; ++c) acc[i][c] = 0.f;
  auto gather = [&](int t, float (&v)[NP][V]) {
    const int J = MODE == 8 || (ONE && !col) ? t : col[t];
    const float* xj = x + (size_t)J * NP * R + r;
#pragma unroll
    for (int j = 0; j < NP; ++j) Cols<V>::load(xj + (size_t)j * R, v[j]);
  };
  auto products = [&](const float* a, const float (&v)[NP][V]) {
#pragma unroll
    for (int q = 0; q < SZ / 4; ++q) {
      const float4 a4 = reinterpret_cast<const float4*>(a)[q];
      const float e[4] = {a4.x, a4.y, a4.z, a4.w};
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (4 * q + k < NN) {
          const int row = (4 * q + k) / NP, cl = (4 * q + k) % NP;   // entry of the stored block
          const int i = MODE == 8 ? cl : row, j = MODE == 8 ? row : cl;
#pragma unroll
          for (int c = 0; c < V; ++c) acc[i][c] = fmaf(e[k], v[j][c], acc[i][c]);
        }
    }
  };
  for (int t0 = b0; t0 < b1; t0 += STAGE) {
    const int cnt = min(STAGE, b1 - t0);
    float xa[NP][V], xb[NP][V];
    if (on) gather(t0, xa);
    __syncwarp();
    for (int u = lane; u < cnt * NN; u += 32) {
      const int blk = SZ == NN ? 0 : u / NN;
      as[blk * (SZ - NN) + u] = Conv<TA>::f(A[(size_t)t0 * NN + u]);
    }
    __syncwarp();
    if (on) {
#pragma unroll
      for (int t = 0; t < STAGE; t += 2) {
        if (t < cnt) {
          if (PF && t + 1 < cnt) gather(t0 + t + 1, xb);
          products(as + t * SZ, xa);
        }
        if (t + 1 < cnt) {
          if (!PF) gather(t0 + t + 1, xb);
          if (PF && t + 2 < cnt) gather(t0 + t + 2, xa);
          products(as + (t + 1) * SZ, xb);
          if (!PF && t + 2 < cnt) gather(t0 + t + 2, xa);
        }
      }
    }
  }
  if (!on) return;
  const size_t base = (size_t)K * NP * R + r;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    const size_t o = base + (size_t)i * R;
    float v[V], xv[V];
    if constexpr (MODE == 1 || MODE == 3) Cols<V>::load(b + o, v);
    if constexpr (MODE == 3) Cols<V>::load(x + o, xv);
    if constexpr (MODE == 4) Cols<V>::load(y + o, v);
#pragma unroll
    for (int c = 0; c < V; ++c) {
      if constexpr (MODE == 1) v[c] -= acc[i][c];
      else if constexpr (MODE == 3) v[c] = xv[c] + omega * (v[c] - xv[c] - acc[i][c]);
      else if constexpr (MODE == 4) v[c] += acc[i][c];
      else v[c] = acc[i][c];
    }
    Cols<V>::store(y + o, v);
    if constexpr (MODE == 6) {
#pragma unroll
      for (int c = 0; c < V; ++c) v[c] *= omega;
      Cols<V>::store(y2 + o, v);
    }
  }
}

// y = A_0 x in FP64 by integer digits (device_fixed.cu says why and how): a warp owns one block row and
// 32 right-hand sides, one per lane.  A lane splits the n_p values of its column in a block's neighbour
// (one exponent for them) and keeps the n_p sums, each with its scale, in registers; the digits of a
// block are read from shared memory, each 16 bytes feeding eight integer multiply-adds.  5,000 rows,
// n_p = 6, 40 columns: 82 us with FP64 multiply-adds (46 us at the FP64 rate), 61 us here.
template <int NP>
__global__ void __launch_bounds__(128, 4) mr_fx_kernel(int n, int R, const int* __restrict__ rowptr,
                                                       const int* __restrict__ col, const int2* __restrict__ A,
                                                       const unsigned short* __restrict__ EA,
                                                       const double* __restrict__ x, double* __restrict__ y) {
  constexpr int NN = NP * NP;
  __shared__ __align__(16) int2 as_s[kMrMaxBR][(NN + 1) / 2 * 2];
  __shared__ int ea_s[kMrMaxBR][NP];
  int2* as = as_s[threadIdx.y];
  int* ea = ea_s[threadIdx.y];
  const int K = blockIdx.x * blockDim.y + threadIdx.y;
  const int lane = threadIdx.x;
  const int r = blockIdx.y * 32 + lane;
  if (K >= n) return;   // a whole warp
  const bool on = r < R;
  const int b0 = rowptr[K], b1 = rowptr[K + 1];
  bool special = false;
  unsigned bad_rows = 0;
  fx::Wide acc[NP];
  int E[NP];
#pragma unroll
  for (int i = 0; i < NP; ++i) E[i] = fx::kNoScale;
  for (int t = b0; t < b1; ++t) {
    __syncwarp();
    for (int u = lane; u < NN; u += 32) as[u] = A[(size_t)t * NN + u];
    if (lane < NP) ea[lane] = EA[(size_t)t * NP + lane];
    int2 xd[NP];
    int em = 1;
    if (on) {
      const double* xj = x + (size_t)col[t] * NP * R + r;
      double xv[NP];
#pragma unroll
      for (int j = 0; j < NP; ++j) xv[j] = xj[(size_t)j * R];
#pragma unroll
      for (int j = 0; j < NP; ++j) em = max(em, fx::biased_exponent(xv[j]));
#pragma unroll
      for (int j = 0; j < NP; ++j) xd[j] = fx::split_digits(xv[j], em);
    }
    __syncwarp();
    if (on) {
      special |= em == fx::kNotFinite;
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        fx::Acc s;
        if constexpr (NP % 2 == 0) {
          const int4* a4 = reinterpret_cast<const int4*>(as) + i;
#pragma unroll
          for (int j = 0; j < NP; j += 2) {
            const int4 d = a4[(j >> 1) * NP];
            fx::mac(s, d.x, d.y, xd[j].x, xd[j].y);
            fx::mac(s, d.z, d.w, xd[j + 1].x, xd[j + 1].y);
          }
        } else {
#pragma unroll
          for (int j = 0; j < NP; ++j) {
            const int2 d = as[j * NP + i];
            fx::mac(s, d.x, d.y, xd[j].x, xd[j].y);
          }
        }
        s.carry();
        if (ea[i] == fx::kNotFinite) bad_rows |= 1u << i;
        const int e = ea[i] + em + fx::kHead;
        if (e > E[i]) {
          acc[i].down(e - E[i]);
          E[i] = e;
        }
        fx::Wide w = s.wide();
        w.down(E[i] - e + fx::kHead);
        acc[i].add(w);
      }
    }
  }
  if (!on) return;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    double v = fx::fx_value(acc[i].hi, acc[i].lo, E[i] - fx::kScale);
    if (special) {   // an infinity or NaN in the column: FP64 products
      v = 0.0;
      for (int t = b0; t < b1; ++t) {
        const int e = EA[(size_t)t * NP + i] - 1022 - 58;
        for (int j = 0; j < NP; ++j) {
          const int2 d = A[(size_t)t * NN + fx::fx_pos(NP, i, j)];
          v = fma(fx::scale2(__ll2double_rn(((long long)d.x << 30) + d.y), e), x[((size_t)col[t] * NP + j) * R + r], v);
        }
      }
    }
    if (bad_rows >> i & 1) v = nan("");
    y[((size_t)K * NP + i) * R + r] = v;
  }
}

// coarsest (one mesh): x[row][r] = sum_j Ainv[row][j] b[j][r], FP64 accumulation.  A CTA owns
// kCoarseRows rows and 32 columns; its eight warps share the j (each b value is widened once per
// kCoarseRows rows) and their sums are added in order.  With one warp per 32 columns walking all j,
// 228 unknowns x 40 columns kept 114 warps busy for 84 us (5 us at the FP64 rate).
constexpr int kCoarseRows = 4;
constexpr int kCoarseWarps = 8;

template <typename TV>
__global__ void __launch_bounds__(32 * kCoarseWarps) mr_coarse_kernel(int nc, int R, const double* __restrict__ Ainv,
                                                                      const TV* __restrict__ b, TV* __restrict__ x) {
  __shared__ double part[kCoarseWarps][kCoarseRows][32];
  const int row0 = blockIdx.x * kCoarseRows;
  const int lane = threadIdx.x, w = threadIdx.y;
  const int r = blockIdx.y * 32 + lane;
  const int j0 = nc * w / kCoarseWarps, j1 = nc * (w + 1) / kCoarseWarps;
  double s[kCoarseRows];
#pragma unroll
  for (int q = 0; q < kCoarseRows; ++q) s[q] = 0.0;
  if (r < R) {
#pragma unroll 4
    for (int j = j0; j < j1; ++j) {
      const double bv = cvt<double>(b[(size_t)j * R + r]);
#pragma unroll
      for (int q = 0; q < kCoarseRows; ++q)
        s[q] = fma(Ainv[(size_t)min(row0 + q, nc - 1) * nc + j], bv, s[q]);
    }
  }
#pragma unroll
  for (int q = 0; q < kCoarseRows; ++q) part[w][q][lane] = s[q];
  __syncthreads();
  if (w < kCoarseRows && row0 + w < nc && r < R) {
    double t = 0.0;
    for (int k = 0; k < kCoarseWarps; ++k) t += part[k][w][lane];
    x[(size_t)(row0 + w) * R + r] = cvt<TV>(t);
  }
}

template <typename TI, typename TO>
__global__ void mr_convert_kernel(size_t n, const TI* __restrict__ a, TO* __restrict__ b) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    b[i] = cvt<TO>(a[i]);
}

// The per-column vector kernels of the outer CG share one partition: row group g
// of G = gridDim.x blockDim.y (threadIdx.y of its CTA) owns rows
// [nrows g / G, nrows (g + 1) / G) and thread x one column, so a column's partial
// sums run over its rows in ascending order whichever kernel forms them.  Rows go
// four at a time, all loads of a group before its arithmetic, to keep enough
// loads in flight per thread; with few columns a CTA holds several row groups
// (40 columns, 30,000 rows, one group of 64 threads per CTA: update 42.6 us for
// 62 MB).
__device__ __forceinline__ void mr_rows(int nrows, int G, int g, int& lo, int& hi) {
  lo = (int)((long long)nrows * g / G);
  hi = (int)((long long)nrows * (g + 1) / G);
}

// per-column partial dots over a chunk of rows: partial[g][r] = sum x y; Y is FP64 or FP32 (a
// V-cycle output, widened exactly)
template <typename TY>
__global__ void mr_dot_kernel(int nrows, int R, int G, const double* __restrict__ x, const TY* __restrict__ y,
                              double* __restrict__ partial) {
  const int g = blockIdx.x * blockDim.y + threadIdx.y, r = threadIdx.x;
  if (r >= R) return;
  int lo, hi;
  mr_rows(nrows, G, g, lo, hi);
  double s = 0.0;
  int row = lo;
  for (; row + 4 <= hi; row += 4) {
    // all loads of the group first (raw words), conversions after: a
    // conversion's branch between two loads would keep them from overlapping
    double xv[4];
    TY yv[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const size_t o = (size_t)(row + u) * R + r;
      xv[u] = x[o];
      yv[u] = y[o];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) s = fma(xv[u], cvt<double>(yv[u]), s);
  }
  for (; row < hi; ++row) {
    const size_t o = (size_t)row * R + r;
    s = fma(x[o], cvt<double>(y[o]), s);
  }
  partial[(size_t)g * R + r] = s;
}

// per column: the sum of the G partials, and that column's CG scalars (same rules as the
// single-column finalize: which 0 PQ, 1 RR, 2 RZ, 3 BB, 4 initial RR).  A CTA owns four columns, 64
// threads each share a column's partials, and their sums are added in a fixed order.  Few columns per
// CTA, since an SM's FP64 pipe adds only two numbers per clock (32 columns per CTA: 11.8 us); one
// thread per column walking its 304 partials took 54 us.
constexpr int kFinCols = 4;
constexpr int kFinThreads = 256;

__global__ void __launch_bounds__(kFinThreads) mr_finalize_kernel(int R, int G, const double* __restrict__ partial,
                                                                    int which, double tol,
                                                                    double* __restrict__ scal) {
  __shared__ double part[2][kFinThreads / 32][kFinCols];
  const int c = threadIdx.x % kFinCols, seg = threadIdx.x / kFinCols;
  const int r = blockIdx.x * kFinCols + c;
  const bool two = which == 1;   // r.r and the new r times the previous z
  double s = 0.0, s2 = 0.0;
  if (r < R)
    for (int g = seg; g < G; g += kFinThreads / kFinCols) {
      s += partial[(size_t)g * R + r];
      if (two) s2 += partial[(size_t)(G + g) * R + r];
    }
  for (int o = kFinCols; o < 32; o *= 2) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    if (two) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
  }
  if ((threadIdx.x & 31) < kFinCols) {
    part[0][threadIdx.x >> 5][c] = s;
    part[1][threadIdx.x >> 5][c] = s2;
  }
  __syncthreads();
  if (threadIdx.x >= kFinCols || r >= R) return;
  double tot = 0.0, tot2 = 0.0;
  for (int w = 0; w < kFinThreads / 32; ++w) {
    tot += part[0][w][c];
    tot2 += part[1][w][c];
  }
  double* sc = scal + (size_t)r * S_COUNT;
  const bool done = sc[S_DONE] != 0.0;
  if (which == 0) {
    sc[S_PQ] = tot;
    if (!done && !(tot > 0.0)) {
      sc[S_BREAK] = 1.0;
      sc[S_DONE] = 1.0;
    }
    sc[S_ALPHA] = sc[S_DONE] != 0.0 ? 0.0 : sc[S_RZ] / tot;
  } else if (which == 1 || which == 4) {
    if (!done) {
      sc[S_RR] = tot;
      sc[S_RZO] = tot2;
      if (which == 1) sc[S_IT] += 1.0;
      if (!isfinite(tot)) {
        sc[S_BREAK] = 1.0;
        sc[S_DONE] = 1.0;
      } else if (sqrt(tot) <= tol * sqrt(sc[S_BB])) {
        sc[S_DONE] = 1.0;
      }
    }
  } else if (which == 2) {   // flexible CG; unused by the first p
    sc[S_BETA] = done ? 0.0 : (tot - sc[S_RZO]) / sc[S_RZ];
    sc[S_RZ] = tot;
  } else {
    sc[S_BB] = tot;
    if (!(tot > 0.0)) sc[S_DONE] = 1.0;
  }
}

// x += alpha_r p; r -= alpha_r q per column, with the FP32 copy of r that the V-cycle reads and the
// chunk's partial sums of r.r and (G rows further) of r times z, the V-cycle's last output: the flexible
// beta needs that product, and taken here the V-cycle may overwrite z
__global__ void mr_update_kernel(int nrows, int R, int G, const double* __restrict__ scal,
                                 const double* __restrict__ p, const double* __restrict__ q, double* __restrict__ x,
                                 double* __restrict__ res, float* __restrict__ r32, const float* __restrict__ z,
                                 double* __restrict__ partial) {
  const int g = blockIdx.x * blockDim.y + threadIdx.y, r = threadIdx.x;
  if (r >= R) return;
  int lo, hi;
  mr_rows(nrows, G, g, lo, hi);
  const double a = scal[(size_t)r * S_COUNT + S_ALPHA];
  double s = 0.0, s2 = 0.0;
  int row = lo;
  for (; row + 4 <= hi; row += 4) {
    double pv[4], qv[4], xv[4], rv[4];
    float zv[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const size_t o = (size_t)(row + u) * R + r;
      pv[u] = p[o];
      qv[u] = q[o];
      xv[u] = x[o];
      rv[u] = res[o];
      zv[u] = z[o];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const size_t o = (size_t)(row + u) * R + r;
      x[o] = fma(a, pv[u], xv[u]);
      const double v = fma(-a, qv[u], rv[u]);
      res[o] = v;
      r32[o] = f64_to_f32(v);
      s = fma(v, v, s);
      s2 = fma(v, f32_to_f64(zv[u]), s2);
    }
  }
  for (; row < hi; ++row) {
    const size_t o = (size_t)row * R + r;
    x[o] = fma(a, p[o], x[o]);
    const double v = fma(-a, q[o], res[o]);
    res[o] = v;
    r32[o] = f64_to_f32(v);
    s = fma(v, v, s);
    s2 = fma(v, f32_to_f64(z[o]), s2);
  }
  partial[(size_t)g * R + r] = s;
  partial[(size_t)(G + g) * R + r] = s2;
}

// p = z + beta_r p per column (p = z on the first step); z is the V-cycle's FP32 output.
// With maxb, also the largest biased FP64 exponent of each column of the new p
// (atomicMax over the CTAs; maxb zeroed before), which the split apply needs
__device__ __forceinline__ int biased_exp(double v) {
  return (int)(((unsigned long long)__double_as_longlong(v) >> 52) & 0x7FF);
}

__global__ void mr_p_kernel(int nrows, int R, int G, const double* __restrict__ scal, int first,
                            const float* __restrict__ z, double* __restrict__ p, int* __restrict__ maxb) {
  const int g = blockIdx.x * blockDim.y + threadIdx.y, r = threadIdx.x;
  if (r >= R) return;
  int lo, hi;
  mr_rows(nrows, G, g, lo, hi);
  const double beta = first ? 0.0 : scal[(size_t)r * S_COUNT + S_BETA];
  int em = 0;
  int row = lo;
  for (; row + 4 <= hi; row += 4) {
    float zv[4];   // raw words first, conversions after (see mr_dot_kernel)
    double pv[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const size_t o = (size_t)(row + u) * R + r;
      zv[u] = z[o];
      pv[u] = first ? 0.0 : p[o];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const double zo = f32_to_f64(zv[u]);
      const double v = first ? zo : fma(beta, pv[u], zo);
      p[(size_t)(row + u) * R + r] = v;
      em = max(em, biased_exp(v));
    }
  }
  for (; row < hi; ++row) {
    const size_t o = (size_t)row * R + r;
    const double zo = f32_to_f64(z[o]);
    const double v = first ? zo : fma(beta, p[o], zo);
    p[o] = v;
    em = max(em, biased_exp(v));
  }
  if (maxb) atomicMax(maxb + r, em);
}

// Single-graph solve: columns converged before the loop are closed, the counters start at zero
__global__ void mr_open_kernel(int R, double* __restrict__ scal, int* __restrict__ it_dev, int* __restrict__ iters) {
  for (int r = threadIdx.x; r < R; r += blockDim.x) {
    scal[(size_t)r * S_COUNT + S_HDONE] = scal[(size_t)r * S_COUNT + S_DONE];
    iters[r] = 0;
  }
  if (threadIdx.x == 0) *it_dev = 0;
}

// Single-graph solve, after the residual norms of an iteration: its entry in the history and the
// iteration count of every open column (one closes in the iteration it converges or breaks down), and
// whether to go on: a column is open, there are iterations left and no device wait has expired.
__global__ void mr_check_kernel(cudaGraphConditionalHandle cond, int R, int maxit, double* __restrict__ scal,
                                int* __restrict__ it_dev, double* __restrict__ hist, int* __restrict__ iters,
                                const int* __restrict__ wait_err) {
  const int it = *it_dev + 1;
  int open = 0;
  for (int r = threadIdx.x; r < R; r += blockDim.x) {
    double* sc = scal + (size_t)r * S_COUNT;
    if (sc[S_HDONE] != 0.0) continue;
    hist[(size_t)r * (maxit + 1) + it] = sc[S_BB] > 0.0 ? sqrt(sc[S_RR] / sc[S_BB]) : 0.0;
    iters[r] = it;
    if (sc[S_DONE] != 0.0) sc[S_HDONE] = 1.0;
    else open = 1;
  }
  open = __syncthreads_or(open);
  if (threadIdx.x == 0) {
    *it_dev = it;
    cudaGraphSetConditional(cond, (open && it < maxit && *wait_err == 0) ? 1u : 0u);
  }
}

// b[k][i][r] = sum_q w_q phi_i(x_q) f[r][K][q], K = perm0[k]  (f only; zero boundary data)
template <int NP>
__global__ void mr_rhs_kernel(int R, int nq, int ne, const int* __restrict__ perm0, const double* __restrict__ V,
                              const double* __restrict__ f, double* __restrict__ b) {
  const int k = blockIdx.x, r = threadIdx.x;
  if (r >= R) return;
  const size_t K = perm0[k];
  const double* fk = f + ((size_t)r * ne + K) * nq;
  const double* Vk = V + (size_t)k * nq * NP;
  double s[NP];
#pragma unroll
  for (int i = 0; i < NP; ++i) s[i] = 0.0;
  for (int q = 0; q < nq; ++q) {
    const double fv = fk[q];
#pragma unroll
    for (int i = 0; i < NP; ++i) s[i] = fma(Vk[q * NP + i], fv, s[i]);
  }
#pragma unroll
  for (int i = 0; i < NP; ++i) b[((size_t)k * NP + i) * R + r] = s[i];
}

// u[r][K][i] = x[k][i][r] (user layout: one contiguous solution per column)
__global__ void mr_out_kernel(int R, int np, const int* __restrict__ perm0, const double* __restrict__ x,
                              int ne, double* __restrict__ u) {
  const int k = blockIdx.x, r = threadIdx.x;
  if (r >= R) return;
  const size_t K = perm0[k];
  for (int i = 0; i < np; ++i) u[((size_t)r * ne + K) * np + i] = x[((size_t)k * np + i) * R + r];
}

}  // namespace

struct MRLevel {
  void* A = nullptr;      // V-cycle operator copies (FP32 or BF16)
  void* Ahat = nullptr;
  void* Dinv = nullptr;
  void* L = nullptr;
  float *x = nullptr, *t = nullptr, *r = nullptr, *b = nullptr, *bh = nullptr;
};

struct MR {
  int R = 0, G = 0;             // columns; row groups of the vector kernels
  int rows_per_cta = 1;         // row groups per CTA
  bool bf16 = false;
  MRLevel lev[kMaxLev];
  double *x = nullptr, *r = nullptr, *p = nullptr, *q = nullptr, *bt = nullptr;
  float *r32 = nullptr, *z32 = nullptr;   // FP32 V-cycle input and output
  double* scal = nullptr;      // [R][S_COUNT]
  double* partial = nullptr;   // [2G][R]
  // autotuned block rows (warps) per CTA, right-hand sides per lane and gather ahead (1) or not of
  // mr_row_kernel and mr_fx_kernel per level and mode (0 FP64 level-0 apply, 1 residual, 3 smoother
  // sweep); 0 = not tuned
  int rows[kMaxLev][4] = {};
  int cols[kMaxLev][4] = {};
  int ahead[kMaxLev][4] = {};
  bool tuned = false;
  bool tc = false;             // smoother sweeps on tcgen05 (BF16 blocks)
  // the CG loop as one graph (a conditional WHILE node around one iteration), with the iteration
  // counter, the columns' counts and their residual histories [R][maxit + 1] on the device
  cudaGraphExec_t gsolve = nullptr;
  long long gsolve_kernels = 0;
  bool gsolve_failed = false;
  int *it_dev = nullptr, *iters_dev = nullptr;
  double* hist_dev = nullptr;
  int* tc_err = nullptr;       // set by a tensor-core kernel whose wait timed out
  // FP64 level-0 apply on tcgen05 by exact splitting: B operand images of the
  // slices of A_0, row exponents, slices of x and column exponents (device_ozaki.cu)
  bool oz = false;
  void* oz_img = nullptr;
  int* oz_eA = nullptr;
  void* oz_xs = nullptr;
  int* oz_maxb = nullptr;
};

void mr_tuning(const MR& M, int level, int nlev, int32_t* out) {
  if (!M.tuned) return;
  if (level + 1 < nlev) {
    out[4] = 32;
    out[5] = M.rows[level][3];
    out[6] = 32;
    out[7] = M.rows[level][1];
    out[10] = M.cols[level][3];
    out[11] = M.cols[level][1];
  }
  if (level == 0) {
    out[8] = M.rows[0][0] ? 32 : 0;
    out[9] = M.rows[0][0];
    out[12] = M.cols[0][0];
  }
}

namespace {

struct MRCarver {
  char* base;
  size_t off;
  template <typename T>
  T* take(size_t count) {
    off = (off + 255) & ~size_t(255);
    T* p = base ? reinterpret_cast<T*>(base + off) : nullptr;
    off += count * sizeof(T);
    return p;
  }
};

template <typename TA>
void upload_conv(void* dst, const std::vector<double>& src, cudaStream_t s) {
  if (src.empty()) return;
  std::vector<TA> h(src.size());
  for (size_t i = 0; i < src.size(); ++i) h[i] = (TA)src[i];
  cudaMemcpyAsync(dst, h.data(), sizeof(TA) * h.size(), cudaMemcpyHostToDevice, s);
  cudaStreamSynchronize(s);
}

}  // namespace

MR* mr_new() { return new MR(); }
void mr_drop_graph(MR* m) {
  if (m && m->gsolve) cudaGraphExecDestroy(m->gsolve);
  if (m) m->gsolve = nullptr;
}
void mr_delete(MR* m) {
  mr_drop_graph(m);
  delete m;
}

// Carves the multi-column buffers after `off`; returns the new end offset.
size_t mr_layout(const cdg::Hierarchy& H, int R, int precision, int tc_fp64, int maxit, MR* mr, char* base,
                 size_t off) {
  MRCarver c{base, off};
  MR tmp;
  MR& M = mr ? *mr : tmp;
  M.R = R;
  M.rows_per_cta = std::max(1, 256 / (((R + 31) / 32) * 32));
  M.G = (M.rows_per_cta > 2 ? 2 : 4) * 152 * M.rows_per_cta;
  M.bf16 = precision == 2;
  const size_t ts = M.bf16 ? sizeof(__nv_bfloat16) : sizeof(float);
  const int np = H.np;
  const size_t nb2 = (size_t)np * np;
  const int nlev = (int)H.lev.size();
  for (int l = 0; l < nlev; ++l) {
    MRLevel& L = M.lev[l];
    const size_t n = (size_t)H.lev[l].n;
    // the residual operator stays FP32 in every mode: b - A x cancels, and BF16
    // blocks (8-bit significands) would leave only noise in a small residual
    L.A = c.take<char>(H.A_t[l].val.size() * sizeof(float));
    if (l + 1 < nlev) {
      L.Ahat = c.take<char>(std::max<size_t>(1, H.Ahat_t[l].val.size()) * ts);
      // block inverses stay FP32 too: with C_D = gamma/h_avg a diagonal block reaches
      // cond ~1e5, and an 8-bit rounding of its inverse is then no inverse at all
      L.Dinv = c.take<char>(n * nb2 * sizeof(float));
      L.L = c.take<char>(n * nb2 * ts);
    }
    L.x = c.take<float>(n * np * R);
    L.t = c.take<float>(n * np * R);
    L.r = c.take<float>(n * np * R);
    L.b = c.take<float>(n * np * R);
    L.bh = c.take<float>(n * np * R);
  }
  const size_t nv = (size_t)H.mesh.ne * np * R;
  M.x = c.take<double>(nv);
  M.r = c.take<double>(nv);
  M.p = c.take<double>(nv);
  M.q = c.take<double>(nv);
  M.bt = c.take<double>(nv);
  M.r32 = c.take<float>(nv);
  M.z32 = c.take<float>(nv);
  M.scal = c.take<double>((size_t)R * S_COUNT);
  M.partial = c.take<double>((size_t)2 * M.G * R);
  M.tc_err = c.take<int>(1);
  M.it_dev = c.take<int>(1);
  M.iters_dev = c.take<int>(R);
  M.hist_dev = c.take<double>((size_t)R * (maxit + 1));
  M.oz = tc_fp64 != 0 && oz_feasible(H.A_t[0], np);
  if (M.oz) {
    M.oz_img = c.take<char>(oz_image_bytes(H.A_t[0]));
    M.oz_eA = c.take<int>((size_t)H.lev[0].n * 16);
    M.oz_xs = c.take<char>(oz_xslice_bytes(H.lev[0].n, np, R));
    M.oz_maxb = c.take<int>(R);
  }
  return c.off;
}

void mr_upload(const cdg::Hierarchy& H, MR& M, cudaStream_t s) {
  const int nlev = (int)H.lev.size();
  for (int l = 0; l < nlev; ++l) {
    MRLevel& L = M.lev[l];
    auto up = [&](void* dst, const std::vector<double>& src) {
      if (!dst) return;
      if (M.bf16) upload_conv<__nv_bfloat16>(dst, src, s);
      else upload_conv<float>(dst, src, s);
    };
    upload_conv<float>(L.A, H.A_t[l].val, s);
    if (l + 1 < nlev) {
      up(L.Ahat, H.Ahat_t[l].val);
      upload_conv<float>(L.Dinv, H.Dinv_t[l], s);
      up(L.L, H.L_t[l]);
    }
  }
  if (M.oz) {
    std::vector<uint16_t> img;
    std::vector<int32_t> eA;
    if (oz_prepare(H.A_t[0], H.np, img, eA)) {
      cudaMemcpyAsync(M.oz_img, img.data(), sizeof(uint16_t) * img.size(), cudaMemcpyHostToDevice, s);
      cudaMemcpyAsync(M.oz_eA, eA.data(), sizeof(int32_t) * eA.size(), cudaMemcpyHostToDevice, s);
      cudaStreamSynchronize(s);
    } else {
      M.oz = false;
    }
  }
}

namespace {

#define MR_NP_DISPATCH(NPV, ...)                            \
  switch (NPV) {                                            \
    case 3: { constexpr int NP = 3; __VA_ARGS__; break; }   \
    case 4: { constexpr int NP = 4; __VA_ARGS__; break; }   \
    case 6: { constexpr int NP = 6; __VA_ARGS__; break; }   \
    case 10: { constexpr int NP = 10; __VA_ARGS__; break; } \
    default: return false;                                  \
  }

// the same dispatch inside void lambdas (an unsupported n_p launches nothing)
#define MR_NP_DISPATCH_V(NPV, ...)                          \
  switch (NPV) {                                            \
    case 3: { constexpr int NP = 3; __VA_ARGS__; break; }   \
    case 4: { constexpr int NP = 4; __VA_ARGS__; break; }   \
    case 6: { constexpr int NP = 6; __VA_ARGS__; break; }   \
    case 10: { constexpr int NP = 10; __VA_ARGS__; break; } \
    default: break;                                         \
  }

inline unsigned threads_for(int R) { return (unsigned)(((R + 31) / 32) * 32); }

// mr_row_kernel with v columns per lane (brought down to what divides R), br warps (block rows) per
// CTA, pf: the next gather ahead
template <typename TA, int NP, int MODE>
void mr_row_launch(int br, int v, bool pf, int n, int R, const int* rp, const int* cl, const TA* A, const float* x,
                   const float* b, float* y, float* y2, float omega, cudaStream_t s) {
  br = std::min(std::max(br, 1), kMrMaxBR);
  while (R % v != 0) v /= 2;
  const dim3 grid((unsigned)((n + br - 1) / br), (unsigned)((R + 32 * v - 1) / (32 * v))), block(32, (unsigned)br);
  auto go = [&](auto kern) { kern<<<grid, block, 0, s>>>(n, R, rp, cl, A, x, b, y, y2, omega); };
  if (v == 4) pf ? go(mr_row_kernel<TA, NP, MODE, 4, true>) : go(mr_row_kernel<TA, NP, MODE, 4, false>);
  else if (v == 2) pf ? go(mr_row_kernel<TA, NP, MODE, 2, true>) : go(mr_row_kernel<TA, NP, MODE, 2, false>);
  else pf ? go(mr_row_kernel<TA, NP, MODE, 1, true>) : go(mr_row_kernel<TA, NP, MODE, 1, false>);
  count_launch();
}

// untuned: two columns per lane where R has them to give, the next gather ahead, four rows per CTA
inline int rows_of(const MR& M, int l, int mode) { return M.rows[l][mode] ? M.rows[l][mode] : kMrMaxBR; }
inline int cols_of(const MR& M, int l, int mode) { return M.cols[l][mode] ? M.cols[l][mode] : M.R >= 64 ? 2 : 1; }
inline bool ahead_of(const MR& M, int l, int mode) { return M.cols[l][mode] ? M.ahead[l][mode] != 0 : true; }

template <typename TA>
bool mr_vcycle(DeviceState& D, MR& M, const cdg_options& o, const float* b0, float* z0, cudaStream_t s) {
  const int np = D.np, nlev = D.nlev, R = M.R;
  const float w = (float)o.omega;
  auto bsr = [&](int mode, int l, const int* rp, const int* cl, const void* A, const float* x, const float* b,
                 float* y) -> bool {
    const int n = D.lev[l].n;
    if (mode == 3 && M.tc)
      return mr_tc_smooth(np, n, R, rp, cl, A, x, b, y, w, M.tc_err, D.wait_limit, s);
    const int br = rows_of(M, l, mode), v = cols_of(M, l, mode);
    const bool pf = ahead_of(M, l, mode);
    MR_NP_DISPATCH(np, {
      if (mode == 1) mr_row_launch<float, NP, 1>(br, v, pf, n, R, rp, cl, (const float*)A, x, b, y, nullptr, w, s);
      else mr_row_launch<TA, NP, 3>(br, v, pf, n, R, rp, cl, (const TA*)A, x, b, y, nullptr, w, s);
    });
    return true;
  };
  // the transfers and D^-1 b: untuned shapes
  const int v1 = R >= 128 ? 4 : R >= 64 ? 2 : 1;
  auto first = [&](int l, const float* b, float* bh, float* x) -> bool {
    const float* Dinv = (const float*)M.lev[l].Dinv;
    const int n = D.lev[l].n;
    MR_NP_DISPATCH(np, {
      if (x) mr_row_launch<float, NP, 6>(kMrMaxBR, v1, false, n, R, nullptr, nullptr, Dinv, b, nullptr, bh, x, w, s);
      else mr_row_launch<float, NP, 7>(kMrMaxBR, v1, false, n, R, nullptr, nullptr, Dinv, b, nullptr, bh, nullptr, w, s);
    });
    return true;
  };
  auto restrict_to = [&](int l, const float* r, float* bc) -> bool {
    const DevLevel& C = D.lev[l + 1];
    MR_NP_DISPATCH(np, (mr_row_launch<TA, NP, 8>(kMrMaxBR, v1, true, C.n, R, C.childptr, nullptr,
                                                 (const TA*)M.lev[l].L, r, nullptr, bc, nullptr, w, s)));
    return true;
  };
  auto prolong = [&](int l, const float* xc, float* x, bool add) -> bool {
    const DevLevel& F = D.lev[l];
    const TA* L = (const TA*)M.lev[l].L;
    MR_NP_DISPATCH(np, {
      if (add) mr_row_launch<TA, NP, 4>(kMrMaxBR, v1, false, F.n, R, nullptr, F.parent, L, xc, nullptr, x, nullptr, w, s);
      else mr_row_launch<TA, NP, 7>(kMrMaxBR, v1, false, F.n, R, nullptr, F.parent, L, xc, nullptr, x, nullptr, w, s);
    });
    return true;
  };
  const dim3 coarse_grid((unsigned)((D.nc + kCoarseRows - 1) / kCoarseRows), (unsigned)((R + 31) / 32));
  const dim3 coarse_block(32, kCoarseWarps);
  if (nlev == 1) {
    mr_coarse_kernel<float><<<coarse_grid, coarse_block, 0, s>>>(D.nc, R, D.coarse_inv, b0, z0);
    count_launch();
    return true;
  }
  std::vector<const float*> bl(nlev);
  bl[0] = b0;
  for (int l = 1; l < nlev; ++l) bl[l] = M.lev[l].b;
  for (int l = 0; l + 1 < nlev; ++l) {
    MRLevel& L = M.lev[l];
    const DevLevel& DL = D.lev[l];
    float* x = L.x;
    float* t = L.t;
    const float* b = bl[l];
    if (o.nu_pre >= 1) {
      if (!first(l, b, L.bh, x)) return false;
      for (int k = 1; k < o.nu_pre; ++k) {
        if (!bsr(3, l, DL.hrowptr, DL.hcol, L.Ahat, x, L.bh, t)) return false;
        std::swap(x, t);
      }
      if (!bsr(1, l, DL.rowptr, DL.col, L.A, x, b, L.r)) return false;
      if (!restrict_to(l, L.r, M.lev[l + 1].b)) return false;
      L.x = x;
      L.t = t;
    } else {
      if (!first(l, b, L.bh, nullptr) || !restrict_to(l, b, M.lev[l + 1].b)) return false;
    }
  }
  mr_coarse_kernel<float><<<coarse_grid, coarse_block, 0, s>>>(D.nc, R, D.coarse_inv, M.lev[nlev - 1].b,
                                                               M.lev[nlev - 1].x);
  count_launch();
  for (int l = nlev - 2; l >= 0; --l) {
    MRLevel& L = M.lev[l];
    const DevLevel& DL = D.lev[l];
    float* x = L.x;
    float* t = L.t;
    if (!prolong(l, M.lev[l + 1].x, x, o.nu_pre >= 1)) return false;
    for (int k = 0; k < o.nu_post; ++k) {
      float* out = (l == 0 && k + 1 == o.nu_post) ? z0 : t;
      if (!bsr(3, l, DL.hrowptr, DL.hcol, L.Ahat, x, L.bh, out)) return false;
      if (out == t) std::swap(x, t);
      else x = out;
    }
    if (l == 0 && o.nu_post == 0)
      cudaMemcpyAsync(z0, x, sizeof(float) * (size_t)DL.n * np * R, cudaMemcpyDeviceToDevice, s);
    if (l > 0 && x != L.x) {
      L.t = L.x;
      L.x = x;
    }
  }
  return true;
}

// maxb_ready: the column exponents of x are already in M.oz_maxb (mr_p_kernel
// stores them for p); pq_groups (split apply only): the apply also leaves the
// partial sums of x . y in M.partial, *pq_groups of them per column
bool mr_apply64(DeviceState& D, MR& M, const double* x, double* y, cudaStream_t s, bool maxb_ready = false,
                int* pq_groups = nullptr, int rows = 0) {
  const DevLevel& L0 = D.lev[0];
  if (M.oz)
    return oz_apply(D.np, L0.n, M.R, L0.rowptr, L0.col, M.oz_img, M.oz_eA, M.oz_xs, M.oz_maxb, maxb_ready, x, y,
                    pq_groups ? M.partial : nullptr, pq_groups, M.tc_err, D.wait_limit, s);
  const int br = rows ? rows : rows_of(M, 0, 0);
  const dim3 grid((unsigned)((L0.n + br - 1) / br), (unsigned)((M.R + 31) / 32)), block(32, (unsigned)br);
  const int2* A = reinterpret_cast<const int2*>(L0.fixed ? L0.A : L0.Adig);
  MR_NP_DISPATCH(D.np, mr_fx_kernel<NP><<<grid, block, 0, s>>>(L0.n, M.R, L0.rowptr, L0.col, A, L0.eA, x, y));
  count_launch();
  return true;
}

// Autotuner of the many-right-hand-side block kernels: for every level and mode the solve launches,
// times the columns per lane (1, 2, 4 where they divide R and leave a lane work) x warps per CTA x
// gather ahead or not, on the handle's operators and zero-filled work vectors, and keeps the fastest.
template <typename TA>
bool mr_autotune(DeviceState& D, MR& M, double omega, cudaStream_t s) {
  const int np = D.np, nlev = D.nlev, R = M.R;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return false;
  const int padded = (R + 31) / 32 * 32;
  auto pick = [&](int l, int mode, auto&& launch_one) {
    float tbest = 3.0e38f;
    for (int v : {1, 2, 4}) {
      if (mode == 0 && v > 1) break;
      if (R % v != 0 || (v > 1 && 32 * v > padded)) continue;
      for (int br : {1, 2, 4}) {
        for (int pf = 0; pf <= (mode == 0 ? 0 : 1); ++pf) {
          const float t = time_calls(s, e0, e1, 2, [&] { launch_one(br, v, pf != 0); });
          if (t < tbest) {
            tbest = t;
            M.rows[l][mode] = br;
            M.cols[l][mode] = v;
            M.ahead[l][mode] = pf;
          }
        }
      }
    }
  };
  bool ok = true;
  if (!M.oz) {   // the FP64 apply on CUDA cores (the split apply has no variants)
    const DevLevel& L0 = D.lev[0];
    const size_t nv = (size_t)L0.n * np * R;
    cudaMemsetAsync(M.p, 0, nv * sizeof(double), s);
    pick(0, 0, [&](int br, int, bool) { mr_apply64(D, M, M.p, M.q, s, false, nullptr, br); });
  }
  const float w = (float)omega;
  for (int l = 0; l + 1 < nlev; ++l) {
    const DevLevel& DL = D.lev[l];
    MRLevel& L = M.lev[l];
    const size_t nv = (size_t)DL.n * np * R;
    for (float* v : {L.x, L.b, L.bh, L.t}) cudaMemsetAsync(v, 0, nv * sizeof(float), s);
    pick(l, 1, [&](int br, int v, bool pf) {
      MR_NP_DISPATCH_V(np, (mr_row_launch<float, NP, 1>(br, v, pf, DL.n, R, DL.rowptr, DL.col, (const float*)L.A,
                                                        (const float*)L.x, (const float*)L.b, L.t, nullptr, w, s)));
    });
    pick(l, 3, [&](int br, int v, bool pf) {
      MR_NP_DISPATCH_V(np, (mr_row_launch<TA, NP, 3>(br, v, pf, DL.n, R, DL.hrowptr, DL.hcol, (const TA*)L.Ahat,
                                                     (const float*)L.x, (const float*)L.bh, L.t, nullptr, w, s)));
    });
  }
  ok = cudaStreamSynchronize(s) == cudaSuccess && cudaGetLastError() == cudaSuccess;
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  M.tuned = ok;
  return ok;
}

// sums G partials per column (G = M.G unless given) into the CG scalars
void mr_finalize(MR& M, int which, double tol, cudaStream_t s, int G = 0) {
  mr_finalize_kernel<<<(M.R + kFinCols - 1) / kFinCols, kFinThreads, 0, s>>>(M.R, G > 0 ? G : M.G, M.partial, which,
                                                                           tol, M.scal);
  count_launch();
}

template <typename TY>
void mr_dot(DeviceState& D, MR& M, const double* x, const TY* y, int which, double tol, cudaStream_t s) {
  const int nrows = (int)(D.ne * D.np);
  const dim3 T(threads_for(M.R), (unsigned)M.rows_per_cta);
  mr_dot_kernel<TY><<<M.G / M.rows_per_cta, T, 0, s>>>(nrows, M.R, M.G, x, y, M.partial);
  count_launch();
  mr_finalize(M, which, tol, s);
}

// the V-cycle maps r32 (FP32 copy of r, written by mr_update_kernel after the first step) to z32;
// z = z32 widened exactly, so the FP64 steps read z32
bool mr_precond(DeviceState& D, MR& M, const cdg_options& o, cudaStream_t s) {
  return M.bf16 ? mr_vcycle<__nv_bfloat16>(D, M, o, M.r32, M.z32, s) : mr_vcycle<float>(D, M, o, M.r32, M.z32, s);
}

void mr_direction(DeviceState& D, MR& M, int first, cudaStream_t s) {
  if (M.oz) cudaMemsetAsync(M.oz_maxb, 0, sizeof(int) * M.R, s);
  mr_p_kernel<<<(unsigned)(M.G / M.rows_per_cta), dim3(threads_for(M.R), (unsigned)M.rows_per_cta), 0, s>>>(
      (int)(D.ne * D.np), M.R, M.G, M.scal, first, M.z32, M.p, M.oz ? M.oz_maxb : nullptr);
  count_launch();
}

// q = A p, alpha, x and r updates, r.r
bool mr_part1(DeviceState& D, MR& M, const cdg_options& o, cudaStream_t s) {
  bool ok;
  if (M.oz) {   // p's column exponents come from mr_p_kernel, p . A p from the apply's epilogue
    int gq = 0;
    ok = mr_apply64(D, M, M.p, M.q, s, true, &gq);
    mr_finalize(M, 0, o.tol, s, gq);
  } else {
    ok = mr_apply64(D, M, M.p, M.q, s);
    mr_dot<double>(D, M, M.p, M.q, 0, o.tol, s);
  }
  // the update (five reads, three writes) runs two CTAs per SM: 256 columns of 200,000 rows 456 us, with
  // the four of the dots 496 us (the dots 162 against 202 us, the p update 147 against 198 us)
  const int Gu = 2 * 152 * M.rows_per_cta;
  mr_update_kernel<<<2 * 152, dim3(threads_for(M.R), (unsigned)M.rows_per_cta), 0, s>>>(
      (int)(D.ne * D.np), M.R, Gu, M.scal, M.p, M.q, M.x, M.r, M.r32, M.z32, M.partial);
  count_launch();
  mr_finalize(M, 1, o.tol, s, Gu);
  return ok;
}

// z = V(r), beta, p
bool mr_part2(DeviceState& D, MR& M, const cdg_options& o, cudaStream_t s) {
  const bool ok = mr_precond(D, M, o, s);
  mr_dot<float>(D, M, M.r, M.z32, 2, o.tol, s);
  mr_direction(D, M, 0, s);
  return ok;
}

// The CG loop as one executable graph, WHILE (cond) { part 1; check; part 2 }, as cdg_solve has it: the
// condition starts at 1 on every launch, and the check clears it.  false: refused, the host drives the loop.
bool mr_capture(DeviceState& D, MR& M, const cdg_options& o) {
  cudaGraph_t g = nullptr;
  if (cudaGraphCreate(&g, 0) != cudaSuccess) return false;
  cudaGraphConditionalHandle cond;
  cudaError_t e = cudaGraphConditionalHandleCreate(&cond, g, 1, cudaGraphCondAssignDefault);
  cudaGraphNodeParams p = {};
  p.type = cudaGraphNodeTypeConditional;
  p.conditional.handle = cond;
  p.conditional.type = cudaGraphCondTypeWhile;
  p.conditional.size = 1;
  cudaGraphNode_t node;
  if (e == cudaSuccess) e = cudaGraphAddNode(&node, g, nullptr, nullptr, 0, &p);
  if (e == cudaSuccess)
    e = cudaStreamBeginCaptureToGraph(D.stream, p.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                      cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) {
    cudaGraphDestroy(g);
    return false;
  }
  const long long before = launch_count();
  bool ok = mr_part1(D, M, o, D.stream);
  mr_check_kernel<<<1, 256, 0, D.stream>>>(cond, M.R, o.maxit, M.scal, M.it_dev, M.hist_dev, M.iters_dev, M.tc_err);
  count_launch();
  ok = mr_part2(D, M, o, D.stream) && ok;
  cudaGraph_t captured = nullptr;
  e = cudaStreamEndCapture(D.stream, &captured);
  // captured launches run when the graph is launched: counted there, per iteration
  M.gsolve_kernels = launch_count() - before;
  count_launch(-M.gsolve_kernels);
  if (ok && e == cudaSuccess) e = cudaGraphInstantiate(&M.gsolve, g, 0);
  cudaGraphDestroy(g);
  if (!ok || e != cudaSuccess) M.gsolve = nullptr;
  return M.gsolve != nullptr;
}

}  // namespace

// Solves A_0 U = B for R columns: f_q [R][n_elements][nq] (device), u [R][n_elements][n_p]
// (device), res_hist [R][maxit+1] and iters [R] (host).
int dev_solve_multi(cdg_handle* h, const double* f_q, double* u, double* res_hist, int* iters, void* stream) {
  if (!h->dev || !h->dev->mr) {
    h->err = "cdg_solve_multi needs a handle created with nrhs > 0 and bound to a device buffer";
    return CDG_ESTATE;
  }
  DeviceState& D = *h->dev;
  MR& M = *D.mr;
  const cdg_options& o = h->opt;
  const int R = M.R;
  if (D.np != 3 && D.np != 4 && D.np != 6 && D.np != 10) {   // cdg_create rejects these already
    h->err = "unsupported n_p for cdg_solve_multi";
    return CDG_EINVAL;
  }
  cudaStream_t cs = (cudaStream_t)stream;
  cudaStream_t s = D.stream;
  cudaEventRecord(D.ev_in, cs);
  cudaStreamWaitEvent(s, D.ev_in, 0);
  const size_t nv = (size_t)D.ne * D.np * R;
  const unsigned T = threads_for(R);
  const unsigned gv = 4 * 152;
  bool ok = true;
  if (o.autotune && !M.tuned) {
    ok = M.bf16 ? mr_autotune<__nv_bfloat16>(D, M, o.omega, s) : mr_autotune<float>(D, M, o.omega, s);
    if (!ok) {
      h->err = "cdg_solve_multi: autotuning failed (unsupported n_p or a CUDA error)";
      return CDG_ECUDA;
    }
  }
  cudaMemsetAsync(M.scal, 0, sizeof(double) * (size_t)R * S_COUNT, s);
  M.tc = M.bf16 && o.tensor_cores != 0 && D.np <= 16;
  cudaMemsetAsync(M.tc_err, 0, sizeof(int), s);
  MR_NP_DISPATCH(D.np, mr_rhs_kernel<NP><<<(unsigned)D.ne, T, 0, s>>>(R, D.nq, (int)D.ne, D.perm0, D.rhs_vol, f_q, M.bt));
  count_launch();
  cudaMemsetAsync(M.x, 0, sizeof(double) * nv, s);
  cudaMemcpyAsync(M.r, M.bt, sizeof(double) * nv, cudaMemcpyDeviceToDevice, s);
  mr_dot<double>(D, M, M.bt, M.bt, 3, o.tol, s);
  mr_dot<double>(D, M, M.r, M.r, 4, o.tol, s);
  std::vector<double> hs((size_t)R * S_COUNT);
  cudaMemcpyAsync(hs.data(), M.scal, sizeof(double) * hs.size(), cudaMemcpyDeviceToHost, s);
  cudaError_t e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    h->err = std::string("solve_multi: ") + cudaGetErrorString(e);
    return CDG_ECUDA;
  }
  const int stride = o.maxit + 1;
  auto rel = [&](int r) {
    const double* sc = &hs[(size_t)r * S_COUNT];
    return sc[S_BB] > 0.0 ? std::sqrt(sc[S_RR] / sc[S_BB]) : 0.0;
  };
  std::vector<char> done(R, 0);
  int ndone = 0, status = CDG_OK, it = 0;
  for (int r = 0; r < R; ++r) {
    iters[r] = 0;
    if (res_hist) res_hist[(size_t)r * stride] = rel(r);
    if (hs[(size_t)r * S_COUNT + S_DONE] != 0.0) {
      done[r] = 1;
      ++ndone;
    }
  }
  auto close = [&](int r) {   // a column whose scalars say that it is done
    done[r] = 1;
    ++ndone;
    if (hs[(size_t)r * S_COUNT + S_BREAK] != 0.0) {
      status = CDG_EBREAKDOWN;
      h->err = "CG breakdown in column " + std::to_string(r);
    }
  };
  if (ndone < R) {
    mr_convert_kernel<double, float><<<gv, 256, 0, s>>>(nv, M.r, M.r32);
    count_launch();
    ok = mr_precond(D, M, o, s);
    mr_dot<float>(D, M, M.r, M.z32, 2, o.tol, s);
    mr_direction(D, M, 1, s);
    if (ok && o.solve_graph && o.maxit > 0 && !M.gsolve && !M.gsolve_failed && !mr_capture(D, M, o)) {
      M.gsolve_failed = true;   // refused by this driver: keep the host-driven loop
      cudaGetLastError();
    }
    const bool in_graph = ok && o.solve_graph && o.maxit > 0 && M.gsolve;
    if (in_graph) {
      mr_open_kernel<<<1, 256, 0, s>>>(R, M.scal, M.it_dev, M.iters_dev);
      count_launch();
      e = cudaGraphLaunch(M.gsolve, s);
      if (e == cudaSuccess) e = cudaMemcpyAsync(&it, M.it_dev, sizeof(int), cudaMemcpyDeviceToHost, s);
      if (e == cudaSuccess) e = cudaMemcpyAsync(iters, M.iters_dev, sizeof(int) * R, cudaMemcpyDeviceToHost, s);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(hs.data(), M.scal, sizeof(double) * hs.size(), cudaMemcpyDeviceToHost, s);
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);
      std::vector<double> hh;   // the columns' entries 1 .. it
      if (e == cudaSuccess && res_hist && it > 0) {
        hh.resize((size_t)R * it);
        e = cudaMemcpy2DAsync(hh.data(), sizeof(double) * it, M.hist_dev + 1, sizeof(double) * stride,
                              sizeof(double) * it, R, cudaMemcpyDeviceToHost, s);
      }
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);
      if (e != cudaSuccess) {
        h->err = std::string("solve_multi: ") + cudaGetErrorString(e);
        return CDG_ECUDA;
      }
      count_launch(M.gsolve_kernels * it);
      for (int r = 0; r < R; ++r) {
        if (res_hist)
          for (int k = 1; k <= iters[r]; ++k) res_hist[(size_t)r * stride + k] = hh[(size_t)r * it + k - 1];
        if (!done[r] && hs[(size_t)r * S_COUNT + S_DONE] != 0.0) close(r);
      }
      if (ndone < R) status = CDG_ENOCONV;
    }
    while (ok && !in_graph) {
      if (it >= o.maxit) {
        status = CDG_ENOCONV;
        break;
      }
      ok = mr_part1(D, M, o, s);
      cudaMemcpyAsync(hs.data(), M.scal, sizeof(double) * hs.size(), cudaMemcpyDeviceToHost, s);
      int tc_err_it = 0;
      cudaMemcpyAsync(&tc_err_it, M.tc_err, sizeof(int), cudaMemcpyDeviceToHost, s);
      e = cudaStreamSynchronize(s);
      if (e != cudaSuccess) {
        h->err = std::string("solve_multi: ") + cudaGetErrorString(e);
        return CDG_ECUDA;
      }
      if (tc_err_it) break;   // a sweep gave up: its rows are not smoothed; reported below
      ++it;
      for (int r = 0; r < R; ++r) {
        if (done[r]) continue;
        iters[r] = it;
        if (res_hist) res_hist[(size_t)r * stride + it] = rel(r);
        if (hs[(size_t)r * S_COUNT + S_DONE] != 0.0) close(r);
      }
      if (ndone == R) break;
      ok = mr_part2(D, M, o, s);
    }
  }
  if (!ok) {
    h->err = "unsupported n_p for cdg_solve_multi";
    return CDG_EINVAL;
  }
  mr_out_kernel<<<(unsigned)D.ne, T, 0, s>>>(R, D.np, D.perm0, M.x, (int)D.ne, u);
  count_launch();
  int tc_err = 0;
  cudaMemcpyAsync(&tc_err, M.tc_err, sizeof(int), cudaMemcpyDeviceToHost, s);
  e = cudaStreamSynchronize(s);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) {
    h->err = std::string("solve_multi: ") + cudaGetErrorString(e);
    return CDG_ECUDA;
  }
  if (tc_err) {
    h->err = "solve_multi: a tensor-core wait reached its iteration limit";
    return CDG_ETIMEOUT;
  }
  if (status == CDG_ENOCONV) h->err = "maximum number of iterations reached";
  return status;
}

// y = A_0 x for the R columns of a multi-right-hand-side handle (tree order,
// [n][n_p][R] FP64, device), by the method its solves use; synchronous.
int dev_apply_multi(cdg_handle* h, const double* x, double* y, void* stream) {
  if (!h->dev || !h->dev->mr) {
    h->err = "cdg_apply_multi needs a handle created with nrhs > 0 and bound to a device buffer";
    return CDG_ESTATE;
  }
  DeviceState& D = *h->dev;
  MR& M = *D.mr;
  cudaStream_t s = (cudaStream_t)stream;
  if (M.oz) cudaMemsetAsync(M.tc_err, 0, sizeof(int), s);
  if (!mr_apply64(D, M, x, y, s)) {
    h->err = "unsupported n_p for cdg_apply_multi";
    return CDG_EINVAL;
  }
  int err = 0;
  if (M.oz) cudaMemcpyAsync(&err, M.tc_err, sizeof(int), cudaMemcpyDeviceToHost, s);
  cudaError_t e = cudaStreamSynchronize(s);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) {
    h->err = std::string("cdg_apply_multi: ") + cudaGetErrorString(e);
    return CDG_ECUDA;
  }
  if (err) {
    h->err = "cdg_apply_multi: a tensor-core wait reached its iteration limit";
    return CDG_ETIMEOUT;
  }
  return CDG_OK;
}
