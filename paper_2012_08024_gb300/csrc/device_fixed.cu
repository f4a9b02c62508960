// FP64 block-sparse products by exact integer arithmetic.
//
// The FP64 pipe of this GPU completes two fused multiply-adds per clock and SM
// (a warp's DFMA occupies its quadrant for 64 clocks, measured 70.7 in a
// dependent chain), a fiftieth of the FP32 rate, and it, not HBM, bounded every
// FP64 block kernel: 0.89 of the FP64 rate at 0.69 of the copy bandwidth, and
// 10-15 us on the small levels, whose few CTAs each ran their FMAs through one
// SM's pipe.  A 32 x 32 + 64 -> 64 bit integer multiply-add (mad.wide) takes 4
// clocks.  So an operator entry is kept as two signed integer digits (the same
// 8 bytes as a double),
//     a = 2^(EA - 58) (ah 2^30 + al),   |ah| <= 2^28,  |al| <= 2^29,
// with one exponent EA per scalar row, every entry rounded to 2^-59 of the
// row's power-of-two bound, and the n_p values of a neighbour's x_J are split
// likewise with one exponent of their own.  Four integer multiply-adds give a
// product of digits exactly, the sum over a block is exact, the blocks' sums are
// brought to the scale of the largest (nothing above 2^-96 of it is lost), and
// one rounding to FP64 ends the row: 16 clocks in the place of 64.  A row's
// result depends on the values that it multiplies and on no others: with one
// exponent for all that a warp gathers, rows of two meshes of a batch shared one,
// and a mesh with small data beside one with large data got a wrong solution.
// (The exponents per block cost 2-4%: apply 72.4 -> 74.3 us, V-cycle of the
// 128^2 (p = 3) mesh 199 -> 207 us, 64 meshes 52.4 -> 54.5 ms.)  The
// method is the splitting of Ozaki, Ogita, Oishi and Rump (2012) with integer
// digits.  58 bits, not fewer, since A x cancels for smooth x, where the small
// constant-mode entries of A meet the largest values of x: on solutions of the
// 32^2 (p = 1, 2, 3) and 6^3 (p = 1, 2) meshes FP64 sums are 0.5-4.1e-12 off in
// the 2-norm, 54-bit digits 1.7-44e-12, 58-bit digits 0.07-2.4e-12 (each below
// FP64's on the same mesh); random vectors 1.0-2.0e-16 against 0.4-0.7e-17.
//
// The sums, over the T <= 28 terms of a block: |sum al xl| <= 2^58 T,
// |sum (ah xl + al xh)| <= 2^58 T; both are then carried into the next higher
// one, and |sum ah xh| <= 2^56 T.
//
// Mapping: the n_p lanes of a group own the n_p scalar rows of one block row; a
// lane loads one value of each x_J, splits it and leaves the digits in shared
// memory for its group, and reads its matrix row digit pairs from a layout in
// which the lanes of a group read consecutive 16 (even n_p) or 8 bytes.
// Packed: floor(32 / n_p) block rows per warp.  WPR: one block row per warp,
// its blocks dealt to the groups (levels with few rows).  A warp strides over
// its packs; the padded column table lets the gathers of x start with the row
// pointers.  The kernel waits for memory (issue slots a third used), so resident
// warps count: 64 registers, 32 warps per SM.  Measured, 131,072 rows of 4
// blocks at n_p = 10: apply 102.7 -> 76.9 us, level of 1,044 rows 12.6 -> 4.7 us
// (72.7 us, 6.1 TB/s, and 3.2 us with dependent launches); 80 registers 84.7 us; digits streamed through shared memory by
// cp.async, one or two packs ahead, 85-104 us (fewer warps fit); 48 registers 90 us.
#include <cuda_runtime.h>

#include <algorithm>

#include "device_fixed.cuh"
#include "device_kernels.cuh"
#include "device_state.h"

namespace {

using namespace fx;

template <int NP, int MODE, bool WPR>
__global__ void __launch_bounds__(kFxThreads, fx_ctas_per_sm(NP)) fx_kernel(const __grid_constant__ FxOp q) {
  using P = Pack<NP, MODE, WPR>;
  __shared__ __align__(16) int2 digits[kFxWarps][P::DIGITS];
  const int packs = WPR ? q.n : (q.n + P::RPW - 1) / P::RPW;
  const int stride = gridDim.x * kFxWarps;
  double dsum = 0.0;
  bool waited = false;
  for (int pack = blockIdx.x * kFxWarps + (threadIdx.x >> 5); pack < packs; pack += stride)
    dsum = fx_pack<NP, MODE, WPR, false>(q, pack, digits[threadIdx.x >> 5], dsum, waited);
  if (!waited) cdgk::wait_for_inputs();   // a warp without rows
  if constexpr (MODE == 0 || MODE == 3)
    if (q.dot) {
      __shared__ double red[kFxThreads];
      dsum = cdgk::cta_sum<kFxWarps>(dsum, red);
      if ((int)threadIdx.x == cdgk::summing_warp<kFxWarps>() * 32) q.dot[blockIdx.x] = dsum;
    }
}

// FP64 blocks to digits, in place: one warp per block row (the row exponents
// first, then block by block through registers)
template <int NP>
__global__ void __launch_bounds__(kFxThreads) fx_encode_kernel(int n, const int* __restrict__ rowptr,
                                                               double* A, int* __restrict__ EA) {
  constexpr int PER = (NP * NP + 31) / 32;
  __shared__ int ex[kFxWarps][NP];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int K = blockIdx.x * kFxWarps + w;
  if (K >= n) return;
  const int b0 = rowptr ? rowptr[K] : K, b1 = rowptr ? rowptr[K + 1] : K + 1;
  for (int i = lane; i < NP; i += 32) ex[w][i] = 1;
  __syncwarp();
  for (int bb = b0; bb < b1; ++bb)
    for (int t = lane; t < NP * NP; t += 32) atomicMax(&ex[w][t / NP], biased_exponent(A[(size_t)bb * NP * NP + t]));
  __syncwarp();
  for (int i = lane; i < NP; i += 32) EA[(size_t)K * NP + i] = ex[w][i] == 0x7FF ? kNotFinite : ex[w][i] - 1022;
  for (int bb = b0; bb < b1; ++bb) {
    double v[PER];
#pragma unroll
    for (int c = 0; c < PER; ++c) {
      const int t = c * 32 + lane;
      v[c] = t < NP * NP ? A[(size_t)bb * NP * NP + t] : 0.0;
    }
    __syncwarp();
    int2* d = reinterpret_cast<int2*>(A) + (size_t)bb * NP * NP;
#pragma unroll
    for (int c = 0; c < PER; ++c) {
      const int t = c * 32 + lane;
      if (t < NP * NP) d[fx_pos(NP, t / NP, t % NP)] = split_digits(v[c], ex[w][t / NP]);
    }
    __syncwarp();
  }
}

#define FX_NP_DISPATCH(NPV, ...)                            \
  switch (NPV) {                                            \
    case 3: { constexpr int NP = 3; __VA_ARGS__; break; }   \
    case 4: { constexpr int NP = 4; __VA_ARGS__; break; }   \
    case 6: { constexpr int NP = 6; __VA_ARGS__; break; }   \
    case 10: { constexpr int NP = 10; __VA_ARGS__; break; } \
    case 15: { constexpr int NP = 15; __VA_ARGS__; break; } \
    case 20: { constexpr int NP = 20; __VA_ARGS__; break; } \
    case 21: { constexpr int NP = 21; __VA_ARGS__; break; } \
    case 28: { constexpr int NP = 28; __VA_ARGS__; break; } \
    default: return false;                                  \
  }

template <int NP, int MODE>
unsigned go(const FxOp& o, cudaStream_t s, bool launch) {
  const bool wpr = !fx_one(MODE) && warp_per_row(NP, o.n, o.blocks);
  const int packs = wpr ? o.n : (o.n + 32 / NP - 1) / (32 / NP);
  const unsigned g =
      (unsigned)std::max(1, std::min((packs + kFxWarps - 1) / kFxWarps, kFxSms * fx_ctas_per_sm(NP)));
  if (!launch) return g;
  if (wpr) {
    if constexpr (!fx_one(MODE) && 32 / NP > 1)
      launch_dep(fx_kernel<NP, MODE, true>, g, kFxThreads, s, o);
  } else {
    launch_dep(fx_kernel<NP, MODE, false>, g, kFxThreads, s, o);
  }
  return g;
}

template <int NP>
unsigned go_mode(const FxOp& o, cudaStream_t s, bool launch) {
  switch (o.mode) {
    case 0: return go<NP, 0>(o, s, launch);
    case 1: return go<NP, 1>(o, s, launch);
    case 3: return go<NP, 3>(o, s, launch);
    case 4: return go<NP, 4>(o, s, launch);
    case 6: return go<NP, 6>(o, s, launch);
    case 7: return go<NP, 7>(o, s, launch);
    case 8: return go<NP, 8>(o, s, launch);
    default: return 0;
  }
}

unsigned dispatch(const FxOp& o, cudaStream_t s, bool launch) {
  FX_NP_DISPATCH(o.np, return go_mode<NP>(o, s, launch));
  return 0;
}

}  // namespace

FxOp operator_op(const DevLevel& L, int mode) {
  const bool hat = mode == 3;
  FxOp o;
  o.mode = mode;
  o.np = L.np;
  o.n = L.n;
  o.blocks = hat ? L.hnnzb : L.nnzb;
  o.rowptr = hat ? L.hrowptr : L.rowptr;
  o.cols = hat ? L.hell : L.ell;
  o.width = hat ? L.whell : L.well;
  o.A = hat ? L.Ahat : L.A;
  o.EA = hat ? L.eH : L.eA;
  return o;
}

// one block per row
FxOp diagonal_op(const DevLevel& L, int mode, const double* blocks, const int* exps) {
  FxOp o;
  o.mode = mode;
  o.np = L.np;
  o.n = L.n;
  o.blocks = L.n;
  o.A = blocks;
  o.EA = exps;
  return o;
}

FxOp prolong_op(const DevLevel& F, int mode) {
  FxOp o = diagonal_op(F, mode, F.Lx, F.eL);
  o.cols = F.parent;
  return o;
}

FxOp restrict_op(const DevLevel& F, const DevLevel& C) {
  FxOp o;
  o.mode = 8;
  o.np = F.np;
  o.n = C.n;
  o.blocks = F.n;
  o.rowptr = C.childptr;
  o.A = F.Rx;
  o.EA = F.eR;
  return o;
}

unsigned fx_grid(const FxOp& o) { return dispatch(o, nullptr, false); }
bool fx_run(const FxOp& o, cudaStream_t s) { return dispatch(o, s, true) > 0; }

bool fx_encode(int np, int n, const int* rowptr, double* A, int* EA, cudaStream_t s) {
  if (n < 1) return true;
  FX_NP_DISPATCH(np, (fx_encode_kernel<NP><<<(unsigned)((n + kFxWarps - 1) / kFxWarps), kFxThreads, 0, s>>>(n, rowptr,
                                                                                                          A, EA)));
  count_launch();
  return true;
}
