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
// with one exponent EA per scalar row of a block, every entry rounded to 2^-59
// of the power of two above that row's largest, and the n_p values of a
// neighbour's x_J are split likewise with one exponent of their own.  Four
// integer multiply-adds give a product of digits exactly, the sum over a block is
// exact, the blocks' sums are brought to the scale of the largest (nothing above
// 2^-96 of it is lost), and one rounding to FP64 ends the row: 16 clocks in the
// place of 64.  The method is the splitting of Ozaki, Ogita, Oishi and Rump
// (2012) with integer digits.
//
// Why an exponent per block and not a wider one: with one per scalar row of A and
// one for all the values that a warp gathers, blocks that kappa makes small lost
// their low digits, a row's result depended on rows that it has no block with,
// and a mesh of a batch whose data were small beside its neighbour's got a wrong
// solution.  Now a row is off by no more than 2^-57 n_p sum_J max|a_J| max|x_J|
// and one rounding.  It costs 0-5% (against the wider exponents: apply of 256^2,
// p = 3, 72.6 -> 75.4 us; V-cycle of 128^2, p = 3, 198 -> 196 us; 64 meshes at
// p = 2 52.2 -> 53.3 ms; 32^2 at p = 2 4.24 -> 4.36 ms).
// Why 58 bits and not fewer: A x cancels for smooth x, where the small
// constant-mode entries of A meet the largest values of x.  On solutions of the
// 32^2 (p = 1, 2, 3) and 6^3 (p = 1, 2) meshes FP64 sums are 0.3-3.1e-12 off in
// the 2-norm, the digits 0.01-0.36e-12, with kappa from 1e-4 to 1e4 at random
// (24^2, p = 2, 3) 3.3-8.1e-9 against 0.1-0.4e-9, random vectors 0.8-1.9e-16
// against 0.5e-16; relative to sum |a| |x| of its own row the worst row of these
// is 7e-16 off with FP64 sums and 4e-15 with digits.  V-cycles of random r against
// the exact cycle: 128^2, p = 3, 0.9-1.2e-12 and 0.9-1.4e-13, 64^2, p = 2, 2.3-5.5e-13 and 1.9-3.1e-14.
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
// (75.2 us, 6.0 TB/s, and 3.3 us with dependent launches); with 80 registers 79.0 us, with 48 137 us; digits
// streamed through shared memory by cp.async, one or two packs ahead, 85-104 us (fewer warps fit).
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

// FP64 blocks to digits, in place: one warp per block (its rows' exponents first, then through registers)
template <int NP>
__global__ void __launch_bounds__(kFxThreads) fx_encode_kernel(int64_t blocks, double* A, unsigned short* EA) {
  constexpr int PER = (NP * NP + 31) / 32;
  __shared__ int ex[kFxWarps][NP];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t b = (int64_t)blockIdx.x * kFxWarps + w;
  if (b >= blocks) return;
  for (int i = lane; i < NP; i += 32) ex[w][i] = 1;
  __syncwarp();
  double v[PER];
#pragma unroll
  for (int c = 0; c < PER; ++c) {
    const int t = c * 32 + lane;
    v[c] = t < NP * NP ? A[(size_t)b * NP * NP + t] : 0.0;
    if (t < NP * NP) atomicMax(&ex[w][t / NP], biased_exponent(v[c]));
  }
  __syncwarp();
  for (int i = lane; i < NP; i += 32) EA[(size_t)b * NP + i] = (unsigned short)ex[w][i];
  int2* d = reinterpret_cast<int2*>(A) + (size_t)b * NP * NP;
#pragma unroll
  for (int c = 0; c < PER; ++c) {
    const int t = c * 32 + lane;
    if (t < NP * NP) d[fx_pos(NP, t / NP, t % NP)] = split_digits(v[c], ex[w][t / NP]);
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
FxOp diagonal_op(const DevLevel& L, int mode, const double* blocks, const unsigned short* exps) {
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

bool fx_encode(int np, int64_t blocks, double* A, unsigned short* EA, cudaStream_t s) {
  if (blocks < 1) return true;
  FX_NP_DISPATCH(np, (fx_encode_kernel<NP><<<(unsigned)((blocks + kFxWarps - 1) / kFxWarps), kFxThreads, 0, s>>>(
                         blocks, A, EA)));
  count_launch();
  return true;
}
