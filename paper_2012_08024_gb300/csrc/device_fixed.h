// FP64 block-sparse products by exact integer arithmetic (device_fixed.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

// One product with a block-sparse matrix in digit form and what is done with it:
// mode 0 y = A x (dot: per-CTA partials of x . y, fx_grid of them), 1 y = b - A x,
// 3 y = x + omega (b - x - A x) (dot: partials of y . dotv), 8 y = A x with block t meeting element t; with one block per row
// (no rowptr): 4 y += A x, 6 y = A x and y2 = omega A x, 7 y = A x.
// x and y do not overlap.
struct FxOp {
  int mode = 0, np = 0, n = 0;
  int64_t blocks = 0;         // blocks of the matrix
  const int* rowptr = nullptr;
  const int* cols = nullptr;  // [n][width], -1 behind a row's last block; one-block modes: [n] or nullptr (K)
  int width = 0;
  const void* A = nullptr;    // digits
  const unsigned short* EA = nullptr;   // [blocks][np] exponents of the digits (fx_encode)
  const double* x = nullptr;
  const double* b = nullptr;
  double* y = nullptr;
  double* y2 = nullptr;
  double omega = 0.0;
  double* dot = nullptr;
  const double* dotv = nullptr;
};

constexpr int kFxSms = 152;

// Whether a level's block rows take a warp each: while they then fit on the GPU at once (32 warps per
// SM; 16 above n_p = 10), or, up to four times as many, are long (three and more blocks per group of
// n_p lanes): a row's blocks, not the number of rows, are what there is to spread.  FP64, 256^2, p = 3:
// 4,135 rows of 7 blocks 7.4 -> 6.4 us; 24^3 tetrahedra, p = 2: 4,875 rows of 10 blocks 12.2 -> 8.8 us;
// but 8,102 rows of 7 blocks at p = 2 (five groups share a row) 6.7 -> 8.9 us.
inline bool warp_per_row(int np, int n, int64_t blocks) {
  const int groups = 32 / np, resident = kFxSms * (np > 10 ? 16 : 32);
  return groups > 1 && (n <= resident || (blocks >= (int64_t)n * 3 * groups && n <= 4 * resident));
}

struct DevLevel;
// products with a level's operators: A (modes 0, 1) or Ahat (3); a diagonal of blocks (6, 7); the
// prolongation to level F from its parents (4, 7); the restriction from F to the next level C (8)
FxOp operator_op(const DevLevel& L, int mode);
FxOp diagonal_op(const DevLevel& L, int mode, const double* blocks, const unsigned short* exps);
FxOp prolong_op(const DevLevel& F, int mode = 4);
FxOp restrict_op(const DevLevel& F, const DevLevel& C);

unsigned fx_grid(const FxOp& o);                  // CTAs of fx_run
bool fx_run(const FxOp& o, cudaStream_t s);       // false: no instance for this np
// FP64 blocks [blocks][np][np] to digits, in place; EA [blocks][np]: the exponent field of the largest entry
// of each of their scalar rows
bool fx_encode(int np, int64_t blocks, double* A, unsigned short* EA, cudaStream_t s);
