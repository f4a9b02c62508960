// Device helpers shared by the solve-phase kernels: read-only loads, aligned
// vector loads of n_p consecutive values, and row i of (A x)_K of a block-sparse
// operator (n_p x n_p row-major blocks, element-major vectors).
#pragma once

#include <cuda_runtime.h>

namespace cdgk {
// Programmatic dependent launch: a kernel launched with launch_dep may start while the kernel before it
// in the stream still runs.  Before this it may only read what no kernel of a solve writes (row
// pointers, columns, matrix blocks); every thread passes here before it reads or writes anything else,
// or returns: the wait ends when all earlier kernels are complete and their writes visible.  Then the
// next kernel may start in the same way.  What an earlier kernel writes is not read-only for the life of
// this one: its pointers carry no __restrict__, which would let the compiler take the read-only path.
__device__ __forceinline__ void wait_for_inputs() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename T>
__device__ __forceinline__ T ldg(const T* p) { return __ldg(p); }

// Conversions between binary32 and binary64 built from the IEEE 754 bit
// fields with integer operations.  On this GPU a conversion instruction to or
// from FP64 runs at the rate of the FP64 pipe (about two per clock per SM),
// as slow as an FP64 FMA; the vector kernels of the FP64 CG would spend as
// much time converting as computing.  Both functions give the correctly
// rounded IEEE result; the cases outside the common range (zero is handled
// here; subnormals, infinities and NaN) fall back to the conversion
// instruction.
//
// binary32 -> binary64 is exact: sign, exponent rebiased by 1023 - 127,
// the 23 fraction bits placed at the top of the 52.
__device__ __forceinline__ double f32_to_f64(float f) {
  const unsigned int u = __float_as_uint(f);
  const unsigned int e = (u >> 23) & 0xFFu;
  const unsigned long long sgn = (unsigned long long)(u & 0x80000000u) << 32;
  if (e - 1u < 0xFEu)   // 1 <= e <= 254: a normal number
    return __longlong_as_double(
        (long long)(sgn | ((unsigned long long)(e + 896u) << 52) | ((unsigned long long)(u & 0x7FFFFFu) << 29)));
  if ((u & 0x7FFFFFFFu) == 0u) return __longlong_as_double((long long)sgn);   // +-0
  return (double)f;
}

// binary64 -> binary32, round to nearest, ties to even: for a result in the
// normal binary32 range keep the top 23 fraction bits and add one unit when
// the 29 dropped bits exceed half a unit, or equal it with an odd kept part.
// The carry of that addition moves into the exponent field as it should, and
// from the largest finite value into the infinity encoding.
__device__ __forceinline__ float f64_to_f32(double d) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
  const unsigned int sgn = (unsigned int)(b >> 32) & 0x80000000u;
  const int e = (int)((b >> 52) & 0x7FF) - 1023;
  if (e >= -126 && e <= 127) {
    const unsigned long long m = b & 0xFFFFFFFFFFFFFull;
    const unsigned int kept = (unsigned int)(m >> 29);
    const unsigned int rest = (unsigned int)(m & 0x1FFFFFFFull);
    unsigned int r = ((unsigned int)(e + 127) << 23) | kept;
    if (rest > 0x10000000u || (rest == 0x10000000u && (kept & 1u))) r += 1u;
    return __uint_as_float(sgn | r);
  }
  if ((b << 1) == 0ull) return __uint_as_float(sgn);   // +-0
  return (float)d;
}

template <typename TO, typename TI>
__device__ __forceinline__ TO cvt(TI v) {
  if constexpr (sizeof(TO) == 8 && sizeof(TI) == 4) return f32_to_f64(v);
  else if constexpr (sizeof(TO) == 4 && sizeof(TI) == 8) return f64_to_f32(v);
  else return (TO)v;
}

// How vector values are read: kReadOnly (ld.global.nc) for what nothing writes while the kernel is
// resident; kPlain for what the kernel before may still be writing when this one starts
// (wait_for_inputs); kCoherent through L2 only, for what other CTAs of the same kernel write.
enum Access { kReadOnly, kPlain, kCoherent };

template <Access A>
__device__ __forceinline__ float ld(const float* p) {
  if constexpr (A == kReadOnly) return __ldg(p);
  if constexpr (A == kCoherent) return __ldcg(p);
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
template <Access A>
__device__ __forceinline__ double ld(const double* p) {
  if constexpr (A == kReadOnly) return __ldg(p);
  if constexpr (A == kCoherent) return __ldcg(p);
  double v;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}
template <Access A>
__device__ __forceinline__ float2 ld(const float2* p) {
  if constexpr (A == kReadOnly) return __ldg(p);
  if constexpr (A == kCoherent) return __ldcg(p);
  float2 v;
  asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}
template <Access A>
__device__ __forceinline__ double2 ld(const double2* p) {
  if constexpr (A == kReadOnly) return __ldg(p);
  if constexpr (A == kCoherent) return __ldcg(p);
  double2 v;
  asm volatile("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
  return v;
}

// NP consecutive values as aligned vector loads
template <typename T, int NP, Access A = kReadOnly>
struct VecLoad;
template <int NP, Access A>
struct VecLoad<float, NP, A> {
  static __device__ __forceinline__ void load(const float* p, float* v) {
    if constexpr (NP % 2 == 0) {
#pragma unroll
      for (int j = 0; j < NP; j += 2) {
        const float2 t = ld<A>(reinterpret_cast<const float2*>(p + j));
        v[j] = t.x;
        v[j + 1] = t.y;
      }
    } else {
#pragma unroll
      for (int j = 0; j < NP; ++j) v[j] = ld<A>(p + j);
    }
  }
};
template <int NP, Access A>
struct VecLoad<double, NP, A> {
  static __device__ __forceinline__ void load(const double* p, double* v) {
    if constexpr (NP % 2 == 0) {
#pragma unroll
      for (int j = 0; j < NP; j += 2) {
        const double2 t = ld<A>(reinterpret_cast<const double2*>(p + j));
        v[j] = t.x;
        v[j + 1] = t.y;
      }
    } else {
#pragma unroll
      for (int j = 0; j < NP; ++j) v[j] = ld<A>(p + j);
    }
  }
};

// Row i of (A x)_K for block row K: sum over the blocks of the row, block by
// block and column by column (the same order for every UNR).
template <typename T, int NP, bool VEC, int UNR, bool COHERENT = false>
__device__ __forceinline__ T row_acc(int K, int i, const int* __restrict__ rowptr, const int* __restrict__ col,
                                     const T* __restrict__ A, const T* x) {
  constexpr Access X = COHERENT ? kCoherent : kPlain;
  T acc = T(0);
  const int b0 = rowptr[K], b1 = rowptr[K + 1];
  if constexpr (VEC) {
    // even n_p: the row of the block and x_J are 8-byte (FP32) / 16-byte
    // (FP64) aligned runs, read as float2 / double2; UNR blocks per step
    // keep UNR times the loads in flight
    int bb = b0;
    for (; bb + UNR <= b1; bb += UNR) {
      T av[UNR][NP], xv[UNR][NP];
#pragma unroll
      for (int u = 0; u < UNR; ++u) {
        const int J = ldg(col + bb + u);
        VecLoad<T, NP>::load(A + (size_t)(bb + u) * NP * NP + i * NP, av[u]);
        VecLoad<T, NP, X>::load(x + (size_t)J * NP, xv[u]);
      }
#pragma unroll
      for (int u = 0; u < UNR; ++u)
#pragma unroll
        for (int j = 0; j < NP; ++j) acc = fma(av[u][j], xv[u][j], acc);
    }
    for (; bb < b1; ++bb) {
      T av[NP], xv[NP];
      VecLoad<T, NP>::load(A + (size_t)bb * NP * NP + i * NP, av);
      VecLoad<T, NP, X>::load(x + (size_t)ldg(col + bb) * NP, xv);
#pragma unroll
      for (int j = 0; j < NP; ++j) acc = fma(av[j], xv[j], acc);
    }
  } else {
    for (int bb = b0; bb < b1; ++bb) {
      const T* a = A + (size_t)bb * NP * NP + i * NP;
      const T* xj = x + (size_t)ldg(col + bb) * NP;
#pragma unroll
      for (int j = 0; j < NP; ++j) acc = fma(ldg(a + j), ld<X>(xj + j), acc);
    }
  }
  return acc;
}

// Sums over a CTA of WARPS warps (threads x), done by one warp: the FP64 pipe of this GPU takes 64 clocks
// for a warp's addition, so a shuffle reduction in every warp of every CTA costs microseconds (64 warps
// per SM, five additions each: 2.5 us per sum).  One warp adds the other warps' lanes pairwise and then
// its own lanes: WARPS + 4 additions per CTA; CTAs on one SM take different warps, and so quadrants.
template <int WARPS>
__device__ __forceinline__ int summing_warp() { return (int)(blockIdx.x + blockIdx.x / 152) % WARPS; }

__device__ __forceinline__ double lanes_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// the sum of v over the CTA, valid in the summing warp; red: [32 WARPS] in shared memory
template <int WARPS>
__device__ __forceinline__ double cta_sum(double v, double* red) {
  __syncthreads();   // red may still be read
  red[threadIdx.x] = v;
  __syncthreads();
  if ((int)(threadIdx.x >> 5) != summing_warp<WARPS>()) return 0.0;
  double t[WARPS];
#pragma unroll
  for (int w = 0; w < WARPS; ++w) t[w] = red[w * 32 + (threadIdx.x & 31)];
#pragma unroll
  for (int h = 1; h < WARPS; h *= 2)
#pragma unroll
    for (int w = 0; w + h < WARPS; w += 2 * h) t[w] += t[w + h];
  return lanes_sum(t[0]);
}

// The same for a whole warp on one block row: floor(32 / n_p) groups of n_p lanes share its blocks
// (group g takes blocks g, g + G, ...; two at a time in flight), lane i of a group row i; the sums
// of the groups are added in a fixed order.  Valid in the lanes of group 0.  x aligned for VecLoad.
template <typename T, int NP, bool COHERENT = false>
__device__ __forceinline__ T split_row_acc(int K, const int* __restrict__ rowptr, const int* __restrict__ col,
                                           const T* __restrict__ A, const T* x) {
  constexpr int G = 32 / NP;
  constexpr Access X = COHERENT ? kCoherent : kPlain;
  const int lane = threadIdx.x & 31;
  const int sub = lane / NP, i = lane - sub * NP;
  T acc = T(0);
  if (sub < G) {
    const int b1 = ldg(rowptr + K + 1);
    int bb = ldg(rowptr + K) + sub;
    for (; bb + G < b1; bb += 2 * G) {
      T av[2][NP], xv[2][NP];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        VecLoad<T, NP>::load(A + (size_t)(bb + u * G) * NP * NP + i * NP, av[u]);
        VecLoad<T, NP, X>::load(x + (size_t)ldg(col + bb + u * G) * NP, xv[u]);
      }
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int j = 0; j < NP; ++j) acc = fma(av[u][j], xv[u][j], acc);
    }
    if (bb < b1) {
      T av[NP], xv[NP];
      VecLoad<T, NP>::load(A + (size_t)bb * NP * NP + i * NP, av);
      VecLoad<T, NP, X>::load(x + (size_t)ldg(col + bb) * NP, xv);
#pragma unroll
      for (int j = 0; j < NP; ++j) acc = fma(av[j], xv[j], acc);
    }
  }
#pragma unroll
  for (int m = G; m > 1; m = (m + 1) / 2) {
    const int h = (m + 1) / 2;
    const T t = __shfl_down_sync(0xffffffffu, acc, h * NP);
    if (sub + h < m) acc += t;
  }
  return acc;
}

// Brings the first blocks that the warp will multiply, and their columns, towards it (split_row_acc).
template <typename T, int NP>
__device__ __forceinline__ void touch_row(int K, const int* __restrict__ rowptr, const int* __restrict__ col,
                                          const T* __restrict__ A) {
  constexpr int G = 32 / NP;
  const int lane = threadIdx.x & 31;
  const int bb = ldg(rowptr + K) + lane / NP;
  if (lane / NP < G && bb < ldg(rowptr + K + 1)) {
    asm volatile("prefetch.global.L1 [%0];" ::"l"(col + bb));
    asm volatile("prefetch.global.L1 [%0];" ::"l"(A + (size_t)bb * NP * NP + (lane % NP) * NP));
  }
}

// The sum over the children K of agglomerate Ag of (L_K^T r_K)_i, its children shared by the groups
// of the warp in the same way; valid in the lanes of group 0.
template <typename T, int NP, bool COHERENT = false>
__device__ __forceinline__ T split_restrict(int Ag, const int* __restrict__ childptr, const T* __restrict__ L,
                                            const T* r) {
  constexpr int G = 32 / NP;
  constexpr Access X = COHERENT ? kCoherent : kPlain;
  const int lane = threadIdx.x & 31;
  const int sub = lane / NP, i = lane - sub * NP;
  T acc = T(0);
  if (sub < G) {
    const int k1 = ldg(childptr + Ag + 1);
    for (int K = ldg(childptr + Ag) + sub; K < k1; K += G) {
      const T* LK = L + (size_t)K * NP * NP + i;
      const T* rk = r + (size_t)K * NP;
#pragma unroll
      for (int j = 0; j < NP; ++j) acc = fma(ldg(LK + j * NP), ld<X>(rk + j), acc);
    }
  }
#pragma unroll
  for (int m = G; m > 1; m = (m + 1) / 2) {
    const int h = (m + 1) / 2;
    const T t = __shfl_down_sync(0xffffffffu, acc, h * NP);
    if (sub + h < m) acc += t;
  }
  return acc;
}

}  // namespace cdgk
