// Device side of the FP64 block products in integer digits (device_fixed.cu says why and how): the
// digits, their products and the work of one warp on one pack of rows, shared by the kernels of
// device_fixed.cu and the persistent V-cycle (device_persist.cu), whose results are therefore the same.
#pragma once

#include <cuda_runtime.h>

#include "device_fixed.h"
#include "device_kernels.cuh"

namespace fx {

constexpr int kFxThreads = 128;
constexpr int kFxWarps = kFxThreads / 32;
constexpr int kNotFinite = 0x7FF;     // exponent field of an infinity or NaN
constexpr int kScale = 2 * 1022;      // a sum's scale is the sum of two exponent fields, E + 1022 each
constexpr int kNoScale = -(1 << 24);  // scale of an empty sum, below every other

// blocks of a row per step of a group: the level-0 rows of A hold five on tetrahedra (Ahat one less)
constexpr int fx_chunk(int np, int mode, bool wpr) {
  return !wpr && mode <= 1 && (np == 4 || np == 10 || np == 20) ? 5 : 4;
}
constexpr bool fx_one(int mode) { return mode == 4 || mode == 6 || mode == 7; }   // one block per row
// resident CTAs of 128 threads per SM that the registers are held to
constexpr int fx_ctas_per_sm(int np) { return np > 10 ? 4 : 8; }

// position of entry (i, j) of a block in the digit layout
__host__ __device__ constexpr int fx_pos(int np, int i, int j) {
  return np % 2 == 0 ? ((j >> 1) * np + i) * 2 + (j & 1) : j * np + i;
}

__device__ __forceinline__ int biased_exponent(double v) {
  return (__double2hiint(v) >> 20) & 0x7FF;
}

// v 2^(58 - E) rounded to an integer, |v| < 2^E, as digits (E = em - 1022, em the biased
// exponent field of the largest value); subnormal values keep their own scale
// (exponent field 1, no implicit bit)
__device__ __forceinline__ int2 split_digits(double v, int em) {
  const long long bits = __double_as_longlong(v);
  const int e = (int)(bits >> 52) & 0x7FF;
  unsigned long long m = (unsigned long long)bits & 0xFFFFFFFFFFFFFull;
  if (e) m |= 1ull << 52;
  const int s = min(em - max(e, 1), 63);
  long long q = (long long)((((m << 6) >> s) + 1) >> 1);
  const long long sg = bits >> 63;
  q = (q ^ sg) - sg;
  const int lo = ((int)((unsigned int)q << 2)) >> 2;   // the low 30 bits, signed
  return make_int2((int)((q - lo) >> 30), lo);
}

// d 2^e: on the exponent field where the result is a normal number
__device__ __forceinline__ double scale2(double d, int e) {
  const int f = biased_exponent(d) + e;
  if (d == 0.0) return d;
  if (f >= 1 && f <= 2046 && biased_exponent(d) != 0)
    return __longlong_as_double(__double_as_longlong(d) + ((long long)e << 52));
  return scalbn(d, e);
}

// hi 2^60 + lo with 0 <= lo < 2^60, in units that its user keeps
struct Wide {
  static constexpr unsigned long long kLow = (1ull << 60) - 1;
  long long hi = 0;
  unsigned long long lo = 0;
  // rounded down to a multiple of 2^d and divided by it, d >= 0
  __device__ __forceinline__ void down(int d) {
    if (d < 60) {
      lo = (((unsigned long long)hi << (60 - d)) & kLow) | (lo >> d);
      hi >>= d;
    } else {
      lo = (unsigned long long)(hi >> min(d - 60, 63)) & kLow;
      hi >>= 63;
    }
  }
  __device__ __forceinline__ void add(const Wide& o) {
    lo += o.lo;
    hi += o.hi + (long long)(lo >> 60);
    lo &= kLow;
  }
};

// Bits between the sum of one block's products (below 2^61 units of hi) and a row's sum: the blocks of a
// row, each at its own scale, are added in units 2^kHead times those of the block of the largest, so
// that 2^26 terms fit and nothing above 2^-96 of that block's bound is lost.
constexpr int kHead = 20;

// A sum of digit products of one scale
struct Acc {
  long long hh = 0, mm = 0, ll = 0;
  // carries of one block's products into the higher sums
  __device__ __forceinline__ void carry() {
    mm += ll >> 30;
    ll &= 0x3FFFFFFF;
    hh += mm >> 30;
    mm &= 0x3FFFFFFF;
  }
  __device__ __forceinline__ unsigned long long low() const { return ((unsigned long long)mm << 30) | ll; }
  __device__ __forceinline__ Wide wide() const {
    Wide w;
    w.hi = hh;
    w.lo = low();
    return w;
  }
};

// (hi 2^60 + lo) 2^(e - 116), rounded once; e = EA + EX of the digits' scales (+ kHead after Wide::down by it)
__device__ __forceinline__ double fx_value(long long hi, unsigned long long lo, int e) {
  const int k = min(60, __clzll(hi ^ (hi >> 63)) - 1);   // low bits that fit beside hi in 63 bits
  long long v = (long long)((unsigned long long)hi << k) | (long long)(lo >> (60 - k));
  if (k < 60 && (lo << (4 + k)) != 0) v |= 1;   // the bits that did not fit, so that no tie is seen where there is none
  return scale2(__ll2double_rn(v), e - 56 - k);
}

template <int NP>
struct DigitRow {
  int h[NP], l[NP];
  // row i of the block at a (digit layout)
  __device__ __forceinline__ void load(const int2* __restrict__ a, int i) {
    if constexpr (NP % 2 == 0) {
      const int4* p = reinterpret_cast<const int4*>(a) + i;
#pragma unroll
      for (int j = 0; j < NP / 2; ++j) {
        const int4 t = __ldg(p + j * NP);
        h[2 * j] = t.x;
        l[2 * j] = t.y;
        h[2 * j + 1] = t.z;
        l[2 * j + 1] = t.w;
      }
    } else {
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        const int2 t = __ldg(a + j * NP + i);
        h[j] = t.x;
        l[j] = t.y;
      }
    }
  }
};

__device__ __forceinline__ void mac(Acc& s, int ah, int al, int xh, int xl) {
  s.hh += (long long)ah * xh;
  s.mm += (long long)ah * xl;
  s.mm += (long long)al * xh;
  s.ll += (long long)al * xl;
}

template <int NP>
__device__ __forceinline__ void fx_mac(const DigitRow<NP>& r, const int2* __restrict__ xs, Acc& s) {
  if constexpr (NP % 2 == 0) {
    const int4* x4 = reinterpret_cast<const int4*>(xs);
#pragma unroll
    for (int j = 0; j < NP / 2; ++j) {
      const int4 t = x4[j];
      mac(s, r.h[2 * j], r.l[2 * j], t.x, t.y);
      mac(s, r.h[2 * j + 1], r.l[2 * j + 1], t.z, t.w);
    }
  } else {
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      const int2 t = xs[j];
      mac(s, r.h[j], r.l[j], t.x, t.y);
    }
  }
  s.carry();
}

// what becomes of a row's sum (modes below); returns the dot partial of modes 0 and 3
template <int MODE>
__device__ __forceinline__ double finish(double acc, size_t o, double xo, double bo, double* y, double* y2,
                                         double omega, double dsum, const double* dotv) {
  if constexpr (MODE == 1) y[o] = bo - acc;
  else if constexpr (MODE == 3) {
    const double v = fma(omega, bo - xo - acc, xo);
    y[o] = v;
    return dotv ? fma(v, dotv[o], dsum) : dsum;
  } else if constexpr (MODE == 4) y[o] = xo + acc;
  else y[o] = acc;
  if constexpr (MODE == 6) y2[o] = omega * acc;
  return MODE == 0 ? fma(xo, acc, dsum) : dsum;
}

template <bool COHERENT>
__device__ __forceinline__ double vload(const double* p) {
  return cdgk::ld<COHERENT ? cdgk::kCoherent : cdgk::kPlain>(p);
}

// digits of one warp's gathered values in shared memory
template <int NP, int MODE, bool WPR>
struct Pack {
  static constexpr int RPW = 32 / NP;
  static constexpr bool ONE = fx_one(MODE);
  static constexpr int CH = ONE ? 1 : fx_chunk(NP, MODE, WPR);
  static constexpr int SPL = WPR ? RPW : 1;                       // groups that share a block row
  static constexpr int GS = CH * NP + 2 + (CH * NP) % 2;          // digits of one group's chunk (padded against bank conflicts)
  static constexpr int DIGITS = RPW * GS;
};

// The largest of the v of a group's n_p lanes, in each of them; v holds two 16-bit fields, each taken by itself
template <int NP>
__device__ __forceinline__ unsigned group_max(unsigned v, int sub, int i) {
  if constexpr (32 / NP == 1) {
    return __reduce_max_sync(0xffffffffu, v & 0xFFFFu) | __reduce_max_sync(0xffffffffu, v >> 16) << 16;
  } else {
#pragma unroll
    for (int o = 1; o < NP; o *= 2)   // the maximum over 2, 4, ... lanes from this one on, around the group
      v = __vmaxu2(v, __shfl_sync(0xffffffffu, v, sub * NP + (i + o < NP ? i + o : i + o - NP)));
    return v;
  }
}

// One warp on one pack of rows: acc = (A x)_(K, i), then by MODE: 0 y = acc; 1 y = b - acc;
// 3 y = x + omega (b - x - acc); 8 y = acc, block t meeting element t; with one block per row (no
// rowptr): 4 y += acc; 6 y = acc, y2 = omega acc; 7 y = acc.  Returns the dot partial of modes 0 and 3.
// q.cols: the rows' columns, q.width of them per row (missing: -1), so that the gathers of x need not
// wait for the row pointer; one-block modes meet element cols[K] (nullptr: K).
// COHERENT: vectors are read through L2 only (written earlier in the same kernel).  waited: whether the
// kernel has passed wait_for_inputs; the first pack's row pointers, columns and digits are read before.
template <int NP, int MODE, bool WPR, bool COHERENT>
__device__ __forceinline__ double fx_pack(const FxOp& q, int pack, int2* __restrict__ digits, double dsum,
                                          bool& waited) {
  using P = Pack<NP, MODE, WPR>;
  constexpr int RPW = P::RPW, CH = P::CH, SPL = P::SPL;
  constexpr bool ONE = P::ONE;
  const int2* A = reinterpret_cast<const int2*>(q.A);
  const int lane = threadIdx.x & 31;
  const int sub = lane / NP;
  const int i = lane - sub * NP;
  const bool grp = sub < RPW;
  int2* xs = digits + (grp ? sub : 0) * P::GS;
  const int K = WPR ? pack : pack * RPW + sub;
  const bool active = grp && K < q.n;
  int b0 = K, nb = active ? 1 : 0;
  if constexpr (!ONE) {
    b0 = active ? __ldg(q.rowptr + K) : 0;
    nb = active ? __ldg(q.rowptr + K + 1) - b0 : 0;
  }
  // blocks of this group: b0 + sub, b0 + sub + SPL, ... (WPR) or all of the row
  const int cnt = !active ? 0 : WPR ? (nb - sub + SPL - 1) / SPL : nb;
  const int first = WPR ? b0 + sub : b0;
  const int maxc = __reduce_max_sync(0xffffffffu, cnt);
  Wide sum;                                        // the row's sum so far, in units of scale E
  int E = kNoScale;
  bool special = false, bad_row = false;           // an infinity or NaN among the values, in the matrix row
  const bool writes = active && (!WPR || sub == 0);
  const size_t o = (size_t)K * NP + i;
  double xo = 0.0, bo = 0.0;                       // the epilogue's operands, on their way early
  auto inputs = [&]() {
    if (!waited) cdgk::wait_for_inputs();
    waited = true;
    if (writes) {
      if constexpr (MODE == 4) xo = vload<COHERENT>(q.y + o);
      if constexpr (MODE == 1 || MODE == 3) bo = vload<COHERENT>(q.b + o);
    }
  };
  if (maxc == 0) inputs();
  for (int base = 0; base < maxc; base += CH) {
    int J[CH];
    double xv[CH];
    unsigned ea[(CH + 1) / 2] = {}, em[(CH + 1) / 2];   // exponent fields of blocks and values, two to a word
    DigitRow<NP> row;
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      const int t = base + c;
      J[c] = -1;
      if constexpr (ONE) {
        if (active) J[c] = q.cols ? __ldg(q.cols + K) : K;
      } else if (q.cols) {
        const int tt = WPR ? sub + t * SPL : t;
        if (active && tt < q.width) J[c] = __ldg(q.cols + (size_t)K * q.width + tt);
      } else if (t < cnt) {
        J[c] = first + t * SPL;
      }
    }
#pragma unroll
    for (int c = 0; c < CH; ++c)
      if (base + c < cnt) ea[c / 2] |= (unsigned)__ldg(q.EA + (size_t)(first + (base + c) * SPL) * NP + i) << (c & 1) * 16;
    if (base < cnt) row.load(A + (size_t)(first + base * SPL) * NP * NP, i);
    if (base == 0) inputs();
#pragma unroll
    for (int c = 0; c < CH; ++c) xv[c] = J[c] >= 0 ? vload<COHERENT>(q.x + (size_t)J[c] * NP + i) : 0.0;
#pragma unroll
    for (int c = 0; c < CH; c += 2) {
      unsigned f = biased_exponent(xv[c]);
      if (c + 1 < CH) f |= (unsigned)biased_exponent(xv[c + 1 < CH ? c + 1 : c]) << 16;
      em[c / 2] = group_max<NP>(f, sub, i);
    }
    unsigned es[(CH + 1) / 2], ma = ea[0], mx = em[0], ms;   // the blocks' scales; the largest of all three
#pragma unroll
    for (int w = 0; w < (CH + 1) / 2; ++w) {
      em[w] = __vmaxu2(em[w], 0x00010001u);
      es[w] = ea[w] + em[w];
      ma = __vmaxu2(ma, ea[w]);
      mx = __vmaxu2(mx, em[w]);
      ms = w == 0 ? es[0] : __vmaxu2(ms, es[w]);
    }
    auto half = [](unsigned v, int c) { return (int)(v >> (c & 1) * 16 & 0xFFFF); };
    bad_row |= max(half(ma, 0), half(ma, 1)) == kNotFinite;
    special |= max(half(mx, 0), half(mx, 1)) == kNotFinite;
    if constexpr (!ONE) {
      const int top = max(E, max(half(ms, 0), half(ms, 1)) + kHead);
      sum.down(top - E);
      E = top;
    } else {
      E = half(ms, 0);
    }
    __syncwarp();
#pragma unroll
    for (int c = 0; c < CH; ++c)
      if (base + c < maxc) {   // the same in every lane
        const int2 d = split_digits(xv[c], half(em[c / 2], c));
        if (grp) xs[c * NP + i] = d;
      }
    __syncwarp();
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      if (base + c < cnt) {
        Acc s;
        fx_mac<NP>(row, xs + c * NP, s);
        if (c + 1 < CH && base + c + 1 < cnt) row.load(A + (size_t)(first + (base + c + 1) * SPL) * NP * NP, i);
        Wide w = s.wide();
        if constexpr (!ONE) w.down(E - half(es[c / 2], c));
        sum.add(w);
      }
    }
  }
  double acc = 0.0;
  if (special) {
    // an infinity or NaN among the values: FP64 products, so that it spreads as IEEE arithmetic says
    for (int t = 0; t < cnt; ++t) {
      const int blk = first + t * SPL;
      const int J = ONE ? (q.cols ? q.cols[K] : K) : q.cols ? q.cols[(size_t)K * q.width + (WPR ? sub + t * SPL : t)] : blk;
      const double* xj = q.x + (size_t)J * NP;
      const int e = __ldg(q.EA + (size_t)blk * NP + i) - 1022 - 58;
      for (int j = 0; j < NP; ++j) {
        const int2 d = A[(size_t)blk * NP * NP + fx_pos(NP, i, j)];
        acc = fma(scale2(__ll2double_rn(((long long)d.x << 30) + d.y), e), vload<COHERENT>(xj + j), acc);
      }
    }
  }
  bool in_fp64 = special;
  if constexpr (WPR && RPW > 1) {
    // sum over the groups of the row: the integer sums, brought to one scale, exactly
    in_fp64 = __any_sync(0xffffffffu, special && grp);
    if (in_fp64) {
      if (!special) acc = fx_value(sum.hi, sum.lo, E - kScale);
#pragma unroll
      for (int m = RPW; m > 1; m = (m + 1) / 2) {
        const int h = (m + 1) / 2;
        const double t = __shfl_down_sync(0xffffffffu, acc, h * NP);
        if (sub + h < m) acc += t;
      }
    } else {
      int top = E;
#pragma unroll
      for (int m = RPW; m > 1; m = (m + 1) / 2) {
        const int h = (m + 1) / 2;
        const int t = __shfl_down_sync(0xffffffffu, top, h * NP);
        if (sub + h < m) top = max(top, t);
      }
      top = __shfl_sync(0xffffffffu, top, i);
      sum.down(max(top - E, 0));   // a lane without a group may hold more than group 0
      E = top;
#pragma unroll
      for (int m = RPW; m > 1; m = (m + 1) / 2) {
        const int h = (m + 1) / 2;
        Wide t;
        t.hi = __shfl_down_sync(0xffffffffu, sum.hi, h * NP);
        t.lo = __shfl_down_sync(0xffffffffu, sum.lo, h * NP);
        if (sub + h < m) sum.add(t);
      }
    }
  }
  if (!in_fp64) acc = fx_value(sum.hi, sum.lo, E - kScale);
  if constexpr (WPR && RPW > 1)
    if (__any_sync(0xffffffffu, bad_row))
#pragma unroll
      for (int m = RPW; m > 1; m = (m + 1) / 2) {
        const int h = (m + 1) / 2;
        const int t = __shfl_down_sync(0xffffffffu, (int)bad_row, h * NP);
        bad_row |= sub + h < m && t;
      }
  if (bad_row) acc = nan("");
  if (writes && (MODE == 3 || (MODE == 0 && q.dot))) xo = vload<COHERENT>(q.x + o);
  return writes ? finish<MODE>(acc, o, xo, bo, q.y, q.y2, q.omega, dsum, q.dotv) : dsum;
}

}  // namespace fx
