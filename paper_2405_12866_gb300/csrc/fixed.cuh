// FP64 numbers in 64-bit fixed point, for the kernels whose FP64 work is
// products and sums of numbers with a known bound: an FP64 FMA costs a warp 60
// cycles on this chip, a 32 x 32 -> 64 bit integer FMA about 7, and a product
// takes three of them.
#pragma once
#include "qfs_common.cuh"

namespace qfs {

// x with its sign flipped if f (an FP64 negation that is not folded into an
// FMA costs an FP64 instruction; this is integer).
__device__ __forceinline__ double neg_if(double x, bool f) {
  return __hiloint2double(__double2hiint(x) ^ (f ? 0x80000000 : 0), __double2loint(x));
}

// x times 2^e for a finite x, exactly, underflow to zero (FP64 arithmetic is
// scarce; this is integer).
__device__ __forceinline__ double scale_exp(double x, int e) {
  const int hi = __double2hiint(x);
  const int f = ((hi >> 20) & 0x7ff);
  if (f == 0x7ff) return x;  // Inf and NaN stay what they are
  if (f == 0 || f + e <= 0) return 0.0;
  return __hiloint2double(hi + (e << 20), __double2loint(x));
}

// Fixed point: a number is (hi, lo) with value hi 2^30 + lo, |lo| <= 2^29, in
// units of 2^-60; a complex one is int4 {re hi, re lo, im hi, im lo}.
constexpr int kFxBits = 60, kFxLow = 30;
__device__ __forceinline__ int2 fx_split(long long v) {
  return int2{(int)((v + (1LL << (kFxLow - 1))) >> kFxLow), ((int)v << (32 - kFxLow)) >> (32 - kFxLow)};
}
__device__ __forceinline__ long long fx_value(int hi, int lo) { return ((long long)hi << kFxLow) + lo; }
// round(x 2^(kFxBits - e)) for |x| < 2^(e + 1), without FP64 instructions.
__device__ __forceinline__ int2 fx_from(double x, int e) {
  const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7ff;
  long long m = ((long long)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(x);
  const int sh = ex - 1075 + kFxBits - e;
  if (sh >= 0) m = ex == 0 ? 0 : m << min(sh, 10);
  else m = sh < -54 ? 0 : (m + (1LL << (-sh - 1))) >> -sh;
  return fx_split(hi < 0 ? -m : m);
}
__device__ __forceinline__ int4 fx_from2(double2 z, int e) {
  const int2 x = fx_from(z.x, e), y = fx_from(z.y, e);
  return int4{x.x, x.y, y.x, y.y};
}
// Whether exponent field t of a matrix' largest entry (0: all zeros) is too far
// out for products scaled back by scale_exp (which knows neither overflow nor
// denormals); so are Inf and NaN.
__device__ __forceinline__ bool fx_out_of_range(int t) { return t != 0 && (t < 500 || t > 1500); }
// acc + a b of 32-bit numbers, in 64 bits.
__device__ __forceinline__ long long mad64(int a, int b, long long acc) { return (long long)a * b + acc; }
// A sum of products of fixed-point numbers: high x high, and the cross terms
// 2^-30 below.  (low x low, 2^-60 below, is left out.)
struct FxSum {
  long long h = 0, c = 0, d = 0;
  __device__ __forceinline__ void add(int ah, int al, int bh, int bl) {
    h = mad64(ah, bh, h);
    c = mad64(ah, bl, c);
    d = mad64(al, bh, d);
  }
  __device__ __forceinline__ long long value() const {
    return h + ((c + d + (1LL << (kFxLow - 1))) >> kFxLow);
  }
};

// The entries of a matrix product of 2^n terms, one component per thread, with a
// scale for every row of the left matrix and every column of the right one, from
// their largest exponent fields t, and room for 2 2^n terms: the high sums stay
// below 2^62, each cross sum below 2^62 and both together below 2^63.  That room
// puts the result's scale up to 2^9 above the result, so the low x low products
// and the bits of the cross sums below 2^-60 count here.
__device__ __forceinline__ int fx_top(double2 z) {
  return max((__double2hiint(z.x) >> 20) & 0x7ff, (__double2hiint(z.y) >> 20) & 0x7ff);
}
__device__ __forceinline__ int fx_row_exp(int t, int n) { return t - 1022 + n - 1; }
__device__ __forceinline__ int fx_col_exp(int t, int n) { return t - 1022 + max(n - 2, 1); }
struct FxDot {
  FxSum t;
  long long low = 0;  // low x low, in units of 2^-88
  // Component im of x y; its low x low part goes to l (two times up to 2^26).
  __device__ __forceinline__ void add(int4 x, int4 y, int im, int& l) {
    const int b1 = im ? y.w : y.y, a2 = im ? x.w : -x.w, b2 = im ? y.y : y.w;
    t.add(x.x, x.y, im ? y.z : y.x, b1);
    t.add(im ? x.z : -x.z, a2, im ? y.x : y.z, b2);
    l += __mulhi(x.y, b1) + __mulhi(a2, b2);
  }
  // Terms k = first, first + STEP, ... < n of row x and column y, which has its
  // entries `ld` apart.  (The low x low parts of eight terms are summed in 32 bits:
  // in 64, with a shift for each, the batched set-up took 60 us instead of 52.)
  template <int STEP>
  __device__ __forceinline__ void run(const int4* x, const int4* y, int ld, int first, int n, int im) {
    int k = first;
    for (; k + 7 * STEP < n; k += 8 * STEP) {
      int l = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) add(x[k + i * STEP], y[(k + i * STEP) * ld], im, l);
      low += l;
    }
    int l = 0;
    for (; k < n; k += STEP) add(x[k], y[k * ld], im, l);
    low += l;
  }
  __device__ __forceinline__ long long cross() const { return t.c + t.d + (low << 2); }
};
__device__ __forceinline__ double fx_dot_value(long long high, long long cross, int e) {
  return scale_exp(fma((double)cross, 1.0 / (1LL << kFxLow), (double)high), e - kFxBits);
}

// Where entry e = (column << n) | row of a slice sits: bits 4 and 5 are folded
// into the bank bits, so that the units of a gate on any two neighbouring row
// bits (whose lanes skip those bits) spread over the banks.  Linear over XOR,
// and a permutation of every 16 entries: below 16 rows a slice need not be a
// multiple of that, so there nothing is folded (fold = 0).
__device__ __forceinline__ uint32_t swz(uint32_t e, uint32_t fold) {
  return e ^ (((e >> 4) & fold) * 5u) ^ (((e >> 5) & fold) * 10u);
}
__device__ __forceinline__ uint32_t swz_fold(int n) { return n >= 4 ? 1u : 0u; }

// The row bits of a gate's two qubits.
struct PairBits {
  int pa, pb, lo, hi;
};
__device__ __forceinline__ PairBits pair_bits(int pa, int pb) { return PairBits{pa, pb, min(pa, pb), max(pa, pb)}; }

// Fixed point: out = G in (adj: G^dagger in) on a slice of `units` units, one
// component of one output row per lane.  out = sum p v.x + q v.y in three
// integer FMAs per product.  In place when out = in.
template <int NT>
__device__ __forceinline__ void fx_apply(const int4* in, int4* out, const int4* gate, const PairBits& g, bool adj, int units, int n) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, rbits = n - 2;
  const uint32_t fold = swz_fold(n);
  const int x = (lane >> 1) & 3, im = lane & 1;
  int2 p[4], q[4];
  uint32_t xo[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int4 w = gate[adj ? 4 * j + x : 4 * x + j];
    const int sy = adj ? -1 : 1;  // conj(G) for the adjoint
    const int2 re{w.x, w.y}, iy{sy * w.z, sy * w.w};
    p[j] = im ? iy : re;
    q[j] = im ? re : int2{-iy.x, -iy.y};
    xo[j] = swz(((uint32_t)(j >> 1) << g.pa) | ((uint32_t)(j & 1) << g.pb), fold);
  }
  const uint32_t mine = xo[x];
  for (int u0 = warp * 4; u0 < units; u0 += NT / 8) {
    const int u = u0 + (lane >> 3);
    const uint32_t b = swz(((uint32_t)(u >> rbits) << n) |
                           insert_two_zero_bits((uint32_t)u & ((1u << rbits) - 1u), g.lo, g.hi), fold);
    FxSum t;
    if (u < units) {
      int4 v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = in[b ^ xo[j]];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        t.add(p[j].x, p[j].y, v[j].x, v[j].y);
        t.add(q[j].x, q[j].y, v[j].z, v[j].w);
      }
    }
    const int2 r = fx_split(t.value());
    __syncwarp();  // (in place: the eight lanes of a unit have read it)
    if (u < units) reinterpret_cast<int2*>(out + (b ^ mine))[im] = r;
  }
}

}  // namespace qfs
