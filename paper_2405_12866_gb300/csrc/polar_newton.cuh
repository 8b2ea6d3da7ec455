// The gate update (Eq. 2 of the paper) of the sweep kernels that update a gate
// from one CTA: the unitary polar factor of A = E^dagger by a scaled Newton
// iteration in FP32 and corrections in 64-bit fixed point, on one warp.
//
// What bounds it is latency: one 4x4 matrix and a serial chain, in which an
// FP64 instruction costs 60 cycles (a 32 x 32 -> 64 bit integer FMA about 5),
// a shuffle 25.  So the iteration is FP32, and residuals that need more digits
// than FP32 holds are formed from integers.
//
//  1. Newton: X <- (z X + X^{-H} / z) / 2 from X = A (Higham, "Functions of
//     Matrices", ch. 8).  X^{-H} = conj(cofactor matrix) / conj(det), one
//     cofactor per lane, so no pivoting and no serial elimination.  The
//     scaling z follows Byers and Xu (SIAM J. Matrix Anal. Appl. 30, 2008):
//     from a >= sigma_max and b <= sigma_min, measured once, the interval that
//     holds the singular values is known for every later step, so the number
//     of steps is known too and no step measures convergence.
//  2. Corrections: with R = I - Q^H Q and K the skew part of Q^H A, Q <- Q +
//     Q R / 2 + D, where D is the derivative of the polar factor in the
//     direction Q K.  That derivative is the Newton iteration differentiated:
//     D <- (z D - Y D^H Y / z) / 2 with the inverses Y of step 1, in FP32.  A
//     correction of size d leaves ~d^2 + 1e-7 d.
//
// complex64 sweeps need the unitary factor only (their environments carry
// FP32 rounding), so they correct R and leave K out.
//
// One update on GB300, alone on its SM: 2400 cycles (complex64) and 6700 (FP64),
// of which the Newton steps take 380 each and a correction of K 2000; the
// update by a whole CTA that it replaced, with a one-sided FP32 Jacobi (7000
// cycles on a random matrix from the identity) and FP64 products, took 10,400
// and 15,400.
#pragma once
#include "fixed.cuh"
#include "polar4.cuh"

#include <limits.h>

namespace qfs {

constexpr int kNewtonMaxIt = 5;
// ||A||_F ||A^-1||_F above which the FP32 iteration is not used (the FP64
// Jacobi takes over).  The singular value ratio is then above 1000.
constexpr float kNewtonMaxCond = 4000.f;
// Scalings (z / 2, 1 / (2 z)) of steps 1, 2, ... for three ranges of that
// number: up to 4.6 (3 steps), 83 (4 steps) and 4000 (5 steps).  With the
// singular values in [1, u] before a step, z = 1 / sqrt(u) and u becomes
// (sqrt(u) + 1 / sqrt(u)) / 2; the steps end at u - 1 <= 1e-5, a distance from
// unitarity that two corrections square to rounding.  Constants instead of a
// running u: its square roots and reciprocals would be a second serial chain.
static __constant__ float2 kNewtonZ[3][kNewtonMaxIt - 1] = {
    {{0.437603f, 0.571294f}, {0.497790f, 0.502219f}, {0.5f, 0.5f}, {0.5f, 0.5f}},
    {{0.232871f, 1.073557f}, {0.437449f, 0.571496f}, {0.497779f, 0.502231f}, {0.5f, 0.5f}},
    {{0.088903f, 2.812059f}, {0.293562f, 0.851611f}, {0.467234f, 0.535064f}, {0.499427f, 0.500574f}}};

// Scratch of one update.  4x4 matrices have entry [r][c] at 4c + r.
struct NewtonSh {
  int4 A[16];                   // A scaled by a power of two, fixed point (corrections of K only)
  int4 Q[16];                   // the iterate, fixed point
  float2 Y[kNewtonMaxIt][16];   // X^{-H} of each step
  float2 z[kNewtonMaxIt];       // its scaling: z / 2, 1 / (2 z)
  double2 polar[32];            // scratch of the FP64 Jacobi
};

// Reciprocal and reciprocal square root of the hardware (about 1 ulp).
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// TwoSum (Knuth): hi + lo = a + b exactly.
__device__ __forceinline__ void two_sum(float a, float b, float& hi, float& lo) {
  hi = __fadd_rn(a, b);
  const float t = __fsub_rn(hi, a);
  lo = __fadd_rn(__fsub_rn(a, __fsub_rn(hi, t)), __fsub_rn(b, t));
}

// Shuffles within each 16-lane half of the warp, and 4x4 products there
// (entry [r][c] at lane 4c + r of the half).
__device__ __forceinline__ float2 shfl16(float2 v, int src) {
  return float2{__shfl_sync(FULL, v.x, src, 16), __shfl_sync(FULL, v.y, src, 16)};
}
__device__ __forceinline__ float2 mm16(float2 a, float2 b, int row, int col) {
  float2 acc{0.f, 0.f};
#pragma unroll
  for (int k = 0; k < 4; ++k) acc = cfma(shfl16(a, 4 * k + row), shfl16(b, 4 * col + k), acc);
  return acc;
}
__device__ __forceinline__ float2 mm16_ah(float2 a, float2 b, int row, int col) {
  float2 acc{0.f, 0.f};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float2 ak = shfl16(a, 4 * row + k), bk = shfl16(b, 4 * col + k);
    acc = cfma(float2{ak.x, -ak.y}, bk, acc);
  }
  return acc;
}

// Step 1, one warp: each 16-lane half holds a matrix A in x, its own (HALVES)
// or both the same.  On success x is the FP32 polar factor and (KEEP; one
// matrix) the inverses and scalings are in s.  Returns the steps, 0 in a half
// whose A is singular or too ill-conditioned.  (A butterfly sum is bitwise the
// same in every lane of a half, so every branch is uniform there.)
template <bool KEEP, bool HALVES>
__device__ __forceinline__ int newton_polar32(float2& x, NewtonSh* s) {
  const int lane = threadIdx.x & 31;
  const int l16 = lane & 15, row = l16 & 3, col = l16 >> 2;
  const int r0 = row == 0 ? 1 : 0, r1 = row <= 1 ? 2 : 1, r2 = row <= 2 ? 3 : 2;
  const int c0 = 4 * (col == 0 ? 1 : 0), c1 = 4 * (col <= 1 ? 2 : 1), c2 = 4 * (col <= 2 ? 3 : 2);
  const bool odd = (row + col) & 1;
  float2 y;
  float nc = 0.f, inv;
  // y = X^{-H}: the conjugate of (cofactor / determinant).
  auto inverse = [&](bool norm) {
    // The 3x3 minor without this lane's row and column, along its first row.
    const float2 a11 = shfl16(x, c1 + r1), a22 = shfl16(x, c2 + r2), a12 = shfl16(x, c2 + r1), a21 = shfl16(x, c1 + r2);
    const float2 a10 = shfl16(x, c0 + r1), a20 = shfl16(x, c0 + r2);
    const float2 a00 = shfl16(x, c0 + r0), a01 = shfl16(x, c1 + r0), a02 = shfl16(x, c2 + r0);
    const float2 m0 = cfma(a11, a22, cmul(float2{-a12.x, -a12.y}, a21));
    const float2 m1 = cfma(a12, a20, cmul(float2{-a10.x, -a10.y}, a22));
    const float2 m2 = cfma(a10, a21, cmul(float2{-a11.x, -a11.y}, a20));
    float2 cf = cmul(a00, m0);
    const float2 cg = cfma(a02, m2, cmul(a01, m1));
    cf.x += cg.x;
    cf.y += cg.y;
    if (odd) cf = float2{-cf.x, -cf.y};
    float2 det = cmul(x, cf);  // summed over a row
    if (norm) nc = fmaf(cf.x, cf.x, cf.y * cf.y);
    det.x += __shfl_xor_sync(FULL, det.x, 4);
    det.y += __shfl_xor_sync(FULL, det.y, 4);
    det.x += __shfl_xor_sync(FULL, det.x, 8);
    det.y += __shfl_xor_sync(FULL, det.y, 8);
    inv = rcp_approx(fmaf(det.x, det.x, det.y * det.y));
    const float dx = det.x * inv, dy = det.y * inv;
    y = float2{fmaf(cf.x, dx, cf.y * dy), fmaf(cf.x, dy, -cf.y * dx)};
  };
  // The first step measures both norms and picks the range.
  float nx = fmaf(x.x, x.x, x.y * x.y);
  inverse(true);
#pragma unroll
  for (int m = 1; m <= 8; m <<= 1) {
    nx += __shfl_xor_sync(FULL, nx, m);
    nc += __shfl_xor_sync(FULL, nc, m);
  }
  const float inv0 = __shfl_sync(FULL, inv, 0, 16), ny = nc * inv0;
  const float cond2 = nx * ny;
  // (NaN included.)  Cofactors carry rounding of 1e-7 |A|^3, the determinant
  // 1e-7 |A|^4: below 2e-6 |A|^4 it is not known, and of a matrix of rank 2
  // both are rounding, whose quotient says nothing about the condition.
  const float n2 = nx * nx;
  const bool ok = cond2 < kNewtonMaxCond * kNewtonMaxCond && n2 * n2 * inv0 < 2.5e11f;
  if (!HALVES && !ok) return 0;
  const int range = cond2 <= 4.6f * 4.6f ? 0 : cond2 <= 83.f * 83.f ? 1 : 2;
  // The other half may need more steps: further ones only converge further.
  const int last = 2 + (HALVES ? __reduce_max_sync(FULL, ok ? range : 0) : range);
  // z = (ny / nx)^(1/4) brings the singular values around 1.
  const float t = rsqrt_approx(ny * rcp_approx(nx)), z = rsqrt_approx(t);
  float2 h{0.5f * z, 0.5f * t * z};
  int it = 0;
#pragma unroll 1
  for (;;) {
    if (KEEP && lane < 16) {
      s->Y[it][l16] = y;
      if (lane == 0) s->z[it] = h;
    }
    x = float2{fmaf(h.x, x.x, h.y * y.x), fmaf(h.x, x.y, h.y * y.y)};
    if (it == last) break;
    h = kNewtonZ[range][it];
    ++it;
    inverse(false);
  }
  return ok ? it + 1 : 0;
}

// The Hermitian R = I - Q^H Q as 16 real values, one per lane of a half warp:
// 4 diagonal entries, then re and im of (0,1) (0,2) (0,3) (1,2) (1,3) (2,3).
struct NewtonPair {
  int c1, c2;   // columns of value lane & 15
  bool im, diag;
  int re_lane, im_lane;  // the values that hold entry [row][col] of this lane
  bool conj;             // ... which is below the diagonal
};
__device__ __forceinline__ NewtonPair newton_pair() {
  NewtonPair w;
  const int v = threadIdx.x & 15, row = v & 3, col = v >> 2;
  w.diag = v < 4;
  const int p = (v - 4) >> 1;
  w.im = !w.diag && ((v - 4) & 1);
  w.c1 = w.diag ? v : p < 3 ? 0 : p < 5 ? 1 : 2;
  w.c2 = w.diag ? v : p < 3 ? p + 1 : p < 5 ? p - 1 : 3;
  const int a = min(row, col), b = max(row, col), i = a == 0 ? b - 1 : a == 1 ? b + 1 : 5;
  w.re_lane = a == b ? a : 4 + 2 * i;
  w.im_lane = a == b ? -1 : 5 + 2 * i;
  w.conj = row > col;
  return w;
}
// Entry [row][col] of this lane from the lanes' values.
__device__ __forceinline__ float2 newton_entry(const NewtonPair& w, float r) {
  const float x = __shfl_sync(FULL, r, w.re_lane), y = __shfl_sync(FULL, r, max(w.im_lane, 0));
  return float2{x, w.im_lane < 0 ? 0.f : w.conj ? -y : y};
}

// R of an FP32 matrix (lanes as x of newton_polar32) by one warp in FP32 with
// exact products and a compensated sum (Ogita, Rump and Oishi's Dot2; error
// about 1e-14): two lanes per value, two rows each.
__device__ __forceinline__ float newton_residual32(float2 x, const NewtonPair& w) {
  const int h = (threadIdx.x >> 4) & 1;
  float s = w.diag && h == 0 ? -1.f : 0.f, e = 0.f;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const float2 q1 = shfl_c(x, 4 * w.c1 + 2 * h + k), q2 = shfl_c(x, 4 * w.c2 + 2 * h + k);
    const float b1 = w.im ? q2.y : q2.x, a2 = w.im ? -q1.y : q1.y, b2 = w.im ? q2.x : q2.y;
    const float p1 = q1.x * b1, p2 = a2 * b2;
    float f1, f2;
    e += fmaf(q1.x, b1, -p1) + fmaf(a2, b2, -p2);
    two_sum(s, p1, s, f1);
    two_sum(s, p2, s, f2);
    e += f1 + f2;
  }
  float f;
  two_sum(s, __shfl_xor_sync(FULL, s, 16), s, f);
  e += f + __shfl_xor_sync(FULL, e, 16);
  return -(s + e);
}

// R of s.Q by one warp, exact to 2^-59: two lanes per value, two rows each.
__device__ __forceinline__ float newton_residual_fx(const NewtonSh& s, const NewtonPair& w) {
  const int h = (threadIdx.x >> 4) & 1;
  FxSum t;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int4 q1 = s.Q[4 * w.c1 + 2 * h + k], q2 = s.Q[4 * w.c2 + 2 * h + k];
    // conj(q1) q2: re = x x + y y, im = x y - y x
    t.add(q1.x, q1.y, w.im ? q2.z : q2.x, w.im ? q2.w : q2.y);
    t.add(w.im ? -q1.z : q1.z, w.im ? -q1.w : q1.w, w.im ? q2.x : q2.z, w.im ? q2.y : q2.w);
  }
  long long v = t.value();
  v += __shfl_xor_sync(FULL, v, 16);
  return (float)((w.diag ? 1LL << kFxBits : 0LL) - v) * (1.f / (1LL << kFxBits));
}

// B = s.Q^H s.A and its skew part by one warp, in 2^-60: a lane forms one
// component (lanes 0..15 real parts) and gets the other.
__device__ __forceinline__ void newton_residual_polar(const NewtonSh& s, float2& b32, float2& k32) {
  const int lane = threadIdx.x & 31, l16 = lane & 15, im = lane >> 4, row = l16 & 3, col = l16 >> 2;
  FxSum t;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int4 q = s.Q[4 * row + r], a = s.A[4 * col + r];
    t.add(q.x, q.y, im ? a.z : a.x, im ? a.w : a.y);
    t.add(im ? -q.z : q.z, im ? -q.w : q.w, im ? a.x : a.z, im ? a.y : a.w);
  }
  const long long b = t.value();
  const long long o = __shfl_sync(FULL, b, 4 * row + col + 16 * im);  // B[col][row]
  const float k = (float)(im ? b + o : b - o) * (0.5f / (1LL << kFxBits)), bf = (float)b * (1.f / (1LL << kFxBits));
  const float ko = __shfl_xor_sync(FULL, k, 16), bo = __shfl_xor_sync(FULL, bf, 16);
  b32 = im ? float2{bo, bf} : float2{bf, bo};
  k32 = im ? float2{ko, k} : float2{k, ko};
}

// Unitary correction of an FP32 matrix x (lanes 0..15, and a copy in lanes
// 16..31) that is unitary to 1e-4 or better: q as newton_update returns it.
// x is left unitary to FP32 rounding.
__device__ __forceinline__ void newton_unitary(float2& x, NewtonSh& s, const NewtonPair& w, long long& q, bool last) {
  const int lane = threadIdx.x & 31;
  const int l16 = lane & 15, row = l16 & 3, col = l16 >> 2, im = lane >> 4;
  constexpr float kUnit = (float)(1LL << kFxBits);
  // The first correction needs R to FP32 digits only.
  float2 d = mm(x, newton_entry(w, newton_residual32(x, w)), row, col);
  q = __float2ll_rn((im ? x.y : x.x) * kUnit) + __float2ll_rn((im ? d.y : d.x) * (0.5f * kUnit));
  x = float2{fmaf(0.5f, d.x, x.x), fmaf(0.5f, d.y, x.y)};
  reinterpret_cast<int2*>(&s.Q[l16])[im] = fx_split(q);
  __syncwarp();
  if (!last) return;
  d = mm(x, newton_entry(w, newton_residual_fx(s, w)), row, col);
  q += __float2ll_rn((im ? d.y : d.x) * (0.5f * kUnit));
}

// Steps 1 and 2 in one warp for the matrix a32 (E^dagger scaled, its largest
// entry in [1/2, 2); lanes 0..15 hold [r][c] at 4c + r, lanes 16..31 a copy).
// POLISH: polar to 2^-59 for the fixed-point matrix in s.A; otherwise unitary
// to 2^-59 and polar to FP32.  False when the matrix is ill-conditioned (zero:
// a32 = 0) or the corrections do not converge; else q is a component of the
// factor's entry (real parts in lanes 0..15, imaginary parts of the same
// entries in lanes 16..31) in units of 2^-60.
template <bool POLISH>
__device__ __forceinline__ bool newton_update(float2 a32, NewtonSh& s, const NewtonPair& w, long long& q) {
  const int lane = threadIdx.x & 31;
  const int l16 = lane & 15, row = l16 & 3, col = l16 >> 2, im = lane >> 4;
  float2 x = a32;
  const int its = newton_polar32<POLISH, false>(x, &s);
  if (!its) return false;
  constexpr float kUnit = (float)(1LL << kFxBits);
  newton_unitary(x, s, w, q, !POLISH);
  if (!POLISH) return true;
  bool ok = true;
#pragma unroll 1
  for (int it = 0;; ++it) {
    float2 b, k;
    newton_residual_polar(s, b, k);
    const float2 r32 = newton_entry(w, newton_residual_fx(s, w));
    // The skew part of (I + R/2) B: what is left of it once Q is unitary.
    const float2 t = mm(r32, b, row, col);
    const float2 qr = mm(x, r32, row, col);
    const float2 tt = shfl_c(t, 4 * row + col);
    k.x = fmaf(0.25f, t.x - tt.x, k.x);
    k.y = fmaf(0.25f, t.y + tt.y, k.y);
    float2 d = mm(x, k, row, col);
    float2 y = s.Y[0][l16], h = s.z[0];
#pragma unroll 1
    for (int j = 1;; ++j) {
      const float2 v = mm(y, mm_ah(d, y, row, col), row, col);
      d = float2{fmaf(h.x, d.x, -h.y * v.x), fmaf(h.x, d.y, -h.y * v.y)};
      if (j == its) break;
      y = s.Y[j][l16];
      h = s.z[j];
    }
    d.x = fmaf(0.5f, qr.x, d.x);
    d.y = fmaf(0.5f, qr.y, d.y);
    // (For floats >= 0 the order of the bits is the order of the values.)
    const float big = __uint_as_float(__reduce_max_sync(FULL, __float_as_uint(fmaxf(fabsf(d.x), fabsf(d.y)))));
    ok = big < 1e-2f && !(it == 5 && big >= 1e-10f);
    if (!ok) break;
    q += __float2ll_rn((im ? d.y : d.x) * kUnit);
    if (big < 1e-10f) break;
    x = float2{x.x + d.x, x.y + d.y};
    reinterpret_cast<int2*>(&s.Q[l16])[im] = fx_split(q);
    __syncwarp();
  }
  return ok;
}

// The entry of lane l16 (lanes 0..15) from newton_update's components.
__device__ __forceinline__ double2 newton_entry64(long long q) {
  const double c = scale_exp((double)q, -kFxBits);
  return double2{c, __shfl_down_sync(FULL, c, 16)};
}

// The power of two that brings the largest entry of a matrix to [1, 2): minus
// its exponent (INT_MIN for a zero matrix), from the lanes' FP64 entries.
__device__ __forceinline__ int newton_exponent(double2 a) {
  const int ex = (__double2hiint(a.x) >> 20) & 0x7ff, ey = (__double2hiint(a.y) >> 20) & 0x7ff;
  const int e = __reduce_max_sync(FULL, max(ex, ey));
  return e == 0 ? INT_MIN : 1023 - e;
}

// newton_update's input E^dagger from the environment: value j (2 (4x + y) +
// {re, im}) of E in lane j, FP32, ...
__device__ __forceinline__ float2 newton_input32(float e) {
  const int l16 = threadIdx.x & 15;
  const float2 a{__shfl_sync(FULL, e, 2 * l16), -__shfl_sync(FULL, e, 2 * l16 + 1)};
  const int ex = (__float_as_int(a.x) >> 23) & 0xff, ey = (__float_as_int(a.y) >> 23) & 0xff;
  const int m = __reduce_max_sync(FULL, max(ex, ey));
  const float sc = m == 0 ? 0.f : __int_as_float(max(254 - m, 1) << 23);
  return float2{a.x * sc, a.y * sc};
}
// ... or the FP64 matrix m (entry 4x + y in lane 4x + y; E or its damped form),
// whose fixed-point copy goes to s.A too.
__device__ __forceinline__ float2 newton_input64(double2 m, NewtonSh& s) {
  const int lane = threadIdx.x & 31;
  const int expo = newton_exponent(m), ex = expo == INT_MIN ? 0 : expo - 1;  // largest entry to [1/2, 1)
  const double2 A{scale_exp(m.x, ex), neg_if(scale_exp(m.y, ex), true)};
  if (lane < 16) s.A[lane] = fx_from2(A, 0);
  __syncwarp();
  return expo == INT_MIN ? float2{0.f, 0.f} : float2{(float)A.x, (float)A.y};
}
// E (entry l16 in lanes l16 and l16 + 16) from its values in lanes 0..31, and
// (1 - beta) E + beta g^dagger (Appendix A of the paper; g: the old gate).
__device__ __forceinline__ double2 newton_env(double e) {
  const int l16 = threadIdx.x & 15;
  return double2{__shfl_sync(FULL, e, 2 * l16), __shfl_sync(FULL, e, 2 * l16 + 1)};
}
__device__ __forceinline__ double2 newton_damp(double2 m, double beta, const double2* g) {
  const int l16 = threadIdx.x & 15;
  const double2 go = g[4 * (l16 & 3) + (l16 >> 2)];
  return double2{(1.0 - beta) * m.x + beta * go.x, (1.0 - beta) * m.y - beta * go.y};
}
// The FP64 Jacobi for what newton_update does not take (it also completes
// rank-deficient matrices): the factor's entry of lane l16.
__device__ __forceinline__ double2 newton_fallback(double2 m, NewtonSh& s) {
  const int l16 = threadIdx.x & 15;
  return warp_polar4(double2{m.x, neg_if(m.y, true)}, double2{(l16 & 3) == (l16 >> 2) ? 1.0 : 0.0, 0.0}, s.polar, nullptr);
}

}  // namespace qfs
