// Elementwise and reduction kernels of the learned warm start (the network
// proposes initial gates; the sweep judges them).  The matrix products run
// on the tensor cores (mlp_gemm.cu); these kernels build the features, cast
// and transpose operands, form the loss gradient, back-propagate GELU, sum
// bias gradients and apply Adam.
#include <cuda_bf16.h>

#include "qfs_common.cuh"
#include "qfs_kernels.h"

#include <algorithm>

namespace qfs {

namespace {
// Derivative of the tanh form of GELU, 0.5 x (1 + tanh u) with u =
// k0 (x + k1 x^3): with s = 1 / (1 + exp(-2u)) = (1 + tanh u) / 2 it is
// s + 2 x s (1 - s) k0 (1 + 3 k1 x^2) (1 - tanh^2 u = 4 s (1 - s), free of
// the cancellation of 1 - t^2); ~1e-6 relative.  exp(-2u) = inf gives s = 0.
__device__ __forceinline__ float gelu_grad_f(float x) {
  const float k0 = 0.7978845608028654f, k1 = 0.044715f;
  const float u = k0 * fmaf(k1 * x, x * x, x);
  const float s = __fdividef(1.f, 1.f + __expf(-2.f * u));
  return fmaf(2.f * x * s * (1.f - s), k0 * fmaf(3.f * k1, x * x, 1.f), s);
}
}  // namespace

// A double as the unevaluated sum of two floats, hi its truncation to 24 bits,
// by integer operations and one integer conversion: FP64 conversions run at
// 1/64 of FP32's rate.  ok is cleared where the split or a product of two such
// pairs could leave FP32's normal range (0 itself is fine).
__device__ __forceinline__ float2 split_f32(double x, bool& ok) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const unsigned up = (unsigned)(u >> 32), ex = (up >> 20) & 0x7FFu;
  if ((u << 1) == 0) return float2{__uint_as_float(up & 0x80000000u), 0.f};
  ok &= ex - (1023u - 40u) <= 60u;  // 2^-40 <= |x| < 2^21
  const unsigned sign = up & 0x80000000u, e32 = ex - 896u;
  const float hi = __uint_as_float(sign | (e32 << 23) | ((unsigned)(u >> 29) & 0x7FFFFFu));
  // The low 29 bits, in units of 2^-52 of x's binade.
  const float lo = __fmul_rn((float)((unsigned)u & 0x1FFFFFFFu), __uint_as_float(sign | ((e32 - 52u) << 23)));
  return float2{hi, lo};
}

// a b as p + e, e exact to 2^-24 of itself (2^-47 of the product).
__device__ __forceinline__ float2 mul_pair(float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  return float2{p, __fmaf_rn(a.x, b.y, __fmaf_rn(a.y, b.x, __fmaf_rn(a.x, b.x, -p)))};
}
// d + e rounded to a float; sure is cleared where a number within 2^-43 size of
// d + e rounds to another one.  The pairs are good to that at worst and FP64
// arithmetic to 2^-52, so where sure stands both round to the same float.
__device__ __forceinline__ float round_pair(float d, float e, float size, bool& sure) {
  constexpr float kSlack = 1.f / (1LL << 43);
  const float r = __fadd_rn(d, __fmaf_rn(size, kSlack, e));
  sure &= r == __fadd_rn(d, __fmaf_rn(size, -kSlack, e));
  return r;
}
// The float next to s - t.
__device__ __forceinline__ float sub_pair(float2 s, float2 t, bool& sure) {
  const float d = __fsub_rn(s.x, t.x), v = __fsub_rn(d, s.x);
  const float err = __fsub_rn(__fsub_rn(s.x, __fsub_rn(d, v)), __fadd_rn(t.x, v));
  return round_pair(d, __fadd_rn(err, __fsub_rn(s.y, t.y)), __fadd_rn(fabsf(s.x), fabsf(t.x)), sure);
}
// A float of normal size (or 0) as a double, by integer operations.
__device__ __forceinline__ double widen(float x) {
  const unsigned u = __float_as_uint(x);
  return x == 0.f ? 0.0 : __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7FFFFFFFu) >> 3) + (896u << 20))), (int)(u << 29));
}

// Features of target t: the 16 x 8 complex matrix U_t Phi_fix as 256 reals
// (row-major, re/im interleaved), bf16, row t of X (ld = 256).  Rows
// count..rows-1 are zero.  Every product of two complex entries is rounded to
// FP32 and the 16 of an output are added in FP32.
//
// The products in FP64 were bound by that pipe (95 us for 4096 targets; the
// targets are 17 MB, 2.5 us of memory time), so they are formed from pairs of
// floats, which give the same rounded float except next to the middle between
// two: an output with such a product (one in ~2000) takes FP64 products, and so does
// a target with an entry outside the pairs' range.  A block walks over targets: its
// 128 threads, one per output, keep their column of Phi_fix in registers and share
// the split target.  24 us (without the check 22).
constexpr int kFeatStride = 17;  // float4s a row: four rows' reads lie in different banks
__global__ void __launch_bounds__(128) k_ws_features(const double2* __restrict__ U, const double2* __restrict__ phif,
                                                     int count, int rows, __nv_bfloat16* __restrict__ X) {
  __shared__ float4 su[16 * kFeatStride];
  const int k = threadIdx.x, i = k / 8, j = k % 8;
  float2 bx[16], by[16];
  bool phi_ok = true;
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    const double2 b = phif[q * 8 + j];
    bx[q] = split_f32(b.x, phi_ok);
    by[q] = split_f32(b.y, phi_ok);
  }
  double2 next[2];
  auto fetch = [&](int t) {
#pragma unroll
    for (int h = 0; h < 2; ++h) next[h] = t < count ? __ldg(U + (size_t)t * 256 + k + 128 * h) : double2{0.0, 0.0};
  };
  fetch(blockIdx.x);
  for (int t = blockIdx.x; t < rows; t += gridDim.x) {
    float re = 0.f, im = 0.f;
    if (t < count) {
      bool ok = phi_ok;
      float4 mine[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float2 ax = split_f32(next[h].x, ok), ay = split_f32(next[h].y, ok);
        mine[h] = make_float4(ax.x, ax.y, ay.x, ay.y);
      }
      __syncthreads();  // the last target's entries are read
#pragma unroll
      for (int h = 0; h < 2; ++h) su[((k + 128 * h) / 16) * kFeatStride + (k & 15)] = mine[h];
      const bool pairs = __syncthreads_and(ok);
      fetch(t + gridDim.x);  // (under this target's products)
      if (pairs) {
        bool sure = true;
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          const float4 a = su[i * kFeatStride + q];
          const float2 ax{a.x, a.y}, ay{a.z, a.w}, nby{-by[q].x, -by[q].y};
          re = __fadd_rn(re, sub_pair(mul_pair(ax, bx[q]), mul_pair(ay, by[q]), sure));
          im = __fadd_rn(im, sub_pair(mul_pair(ay, bx[q]), mul_pair(ax, nby), sure));
        }
        // Outputs (about one in 2000) with an unsure product, a warp at a time: a
        // lane forms one component of one product in FP64.
        for (unsigned todo = __ballot_sync(FULL, !sure); todo; todo &= todo - 1) {
          const int lane = k & 31, src = __ffs(todo) - 1, o = (k & ~31) | src, q = lane >> 1;
          const double2 x = U[(size_t)t * 256 + o / 8 * 16 + q], y = phif[q * 8 + o % 8];
          const float v = (float)(lane & 1 ? x.x * y.y + x.y * y.x : x.x * y.x - x.y * y.y);
          float sx = 0.f, sy = 0.f;
#pragma unroll
          for (int p = 0; p < 16; ++p) {
            sx = __fadd_rn(sx, __shfl_sync(FULL, v, 2 * p));
            sy = __fadd_rn(sy, __shfl_sync(FULL, v, 2 * p + 1));
          }
          if (lane == src) {
            re = sx;
            im = sy;
          }
        }
      } else {
        const double2* u = U + (size_t)t * 256 + i * 16;
        for (int q = 0; q < 16; ++q) {
          const double2 a = u[q], b = phif[q * 8 + j];
          re += (float)(a.x * b.x - a.y * b.y);
          im += (float)(a.x * b.y + a.y * b.x);
        }
      }
    }
    // Scaled by sqrt(16) = 4 so that the features have unit variance per
    // complex entry (the columns of U Phi_fix are unit vectors of length 16).
    *reinterpret_cast<__nv_bfloat162*>(X + (size_t)t * 256 + 2 * k) = __floats2bfloat162_rn(4.f * re, 4.f * im);
  }
}

// dst[c][r] = src[r][c] (bf16), 32 x 32 tiles; R, C multiples of 32.
// dst (C x R) = src (R x C)^T, both bf16 row-major, R and C multiples of 64:
// 64 x 64 tiles, two elements per access (128-byte rows per warp on both
// sides); the shared tile's rows are padded by one word.
__global__ void k_transpose_bf16_64(const __nv_bfloat16* __restrict__ src, int R, int C,
                                    __nv_bfloat16* __restrict__ dst) {
  __shared__ __nv_bfloat16 tile[64][66];
  const int c0 = blockIdx.x * 64, r0 = blockIdx.y * 64;
  const int tx = threadIdx.x, ty = threadIdx.y;
  for (int y = ty; y < 64; y += 8) {
    const __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162*>(src + (size_t)(r0 + y) * C + c0 + 2 * tx);
    tile[y][2 * tx] = v.x;
    tile[y][2 * tx + 1] = v.y;
  }
  __syncthreads();
  for (int y = ty; y < 64; y += 8) {
    __nv_bfloat162 v;
    v.x = tile[2 * tx][y];
    v.y = tile[2 * tx + 1][y];
    *reinterpret_cast<__nv_bfloat162*>(dst + (size_t)(c0 + y) * R + r0 + 2 * tx) = v;
  }
}

__global__ void k_transpose_bf16(const __nv_bfloat16* __restrict__ src, int R, int C,
                                 __nv_bfloat16* __restrict__ dst) {
  __shared__ __nv_bfloat16 tile[32][33];
  const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  for (int y = threadIdx.y; y < 32; y += 8) tile[y][threadIdx.x] = src[(size_t)(r0 + y) * C + c0 + threadIdx.x];
  __syncthreads();
  for (int y = threadIdx.y; y < 32; y += 8) dst[(size_t)(c0 + y) * R + r0 + threadIdx.x] = tile[threadIdx.x][y];
}

__global__ void k_cast_f32_bf16(const float* __restrict__ a, __nv_bfloat16* __restrict__ b, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    b[i] = __float2bfloat16(a[i]);
}

__global__ void k_cast_f64_f32(const double* __restrict__ a, float* __restrict__ b, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    b[i] = (float)a[i];
}

// A 64 x 64 tile of a layer's output gradient G (256 threads; thread (tx, ty)
// holds columns 4 tx .. + 3 of rows ty, ty + 16, ...): what the two products of
// the layer's backward pass and its bias gradient need of it, while it is in
// registers.  bf16 rows to G16 (rows x cols), the transposed tile to GT16 (cols
// x rows) through shared memory, the column sums to db (zero before) by one
// atomic per column and tile.
//
// As four kernels (gradient in FP32 and bf16, column sums, transpose, each
// reading what the last one wrote) a hidden layer of 4096 x 1024 took 19.0 us
// and the output layer 35; memory traffic 84 MB, here 50 (L2 holds most of
// it).  Now 8.2 and 17 us, each with its column sums' memset (1.7 us).
struct GradTile {
  __nv_bfloat162 t[64][33];  // row stride 33 words: 2-way conflicts at most in the transposed reads
  float sum[16][64];
};
__device__ __forceinline__ void grad_tile_row(GradTile& s, int r, int tx, float4 g, float4& acc,
                                              __nv_bfloat16* __restrict__ row16) {
  const __nv_bfloat162 a = __floats2bfloat162_rn(g.x, g.y), b = __floats2bfloat162_rn(g.z, g.w);
  *reinterpret_cast<uint2*>(row16 + 4 * tx) =
      make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
  s.t[r][2 * tx] = a;
  s.t[r][2 * tx + 1] = b;
  acc.x += g.x;
  acc.y += g.y;
  acc.z += g.z;
  acc.w += g.w;
}
__device__ __forceinline__ void grad_tile_end(GradTile& s, int tid, float4 acc, int r0, int c0, int rows,
                                              __nv_bfloat16* __restrict__ GT16, float* __restrict__ db) {
  *reinterpret_cast<float4*>(&s.sum[tid >> 4][4 * (tid & 15)]) = acc;
  __syncthreads();
  if (tid < 64) {
    float t = 0.f;
#pragma unroll
    for (int y = 0; y < 16; ++y) t += s.sum[y][tid];
    atomicAdd(db + c0 + tid, t);
  }
  const __nv_bfloat16* tile = reinterpret_cast<const __nv_bfloat16*>(s.t);
  const int lane = tid & 31;
#pragma unroll
  for (int c = tid >> 5; c < 64; c += 8) {
    __nv_bfloat162 v;
    v.x = tile[(2 * lane) * 66 + c];
    v.y = tile[(2 * lane + 1) * 66 + c];
    *reinterpret_cast<__nv_bfloat162*>(GT16 + (size_t)(c0 + c) * rows + r0 + 2 * lane) = v;
  }
}

// Output gradient of the mean squared error over the first n_out columns of
// the first B_valid rows: G = 2 (Y - T) / (B_valid n_out), zero elsewhere;
// loss partial sums per block into loss_part[block] (at most 1024).  Block
// column x walks the row tiles y, y + gridDim.y, ...
//
// Y - T is a pair of floats (exactly) and so is its scaled value, which gives the
// same rounded float as FP64 except next to the middle between two, and there it
// takes FP64; the sum of squares is FP64's, of differences widened by integer
// operations.  (Squares as pairs, 16 to a sum: 1.6e-15 of the loss away from the
// exact one; so 2e-16.)  FP64 conversions and products for everything were 24 us of
// that pipe.  Differences outside the pairs' range take FP64.
__global__ void __launch_bounds__(256)
    k_ws_loss_grad(const float* __restrict__ Y, int ldy, const float* __restrict__ T, int n_out, int rows, int B_valid,
                   double scale, __nv_bfloat16* __restrict__ G16, __nv_bfloat16* __restrict__ GT16, float* __restrict__ db,
                   double* __restrict__ loss_part) {
  __shared__ GradTile s;
  __shared__ double red[8];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, c0 = blockIdx.x * 64;
  const float sh = (float)scale, sl = (float)(scale - (double)sh);
  double acc[2] = {0.0, 0.0};
  for (int r0 = 64 * blockIdx.y; r0 < rows; r0 += 64 * gridDim.y) {
    float4 col = make_float4(0.f, 0.f, 0.f, 0.f);
    const int c = c0 + 4 * tx;
    float4 ly[4], lt[4];
#pragma unroll
    for (int y = 0; y < 4; ++y) {
      const int r = r0 + ty + 16 * y;
      const bool in = r < B_valid && c < n_out;
      ly[y] = in ? *reinterpret_cast<const float4*>(Y + (size_t)r * ldy + c) : make_float4(0.f, 0.f, 0.f, 0.f);
      lt[y] = in ? *reinterpret_cast<const float4*>(T + (size_t)r * n_out + c) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int y = 0; y < 4; ++y) {
      const int r = r0 + ty + 16 * y;
      const float4 v = ly[y], w = lt[y];
      const float vy[4] = {v.x, v.y, v.z, v.w}, vt[4] = {w.x, w.y, w.z, w.w};
      float g[4];  // (0 where the loads gave 0)
      double dd[4];
      bool sure = true;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        // d + de = Y - T exactly.
        const float d = __fsub_rn(vy[e], vt[e]), b = __fsub_rn(d, vy[e]);
        const float de = __fsub_rn(__fsub_rn(vy[e], __fsub_rn(d, b)), __fadd_rn(vt[e], b));
        const float m = fabsf(d), p = __fmul_rn(d, sh);
        sure &= d == 0.f || (m >= 1e-18f && m <= 1e18f);
        g[e] = round_pair(p, __fmaf_rn(de, sh, __fmaf_rn(d, sl, __fmaf_rn(d, sh, -p))), fabsf(p), sure);
        dd[e] = widen(d) + widen(de);
      }
      if (!sure) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          dd[e] = (double)vy[e] - (double)vt[e];
          g[e] = (float)(scale * dd[e]);
        }
      }
      if (c < n_out) {  // (n_out is a multiple of 64: whole blocks)
        acc[0] = fma(dd[0], dd[0], acc[0]);
        acc[1] = fma(dd[1], dd[1], acc[1]);
        acc[0] = fma(dd[2], dd[2], acc[0]);
        acc[1] = fma(dd[3], dd[3], acc[1]);
      }
      grad_tile_row(s, ty + 16 * y, tx, make_float4(g[0], g[1], g[2], g[3]), col, G16 + (size_t)r * ldy + c0);
    }
    grad_tile_end(s, tid, col, r0, c0, rows, GT16, db);
    __syncthreads();
  }
  double sum = acc[0] + acc[1];
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) sum += __shfl_xor_sync(~0u, sum, m);
  if ((tid & 31) == 0) red[tid >> 5] = sum;
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < 8; ++w) sum += red[w];
    loss_part[blockIdx.y * gridDim.x + blockIdx.x] = sum;
  }
}

// G = dH * gelu'(Z) of a hidden layer, rows >= B_valid zero.
__global__ void __launch_bounds__(256)
    k_gelu_back(const float* __restrict__ dH, const float* __restrict__ Z, int rows, int cols, int B_valid,
                __nv_bfloat16* __restrict__ G16, __nv_bfloat16* __restrict__ GT16, float* __restrict__ db) {
  __shared__ GradTile s;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, c0 = blockIdx.x * 64, r0 = blockIdx.y * 64;
  float4 col = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int y = 0; y < 4; ++y) {
    const int r = r0 + ty + 16 * y;
    const size_t at = (size_t)r * cols + c0 + 4 * tx;
    float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < B_valid) {
      const float4 h = *reinterpret_cast<const float4*>(dH + at), z = *reinterpret_cast<const float4*>(Z + at);
      g = make_float4(h.x * gelu_grad_f(z.x), h.y * gelu_grad_f(z.y), h.z * gelu_grad_f(z.z), h.w * gelu_grad_f(z.w));
    }
    grad_tile_row(s, ty + 16 * y, tx, g, col, G16 + (size_t)r * cols + c0);
  }
  grad_tile_end(s, tid, col, r0, c0, rows, GT16, db);
}

// acc += (sum of parts[0..n)) * scale (one block).
__global__ void k_loss_accumulate(const double* __restrict__ parts, int n, double scale, double* __restrict__ acc) {
  __shared__ double red[256];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s += parts[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int h = blockDim.x / 2; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) *acc += red[0] * scale;
}

// Adam (Kingma & Ba 2015) on fp32 master parameters with a bf16 copy.
// With `sched` (device, 3 floats per step: lr, bc1, bc2) the step's values
// are read at index *sched_step, so that one captured graph serves every
// step; otherwise the arguments are used.
__global__ void k_adam(float* __restrict__ w, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ g, long long n, float lr, float b1, float b2, float eps,
                       float bc1, float bc2, __nv_bfloat16* __restrict__ w16, const float* __restrict__ sched,
                       const int* __restrict__ sched_step) {
  if (sched) {
    const int s = *sched_step;
    lr = sched[3 * s];
    bc1 = sched[3 * s + 1];
    bc2 = sched[3 * s + 2];
  }
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
    w[i] = wi;
    if (w16) w16[i] = __float2bfloat16(wi);
  }
}

// Network outputs -> 6 gates per row (G[r][c] from outputs 2(16g + 4r + c),
// +1) -> E = G^dagger, so that the polar update (which returns the polar
// factor of E^dagger) projects G onto U(4).
__global__ void k_ws_gates_adjoint(const float* __restrict__ Y, int ldy, int count, double2* __restrict__ E) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= (long long)count * 96) return;
  const int t = (int)(e / 96), q = (int)(e % 96), g = q / 16, x = (q % 16) / 4, y = q % 4;
  const float* row = Y + (size_t)t * ldy + 32 * g;
  // E[x][y] = conj(G[y][x])
  E[e] = double2{(double)row[2 * (4 * y + x)], -(double)row[2 * (4 * y + x) + 1]};
}

// Mini-batch gather: rows idx[0..bv) of the device training set into the
// batch buffers; rows bv..B-1 of X are zeroed.
// Rows idx[0 .. bv) of the training set, after advancing idx by
// *jstep * batch when jstep is given (the step within the epoch, read on the
// device so that one captured graph serves every step).
__global__ void k_ws_gather(const __nv_bfloat16* __restrict__ Xall, const float* __restrict__ Tall,
                            const int* __restrict__ idx, int bv, int B, __nv_bfloat16* __restrict__ X,
                            float* __restrict__ T, const int* __restrict__ jstep, int batch) {
  if (jstep) idx += (long long)*jstep * batch;
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e < (long long)B * 256) {
    const int r = (int)(e / 256), c = (int)(e % 256);
    X[e] = r < bv ? Xall[(size_t)idx[r] * 256 + c] : __float2bfloat16(0.f);
  }
  if (e < (long long)bv * 192) {
    const int r = (int)(e / 192), c = (int)(e % 192);
    T[e] = Tall[(size_t)idx[r] * 192 + c];
  }
}

// The end of a training step: the step within the epoch and the step of
// the call advance.
__global__ void k_ws_step_advance(int* jstep, int* gstep) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    *jstep += 1;
    *gstep += 1;
  }
}

static int blocks_for(long long n, int threads = 256, int cap = 4096) {
  long long b = (n + threads - 1) / threads;
  return (int)(b > cap ? cap : (b < 1 ? 1 : b));
}

void launch_ws_features(const double2* U, const double2* phif, int count, int rows, __nv_bfloat16* X,
                        cudaStream_t st) {
  // (two blocks an SM by their registers; each splits Phi_fix once)
  k_ws_features<<<std::min(rows, 304), 128, 0, st>>>(U, phif, count, rows, X);
}
void launch_ws_gates_adjoint(const float* Y, int ldy, int count, double2* E, cudaStream_t st) {
  const long long n = (long long)count * 96;
  k_ws_gates_adjoint<<<(int)((n + 255) / 256), 256, 0, st>>>(Y, ldy, count, E);
}
void launch_ws_gather(const __nv_bfloat16* Xall, const float* Tall, const int* idx, int bv, int B,
                      __nv_bfloat16* X, float* T, cudaStream_t st, const int* jstep, int batch) {
  const long long n = (long long)B * 256;
  k_ws_gather<<<(int)((n + 255) / 256), 256, 0, st>>>(Xall, Tall, idx, bv, B, X, T, jstep, batch);
}
void launch_ws_step_advance(int* jstep, int* gstep, cudaStream_t st) { k_ws_step_advance<<<1, 32, 0, st>>>(jstep, gstep); }
void launch_transpose_bf16(const __nv_bfloat16* src, int R, int C, __nv_bfloat16* dst, cudaStream_t st) {
  if (R % 64 == 0 && C % 64 == 0)
    k_transpose_bf16_64<<<dim3(C / 64, R / 64), dim3(32, 8), 0, st>>>(src, R, C, dst);
  else
    k_transpose_bf16<<<dim3(C / 32, R / 32), dim3(32, 8), 0, st>>>(src, R, C, dst);
}
void launch_cast_f32_bf16(const float* a, __nv_bfloat16* b, long long n, cudaStream_t st) {
  k_cast_f32_bf16<<<blocks_for(n), 256, 0, st>>>(a, b, n);
}
void launch_cast_f64_f32(const double* a, float* b, long long n, cudaStream_t st) {
  k_cast_f64_f32<<<blocks_for(n), 256, 0, st>>>(a, b, n);
}
int launch_ws_loss_grad(const float* Y, int ldy, const float* T, int n_out, int rows, int B_valid, __nv_bfloat16* G16,
                        __nv_bfloat16* GT16, float* db, double* loss_part, cudaStream_t st) {
  const dim3 grid(ldy / 64, std::min(rows / 64, 1024 / (ldy / 64)));
  cudaMemsetAsync(db, 0, sizeof(float) * (size_t)ldy, st);
  k_ws_loss_grad<<<grid, 256, 0, st>>>(Y, ldy, T, n_out, rows, B_valid, 2.0 / ((double)B_valid * n_out), G16, GT16, db,
                                       loss_part);
  return (int)(grid.x * grid.y);
}
void launch_gelu_back(const float* dH, const float* Z, int rows, int cols, int B_valid, __nv_bfloat16* G16,
                      __nv_bfloat16* GT16, float* db, cudaStream_t st) {
  cudaMemsetAsync(db, 0, sizeof(float) * (size_t)cols, st);
  k_gelu_back<<<dim3(cols / 64, rows / 64), 256, 0, st>>>(dH, Z, rows, cols, B_valid, G16, GT16, db);
}
void launch_loss_accumulate(const double* parts, int n, double scale, double* acc, cudaStream_t st) {
  k_loss_accumulate<<<1, 256, 0, st>>>(parts, n, scale, acc);
}
void launch_adam(float* w, float* m, float* v, const float* g, long long n, float lr, float b1, float b2, float eps,
                 float bc1, float bc2, __nv_bfloat16* w16, cudaStream_t st, const float* sched,
                 const int* sched_step) {
  k_adam<<<blocks_for(n), 256, 0, st>>>(w, m, v, g, n, lr, b1, b2, eps, bc1, bc2, w16, sched, sched_step);
}

}  // namespace qfs
