// Phi_L = U Psi (Section 3 of the paper, the A tensor) to FP64 accuracy on the
// tensor cores: every number is cut into seven signed 8-bit digits, products
// of digits are exact in f16 x f16 -> FP32, and sums of products are exact as
// long as they stay below 2^24 (the error-free splitting of Ozaki, Ogita,
// Oishi and Rump, Numer. Algorithms 59, 2012, for matrix products).
//
// Why: FP64 arithmetic runs at 1/64 of FP32's rate here.  The FP64 kernel was
// at 84% of that pipe's peak (4.28 ms at n = 12, M = 32); the same product in
// digits is 34 f16 products of the same shape, 73 us of tcgen05 at its peak,
// beside 40 us to read U once.
//
// As a real product: U as it lies in memory is N x 2N reals (re, im
// interleaved), and Psi becomes 2N x 2M with columns (pr, -pi), (pi, pr), so
// that columns 2j, 2j + 1 of the result are re and im of column j.
//
// Digits: x = sum_i a_i 2^(-6 - 8i), a_i in [-128, 127] for i > 0, from
// round(x 2^54); Psi's columns are first scaled by a power of two to [1/2, 1).
// D_d = sum over i + j = d of (a_i b_j), d = 0..7, is one TMEM accumulator of
// NB columns, and since the digits of Psi lie side by side along the columns
// of one shared-memory operand, a_i times b_j, b_{j+1}, ... is one MMA that
// adds into D_{i+j}, D_{i+j+1}, ...  The digits of U are formed on the fly by
// the warps that load it.  D_0..D_4 are emptied into 64-bit integers before they
// can pass 2^24, D_4 after every 256 products, and D_5 with it (81920 a product at
// most, so its last additions may round to 2^-52 where every digit is extreme);
// D_6, 2^-48 of D_0, after every 4096.  D_7 may round, and what is left out (d > 7)
// is below 2^-60 of the result's scale.  (With D_4 and D_5 read only at the end the
// sums of constant rows and columns were off in splits of 4096 products and more, by
// up to 1e-11 at n = 13.)
//
// Up to 256 rows there are at most two tiles to fill: unless 256 rows meet many
// columns, k_fx_product forms the product in 64-bit fixed point (fixed.cuh), a
// component by one or two threads (n = 6, M = 16: 50 us as FP64, 6 us so).
//
// U's digits have a fixed scale, so its rows have to have a norm near 1, as a
// unitary's do.  The kernel sums their squares on the way; if any is outside
// [0.81, 1.21], a second pass scales every row by a power of two (n = 12, M = 32,
// such a target: 4.5 ms with the FP64 kernel for it, 0.37 so).  Rows out of
// FP32's range, Inf and NaN take the FP64 kernel, and so does a product whose
// bounded waits ran out.
//
// Scratch: the digits of Psi and the splits' sums, for as many columns at a time as
// fit kOzScratch (n = 12, M = 4096: 1.2 GB in one go).
#include <cuda_fp16.h>

#include "fixed.cuh"
#include "qfs_kernels.h"

#include <algorithm>

namespace qfs {

namespace {

constexpr int kDig = 7;          // digits of a number
constexpr int kOzK = 32;         // reals of one pipeline step
constexpr int kOzChunk = 8;      // steps between two readings of D_3..D_5 (D_0..D_2: fewer)
constexpr int kOzLow = 16;       // chunks between two readings of D_6
constexpr int kOzThreads = 288;  // eight warps for digits and sums, one for the MMAs
constexpr int kOzProd = 256;
constexpr int kABytes = kDig * 128 * kOzK * 2;
constexpr long long kOzWait = 1LL << 24;
constexpr size_t kOzScratch = (size_t)256 << 20;

__host__ __device__ constexpr int oz_bbytes(int nb) { return kDig * nb * kOzK * 2; }
constexpr int oz_smem(int nb) { return 2 * (kABytes + oz_bbytes(nb)) + 128; }

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(uint64_t* b, int n) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(b)), "r"(n) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(b)) : "memory");
}
__device__ __forceinline__ bool bar_wait(uint64_t* b, unsigned parity) {
  for (long long i = 0; i < kOzWait; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(su32(b)), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

// The digits of two numbers 2^-e x, |x| < 2^(e + 1), as seven f16 pairs, most significant first.
// The kernel's producers are bound by these instructions, so: two 32-bit
// funnel shifts instead of a 64-bit shift by a variable, no conversions.
__device__ __forceinline__ void digits2(double x0, double x1, int e, uint32_t (&d)[kDig]) {
  unsigned long long t[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const double x = k ? x1 : x0;
    const int h = __double2hiint(x);
    const uint32_t l = (uint32_t)__double2loint(x), mh = ((uint32_t)h & 0xfffffu) | 0x100000u;
    // |x| 2^(55 - e) = (m << 3) >> (1023 + e - exponent field) for the 53-bit mantissa m.
    const uint32_t m1 = mh << 3 | l >> 29, m0 = l << 3;
    const int sh = min(max(1023 + e - ((h >> 20) & 0x7ff), 0), 63);
    const bool far = sh >= 32;
    const uint32_t a1 = far ? 0u : m1, a0 = far ? m1 : m0;
    const unsigned long long y = (unsigned long long)(a1 >> (sh & 31)) << 32 | __funnelshift_r(a0, a1, sh);
    const unsigned long long v = (y + 1) >> 1;  // rounded to 2^-54
    // Plus 128 in every byte: the bytes are the digits plus 128 (the top one,
    // which may need a ninth bit, is taken from the upper bits).
    t[k] = (h < 0 ? 0 - v : v) + 0x0080808080808080ULL;
  }
  const uint32_t l0 = (uint32_t)t[0], l1 = (uint32_t)t[1], h0 = (uint32_t)(t[0] >> 32), h1 = (uint32_t)(t[1] >> 32);
  // f16 0x6400 | b is 1024 + b; minus 1152 leaves the digit.
  const __half2 off = __half2half2(__ushort_as_half(0x6480));
  auto put = [&](int i, uint32_t w0, uint32_t w1, int byte) {
    const uint32_t p = __byte_perm(w0, w1, byte | (byte + 4) << 4) & 0xffffu;  // bytes: b(w0), b(w1)
    const uint32_t q = __byte_perm(p, 0x64646464u, 0x4140);                    // b0 64 b1 64
    const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&q), off);
    d[i] = *reinterpret_cast<const uint32_t*>(&h);
  };
  const int top0 = ((int)h0 >> 16) - 128, top1 = ((int)h1 >> 16) - 128;
  const __half2 th = __halves2half2(__int2half_rn(top0), __int2half_rn(top1));
  d[0] = *reinterpret_cast<const uint32_t*>(&th);
  put(1, h0, h1, 1);
  put(2, h0, h1, 0);
  put(3, l0, l1, 3);
  put(4, l0, l1, 2);
  put(5, l0, l1, 1);
  put(6, l0, l1, 0);
}

// x rounded toward zero to FP32 (zero below 2^-126), from its bits: an FP64
// conversion occupies the FP64 pipe.
__device__ __forceinline__ float trunc32(double x) {
  const int h = __double2hiint(x), f = ((h >> 20) & 0x7ff) - 896;
  const uint32_t m = ((uint32_t)h & 0xfffffu) << 3 | (uint32_t)__double2loint(x) >> 29;
  return __uint_as_float(f <= 0 ? 0u : (uint32_t)min(f, 255) << 23 | m);  // (Inf or NaN stays one; the sign is not wanted)
}

// The scale of a row in the second pass: 2^e with norm^2 in [2^(2e - 1), 2^(2e + 1)).
__device__ __forceinline__ bool oz_row_ok(float n2) { return n2 > 0x1p-100f && n2 < 0x1p100f; }
__device__ __forceinline__ int oz_row_exp(float n2) { return oz_row_ok(n2) ? ((int)(__float_as_uint(n2) >> 23) - 126) >> 1 : 0; }

// K-major operand without swizzle: 8 rows x 16 bytes are contiguous, `lead`
// bytes lie between neighbours along K, 128 between groups of 8 rows.
__device__ __forceinline__ uint64_t oz_desc(uint32_t saddr, uint32_t lead) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | (uint64_t)(lead >> 4) << 16 | (uint64_t)(128 >> 4) << 32 | (uint64_t)1 << 46;
}

__device__ __forceinline__ void tmem_ld16(uint32_t addr, uint32_t (&w)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7]), "=r"(w[8]),
        "=r"(w[9]), "=r"(w[10]), "=r"(w[11]), "=r"(w[12]), "=r"(w[13]), "=r"(w[14]), "=r"(w[15])
      : "r"(addr)
      : "memory");
}
// Loads done; the registers stand here so that nothing reads them before.
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&w)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(w[0]), "+r"(w[1]), "+r"(w[2]), "+r"(w[3]), "+r"(w[4]), "+r"(w[5]), "+r"(w[6]), "+r"(w[7]),
                 "+r"(w[8]), "+r"(w[9]), "+r"(w[10]), "+r"(w[11]), "+r"(w[12]), "+r"(w[13]), "+r"(w[14]), "+r"(w[15])
               :
               : "memory");
}
// Zeros into 16 columns of this warp's 32 lanes.
__device__ __forceinline__ void tmem_zero16(uint32_t addr) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(addr),
      "r"(0)
      : "memory");
}

}  // namespace

// Digits of M columns of Psi (rows of ld) in the order of the product kernel's
// stages: [column block][step][K group of 8][digit][column][8].  Block j takes
// column j (j >= M: zeros that fill up the last column block) and a chunk of the
// rows (blockIdx.y; all of them look over the whole column for its scale expo[j]).
// With row2 (nullable) they also zero it and the flags.
__global__ void __launch_bounds__(256) k_oz_prep(const double2* __restrict__ Psi, int ld, int N, int M, int NB, __half* dig,
                                                  int* expo, float* row2, int* flags) {
  const int j = blockIdx.x, tid = threadIdx.x;
  if (row2 != nullptr) {
    for (int i = (blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + tid; i < N; i += gridDim.x * gridDim.y * blockDim.x)
      row2[i] = 0.f;
    if (j == 0 && blockIdx.y == 0 && tid < 2) flags[tid] = 0;
  }
  int top = 0;  // exponent field of the column's largest entry
  if (j < M)
    for (int i = tid; i < N; i += 256) {
      const double2 z = Psi[(long long)i * ld + j];
      top = max(top, max((__double2hiint(z.x) >> 20) & 0x7ff, (__double2hiint(z.y) >> 20) & 0x7ff));
    }
  __shared__ int red[8];
  top = __reduce_max_sync(FULL, top);
  if ((tid & 31) == 0) red[tid >> 5] = top;
  __syncthreads();
  for (int w = 0; w < 8; ++w) top = max(top, red[w]);
  const int e = top == 0 ? 0 : top - 1022;  // entries times 2^-e are below 1
  // (Far out, Inf or NaN: 2^20 stands for it, and the FP64 kernel runs.)
  if (tid == 0 && blockIdx.y == 0) expo[j] = top != 0 && (top < 100 || top > 1900) ? 1 << 20 : e;
  auto scaled = [&](double x) {
    const int hi = __double2hiint(x), f = (hi >> 20) & 0x7ff;
    return f == 0 || f - e <= 0 ? 0.0 : __hiloint2double(hi - (e << 20), __double2loint(x));
  };
  const int c0 = 2 * j, cb = c0 / NB, c = c0 % NB, steps = 2 * N / kOzK;
  const int g0 = (int)((long long)blockIdx.y * (N / 4) / gridDim.y), g1 = (int)((long long)(blockIdx.y + 1) * (N / 4) / gridDim.y);
  for (int g = g0 + tid; g < g1; g += 256) {  // a group: 4 complex rows, 8 reals
    double2 z[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      z[r] = j < M ? Psi[(long long)(4 * g + r) * ld + j] : double2{0.0, 0.0};
      z[r] = double2{scaled(z[r].x), scaled(z[r].y)};
    }
    uint32_t a[kDig][4], b[kDig][4];  // columns 2j: (pr, -pi), 2j + 1: (pi, pr)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      uint32_t d[kDig];
      digits2(z[r].x, -z[r].y, 0, d);
#pragma unroll
      for (int i = 0; i < kDig; ++i) a[i][r] = d[i];
      digits2(z[r].y, z[r].x, 0, d);
#pragma unroll
      for (int i = 0; i < kDig; ++i) b[i][r] = d[i];
    }
    const int step = g / (kOzK / 8), k8 = g % (kOzK / 8);
    __half* base = dig + ((long long)cb * steps + step) * (oz_bbytes(NB) / 2) + (long long)k8 * kDig * NB * 8;
#pragma unroll
    for (int i = 0; i < kDig; ++i) {
      *reinterpret_cast<uint4*>(base + (i * NB + c) * 8) = make_uint4(a[i][0], a[i][1], a[i][2], a[i][3]);
      *reinterpret_cast<uint4*>(base + (i * NB + c + 1) * 8) = make_uint4(b[i][0], b[i][1], b[i][2], b[i][3]);
    }
  }
}

// Grid (N / 128 row tiles, K splits, column blocks).  part: [split][column
// block][row][NB] sums in units of 2^-54 of the scaled rows and columns.  row2: the
// sums of the rows' squares, which this launch adds to (norms) or, SCALED, scales by.
template <int NB, bool SCALED>
__global__ void __launch_bounds__(kOzThreads, 1)
    k_oz_product(const double* __restrict__ U, const __half* __restrict__ dig, int N, long long* part, float* row2, int norms,
                 int* flag, int* err) {
  extern __shared__ __align__(128) unsigned char sm[];
  constexpr int kB = oz_bbytes(NB), kStage = kABytes + kB, HC = NB / 2;
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + 2 * kStage);
  uint64_t *empty = full + 2, *accfull = full + 4, *accfree = full + 5;
  uint32_t* slot = reinterpret_cast<uint32_t*>(full + 6);
  volatile int* gave_up = reinterpret_cast<volatile int*>(slot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int steps = 2 * N / kOzK;
  const int k0 = (int)((long long)blockIdx.y * steps / gridDim.y), k1 = (int)((long long)(blockIdx.y + 1) * steps / gridDim.y);
  const int nk = k1 - k0, nchunk = (nk + kOzChunk - 1) / kOzChunk;
  const int row0 = blockIdx.x * 128;

  if (tid == 0) {
    bar_init(&full[0], kOzProd + 1);
    bar_init(&full[1], kOzProd + 1);
    bar_init(&empty[0], 1);
    bar_init(&empty[1], 1);
    bar_init(accfull, 1);
    bar_init(accfree, kOzProd);
    *gave_up = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 8) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(slot)), "r"(8 * NB)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *slot;

  if (warp == 8) {
    // ------------------------------------------------------------- the MMAs
    if (lane == 0) {
      constexpr uint32_t idesc = (1u << 4) | ((uint32_t)(128 >> 4) << 24);
      bool ok = true;
      for (int i = 0; i < nk && ok; ++i) {
        const int s = i & 1;
        if (i % kOzChunk == 0) ok = bar_wait(accfree, (unsigned)(i / kOzChunk) & 1u);
        ok = ok && bar_wait(&full[s], (unsigned)(i >> 1) & 1u) && !*gave_up;
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t a0 = su32(sm + s * kStage), b0 = a0 + kABytes;
        // a_i times digits j .. j + w - 1 of Psi into D_{i+j} ...: at most four
        // digits (256 columns) at a time, D_0..D_3 apart from D_4..D_7.
        auto mma = [&](int kk, int i_, int j, int w) {
          const uint64_t ad = oz_desc(a0 + (uint32_t)(i_ * 128 * kOzK * 2 + kk * 2 * 128 * 16), 128 * 16);
          const uint64_t bd = oz_desc(b0 + (uint32_t)(kk * 2 * kDig * NB * 16 + j * NB * 16), kDig * NB * 16);
          asm volatile(
              "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
              " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem + (uint32_t)((i_ + j) * NB)),
              "l"(ad), "l"(bd), "r"(idesc | (uint32_t)(w * NB >> 3) << 17), "r"(1)
              : "memory");
        };
#pragma unroll
        for (int kk = 0; kk < kOzK / 16; ++kk) {
#pragma unroll
          for (int d = 0; d < kDig; ++d) {
            if (d < 4) mma(kk, d, 0, 4 - d);
            const int j = d < 4 ? 4 - d : 0, last = d == 0 ? 6 : 7 - d;  // i + j from 4 (or i) to 7 (j <= 6)
            mma(kk, d, j, last - j + 1);
          }
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(su32(&empty[s]))
                     : "memory");
        if ((i + 1) % kOzChunk == 0 || i + 1 == nk)
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(su32(accfull))
                       : "memory");
      }
      if (!ok) *gave_up = 1;
    }
    __syncwarp();
  } else {
    // ---------------------------------------------- digits of U, sums of D
    // Lane: row lane & 7 of a group of eight, K group lane >> 3 of four, so
    // that eight lanes store 128 contiguous bytes; two rows per thread.
    const int r = warp * 8 + (lane & 7), k8 = lane >> 3;
    const double* u0 = U + (long long)(row0 + r) * 2 * N + k8 * 8;
    const double* u1 = u0 + 64LL * 2 * N;
    double2 x[2][4];
    float n0 = 0.f, n1 = 0.f;
    const int e0 = SCALED ? oz_row_exp(row2[row0 + r]) : 0, e1 = SCALED ? oz_row_exp(row2[row0 + r + 64]) : 0;
    auto load = [&](int h, int k) {
#pragma unroll
      for (int q = 0; q < 4; ++q) x[h][q] = __ldg(reinterpret_cast<const double2*>((h ? u1 : u0) + (long long)k * kOzK) + q);
    };
    const uint32_t lanes = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * HC);
    long long hi[HC];
#pragma unroll
    for (int c = 0; c < HC; ++c) hi[c] = 0;
    // D_0..D_5 into hi, 16 columns at a time: while one part is added the next is
    // on its way and the last one is zeroed.  Before a sum can pass 2^24: a product
    // adds at most 2^12 to D_0, 2^14 to D_1 (both read after every fourth chunk),
    // 2^15 to D_2 (every second), 49152 to D_3 and 2^16 to D_4 (every one).
    constexpr int P = HC / 16;
    auto at = [&](int q) { return lanes + (uint32_t)(q / P * NB + q % P * 16); };
    auto gather = [&](int chunk, bool clear) {  // clear: another chunk follows
      if (!bar_wait(accfull, (unsigned)chunk & 1u)) return false;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      // (P = 1 takes parts of two sums together: it starts at an even one.)
      const int d0 = !clear || chunk % 4 == 3 ? 0 : P == 1 || chunk % 2 == 1 ? 2 : 3;
      uint32_t wa[16], wb[16];
      tmem_ld16(at(d0 * P), wa);
      auto pair = [&](int q, int weight_a, int weight_b, bool top) {  // parts q and q + 1
        auto add = [&](const uint32_t (&w)[16], int c0, int weight) {
#pragma unroll
          for (int c = 0; c < 16; ++c) {
            const int v = __float2int_rn(__uint_as_float(w[c]));
            if (top) hi[c0 + c] += (long long)(v * weight) << 32;
            else hi[c0 + c] = mad64(v, weight, hi[c0 + c]);
          }
        };
        tmem_wait_ld(wa);
        tmem_ld16(at(q + 1), wb);
        if (clear) tmem_zero16(at(q));
        add(wa, 0, weight_a);
        tmem_wait_ld(wb);
        if (q + 2 < 6 * P) tmem_ld16(at(q + 2), wa);
        if (clear) tmem_zero16(at(q + 1));
        add(wb, P == 2 ? 16 : 0, weight_b);
      };
      // (|D_0| <= 2^22 and |D_1| <= 2^24 weigh 2^40 and 2^32.)
      if (d0 == 0) {
#pragma unroll
        for (int q = 0; q < 2 * P; q += 2) pair(q, 1 << (8 - 8 * (q / P)), 1 << (8 - 8 * ((q + 1) / P)), true);
      }
#pragma unroll 1
      for (int q = max(d0, 2) * P; q < 6 * P; q += 2) pair(q, 1 << (40 - 8 * (q / P)), 1 << (40 - 8 * ((q + 1) / P)), false);
      return true;
    };
    bool ok = true;
    int issued = 0;
    for (int q = 0; q < 8 * P; ++q) tmem_zero16(at(q));
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    bar_arrive(accfree);
    if (nk > 0) {
      load(0, k0);
      load(1, k0);
    }
    for (int i = 0; i < nk; ++i) {
      const int s = i & 1;
      ok = bar_wait(&empty[s], ((unsigned)(i >> 1) & 1u) ^ 1u) && !*gave_up;
      if (!ok) break;
      unsigned char* st = sm + s * kStage;
      if (tid == 0) {
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(&full[s])), "r"(kB) : "memory");
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(su32(st + kABytes)),
            "l"(dig + ((long long)blockIdx.z * steps + k0 + i) * (kB / 2)), "r"(kB), "r"(su32(&full[s]))
            : "memory");
        ++issued;
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t d[4][kDig];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          digits2(x[h][q].x, x[h][q].y, h ? e1 : e0, d[q]);
          if constexpr (!SCALED) {
            const float fx = trunc32(x[h][q].x), fy = trunc32(x[h][q].y);
            (h ? n1 : n0) = fmaf(fx, fx, fmaf(fy, fy, h ? n1 : n0));
          }
        }
#pragma unroll
        for (int p = 0; p < kDig; ++p)
          *reinterpret_cast<uint4*>(st + p * 128 * kOzK * 2 + k8 * 128 * 16 + (r + 64 * h) * 16) =
              make_uint4(d[0][p], d[1][p], d[2][p], d[3][p]);
        // This row's next numbers, at once: 32 KB a CTA stay in flight.
        if (i + 1 < nk) load(h, k0 + i + 1);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      bar_arrive(&full[s]);
      // The previous chunk's sums, with this step's operands already staged.
      if (i > 0 && i % kOzChunk == 0) {
        ok = gather(i / kOzChunk - 1, true);
        if (!ok) break;
        if (i % (kOzChunk * kOzLow) == 0) {
#pragma unroll
          for (int h = 0; h < P; ++h) {
            uint32_t w[16];
            tmem_ld16(at(6 * P + h), w);
            tmem_wait_ld(w);
#pragma unroll
            for (int c = 0; c < 16; ++c) hi[16 * h + c] += (__float2int_rn(__uint_as_float(w[c])) + 128) >> 8;
            tmem_zero16(at(6 * P + h));
          }
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        bar_arrive(accfree);
      }
    }
    if (ok && nk > 0) ok = gather(nchunk - 1, false);
    if (!ok) {
      *gave_up = 1;
      if (tid == 0)  // the copies in flight land first (bounded)
        for (int i = max(0, issued - 2); i < issued; ++i) bar_wait(&full[i & 1], (unsigned)(i >> 1) & 1u);
    } else {
      long long* out = part + (((long long)blockIdx.y * gridDim.z + blockIdx.z) * N + row0 + (warp & 3) * 32 + lane) * NB +
                       (warp >> 2) * HC;
      // hi in 2^-52, D_6 in 2^-60, D_7 in 2^-68; together in 2^-54.
#pragma unroll
      for (int h = 0; h < P; ++h) {
        uint32_t w6[16], w7[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) w6[c] = w7[c] = 0u;
        if (nk > 0) {
          tmem_ld16(at(6 * P + h), w6);
          tmem_ld16(at(7 * P + h), w7);
          tmem_wait_ld(w6);
          tmem_wait_ld(w7);
        }
        auto sum = [&](int c) {
          const long long low = ((long long)__float2int_rn(__uint_as_float(w6[c])) << 8) + __float2int_rn(__uint_as_float(w7[c]));
          return (hi[16 * h + c] << 2) + ((low + (1 << 13)) >> 14);
        };
#pragma unroll
        for (int c = 0; c < 16; c += 2) *reinterpret_cast<longlong2*>(out + 16 * h + c) = longlong2{sum(c), sum(c + 1)};
      }
      if (!SCALED && norms && blockIdx.z == 0) {
        n0 += __shfl_xor_sync(FULL, n0, 8);
        n1 += __shfl_xor_sync(FULL, n1, 8);
        n0 += __shfl_xor_sync(FULL, n0, 16);
        n1 += __shfl_xor_sync(FULL, n1, 16);
        if (lane < 8) {
          atomicAdd(row2 + row0 + r, n0);
          atomicAdd(row2 + row0 + r + 64, n1);
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (tid == 0 && *gave_up) {
    atomicOr(flag, 1);  // (the FP64 kernel forms the product)
    if (err != nullptr) atomicOr(err, 1);
  }
  if (warp == 8) {
    if (lane == 0 && *gave_up) {
      // MMAs already issued finish (bounded) before their accumulator goes.
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(su32(&empty[0]))
                   : "memory");
      for (int i = 0; i < 64; ++i) __nanosleep(1000);
    }
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(8 * NB) : "memory");
  }
}

// The splits' sums (exact), to FP64, into M columns of out (rows of ld).  *flag
// |= 1, and *rows = 1 (nullable), when a row of U or a column was out of scale.
template <bool SCALED>
__global__ void __launch_bounds__(256) k_oz_finish(const long long* __restrict__ part, const int* __restrict__ expo,
                                                    const float* __restrict__ row2, int N, int M, int NB, int splits, int cblocks,
                                                    double2* out, int ld, int* flag, volatile int* rows) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)N * M) return;
  const int row = (int)(i / M), j = (int)(i - (long long)row * M);
  const int cb = 2 * j / NB, c = 2 * j % NB;
  long long re = 0, im = 0;
  for (int s = 0; s < splits; ++s) {
    const longlong2 v =
        __ldcs(reinterpret_cast<const longlong2*>(part + (((long long)s * cblocks + cb) * N + row) * NB + c));
    re += v.x;
    im += v.y;
  }
  const int e = expo[j], er = SCALED ? oz_row_exp(row2[row]) : 0;
  out[(long long)row * ld + j] = double2{scale_exp((double)re, e + er - 54), scale_exp((double)im, e + er - 54)};
  bool bad = e == 1 << 20 && row == 0;
  if (j == 0) {
    const float n2 = row2[row];
    bad |= SCALED ? !oz_row_ok(n2) : !(n2 > 0.81f && n2 < 1.21f);
  }
  if (bad) {
    atomicOr(flag, 1);
    if (rows != nullptr) *rows = 1;
  }
}

// out = U Psi for N <= 256 rows (fixed.cuh: FxDot): grid (N / 8 row tiles (at least 1), column tiles).  Where a row's
// or a column's entries are far from 1, Inf or NaN, its results take FP64 arithmetic.
//
// A warp reads a row of U, so its exponent is one reduction; columns, read along
// rows of Psi, meet in shared memory.  (Without the low x low products 1.3e-15 of
// the norm at n = 6, FP64 arithmetic 3.8e-16; with them 2.2e-16, in the same time.)
//
// At n = 7 and 8 too, in tiles of 8 columns with KS = 2 threads to a component
// (which take every second term each): one launch takes less than the four of the
// digits (a call with M = 24: n = 7 61 -> 33 us, n = 8 53 -> 40, n = 9 by digits 54).
constexpr int kFxRows = 8;
template <int kFxCols, int KS>
__global__ void __launch_bounds__(256) k_fx_product(const double2* __restrict__ U, const double2* __restrict__ Psi,
                                                    double2* __restrict__ out, int n, int M) {
  extern __shared__ int4 su[];  // kFxRows x N, then N x kFxCols
  int4* sp = su + (kFxRows << n);
  __shared__ int tu[kFxRows], tp[kFxCols];  // largest exponent fields
  const int N = 1 << n, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r0 = blockIdx.x * kFxRows, rows = min(kFxRows, N - r0), c0 = blockIdx.y * kFxCols, cols = min(kFxCols, M - c0);
  if (tid < kFxCols) tp[tid] = 0;
  if (warp < rows) {
    int t = 0;
    for (int k = lane; k < N; k += 32) t = max(t, fx_top(U[(long long)(r0 + warp) * N + k]));
    t = __reduce_max_sync(FULL, t);
    if (lane == 0) tu[warp] = t;
  }
  __syncthreads();
  for (int i = tid; i < N * cols; i += 256) atomicMax(&tp[i % cols], fx_top(Psi[(long long)(i / cols) * M + c0 + i % cols]));
  __syncthreads();
  auto eu = [&](int i) { return fx_row_exp(tu[i], n); };
  auto ep = [&](int j) { return fx_col_exp(tp[j], n); };
  for (int i = tid; i < rows * N; i += 256) su[i] = fx_from2(U[(long long)r0 * N + i], eu(i >> n));
  for (int i = tid; i < N * cols; i += 256) sp[i] = fx_from2(Psi[(long long)(i / cols) * M + c0 + i % cols], ep(i % cols));
  __syncthreads();
  for (int e = tid; e < 2 * KS * rows * cols; e += 256) {  // (KS = 2: a multiple of 32, so warps are whole)
    const int c = e / KS, part = e % KS, im = c & 1, i = (c >> 1) / cols, j = (c >> 1) % cols;
    FxDot t;
    t.run<KS>(su + i * N, sp + j, cols, part, N, im);
    long long high = t.t.h, cross = t.cross();
    if constexpr (KS == 2) {
      high += __shfl_xor_sync(FULL, high, 1);
      cross += __shfl_xor_sync(FULL, cross, 1);
      if (part) continue;
    }
    double v = 0.0;
    if (fx_out_of_range(tu[i]) || fx_out_of_range(tp[j])) {
      for (int k = 0; k < N; ++k) {
        const double2 x = U[(long long)(r0 + i) * N + k], y = Psi[(long long)k * M + c0 + j];
        v = im ? fma(x.x, y.y, fma(x.y, y.x, v)) : fma(x.x, y.x, fma(-x.y, y.y, v));
      }
    } else {
      v = fx_dot_value(high, cross, eu(i) + ep(j));
    }
    reinterpret_cast<double*>(out + (long long)(r0 + i) * M + c0 + j)[im] = v;
  }
}

namespace {

struct OzShape {
  int nb, cblocks, splits;  // of a group of columns
  int cols, groups;         // columns of a group (the last one may have fewer)
  size_t dig, part, row2, expo, total;
};
OzShape oz_shape(int N, int M, int num_sms) {
  OzShape s;
  s.nb = 2 * M <= 32 ? 32 : 64;
  const int all = (2 * M + s.nb - 1) / s.nb, steps = 2 * N / kOzK;
  auto up = [](size_t b) { return (b + 255) / 256 * 256; };
  auto shape = [&](int cblocks) {
    s.cblocks = cblocks;
    s.splits = std::max(1, std::min(steps / 2, num_sms / (N / 128 * cblocks)));
    s.dig = up((size_t)cblocks * steps * oz_bbytes(s.nb));
    s.part = up((size_t)s.splits * cblocks * N * s.nb * sizeof(long long));
    s.row2 = up((size_t)N * sizeof(float));
    s.expo = up((size_t)cblocks * s.nb / 2 * sizeof(int) + 2 * sizeof(int));
    s.total = s.dig + s.part + s.row2 + s.expo;
  };
  for (s.groups = 1;; ++s.groups) {
    shape((all + s.groups - 1) / s.groups);
    if (s.total <= kOzScratch || s.cblocks == 1) break;
  }
  s.cols = s.cblocks * s.nb / 2;
  s.groups = (M + s.cols - 1) / s.cols;
  return s;
}

// One pass over all columns: digits of Psi, product, sums.
template <bool SCALED>
cudaError_t oz_pass(const OzShape& s, const double2* U, const double2* Psi, double2* out, int N, int M, void* scratch, int* err,
                    int* rows, cudaStream_t st) {
  char* p = static_cast<char*>(scratch);
  __half* dig = reinterpret_cast<__half*>(p);
  long long* part = reinterpret_cast<long long*>(p + s.dig);
  float* row2 = reinterpret_cast<float*>(p + s.dig + s.part);
  int* flags = reinterpret_cast<int*>(p + s.dig + s.part + s.row2);
  int *flag = flags + SCALED, *expo = flags + 2;
  const auto product = s.nb == 64 ? k_oz_product<64, SCALED> : k_oz_product<32, SCALED>;
  cudaError_t e = allow_smem(product, oz_smem(s.nb));
  for (int c = 0; c < M && e == cudaSuccess; c += s.cols) {
    const int m = std::min(s.cols, M - c), cblocks = (2 * m + s.nb - 1) / s.nb;
    const bool first = !SCALED && c == 0;
    e = launch_kernel(k_oz_prep, dim3(cblocks * s.nb / 2, std::max(1, std::min(16, N / 512))), 256, 0, st, Psi + c, M, N, m, s.nb,
                      dig, expo, first ? row2 : nullptr, flags);
    if (e == cudaSuccess)
      e = launch_kernel(product, dim3(N / 128, s.splits, cblocks), kOzThreads, oz_smem(s.nb), st, (const double*)U, dig, N, part,
                        row2, (int)first, flag, err);
    if (e == cudaSuccess)
      e = launch_kernel(k_oz_finish<SCALED>, (unsigned)(((long long)N * m + 255) / 256), 256, 0, st, part, expo, row2, N, m, s.nb,
                        s.splits, cblocks, out + c, M, flag, rows);
  }
  return e;
}

}  // namespace

// From 512 rows on, and at 256 for more than 96 columns, where fixed point grows
// with M (a call at M = 64: 48 us, 96: 56, 128: 67, 256: 93) and digits take 50 us.
size_t oz_scratch_bytes(int N, int M, int num_sms) {
  return N < 256 || (N == 256 && M <= 96) ? 0 : oz_shape(N, M, num_sms).total;
}
int oz_launches(int N, int M, int num_sms) { return 3 * oz_shape(N, M, num_sms).groups; }

const int* oz_flag(const void* scratch, int N, int M, int num_sms) {
  const OzShape s = oz_shape(N, M, num_sms);
  return reinterpret_cast<const int*>(static_cast<const char*>(scratch) + s.dig + s.part + s.row2);
}

cudaError_t launch_oz_product(const double2* U, const double2* Psi, double2* out, int N, int M, void* scratch, int* err, int* rows,
                              int num_sms, cudaStream_t st) {
  const cudaError_t e = oz_pass<false>(oz_shape(N, M, num_sms), U, Psi, out, N, M, scratch, err, rows, st);
  return e != cudaSuccess || rows != nullptr ? e : launch_gemm_upsi(U, Psi, out, N, M, st, oz_flag(scratch, N, M, num_sms));
}
cudaError_t launch_oz_scaled(const double2* U, const double2* Psi, double2* out, int N, int M, void* scratch, int* err, int num_sms,
                             cudaStream_t st) {
  const cudaError_t e = oz_pass<true>(oz_shape(N, M, num_sms), U, Psi, out, N, M, scratch, err, nullptr, st);
  return e != cudaSuccess ? e : launch_gemm_upsi(U, Psi, out, N, M, st, oz_flag(scratch, N, M, num_sms) + 1);
}

cudaError_t launch_fx_product(const double2* U, const double2* Psi, double2* out, int n, int M, cudaStream_t st) {
  const int cols = n <= 6 ? 32 : 8;
  const size_t smem = sizeof(int4) * (size_t)(kFxRows + cols) << n;  // (n = 8: 64 KB)
  const dim3 grid((unsigned)std::max(1, (1 << n) / kFxRows), (M + cols - 1) / cols);
  if (n <= 6) return launch_kernel(k_fx_product<32, 1>, grid, 256, smem, st, U, Psi, out, n, M);
  const cudaError_t e = allow_smem(k_fx_product<8, 2>, sizeof(int4) * (size_t)(kFxRows + 8) << kFxProductQubits);
  return e != cudaSuccess ? e : launch_kernel(k_fx_product<8, 2>, grid, 256, smem, st, U, Psi, out, n, M);
}

}  // namespace qfs
