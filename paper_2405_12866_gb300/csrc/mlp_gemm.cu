// BF16 GEMMs on the fifth-generation tensor cores (tcgen05) for the learned
// warm start:  C[M x N] = A[M x K] * B[N x K]^T  (+ bias[N], optional GELU),
// A and B bf16 row-major (both K-major), accumulation in FP32 in tensor
// memory (TMEM).
//
// k_gemm_bf16_tma: a warp-specialised, persistent pipeline.  Each CTA walks
// its share of the work items (output tiles x K splits).  Warp 0 issues TMA
// tile loads (128-byte swizzle) into a ring of kStages shared stages, each
// tracked by a "full" mbarrier (transaction bytes) and an "empty" mbarrier,
// running ahead into the next item's tiles; warp 1 owns two TMEM accumulators
// (128 x BN fp32 columns each, used in turn) and one of its threads issues the
// tcgen05.mma chain, releasing each stage with tcgen05.commit; warps 2-9 wait
// for an accumulator's commit and run its epilogue (tcgen05.ld, bias, GELU,
// stores in whole 128-byte lines through shared memory) under the next item's
// products.  With split-K each item reduces a K range and adds its tile into
// C32 with vector atomics (the first split adds the bias).
//
// What bounds it: the tensor pipe at the chip's sustained rate (5.4 us a 128 x
// 256 tile at K = 1024 on all SMs, 1.9 PFLOP/s), plus ~5 us of launch, first
// loads and the last epilogue.  With one tile per CTA the set-up and the
// epilogue stood beside the products in each of the two rounds of 8192 x 1024
// x 1024's 256 tiles, and GELU, 3.6 us a tile with a branch around every
// store, was most of the epilogue (now 1.6 us).  Bias, GELU and a bf16 output:
// 8192 rows 27.2 -> 20.1 us, 4096 rows (one round) 14.4 -> 12.7, 16384 rows
// 53.7 -> 34.3; a split-K product 1024 x 1024 x 4096 11.75 -> 11.3.  (GELU with
// its constants folded, 7 instructions, takes 18.4 us for 8192 rows, but rounds
// differently: 2e-4 of the bf16 activations move by a step.)

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdlib>
#include <mutex>

#include "qfs_kernels.h"

namespace qfs {

namespace {

constexpr long long kGemmWaitLimit = 1LL << 24;

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, unsigned parity) {
  for (long long i = 0; i < kGemmWaitLimit; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(su32(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

// The tanh form of GELU, 0.5 x (1 + tanh u) with u = sqrt(2/pi) (x +
// 0.044715 x^3), evaluated as the equal x / (1 + exp(-2u)): ten instructions,
// two of them special functions, ~1e-6 relative, far below the bf16 rounding of
// the result.  The .ftz forms give 0 where a result is subnormal (PTX ISA): 1 + that
// is 1, and a reciprocal below 2^-126 leaves nothing of x (exp(-2u) = inf for u <
// -44 gives -0).
__device__ __forceinline__ float gelu_tanh(float x) {
  const float k0 = 0.7978845608028654f, k1 = 0.044715f;
  const float u = k0 * fmaf(k1 * x, x * x, x);
  float e, r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"((-2.f * u) * 1.4426950408889634f));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(1.f + e));
  return x * r;
}

}  // namespace

// ------------------------------------------------------------ TMA pipeline

namespace {

// Warp 0: TMA producer; warp 1: MMA issuer; warps 2-9: epilogue (two per
// TMEM lane quadrant, each with half of the tile's columns).
constexpr int kBM = 128, kBK = 64, kStages = 4, kTmaThreads = 320, kEpiWarps = 8;
// An epilogue warp's 32 x 32 fp32 staging block: float4 slot c of row r lies at
// slot c ^ (r & 7), so both a column of rows and a row of slots cover all banks.
constexpr int kTileBytes = 32 * 32 * 4;
__device__ __forceinline__ int tile_slot(int r, int c4) { return 32 * r + 4 * (c4 ^ (r & 7)); }

template <int BN>
struct TmaCfg {
  static constexpr int kABytes = kBM * kBK * 2;
  static constexpr int kBBytes = BN * kBK * 2;
  static constexpr int kStageBytes = kABytes + kBBytes;
  // stages, 1024-byte alignment slack, barriers (256 B), the epilogue's blocks
  static constexpr int kSmem = kStages * kStageBytes + 1024 + 256 + kEpiWarps * kTileBytes;
  static constexpr int kTmemCols = 2 * BN;  // two accumulators
  static constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                                     ((uint32_t)(kBM >> 4) << 24);
};

// K-major operand with the 128-byte swizzle: rows of 64 bf16 (128 B), 8-row
// groups 1024 B apart (stride byte offset); the leading byte offset is not
// used by swizzled K-major layouts.
__device__ __forceinline__ uint64_t desc_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void commit_to(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(su32(bar))
               : "memory");
}

// Work item i of a product: its tile's first row and column and its K steps.
// Items of one split are consecutive, tiles of one row block next to each
// other (they share A's rows in L2).
struct GemmItem {
  int m0, n0, z, kb, ke;
};
template <int BN>
__device__ __forceinline__ GemmItem gemm_item(const GemmArgs& g, int i) {
  const unsigned nx = (unsigned)g.N / BN, tiles = nx * ((unsigned)g.M / kBM), KT = (unsigned)g.K / kBK;
  unsigned z = 0, t = (unsigned)i, kb = 0, ke = KT;
  if (g.splitk > 1) {
    z = t / tiles;
    t -= z * tiles;
    kb = z * KT / (unsigned)g.splitk;
    ke = (z + 1) * KT / (unsigned)g.splitk;
  }
  const unsigned y = t / nx;
  return GemmItem{(int)(y * kBM), (int)((t - y * nx) * BN), (int)z, (int)kb, (int)ke};
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint64_t* bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], "
      "[%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(su32(bar)), "r"(x), "r"(y)
      : "memory");
}

}  // namespace

template <int BN>
__global__ void __launch_bounds__(kTmaThreads, 1)
    k_gemm_bf16_tma(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, GemmArgs g) {
  using Cfg = TmaCfg<BN>;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const uint32_t raw = su32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* sb = smem_raw + (base - raw);
  uint64_t* full = reinterpret_cast<uint64_t*>(sb + kStages * Cfg::kStageBytes);
  uint64_t* empty = full + kStages;
  uint64_t* accf = empty + kStages;  // [2] accumulator complete
  uint64_t* acce = accf + 2;         // [2] accumulator read by every epilogue warp
  uint64_t* drain = acce + 2;        // after a give-up: the MMAs issued are done
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int items = (g.N / BN) * (g.M / kBM) * g.splitk;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], kEpiWarps);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapA)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapB)) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)),
                 "r"(Cfg::kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  // Launched as a programmatic dependent of the previous kernel on the
  // stream: the set-up above may overlap its tail; no global memory is read
  // or written before that kernel has completed and its writes are visible.
  asm volatile("griddepcontrol.wait;" ::: "memory");

  if (warp == 0) {
    // Producer: one thread issues the TMA loads of both operands per stage.
    if (lane == 0) {
      int issued = 0;
      for (int w = blockIdx.x; w < items && !*abort_flag; w += gridDim.x) {
        const GemmItem it = gemm_item<BN>(g, w);
        for (int k = it.kb; k < it.ke; ++k, ++issued) {
          const int s = issued % kStages;
          const unsigned ph = (unsigned)(issued / kStages) & 1u;
          if (!mbar_wait_bounded(&empty[s], ph ^ 1u) || *abort_flag) {
            *abort_flag = 1;
            break;
          }
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(&full[s])),
                       "r"(Cfg::kStageBytes)
                       : "memory");
          const uint32_t dst = base + (uint32_t)(s * Cfg::kStageBytes);
          tma_load_2d(dst, &mapA, &full[s], k * kBK, it.m0);
          tma_load_2d(dst + Cfg::kABytes, &mapB, &full[s], k * kBK, it.n0);
        }
      }
      // After a give-up (which may come from another warp once every load is
      // issued), wait (bounded) for the copies that may be in flight: the last
      // one of each stage.
      if (*abort_flag)
        for (int i = issued > kStages ? issued - kStages : 0; i < issued; ++i)
          mbar_wait_bounded(&full[i % kStages], (unsigned)(i / kStages) & 1u);
    }
    __syncwarp();
  } else if (warp == 1) {
    // MMA issuer.
    if (lane == 0) {
      int step = 0, item = 0;
      for (int w = blockIdx.x; w < items && !*abort_flag; w += gridDim.x, ++item) {
        const GemmItem it = gemm_item<BN>(g, w);
        const int buf = item & 1;
        if (!mbar_wait_bounded(&acce[buf], (((unsigned)item >> 1) & 1u) ^ 1u)) {
          *abort_flag = 1;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t acc_t = tmem + (uint32_t)(buf * BN);
        for (int k = it.kb; k < it.ke; ++k, ++step) {
          const int s = step % kStages;
          const unsigned ph = (unsigned)(step / kStages) & 1u;
          if (!mbar_wait_bounded(&full[s], ph) || *abort_flag) {
            *abort_flag = 1;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t a0 = base + (uint32_t)(s * Cfg::kStageBytes), b0 = a0 + Cfg::kABytes;
#pragma unroll
          for (int kk = 0; kk < kBK / 16; ++kk) {
            const uint64_t ad = desc_sw128(a0 + kk * 32), bd = desc_sw128(b0 + kk * 32);
            const uint32_t acc = (k > it.kb || kk > 0) ? 1u : 0u;
            asm volatile(
                "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(acc_t),
                "l"(ad), "l"(bd), "r"(Cfg::kIdesc), "r"(acc)
                : "memory");
          }
          commit_to(&empty[s]);
        }
        // Arrives once every MMA issued above has completed.
        commit_to(&accf[buf]);
      }
      // Every operand load of this CTA is issued: the next kernel on the
      // stream may start its set-up (it waits for this grid to complete
      // before touching memory).
      asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
    __syncwarp();
  } else {
    // Epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31 (rows of the
    // tile) and columns half * BN/2 .. + BN/2 - 1.
    const int q = warp & 3, half = (warp - 2) >> 2;
    float* stile = reinterpret_cast<float*>(sb + kStages * Cfg::kStageBytes + 256 + (warp - 2) * kTileBytes);
    int item = 0;
    for (int w = blockIdx.x; w < items; w += gridDim.x, ++item) {
      const GemmItem it = gemm_item<BN>(g, w);
      const int buf = item & 1;
      const bool add_bias = g.bias != nullptr && it.z == 0;
      // (the bias is fetched under the products)
      constexpr int HC = BN / 2;
      float4 bias[HC / 32];
#pragma unroll
      for (int b = 0; b < HC / 32; ++b)
        bias[b] = add_bias ? __ldg(reinterpret_cast<const float4*>(g.bias + it.n0 + half * HC + 32 * b) + (lane & 7))
                           : make_float4(0.f, 0.f, 0.f, 0.f);
      if (!mbar_wait_bounded(&accf[buf], ((unsigned)item >> 1) & 1u) || *abort_flag) {
        *abort_flag = 1;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
      for (int c64 = 0; c64 < HC; c64 += 64) {
        const int cb = half * HC + c64;
        uint32_t v[64];
        const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * BN + cb);
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          uint32_t* w32 = v + 32 * hh;
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
              "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
              "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
              : "=r"(w32[0]), "=r"(w32[1]), "=r"(w32[2]), "=r"(w32[3]), "=r"(w32[4]), "=r"(w32[5]), "=r"(w32[6]), "=r"(w32[7]),
                "=r"(w32[8]), "=r"(w32[9]), "=r"(w32[10]), "=r"(w32[11]), "=r"(w32[12]), "=r"(w32[13]), "=r"(w32[14]),
                "=r"(w32[15]), "=r"(w32[16]), "=r"(w32[17]), "=r"(w32[18]), "=r"(w32[19]), "=r"(w32[20]), "=r"(w32[21]),
                "=r"(w32[22]), "=r"(w32[23]), "=r"(w32[24]), "=r"(w32[25]), "=r"(w32[26]), "=r"(w32[27]), "=r"(w32[28]),
                "=r"(w32[29]), "=r"(w32[30]), "=r"(w32[31])
              : "r"(taddr + 32u * hh)
              : "memory");
        }
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (c64 + 64 == HC) {
          // The accumulator is read: the next item but one may overwrite it.
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0)
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(&acce[buf])) : "memory");
        }
        // Each 32 x 32 block goes through this warp's staging block: lane l
        // writes its row, then eight lanes cover one row's 128 bytes per
        // store, so every store writes whole lines.
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          const int col = it.n0 + cb + 32 * hh + 4 * (lane & 7);
#pragma unroll
          for (int j4 = 0; j4 < 8; ++j4)
            *reinterpret_cast<float4*>(stile + tile_slot(lane, j4)) =
                make_float4(__uint_as_float(v[32 * hh + 4 * j4]), __uint_as_float(v[32 * hh + 4 * j4 + 1]),
                            __uint_as_float(v[32 * hh + 4 * j4 + 2]), __uint_as_float(v[32 * hh + 4 * j4 + 3]));
          const float4 bv = bias[c64 / 32 + hh];
          __syncwarp();
          // Without a branch between them, so that the 32 values' chains
          // overlap: GELU is half of the epilogue.
          float4 f[8];
#pragma unroll
          for (int i8 = 0; i8 < 8; ++i8) {
            f[i8] = *reinterpret_cast<const float4*>(stile + tile_slot(4 * i8 + (lane >> 3), lane & 7));
            if (add_bias) {
              f[i8].x += bv.x;
              f[i8].y += bv.y;
              f[i8].z += bv.z;
              f[i8].w += bv.w;
            }
          }
          const int row0 = it.m0 + q * 32 + (lane >> 3), left = g.M_valid - row0;
          const size_t at = (size_t)row0 * g.ldc + col, step = 4 * (size_t)g.ldc;
          if (g.splitk > 1) {
#pragma unroll
            for (int i8 = 0; i8 < 8; ++i8)
              if (4 * i8 < left) atomicAdd(reinterpret_cast<float4*>(g.C32 + at + i8 * step), f[i8]);
          } else {
            if (g.C32) {
#pragma unroll
              for (int i8 = 0; i8 < 8; ++i8)
                if (4 * i8 < left) *reinterpret_cast<float4*>(g.C32 + at + i8 * step) = f[i8];
            }
            if (g.C16) {
              if (g.gelu) {
#pragma unroll
                for (int i8 = 0; i8 < 8; ++i8)
                  f[i8] = make_float4(gelu_tanh(f[i8].x), gelu_tanh(f[i8].y), gelu_tanh(f[i8].z), gelu_tanh(f[i8].w));
              }
#pragma unroll
              for (int i8 = 0; i8 < 8; ++i8) {
                const __nv_bfloat162 p0 = __floats2bfloat162_rn(f[i8].x, f[i8].y),
                                     p1 = __floats2bfloat162_rn(f[i8].z, f[i8].w);
                if (4 * i8 < left)
                  *reinterpret_cast<uint2*>(g.C16 + at + i8 * step) =
                      make_uint2(*reinterpret_cast<const uint32_t*>(&p0), *reinterpret_cast<const uint32_t*>(&p1));
              }
            }
          }
          __syncwarp();
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  // (g.err may be mapped host memory: one plain store, no atomic.)
  if (threadIdx.x == 0 && *abort_flag) *reinterpret_cast<volatile int*>(g.err) = 1;
  if (warp == 1) {
    // After a give-up, let the MMAs already issued finish (bounded) before
    // the accumulators are released.
    if (lane == 0 && *abort_flag) {
      commit_to(drain);
      mbar_wait_bounded(drain, 0);
    }
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(Cfg::kTmemCols) : "memory");
  }
}

namespace {

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = []() -> PFN_cuTensorMapEncodeTiled_v12000 {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) !=
            cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }();
  return fn;
}

// Row-major bf16 matrix (rows x K, leading dimension ld) as TMA tiles of
// box_rows x 64 with the 128-byte swizzle.
bool encode_kmajor(CUtensorMap* map, const void* ptr, int rows, int K, int ld, int box_rows) {
  auto fn = tensor_map_encoder();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Encoded maps of recent operands (the training loop reuses the same
// buffers every step; encoding is host work on every launch otherwise).
// Keyed by everything the encoding reads; small, round-robin replacement.
struct MapKey {
  const void* ptr;
  int rows, K, ld, box_rows;
  bool operator==(const MapKey& o) const {
    return ptr == o.ptr && rows == o.rows && K == o.K && ld == o.ld && box_rows == o.box_rows;
  }
};
bool cached_kmajor(CUtensorMap* map, const void* ptr, int rows, int K, int ld, int box_rows) {
  constexpr int kSlots = 64;
  static std::mutex mu;
  static MapKey keys[kSlots];
  static CUtensorMap maps[kSlots];
  static int used = 0, next = 0;
  const MapKey k{ptr, rows, K, ld, box_rows};
  {
    std::lock_guard<std::mutex> lock(mu);
    for (int i = 0; i < used; ++i)
      if (keys[i] == k) {
        *map = maps[i];
        return true;
      }
  }
  if (!encode_kmajor(map, ptr, rows, K, ld, box_rows)) return false;
  std::lock_guard<std::mutex> lock(mu);
  const int slot = used < kSlots ? used++ : (next++ % kSlots);
  keys[slot] = k;
  maps[slot] = *map;
  return true;
}

template <int BN>
cudaError_t launch_tma(const GemmArgs& g, cudaStream_t st) {
  static const cudaError_t attr = cudaFuncSetAttribute(k_gemm_bf16_tma<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       TmaCfg<BN>::kSmem);
  if (attr != cudaSuccess) return attr;
  CUtensorMap ma, mb;
  if (!cached_kmajor(&ma, g.A, g.M, g.K, g.lda, kBM) || !cached_kmajor(&mb, g.B, g.N, g.K, g.ldb, BN))
    return cudaErrorInvalidValue;
  const long long items = (long long)(g.N / BN) * (g.M / kBM) * g.splitk;
  const long long at_once = g.sms > 0 ? g.sms : 1;  // one CTA per SM: the stages fill its shared memory
  // Programmatic dependent launch: this GEMM's set-up may overlap the tail
  // of the previous kernel on the stream (the kernel waits for it before
  // any memory access).
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)std::min(items, at_once));
  cfg.blockDim = dim3(kTmaThreads);
  cfg.dynamicSmemBytes = TmaCfg<BN>::kSmem;
  cfg.stream = st;
  cudaLaunchAttribute pdl[1];
  pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  pdl[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = pdl;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_gemm_bf16_tma<BN>, ma, mb, g);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace

int gemm_splitk_for(const GemmArgs& g) {
  if (g.C16 || g.gelu || !g.C32) return 1;  // (the bias is added by the first split)
  const int BN = g.N % 256 == 0 ? 256 : 128;
  const int tiles = (g.N / BN) * (g.M / kBM);
  const int KT = g.K / kBK;
  int s = 1;
  while (tiles * s * 2 <= g.sms && KT / (s * 2) >= 4) s *= 2;
  return s;
}

cudaError_t launch_gemm_bf16_tc(const GemmArgs& g, cudaStream_t st) {
  if (g.splitk > 1) {
    // The split CTAs add into C32, which starts from zero.
    const cudaError_t e = cudaMemset2DAsync(g.C32, (size_t)g.ldc * 4, 0, (size_t)g.N * 4, g.M_valid, st);
    if (e != cudaSuccess) return e;
  }
  return g.N % 256 == 0 ? launch_tma<256>(g, st) : launch_tma<128>(g, st);
}

}  // namespace qfs
