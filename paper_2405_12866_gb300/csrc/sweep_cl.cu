// Sweeps (Section 3 of the paper) of starts whose state fits on chip: one
// thread-block cluster per start, no work queue and no global hand-over
// between gate steps.
//
// A gate acts on rows, one sample column at a time, so the C CTAs of a cluster
// take M / C columns each and need nothing from one another but the sum of
// their 4x4 environments: 32 numbers per gate step, sent to every CTA of the
// cluster through distributed shared memory.  Every CTA then runs the gate
// update itself (the same instructions on the same sums, so the same bits) and
// goes on with its own columns.  The state being pushed (B on the way forward,
// Phi on the way back) stays in shared memory for the whole sweep; the B list
// goes to global memory and each B_{k-1} is fetched again while the update of
// gate k + 1 runs.
//
// What bounds it: a start is a chain of 2L - 1 steps and L updates, and at
// these sizes a step is short, so latency decides: the update (polar_newton.cuh)
// and the exchange.  FP64 slices of thousands of entries are bound by the FP64
// pipe instead (2 lanes per clock and SM; 48 FMAs per entry and gate).
//
// complex64: a thread owns a unit (the four rows of one r and one column) of a
// gate step, so steps on shared memory are in place, what it stores of the B
// list it alone reads back (cp.async into its own slots), and E comes from
// registers.  FP64: work is cut to one output component per lane (8 products
// per gate step), and each lane of a warp sums one of the 32 components of E.
//
// FP64 in fixed point (FX).  An FP64 FMA costs a warp 60 cycles on this chip,
// a 32 x 32 -> 64 bit integer one about 7.  The columns of Psi and U Psi have a
// norm that unitary gates keep, so no entry of B_k or Phi_k ever exceeds it,
// and a fixed point of 2^-60 of that norm (kept as high and low 30 bits) holds
// an entry as well as FP64 does: entries of a state on n qubits are about
// 2^(-n/2), where FP64's spacing is 2^(-53 - n/2).  A product takes three
// integer FMAs (the low x low part, below 2^-60, is left out), the sums are
// exact and E is rounded once.  The plain FP64 form remains for inputs without
// that bound (initial gates that are not unitary, columns out of range).
#include "polar_newton.cuh"
#include "qfs_common.cuh"
#include "qfs_kernels.h"

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

namespace qfs {

namespace {

constexpr int kClMaxC = 16;
constexpr int kMaxSmem = 211 * 1024;  // (beside 15 KB of static shared memory)
constexpr int kClRing = 3;  // rounds of B in flight per thread (complex64)

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Eight bytes to shared memory of a CTA of the cluster; they count on its barrier.
__device__ __forceinline__ void st_async8(uint32_t addr, unsigned long long v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(addr), "l"(v), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(smem)), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ int ld_volatile(const int* p) { return *reinterpret_cast<const volatile int*>(p); }

struct ClShared {
  unsigned long long exch[2][kClMaxC][32];  // environment sums of the cluster's CTAs, two exchanges deep
  unsigned long long red[16][32];           // per-warp sums
  unsigned long long mbar[2];
  NewtonSh nw;
  long long out[32];  // the new gate for the warp that writes it out: components of newton_update, or FP64
  int flag, out_fx;
};

// Sum of the CTAs' values: each CTA's warp 0 brings one 8-byte value per lane;
// on return ClShared::exch[par] holds every CTA's.  Bounded: false when a wait
// runs out.
__device__ __forceinline__ bool cl_exchange(ClShared& sh, uint32_t C, uint32_t rank, uint32_t& count, unsigned long long v,
                                            long long limit) {
  const int lane = threadIdx.x & 31;
  const uint32_t par = count & 1u, phase = (count >> 1) & 1u;
  ++count;
  const uint32_t bar = smem_u32(&sh.mbar[par]), slot = smem_u32(&sh.exch[par][rank][lane]);
  if (lane == 0) mbar_expect(bar, C * 256u);
  for (uint32_t c = 0; c < C; ++c) {
    const uint32_t to = (rank + c) % C;
    st_async8(mapa(slot, to), v, mapa(bar, to));
  }
  long long polls = 0;
  while (!mbar_test(bar, phase)) {
    if (++polls > limit) return false;
  }
  return true;
}

// The update of a gate in warp 0 from E, whose value j (2 (4x + y) + {re, im})
// is in lane j: ehi + elo (complex64), v in units of 2^ev (FX) or e64.  Leaves
// the gate in gs (and in gd, the FP64 copy that a damped run needs).  True: q
// is its component as newton_update leaves it; false: p is its entry [l16 & 3]
// [l16 >> 2] in lanes 0..15.
template <typename T, bool FX>
__device__ __forceinline__ bool cl_update(const ClArgs& a, ClShared& sh, double e64, float ehi, float elo, long long v,
                                          const NewtonPair& pair, typename C2<T>::t* gs, double2* gd, long long& q, double2& p) {
  constexpr bool F32 = sizeof(T) == 4;
  const int lane = threadIdx.x & 31;
  const int l16 = lane & 15, im = lane >> 4, at = 4 * (l16 & 3) + (l16 >> 2);
  const bool damp = a.beta != 0.0;
  auto matrix = [&]() {
    if (F32 && !damp) e64 = (double)ehi + (double)elo;
    const double2 m = newton_env(e64);
    return damp ? newton_damp(m, a.beta, F32 || FX ? gd : reinterpret_cast<const double2*>(gs)) : m;
  };
  float2 a32;
  if (damp || (!F32 && !FX)) {
    a32 = newton_input64(matrix(), sh.nw);  // (e64 is set)
  } else if (F32) {
    a32 = newton_input32(ehi);
  } else {
    // Largest entry to [2^59, 2^60).
    const unsigned long long mag = v < 0 ? -(unsigned long long)v : (unsigned long long)v;
    const int msb = __reduce_max_sync(FULL, 63 - __clzll(mag));  // (-1: zero)
    const int sft = kFxBits - 1 - msb;
    const long long w = msb < 0 ? 0 : sft >= 0 ? v << sft : v >> -sft;
    const int2 f = fx_split((lane & 1) ? -w : w);
    // Lane j of E is entry [j >> 3][(j >> 1) & 3]: A[y][x] at 4x + y.
    reinterpret_cast<int2*>(&sh.nw.A[lane >> 1])[lane & 1] = f;
    const float fv = fmaf((float)f.x, 1.f / (1 << (kFxBits - kFxLow)), (float)f.y * (1.f / (1LL << kFxBits)));
    a32 = float2{__shfl_sync(FULL, fv, 2 * l16), __shfl_sync(FULL, fv, 2 * l16 + 1)};
    __syncwarp();
  }
  const bool ok = newton_update<!F32>(a32, sh.nw, pair, q);
  if (ok) {
    if constexpr (F32) {
      reinterpret_cast<float*>(gs)[2 * at + im] = (float)q * (1.f / (1LL << kFxBits));
    } else if constexpr (FX) {
      reinterpret_cast<int2*>(gs)[2 * at + im] = fx_split(q);
    }
    if ((!F32 && !FX) || gd) p = newton_entry64(q);
  } else {
    if (FX && !damp) e64 = (double)v;  // (its scale does not matter)
    p = newton_fallback(matrix(), sh.nw);
    if (lane < 16) {
      if constexpr (F32) gs[at] = float2{(float)p.x, (float)p.y};
      else if constexpr (FX) reinterpret_cast<int4*>(gs)[at] = fx_from2(p, 0);
    }
  }
  if (!F32 && !FX && lane < 16) reinterpret_cast<double2*>(gs)[at] = p;
  if (gd && lane < 16) gd[at] = p;
  __syncwarp();
  return ok;
}

// Sum over the cluster of one FP32 pair per lane (complex64), or of one FP64
// value per lane; warp 0 only.
__device__ __forceinline__ bool cl_sum_pair(ClShared& sh, uint32_t C, uint32_t rank, uint32_t& count, float& hi, float& lo,
                                            long long limit) {
  if (C == 1) return true;
  const int lane = threadIdx.x & 31;
  const uint32_t par = count & 1u;
  const unsigned long long v = ((unsigned long long)__float_as_uint(lo) << 32) | __float_as_uint(hi);
  if (!cl_exchange(sh, C, rank, count, v, limit)) return false;
  float h = 0.f, l = 0.f;
  for (uint32_t c = 0; c < C; ++c) {
    const unsigned long long w = *reinterpret_cast<const volatile unsigned long long*>(&sh.exch[par][c][lane]);
    float e;
    two_sum(h, __uint_as_float((unsigned)w), h, e);
    l += e + __uint_as_float((unsigned)(w >> 32));
  }
  hi = h;
  lo = l;
  return true;
}
__device__ __forceinline__ bool cl_sum_int(ClShared& sh, uint32_t C, uint32_t rank, uint32_t& count, long long& v,
                                           long long limit) {
  if (C == 1) return true;
  const int lane = threadIdx.x & 31;
  const uint32_t par = count & 1u;
  if (!cl_exchange(sh, C, rank, count, (unsigned long long)v, limit)) return false;
  long long t = 0;
  for (uint32_t c = 0; c < C; ++c)
    t += (long long)*reinterpret_cast<const volatile unsigned long long*>(&sh.exch[par][c][lane]);
  v = t;
  return true;
}
__device__ __forceinline__ bool cl_sum_double(ClShared& sh, uint32_t C, uint32_t rank, uint32_t& count, double& v,
                                              long long limit) {
  if (C == 1) return true;
  const int lane = threadIdx.x & 31;
  const uint32_t par = count & 1u;
  if (!cl_exchange(sh, C, rank, count, (unsigned long long)__double_as_longlong(v), limit)) return false;
  double t = 0.0;
  for (uint32_t c = 0; c < C; ++c)
    t += __longlong_as_double((long long)*reinterpret_cast<const volatile unsigned long long*>(&sh.exch[par][c][lane]));
  v = t;
  return true;
}

__device__ __forceinline__ PairBits cl_geo(const ClArgs& a, int k) { return pair_bits(a.pos[k] & 15, a.pos[k] >> 4); }

// What a start that gave up has is not a sweep's: NaN, for a caller that has no
// error word.  (A loop that is not unrolled: unrolled, or as a call, the code around
// it shifts and a chain of short sweeps takes 1% longer, 3815 -> 3850 us at n = 3.)
__device__ __forceinline__ void cl_give_up(const ClArgs& a, int s) {
  const double nan = __longlong_as_double(-1LL);
#pragma unroll 1
  for (int i = threadIdx.x; i < a.L * 16; i += blockDim.x) {
    const long long at = (long long)s * a.L * 16 + i;
    a.g64[at] = double2{nan, nan};
    if (a.envs != nullptr) a.envs[at] = double2{nan, nan};
  }
  if (threadIdx.x == 0) a.costs[s] = nan;
}

}  // namespace

// One cluster per start; a.nsweeps sweeps of it.
//
// Time of a sweep (us), dataflow sweep as it was -> this kernel: n = 3, 4
// gates, M = 4, 1 start, FP64 105 -> 18; n = 7, 21 gates, M = 24, 5 starts,
// FP64 608 -> 121; n = 8, 28 gates, M = 16, 16 starts, FP64 816 -> 232 and
// complex64 443 -> 92; n = 10, 18 gates, M = 32, 8 starts, FP64 788 -> 384.
// A gate of the n = 8 FP64 sweep then takes 16,000 cycles: forward product
// 2400, environment 2400, sums and exchange 1800, update 6700, backward product
// 1800, barriers and hand-over 900.
//
// 256 threads: the phases are short, so more warps only lengthen the barriers;
// 512 for complex64 slices of 4096 entries and more, whose steps are bound by
// shared memory and FP32 issue.
template <typename T, int NT, bool FX>
__global__ void __launch_bounds__(NT, 1) k_sweep_cl(ClArgs a) {
  using T2 = typename C2<T>::t;
  constexpr bool F32 = sizeof(T) == 4;
  constexpr int NW = NT / 32;
  extern __shared__ __align__(16) unsigned char cl_smem[];
  __shared__ ClShared sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t C = a.C, rank = C == 1 ? 0 : cluster_rank();
  const int s = blockIdx.x / C;
  const int n = a.n, L = a.L, M = a.M;
  const uint32_t fold = swz_fold(n);
  // (Uniform over a cluster: an earlier launch set the stop word, or the start is inactive.)
  if (a.stop != nullptr && ld_volatile(a.stop) < a.sweep0) return;
  if (a.active != nullptr && a.active[s] == 0) return;
  // (FP64: the target's scales; a form takes only the targets it is for.)
  int e_psi = 0, e_phi = 0;
  if (sizeof(T) == 8) {
    const int4 sc = a.scale != nullptr ? a.scale[s / a.spt] : int4{1, 0, 0, 0};
    if ((sc.x == 0) != FX) return;
    e_psi = sc.y + a.e_head;
    e_phi = sc.z;
  }
  const int c0 = (int)((long long)M * rank / C), mc = (int)((long long)M * (rank + 1) / C) - c0;
  const int E = mc << n, units = E >> 2, rbits = n - 2;
  const int slice = ((M + C - 1) / C) << n;  // entries of the largest slice
  // Shared memory: gates, (FP64 copies,) row bits, state, second state or ring.
  T2* gates = reinterpret_cast<T2*>(cl_smem);
  double2* gates64 = reinterpret_cast<double2*>(gates + L * 16);
  const bool keep64 = (F32 || FX) && a.beta != 0.0;
  T2* X = reinterpret_cast<T2*>(gates64 + (keep64 ? L * 16 : 0));
  T2* X2 = X + slice;                                  // FP64
  float4* ring = reinterpret_cast<float4*>(X + slice);  // complex64
  double2* g64 = a.g64 + (long long)s * L * 16;
  float2* g32 = F32 ? a.g32 + (long long)s * L * 16 : nullptr;
  const long long sN = (long long)M << n, tgt = (long long)(s / a.spt) * sN;
  const T2* psi = reinterpret_cast<const T2*>(a.psi) + tgt;
  const T2* phil = reinterpret_cast<const T2*>(a.phil) + tgt;
  T2* bl = reinterpret_cast<T2*>(a.blist) + (long long)s * sN + ((long long)c0 << n);
  const long long bstep = (long long)a.S * sN;
  T2* last = reinterpret_cast<T2*>(a.blast) + (long long)s * sN + ((long long)c0 << n);  // complex64: B_{L-1}

  if (C > 1) {
    if (tid == 0) {
      mbar_init(smem_u32(&sh.mbar[0]), 1);
      mbar_init(smem_u32(&sh.mbar[1]), 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    cluster_arrive();
  }
  for (int i = tid; i < L * 16; i += NT) {
    if constexpr (F32) gates[i] = g32[i];
    else if constexpr (FX) reinterpret_cast<int4*>(gates)[i] = fx_from2(g64[i], 0);
    else gates[i] = g64[i];
    if (keep64) gates64[i] = g64[i];
  }
  if (C > 1) cluster_wait();
  uint32_t count = 0;
  bool alive = true;
  const NewtonPair pair = newton_pair();

  // Entries of the slice from a row-major N x M state.
  auto load_slice = [&](const T2* src, T2* dst, int e) {
    for (int i = tid; i < E; i += NT) {
      const int row = i / mc, j = i - row * mc;
      const uint32_t at = swz(((uint32_t)j << n) | (uint32_t)row, fold);
      const T2 v = __ldg(src + (long long)row * M + c0 + j);
      if constexpr (FX) reinterpret_cast<int4*>(dst)[at] = fx_from2(v, e);
      else dst[at] = v;
    }
  };
  // Complex64: this thread's unit of round rd in the B list, as two float4 (rows 0 and 1, rows 2 and 3).
  const int rounds = (units + NT - 1) / NT;
  auto bunit = [&](int k, int h, int u) {
    return reinterpret_cast<float4*>(k + 1 < L ? bl + k * bstep : last) + (long long)h * units + u;
  };
  auto fetch = [&](int q) {  // round q of the whole backward pass: gate L - 1 - q / rounds
    if constexpr (F32) {
      const int k = L - 1 - q / rounds, u = (q % rounds) * NT + tid;
      if (k >= 0 && u < units) {
        float4* slot = ring + (q % kClRing) * 2 * NT + tid;
        cp_async16(slot, bunit(k, 0, u));
        cp_async16(slot + NT, bunit(k, 1, u));
      }
      cp_commit();
    }
  };
  auto fetch_b = [&](int k, T2* dst) {  // FP64: B_k's slice
    for (int i = tid; i < E; i += NT) cp_async16(dst + i, bl + k * bstep + i);
    cp_commit();
  };
  // FP64: out = G in, one component of one output row per lane; ADJ: G^dagger.
  auto apply64 = [&](int k, const T2* in, T2* out, bool adj) {
    if constexpr (!F32) {
      const PairBits g = cl_geo(a, k);
      const int x = (lane >> 1) & 3, im = lane & 1;
      double p[4], q[4];  // out = sum p v.x + q v.y
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        double2 w = adj ? gates[16 * k + 4 * j + x] : gates[16 * k + 4 * x + j];
        const double wy = neg_if(w.y, adj), ny = neg_if(wy, true);
        p[j] = im ? wy : w.x;
        q[j] = im ? w.x : ny;
      }
      uint32_t xo[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) xo[j] = swz(((uint32_t)(j >> 1) << g.pa) | ((uint32_t)(j & 1) << g.pb), fold);
      const uint32_t mine = xo[x];
      const int upr = NT / 8;
      for (int u0 = warp * 4; u0 < units; u0 += 2 * upr) {
        const int ua = u0 + (lane >> 3), ub = ua + upr;
        const bool va = ua < units, vb = ub < units;
        const uint32_t ba = swz(((uint32_t)(ua >> rbits) << n) |
                                insert_two_zero_bits((uint32_t)ua & ((1u << rbits) - 1u), g.lo, g.hi), fold);
        const uint32_t bb = swz(((uint32_t)(ub >> rbits) << n) |
                                insert_two_zero_bits((uint32_t)ub & ((1u << rbits) - 1u), g.lo, g.hi), fold);
        double ra = 0.0, rb = 0.0;
        double2 v[4], w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = va ? in[ba ^ xo[j]] : double2{0.0, 0.0};
        if (u0 + upr < units) {  // (uniform over the warp: FP64 instructions are not issued for nothing)
#pragma unroll
          for (int j = 0; j < 4; ++j) w[j] = vb ? in[bb ^ xo[j]] : double2{0.0, 0.0};
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            ra = fma(p[j], v[j].x, ra);
            rb = fma(p[j], w[j].x, rb);
            ra = fma(q[j], v[j].y, ra);
            rb = fma(q[j], w[j].y, rb);
          }
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            ra = fma(p[j], v[j].x, ra);
            ra = fma(q[j], v[j].y, ra);
          }
        }
        __syncwarp();  // (in place: the eight lanes of a unit have read it)
        if (va) reinterpret_cast<double*>(out + (ba ^ mine))[im] = ra;
        if (vb) reinterpret_cast<double*>(out + (bb ^ mine))[im] = rb;
      }
    }
  };

  for (int sw = 0; sw < a.nsweeps && alive; ++sw) {
    if (sw > 0 && a.stop != nullptr) {  // (one CTA per start)
      if (tid == 0) sh.flag = ld_volatile(a.stop) >= a.sweep0 + sw;
      __syncthreads();
      if (!sh.flag) break;
      __syncthreads();
    }
    T2* Bs = X2;   // FP64: B_k during the backward pass
    T2* Ph = X;    // Phi
    // ---------------------------------------------------------------- forward
    load_slice(psi, X, e_psi);
    __syncthreads();
    if constexpr (F32) {
      for (int k = 0; k < L; ++k) {
        const PairBits g = cl_geo(a, k);
        uint32_t xo[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) xo[j] = swz(((uint32_t)(j >> 1) << g.pa) | ((uint32_t)(j & 1) << g.pb), fold);
        T2 gr[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) gr[i] = gates[16 * k + i];
        for (int u = tid; u < units; u += NT) {
          const uint32_t b = swz(((uint32_t)(u >> rbits) << n) |
                                 insert_two_zero_bits((uint32_t)u & ((1u << rbits) - 1u), g.lo, g.hi), fold);
          T2 v[4];
#pragma unroll
          for (int x = 0; x < 4; ++x) v[x] = X[b ^ xo[x]];
          __stcg(bunit(k, 0, u), float4{v[0].x, v[0].y, v[1].x, v[1].y});
          __stcg(bunit(k, 1, u), float4{v[2].x, v[2].y, v[3].x, v[3].y});
          if (k + 1 < L) {
#pragma unroll
            for (int x = 0; x < 4; ++x) {
              T2 t = cmul(gr[4 * x], v[0]);
#pragma unroll
              for (int j = 1; j < 4; ++j) t = cfma(gr[4 * x + j], v[j], t);
              X[b ^ xo[x]] = t;
            }
          }
        }
        __syncthreads();
      }
#pragma unroll
      for (int q = 0; q < kClRing - 1; ++q) fetch(q);
    } else {
      T2 *in = X, *out = X2;
      for (int k = 0; k + 1 < L; ++k) {
        for (int i = tid; i < E; i += NT) __stcg(bl + k * bstep + i, in[i]);
        if constexpr (FX)
          fx_apply<NT>(reinterpret_cast<const int4*>(in), reinterpret_cast<int4*>(out),
                       reinterpret_cast<const int4*>(gates) + 16 * k, cl_geo(a, k), false, units, n);
        else apply64(k, in, out, false);
        __syncthreads();
        T2* t = in;
        in = out;
        out = t;
      }
      Bs = in;  // B_{L-1}, the first environment's
      Ph = out;
    }
    load_slice(phil, Ph, e_phi);
    __syncthreads();
    // --------------------------------------------------------------- backward
    double cost = 0.0;
    for (int k = L - 1; k >= 0; --k) {
      const PairBits g = cl_geo(a, k);
      uint32_t xo[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) xo[j] = swz(((uint32_t)(j >> 1) << g.pa) | ((uint32_t)(j & 1) << g.pb), fold);
      auto unit_base = [&](int u) {
        return swz(((uint32_t)(u >> rbits) << n) |
                   insert_two_zero_bits((uint32_t)u & ((1u << rbits) - 1u), g.lo, g.hi), fold);
      };
      // Environment of this CTA's columns.
      if constexpr (F32) {
        float acc[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) acc[i] = 0.f;
        for (int rd = 0; rd < rounds; ++rd) {
          const int q = (L - 1 - k) * rounds + rd;
          fetch(q + kClRing - 1);
          cp_wait<kClRing - 1>();
          const int u = rd * NT + tid;
          if (u < units) {
            const uint32_t b = unit_base(u);
            const float4* slot = ring + (q % kClRing) * 2 * NT + tid;
            const float4 b01 = slot[0], b23 = slot[NT];
            const float2 bv[4] = {float2{b01.x, b01.y}, float2{b01.z, b01.w}, float2{b23.x, b23.y}, float2{b23.z, b23.w}};
            float2 ph[4];
#pragma unroll
            for (int y = 0; y < 4; ++y) ph[y] = Ph[b ^ xo[y]];
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
              for (int y = 0; y < 4; ++y)
                cfma_conj(acc[2 * (4 * x + y)], acc[2 * (4 * x + y) + 1], bv[x], ph[y]);
          }
        }
        const float mine = warp_reduce_scatter32<float>(acc, lane);
        reinterpret_cast<float*>(sh.red[warp])[lane] = mine;
      } else if constexpr (FX) {
        cp_wait<0>();
        __syncthreads();
        const int x = lane >> 3, y = (lane >> 1) & 3, im = lane & 1;
        const uint32_t ox = xo[x], oy = xo[y];
        const int4 *Bx = reinterpret_cast<const int4*>(Bs), *Px = reinterpret_cast<const int4*>(Ph);
        // E[x][y] += B[x] conj(Phi[y]): re = b.x p.x + b.y p.y, im = b.y p.x - b.x p.y.
        // The cross sums are folded into s0 often enough that they cannot overflow
        // (Cauchy-Schwarz over four units).
        long long s0 = 0, s1 = 0, s2 = 0;
        auto term = [&](int u) {
          const uint32_t e = unit_base(u);
          const int4 b = Bx[e ^ ox], p = Px[e ^ oy];
          const int2 b1{im ? b.z : b.x, im ? b.w : b.y}, b2{im ? -b.x : b.z, im ? -b.y : b.w};
          s0 = mad64(b1.x, p.x, s0);
          s1 = mad64(b1.x, p.y, s1);
          s2 = mad64(b1.y, p.x, s2);
          s0 = mad64(b2.x, p.z, s0);
          s1 = mad64(b2.x, p.w, s1);
          s2 = mad64(b2.y, p.z, s2);
        };
        auto fold = [&]() {
          const long long c = s1 + s2;
          s0 += c >> kFxLow;
          s1 = c & ((1LL << kFxLow) - 1);
          s2 = 0;
        };
        int u = warp;
        for (; u + 3 * NW < units; u += 4 * NW) {
#pragma unroll
          for (int i = 0; i < 4; ++i) term(u + i * NW);
          fold();
        }
        for (; u < units; u += NW) term(u);
        fold();
        reinterpret_cast<long long*>(sh.red[warp])[lane] = s0;
      } else {
        cp_wait<0>();
        __syncthreads();
        const int slices = units >= 256 ? NW : 4;
        if (warp < slices) {
          const int x = lane >> 3, y = (lane >> 1) & 3, im = lane & 1;
          const uint32_t ox = xo[x], oy = xo[y];
          // E[x][y] += B[x] conj(Phi[y]): re = b.x p.x + b.y p.y, im = b.y p.x - b.x p.y
          double t[4] = {0.0, 0.0, 0.0, 0.0};
          int u = warp;
          for (; u + 3 * slices < units; u += 4 * slices) {
            double2 b[4], p[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const uint32_t e = unit_base(u + i * slices);
              b[i] = Bs[e ^ ox];
              p[i] = Ph[e ^ oy];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) t[i] = fma(im ? b[i].y : b[i].x, p[i].x, t[i]);
#pragma unroll
            for (int i = 0; i < 4; ++i) t[i] = fma(neg_if(im ? b[i].x : b[i].y, im), p[i].y, t[i]);
          }
          for (; u < units; u += slices) {
            const uint32_t e = unit_base(u);
            const double2 b = Bs[e ^ ox], p = Ph[e ^ oy];
            t[0] = fma(im ? b.y : b.x, p.x, t[0]);
            t[0] = fma(neg_if(im ? b.x : b.y, im), p.y, t[0]);
          }
          if (warp + 3 * slices < units) t[0] = (t[0] + t[1]) + (t[2] + t[3]);
          reinterpret_cast<double*>(sh.red[warp])[lane] = t[0];
        }
      }
      __syncthreads();
      if constexpr (!F32) {
        if (k > 0) fetch_b(k - 1, Bs);
      }
      // Sum over the warps and the cluster, update.
      float hi = 0.f, lo = 0.f;
      double e = 0.0;
      long long fx = 0, q = 0;
      double2 p{0.0, 0.0};
      bool isq = false;
      const int e_unit = e_psi + e_phi - kFxBits + a.e_shift;  // FX: the unit of fx
      if (warp == 0) {
        if constexpr (F32) {
#pragma unroll
          for (int w = 0; w < NW; ++w) {
            float t;
            two_sum(hi, reinterpret_cast<const float*>(sh.red[w])[lane], hi, t);
            lo += t;
          }
          alive = cl_sum_pair(sh, C, rank, count, hi, lo, a.wait_limit);
        } else if constexpr (FX) {
          // Exact up to here; a.e_shift makes room for the sum over M columns.
          fx = (1LL << a.e_shift) >> 1;
#pragma unroll
          for (int w = 0; w < NW; ++w) fx += reinterpret_cast<const long long*>(sh.red[w])[lane];
          fx >>= a.e_shift;
          alive = cl_sum_int(sh, C, rank, count, fx, a.wait_limit);
        } else {
          const int slices = units >= 256 ? NW : 4;
          e = reinterpret_cast<const double*>(sh.red[0])[lane];
          for (int w = 1; w < slices; ++w) e += reinterpret_cast<const double*>(sh.red[w])[lane];
          alive = cl_sum_double(sh, C, rank, count, e, a.wait_limit);
        }
        alive = __all_sync(FULL, alive);
        if (F32 && a.beta != 0.0) e = (double)hi + (double)lo;
        if (FX && a.beta != 0.0) e = scale_exp((double)fx, e_unit);
        isq = cl_update<T, FX>(a, sh, e, hi, lo, fx, pair, gates + 16 * k, keep64 ? gates64 + 16 * k : nullptr, q, p);
        if (k == 0) {
          // 2 - (2 / M) Re tr(g E): the factor's entry [r][c] meets E[c][r].
          if (F32) e = (double)hi + (double)lo;
          if (FX) e = scale_exp((double)fx, e_unit);
          if (isq) p = newton_entry64(q);
          const int l16 = lane & 15;
          const double ex = __shfl_sync(FULL, e, 2 * l16), ey = __shfl_sync(FULL, e, 2 * l16 + 1);
          double t = lane < 16 ? (p.x * ex - p.y * ey) : 0.0;
#pragma unroll
          for (int o = 16; o >= 1; o >>= 1) t += __shfl_xor_sync(FULL, t, o);
          if (lane == 0) reinterpret_cast<double&>(sh.red[0][0]) = 2.0 - 2.0 * a.inv_M * t;
        }
        const double py = __shfl_sync(FULL, p.y, lane & 15);
        sh.out[lane] = isq ? q : __double_as_longlong(lane < 16 ? p.x : py);
        if (lane == 0) {
          sh.out_fx = isq;
          sh.flag = alive;
        }
        if (rank == 0 && a.envs != nullptr) {
          if (F32) e = (double)hi + (double)lo;
          if (FX) e = scale_exp((double)fx, e_unit);
          reinterpret_cast<double*>(a.envs + ((long long)s * L + k) * 16)[lane] = e;
        }
      }
      __syncthreads();
      if (warp == NW - 1 && rank == 0) {  // the gate's way out, off warp 0's chain
        const int at = 16 * k + 4 * (lane & 3) + ((lane >> 2) & 3), im = lane >> 4;
        const long long w = sh.out[lane];
        reinterpret_cast<double*>(g64 + at)[im] = sh.out_fx ? scale_exp((double)w, -kFxBits) : __longlong_as_double(w);
        if constexpr (F32) {
          if (lane < 16) g32[at] = gates[at];
        }
      }
      alive = sh.flag != 0;
      if (!alive) break;
      if (k == 0) {
        cost = reinterpret_cast<const double&>(sh.red[0][0]);
        break;
      }
      // Phi_{k-1} = g_k^dagger Phi_k
      if constexpr (F32) {
        T2 gd[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const T2 t = gates[16 * k + 4 * (i & 3) + (i >> 2)];
          gd[i] = T2{t.x, -t.y};
        }
        for (int u = tid; u < units; u += NT) {
          const uint32_t b = unit_base(u);
          T2 v[4];
#pragma unroll
          for (int x = 0; x < 4; ++x) v[x] = Ph[b ^ xo[x]];
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            T2 t = cmul(gd[4 * x], v[0]);
#pragma unroll
            for (int j = 1; j < 4; ++j) t = cfma(gd[4 * x + j], v[j], t);
            Ph[b ^ xo[x]] = t;
          }
        }
        __syncthreads();
      } else {
        if constexpr (FX)
          fx_apply<NT>(reinterpret_cast<const int4*>(Ph), reinterpret_cast<int4*>(Ph),
                       reinterpret_cast<const int4*>(gates) + 16 * k, g, true, units, n);
        else apply64(k, Ph, Ph, true);
        // The next environment waits for it behind its barrier.
      }
    }
    if (!alive) break;
    if constexpr (F32) {
      // The residual cost (1/M) sum |g_1^dagger Phi_1 - Psi|^2, unless the
      // update's estimate is so far above the tolerance that it decides nothing.
      if (!(a.resid_skip > 0.0 && cost > a.resid_skip)) {
        const PairBits g = cl_geo(a, 0);
        T2 gd[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const T2 t = gates[4 * (i & 3) + (i >> 2)];
          gd[i] = T2{t.x, -t.y};
        }
        float r = 0.f;
        for (int u = tid; u < units; u += NT) {
          const uint32_t b = swz(((uint32_t)(u >> rbits) << n) |
                                 insert_two_zero_bits((uint32_t)u & ((1u << rbits) - 1u), g.lo, g.hi), fold);
          const float4 b01 = __ldcg(bunit(0, 0, u)), b23 = __ldcg(bunit(0, 1, u));
          const float2 bv[4] = {float2{b01.x, b01.y}, float2{b01.z, b01.w}, float2{b23.x, b23.y}, float2{b23.z, b23.w}};
          T2 v[4];
#pragma unroll
          for (int x = 0; x < 4; ++x)
            v[x] = Ph[b ^ swz(((uint32_t)(x >> 1) << g.pa) | ((uint32_t)(x & 1) << g.pb), fold)];
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            T2 t = cmul(gd[4 * x], v[0]);
#pragma unroll
            for (int j = 1; j < 4; ++j) t = cfma(gd[4 * x + j], v[j], t);
            const float dx = t.x - bv[x].x, dy = t.y - bv[x].y;
            r = fmaf(dx, dx, fmaf(dy, dy, r));
          }
        }
        double rd = (double)r;
#pragma unroll
        for (int m = 16; m >= 1; m >>= 1) rd += __shfl_xor_sync(FULL, rd, m);
        __syncthreads();  // (red[0] held the estimate)
        if (lane == 0) reinterpret_cast<double&>(sh.red[warp][0]) = rd;
        __syncthreads();
        if (warp == 0) {
          double t = lane < NW ? reinterpret_cast<const double&>(sh.red[lane][0]) : 0.0;
#pragma unroll
          for (int m = 8; m >= 1; m >>= 1) t += __shfl_xor_sync(FULL, t, m);
          t = __shfl_sync(FULL, t, 0);
          alive = cl_sum_double(sh, C, rank, count, t, a.wait_limit);
          alive = __all_sync(FULL, alive);
          if (lane == 0) {
            reinterpret_cast<double&>(sh.red[0][0]) = t * a.inv_M;
            sh.flag = alive;
          }
        }
        __syncthreads();
        alive = sh.flag != 0;
        if (!alive) break;
        cost = reinterpret_cast<const double&>(sh.red[0][0]);
      }
      cp_wait<0>();
    }
    if (rank == 0 && tid == 0) {
      a.costs[s] = cost;
      if (a.cost_rows != nullptr) a.cost_rows[(long long)sw * a.S + s] = cost;
      if (a.stop != nullptr && cost <= a.stop_tol) atomicMin(a.stop, a.sweep0 + sw);
    }
    if (cost <= a.stop_tol && a.nsweeps > 1) break;  // (this start has met the tolerance: it sweeps no further)
    __syncthreads();
  }
  if (!alive && tid == 0 && a.err != nullptr) atomicOr(a.err, 1);
  // No CTA leaves while copies of its own are in flight or a peer may still
  // store to its shared memory.  A CTA that saw every exchange complete has
  // received all there is; one that gave up waits (bounded) for what its peers
  // had sent by the time all of them stopped.
  cp_wait<0>();
  if (C > 1) {
    cluster_arrive();
    cluster_wait();
    if (!alive) {
      cl_give_up(a, s);
#pragma unroll 1
      for (int i = 0; i < 256; ++i) __nanosleep(1000);
    }
  }
}

namespace {

size_t cl_smem_bytes(Real r, int n, int M, int L, int C, int NT, bool keep64) {
  const size_t es = r == R32 ? 8 : 16;
  const size_t slice = ((size_t)(M + C - 1) / C) << n;
  size_t b = (size_t)L * 16 * es + (keep64 ? (size_t)L * 16 * 16 : 0);
  b += slice * es;
  b += r == R32 ? (size_t)kClRing * 2 * NT * 16 : slice * es;
  return b;
}
// Threads of a CTA: enough units (complex64) for 512, else 256.
int cl_threads(Real r, int n, int M, int C) {
  return r == R32 && ((size_t)((M + C - 1) / C) << n) >= 4096 ? 512 : 256;
}
using ClKernel = void (*)(ClArgs);
ClKernel cl_kernel(Real r, int nt, bool fx) {
  if (r == R64) return fx ? k_sweep_cl<double, 256, true> : k_sweep_cl<double, 256, false>;
  return nt == 512 ? k_sweep_cl<float, 512, false> : k_sweep_cl<float, 256, false>;
}
// Clusters of C CTAs that the device holds at once.
int cl_resident(Real r, int nt, bool fx, int C, size_t smem) {
  static std::mutex mu;
  static std::map<std::tuple<int, int, int, int, size_t>, int> known;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  const auto key = std::make_tuple(dev, (int)r * 2 + (int)fx, nt, C, smem);
  {
    std::lock_guard<std::mutex> lock(mu);
    const auto it = known.find(key);
    if (it != known.end()) return it->second;
  }
  int num = 0;
  const ClKernel kernel = cl_kernel(r, nt, fx);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(64 * C));
  cfg.blockDim = dim3((unsigned)nt);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)C;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
  if (e == cudaSuccess && C > 8) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&num, kernel, &cfg);
  if (e != cudaSuccess) {
    cudaGetLastError();
    num = 0;
  }
  std::lock_guard<std::mutex> lock(mu);
  known[key] = num;
  return num;
}

}  // namespace

// The FP64 sample cost (1/M) sum_j ||U psi_j - C psi_j||^2 of one start's gates
// in fixed point: CTA j pushes column j through the circuit in shared memory
// (columns need nothing from one another), so a check is one launch instead of
// one per gate: 33 us against 242 us at n = 8 with 28 gates and 16 columns,
// 159 against 188 us at n = 12 with 17 gates and 32.  The differences are exact, their
// squares are summed in FP64, the columns by the CTA that finishes last.
template <int NT>
__global__ void __launch_bounds__(NT) k_cl_check(ClArgs a, double* parts, unsigned* count) {
  extern __shared__ __align__(16) unsigned char cl_smem[];
  __shared__ double red[NT / 32];
  __shared__ int last;
  const int tid = threadIdx.x, lane = tid & 31, n = a.n, N = 1 << n, M = a.M, j = blockIdx.x;
  const uint32_t fold = swz_fold(n);
  const int4 sc = a.scale[0];
  const int e = max(sc.y, sc.z);  // one scale for both sides of the difference
  int4* gates = reinterpret_cast<int4*>(cl_smem);
  int4* X = gates + a.L * 16;
  for (int i = tid; i < a.L * 16; i += NT) gates[i] = fx_from2(a.g64[i], 0);
  const double2* psi = reinterpret_cast<const double2*>(a.psi);
  const double2* phil = reinterpret_cast<const double2*>(a.phil);
  for (int i = tid; i < N; i += NT) X[swz((uint32_t)i, fold)] = fx_from2(__ldg(psi + (long long)i * M + j), e);
  __syncthreads();
  for (int k = 0; k < a.L; ++k) {
    fx_apply<NT>(X, X, gates + 16 * k, cl_geo(a, k), false, N >> 2, n);
    __syncthreads();
  }
  double t = 0.0;
  for (int i = tid; i < N; i += NT) {
    const int4 x = X[swz((uint32_t)i, fold)], y = fx_from2(__ldg(phil + (long long)i * M + j), e);
    const double dx = (double)(fx_value(y.x, y.y) - fx_value(x.x, x.y)),
                 dy = (double)(fx_value(y.z, y.w) - fx_value(x.z, x.w));
    t = fma(dx, dx, fma(dy, dy, t));
  }
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) t += __shfl_xor_sync(FULL, t, m);
  if (lane == 0) red[tid >> 5] = t;
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < NT / 32; ++w) t += red[w];
    __stcg(parts + j, t);
    __threadfence();
    last = atomicAdd(count, 1u) == (unsigned)M - 1;
  }
  __syncthreads();
  if (last && tid < 32) {
    __threadfence();
    double v = 0.0;
    for (int c = lane; c < M; c += 32) v += __ldcg(parts + c);
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) v += __shfl_xor_sync(FULL, v, m);
    if (lane == 0) {
      a.costs[0] = ldexp(v, 2 * (e - kFxBits)) * a.inv_M;
      *count = 0;
    }
  }
}

// The scales of one target's fixed-point sweeps: out = {plain, e_psi, e_phi, 0},
// plain 0 or the reason why its sweeps take the plain FP64 form (kClPlain...).
// Block j < M: the norm of column j of Psi and of U Psi (FP32 is enough for an
// exponent); the other blocks: whether every initial gate is unitary to 1e-4.
// acc (zero before): the largest squared norms' bits, a not-unitary flag, and
// the finished blocks; the last block turns them into out.
__global__ void k_cl_scale(int N, int M, int gates, const double2* psi, const double2* phil, const double2* g, unsigned* acc,
                           int4* out) {
  const int tid = threadIdx.x, lane = tid & 31;
  if ((int)blockIdx.x < M) {
    float a = 0.f, b = 0.f;
    for (int i = tid; i < N; i += blockDim.x) {
      const double2 u = psi[(long long)i * M + blockIdx.x], v = phil[(long long)i * M + blockIdx.x];
      const float ux = (float)u.x, uy = (float)u.y, vx = (float)v.x, vy = (float)v.y;
      a = fmaf(ux, ux, fmaf(uy, uy, a));
      b = fmaf(vx, vx, fmaf(vy, vy, b));
    }
    __shared__ float s[2][32];
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) {
      a += __shfl_xor_sync(FULL, a, m);
      b += __shfl_xor_sync(FULL, b, m);
    }
    if (lane == 0) {
      s[0][tid >> 5] = a;
      s[1][tid >> 5] = b;
    }
    __syncthreads();
    if (tid == 0) {
      for (int w = 1; w < (int)blockDim.x / 32; ++w) {
        a += s[0][w];
        b += s[1][w];
      }
      atomicMax(acc, __float_as_uint(a));  // (norms are >= 0, and NaN is above every number)
      atomicMax(acc + 1, __float_as_uint(b));
    }
  } else {
    const int i = (blockIdx.x - M) * blockDim.x + tid;
    bool bad = false;
    if (i < gates) {
      float2 q[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const double2 z = g[(long long)i * 16 + j];
        q[j] = float2{(float)z.x, (float)z.y};
      }
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c <= r; ++c) {
          float2 t{0.f, 0.f};
#pragma unroll
          for (int j = 0; j < 4; ++j) t = cfma(q[4 * r + j], float2{q[4 * c + j].x, -q[4 * c + j].y}, t);
          bad |= !(fabsf(t.x - (r == c ? 1.f : 0.f)) < 1e-4f && fabsf(t.y) < 1e-4f);
        }
    }
    if (bad) atomicOr(acc + 2, 1u);
  }
  __shared__ unsigned last;
  __threadfence();
  __syncthreads();
  if (tid == 0) last = atomicAdd(acc + 3, 1u) == gridDim.x - 1;
  __syncthreads();
  if (last && tid == 0) {
    __threadfence();
    int e[2];
    bool range = true;
    for (int k = 0; k < 2; ++k) {
      const float n2 = __uint_as_float(atomicOr(acc + k, 0u));
      const bool ok = n2 > 1e-30f && n2 < 1e30f;
      range &= ok;
      // The least e with norm <= 1.001 2^e.
      e[k] = ok ? (int)ceilf(0.5f * log2f(n2) - 1.4e-3f) : 0;
    }
    *out = int4{!range ? kClPlainRange : atomicOr(acc + 2, 0u) != 0 ? kClPlainGates : 0, e[0], e[1], 0};
  }
}

cudaError_t launch_cl_scale(int n, int M, int gates, const double2* psi, const double2* phil, const double2* g, unsigned* acc,
                            int4* out, cudaStream_t st) {
  const cudaError_t e = cudaMemsetAsync(acc, 0, 4 * sizeof(unsigned), st);
  if (e != cudaSuccess) return e;
  const int nt = n >= 11 ? 1024 : 256;
  return launch_kernel(k_cl_scale, M + (gates + nt - 1) / nt, nt, 0, st, 1 << n, M, gates, psi, phil, g, acc, out);
}

ClPlan cl_plan(Real r, int n, int M, int L, int spt, bool keep64) {
  ClPlan best;
  if (n < 2 || L > kClMaxGates) return best;
  double best_t = 0.0;
  for (int C = 1; C <= kClMaxC && C <= M; ++C) {
    if ((M + C - 1) / C == (M + C - 2) / std::max(C - 1, 1) && C > 1) continue;  // no fewer columns than with C - 1
    const int nt = cl_threads(r, n, M, C);
    const size_t smem = cl_smem_bytes(r, n, M, L, C, nt, keep64);
    if (smem > (size_t)kMaxSmem || (r == R64 && (M + C - 1) / C > 16)) continue;
    const int at_once = cl_resident(r, nt, r == R64, C, smem);
    if (at_once < 1) continue;
    // Microseconds of a gate: update and exchange, then the slice's share of the pipes.
    const double entries = (double)(((size_t)(M + C - 1) / C) << n);
    const double work = entries * (r == R32 ? 0.34e-3 : 6.0e-3);
    const double fixed = (r == R32 ? 1.4 : 3.0) + (C > 1 ? 0.6 : 0.0) + (C > 8 ? 0.2 : 0.0);
    const int waves = (spt + at_once - 1) / at_once;
    const double t = waves * (fixed + work);
    // More than two rounds of complex64 starts of 1 MiB and more: their B
    // lists are in HBM and the dataflow sweep, which overlaps one start's
    // update with another's streaming, is the faster one (a sweep here and
    // there at n = 12, 17 gates, M = 32: 12 starts 207 us and 306, 16: 341 and
    // 344, 20: 408 and 362, 24, two rounds again: 406 and 399, 32: 606 and 458;
    // n = 11, 32 starts 185 and 296).  So it is where a second round of slices of
    // 16,384 entries is a third full or less (n = 9, M = 512: 6 starts 150 and 249,
    // 8: 294 and 272, 10: 294 and 291; 10 to 12 qubits alike).  It takes even M.
    const bool rounds = waves > 2 || (waves == 2 && entries >= 16384.0 && 3 * spt <= 4 * at_once);
    const bool large = r == R32 && rounds && ((size_t)M << n) >= ((size_t)1 << 17) && M % 2 == 0;
    if (best_t == 0.0 || t < best_t) {
      best_t = t;
      best.C = large ? 0 : C;
      best.threads = nt;
      best.smem = smem;
      // Fixed-point sums of E: over a CTA's columns (norm 1 each) below 2^62
      // with up to 4 of them, so more columns take a smaller scale; over all M
      // columns below 2^62 by a shift before the CTAs' sums are added.
      const int mc = (M + C - 1) / C;
      best.e_head = mc <= 4 ? 0 : mc <= 8 ? 1 : 2;
      best.e_shift = 0;
      while (M > (4 << (best.e_shift + best.e_head))) ++best.e_shift;
    }
  }
  return best;
}

cudaError_t launch_sweep_cl(Real r, const ClPlan& p, const ClArgs& a, bool fx, cudaStream_t st) {
  const ClKernel kernel = cl_kernel(r, p.threads, fx);
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
  if (e == cudaSuccess && p.C > 8) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(a.S * p.C));
  cfg.blockDim = dim3((unsigned)p.threads);
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)p.C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  ClArgs args = a;
  args.C = p.C;
  args.e_head = p.e_head;
  args.e_shift = p.e_shift;
  return cudaLaunchKernelEx(&cfg, kernel, args);
}

bool cl_check_fits(int n, int L) {
  return n >= 2 && L <= kClMaxGates && (((size_t)1 << n) + (size_t)L * 16) * sizeof(int4) <= (size_t)kMaxSmem;
}
cudaError_t launch_cl_check(const ClArgs& a, double* parts, unsigned* count, cudaStream_t st) {
  const size_t smem = (((size_t)1 << a.n) + (size_t)a.L * 16) * sizeof(int4);
  const bool wide = a.n >= 9;
  const auto kernel = wide ? k_cl_check<512> : k_cl_check<128>;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
  if (e != cudaSuccess) return e;
  return launch_kernel(kernel, a.M, wide ? 512 : 128, smem, st, a, parts, count);
}

}  // namespace qfs
