// One whole sweep (Section 3 of the paper) of every multistart as a single
// persistent, cooperative launch: a dataflow schedule instead of one launch
// per gate step.
//
// The sweep is a chain of steps per start: L-1 forward steps (B_k = g_k
// B_{k-1}), L backward steps (Phi_k = g_{k+1}^dagger Phi_{k+1}, environment of
// gate k from B_{k-1} and Phi_k, then the polar update of gate k) and, in
// complex64, the residual pass that gives the sample cost.  Steps of
// different starts are independent.  Every (step, start, chunk of rows) is a
// work item; items are numbered step-major, then start, then chunk, and
// handed out by one atomic counter.  An item waits (bounded) until its start
// has finished all earlier steps; the CTA that completes the last chunk of a
// backward step runs the gate update (one warp) and then publishes the step.
// Because items are taken in an order in which every dependency comes first
// and all CTAs are co-resident (cooperative launch), the smallest unfinished
// item can always proceed.  While one start waits for its update, the other
// starts' items keep the memory system busy, and no launch boundary, tail
// wave or idle update kernel sits between gate steps.
//
// Data written inside the launch (B list, Phi, gates, partial sums) is read
// back through L2 (ld.global.cg), never from a possibly stale L1 line.
// Every wait is bounded: when one runs out the CTA sets the run's error word
// and every CTA stops taking items; the host reports QFS_ETIMEOUT.
#include "polar_newton.cuh"
#include "qfs_common.cuh"
#include "qfs_kernels.h"

#include <algorithm>

namespace qfs {

namespace {

// One CTA per SM holding all the warps the registers allow (12 for complex64,
// 8 for complex128): an item is streamed by the whole SM, so the chunks of
// one start finish sooner than with several smaller CTAs sharing the SM.
template <typename T>
__host__ __device__ constexpr int df_threads() {
  return sizeof(T) == 4 ? 512 : 256;
}
constexpr int kDfMaxWarps = 16;

template <typename T, int VEC> struct DfV;
template <> struct DfV<float, 2> { using t = float4; };
template <> struct DfV<float, 1> { using t = float2; };
template <> struct DfV<double, 1> { using t = double2; };

template <typename T, int VEC>
__device__ __forceinline__ void ldg(const typename C2<T>::t* p, typename C2<T>::t (&o)[VEC]) {
  using V = typename DfV<T, VEC>::t;
  const V v = __ldcg(reinterpret_cast<const V*>(p));
  if constexpr (VEC == 2) {
    o[0] = float2{v.x, v.y};
    o[1] = float2{v.z, v.w};
  } else {
    o[0] = v;
  }
}
template <typename T, int VEC>
__device__ __forceinline__ void stg(typename C2<T>::t* p, const typename C2<T>::t (&o)[VEC]) {
  using V = typename DfV<T, VEC>::t;
  if constexpr (VEC == 2) {
    __stcg(reinterpret_cast<V*>(p), V{o[0].x, o[0].y, o[1].x, o[1].y});
  } else {
    __stcg(reinterpret_cast<V*>(p), o[0]);
  }
}

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_u32(unsigned* p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_volatile_i32(const int* p) { return *reinterpret_cast<const volatile int*>(p); }

template <typename T>
struct DfShared {
  typename C2<T>::t gs[16];
  typename C2<T>::t gs2[16];  // the second gate of a two-gate forward step
  double red[kDfMaxWarps][32];
  NewtonSh nw;
  long long item;
  int flag;
};

// Block-wide sum of 32 per-thread values (one per lane slot) into
// partials[slot * 32 + lane] by warp 0.
template <typename T, typename PT>
__device__ __forceinline__ void block_partials32(double mine, DfShared<T>& sh, PT* out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  sh.red[warp][lane] = mine;
  __syncthreads();
  if (warp == 0) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < df_threads<T>() / 32; ++w) t += sh.red[w][lane];
    __stcg(out + lane, (PT)t);
  }
}

// Start s's input and Phi input: per-start stride, plus a per-target stride
// for the arrays one per target (Psi, U Psi) when several targets share the
// launch (start s belongs to target s / spt).
template <typename T2>
__device__ __forceinline__ const T2* df_in(const DfStep& st, int s) {
  return reinterpret_cast<const T2*>(st.in) + s * st.in_stride + (long long)(s / st.spt) * st.in_gstride;
}
template <typename T2>
__device__ __forceinline__ const T2* df_phi_in(const DfStep& st, int s) {
  return reinterpret_cast<const T2*>(st.phi_in) + s * st.phi_in_stride + (long long)(s / st.spt) * st.phi_in_gstride;
}

// Entry i of a gate of start s, or of its adjoint.
template <typename T2>
__device__ __forceinline__ T2 gate_entry(const DfStep& st, const void* gate, int s, int i) {
  const T2 g = __ldcg(reinterpret_cast<const T2*>(gate) + s * st.gate_stride + (st.adj ? 4 * (i & 3) + (i >> 2) : i));
  return T2{g.x, st.adj ? -g.y : g.y};
}
// Gate of this start (16 complex) into shared memory.
template <typename T>
__device__ __forceinline__ void load_gate(const DfStep& st, int s, DfShared<T>& sh) {
  using T2 = typename C2<T>::t;
  if (threadIdx.x < 16) sh.gs[threadIdx.x] = st.gate ? gate_entry<T2>(st, st.gate, s, threadIdx.x) : T2{};
  __syncthreads();
}

// Forward rows of one chunk: Y = (g (x) I) X on the pair of st.fg.
template <typename T, int VEC>
__device__ void df_forward(const DfStep& st, int s, int c, DfShared<T>& sh) {
  using T2 = typename C2<T>::t;
  load_gate<T>(st, s, sh);
  T2 gr[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) gr[i] = sh.gs[i];
  const T2* X = df_in<T2>(st, s);
  T2* Y = reinterpret_cast<T2*>(st.out) + s * st.fg.sN;
  const int MV = st.fg.M / VEC;
  const int u0 = c * st.chunk, u1 = min(u0 + st.chunk, st.units);
  auto offsets = [&](int u, uint32_t (&off)[4]) {
    const int r = u / MV, jv = u - r * MV;
    const uint32_t base = insert_two_zero_bits((uint32_t)r, st.fg.lo, st.fg.hi);
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const uint32_t row = base | ((uint32_t)(x >> 1) << st.fg.pos_a) | ((uint32_t)(x & 1) << st.fg.pos_b);
      off[x] = row * (uint32_t)st.fg.M + (uint32_t)jv * VEC;
    }
  };
  auto apply = [&](const T2 (&v)[4][VEC], const uint32_t (&off)[4]) {
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      T2 o[VEC];
#pragma unroll
      for (int q = 0; q < VEC; ++q) {
        T2 acc = cmul(gr[4 * x], v[0][q]);
#pragma unroll
        for (int xp = 1; xp < 4; ++xp) acc = cfma(gr[4 * x + xp], v[xp][q], acc);
        o[q] = acc;
      }
      stg<T, VEC>(Y + off[x], o);
    }
  };
  // Two units per thread per round: eight loads in flight.
  constexpr int NT = df_threads<T>();
  int u = u0 + threadIdx.x;
  for (; u + NT < u1; u += 2 * NT) {
    uint32_t oa[4], ob[4];
    offsets(u, oa);
    offsets(u + NT, ob);
    T2 va[4][VEC], vb[4][VEC];
#pragma unroll
    for (int x = 0; x < 4; ++x) ldg<T, VEC>(X + oa[x], va[x]);
#pragma unroll
    for (int x = 0; x < 4; ++x) ldg<T, VEC>(X + ob[x], vb[x]);
    apply(va, oa);
    apply(vb, ob);
  }
  if (u < u1) {
    uint32_t oa[4];
    offsets(u, oa);
    T2 va[4][VEC];
#pragma unroll
    for (int x = 0; x < 4; ++x) ldg<T, VEC>(X + oa[x], va[x]);
    apply(va, oa);
  }
}

// Asynchronous 16-byte copies global -> shared (L2 only), in groups.
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)),
               "l"(gmem)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Stages of the backward step's copy pipeline.  Each thread copies the
// sixteen bytes it will itself consume (eight rows of its unit: four of Phi,
// four of B) into its own slots of a stage, so completion needs only the
// thread's own cp.async.wait_group, never a block barrier; with kDfStages
// stages, kDfStages - 1 rounds of loads are in flight per thread while one
// round is computed, held in shared memory instead of registers.  Slot
// (stage, row j, thread t) sits at ((stage * 8 + j) * threads + t) * 16
// bytes: a warp reads 512 contiguous bytes, free of bank conflicts.
constexpr int kDfStages = 3;
template <typename T>
__host__ __device__ constexpr int df_stage_bytes() {
  return kDfStages * 8 * df_threads<T>() * 16;
}

// Two forward steps in one pass over 16-row units (gates k and k+1 on four
// distinct qubits; geometry bg with gate k's pair on local bits 3, 2 and
// gate k+1's on local bits 1, 0): B_k = g_k B_{k-1}, stored where something
// reads it, and B_{k+1} = g_{k+1} B_k.  The same step with the adjoints of two
// updated gates carries Phi past both, in place.  Four lanes share a unit: lane
// quarter qx holds the four rows of one value of gate k+1's bits and applies
// g_k to them; after a transpose over the four lanes it applies g_{k+1}.  (Sixteen
// shuffles a round; fetching every row where it is used took 64, and 16 warps
// of those were the step's bound: 11.9 us an item of 420 KB.)  Rows
// are staged by cp.async into the thread's own slots (kDfFwd2Stages - 1
// rounds in flight).
constexpr int kDfFwd2Stages = 4;
template <typename T, int VEC>
__device__ void df_forward2(const DfStep& st, int s, int c, DfShared<T>& sh, uint4* stage) {
  using T2 = typename C2<T>::t;
  static_assert(sizeof(T2) * VEC == 16, "one 16-byte slot per row");
  static_assert(kDfFwd2Stages * 4 <= kDfStages * 8, "forward stages fit the stage buffer");
  constexpr int NT = df_threads<T>();
  constexpr int NW = NT / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int qx = lane >> 3, v = lane & 7;
  if (threadIdx.x < 16) sh.gs[threadIdx.x] = gate_entry<T2>(st, st.gate, s, threadIdx.x);
  else if (threadIdx.x < 32) sh.gs2[threadIdx.x - 16] = gate_entry<T2>(st, st.gate2, s, threadIdx.x - 16);
  __syncthreads();
  T2 g1[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) g1[i] = sh.gs[i];
  const T2* X = df_in<T2>(st, s);
  T2* Y1 = reinterpret_cast<T2*>(st.out) + s * st.bg.sN;
  T2* Y2 = reinterpret_cast<T2*>(st.out2) + s * st.bg.sN;
  const uint32_t M = (uint32_t)st.bg.M;
  const uint32_t d0 = (1u << st.bg.pos[0]) * M, d1 = (1u << st.bg.pos[1]) * M;
  const uint32_t d2 = (1u << st.bg.pos[2]) * M, d3 = (1u << st.bg.pos[3]) * M;
  const uint32_t xoff = ((qx >> 1) ? d1 : 0u) + ((qx & 1) ? d0 : 0u);
  const uint32_t joff[4] = {0u, d2, d3, d3 + d2};  // j = 2 bit(local 3) + bit(local 2): gate k's index
  const int MV = st.bg.M / VEC;
  const int u0 = c * st.chunk, u1 = min(u0 + st.chunk, st.units);
  constexpr int per_round = 8 * NW;
  const int rounds = (u1 - u0 + per_round - 1) / per_round;
  auto unit_off = [&](int u) {
    const int r = u / MV, jv = u - r * MV;
    uint32_t base = (uint32_t)r;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int p = st.bg.ins[i];
      base = ((base >> p) << (p + 1)) | (base & ((1u << p) - 1u));
    }
    return base * M + (uint32_t)jv * VEC + xoff;
  };
  auto issue = [&](int rd) {
    const int u = u0 + rd * per_round + warp * 8 + v;
    if (rd < rounds && u < u1) {
      uint4* slot = stage + (size_t)((rd % kDfFwd2Stages) * 4) * NT + threadIdx.x;
      const uint32_t o = unit_off(u);
#pragma unroll
      for (int j = 0; j < 4; ++j) cp_async16(slot + (size_t)j * NT, X + o + joff[j]);
    }
    cp_async_commit();
  };
#pragma unroll
  for (int rd = 0; rd < kDfFwd2Stages - 1; ++rd) issue(rd);
  for (int rd = 0; rd < rounds; ++rd) {
    issue(rd + kDfFwd2Stages - 1);
    cp_async_wait<kDfFwd2Stages - 1>();
    const int u = u0 + rd * per_round + warp * 8 + v;
    const bool valid = u < u1;  // (all four lanes of a unit agree)
    T2 b[4][VEC];
    {
      const uint4* slot = stage + (size_t)((rd % kDfFwd2Stages) * 4) * NT + threadIdx.x;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        uint4 w4 = valid ? slot[(size_t)j * NT] : make_uint4(0u, 0u, 0u, 0u);
        const T2* e = reinterpret_cast<const T2*>(&w4);
#pragma unroll
        for (int q = 0; q < VEC; ++q) b[j][q] = e[q];
      }
    }
    const uint32_t o = valid ? unit_off(u) : 0u;
    T2 y[4][VEC];
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int q = 0; q < VEC; ++q) {
        T2 acc = cmul(g1[4 * x], b[0][q]);
#pragma unroll
        for (int xp = 1; xp < 4; ++xp) acc = cfma(g1[4 * x + xp], b[xp][q], acc);
        y[x][q] = acc;
      }
    if (valid && st.out != nullptr) {
#pragma unroll
      for (int x = 0; x < 4; ++x) stg<T, VEC>(Y1 + o + joff[x], y[x]);
    }
    // The quarters' rows change places (4 x 4 transpose of 16-byte entries over
    // the unit's four lanes, two exchanges): lane qx then holds row qx of gate
    // k's index for all four of gate k+1's.
    auto swap = [&](T2 (&p)[VEC], T2 (&q)[VEC], bool upper, int m) {
#pragma unroll
      for (int e = 0; e < VEC; ++e) {
        const T2 send = upper ? p[e] : q[e];
        const T2 got{__shfl_xor_sync(FULL, send.x, m), __shfl_xor_sync(FULL, send.y, m)};
        if (upper) p[e] = got;
        else q[e] = got;
      }
    };
    swap(y[0], y[1], qx & 1, 8);
    swap(y[2], y[3], qx & 1, 8);
    swap(y[0], y[2], qx >> 1, 16);
    swap(y[1], y[3], qx >> 1, 16);
    // z = g_{k+1} y, summed in the order of the one-gate forward step.
    const uint32_t oz = o - xoff + ((qx >> 1) ? d3 : 0u) + ((qx & 1) ? d2 : 0u);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      T2 z[VEC];
#pragma unroll
      for (int q = 0; q < VEC; ++q) {
        T2 acc = cmul(sh.gs2[4 * r], y[0][q]);
#pragma unroll
        for (int xp = 1; xp < 4; ++xp) acc = cfma(sh.gs2[4 * r + xp], y[xp][q], acc);
        z[q] = acc;
      }
      if (valid) stg<T, VEC>(Y2 + oz + ((r >> 1) ? d1 : 0u) + ((r & 1) ? d0 : 0u), z);
    }
  }
  cp_async_wait<0>();
}

// Backward step on 16-row units (gate k+1 and gate k on four distinct
// qubits): four lanes share a unit as in the per-step kernel; the partial
// sums of E_k go to partials slot (s, c).
template <typename T, int VEC>
__device__ void df_backward_q4(const DfStep& st, int s, int c, DfShared<T>& sh, T* part, uint4* stage) {
  using T2 = typename C2<T>::t;
  static_assert(sizeof(T2) * VEC == 16, "one 16-byte slot per row");
  constexpr int NT = df_threads<T>();
  constexpr int NW = NT / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int qx = lane >> 3, v = lane & 7;
  load_gate<T>(st, s, sh);
  T2 gd[16];
#pragma unroll
  for (int y = 0; y < 4; ++y)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const T2 t = sh.gs[4 * j + y];
      gd[4 * y + j] = T2{t.x, -t.y};
    }
  const T2* B = df_in<T2>(st, s);
  const T2* P = df_phi_in<T2>(st, s);
  T2* Po = reinterpret_cast<T2*>(st.phi_out) + s * st.bg.sN;
  const uint32_t M = (uint32_t)st.bg.M;
  const uint32_t d0 = (1u << st.bg.pos[0]) * M, d1 = (1u << st.bg.pos[1]) * M;
  const uint32_t d2 = (1u << st.bg.pos[2]) * M, d3 = (1u << st.bg.pos[3]) * M;
  const uint32_t xoff = ((qx >> 1) ? d1 : 0u) + ((qx & 1) ? d0 : 0u);
  const uint32_t joff[4] = {0u, d2, d3, d3 + d2};
  T acc[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = T(0);
  const int MV = st.bg.M / VEC;
  const int u0 = c * st.chunk, u1 = min(u0 + st.chunk, st.units);
  constexpr int per_round = 8 * NW;  // units of one round (eight per warp)
  const int rounds = (u1 - u0 + per_round - 1) / per_round;
  auto unit_off = [&](int u) {
    const int r = u / MV, jv = u - r * MV;
    uint32_t base = (uint32_t)r;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int p = st.bg.ins[i];
      base = ((base >> p) << (p + 1)) | (base & ((1u << p) - 1u));
    }
    return base * M + (uint32_t)jv * VEC + xoff;
  };
  auto issue = [&](int rd) {
    const int u = u0 + rd * per_round + warp * 8 + v;
    if (rd < rounds && u < u1) {
      uint4* slot = stage + (size_t)((rd % kDfStages) * 8) * NT + threadIdx.x;
      const uint32_t o = unit_off(u);
#pragma unroll
      for (int j = 0; j < 4; ++j) cp_async16(slot + (size_t)j * NT, P + o + joff[j]);
#pragma unroll
      for (int j = 0; j < 4; ++j) cp_async16(slot + (size_t)(4 + j) * NT, B + o + joff[j]);
    }
    cp_async_commit();  // (an empty group keeps the group count uniform)
  };
#pragma unroll
  for (int rd = 0; rd < kDfStages - 1; ++rd) issue(rd);
  for (int rd = 0; rd < rounds; ++rd) {
    issue(rd + kDfStages - 1);
    cp_async_wait<kDfStages - 1>();  // this thread's copies of round rd have landed
    const int u = u0 + rd * per_round + warp * 8 + v;
    const bool valid = u < u1;
    T2 ph[4][VEC], b[4][VEC];
    {
      const uint4* slot = stage + (size_t)((rd % kDfStages) * 8) * NT + threadIdx.x;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        uint4 w4 = valid ? slot[(size_t)j * NT] : make_uint4(0u, 0u, 0u, 0u);
        const T2* e = reinterpret_cast<const T2*>(&w4);
#pragma unroll
        for (int q = 0; q < VEC; ++q) {
          if (j < 4) ph[j][q] = e[q];
          else b[j - 4][q] = e[q];
        }
      }
    }
    const uint32_t base_off = valid ? unit_off(u) : 0u;
    {
      T2 nw[4][VEC];
#pragma unroll
      for (int y = 0; y < 4; ++y)
#pragma unroll
        for (int q = 0; q < VEC; ++q) {
          T2 t = cmul(gd[4 * y], ph[0][q]);
#pragma unroll
          for (int j = 1; j < 4; ++j) t = cfma(gd[4 * y + j], ph[j][q], t);
          nw[y][q] = t;
        }
#pragma unroll
      for (int y = 0; y < 4; ++y)
#pragma unroll
        for (int q = 0; q < VEC; ++q) ph[y][q] = nw[y][q];
      if (valid) {
#pragma unroll
        for (int y = 0; y < 4; ++y) stg<T, VEC>(Po + base_off + joff[y], ph[y]);
      }
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < VEC; ++q) {
          T2 pp = ph[j][q];
          if (m) {
            pp.x = __shfl_xor_sync(FULL, pp.x, 8 * m);
            pp.y = __shfl_xor_sync(FULL, pp.y, 8 * m);
          }
          cfma_conj(acc[2 * m], acc[2 * m + 1], b[j][q], pp);
        }
    }
  }
  cp_async_wait<0>();
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    acc[i] += __shfl_xor_sync(FULL, acc[i], 1);
    acc[i] += __shfl_xor_sync(FULL, acc[i], 2);
    acc[i] += __shfl_xor_sync(FULL, acc[i], 4);
  }
  // Lane (x, 0) holds E[x][x^m]; gather them into lane slots 2(4x+y)+{0,1}.
  if (v == 0) {
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int e = 4 * qx + (qx ^ m);
      sh.red[warp][2 * e] = (double)acc[2 * m];
      sh.red[warp][2 * e + 1] = (double)acc[2 * m + 1];
    }
  }
  __syncthreads();
  if (warp == 0) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < NW; ++w) t += sh.red[w][lane];
    __stcg(part + lane, (T)t);
  }
}

template <int U, int EA, int EB>
__device__ __forceinline__ constexpr int df_spread_rest(int j) {
  int t = 0, bit = 0;
  for (int i = 0; i < U; ++i) {
    if (i == EA || i == EB) continue;
    t |= ((j >> bit) & 1) << i;
    ++bit;
  }
  return t;
}

// Backward step on 2^U-row units, one unit per thread (U = 2 or 3), or the
// residual pass (MODE 1: sum |g^dagger Phi - B|^2 into a double partial).
template <typename T, int VEC, int MODE, int U, int EA, int EB>
__device__ void df_backward_gen(const DfStep& st, int s, int c, DfShared<T>& sh, void* part) {
  using T2 = typename C2<T>::t;
  constexpr int ROWS = 1 << U;
  const int lane = threadIdx.x & 31;
  load_gate<T>(st, s, sh);
  const bool has_gate = st.gate != nullptr;
  auto gd = [&](int y, int yp) {
    const T2 t = sh.gs[4 * yp + y];
    return T2{t.x, -t.y};
  };
  const T2* B = df_in<T2>(st, s);
  const T2* P = df_phi_in<T2>(st, s);
  T2* Po = st.phi_out ? reinterpret_cast<T2*>(st.phi_out) + s * st.bg.sN : nullptr;
  const uint32_t M = (uint32_t)st.bg.M;
  uint32_t dpos[U];
#pragma unroll
  for (int i = 0; i < U; ++i) dpos[i] = (1u << st.bg.pos[i]) * M;
  T acc[MODE == 0 ? 32 : 1];
#pragma unroll
  for (int i = 0; i < (MODE == 0 ? 32 : 1); ++i) acc[i] = T(0);
  const int MV = st.bg.M / VEC;
  const int u0 = c * st.chunk, u1 = min(u0 + st.chunk, st.units);
  for (int u = u0 + threadIdx.x; u < u1; u += df_threads<T>()) {
    const int r = u / MV, jv = u - r * MV;
    uint32_t base = (uint32_t)r;
#pragma unroll
    for (int i = 0; i < U; ++i) {
      const int p = st.bg.ins[i];
      base = ((base >> p) << (p + 1)) | (base & ((1u << p) - 1u));
    }
    const uint32_t base_off = base * M + (uint32_t)jv * VEC;
    auto off = [&](int t) {
      uint32_t o = base_off;
#pragma unroll
      for (int i = 0; i < U; ++i)
        if ((t >> i) & 1) o += dpos[i];
      return o;
    };
    T2 ph[ROWS][VEC];
#pragma unroll
    for (int t = 0; t < ROWS; ++t) ldg<T, VEC>(P + off(t), ph[t]);
    if (has_gate) {
#pragma unroll
      for (int t0 = 0; t0 < ROWS / 4; ++t0) {
        T2 nw[4][VEC];
#pragma unroll
        for (int y = 0; y < 4; ++y)
#pragma unroll
          for (int q = 0; q < VEC; ++q) {
            T2 a2 = cmul(gd(y, 0), ph[(0 << (U - 2)) | t0][q]);
#pragma unroll
            for (int yp = 1; yp < 4; ++yp) a2 = cfma(gd(y, yp), ph[(yp << (U - 2)) | t0][q], a2);
            nw[y][q] = a2;
          }
#pragma unroll
        for (int y = 0; y < 4; ++y)
#pragma unroll
          for (int q = 0; q < VEC; ++q) ph[(y << (U - 2)) | t0][q] = nw[y][q];
      }
      if (Po) {
#pragma unroll
        for (int t = 0; t < ROWS; ++t) stg<T, VEC>(Po + off(t), ph[t]);
      }
    }
    if constexpr (MODE == 0) {
#pragma unroll
      for (int j = 0; j < ROWS / 4; ++j) {
        const int rest = df_spread_rest<U, EA, EB>(j);
        T2 b[4][VEC];
#pragma unroll
        for (int x = 0; x < 4; ++x) ldg<T, VEC>(B + off(rest | ((x >> 1) << EA) | ((x & 1) << EB)), b[x]);
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int y = 0; y < 4; ++y) {
            const int ty = rest | ((y >> 1) << EA) | ((y & 1) << EB);
#pragma unroll
            for (int q = 0; q < VEC; ++q) {
              cfma_conj(acc[2 * (4 * x + y)], acc[2 * (4 * x + y) + 1], b[x][q], ph[ty][q]);
            }
          }
      }
    } else {
#pragma unroll
      for (int t = 0; t < ROWS; ++t) {
        T2 b[VEC];
        ldg<T, VEC>(B + off(t), b);
#pragma unroll
        for (int q = 0; q < VEC; ++q) {
          const T dx = ph[t][q].x - b[q].x, dy = ph[t][q].y - b[q].y;
          acc[0] = fmat(dx, dx, fmat(dy, dy, acc[0]));
        }
      }
    }
  }
  if constexpr (MODE == 0) {
    const double mine = (double)warp_reduce_scatter32<T>(acc, lane);
    block_partials32<T, T>(mine, sh, reinterpret_cast<T*>(part));
  } else {
    double v = (double)acc[0];
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) v += __shfl_xor_sync(FULL, v, m);
    block_partials32<T, double>(lane == 0 ? v : 0.0, sh, reinterpret_cast<double*>(part));
  }
}

// Environments of two gates on four distinct qubits in one pass (complex64):
// F[x][y] = sum B[x] conj(Phi[y]) over the 16 x 16 row pairs of a unit, B the
// state before both gates, Phi carried past everything behind them.  Both 4x4
// environments, the second one with the first gate already updated, are sums
// over F with the other gate (df_update_pair), so B and Phi are read once for
// two gates where a step per gate reads B, reads Phi and writes Phi twice:
// 6 N M s bytes a pair of gates with its forward step and Phi's, against 9.  At
// n = 12, M = 32, 32 starts: 491 -> 477 us a sweep (461 with the transposed forward
// step); what is left is issue-bound, 9.8 us an item of 512 units at 256 FMAs a
// thread and round, not bound by the bytes.
//
// The price is arithmetic, 16 complex FMAs per entry instead of 8, so F is
// formed as a small matrix product: a tile of 16 rows x 64 columns' pairs of B
// and Phi in shared memory (cp.async, kEnvStages deep, rows padded by 32 bytes
// so that the four rows of an access lie in different banks), 16 threads per
// 16 x 16 block with 4 x 4 entries each: 128 FMAs per eight 16-byte reads.
constexpr int kEnvStages = 4, kEnvCols = 64, kEnvRow = kEnvCols * 16 + 32, kEnvStage = 32 * kEnvRow;
static_assert(kEnvStages * kEnvStage <= df_stage_bytes<float>(), "environment stages fit the stage buffer");
static_assert(16 * 512 * 4 + 2 * 512 * 4 <= df_stage_bytes<float>(), "and its sums");

__device__ __forceinline__ void cp_async16_zero(void* smem, const void* gmem, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem),
               "r"(valid ? 16 : 0)
               : "memory");
}

__device__ void df_env16(const DfStep& st, int s, int c, float* part, unsigned char* stage) {
  constexpr int NT = df_threads<float>();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float2* B = df_in<float2>(st, s);
  const float2* P = df_phi_in<float2>(st, s);
  const uint32_t M = (uint32_t)st.bg.M;
  const int MV = st.bg.M / 2;
  const int u0 = c * st.chunk, u1 = min(u0 + st.chunk, st.units);
  const int rounds = (u1 - u0 + kEnvCols - 1) / kEnvCols;
  // Copies: this thread's column pair and four rows, two of B and two of Phi.
  const int col = tid & (kEnvCols - 1), rg = tid >> 6;
  auto row_off = [&](int t) {
    return ((((uint32_t)t & 1u) << st.bg.pos[0]) | (((uint32_t)t >> 1 & 1u) << st.bg.pos[1]) |
            (((uint32_t)t >> 2 & 1u) << st.bg.pos[2]) | (((uint32_t)t >> 3 & 1u) << st.bg.pos[3])) * M;
  };
  const uint32_t ra = row_off(rg), rb = row_off(rg + 8);
  auto issue = [&](int rd) {
    if (rd < rounds) {
      const int u = u0 + rd * kEnvCols + col;
      const bool valid = u < u1;
      const int r = (valid ? u : u0) / MV, jv = (valid ? u : u0) - r * MV;
      uint32_t base = (uint32_t)r;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int p = st.bg.ins[i];
        base = ((base >> p) << (p + 1)) | (base & ((1u << p) - 1u));
      }
      const uint32_t o = base * M + (uint32_t)jv * 2;
      unsigned char* d = stage + (rd % kEnvStages) * kEnvStage + col * 16;
      cp_async16_zero(d + rg * kEnvRow, B + o + ra, valid);
      cp_async16_zero(d + (rg + 8) * kEnvRow, B + o + rb, valid);
      cp_async16_zero(d + (rg + 16) * kEnvRow, P + o + ra, valid);
      cp_async16_zero(d + (rg + 24) * kEnvRow, P + o + rb, valid);
    }
    cp_async_commit();
  };
  // Sums: entries F[4 r + i][4 q + j].
  const int i = tid & 3, j = (tid >> 2) & 3, g = tid >> 4;
  float acc[4][4][2];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[r][q][0] = acc[r][q][1] = 0.f;
  __syncthreads();  // (the stages may still be read as another step's)
#pragma unroll
  for (int rd = 0; rd < kEnvStages - 1; ++rd) issue(rd);
  for (int rd = 0; rd < rounds; ++rd) {
    cp_async_wait<kEnvStages - 2>();
    __syncthreads();  // round rd is there for everybody, round rd - 1 is read
    issue(rd + kEnvStages - 1);
    const unsigned char* d = stage + (rd % kEnvStages) * kEnvStage;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const unsigned char* e = d + (h * 32 + g) * 16;
      float4 b[4], p[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) b[r] = *reinterpret_cast<const float4*>(e + (4 * r + i) * kEnvRow);
#pragma unroll
      for (int q = 0; q < 4; ++q) p[q] = *reinterpret_cast<const float4*>(e + (16 + 4 * q + j) * kEnvRow);
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          cfma_conj(acc[r][q][0], acc[r][q][1], float2{b[r].x, b[r].y}, float2{p[q].x, p[q].y});
          cfma_conj(acc[r][q][0], acc[r][q][1], float2{b[r].z, b[r].w}, float2{p[q].z, p[q].w});
        }
    }
  }
  cp_async_wait<0>();
  // The warp's two groups, then the warps (TwoSum, fixed order).
  float* buf = reinterpret_cast<float*>(stage);
  __syncthreads();
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float re = acc[r][q][0] + __shfl_xor_sync(FULL, acc[r][q][0], 16);
      const float im = acc[r][q][1] + __shfl_xor_sync(FULL, acc[r][q][1], 16);
      if (lane < 16) *reinterpret_cast<float2*>(buf + warp * 512 + 2 * ((4 * r + i) * 16 + 4 * q + j)) = float2{re, im};
    }
  __syncthreads();
  float hi = 0.f, lo = 0.f;
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) {
    float t;
    two_sum(hi, buf[w * 512 + tid], hi, t);
    lo += t;
  }
  __stcg(part + tid, hi + lo);
}

// The update of gate k for start s by warp 0 (polar_newton.cuh) from the summed
// environment, whose value j is in lane j: hi + lo (complex64 sweeps) or e.
template <typename T>
__device__ void df_update(const UpdateArgs& ua, int s, DfShared<T>& sh, float hi, float lo, double e, float2* keep = nullptr) {
  constexpr bool F32 = sizeof(T) == 4;
  const int lane = threadIdx.x & 31, l16 = lane & 15, at = 4 * (l16 & 3) + (l16 >> 2);
  double2* g64 = ua.g64 + s * ua.g_stride;
  const bool damp = ua.beta != 0.0;
  auto env = [&]() { return newton_env(F32 ? (double)hi + (double)lo : e); };
  auto matrix = [&]() { return damp ? newton_damp(env(), ua.beta, g64) : env(); };
  const float2 a32 = F32 && !damp ? newton_input32(hi) : newton_input64(matrix(), sh.nw);
  long long q;
  const double2 p = newton_update<!F32>(a32, sh.nw, newton_pair(), q) ? newton_entry64(q) : newton_fallback(matrix(), sh.nw);
  if (lane < 16) {
    g64[at] = p;
    const float2 pf{(float)p.x, (float)p.y};
    if (ua.g32) (ua.g32 + s * ua.g_stride)[at] = pf;
    if (keep) keep[at] = pf;
  }
  if (ua.env_out) {
    const double2 m = env();
    if (lane < 16) ua.env_out[s * ua.env_stride + l16] = m;
  }
  if (ua.cost_out) {
    const double2 m = env();
    double t = lane < 16 ? (p.x * m.x - p.y * m.y) : 0.0;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) t += __shfl_xor_sync(FULL, t, o);
    if (lane == 0) ua.cost_out[s] = 2.0 - 2.0 * ua.inv_M * t;
  }
}

// The two updates behind df_env16, by warp 0: F (hi + lo, 16 x 16 complex) in
// shared memory, gate k on the upper index pair of x = 4 xa + xb, gate k - 1 on
// the lower.  E_k[xa][ya] = sum g_{k-1}[z][xb] F[xa xb][ya z] with the old gate
// k - 1 (it makes B_{k-1} of B_{k-2}), E_{k-1}[xb][yb] = sum g_k[ya][z]
// F[z xb][ya yb] with the new gate k (its adjoint makes Phi_{k-1} of Phi_k).
__device__ void df_update_pair(const UpdateArgs& up, const UpdateArgs& lower, int s, DfShared<float>& sh, const float2* fh,
                               const float2* fl) {
  const int lane = threadIdx.x & 31, x = lane >> 3, y = (lane >> 1) & 3, im = lane & 1;
  if (lane < 16) sh.gs[lane] = __ldcg(lower.g32 + s * lower.g_stride + lane);
  __syncwarp();
  auto term = [&](float2 g, float2 f, float& acc) {  // component im of g f
    acc = fmaf(g.x, im ? f.y : f.x, acc);
    acc = fmaf(im ? g.y : -g.y, im ? f.x : f.y, acc);
  };
  float a = 0.f, b = 0.f, l = 0.f, hi, lo;
#pragma unroll
  for (int z = 0; z < 4; ++z)
#pragma unroll
    for (int xb = 0; xb < 4; ++xb) {
      const int at = (4 * x + xb) * 16 + 4 * y + z;
      term(sh.gs[4 * z + xb], fh[at], (xb & 1) ? b : a);
      term(sh.gs[4 * z + xb], fl[at], l);
    }
  two_sum(a, b, hi, lo);
  df_update<float>(up, s, sh, hi, lo + l, 0.0, sh.gs2);
  __syncwarp();
  a = b = l = 0.f;
#pragma unroll
  for (int z = 0; z < 4; ++z)
#pragma unroll
    for (int ya = 0; ya < 4; ++ya) {
      const int at = (4 * z + x) * 16 + 4 * ya + y;
      term(sh.gs2[4 * ya + z], fh[at], (ya & 1) ? b : a);
      term(sh.gs2[4 * ya + z], fl[at], l);
    }
  two_sum(a, b, hi, lo);
  df_update<float>(lower, s, sh, hi, lo + l, 0.0);
}

// Partial-sum slots: start s owns slots s * stride .. s * stride + stride - 1
// (stride = the most chunks of any step), so starts that are at different
// steps, with different chunk counts, never share a slot.
template <typename T>
__device__ void df_process(const DfStep& st, int s, int c, DfShared<T>& sh, void* partials, double* resid,
                           int stride, int len, uint4* stage) {
  constexpr int V2 = sizeof(T) == 4 ? 2 : 1;  // samples per thread for 4- and 16-row units
  T* part = reinterpret_cast<T*>(partials) + ((long long)s * stride + c) * len;
  double* part64 = resid + ((long long)s * stride + c) * 32;
  switch (st.kind) {
    case DF_FWD: df_forward<T, V2>(st, s, c, sh); break;
    case DF_FWD2: df_forward2<T, V2>(st, s, c, sh, stage); break;
    case DF_BWD4: df_backward_q4<T, V2>(st, s, c, sh, part, stage); break;
    case DF_BWD2_10: df_backward_gen<T, V2, 0, 2, 1, 0>(st, s, c, sh, part); break;
    case DF_BWD2_01: df_backward_gen<T, V2, 0, 2, 0, 1>(st, s, c, sh, part); break;
    case DF_BWD3_20: df_backward_gen<T, 1, 0, 3, 2, 0>(st, s, c, sh, part); break;
    case DF_BWD3_02: df_backward_gen<T, 1, 0, 3, 0, 2>(st, s, c, sh, part); break;
    case DF_BWD3_10: df_backward_gen<T, 1, 0, 3, 1, 0>(st, s, c, sh, part); break;
    case DF_BWD3_01: df_backward_gen<T, 1, 0, 3, 0, 1>(st, s, c, sh, part); break;
    case DF_RESID: df_backward_gen<T, V2, 1, 2, 1, 0>(st, s, c, sh, part64); break;
    case DF_ENV16:
      if constexpr (sizeof(T) == 4) df_env16(st, s, c, part, reinterpret_cast<unsigned char*>(stage));
      break;
    default: break;
  }
}

}  // namespace

template <typename T>
__global__ void __launch_bounds__(df_threads<T>(), 1) k_sweep_df(DfArgs a) {
  __shared__ DfShared<T> sh;
  extern __shared__ __align__(16) uint4 df_stage[];  // df_stage_bytes<T>() of copy stages
  constexpr int NW = df_threads<T>() / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // Thread 0 takes the next item when the CTA is free (a reservation held
  // while the current item runs would delay that item by a whole item).
  // A CTA's items increase, so the step search resumes where it stopped.
  // The next sweep's control words (a slot this sweep does not use).
  if (a.zero_next != nullptr)
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < a.zero_count; k += gridDim.x * blockDim.x)
      a.zero_next[k] = 0u;
  // A sweep queued behind one that met the tolerance does nothing.
  if (a.stop != nullptr && ld_volatile_i32(a.stop)) return;
  int i = 0;
  for (;;) {
    if (threadIdx.x == 0) {
      long long w = -1;
      if (!ld_volatile_i32(a.err)) {
        const unsigned x = atomicAdd(a.queue, 1u);
        if ((long long)x < a.total_items) w = x;
      }
      sh.item = w;
    }
    __syncthreads();
    const long long w = sh.item;
    if (w < 0) return;
    while (i + 1 < a.nsteps && a.steps[i + 1].item0 <= w) ++i;
    const DfStep& st = a.steps[i];
    const int rel = (int)(w - st.item0);
    const int s = rel / st.nchunk, c = rel - s * st.nchunk;
    unsigned long long* itr = a.item_trace ? a.item_trace + w * 4 : nullptr;
    if (itr && threadIdx.x == 0) {
      itr[0] = globaltimer_ns();
      itr[3] = ((unsigned long long)blockIdx.x << 40) | ((unsigned long long)i << 20) | (unsigned)s;
    }
    // Wait until start s has completed steps 0 .. i-1.
    if (threadIdx.x == 0) {
      int ok = 1;
      long long polls = 0;
      while (ld_acquire_u32(a.done + s) < (unsigned)i) {
        if (++polls > a.wait_limit || ld_volatile_i32(a.err)) {
          ok = 0;
          break;
        }
        __nanosleep(32);
      }
      if (!ok) atomicOr(a.err, 1);
      sh.flag = ok;
    }
    __syncthreads();
    if (!sh.flag) return;
    // The residual pass of a start whose cost estimate from the gate-1
    // update is far above the tolerance is skipped: it could not decide
    // anything (the estimate, accurate to ~1e-7 absolute, stands).
    const bool act = (a.active == nullptr || a.active[s] != 0) &&
                     !(st.resid && a.resid_skip > 0.0 && __ldcg(a.resid_cost + s) > a.resid_skip);
    if (a.trace && threadIdx.x == 0 && c == 0) a.trace[((long long)i * a.S + s) * 4] = globaltimer_ns();
    if (itr && threadIdx.x == 0) itr[1] = globaltimer_ns();
    if (act) df_process<T>(st, s, c, sh, a.partials, a.resid_partials, a.part_stride, a.part_len, df_stage);
    // Publish this chunk; the last chunk of (step, start) finishes the step.
    __syncthreads();
    if (threadIdx.x == 0) {
      if (itr) itr[2] = globaltimer_ns();
      __threadfence();
      const unsigned old = atomicAdd(a.chunk_cnt + (long long)i * a.S + s, 1u);
      sh.flag = old == (unsigned)(st.nchunk - 1);
    }
    __syncthreads();
    if (sh.flag) {
      unsigned long long* tr = a.trace ? a.trace + ((long long)i * a.S + s) * 4 : nullptr;
      if (tr && threadIdx.x == 0) tr[1] = globaltimer_ns();
      if (act && st.kind != DF_FWD && st.kind != DF_FWD2) {
        __threadfence();
        if (st.kind == DF_RESID) {
          if (warp == 0) {
            const double* pp = a.resid_partials + (long long)s * a.part_stride * 32;
            double t = 0.0;
            for (int b = lane; b < st.nchunk; b += 32) t += __ldcg(pp + (long long)b * 32);
#pragma unroll
            for (int m = 16; m >= 1; m >>= 1) t += __shfl_xor_sync(FULL, t, m);
            if (lane == 0) {
              a.resid_cost[s] = t * a.inv_M;
              if (a.cost_row != nullptr) a.cost_row[s] = t * a.inv_M;
              if (a.stop != nullptr && t * a.inv_M <= a.stop_tol) atomicExch(a.stop, 1);
            }
          }
        } else if (sizeof(T) == 4 && st.kind == DF_ENV16) {
          if constexpr (sizeof(T) == 4) {
            // One of the 512 values of F per thread, over the chunks.
            float* fh = reinterpret_cast<float*>(df_stage);
            float* fl = fh + 512;
            const float* pp = reinterpret_cast<const float*>(a.partials) + (long long)s * a.part_stride * a.part_len + threadIdx.x;
            float hi = 0.f, lo = 0.f;
            for (int b0 = 0; b0 < st.nchunk; b0 += 8) {  // (eight loads in flight)
              float v[8];
#pragma unroll
              for (int b = 0; b < 8; ++b) v[b] = b0 + b < st.nchunk ? __ldcg(pp + (long long)(b0 + b) * a.part_len) : 0.f;
#pragma unroll
              for (int b = 0; b < 8; ++b) {
                float t;
                two_sum(hi, v[b], hi, t);
                lo += t;
              }
            }
            fh[threadIdx.x] = hi;
            fl[threadIdx.x] = lo;
            __syncthreads();
            if (tr && threadIdx.x == 0) tr[2] = globaltimer_ns();
            if (warp == 0)
              df_update_pair(st.upd, st.upd2, s, sh, reinterpret_cast<const float2*>(fh), reinterpret_cast<const float2*>(fl));
            if (st.upd2.cost_out != nullptr && threadIdx.x == 0 && a.cost_row != nullptr)
              a.cost_row[s] = st.upd2.cost_out[s];
          }
        } else {
          // The chunk partials summed by all warps (warp w takes chunks w, w
          // + NW, ...; fixed order), then over the warps: complex64 sums in
          // FP32 with their rounding kept (TwoSum), 16 FP64 additions being a
          // chain of 1000 cycles.
          const T* pp = reinterpret_cast<const T*>(a.partials) + (long long)s * a.part_stride * a.part_len;
          T acc[4] = {T(0), T(0), T(0), T(0)};
          int b = warp;
          for (; b + 3 * NW < st.nchunk; b += 4 * NW) {
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[q] += __ldcg(pp + (long long)(b + q * NW) * a.part_len + lane);
          }
          for (; b < st.nchunk; b += NW) acc[0] += __ldcg(pp + (long long)b * a.part_len + lane);
          const T mine = (acc[0] + acc[1]) + (acc[2] + acc[3]);
          if constexpr (sizeof(T) == 4) reinterpret_cast<float*>(sh.red[warp])[lane] = mine;
          else sh.red[warp][lane] = mine;
          __syncthreads();
          if (tr && threadIdx.x == 0) tr[2] = globaltimer_ns();
          // complex64 sweeps: the polar factor to FP32 accuracy, the accuracy
          // of their environments; FP64 sweeps: polar to FP64 rounding.
          if (warp == 0) {
            float hi = 0.f, lo = 0.f;
            double e = 0.0;
            if constexpr (sizeof(T) == 4) {
#pragma unroll
              for (int w = 0; w < NW; ++w) {
                float t;
                two_sum(hi, reinterpret_cast<const float*>(sh.red[w])[lane], hi, t);
                lo += t;
              }
            } else {
#pragma unroll
              for (int w = 0; w < NW; ++w) e += sh.red[w][lane];
            }
            df_update<T>(st.upd, s, sh, hi, lo, e);
          }
          if (st.upd.cost_out != nullptr && threadIdx.x == 0) {
            const double cost = st.upd.cost_out[s];
            if (a.cost_row != nullptr) a.cost_row[s] = cost;
            if (a.stop != nullptr && a.stop_from_update && cost <= a.stop_tol) atomicExch(a.stop, 1);
          }
        }
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        __threadfence();
        if (tr) tr[3] = globaltimer_ns();
        st_release_u32(a.done + s, (unsigned)(i + 1));
      }
    }
    __syncthreads();
  }
}

int df_blocks_per_sm(Real r) {
  static int cache[2] = {0, 0};
  int& c = cache[r == R32 ? 0 : 1];
  if (c) return c;
  int b = 0;
  cudaError_t e;
  if (r == R32) {
    e = cudaFuncSetAttribute(k_sweep_df<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, df_stage_bytes<float>());
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_sweep_df<float>, df_threads<float>(),
                                                        df_stage_bytes<float>());
  } else {
    e = cudaFuncSetAttribute(k_sweep_df<double>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             df_stage_bytes<double>());
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_sweep_df<double>, df_threads<double>(),
                                                        df_stage_bytes<double>());
  }
  if (e != cudaSuccess || b < 1) {
    cudaGetLastError();
    return 0;
  }
  c = b;
  return c;
}

cudaError_t launch_sweep_df(Real r, const DfArgs& a, int num_sms, cudaStream_t st) {
  const int bps = df_blocks_per_sm(r);
  if (bps < 1) return cudaErrorLaunchOutOfResources;
  const int grid = (int)std::min<long long>((long long)bps * num_sms, std::max<long long>(a.total_items, 1));
  DfArgs args = a;
  void* params[] = {&args};
  return r == R32 ? cudaLaunchCooperativeKernel((const void*)k_sweep_df<float>, dim3(grid),
                                                dim3(df_threads<float>()), params, df_stage_bytes<float>(), st)
                  : cudaLaunchCooperativeKernel((const void*)k_sweep_df<double>, dim3(grid),
                                                dim3(df_threads<double>()), params, df_stage_bytes<double>(), st);
}

// Chunking of one step: about `target` bytes of streaming per item, a
// multiple of 32 units per chunk.
void df_chunking(DfStep& st, double bytes_per_unit, double target) {
  long long nchunk = (long long)((st.units * bytes_per_unit + target - 1) / target);
  nchunk = std::max<long long>(1, std::min<long long>(nchunk, (st.units + 31) / 32));
  long long chunk = (st.units + nchunk - 1) / nchunk;
  chunk = (chunk + 31) / 32 * 32;
  st.chunk = (int)chunk;
  st.nchunk = (int)((st.units + chunk - 1) / chunk);
}

}  // namespace qfs
