// Batched QFactor-Sample: many small instantiation problems (3-5 qubits,
// 2-10 two-qubit gates each) and their multistarts in one persistent launch.
//
// Work is handed out in units: a unit is one problem and 32/G of its starts,
// run by one warp with G lanes per start (G = 32: a warp per start; G = 16,
// 8 or 4: two, four or eight starts share a warp).  Each start keeps its
// running state B and Phi (N x M complex, N <= 32, M <= 16) and its gates in
// its own slice of shared memory and sweeps as in Section 3 of the paper; the list of
// intermediate states is replaced by walking B back with the old gate
// (B_{k-1} = g_k^dagger B_k), so nothing leaves the SM between sweeps.  The
// starts' state arithmetic (gate applications, environment sums) runs side
// by side in their lane groups; each group reduces its environment over its
// own lanes, and the warp then updates the unit's gates one after another
// (Eq. 2: the FP32 Newton polar factor, FP64 Jacobi for ill-conditioned
// environments).  Units come from an atomic work
// queue ordered largest problem first; the schedule G (and the warps per
// block) of each class of problems (n, L, M) is chosen by the host's
// autotuner.  The run's stop rule is kept without any waiting: a start stops
// when it converges or once its sweep passes the earliest converged sweep of
// its problem (an atomicMin); the lowest-cost start among those that
// converged at that sweep is the problem's answer, which is what lock-step
// multistarts would return.  A finishing kernel then makes the selected
// gates unitary in FP64, checks the cost in FP64 and, if needed, refines
// with FP64 sweeps.
#include "polar_newton.cuh"
#include "qfs_common.cuh"
#include "qfs_kernels.h"

#include <climits>
#include <map>
#include <mutex>
#include <tuple>

namespace qfs {

namespace {

// Polar factor in FP32 (batched complex64 sweeps): each 16-lane half of the
// warp holds a matrix A (entry [r][c] at lane 4c + r), its own (HALVES) or
// both the same.  The scaled Newton iteration of polar_newton.cuh and one
// Newton-Schulz step, which leaves the factor unitary to FP32 rounding (the
// finishing kernel makes the answer unitary in FP64).  False in a half whose
// matrix is singular or too ill-conditioned (the caller then takes the FP64
// Jacobi, which also completes rank-deficient cases).
//
// Against the one-sided Jacobi with the gate's previous singular vectors as
// start that it replaces, an update needs no state between sweeps and a fixed
// 3 to 5 steps of 380 cycles where a Jacobi sweep took 750 and three to five
// of them were needed in the first sweeps of a run.
template <bool HALVES>
__device__ __forceinline__ bool batch_polar32(float2 a, float2* q_out) {
  const int l16 = threadIdx.x & 15, row = l16 & 3, col = l16 >> 2;
  const int its = newton_polar32<false, HALVES>(a, nullptr);
  if (!HALVES && !its) return false;
  const float2 g = mm16_ah(a, a, row, col);
  const float2 t{(row == col ? 1.5f : 0.f) - 0.5f * g.x, -0.5f * g.y};
  *q_out = mm16(a, t, row, col);
  return its != 0;
}

template <typename T> struct BT;
template <> struct BT<float> { using t2 = float2; };
template <> struct BT<double> { using t2 = double2; };

__device__ __forceinline__ uint32_t ins2(uint32_t r, int lo, int hi) {
  r = ((r >> lo) << (lo + 1)) | (r & ((1u << lo) - 1u));
  r = ((r >> hi) << (hi + 1)) | (r & ((1u << hi) - 1u));
  return r;
}

// X <- g X (dag = false) or X <- g^dagger X (dag = true) on qubits (qa, qb),
// X an N x M state in shared memory, by the G lanes of one group (gl = lane
// within the group).  The caller synchronises the warp.
template <int G, typename T2>
__device__ void group_apply(T2* X, const T2* g, int n, int M, int qa, int qb, bool dag, int gl) {
  const int pa = n - 1 - qa, pb = n - 1 - qb;
  const int lo = min(pa, pb), hi = max(pa, pb);
  const int groups = (1 << (n - 2)) * M;
  // The operator in registers (the state writes below could alias it for
  // the compiler): gg[4y + x] = (g or g^dagger)[y][x].
  T2 gg[16];
#pragma unroll
  for (int y = 0; y < 4; ++y)
#pragma unroll
    for (int x = 0; x < 4; ++x) gg[4 * y + x] = dag ? T2{g[4 * x + y].x, -g[4 * x + y].y} : g[4 * y + x];
  for (int w = gl; w < groups; w += G) {
    const int r = w / M, j = w - r * M;
    const uint32_t base = ins2((uint32_t)r, lo, hi);
    int off[4];
    T2 v[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      off[x] = (int)((base | ((uint32_t)(x >> 1) << pa) | ((uint32_t)(x & 1) << pb)) * M + j);
      v[x] = X[off[x]];
    }
#pragma unroll
    for (int y = 0; y < 4; ++y) {
      T2 t{0, 0};
#pragma unroll
      for (int x = 0; x < 4; ++x) t = cfma(gg[4 * y + x], v[x], t);
      X[off[y]] = t;
    }
  }
}

// Reduce-scatter of 32 per-lane values over the G lanes of a group: on
// return lane gl holds, in v[0 .. 32/G - 1], the group's sums of the values
// base .. base + 32/G - 1, base returned.
template <int G, typename T>
__device__ __forceinline__ int group_reduce_scatter(T (&v)[32], int gl) {
  int base = 0;
  int cnt = 32;
#pragma unroll
  for (int o = G / 2; o >= 1; o >>= 1) {
    cnt >>= 1;
    const bool upper = (gl & o) != 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      if (i < cnt) {
        const T send = upper ? v[i] : v[i + cnt];
        const T keep = upper ? v[i + cnt] : v[i];
        v[i] = keep + __shfl_xor_sync(FULL, send, o);
      }
    }
    if (upper) base += cnt;
  }
  return base;
}

// Environment partial sums of one start over its group's lanes:
// acc[2(4x+y)+{0,1}] += B[x] conj(Phi[y]) over the groups of (qa, qb).
template <int G, typename T, typename T2>
__device__ void group_env_acc(const T2* Bs, const T2* Ph, int n, int M, int qa, int qb, int gl, T (&acc)[32]) {
  const int pa = n - 1 - qa, pb = n - 1 - qb;
  const int lo = min(pa, pb), hi = max(pa, pb);
  const int groups = (1 << (n - 2)) * M;
  for (int w = gl; w < groups; w += G) {
    const int r = w / M, j = w - r * M;
    const uint32_t base = ins2((uint32_t)r, lo, hi);
    T2 b[4], p[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const int off = (int)((base | ((uint32_t)(x >> 1) << pa) | ((uint32_t)(x & 1) << pb)) * M + j);
      b[x] = Bs[off];
      p[x] = Ph[off];
    }
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        cfma_conj(acc[2 * (4 * x + y)], acc[2 * (4 * x + y) + 1], b[x], p[y]);
      }
  }
}

// New gate from E (E[c][r] in lane 4c + r of both halves): the polar factor
// of E^dagger.
__device__ void warp_update(float2 e, float2* g, double2* sm) {
  const int lane = threadIdx.x & 31;
  const int l16 = lane & 15, r = l16 & 3, c = l16 >> 2;
  const float2 a32{e.x, -e.y};  // A[r][c] = conj(E[c][r])
  float2 q;
  if (!batch_polar32<false>(a32, &q)) {
    const double2 p =
        warp_polar4(double2{(double)e.x, -(double)e.y}, double2{r == c ? 1.0 : 0.0, 0.0}, sm, nullptr);
    q = float2{(float)p.x, (float)p.y};
  }
  if (lane < 16) g[4 * r + c] = q;
  __syncwarp();
}
__device__ void warp_update64(double2 e, double2* g, double2* sm) {
  double2 p;
  polar_update_warp<2>(e, nullptr, 0.0, sm, g, nullptr, &p, nullptr);
  __syncwarp();
}

// The unit's two gate updates at once (16 lanes per start): half h updates
// the gate of start h from its environment e (E[c][r] at lane 4c + r of the
// half).  A half whose fast path fails takes the FP64 Jacobi (warp-wide, one
// half after the other), as warp_update does.
__device__ void halfwarp_update(float2 e, float2* g, double2* sm, bool act) {
  const int lane = threadIdx.x & 31;
  const int l16 = lane & 15, r = l16 & 3, c = l16 >> 2, h = lane >> 4;
  // A[r][c] = conj(E[c][r]); an idle half carries the identity along.
  const float2 a32 = act ? float2{e.x, -e.y} : float2{r == c ? 1.f : 0.f, 0.f};
  float2 q;
  const bool fine = batch_polar32<true>(a32, &q);
  const unsigned bad = __ballot_sync(FULL, !fine);
  for (int hh = 0; hh < 2; ++hh) {
    if (!((bad >> (16 * hh)) & 1u)) continue;
    // The FP64 Jacobi of half hh's matrix on the whole warp: A in lanes 0..15.
    const float2 ah{__shfl_sync(FULL, a32.x, 16 * hh + l16), __shfl_sync(FULL, a32.y, 16 * hh + l16)};
    const double2 p = warp_polar4(double2{(double)ah.x, (double)ah.y}, double2{r == c ? 1.0 : 0.0, 0.0}, sm, nullptr);
    const float2 pf{(float)p.x, (float)p.y};
    const float2 pq{__shfl_sync(FULL, pf.x, l16), __shfl_sync(FULL, pf.y, l16)};
    if (h == hh) q = pq;
  }
  if (act) g[4 * r + c] = q;
  __syncwarp();
}

// Per-start smem slice (complex64): B (E_max), Phi (E_max), gates (16 L_max),
// environment (16).
__host__ __device__ __forceinline__ int batch_slice_f2(int max_elems, int max_L) {
  return 2 * max_elems + 16 * max_L + 16;
}

// One sweep (Section 3) of every active start of a unit: forward to B_{L-1}
// with the current gates, then k = L..1: environment from (B_{k-1}, Phi_k),
// update gate k, B_{k-2} = g_{k-1}^dagger B_{k-1} (old gate), Phi_{k-1} =
// g_k^dagger Phi_k (new gate).  Returns, in every lane of a group, the
// residual (1/M) sum |g_1^dagger Phi_1 - Psi|^2 of its start's swept gates,
// as an FP32 sum of squares (no cancellation; relative error ~1e-6, far
// below what the FP64 check at dist_tol needs).  `act` is this group's
// start being active; `act_mask` has bit j set when group j is active.
template <int G>
__device__ float group_sweep(float2* slice, int slice_f2, int E_max, int L_max, const float2* psi,
                             const float2* phil, const int* pairs, int n, int M, int L, double2* sm, bool act,
                             unsigned act_mask) {
  constexpr int NG = 32 / G;
  const int lane = threadIdx.x & 31;
  const int gi = lane / G, gl = lane % G;
  float2* Bs = slice + gi * slice_f2;
  float2* Ph = Bs + E_max;
  float2* Gt = Ph + E_max;
  float* Env = reinterpret_cast<float*>(Gt + 16 * L_max);
  const int E = M << n;
  if (act) {
    for (int i = gl; i < E; i += G) {
      Bs[i] = psi[i];
      Ph[i] = phil[i];
    }
  }
  __syncwarp();
  for (int k = 1; k <= L - 1; ++k) {
    if (act) group_apply<G, float2>(Bs, Gt + 16 * (k - 1), n, M, pairs[2 * (k - 1)], pairs[2 * (k - 1) + 1], false, gl);
    __syncwarp();
  }
  for (int k = L; k >= 1; --k) {
    const int qa = pairs[2 * (k - 1)], qb = pairs[2 * (k - 1) + 1];
    float acc[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = 0.f;
    if (act) group_env_acc<G, float, float2>(Bs, Ph, n, M, qa, qb, gl, acc);
    if constexpr (G == 32) {
      const float v = warp_reduce_scatter32<float>(acc, lane);
      const int l16 = lane & 15;
      const float2 e{__shfl_sync(FULL, v, 2 * l16), __shfl_sync(FULL, v, 2 * l16 + 1)};
      if (act) warp_update(e, Gt + 16 * (k - 1), sm);
    } else if constexpr (G == 16) {
      // After the reduce-scatter lane gl holds two of its start's 32
      // environment floats; gather E[c][r] to lane 4c + r of each half
      // through shared memory, then both starts' updates run side by side.
      const int base = group_reduce_scatter<G, float>(acc, gl);
      Env[base] = acc[0];
      Env[base + 1] = acc[1];
      __syncwarp();
      const float2 e{Env[2 * gl], Env[2 * gl + 1]};
      halfwarp_update(e, Gt + 16 * (k - 1), sm, act);
    } else {
      const int base = group_reduce_scatter<G, float>(acc, gl);
#pragma unroll
      for (int i = 0; i < 32 / G; ++i) Env[base + i] = acc[i];
      __syncwarp();
      // The warp updates the unit's gates one start after another.
      const int l16 = lane & 15;
#pragma unroll 1
      for (int j = 0; j < NG; ++j) {
        if (!((act_mask >> j) & 1u)) continue;
        float2* sj = slice + j * slice_f2;
        const float* envj = reinterpret_cast<const float*>(sj + 2 * E_max + 16 * L_max);
        const float2 e{envj[2 * l16], envj[2 * l16 + 1]};
        warp_update(e, sj + 2 * E_max + 16 * (k - 1), sm);
      }
    }
    __syncwarp();
    if (k > 1 && act) {
      group_apply<G, float2>(Bs, Gt + 16 * (k - 2), n, M, pairs[2 * (k - 2)], pairs[2 * (k - 2) + 1], true, gl);
      group_apply<G, float2>(Ph, Gt + 16 * (k - 1), n, M, qa, qb, true, gl);
    }
    __syncwarp();
  }
  float r = 0.f;
  if (act) group_apply<G, float2>(Ph, Gt, n, M, pairs[0], pairs[1], true, gl);
  __syncwarp();
  if (act) {
    for (int i = gl; i < E; i += G) {
      const float2 p = Ph[i], q = psi[i];
      const float dx = p.x - q.x, dy = p.y - q.y;
      r = fmaf(dx, dx, fmaf(dy, dy, r));
    }
  }
#pragma unroll
  for (int o = G / 2; o >= 1; o >>= 1) r += __shfl_xor_sync(FULL, r, o);
  __syncwarp();
  return r * (1.f / (float)M);
}

// One FP64 sweep of one start by a whole warp (the refinement sweeps of the
// finishing kernel), as group_sweep with G = 32, B and Phi in Bs and Ph.
__device__ void warp_sweep64(double2* Bs, double2* Ph, double2* G, const double2* psi, const double2* phil,
                             const int* pairs, int n, int M, int L, double2* sm) {
  const int lane = threadIdx.x & 31;
  const int E = M << n;
  for (int i = lane; i < E; i += 32) {
    Bs[i] = psi[i];
    Ph[i] = phil[i];
  }
  __syncwarp();
  for (int k = 1; k <= L - 1; ++k) {
    group_apply<32, double2>(Bs, G + 16 * (k - 1), n, M, pairs[2 * (k - 1)], pairs[2 * (k - 1) + 1], false, lane);
    __syncwarp();
  }
  for (int k = L; k >= 1; --k) {
    const int qa = pairs[2 * (k - 1)], qb = pairs[2 * (k - 1) + 1];
    double acc[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = 0.0;
    group_env_acc<32, double, double2>(Bs, Ph, n, M, qa, qb, lane, acc);
    const double v = warp_reduce_scatter32<double>(acc, lane);
    const int l16 = lane & 15;
    const double2 e{__shfl_sync(FULL, v, 2 * l16), __shfl_sync(FULL, v, 2 * l16 + 1)};
    warp_update64(e, G + 16 * (k - 1), sm);
    if (k > 1) {
      group_apply<32, double2>(Bs, G + 16 * (k - 2), n, M, pairs[2 * (k - 2)], pairs[2 * (k - 2) + 1], true, lane);
      group_apply<32, double2>(Ph, G + 16 * (k - 1), n, M, qa, qb, true, lane);
    }
    __syncwarp();
  }
}

}  // namespace

namespace {
// Largest exponent field of `count` complex numbers, by a whole block.
__device__ int block_exponent(const double2* z, int count, int* red) {
  int top = 0;
  for (int i = threadIdx.x; i < count; i += blockDim.x) {
    const double2 v = z[i];
    top = max(top, max((__double2hiint(v.x) >> 20) & 0x7ff, (__double2hiint(v.y) >> 20) & 0x7ff));
  }
  top = __reduce_max_sync(FULL, top);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = top;
  __syncthreads();
  for (int w = 0; w < (int)blockDim.x / 32; ++w) top = max(top, red[w]);
  return top;
}
}  // namespace

// Per-problem set-up: Phi_L = U Psi to FP64 accuracy and complex64 copies of
// Psi and Phi_L.  One block per problem, one component of the product per
// thread at a time, in fixed point with a scale for every row of U and column
// of Psi (fixed.cuh: FxDot).  (1024 problems of 3 to 5 qubits: 110 us in FP64,
// whose pipe it filled by a third, 52 so; 96 problems 20.)  Error relative to the product's norm
// at n = 6: FP64 3.9e-16, with one scale for all of U and all of Psi and without
// the low x low products 1.2e-15, so 6e-17.  Rows and columns out of the scales'
// range (Inf, NaN) take the FP64 form.
__global__ void __launch_bounds__(128) k_batch_prep(BatchArgs a) {
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ int tu[1 << kBatchMaxQubits], tp[1 << kBatchMaxQubits];  // largest exponent fields (M <= N)
  const int p = blockIdx.x;
  if (p >= a.P) return;
  const BatchProblem pr = a.probs[p];
  const int n = pr.n, N = 1 << n, M = pr.M, lane = threadIdx.x & 31;
  const double2* U = a.targets + pr.target_off;
  const double2* psi = a.psi64 + pr.state_off;
  if (threadIdx.x == 0) a.s_star[p] = INT_MAX;
  int4* su = reinterpret_cast<int4*>(dsm);
  int4* sp = su + N * N;
  for (int j = threadIdx.x; j < M; j += blockDim.x) tp[j] = 0;
  __syncthreads();
  for (int e = threadIdx.x; e < N * M; e += blockDim.x) {
    const double2 s = psi[e];
    a.psi32[pr.state_off + e] = float2{(float)s.x, (float)s.y};
    atomicMax(&tp[e % M], fx_top(s));
  }
  // A warp takes four rows of U at a time: their loads, then their exponents.
  for (int r = 4 * (threadIdx.x >> 5); r < N; r += 16) {
    double2 z[4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int h = 0; h < 2; ++h) z[i][h] = lane + 32 * h < N ? U[(r + i) * N + lane + 32 * h] : double2{0.0, 0.0};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int t = __reduce_max_sync(FULL, max(fx_top(z[i][0]), fx_top(z[i][1])));
      if (lane == 0) tu[r + i] = t;
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (lane + 32 * h < N) su[(r + i) * N + lane + 32 * h] = fx_from2(z[i][h], fx_row_exp(t, n));
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < N * M; e += blockDim.x) sp[e] = fx_from2(psi[e], fx_col_exp(tp[e % M], n));
  __syncthreads();
  for (int c = threadIdx.x; c < 2 * N * M; c += blockDim.x) {
    const int e = c >> 1, im = c & 1, i = e / M, j = e - i * M;
    double v = 0.0;
    if (fx_out_of_range(tu[i]) || fx_out_of_range(tp[j])) {
      for (int k = 0; k < N; ++k) {
        const double2 x = U[i * N + k], y = psi[k * M + j];
        v = im ? fma(x.x, y.y, fma(x.y, y.x, v)) : fma(x.x, y.x, fma(-x.y, y.y, v));
      }
    } else {
      FxDot t;
      t.run<1>(su + i * N, sp + j, M, 0, N, im);
      v = fx_dot_value(t.t.h, t.cross(), fx_row_exp(tu[i], n) + fx_col_exp(tp[j], n));
    }
    reinterpret_cast<double*>(a.phil64 + pr.state_off + e)[im] = v;
    reinterpret_cast<float*>(a.phil32 + pr.state_off + e)[im] = (float)v;
  }
}

// One unit (a problem and up to 32/G of its starts) swept by the warp to
// its end, in `region` (the warp's shared memory, laid out for this
// problem: a slice of batch_slice_f2(N M, L) float2 per start).
template <int G>
__device__ __forceinline__ void batch_run_unit(const BatchArgs& a, const BatchUnit& u, float2* region,
                                               double2* sm_polar) {
  constexpr int NG = 32 / G;
  const int lane = threadIdx.x & 31;
  const int gi = lane / G, gl = lane % G;
  const int p = u.p;
  const BatchProblem pr = a.probs[p];
  const int* pairs = a.pairs + pr.pair_off;
  const int E = pr.M << pr.n, L = pr.L;
  const int sf = batch_slice_f2(E, L);
  const int s = u.s0 + gi;
  bool act = gi < u.ns;
  float2* mine = region + gi * sf;
  float2* Gt = mine + 2 * E;
  const size_t goff = pr.gate_off + (size_t)s * L * 16;
  if (act) {
    for (int i = gl; i < 16 * L; i += G) {
      const double2 g = a.init_gates[goff + i];
      Gt[i] = float2{(float)g.x, (float)g.y};
    }
  }
  __syncwarp();
  const float2* psi = a.psi32 + pr.state_off;
  const float2* phil = a.phil32 + pr.state_off;
  int conv = INT_MAX, sweeps = 0, stall = 0;
  // The sweep's cost and the plateau test stay in FP32 (the FP64 pipe
  // costs 64 cycles per warp instruction); only the tolerance test is FP64.
  float cost = 4.f, prev = -1.f;
  const float dtr = (float)a.diff_tol_r;
  for (int sw = 1; sw <= a.max_sweeps; ++sw) {
    // A start that has not converged by its problem's earliest converged
    // sweep can no longer be selected.
    if (sw > *(volatile int*)(a.s_star + p)) act = false;
    const unsigned ballot = __ballot_sync(FULL, act && gl == 0);
    unsigned mask = 0;
#pragma unroll
    for (int j = 0; j < NG; ++j) mask |= ((ballot >> (j * G)) & 1u) << j;
    if (!mask) break;
    const float c = group_sweep<G>(region, sf, E, L, psi, phil, pairs, pr.n, pr.M, L, sm_polar, act, mask);
    if (act) {
      cost = c;
      sweeps = sw;
      if ((double)cost <= a.tol) {
        conv = sw;
        if (gl == 0) atomicMin(a.s_star + p, sw);
        act = false;
      } else if (a.plateau_window > 0 && prev >= 0.f) {
        // Plateau (App. A): no relative improvement > diff_tol_r for
        // plateau_window sweeps in a row stops this start.
        stall = fabsf(prev) - fabsf(cost) > dtr * fabsf(cost) ? 0 : stall + 1;
        if (stall >= a.plateau_window && sw >= a.min_sweeps) act = false;
      }
      prev = cost;
    }
  }
  if (gi < u.ns) {
    const size_t ri = (size_t)p * a.S + s;
    if (gl == 0) {
      a.conv_sweep[ri] = conv;
      a.final_cost[ri] = (double)cost;
      a.sweeps_run[ri] = sweeps;
    }
    for (int i = gl; i < 16 * L; i += G) a.gates32[goff + i] = Gt[i];
  }
  __syncwarp();
}

// Persistent sweep kernel with G lanes per start: warps take units until
// the queue is empty.  region_f2: each warp's shared memory in float2 (at
// least (32/G) batch_slice_f2(N M, L) for every unit it may take).
template <int G>
__global__ void k_batch_sweep(BatchArgs a, const BatchUnit* units, int nunits, int* queue, int region_f2) {
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ double2 sm_polar[kBatchMaxWarps][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* region = reinterpret_cast<float2*>(dsm) + (size_t)warp * region_f2;
  while (true) {
    int item = 0;
    if (lane == 0) item = atomicAdd(queue, 1);
    item = __shfl_sync(FULL, item, 0);
    if (item >= nunits) break;
    const unsigned long long t0 = a.unit_trace ? globaltimer_ns() : 0ull;
    batch_run_unit<G>(a, units[item], region, sm_polar[warp]);
    if (a.unit_trace && lane == 0) {
      const BatchUnit u = units[item];
      unsigned sm;
      asm volatile("mov.u32 %0, %%smid;" : "=r"(sm));
      unsigned long long* r = a.unit_trace + 4 * (size_t)item;
      r[0] = t0;
      r[1] = globaltimer_ns();
      r[2] = (unsigned long long)u.p;
      r[3] = ((unsigned long long)sm << 32) | ((unsigned long long)u.s0 << 16) | ((unsigned)u.ns << 8) | G;
    }
  }
}

// One block per problem: pick the start, make its gates unitary, check the
// cost, FP64 refinement sweeps while the cost is above tol.
//
// Gates are made unitary by one warp each and the cost's circuit is applied in
// fixed point (fixed.cuh), each to FP64 accuracy: bound by integer issue.  As
// one warp of FP64 instructions a problem took 30 to 80 us (1024 problems of 3
// to 5 qubits: 172 us).
__global__ void __launch_bounds__(128) k_batch_finalize(BatchArgs a) {
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ NewtonSh nw[4];
  __shared__ double red[4];
  __shared__ int redi[4];
  const int p = blockIdx.x;
  if (p >= a.P) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int l16 = lane & 15, row = l16 & 3, col = l16 >> 2, im = lane >> 4;
  const BatchProblem pr = a.probs[p];
  const int E = pr.M << pr.n, n = pr.n, M = pr.M;
  double2* Bs = reinterpret_cast<double2*>(dsm);  // (refinement sweeps)
  double2* Ph = Bs + a.max_elems;
  double2* G = Ph + a.max_elems;
  int4* X = reinterpret_cast<int4*>(G + 16 * a.max_L);
  int4* GX = X + a.max_elems;
  // Selection: among starts converged at the earliest converged sweep, the
  // lowest cost (lowest index on ties); if none converged, the lowest cost.
  const int sst = a.s_star[p];
  int best = 0;
  double bc = 1e300;
  for (int s = lane; s < a.S; s += 32) {
    const size_t ri = (size_t)p * a.S + s;
    const double c = a.final_cost[ri];
    if ((sst == INT_MAX || a.conv_sweep[ri] == sst) && c < bc) {
      bc = c;
      best = s;
    }
  }
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) {
    const double oc = __shfl_xor_sync(FULL, bc, m);
    const int ob = __shfl_xor_sync(FULL, best, m);
    if (oc < bc || (oc == bc && ob < best)) {
      bc = oc;
      best = ob;
    }
  }
  const int sweeps = sst == INT_MAX ? a.sweeps_run[(size_t)p * a.S + best] : sst;
  const size_t goff = pr.gate_off + (size_t)best * pr.L * 16;
  const NewtonPair pair = newton_pair();
  for (int k = warp; k < pr.L; k += 4) {
    float2 x = a.gates32[goff + 16 * k + (4 * row + col)];  // lane 4col+row holds g[row][col]
    long long q;
    newton_unitary(x, nw[warp], pair, q, true);
    reinterpret_cast<int2*>(GX + 16 * k + 4 * row + col)[im] = fx_split(q);
    reinterpret_cast<double*>(G + 16 * k + 4 * row + col)[im] = scale_exp((double)q, -kFxBits);
    __syncwarp();
  }
  const int* pairs = a.pairs + pr.pair_off;
  const double2* psi = a.psi64 + pr.state_off;
  const double2* phil = a.phil64 + pr.state_off;
  // FP64 cost: (1/M) || Phi_L - C Psi ||^2.  One scale for both sides, with
  // room for an entry to grow to its column's norm (3 bits).
  const int top = max(block_exponent(psi, E, redi), block_exponent(phil, E, redi));
  double c;
  auto cost64 = [&]() {  // (warp 0, in FP64: refined gates, and numbers out of the scale's range)
    for (int i = lane; i < E; i += 32) Bs[i] = psi[i];
    __syncwarp();
    for (int k = 1; k <= pr.L; ++k) {
      group_apply<32, double2>(Bs, G + 16 * (k - 1), n, M, pairs[2 * (k - 1)], pairs[2 * (k - 1) + 1], false, lane);
      __syncwarp();
    }
    double acc = 0.0;
    for (int i = lane; i < E; i += 32) {
      const double dx = phil[i].x - Bs[i].x, dy = phil[i].y - Bs[i].y;
      acc += dx * dx + dy * dy;
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) acc += __shfl_xor_sync(FULL, acc, o);
    return acc / M;
  };
  if (!fx_out_of_range(top)) {
    const int e = top - 1022 + 3;
    const uint32_t fold = swz_fold(n);
    for (int i = tid; i < E; i += 128) {
      const int r = i / M, j = i - r * M;
      X[swz(((uint32_t)j << n) | (uint32_t)r, fold)] = fx_from2(psi[i], e);
    }
    __syncthreads();
    for (int k = 0; k < pr.L; ++k) {
      fx_apply<128>(X, X, GX + 16 * k, pair_bits(n - 1 - pairs[2 * k], n - 1 - pairs[2 * k + 1]), false, E >> 2, n);
      __syncthreads();
    }
    double acc = 0.0;
    for (int i = tid; i < E; i += 128) {
      const int r = i / M, j = i - r * M;
      const int4 x = X[swz(((uint32_t)j << n) | (uint32_t)r, fold)], y = fx_from2(phil[i], e);
      const double dx = (double)(fx_value(y.x, y.y) - fx_value(x.x, x.y)), dy = (double)(fx_value(y.z, y.w) - fx_value(x.z, x.w));
      acc = fma(dx, dx, fma(dy, dy, acc));
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) acc += __shfl_xor_sync(FULL, acc, o);
    if (lane == 0) red[warp] = acc;
    __syncthreads();
    c = ldexp((red[0] + red[1]) + (red[2] + red[3]), 2 * (e - kFxBits)) / M;
  } else {
    __syncthreads();
    if (warp == 0) {
      c = cost64();
      if (lane == 0) red[0] = c;
    }
    __syncthreads();
    c = red[0];
  }
  int refine = 0;
  if (warp == 0) {
    while (c > a.tol && refine < a.refine_max && (sst != INT_MAX || a.refine_unconverged)) {
      warp_sweep64(Bs, Ph, G, psi, phil, pairs, n, M, pr.L, nw[0].polar);
      ++refine;
      c = cost64();
    }
  }
  __syncthreads();
  for (int i = tid; i < 16 * pr.L; i += 128) a.gates_out[pr.gate_out_off + i] = G[i];
  if (tid == 0) {
    a.res_cost[p] = c;
    a.res_sweeps[p] = sweeps;
    a.res_best[p] = best;
    a.res_refine[p] = refine;
  }
}

cudaError_t launch_batch_prep(const BatchArgs& a, cudaStream_t st) {
  const cudaError_t e = allow_smem(k_batch_prep, kBatchPrepSmem);
  return e != cudaSuccess ? e : launch_kernel(k_batch_prep, a.P, 128, (size_t)a.max_prep * sizeof(int4), st, a);
}

int batch_region_f2(int G, int max_elems, int max_L) { return (32 / G) * batch_slice_f2(max_elems, max_L); }

size_t batch_sweep_smem(int G, int warps, int max_elems, int max_L) {
  return (size_t)warps * batch_region_f2(G, max_elems, max_L) * sizeof(float2);
}

namespace {
template <int G>
int blocks_per_sm_g(int warps, size_t smem) {
  allow_smem(k_batch_sweep<G>, kBatchSweepSmem);
  int b = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_batch_sweep<G>, 32 * warps, smem) != cudaSuccess) {
    cudaGetLastError();
    b = 0;
  }
  return b;
}
}  // namespace

// (Asked about 180 times a call of a thousand problems in 21 classes; the driver's
// two calls behind an answer took 190 us of the call together, so answers are
// kept, by device and launch shape.)
int batch_sweep_blocks_per_sm(int G, int warps, size_t smem) {
  static std::mutex mu;
  static std::map<std::tuple<int, int, int, size_t>, int> known;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  const auto key = std::make_tuple(dev, G, warps, smem);
  std::lock_guard<std::mutex> lock(mu);
  const auto it = known.find(key);
  if (it != known.end()) return it->second;
  int b = 0;
  switch (G) {
    case 4: b = blocks_per_sm_g<4>(warps, smem); break;
    case 8: b = blocks_per_sm_g<8>(warps, smem); break;
    case 16: b = blocks_per_sm_g<16>(warps, smem); break;
    case 32: b = blocks_per_sm_g<32>(warps, smem); break;
    default: break;
  }
  if (known.size() >= 4096) known.clear();
  known[key] = b;
  return b;
}

cudaError_t launch_batch_sweep(int G, const BatchArgs& a, const BatchUnit* units, int nunits, int* queue, int blocks,
                               int warps, int region_f2, cudaStream_t st) {
  const size_t smem = (size_t)warps * region_f2 * sizeof(float2);
  const auto kernel = G == 4 ? k_batch_sweep<4> : G == 8 ? k_batch_sweep<8> : G == 16 ? k_batch_sweep<16> : k_batch_sweep<32>;
  const cudaError_t e = allow_smem(kernel, kBatchSweepSmem);
  return e != cudaSuccess ? e : launch_kernel(kernel, blocks, 32 * warps, smem, st, a, units, nunits, queue, region_f2);
}

cudaError_t launch_batch_finalize(const BatchArgs& a, cudaStream_t st) {
  const size_t smem = (size_t)(3 * a.max_elems + 32 * a.max_L) * sizeof(double2);
  const cudaError_t e = allow_smem(k_batch_finalize, kBatchFinalizeSmem);
  return e != cudaSuccess ? e : launch_kernel(k_batch_finalize, a.P, 128, smem, st, a);
}

}  // namespace qfs
