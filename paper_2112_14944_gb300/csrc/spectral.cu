// Graph analysis for the deflated Chebyshev sweeps of the FP32 propagation.
//
// The walk matrix P of an undirected graph is self-adjoint in the inner
// product <u, v>_D = sum_i dw_i u_i v_i, so its spectrum is real. Each
// connected component C contributes the eigenvalue 1 (right eigenvector 1_C,
// left eigenvector the stationary vector dw 1_C / m_C, m_C = sum_{i in C} dw_i);
// a node without edges is a component of its own (its walk stays put). For the
// PPR system x (I - cP) = alpha e_s the coefficient of x on the stationary
// vector of C(s) is exactly x 1_C = 1 (multiply the system by 1_C), so the
// propagation can start from that vector and leave only the other modes,
// whose eigenvalues lie in [-b, b] for some b <= 1. Chebyshev semi-iteration
// on [1 - cb, 1 + cb] then converges at rate (1 - sqrt(1 - (cb)^2)) / (cb)
// instead of the rate for b = 1.
//
// This file computes, once per graph:
//  * the component root of every node (the smallest node id of its
//    component; hooking of larger roots under smaller ones with atomicMin,
//    then pointer jumping, until no edge joins two roots), and m_C per root;
//  * an estimate of b: power iteration with P^2 from v_0 = (P - I) u (which
//    has no component on any eigenvalue-1 mode, since (P - I) 1_C = 0 and P
//    is self-adjoint in <,>_D), then the Rayleigh quotient
//    b^2 ~ <P v, P v>_D / <v, v>_D. It is a lower estimate (a weighted mean
//    of lambda^2), so a margin is added; an underestimate only slows the
//    modes above it, it never breaks convergence, and the FP64 residual
//    certificate decides when a row is done.
// All reductions run in a fixed order, so the estimate (and every result
// downstream of it) is the same on every run.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"

namespace pprviz {

namespace {
constexpr int kSpecBlocks = 256;  // blocks of the partial-sum reductions
constexpr int kSpecIters = 12;    // P^2 power steps
constexpr int kCcMaxRounds = 64;  // hooking rounds before giving up

__global__ void k_cc_init(int64_t n, int32_t *__restrict__ parent) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) parent[i] = (int32_t)i;
}

// bounded walk to the root (parent[x] <= x always, so at most x steps)
template <typename P>
__device__ __forceinline__ int32_t cc_root(P parent, int32_t x) {
  for (int it = 0; it < (1 << 20); ++it) {
    const int32_t p = parent[x];
    if (p == x) break;
    x = p;
  }
  return x;
}

// One warp per node u: for every edge (u, v) with u < v, hook the larger root
// under the smaller one.
__global__ void k_cc_hook(int64_t n, const int64_t *__restrict__ rp, const int32_t *__restrict__ col,
                          int32_t *parent, int *__restrict__ changed) {
  const int64_t u = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (u >= n) return;
  int ch = 0;
  for (int64_t p = rp[u] + lane; p < rp[u + 1]; p += 32) {
    const int32_t v = col[p];
    if ((int64_t)v <= u) continue;
    const int32_t ru = cc_root(parent, (int32_t)u), rv = cc_root(parent, v);
    if (ru != rv) {
      atomicMin(&parent[max(ru, rv)], min(ru, rv));
      ch = 1;
    }
  }
  if (__any_sync(0xffffffffu, ch) && lane == 0) atomicOr(changed, 1);
}

__global__ void k_cc_compress(int64_t n, int32_t *parent) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) parent[i] = cc_root(parent, parent[i]);
}

// deterministic start vector u_i in [-0.5, 0.5) (SplitMix64 finaliser of i)
__device__ __forceinline__ double start_u(int64_t i) {
  uint64_t z = (uint64_t)i + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  return (double)(z >> 11) * (1.0 / 9007199254740992.0) - 0.5;
}

// out = P v (or P u - u with the start vector when v == nullptr), FP64, one warp per row:
// (P v)_j = (1 / dw_j) sum_{i in N(j)} w_ji v_i, and v_j for a node without edges.
__global__ void k_spec_spmv(int64_t n, const int64_t *__restrict__ rp, const int32_t *__restrict__ col,
                            const float *__restrict__ w, const double *__restrict__ invdw,
                            const double *__restrict__ v, double *__restrict__ out) {
  const int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (j >= n) return;
  const int64_t b = rp[j], e = rp[j + 1];
  double acc = 0.0;
  for (int64_t p = b + lane; p < e; p += 32) {
    const int32_t i = col[p];
    const double vi = v ? v[i] : start_u(i);
    acc += (w ? (double)w[p] : 1.0) * vi;
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) {
    const double vj = v ? v[j] : start_u(j);
    const double pv = (e == b) ? vj : acc * invdw[j];
    out[j] = v ? pv : pv - vj;
  }
}

// part[blk] = sum over the block's strided share of dw_i a_i b_i (dw = 1 / invdw)
__global__ void k_spec_dot(int64_t n, const double *__restrict__ invdw, const double *__restrict__ a,
                           const double *__restrict__ b, double *__restrict__ part) {
  __shared__ double red[256];
  double s = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    s += a[i] * b[i] / invdw[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// out[0] = sum of part[0 .. np) in a fixed order
__global__ void k_spec_sum(int np, const double *__restrict__ part, double *__restrict__ out) {
  __shared__ double red[256];
  double s = 0.0;
  for (int i = threadIdx.x; i < np; i += blockDim.x) s += part[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[0] = red[0];
}

// v /= sqrt(nrm2[0]) when it is positive (keeps the power iterates in range)
__global__ void k_spec_normalise(int64_t n, const double *__restrict__ nrm2, double *__restrict__ v) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const double s = nrm2[0];
  if (i < n && s > 0.0) v[i] *= 1.0 / sqrt(s);
}

// Sum over the CTA (1,024 threads), the same value in every thread.
__device__ __forceinline__ double block_sum(double s, double *red) {
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  __syncthreads();  // red is free
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  double t = red[threadIdx.x & 31];
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// The whole analysis of a small graph (n <= kSpecSmall, few edges) by one CTA: components,
// then the power steps, with the vectors in shared memory and 8 lanes per row.
// The separate kernels below cost a launch per step and a host wait per
// component round, ~345 us for a 150-node view; this one about 130 us with its read-back.
// out: [0] <v, v>, [1] <P v, P v>, [2] 1 when the components are resolved, then
// 1 / dw of the n nodes, then the component roots (int32).
constexpr int64_t kSpecSmall = 512;
__global__ void __launch_bounds__(1024)
k_spec_small(int n, const int64_t *__restrict__ rp, const int32_t *__restrict__ col, const float *__restrict__ w,
             const double *__restrict__ invdw, int32_t *__restrict__ comp, double *__restrict__ out) {
  __shared__ int32_t parent[kSpecSmall];
  __shared__ double va[kSpecSmall], vb[kSpecSmall], red[32];
  const int g8 = threadIdx.x >> 3, l8 = threadIdx.x & 7;  // row group and lane in it
  for (int i = threadIdx.x; i < n; i += 1024) parent[i] = i;
  __syncthreads();
  bool done = false;
  for (int round = 0; round < kCcMaxRounds && !done; ++round) {
    int ch = 0;
    for (int u = g8; u < n; u += 128)
      for (int64_t p = rp[u] + l8; p < rp[u + 1]; p += 8) {
        const int32_t v = col[p];
        if (v <= u) continue;
        const int32_t ru = cc_root((volatile int32_t *)parent, u), rv = cc_root((volatile int32_t *)parent, v);
        if (ru != rv) {
          atomicMin(&parent[max(ru, rv)], min(ru, rv));
          ch = 1;
        }
      }
    done = __syncthreads_or(ch) == 0;
    for (int i = threadIdx.x; i < n; i += 1024) {
      const int32_t r = cc_root((volatile int32_t *)parent, i);
      *(volatile int32_t *)&parent[i] = r;
    }
    __syncthreads();
  }
  int32_t *comp_out = reinterpret_cast<int32_t *>(out + 3 + n);
  for (int i = threadIdx.x; i < n; i += 1024) {
    comp[i] = parent[i];
    comp_out[i] = parent[i];
    out[3 + i] = invdw[i];
  }
  // dst = P src (FIRST: (P - I) u with the start vector)
  auto step = [&](const double *src, double *dst) {
    for (int j0 = 0; j0 < n; j0 += 128) {
      const int j = j0 + g8;
      double acc = 0.0;
      int64_t b = 0, e = 0;
      if (j < n) {
        b = rp[j];
        e = rp[j + 1];
        for (int64_t p = b + l8; p < e; p += 8) {
          const int32_t i = col[p];
          acc += (w ? (double)w[p] : 1.0) * (src ? src[i] : start_u(i));
        }
      }
      for (int o = 4; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (j < n && l8 == 0) {
        const double vj = src ? src[j] : start_u(j);
        const double pv = (e == b) ? vj : acc * invdw[j];
        dst[j] = src ? pv : pv - vj;
      }
    }
    __syncthreads();
  };
  auto dot = [&](const double *a) {
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += 1024) s += a[i] * a[i] / invdw[i];
    return block_sum(s, red);
  };
  step(nullptr, va);
  for (int it = 0; it < kSpecIters; ++it) {
    step(va, vb);
    step(vb, va);
    if (it % 4 == 3) {
      const double s = dot(va);
      if (s > 0.0)
        for (int i = threadIdx.x; i < n; i += 1024) va[i] *= 1.0 / sqrt(s);
      __syncthreads();
    }
  }
  step(va, vb);
  const double vv = dot(va), pp = dot(vb);
  if (threadIdx.x == 0) {
    out[0] = vv;
    out[1] = pp;
    out[2] = done ? 1.0 : 0.0;
  }
}

// Directed graphs, the walk T among the nodes with out-edges (a dangling node
// keeps its walk and feeds nobody; it counts as 0 here):
// LEFT: out_j = sum_{i -> j} w_ij v_i / dw_i over the pull rows (the dangling
// nodes' own entries weigh 0); at a dangling j 0, or with `keep` what flows in.
// Right: out_i = (1 / dw_i) sum_{i -> j} w_ij v_j over the out rows. One warp per row.
template <bool LEFT>
__global__ void k_dir_spmv(int64_t n, const int64_t *__restrict__ orp, const int64_t *__restrict__ rp,
                           const int32_t *__restrict__ col, const float *__restrict__ w,
                           const double *__restrict__ invdw, const double *__restrict__ v, double *__restrict__ out,
                           bool keep) {
  const int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (j >= n) return;
  const bool dangling = orp[j] == orp[j + 1];
  double acc = 0.0;
  for (int64_t p = rp[j] + lane; p < rp[j + 1]; p += 32) {
    const int32_t i = col[p];
    const double wi = w ? (double)w[p] : 1.0;
    acc += LEFT ? wi * (v[i] * invdw[i]) : wi * v[i];
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) out[j] = (dangling && !keep) ? 0.0 : LEFT ? acc : acc * invdw[j];
}

// the starts: 1, or the hashed vector of the spectral bound, on nodes with out-edges
__global__ void k_dir_start(int64_t n, const int64_t *__restrict__ orp, bool hashed, double *__restrict__ v) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) v[i] = orp[i] == orp[i + 1] ? 0.0 : hashed ? start_u(i) : 1.0;
}

// part[blk] = the block's strided share of sum_i a_i b_i
__global__ void k_dir_dot(int64_t n, const double *__restrict__ a, const double *__restrict__ b,
                          double *__restrict__ part) {
  __shared__ double red[256];
  double s = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    s += a[i] * b[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// z -= (zu / vu) v
__global__ void k_dir_project(int64_t n, const double *__restrict__ zu, const double *__restrict__ vu,
                              const double *__restrict__ v, double *__restrict__ z) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n && vu[0] > 0.0) z[i] -= zu[0] / vu[0] * v[i];
}

// What graph_perron judges the pair by, per block: v v, v (v T), |v T|^2, u u,
// u (T u), |T u|^2, sum v, max u (all vectors >= 0). One pass over the four
// vectors instead of a dot and its sum each; the host adds the blocks in order.
constexpr int kDirSums = 8;
__global__ void __launch_bounds__(256)
k_dir_quality(int64_t n, const double *__restrict__ v, const double *__restrict__ vt, const double *__restrict__ u,
              const double *__restrict__ tu, double *__restrict__ part) {
  __shared__ double red[8][kDirSums];
  double s[kDirSums] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double a = v[i], b = vt[i], c = u[i], d = tu[i];
    s[0] += a * a;
    s[1] += a * b;
    s[2] += b * b;
    s[3] += c * c;
    s[4] += c * d;
    s[5] += d * d;
    s[6] += a;
    s[7] = c > s[7] ? c : s[7];
  }
#pragma unroll
  for (int q = 0; q < kDirSums; ++q) {
    for (int o = 16; o > 0; o >>= 1) {
      const double x = __shfl_xor_sync(0xffffffffu, s[q], o);
      s[q] = q < 7 ? s[q] + x : (x > s[q] ? x : s[q]);
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][q] = s[q];
  }
  __syncthreads();
  if (threadIdx.x < kDirSums) {
    double t = red[0][threadIdx.x];
    for (int w = 1; w < 8; ++w) {
      const double x = red[w][threadIdx.x];
      t = threadIdx.x < 7 ? t + x : (x > t ? x : t);
    }
    part[blockIdx.x * kDirSums + threadIdx.x] = t;
  }
}

// vy = v / dw (non-dangling), the inflow (dangling); u scaled to v u = 1, rounded to float
__global__ void k_dir_finish(int64_t n, const int64_t *__restrict__ orp, const double *__restrict__ invdw,
                             const double *__restrict__ v, const double *__restrict__ flow,
                             const double *__restrict__ u, double vu, float *__restrict__ vy, float *__restrict__ uf) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  vy[i] = (float)(orp[i] == orp[i + 1] ? flow[i] : v[i] * invdw[i]);
  uf[i] = (float)(u[i] / vu);
}
}  // namespace

// The dominant mode of the walk among the non-dangling nodes: left and right
// power iterations in FP64 (normalised every 8 steps), lambda by the two-sided
// Rayleigh quotient, then the decay of a hashed vector without that mode gives
// the rate of the rest. The pair is used only if it comes near a mode:
//  * the condition |v|_1 max u / (v u) at most kModeCondition: the start is that
//    many times the solution at most, so its FP32 rounding (2^-24 of it) stays
//    within the main solve's 1e-5. Without cycles (every eigenvalue 0) the
//    iterations leave no eigenvector and v u is a leftover: 1e24 and more on
//    acyclic power-law and random graphs, 1e6 with a few cycles in one, 1 to 66
//    where there is a mode to use. It also bounds u / (v u), which goes to FP32,
//    since |v|_1 >= |v|;
//  * |v T - lambda v| and |T u - lambda u| at most kModeResidual lambda |v|, |u|:
//    above 1 without cycles. A pair that is still on its way (1e-3 to 0.1 on
//    power-law graphs of few edges per node, whose next mode is nearly as slow)
//    takes most of the slow modes out of the start at the plain rate: 1 to 13 %
//    fewer sweeps on large graphs, 1 to 4 % more on small periodic ones.
// Otherwise, as for a walk without any mode, the solves start plainly.
constexpr double kModeResidual = 0.5, kModeCondition = 100.0;
int graph_perron(pprviz_ctx *ctx, const pprviz_graph *g) {
  if (g->per_ready) return PPRVIZ_OK;
  std::lock_guard<std::mutex> lock(g->lazy);
  if (g->per_ready) return PPRVIZ_OK;
  constexpr int STEPS = 40, DECAY = 8;
  const int64_t n = g->n;
  const unsigned nb = (unsigned)((n + 255) / 256), wb = (unsigned)((n * 32 + 255) / 256);
  PPRVIZ_CUDA(ctx, g->per_vy.ensure(sizeof(float) * (size_t)n));
  PPRVIZ_CUDA(ctx, g->per_u.ensure(sizeof(float) * (size_t)n));
  PPRVIZ_TRY(ws_ensure(ctx, WS_SPEC, sizeof(double) * (size_t)(4 * n + (1 + kDirSums) * kSpecBlocks + 8)));
  double *v = ctx->ws[WS_SPEC].as<double>(), *u = v + n, *z = u + n, *t = z + n, *part = t + n,
         *sc = part + kSpecBlocks, *qual = sc + 8;
  const int64_t *orp = g->rp.as<int64_t>();
  const double *invdw = g->invdw_d.as<double>();
  auto left = [&](const double *in, double *out, bool keep) -> int {
    PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH);
    k_dir_spmv<true><<<wb, 256, 0, ctx->stream>>>(n, orp, g->prp.as<int64_t>(), g->pcol.as<int32_t>(),
                                                  g->pws.as<float>(), invdw, in, out, keep);
    PPRVIZ_LAUNCHED(ctx);
    return PPRVIZ_OK;
  };
  auto right = [&](const double *in, double *out) -> int {
    PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH);
    k_dir_spmv<false><<<wb, 256, 0, ctx->stream>>>(n, orp, orp, g->col.as<int32_t>(),
                                                   g->weighted ? g->w.as<float>() : nullptr, invdw, in, out, false);
    PPRVIZ_LAUNCHED(ctx);
    return PPRVIZ_OK;
  };
  auto dot = [&](const double *a, const double *b, double *out) -> int {
    { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_dir_dot<<<kSpecBlocks, 256, 0, ctx->stream>>>(n, a, b, part); }
    PPRVIZ_LAUNCHED(ctx);
    { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_spec_sum<<<1, 256, 0, ctx->stream>>>(kSpecBlocks, part, out); }
    PPRVIZ_LAUNCHED(ctx);
    return PPRVIZ_OK;
  };
  auto start = [&](double *out, bool hashed) -> int {
    { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_dir_start<<<nb, 256, 0, ctx->stream>>>(n, orp, hashed, out); }
    PPRVIZ_LAUNCHED(ctx);
    return PPRVIZ_OK;
  };
  auto power = [&](double *x, bool is_left) -> int {
    PPRVIZ_TRY(start(x, false));
    for (int it = 0; it < STEPS; it += 2) {
      PPRVIZ_TRY(is_left ? left(x, t, false) : right(x, t));
      PPRVIZ_TRY(is_left ? left(t, x, false) : right(t, x));
      if (it % 8 == 6) {
        PPRVIZ_TRY(dot(x, x, sc));
        { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_spec_normalise<<<nb, 256, 0, ctx->stream>>>(n, sc, x); }
        PPRVIZ_LAUNCHED(ctx);
      }
    }
    return PPRVIZ_OK;
  };
  PPRVIZ_TRY(power(v, true));
  PPRVIZ_TRY(power(u, false));
  PPRVIZ_TRY(dot(v, u, sc));        // v u
  PPRVIZ_TRY(right(u, t));
  PPRVIZ_TRY(dot(v, t, sc + 1));    // v T u
  PPRVIZ_TRY(left(v, z, false));
  { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_dir_quality<<<kSpecBlocks, 256, 0, ctx->stream>>>(n, v, z, u, t, qual); }
  PPRVIZ_LAUNCHED(ctx);
  // the rest: DECAY steps to shed the fast modes, DECAY more are measured
  PPRVIZ_TRY(start(z, true));
  auto project = [&]() -> int {
    PPRVIZ_TRY(dot(z, u, sc + 2));
    { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_dir_project<<<nb, 256, 0, ctx->stream>>>(n, sc + 2, sc, v, z); }
    PPRVIZ_LAUNCHED(ctx);
    return PPRVIZ_OK;
  };
  for (int half = 0; half < 2; ++half) {
    PPRVIZ_TRY(project());
    for (int it = 0; it < DECAY; it += 2) {
      PPRVIZ_TRY(left(z, t, false));
      PPRVIZ_TRY(left(t, z, false));
    }
    PPRVIZ_TRY(project());
    PPRVIZ_TRY(dot(z, z, sc + 3 + half));
  }
  PPRVIZ_TRY(left(v, t, true));  // what the left vector sends to the dangling nodes
  double hs[5] = {0, 0, 0, 0, 0};
  std::vector<double> hq((size_t)kSpecBlocks * kDirSums);
  PPRVIZ_CUDA(ctx, cudaMemcpyAsync(hs, sc, sizeof(hs), cudaMemcpyDeviceToHost, ctx->stream));
  PPRVIZ_CUDA(ctx, cudaMemcpyAsync(hq.data(), qual, sizeof(double) * hq.size(), cudaMemcpyDeviceToHost, ctx->stream));
  PPRVIZ_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  double q[kDirSums] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (int b = 0; b < kSpecBlocks; ++b)
    for (int e = 0; e < kDirSums; ++e) {
      const double x = hq[(size_t)b * kDirSums + e];
      q[e] = e < 7 ? q[e] + x : std::max(q[e], x);
    }
  const double lambda = hs[0] > 0.0 ? hs[1] / hs[0] : 0.0;
  // (comparisons that a NaN fails)
  auto settled = [lambda](double xx, double xy, double yy) {  // |y - lambda x| <= kModeResidual lambda |x|
    return xx > 0.0 && yy - 2.0 * lambda * xy + lambda * lambda * xx <= kModeResidual * kModeResidual * lambda * lambda * xx;
  };
  const double decay = hs[3] > 0.0 && hs[4] >= 0.0 ? pow(hs[4] / hs[3], 0.5 / DECAY) : 1.0;
  const double rest = 1.05 * decay + 0.02;  // estimate + margin
  g->per_ok = lambda > 1e-3 && lambda < 1.0 + 1e-9 && settled(q[0], q[1], q[2]) && settled(q[3], q[4], q[5]) &&
              q[6] * q[7] <= kModeCondition * hs[0];
  g->per_b = 1.0;
  if (g->per_ok) {
    g->per_lambda = std::min(lambda, 1.0);
    g->per_b = std::min(1.0, rest);
    { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_dir_finish<<<nb, 256, 0, ctx->stream>>>(
        n, orp, invdw, v, t, u, hs[0], g->per_vy.as<float>(), g->per_u.as<float>()); }
    PPRVIZ_LAUNCHED(ctx);
    g->h_u.resize((size_t)n);
    PPRVIZ_CUDA(ctx, cudaMemcpyAsync(g->h_u.data(), g->per_u.p, sizeof(float) * (size_t)n, cudaMemcpyDeviceToHost,
                                     ctx->stream));
    PPRVIZ_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  }
  g->per_ready = true;
  return PPRVIZ_OK;
}

int graph_spectral(pprviz_ctx *ctx, const pprviz_graph *g) {
  if (g->spec_ready) return PPRVIZ_OK;
  std::lock_guard<std::mutex> lock(g->lazy);
  if (g->spec_ready) return PPRVIZ_OK;
  const int64_t n = g->n;
  const unsigned nb = (unsigned)((n + 255) / 256), wb = (unsigned)((n * 32 + 255) / 256);
  PPRVIZ_CUDA(ctx, g->comp.ensure(sizeof(int32_t) * (size_t)n));
  PPRVIZ_TRY(ws_ensure(ctx, WS_SPEC, sizeof(double) * (size_t)(3 * n + kSpecBlocks + 8)));
  PPRVIZ_TRY(ws_ensure(ctx, WS_FLAG, 64));
  int32_t *parent = g->comp.as<int32_t>();
  int *changed = ctx->ws[WS_FLAG].as<int>();
  const int64_t *rp = g->rp.as<int64_t>();
  const int32_t *col = g->col.as<int32_t>();
  const float *w = g->weighted ? g->w.as<float>() : nullptr;
  const double *invdw = g->invdw_d.as<double>();

  // |lambda| <= b off the stationary modes, from <v, v>_D and <P v, P v>_D
  auto bound = [&](bool resolved, double vv, double pp) {
    double b = 1.0;
    if (!resolved) {
      b = 1.0;  // components unresolved: keep the full interval and no deflation
    } else if (vv > 0.0 && std::isfinite(vv) && std::isfinite(pp)) {
      b = std::min(1.0, 1.05 * sqrt(std::max(0.0, pp / vv)) + 0.02);
    } else {
      b = 0.02;  // no non-stationary mode reached: every component is trivial
    }
    g->spec_b = b;
    g->spec_deflate = resolved;
    g->spec_ready = true;
  };
  // One SM's rate against launches: 150 nodes and 3,000 edges 212 us (311 by the
  // separate kernels), 12,000 edges 282 (333); 400 nodes and 4,000 edges 296
  // (316), 8,000 edges 367 (319); 1,000 nodes and 5,000 edges 490 (335). The
  // line 16 n + edges = 12,000 keeps to the side where the one launch is faster.
  if (n <= kSpecSmall && 16 * n + g->nnz <= 12000) {
    double *out = ctx->ws[WS_SPEC].as<double>();
    { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_spec_small<<<1, 1024, 0, ctx->stream>>>((int)n, rp, col, w, invdw, parent, out); }
    PPRVIZ_LAUNCHED(ctx);
    std::vector<double> h((size_t)(3 + n + (n + 1) / 2));
    PPRVIZ_CUDA(ctx, cudaMemcpyAsync(h.data(), out, sizeof(double) * h.size(), cudaMemcpyDeviceToHost, ctx->stream));
    PPRVIZ_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    g->h_comp.resize((size_t)n);
    memcpy(g->h_comp.data(), h.data() + 3 + n, sizeof(int32_t) * (size_t)n);
    g->h_mc.assign((size_t)n, 0.0);
    for (int64_t i = 0; i < n; ++i) g->h_mc[(size_t)g->h_comp[i]] += 1.0 / h[(size_t)(3 + i)];
    bound(h[2] != 0.0, h[0], h[1]);
    return PPRVIZ_OK;
  }

  // ---- connected components
  { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_cc_init<<<nb, 256, 0, ctx->stream>>>(n, parent); }
  PPRVIZ_LAUNCHED(ctx);
  bool done = false;
  for (int round = 0; round < kCcMaxRounds && !done; ++round) {
    PPRVIZ_CUDA(ctx, cudaMemsetAsync(changed, 0, sizeof(int), ctx->stream));
    { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_cc_hook<<<wb, 256, 0, ctx->stream>>>(n, rp, col, parent, changed); }
    PPRVIZ_LAUNCHED(ctx);
    { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_cc_compress<<<nb, 256, 0, ctx->stream>>>(n, parent); }
    PPRVIZ_LAUNCHED(ctx);
    int hc = 0;
    PPRVIZ_CUDA(ctx, cudaMemcpyAsync(&hc, changed, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    PPRVIZ_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    done = hc == 0;
  }
  g->h_comp.resize((size_t)n);
  std::vector<double> h_invdw((size_t)n);
  PPRVIZ_CUDA(ctx, cudaMemcpyAsync(g->h_comp.data(), parent, sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToHost,
                                   ctx->stream));
  PPRVIZ_CUDA(ctx, cudaMemcpyAsync(h_invdw.data(), invdw, sizeof(double) * (size_t)n, cudaMemcpyDeviceToHost,
                                   ctx->stream));
  PPRVIZ_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  // m_C per root, summed in node order (the stationary vector's normaliser)
  g->h_mc.assign((size_t)n, 0.0);
  for (int64_t i = 0; i < n; ++i) g->h_mc[(size_t)g->h_comp[i]] += 1.0 / h_invdw[(size_t)i];

  // ---- spectral bound of the non-stationary modes
  double *va = ctx->ws[WS_SPEC].as<double>(), *vb = va + n, *part = va + 3 * n, *scal = part + kSpecBlocks;
  { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_spec_spmv<<<wb, 256, 0, ctx->stream>>>(n, rp, col, w, invdw, nullptr, va); }
  PPRVIZ_LAUNCHED(ctx);
  for (int it = 0; it < kSpecIters; ++it) {
    { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_spec_spmv<<<wb, 256, 0, ctx->stream>>>(n, rp, col, w, invdw, va, vb); }
    PPRVIZ_LAUNCHED(ctx);
    { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_spec_spmv<<<wb, 256, 0, ctx->stream>>>(n, rp, col, w, invdw, vb, va); }
    PPRVIZ_LAUNCHED(ctx);
    if (it % 4 == 3) {
      { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_spec_dot<<<kSpecBlocks, 256, 0, ctx->stream>>>(n, invdw, va, va, part); }
      PPRVIZ_LAUNCHED(ctx);
      { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_spec_sum<<<1, 256, 0, ctx->stream>>>(kSpecBlocks, part, scal); }
      PPRVIZ_LAUNCHED(ctx);
      { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_spec_normalise<<<nb, 256, 0, ctx->stream>>>(n, scal, va); }
      PPRVIZ_LAUNCHED(ctx);
    }
  }
  { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_spec_spmv<<<wb, 256, 0, ctx->stream>>>(n, rp, col, w, invdw, va, vb); }
  PPRVIZ_LAUNCHED(ctx);
  { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_spec_dot<<<kSpecBlocks, 256, 0, ctx->stream>>>(n, invdw, va, va, part); }
  PPRVIZ_LAUNCHED(ctx);
  { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_spec_sum<<<1, 256, 0, ctx->stream>>>(kSpecBlocks, part, scal); }
  PPRVIZ_LAUNCHED(ctx);
  { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_spec_dot<<<kSpecBlocks, 256, 0, ctx->stream>>>(n, invdw, vb, vb, part); }
  PPRVIZ_LAUNCHED(ctx);
  { PPRVIZ_PROF(ctx, PPRVIZ_K_GRAPH); k_spec_sum<<<1, 256, 0, ctx->stream>>>(kSpecBlocks, part, scal + 1); }
  PPRVIZ_LAUNCHED(ctx);
  double hs[2] = {0.0, 0.0};
  PPRVIZ_CUDA(ctx, cudaMemcpyAsync(hs, scal, sizeof(hs), cudaMemcpyDeviceToHost, ctx->stream));
  PPRVIZ_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  bound(done, hs[0], hs[1]);
  return PPRVIZ_OK;
}

}  // namespace pprviz
