// P4/P5/P6 - stress energy, gradients and stress-majorization layout.
//
// Paper (Sec. 5, Eq. (7); Appendix A.1, Eqs. (8)-(10)):
//   L(X | Delta) = sum_{i<j} (1 - |X_i - X_j| / Delta_ij)^2
//   L^w[i][j] = -1/Delta_ij^2 (i != j), L^w[i][i] = sum_{k != i} 1/Delta_ik^2
//   L^Y[i][j] = -1/(Delta_ij |Y_i - Y_j|) (i != j, Y_i != Y_j), L^Y[i][i] = -row sum
//   X <- (L^w)^-1 L^Y(Y) Y                                    (Eq. (10))
//
// GB300 design:
//  * L^w does not depend on X, so it is inverted once per view. L^w is a
//    Laplacian (singular on the ones vector); A = L^w + J/k is SPD with
//    A 1 = 1, and for b = L^Y Y (zero column sums) A^-1 b is exactly the
//    centred Moore-Penrose solution. A is inverted once in place by the
//    symmetric block sweep of factor.cu.
//  * The layout works on the symmetric part Delta_s = (Delta + Delta^T)/2 (equal
//    to Delta for the symmetric PDist of Eq. (1)), so 1/Delta_s and M = A^-1 are
//    symmetric and each update reads only their upper-triangle 128 x 128 tiles:
//    a tile (I, J), I < J, adds its row sums to rows I and its column sums to
//    rows J. Two streaming passes per update (b = L^Y X over 1/Delta_s, then
//    X = M b) read half of each k x k matrix once. Partial sums are written
//    per (tile, row) and added in a fixed order: no atomics, reproducible.
//  * The energy and its gradients recompute every pair from X and Delta; no
//    k x k intermediate is stored.
#include <cuda.h>
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "recip.cuh"

namespace pprviz {

constexpr int ST = 128;       // symmetric pass tile edge

template <typename T> struct T2;
template <> struct T2<float> { using type = float2; };
template <> struct T2<double> { using type = double2; };

// ---------------------------------------------------------------------------
// Build from Delta_s = (Delta + Delta^T) / 2, in 32 x 32 tiles with the mirrored
// tile staged in shared memory:
//   W1[i][j] = 1/Delta_s (0 on the diagonal and in the padding),
//   A[i][j]  = 1/k - 1/Delta_s^2 off the diagonal, identity on padded rows,
//   rowpart[J][i] = sum over the tile's 32 columns of 1/Delta_s^2 (FP64);
// k_build_diag then sets A[i][i] = sum_J rowpart[J][i] + 1/k in a fixed order.
// Every consumer reads the upper triangle of 128-row blocks (diagonal 128
// blocks in full), so tiles below the diagonal 128 blocks are not written: the
// mirrored tile above supplies their row sums as its column sums (W1 and A are
// symmetric entry by entry), and checks the mirrored inputs. One thread per row
// and column adds the tile's squares (one FP64 shuffle sum per element bounded
// the pass on the FP64 pipe): k = 10,000 (0.8 GB), 891 -> 228 us.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ T recip(T d) { return T(1) / d; }
template <>
__device__ __forceinline__ float recip<float>(float d) { return __frcp_rn(d); }

// Sum of 32 values p[0], p[stride], ...: FP64 additions, or, for floats, a float
// sum with its exact rounding errors (TwoSum, Knuth), good to ~2^-50 of the sum
// (it becomes part of an FP32 diagonal entry) and off GB300's narrow FP64 pipe.
__device__ __forceinline__ double sum32(const double *p, int stride) {
  double s = 0.0;
  for (int e = 0; e < 32; ++e) s += p[e * stride];
  return s;
}
__device__ __forceinline__ double sum32(const float *p, int stride) {
  float s = 0.0f, c = 0.0f;
#pragma unroll
  for (int e = 0; e < 32; ++e) {
    const float q = p[e * stride];
    const float t = __fadd_rn(s, q);
    const float bb = __fsub_rn(t, s);
    c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, bb)), __fsub_rn(q, bb)));
    s = t;
  }
  return (double)s + (double)c;
}

template <typename TI, typename T>
__global__ void k_build_sym(int32_t k, int32_t kp, const TI *__restrict__ D, T *__restrict__ W1,
                            T *__restrict__ A, double *__restrict__ rowpart, int *__restrict__ flag) {
  const int by = blockIdx.y, bx = blockIdx.x;
  if ((by >> 2) > (bx >> 2)) return;  // below the diagonal 128 blocks
  const bool mirror = (by >> 2) < (bx >> 2);
  __shared__ TI tr[32][33];
  __shared__ T sq[32][33];  // 1/Delta_s^2
  const int i0 = by * 32, j0 = bx * 32;
  const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
  TI own[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int jj = ty + 8 * e, j = j0 + jj, i = i0 + tx;
    tr[jj][tx] = (j < k && i < k) ? D[(int64_t)j * k + i] : TI(0);
    const int io = i0 + jj, jo = j0 + tx;
    own[e] = (io < k && jo < k) ? D[(int64_t)io * k + jo] : TI(0);
  }
  __syncthreads();
  const T invk = (T)(1.0 / (double)k);
  int bad = 0;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int ii = ty + 8 * e, i = i0 + ii, j = j0 + tx;
    T wsq = T(0);
    if (i < k && j < k && i != j) {
      const TI a = own[e], b = tr[tx][ii];
      // every input entry must itself be a valid distance (this element checks
      // a; b is checked by the element (j, i), or here when that tile is not built)
      if (!(a > TI(0)) || !isfinite(a)) bad = 1;
      if (mirror && (!(b > TI(0)) || !isfinite(b))) bad = 1;
      const T d = (T)((a + b) * TI(0.5));
      const T w1 = recip(d);
      wsq = w1 * w1;
      W1[(int64_t)i * kp + j] = w1;
      A[(int64_t)i * kp + j] = invk - wsq;
    } else {
      W1[(int64_t)i * kp + j] = T(0);
      if (i != j || i >= k) A[(int64_t)i * kp + j] = (i == j) ? T(1) : T(0);
    }
    sq[ii][tx] = wsq;
  }
  __syncthreads();
  if (ty == 0) rowpart[(int64_t)bx * kp + i0 + tx] = sum32(&sq[tx][0], 1);
  // the row sums of the tile (bx, by) below: this tile's column sums
  if (mirror && ty == 1) rowpart[(int64_t)by * kp + j0 + tx] = sum32(&sq[0][tx], 33);
  if (bad) atomicOr(flag, 1);
}

template <typename T>
__global__ void k_build_diag(int32_t k, int32_t kp, const double *__restrict__ rowpart, T *__restrict__ A) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= k) return;
  double s = 0.0;
  for (int b = 0; b < kp / 32; ++b) s += rowpart[(int64_t)b * kp + i];
  A[(int64_t)i * kp + i] = (T)(s + 1.0 / (double)k);
}

// ---------------------------------------------------------------------------
// FP64 symmetric pair pass over the upper-triangle ST64 x ST64 tiles of a
// symmetric kp x kp matrix Mat (zero beyond k), one CTA per tile (I, J), I <= J,
// 8 warps: warp w owns tile rows 8w..8w+7, lane l the columns 2l and 2l + 1.
// With v = the vector (x for MODE 0, b for MODE 1):
//   MODE 0 (L^Y): t_ij = Mat_ij (v_i - v_j) / |v_i - v_j|; row i gets +t_ij,
//                 column j gets -t_ij (since t_ji = -t_ij)
//   MODE 1 (apply M): row i gets Mat_ij v_j, column j gets Mat_ij v_i
// Row sums go to Part[J][i], column sums (off-diagonal tiles only) to Part[I][j].
// Bound by the FP64 pipe (2 operations per cycle and SM; 15 per pair in MODE 0,
// 5 in MODE 1), so what counts is that every SM has a tile: 64 x 64 tiles give
// a view of 1,000 nodes 136 CTAs (128 x 128 gave it 36). The tile is loaded
// before the wait for the previous pass (programmatic dependent launch).
// k = 1,000: one update (both passes) 137 -> 39 us, of which the FP64 pipe needs
// about 21.
// ---------------------------------------------------------------------------
constexpr int ST64 = 64;

// The halving steps of lanes_transpose_sum: value index lane / (32 / NV) summed
// over the lanes of equal lane % (32 / NV).
template <int NV, typename T>
__device__ __forceinline__ T lanes_fold(T (&v)[NV], int lane) {
  constexpr int LOG = NV == 32 ? 5 : NV == 16 ? 4 : NV == 8 ? 3 : NV == 4 ? 2 : NV == 2 ? 1 : 0;
#pragma unroll
  for (int s = 0; s < LOG; ++s) {
    const int off = 16 >> s;
    const int half = (NV >> s) / 2;
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const T send = up ? v[i] : v[i + half];
      const T keep = up ? v[i + half] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
  return v[0];
}

// Sum over the 32 lanes of NV values per lane; returns, in every lane, the
// total of value index lane / (32 / NV). Recursive halving: 31 shuffles for
// NV = 32, 15 + 1 for NV = 16.
template <int NV, typename T>
__device__ __forceinline__ T lanes_transpose_sum(T (&v)[NV], int lane) {
  constexpr int LOG = NV == 32 ? 5 : NV == 16 ? 4 : NV == 8 ? 3 : NV == 4 ? 2 : NV == 2 ? 1 : 0;
  T r = lanes_fold<NV, T>(v, lane);
#pragma unroll
  for (int off = 16 >> LOG; off > 0; off >>= 1) r += __shfl_xor_sync(0xffffffffu, r, off);
  return r;
}

// sum_{o < nb} p[o * kp] in order o = 0, 1, ...; the loads (L2, since other
// CTAs wrote them) are issued 4 at a time so that their latencies overlap,
// the additions keep the order
template <typename V2>
__device__ __forceinline__ V2 sum_parts_in_order(const V2 *p, int64_t kp, int nb) {
  V2 s = __ldcg(p);
  for (int o0 = 1; o0 < nb; o0 += 4) {
    V2 u[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (o0 + q < nb) u[q] = __ldcg(p + (int64_t)(o0 + q) * kp);
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (o0 + q < nb) {
        s.x += u[q].x;
        s.y += u[q].y;
      }
  }
  return s;
}

// After its partial sums are written, the tile counts itself in for row
// block I (and, off the diagonal, for row block J); every row block receives
// exactly nbt partials (one per slot), so the CTA that brings a block's count
// to nbt sums that block's partials in slot order into Vout and resets the
// count for the next pass (a deterministic result, independent of which CTA
// finishes last). One thread per CTA fences after the block barrier before
// counting (release) and after a last count (acquire); the reducer reads
// through L2.
template <int MODE>
__global__ void __launch_bounds__(256)
k_sympass64(int32_t kp, int nbt, const int2 *__restrict__ tiles, const double *__restrict__ Mat, const double2 *V,
            double2 *Part, int *cnt, double2 *Vout) {
  constexpr int RPW64 = 8;
  __shared__ double2 sVi[ST64];
  __shared__ double colred[8][2 * ST64];
  __shared__ int last[2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int I = tiles[blockIdx.x].x, J = tiles[blockIdx.x].y;
  const int64_t i0 = (int64_t)I * ST64, j0 = (int64_t)J * ST64;
  double2 m[RPW64];
#pragma unroll
  for (int r = 0; r < RPW64; ++r)
    m[r] = __ldg(reinterpret_cast<const double2 *>(Mat + (i0 + warp * RPW64 + r) * kp + j0) + lane);
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the previous pass's vector and partials
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (threadIdx.x < ST64) sVi[threadIdx.x] = __ldcg(V + i0 + threadIdx.x);
  const double2 va = __ldcg(V + j0 + 2 * lane), vb = __ldcg(V + j0 + 2 * lane + 1);
  __syncthreads();
  double cx[2] = {0.0, 0.0}, cy[2] = {0.0, 0.0}, acc[2 * RPW64];
#pragma unroll
  for (int r = 0; r < RPW64; ++r) {
    const double2 vi = sVi[warp * RPW64 + r];
    double ax, ay;
    if (MODE == 0) {
      const double dxa = vi.x - va.x, dya = vi.y - va.y, dxb = vi.x - vb.x, dyb = vi.y - vb.y;
      const double ca = m[r].x * rsqrt_pos(fma(dxa, dxa, dya * dya));
      const double cb = m[r].y * rsqrt_pos(fma(dxb, dxb, dyb * dyb));
      ax = fma(cb, dxb, ca * dxa);
      ay = fma(cb, dyb, ca * dya);
      cx[0] = fma(-ca, dxa, cx[0]);
      cy[0] = fma(-ca, dya, cy[0]);
      cx[1] = fma(-cb, dxb, cx[1]);
      cy[1] = fma(-cb, dyb, cy[1]);
    } else {
      ax = fma(m[r].y, vb.x, m[r].x * va.x);
      ay = fma(m[r].y, vb.y, m[r].x * va.y);
      cx[0] = fma(m[r].x, vi.x, cx[0]);
      cy[0] = fma(m[r].x, vi.y, cy[0]);
      cx[1] = fma(m[r].y, vi.x, cx[1]);
      cy[1] = fma(m[r].y, vi.y, cy[1]);
    }
    acc[2 * r] = ax;
    acc[2 * r + 1] = ay;
  }
  double *part = reinterpret_cast<double *>(Part);
  const double tot = lanes_transpose_sum<2 * RPW64, double>(acc, lane);
  if (lane % 2 == 0) part[((int64_t)J * kp + i0 + warp * RPW64) * 2 + lane / 2] = tot;
  if (I != J) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      colred[warp][(lane * 2 + u) * 2] = cx[u];
      colred[warp][(lane * 2 + u) * 2 + 1] = cy[u];
    }
    __syncthreads();
    if (threadIdx.x < 2 * ST64) {
      double s = 0.0;
#pragma unroll
      for (int w = 0; w < 8; ++w) s += colred[w][threadIdx.x];
      part[((int64_t)I * kp + j0) * 2 + threadIdx.x] = s;
    }
  }
  __syncthreads();  // every thread's partials are written (CTA scope)
  if (threadIdx.x == 0) {
    __threadfence();  // release, cumulative over the barrier
    last[0] = atomicAdd(&cnt[I], 1) == nbt - 1;
    last[1] = (I != J) ? (atomicAdd(&cnt[J], 1) == nbt - 1) : 0;
    if (last[0] || last[1]) __threadfence();  // acquire before the block reads other CTAs' partials
  }
  __syncthreads();
  // threads 0..63 reduce row block I, threads 64..127 row block J
  if (threadIdx.x < 2 * ST64) {
    const int side = threadIdx.x / ST64;
    if (last[side]) {
      const int R = side ? J : I;
      const int64_t row = (int64_t)R * ST64 + threadIdx.x % ST64;
      Vout[row] = sum_parts_in_order(Part + row, (int64_t)kp, nbt);
      if (threadIdx.x % ST64 == 0) cnt[R] = 0;
    }
  }
}

// Views of a pass: a view's matrix, vector and partial-sum slices.
// A single view is the case of one descriptor.
struct BatchView {
  int64_t mat_off;   // elements into the batched kp x kp matrices
  int64_t vec_off;   // 2-vectors into the batched coordinate / b vectors (kp each)
  int64_t part_off;  // 2-vectors into the batched partial sums (nbt x kp each)
  int32_t kp, nbt, k;
};

// ---------------------------------------------------------------------------
// FP32 symmetric pass, persistent, pipelined and warp-specialized (the FP32
// path of the single and the batched layout). One CTA per SM: a producer warp
// and 16 consumer warps. Each CTA takes a contiguous chunk of the tile table,
// which lists every view's upper-triangle tiles column by column (J, then
// I = 0..J). The producer brings each 128 x 128 tile (64 KiB) into a
// shared-memory stage with one TMA tensor copy (cp.async.bulk.tensor.2d; a
// tensor map per view and matrix), together with the two 1 KiB coordinate
// slices it needs (plain bulk copies), all completing on the stage's "full"
// mbarrier; it refills a stage once the stage's "empty" mbarrier has seen all
// 16 consumer warps. With PS stages the copies of PS tiles are in flight.
// The consumer warps never wait for each other: warp w takes tile rows
// 8w..8w+7 (lane l the columns 4l..4l+3, one conflict-free 16-byte
// shared-memory read per row), sums its rows across lanes and stores them per
// tile (row block I, slot J), and keeps its column sums in registers while
// consecutive tiles of the chunk share the column block J (a "run"); it
// writes them once per run to the run's slot. A separate launch
// (k_reduce_rows) adds slots and runs in a fixed order. Per pair:
//   MODE 0 (L^Y): t_ij = Mat_ij (v_i - v_j) / |v_i - v_j|: row i +t, column j -t
//   MODE 1 (apply M): row i gets Mat_ij v_j, column j gets Mat_ij v_i
// (the diagonal tile adds its rows only: it is stored in full). Lane l's four
// columns are processed as two pairs with Blackwell's paired FP32
// instructions (two lanes of work per issue slot).
// Every mbarrier wait has an iteration limit: on expiry the warp sets *err and
// stops; the producer then waits (again bounded) for the copies it issued.
// ---------------------------------------------------------------------------
namespace spipe {
constexpr int PS = 3;                           // pipeline stages
constexpr int CWARPS = 16;                      // consumer warps
constexpr int THREADS = (CWARPS + 1) * 32;      // + the producer warp
constexpr int PRW = ST / CWARPS;                // tile rows per consumer warp
constexpr uint32_t TILE_BYTES = ST * ST * 4;    // one FP32 tile
constexpr uint32_t VEC_BYTES = ST * 8;          // 128 coordinate pairs
constexpr uint32_t STAGE_BYTES = TILE_BYTES + 2 * VEC_BYTES;  // tile, rows' and columns' vector slices
constexpr int SMEM = PS * (int)STAGE_BYTES + 1024;  // stages + alignment slack
constexpr long WAIT_LIMIT = 1L << 24;           // mbarrier polls before giving up

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity) {
  uint32_t done = 0;
  for (long it = 0; it < WAIT_LIMIT && !done; ++it) {
    asm volatile(
        "{\n\t.reg .pred q;\n\tmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\n\tselp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
  }
  return done != 0;
}

// One thread: tile (I, J) of the matrix behind `map` and the vector slices
// V[I 128 ..] and V[J 128 ..] (V is the view's vector) into the stage at dst,
// all completing on bar (armed with their byte count first). The maps sit in
// global memory, written by a host copy before the launch; the first use of
// each map by a CTA is preceded by a tensor-map acquire fence (`fenced`
// remembers the last map fenced).
__device__ __forceinline__ void tile_copy(uint32_t dst, uint32_t b, const CUtensorMap *map, int I, int J,
                                          uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint "
      "[%0], [%1, {%2, %3}], [%4], %5;" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(J * ST), "r"(I * ST), "r"(b), "l"(policy)
      : "memory");
}

__device__ __forceinline__ void issue_tile(uint32_t dst, uint64_t *bar, const CUtensorMap *map, const float2 *V,
                                           int I, int J, const CUtensorMap *&fenced, uint64_t policy) {
  if (map != fenced) {
    asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(reinterpret_cast<uint64_t>(map))
                 : "memory");
    fenced = map;
  }
  const uint32_t b = smem_u32(bar);
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(STAGE_BYTES) : "memory");
  tile_copy(dst, b, map, I, J, policy);
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   dst + TILE_BYTES),
               "l"(V + (int64_t)I * ST), "r"(VEC_BYTES), "r"(b)
               : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   dst + TILE_BYTES + VEC_BYTES),
               "l"(V + (int64_t)J * ST), "r"(VEC_BYTES), "r"(b)
               : "memory");
}

// 1/sqrt(max(d2, 2^-100)) on the special-function unit. For coincident points
// (d2 = 0) the pair's dx, dy are 0, so its term is 0, as the L^Y definition
// sets it; padding entries carry a zero matrix entry.
__device__ __forceinline__ float rsqrt_clamped(float d2) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(fmaxf(d2, 0x1p-100f)));
  return r;
}
}  // namespace spipe

// A tile of the FP32 pass: view v, tile (I, J) of its kp x kp matrices, the
// view's vector offset / 128, its row-sum slots (2-vectors) and the run slot
// of its column sums (-1 for a diagonal tile).
struct __align__(16) TileRec {
  int32_t v, I, J, vblk;
  int32_t kp, run;
  int64_t part_off;
};

// Run slot r holds, per consumer warp w, that warp's column sums of the run:
// RunPart[(r CWARPS + w) 128 + c], c the column within block J.
template <int MODE>
__global__ void __launch_bounds__(spipe::THREADS, 1)
k_sympass_pipe(int ntile, int npin /* per CTA */, const TileRec *__restrict__ tiles, const CUtensorMap *__restrict__ maps,
               const float2 *__restrict__ V, float2 *__restrict__ Part, float2 *__restrict__ RunPart,
               int *__restrict__ err) {
  using namespace spipe;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full[PS], empty[PS];
  __shared__ TileRec srec[PS];  // the record of the tile in each stage, written by the producer
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int first = (int)((int64_t)blockIdx.x * ntile / gridDim.x);
  const int mine = (int)((int64_t)(blockIdx.x + 1) * ntile / gridDim.x) - first;
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;  // TMA destinations 1024-byte aligned
  const unsigned char *sgen = smem_raw + (sbase - smem_u32(smem_raw));
  if (threadIdx.x == 0) {
    for (int s = 0; s < PS; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&full[s])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&empty[s])), "r"(CWARPS));
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();  // the only CTA-wide barrier
  // the launch that follows (the reduce) may be scheduled from now on; it
  // waits for this grid's completion itself
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (warp == CWARPS) {
    // ---- producer
    if (lane == 0) {
      const CUtensorMap *fenced = nullptr;
      // L2 policies: the first npin tiles of every CTA's chunk stay resident
      // across passes (evict_last), so that each CTA reads the same share
      // from L2; the rest stream through (evict_first)
      uint64_t keep, stream;
      asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(keep));
      asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(stream));
      // The matrix tiles do not depend on the previous launch: the first PS
      // are requested before waiting for it (expect_tx without the arrival,
      // so the stage cannot complete early); their vector slices, which the
      // previous launch writes, after it.
      const int npre = mine < PS ? mine : PS;
      for (int n = 0; n < npre; ++n) {
        const TileRec t = tiles[first + n];
        const CUtensorMap *map = maps + 2 * t.v + MODE;
        if (map != fenced) {
          asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(reinterpret_cast<uint64_t>(map))
                       : "memory");
          fenced = map;
        }
        const uint32_t b = smem_u32(&full[n]);
        asm volatile("mbarrier.expect_tx.shared::cta.b64 [%0], %1;" ::"r"(b), "r"(TILE_BYTES) : "memory");
        tile_copy(sbase + (uint32_t)n * STAGE_BYTES, b, map, t.I, t.J, n < npin ? keep : stream);
      }
      asm volatile("griddepcontrol.wait;" ::: "memory");
      for (int n = 0; n < npre; ++n) {
        const TileRec t = tiles[first + n];
        const float2 *Vv = V + (int64_t)t.vblk * ST;
        const uint32_t dst = sbase + (uint32_t)n * STAGE_BYTES, b = smem_u32(&full[n]);
        srec[n] = t;  // released to the consumers by the arrive below
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(2 * VEC_BYTES) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         dst + TILE_BYTES),
                     "l"(Vv + (int64_t)t.I * ST), "r"(VEC_BYTES), "r"(b)
                     : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         dst + TILE_BYTES + VEC_BYTES),
                     "l"(Vv + (int64_t)t.J * ST), "r"(VEC_BYTES), "r"(b)
                     : "memory");
      }
      int issued = npre;
      bool ok = true;
      for (int n = npre; n < mine; ++n) {
        const int s = n % PS;
        const TileRec t = tiles[first + n];
        if (!mbar_wait(&empty[s], (uint32_t)(((n - PS) / PS) & 1))) {
          ok = false;
          break;
        }
        srec[s] = t;  // released to the consumers by the arrive below
        issue_tile(sbase + (uint32_t)s * STAGE_BYTES, &full[s], maps + 2 * t.v + MODE, V + (int64_t)t.vblk * ST, t.I,
                   t.J, fenced, n < npin ? keep : stream);
        issued = n + 1;
      }
      if (!ok) {
        atomicOr(err, 1);
        // copies of the last PS issued tiles may still be landing
        for (int n = issued > PS ? issued - PS : 0; n < issued; ++n)
          (void)mbar_wait(&full[n % PS], (uint32_t)((n / PS) & 1));
      }
    }
    return;
  }
  // ---- consumers
  const int rbase = warp * PRW;
  const float sg = MODE == 0 ? -1.0f : 1.0f;
  float2 rxA = make_float2(0.0f, 0.0f), rxB = rxA, ryA = rxA, ryB = rxA;  // column sums of the current run
  int cur_run = -1;
#pragma unroll 1
  for (int n = 0; n < mine; ++n) {
    const int s = n % PS;
    if (!mbar_wait(&full[s], (uint32_t)((n / PS) & 1))) {
      if (lane == 0) atomicOr(err, 1);
      return;
    }
    const TileRec t = srec[s];
    if (t.run != cur_run) {
      if (cur_run >= 0) {
        float4 *o = reinterpret_cast<float4 *>(RunPart + ((int64_t)cur_run * CWARPS + warp) * ST + lane * 4);
        o[0] = make_float4(sg * rxA.x, sg * ryA.x, sg * rxA.y, sg * ryA.y);
        o[1] = make_float4(sg * rxB.x, sg * ryB.x, sg * rxB.y, sg * ryB.y);
      }
      rxA = rxB = ryA = ryB = make_float2(0.0f, 0.0f);
      cur_run = t.run;
    }
    const unsigned char *stage = sgen + (size_t)s * STAGE_BYTES;
    const float *stile = reinterpret_cast<const float *>(stage) + rbase * ST + lane * 4;
    const float2 *svi = reinterpret_cast<const float2 *>(stage + TILE_BYTES) + rbase;
    const float4 *svj = reinterpret_cast<const float4 *>(stage + TILE_BYTES + VEC_BYTES) + lane * 2;
    // columns 4l..4l+3 as pairs A = (4l, 4l+1), B = (4l+2, 4l+3); MODE 0 keeps
    // the column coordinates negated
    const float4 c01 = svj[0], c23 = svj[1];  // (x0, y0, x1, y1), (x2, y2, x3, y3)
    const float2 xA = make_float2(sg * c01.x, sg * c01.z), yA = make_float2(sg * c01.y, sg * c01.w);
    const float2 xB = make_float2(sg * c23.x, sg * c23.z), yB = make_float2(sg * c23.y, sg * c23.w);
    float2 cxA = make_float2(0.0f, 0.0f), cxB = cxA, cyA = cxA, cyB = cxA;
    float acc[2 * PRW];
#pragma unroll
    for (int r = 0; r < PRW; ++r) {
      const float4 m4 = *reinterpret_cast<const float4 *>(stile + r * ST);
      const float2 vi = svi[r];
      const float2 mA = make_float2(m4.x, m4.y), mB = make_float2(m4.z, m4.w);
      const float2 vx = make_float2(vi.x, vi.x), vy = make_float2(vi.y, vi.y);
      float2 ra, rb;
      if (MODE == 0) {
        const float2 dxA = __fadd2_rn(vx, xA), dyA = __fadd2_rn(vy, yA);
        const float2 dxB = __fadd2_rn(vx, xB), dyB = __fadd2_rn(vy, yB);
        const float2 qA = __ffma2_rn(dyA, dyA, __fmul2_rn(dxA, dxA));
        const float2 qB = __ffma2_rn(dyB, dyB, __fmul2_rn(dxB, dxB));
        const float2 kA = __fmul2_rn(mA, make_float2(rsqrt_clamped(qA.x), rsqrt_clamped(qA.y)));
        const float2 kB = __fmul2_rn(mB, make_float2(rsqrt_clamped(qB.x), rsqrt_clamped(qB.y)));
        ra = __ffma2_rn(kB, dxB, __fmul2_rn(kA, dxA));
        rb = __ffma2_rn(kB, dyB, __fmul2_rn(kA, dyA));
        cxA = __ffma2_rn(kA, dxA, cxA);  // sums of +t; negated when stored
        cxB = __ffma2_rn(kB, dxB, cxB);
        cyA = __ffma2_rn(kA, dyA, cyA);
        cyB = __ffma2_rn(kB, dyB, cyB);
      } else {
        ra = __ffma2_rn(mB, xB, __fmul2_rn(mA, xA));
        rb = __ffma2_rn(mB, yB, __fmul2_rn(mA, yA));
        cxA = __ffma2_rn(mA, vx, cxA);
        cxB = __ffma2_rn(mB, vx, cxB);
        cyA = __ffma2_rn(mA, vy, cyA);
        cyB = __ffma2_rn(mB, vy, cyB);
      }
      acc[2 * r] = ra.x + ra.y;
      acc[2 * r + 1] = rb.x + rb.y;
    }
    // every lane's reads of stage s (and of srec[s]) are done (their values
    // are in use above)
    __syncwarp();
    if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&empty[s])) : "memory");
    if (t.run >= 0) {
      rxA = __fadd2_rn(rxA, cxA);
      rxB = __fadd2_rn(rxB, cxB);
      ryA = __fadd2_rn(ryA, cyA);
      ryB = __fadd2_rn(ryB, cyB);
    }
    const float tot = lanes_transpose_sum<2 * PRW, float>(acc, lane);
    constexpr int REP = 32 / (2 * PRW);
    if (lane % REP == 0) {
      const int idx = lane / REP;
      float *part = reinterpret_cast<float *>(Part + t.part_off);
      part[((int64_t)t.J * t.kp + (int64_t)t.I * ST + rbase + (idx >> 1)) * 2 + (idx & 1)] = tot;
    }
  }
  if (cur_run >= 0) {
    float4 *o = reinterpret_cast<float4 *>(RunPart + ((int64_t)cur_run * CWARPS + warp) * ST + lane * 4);
    o[0] = make_float4(sg * rxA.x, sg * ryA.x, sg * rxA.y, sg * ryA.y);
    o[1] = make_float4(sg * rxB.x, sg * ryB.x, sg * rxB.y, sg * ryB.y);
  }
}

// Row block R of view v, (v, R) = blocks[blockIdx.x]:
//   Vout[R 128 + row] = sum_{J = R}^{nbt - 1} Part[J][R 128 + row]        (row sums of tiles (R, J))
//                     + sum over the runs of column block R and their warps
//                       of RunPart[(r CWARPS + w) 128 + row]                (column sums of tiles (I < R, R))
// The items are numbered in that order; thread (g, row) adds items g, g + 8,
// ... in order, then the eight group sums are added in order (a fixed order:
// the same result on every run).
__global__ void __launch_bounds__(1024)
k_reduce_rows(const int2 *__restrict__ blocks, const BatchView *__restrict__ views, const int *__restrict__ run_ptr,
              const int *__restrict__ run_idx, const float2 *__restrict__ Part, const float2 *__restrict__ RunPart,
              float2 *__restrict__ Vout) {
  constexpr int NG = 8, UN = 10;
  __shared__ float2 red[NG][ST];
  // launched as a programmatic dependent of the pass: wait for it to complete
  // (its partial sums visible); the next pass may be scheduled meanwhile
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int2 b = blocks[blockIdx.x];
  const BatchView bv = views[b.x];
  const int row = threadIdx.x & (ST - 1), g = threadIdx.x >> 7;
  const int64_t r = (int64_t)b.y * ST + row;
  const int nrow = bv.nbt - b.y;
  const int r0 = run_ptr[blockIdx.x], nitem = nrow + (run_ptr[blockIdx.x + 1] - r0) * spipe::CWARPS;
  float2 acc = make_float2(0.0f, 0.0f);
#pragma unroll 1
  for (int i0 = g; i0 < nitem; i0 += NG * UN) {
    float2 u[UN];
#pragma unroll
    for (int e = 0; e < UN; ++e) {
      const int i = i0 + NG * e;
      if (i < nrow) {
        u[e] = __ldcg(Part + bv.part_off + (int64_t)(b.y + i) * bv.kp + r);
      } else if (i < nitem) {
        const int q = i - nrow;
        const int run = run_idx[r0 + q / spipe::CWARPS];
        u[e] = __ldcg(RunPart + ((int64_t)run * spipe::CWARPS + q % spipe::CWARPS) * ST + row);
      }
    }
#pragma unroll
    for (int e = 0; e < UN; ++e)
      if (i0 + NG * e < nitem) {
        acc.x += u[e].x;
        acc.y += u[e].y;
      }
  }
  red[g][row] = acc;
  __syncthreads();
  if (threadIdx.x < ST) {
    float2 v = red[0][row];
#pragma unroll
    for (int e = 1; e < NG; ++e) {
      v.x += red[e][row].x;
      v.y += red[e][row].y;
    }
    Vout[bv.vec_off + r] = v;
  }
}

// ---------------------------------------------------------------------------
// FP32 updates of a view whose two matrices fit into the shared memories of
// the GPU (2 k^2 floats: k up to about 2,000): one cooperative launch for all
// updates. CTA c owns rows [c nr, (c + 1) nr) and keeps them, of 1/Delta_s and
// of M, in shared memory; thread t owns the columns 4t..4t+3. Per update
//   b_i = sum_j W_ij (x_i - x_j) / |x_i - x_j|   for the CTA's rows,
//   grid barrier, x_i = sum_j M_ij b_j, grid barrier,
// every row summed by its CTA alone (threads in column order, a fixed tree), so
// there are no partial sums to reduce, and nothing but the 2 k coordinates
// moves between CTAs. Reading both triangles doubles the arithmetic of the
// streaming passes, which is small here; what bounds an update is the latency
// of its two barriers and of the reads behind them. The streaming pipeline
// spends four launches on it: k = 1,999, 21 -> 7.5 us an update;
// k = 150, 19 -> 3.9 us. Above the limit the matrices stream from L2 or HBM
// and the pipeline's half of the bytes counts.
// Every barrier wait ends after a global-timer deadline: the CTA then records
// the error and leaves, and so does every CTA that sees it.
// ---------------------------------------------------------------------------
namespace resident {
constexpr int NRMAX = 16;                 // rows per CTA at most (2 NRMAX sums per thread)
constexpr uint32_t GAVE_UP = 0x80000000u; // barrier word: a wait expired somewhere

__device__ __forceinline__ uint64_t gtimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Grid barrier number `n` (1, 2, ...) of `ctas` CTAs on a counter that starts at
// 0; false once a wait has expired. All threads of the CTA call it.
__device__ __forceinline__ bool grid_barrier(uint32_t *bar, uint32_t n, uint32_t ctas, uint64_t limit_ns) {
  __shared__ int ok_sh;
  __syncthreads();  // the CTA's writes come before its arrival
  if (threadIdx.x == 0) {
    int ok = 1;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    const uint64_t t0 = gtimer();
    for (uint32_t it = 0;; ++it) {
      uint32_t v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if (v & GAVE_UP) {
        ok = 0;
        break;
      }
      if (v >= n * ctas) break;
      if ((it & 255) == 255 && gtimer() - t0 > limit_ns) {
        atomicOr(bar, GAVE_UP);
        ok = 0;
        break;
      }
    }
    ok_sh = ok;
  }
  __syncthreads();
  return ok_sh != 0;
}

// sums of the rows over all columns: acc[2 r], acc[2 r + 1] per thread -> out[r0 + r]
template <int NR>
__device__ __forceinline__ void row_sums(float (&acc)[2 * NR], float *red, int nr, float2 *out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  constexpr int REP = 32 / (2 * NR);
  const float tot = lanes_transpose_sum<2 * NR, float>(acc, lane);
  if (lane % REP == 0) red[warp * 2 * NR + lane / REP] = tot;
  __syncthreads();
  if ((int)threadIdx.x < 2 * nr) {
    float s = red[threadIdx.x];
    for (int w = 1; w < warps; ++w) s += red[w * 2 * NR + threadIdx.x];
    __stcg(reinterpret_cast<float *>(out) + threadIdx.x, s);
  }
}
}  // namespace resident

// kq: columns rounded up to 4 (a row's stride in shared memory); blockDim.x >= kq / 4
template <int NR>
__global__ void __launch_bounds__(512, 1)
k_layout_resident(int32_t k, int32_t kp, int32_t kq, int nrows, int iters, const float *__restrict__ W1,
                  const float *__restrict__ M, float2 *X, float2 *B, uint32_t *bar, int *__restrict__ err,
                  uint64_t limit_ns, int withhold) {
  using namespace resident;
  if (withhold && blockIdx.x + 1 == gridDim.x) return;  // (a test of the barrier's expiry: this CTA never arrives)
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  float *sW = reinterpret_cast<float *>(smem_raw);  // [nrows][kq]
  float *sM = sW + (size_t)nrows * kq;              // [nrows][kq]
  float *red = sM + (size_t)nrows * kq;             // [warps][2 NR]
  __shared__ float2 sx[NR];
  const int r0 = (int)blockIdx.x * nrows, nr = min(nrows, k - r0);
  // the rows, from the stored upper triangle of 128-blocks: element (r, j) is
  // at (j, r) where j's block comes before r's
  for (int e = threadIdx.x; e < nr * kq; e += blockDim.x) {
    const int r = e / kq, j = e - r * kq;
    float w = 0.0f, m = 0.0f;
    if (j < k && (j >> 7) >= ((r0 + r) >> 7)) {
      w = W1[(int64_t)(r0 + r) * kp + j];
      m = M[(int64_t)(r0 + r) * kp + j];
    }
    sW[e] = w;
    sM[e] = m;
  }
  __syncthreads();
  const int jlow = (((r0 + nr - 1) >> 7) << 7);  // columns of earlier blocks, for some row
  for (int e = threadIdx.x; e < nr * jlow; e += blockDim.x) {
    const int j = e / nr, r = e - j * nr;
    if ((j >> 7) < ((r0 + r) >> 7)) {
      sW[r * kq + j] = W1[(int64_t)j * kp + r0 + r];
      sM[r * kq + j] = M[(int64_t)j * kp + r0 + r];
    }
  }
  const int c0 = 4 * (int)threadIdx.x;
  const bool has = c0 < kq;  // X and B are zero up to kp >= kq, and so are the matrices' padded columns
  uint32_t nbar = 0;
  for (int it = 0; it < iters; ++it) {
    float acc[2 * NR];
    // ---- b = L^Y(X) X
    float4 v01 = make_float4(0.0f, 0.0f, 0.0f, 0.0f), v23 = v01;
    if (has) {
      v01 = __ldcg(reinterpret_cast<const float4 *>(X + c0));
      v23 = __ldcg(reinterpret_cast<const float4 *>(X + c0) + 1);
    }
    if ((int)threadIdx.x < nr) sx[threadIdx.x] = __ldcg(X + r0 + threadIdx.x);
    __syncthreads();
    {
      const float2 xA = make_float2(-v01.x, -v01.z), yA = make_float2(-v01.y, -v01.w);
      const float2 xB = make_float2(-v23.x, -v23.z), yB = make_float2(-v23.y, -v23.w);
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        acc[2 * r] = acc[2 * r + 1] = 0.0f;
        if (r < nr && has) {
          const float4 m4 = *reinterpret_cast<const float4 *>(sW + r * kq + c0);
          const float2 vi = sx[r];
          const float2 vx = make_float2(vi.x, vi.x), vy = make_float2(vi.y, vi.y);
          const float2 dxA = __fadd2_rn(vx, xA), dyA = __fadd2_rn(vy, yA);
          const float2 dxB = __fadd2_rn(vx, xB), dyB = __fadd2_rn(vy, yB);
          const float2 qA = __ffma2_rn(dyA, dyA, __fmul2_rn(dxA, dxA));
          const float2 qB = __ffma2_rn(dyB, dyB, __fmul2_rn(dxB, dxB));
          const float2 kA = __fmul2_rn(make_float2(m4.x, m4.y),
                                       make_float2(spipe::rsqrt_clamped(qA.x), spipe::rsqrt_clamped(qA.y)));
          const float2 kB = __fmul2_rn(make_float2(m4.z, m4.w),
                                       make_float2(spipe::rsqrt_clamped(qB.x), spipe::rsqrt_clamped(qB.y)));
          const float2 ra = __ffma2_rn(kB, dxB, __fmul2_rn(kA, dxA));
          const float2 rb = __ffma2_rn(kB, dyB, __fmul2_rn(kA, dyA));
          acc[2 * r] = ra.x + ra.y;
          acc[2 * r + 1] = rb.x + rb.y;
        }
      }
    }
    row_sums<NR>(acc, red, nr, B + r0);
    if (!grid_barrier(bar, ++nbar, gridDim.x, limit_ns)) break;
    // ---- X = M b
    if (has) {
      v01 = __ldcg(reinterpret_cast<const float4 *>(B + c0));
      v23 = __ldcg(reinterpret_cast<const float4 *>(B + c0) + 1);
    }
    {
      const float2 xA = make_float2(v01.x, v01.z), yA = make_float2(v01.y, v01.w);
      const float2 xB = make_float2(v23.x, v23.z), yB = make_float2(v23.y, v23.w);
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        acc[2 * r] = acc[2 * r + 1] = 0.0f;
        if (r < nr && has) {
          const float4 m4 = *reinterpret_cast<const float4 *>(sM + r * kq + c0);
          const float2 mA = make_float2(m4.x, m4.y), mB = make_float2(m4.z, m4.w);
          const float2 ra = __ffma2_rn(mB, xB, __fmul2_rn(mA, xA));
          const float2 rb = __ffma2_rn(mB, yB, __fmul2_rn(mA, yA));
          acc[2 * r] = ra.x + ra.y;
          acc[2 * r + 1] = rb.x + rb.y;
        }
      }
    }
    row_sums<NR>(acc, red, nr, X + r0);
    if (!grid_barrier(bar, ++nbar, gridDim.x, limit_ns)) break;
  }
  // (an expired wait leaves its mark in the barrier word)
  if (threadIdx.x == 0 && blockIdx.x == 0 && nbar > 0) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
    if (v & GAVE_UP) atomicOr(err, 1);
  }
}

// X (kp x 2) = x0 for rows < k, zero on the padding.
template <typename TI, typename T>
__global__ void k_load_x(int32_t k, int32_t kp, const TI *__restrict__ x, typename T2<T>::type *__restrict__ X) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= kp) return;
  typename T2<T>::type v;
  v.x = i < k ? (T)x[2 * i] : T(0);
  v.y = i < k ? (T)x[2 * i + 1] : T(0);
  X[i] = v;
}

// Centre X (FP64 mean, one block, fixed order) and convert to the output type.
template <typename T, typename TO>
__global__ void k_finish(int32_t k, const typename T2<T>::type *__restrict__ X, TO *__restrict__ out,
                         typename T2<T>::type *__restrict__ Xc) {
  __shared__ double sx[1024], sy[1024];
  double mx = 0.0, my = 0.0;
  for (int64_t i = threadIdx.x; i < k; i += blockDim.x) {
    mx += (double)X[i].x;
    my += (double)X[i].y;
  }
  sx[threadIdx.x] = mx;
  sy[threadIdx.x] = my;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      sx[threadIdx.x] += sx[threadIdx.x + o];
      sy[threadIdx.x] += sy[threadIdx.x + o];
    }
    __syncthreads();
  }
  const double ax = sx[0] / k, ay = sy[0] / k;
  for (int64_t i = threadIdx.x; i < k; i += blockDim.x) {
    const T cx = (T)((double)X[i].x - ax), cy = (T)((double)X[i].y - ay);
    out[2 * i] = (TO)cx;
    out[2 * i + 1] = (TO)cy;
    if (Xc) {
      typename T2<T>::type w;
      w.x = cx;
      w.y = cy;
      Xc[i] = w;
    }
  }
}

// ---------------------------------------------------------------------------
// Energy and gradients by pair recomputation. Per pair i != j with
// d = |x_i - x_j|, u = 1/Delta_ij, e = 1 - d u:
//   energy += e^2 (halved at the end: Eq. (7) sums i < j)
//   grad_x_i += -2 e u / d (x_i - x_j)      (0 when d = 0)
//   grad_pdist_ij = e d u^2
//
// A block owns ERPB rows at a time (block-stride over row groups, at most
// EBLOCKS blocks) and its 256 threads share the columns, so a view of a few
// thousand nodes already fills the GPU; the coordinates (8 k bytes) come from
// L1. The pass is meant to be bound by reading Delta (and writing
// grad_pdist). What it must not spend is GB300's FP64 pipe (2 operations per
// cycle and SM): one FP64 add and one conversion per pair alone cost five
// times the read. In FP32 the squares e^2 are therefore summed as a float and
// its exact rounding errors (TwoSum, Knuth), two rows at a time with the
// paired FP32 instructions, and go to an FP64 sum every QCH columns: over so
// few terms the roundings of the error word come to ~2^-49 of them (FP64
// additions: 2^-53 each; the squares themselves are rounded to 2^-24).
// 1/Delta, d and (-2 e u) / d start from the special-function unit, each
// followed by one correction from its residual (Newton's iteration), so that
// each is rounded about once, as in the plain formulas. Pairs outside
// the range in which those steps are safe (coincident or extremely close
// points, huge or tiny values, infinities, NaN, the diagonal) and a last
// group of fewer than ERPB rows take the plain formulas.
// Measured at k = 8,192 on one GB300 (read 268 MB, write 268 MB with
// grad_pdist), before -> now, with the reduce: energy alone 581 -> 104 us, both
// gradients 701 -> 161 us. It now issues ~30 instructions per pair, most of them on
// the FMA pipe, and waits on loads for the rest.
// ---------------------------------------------------------------------------
constexpr int ERPB = 4;                 // rows of a row group
constexpr int ETHREADS = 256;           // threads per block
constexpr int EBLOCKS = 608;            // blocks (and FP64 partials) at most: four per SM, so that the FP64
                                        // reduction at a block's end runs once per several row groups
inline unsigned energy_blocks(int64_t k) {
  return (unsigned)std::min<int64_t>((k + ERPB - 1) / ERPB, EBLOCKS);
}

// per-thread energy sums: a paired float sum with its rounding errors (FP32
// pairs on the fast path) and an FP64 sum (everything else)
template <typename T>
struct EAcc {
  float2 s = make_float2(0.0f, 0.0f), c = make_float2(0.0f, 0.0f);
  double d = 0.0;
  __device__ __forceinline__ void add2(float2 q) {  // TwoSum, both halves
    const float2 n = make_float2(-1.0f, -1.0f);
    const float2 t = __fadd2_rn(s, q);
    const float2 bb = __ffma2_rn(n, s, t);                       // t - s
    const float2 e0 = __ffma2_rn(n, __ffma2_rn(n, bb, t), s);    // s - (t - bb)
    const float2 e1 = __ffma2_rn(n, bb, q);                      // q - bb
    c = __fadd2_rn(c, __fadd2_rn(e0, e1));
    s = t;
  }
  // to the FP64 sum, before the roundings of c add up to one of its
  __device__ __forceinline__ void flush() {
    d += ((double)s.x + (double)s.y) + ((double)c.x + (double)c.y);
    s = c = make_float2(0.0f, 0.0f);
  }
};

// The shares of a row's gradient are added up with their rounding errors from
// groups of eight threads on: a row has 256 shares, at k = 1,000 one for every
// four terms, and plain sums of them lost more than 32 shares a row did. Root
// mean square error of a gradient at k = 1,000, 32 plain shares, 256 plain, now:
// FP32 4.4e-8, 5.2e-8, 2.9e-8; FP64 (k = 700) 7.7e-17, 9.6e-17, 5.2e-17. Both
// gradients at k = 8,192: 153 -> 161 us.
template <typename T>
struct Sum2 {  // a sum and its rounding errors (TwoSum, Knuth)
  T s, c;
  __device__ __forceinline__ Sum2 operator+(Sum2 b) const {
    const T t = s + b.s, bb = t - s;
    return {t, ((s - (t - bb)) + (b.s - bb)) + (c + b.c)};
  }
};

// one pair by the plain formulas; row i, column j
template <typename T, bool GX, bool GD>
__device__ __forceinline__ void energy_pair(int64_t i, int64_t j, int64_t k, T del, T dx, T dy, T scale, double &eacc,
                                            T &gxx, T &gxy, T *__restrict__ gD, int &bad) {
  if (i == j) {
    if (GD) gD[i * k + j] = T(0);
    return;
  }
  if (!(del > T(0))) bad = 1;
  const T d = sqrt(dx * dx + dy * dy);
  const T u = T(1) / del;
  const T e = T(1) - d * u;
  eacc += (double)(e * e);
  if (GX && d > T(0)) {
    const T coef = T(-2) * e * u / d;
    gxx += coef * dx;
    gxy += coef * dy;
  }
  if (GD) gD[i * k + j] = scale * e * d * u * u;
}

// All of a, b, c, d in [2^lo, 2^hi], as bit patterns of positive floats (zero,
// negative and NaN values fall outside).
__device__ __forceinline__ bool all_in_range(const float (&v)[4], int lo, int hi) {
  const int a = __float_as_int(v[0]), b = __float_as_int(v[1]), c = __float_as_int(v[2]), d = __float_as_int(v[3]);
  return min(min(a, b), min(c, d)) >= ((127 + lo) << 23) && max(max(a, b), max(c, d)) <= ((127 + hi) << 23);
}
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

template <typename T, bool GX, bool GD>
__global__ void __launch_bounds__(ETHREADS, std::is_same<T, float>::value ? 4 : 2)
k_energy(int32_t k, const T *__restrict__ Delta, const typename T2<T>::type *__restrict__ X, T scale,
         double *__restrict__ eparts, T *__restrict__ gx, T *__restrict__ gD, int *__restrict__ flag) {
  using V2 = typename T2<T>::type;
  constexpr int WARPS = ETHREADS / 32;
  constexpr int QCH = 32;  // columns per thread between two runs of the plain formulas (bits of `plain`)
  __shared__ double se[WARPS];
  __shared__ Sum2<T> sg[WARPS][2 * ERPB];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  EAcc<T> acc;
  int bad = 0;
  for (int64_t r0 = (int64_t)blockIdx.x * ERPB; r0 < k; r0 += (int64_t)gridDim.x * ERPB) {
    const int nr = (int)min((int64_t)ERPB, k - r0);
    const T *D0 = Delta + r0 * k;
    V2 xi[ERPB];
    T gxx[ERPB], gxy[ERPB];
#pragma unroll
    for (int r = 0; r < ERPB; ++r) {
      xi[r] = X[min((int)r0 + r, k - 1)];
      gxx[r] = gxy[r] = T(0);
    }
    for (int64_t c0 = threadIdx.x; c0 < k; c0 += QCH * ETHREADS) {
      const int nq = (int)min((int64_t)QCH, (k - c0 + ETHREADS - 1) / ETHREADS);
      uint32_t plain = nq == QCH ? 0xffffffffu : (1u << nq) - 1u;  // columns left to the plain formulas
      if constexpr (std::is_same<T, float>::value) {
        if (nr == ERPB) {
          const float2 n = make_float2(-1.0f, -1.0f), one = make_float2(1.0f, 1.0f), half = make_float2(0.5f, 0.5f);
          const T *Dc = D0 + c0;
          const V2 *Xc = X + c0;
          const int jd = (int)(r0 - c0);  // columns jd .. jd + 3 (from c0) hold the diagonal
          // the next column's loads are in flight while a column is computed
          float nd[ERPB];
          V2 nx = Xc[0];
#pragma unroll
          for (int r = 0; r < ERPB; ++r) nd[r] = __ldcs(Dc + (int64_t)r * k);
#pragma unroll 2
          for (int q = 0; q < nq; ++q) {
            float del[ERPB], d2a[ERPB];
            const V2 xj = nx;
#pragma unroll
            for (int r = 0; r < ERPB; ++r) del[r] = nd[r];
            if (q + 1 < nq) {
              nx = Xc[(q + 1) * ETHREADS];
#pragma unroll
              for (int r = 0; r < ERPB; ++r) nd[r] = __ldcs(Dc + (int64_t)r * k + (q + 1) * ETHREADS);
            }
            float2 dx[ERPB / 2], dy[ERPB / 2], d2[ERPB / 2];
            const float2 xj2 = make_float2(xj.x, xj.x), yj2 = make_float2(xj.y, xj.y);
#pragma unroll
            for (int p = 0; p < ERPB / 2; ++p) {  // rows 2p, 2p + 1
              dx[p] = __ffma2_rn(n, xj2, make_float2(xi[2 * p].x, xi[2 * p + 1].x));
              dy[p] = __ffma2_rn(n, yj2, make_float2(xi[2 * p].y, xi[2 * p + 1].y));
              d2[p] = __ffma2_rn(dx[p], dx[p], __fmul2_rn(dy[p], dy[p]));
              d2a[2 * p] = d2[p].x;
              d2a[2 * p + 1] = d2[p].y;
            }
            if (!all_in_range(d2a, -80, 40) || !all_in_range(del, -20, 60) ||
                (unsigned)(q * ETHREADS - jd) < (unsigned)ERPB)
              continue;
            plain &= ~(1u << q);
#pragma unroll
            for (int p = 0; p < ERPB / 2; ++p) {
              const float2 dl = make_float2(del[2 * p], del[2 * p + 1]);
              const float2 u0 = make_float2(rcp_approx(dl.x), rcp_approx(dl.y));
              const float2 y0 = make_float2(rsqrt_approx(d2[p].x), rsqrt_approx(d2[p].y));
              // u0 + u0 (1 - Delta u0)
              const float2 u = __ffma2_rn(__ffma2_rn(__fmul2_rn(n, dl), u0, one), u0, u0);
              const float2 s0 = __fmul2_rn(d2[p], y0);
              // d = s0 + (d2 - s0^2) / (2 s0), 1 / s0 ~ y0
              const float2 res = __ffma2_rn(__fmul2_rn(n, s0), s0, d2[p]);
              const float2 d = __ffma2_rn(__fmul2_rn(half, y0), res, s0);
              const float2 e = __ffma2_rn(__fmul2_rn(n, d), u, one);
              acc.add2(__fmul2_rn(e, e));
              if (GX) {
                // (-2 e u) / d = q0 + y0 (t - d q0)
                const float2 t = __fmul2_rn(__fmul2_rn(make_float2(-2.0f, -2.0f), e), u);
                const float2 q0 = __fmul2_rn(t, y0);
                const float2 cf = __ffma2_rn(__ffma2_rn(__fmul2_rn(n, d), q0, t), y0, q0);
                const float2 gX = __ffma2_rn(cf, dx[p], make_float2(gxx[2 * p], gxx[2 * p + 1]));
                const float2 gY = __ffma2_rn(cf, dy[p], make_float2(gxy[2 * p], gxy[2 * p + 1]));
                gxx[2 * p] = gX.x;
                gxx[2 * p + 1] = gX.y;
                gxy[2 * p] = gY.x;
                gxy[2 * p + 1] = gY.y;
              }
              if (GD) {  // ((scale e) d u) u, the order of the plain formula
                const float2 g = __fmul2_rn(__fmul2_rn(__fmul2_rn(__fmul2_rn(make_float2(scale, scale), e), d), u), u);
                T *o = gD + (r0 + 2 * p) * k + c0 + q * ETHREADS;
                __stcs(o, g.x);
                __stcs(o + k, g.y);
              }
            }
          }
          acc.flush();
        }
      }
      while (plain) {
        const int q = __ffs((int)plain) - 1;
        plain &= plain - 1u;
        const int64_t j = c0 + q * ETHREADS;
        const V2 xj = X[j];
#pragma unroll
        for (int r = 0; r < ERPB; ++r)
          if (r < nr)
            energy_pair<T, GX, GD>(r0 + r, j, k, D0[(int64_t)r * k + j], xi[r].x - xj.x, xi[r].y - xj.y, scale, acc.d,
                                   gxx[r], gxy[r], gD, bad);
      }
    }
    if (GX) {
      T v[2 * ERPB];
#pragma unroll
      for (int r = 0; r < ERPB; ++r) {
        v[2 * r] = gxx[r];
        v[2 * r + 1] = gxy[r];
      }
      constexpr int REP = 32 / (2 * ERPB);
      Sum2<T> tot{lanes_fold<2 * ERPB, T>(v, lane), T(0)};
#pragma unroll
      for (int off = REP / 2; off > 0; off >>= 1)
        tot = tot + Sum2<T>{__shfl_xor_sync(0xffffffffu, tot.s, off), __shfl_xor_sync(0xffffffffu, tot.c, off)};
      if (lane % REP == 0) sg[warp][lane / REP] = tot;
      __syncthreads();
      if (threadIdx.x < 2 * ERPB && r0 + (threadIdx.x >> 1) < k) {
        Sum2<T> s = sg[0][threadIdx.x];
#pragma unroll
        for (int w = 1; w < WARPS; ++w) s = s + sg[w][threadIdx.x];
        gx[2 * r0 + threadIdx.x] = scale * (s.s + s.c);
      }
      __syncthreads();  // before the next group's sums
    }
  }
  double e = acc.d;
  for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
  if (lane == 0) se[warp] = e;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < WARPS; ++w) s += se[w];
    eparts[blockIdx.x] = s;
  }
  if (bad) atomicOr(flag, 1);
}

__global__ void k_reduce_energy(int nparts, const double *__restrict__ eparts, double *__restrict__ out) {
  __shared__ double s[256];
  double a = 0.0;
  for (int i = threadIdx.x; i < nparts; i += blockDim.x) a += eparts[i];
  s[threadIdx.x] = a;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = 0.5 * s[0];
}

template <typename TI, typename T>
__global__ void k_convert(int64_t cnt, const TI *__restrict__ in, T *__restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < cnt) out[i] = (T)in[i];
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
namespace {

// Grid and shared-memory setup of the pipelined FP32 pass: one CTA per SM
// (fewer when the table is shorter).
int sympass_pipe_grid(pprviz_ctx *ctx, size_t ntile, unsigned *grid) {
  int nsm = 0;
  PPRVIZ_CUDA(ctx, cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device));
  PPRVIZ_CUDA(ctx, cudaFuncSetAttribute(k_sympass_pipe<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, spipe::SMEM));
  PPRVIZ_CUDA(ctx, cudaFuncSetAttribute(k_sympass_pipe<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, spipe::SMEM));
  *grid = (unsigned)std::min<size_t>(ntile, (size_t)std::max(nsm, 1));
  return PPRVIZ_OK;
}

// cuTensorMapEncodeTiled through the runtime's driver entry point (the
// library links only the runtime).
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The kp x kp row-major FP32 matrix at base as a 2-D tensor with 128 x 128
// boxes, no swizzle (a box lands row-major in shared memory).
int tile_map(pprviz_ctx *ctx, const float *base, int32_t kp, CUtensorMap *out) {
  static EncodeTiledFn encode = nullptr;
  if (!encode) {
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    const cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn)
      return set_err(ctx, PPRVIZ_E_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
    encode = reinterpret_cast<EncodeTiledFn>(fn);
  }
  const cuuint64_t dims[2] = {(cuuint64_t)kp, (cuuint64_t)kp};
  const cuuint64_t strides[1] = {(cuuint64_t)kp * sizeof(float)};
  const cuuint32_t box[2] = {(cuuint32_t)ST, (cuuint32_t)ST};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = encode(out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float *>(base), dims, strides, box,
                            estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return set_err(ctx, PPRVIZ_E_CUDA, "cuTensorMapEncodeTiled failed for a layout matrix");
  return PPRVIZ_OK;
}

// Tables of the pipelined FP32 pass for a grid of G CTAs (device slots
// WS_TREC, WS_TROWS):
//  * tile records of every view's upper-triangle tiles, view by view, column
//    by column (J, then I = 0..J), with the run slot of each off-diagonal
//    tile: consecutive tiles of one column block in one CTA's chunk
//    [b ntile / G, (b + 1) ntile / G) share a run;
//  * the (view, row block) pairs, one per k_reduce_rows block (view order,
//    then R), and for each the runs of column block R (CSR: run_ptr, run_idx).
struct PassTables {
  const TileRec *recs = nullptr;
  int ntile = 0;
  const int2 *blocks = nullptr;
  const int *run_ptr = nullptr, *run_idx = nullptr;
  int nblocks = 0, nruns = 0;
};

int upload_pass_tables(pprviz_ctx *ctx, const std::vector<BatchView> &bv, unsigned G, PassTables *pt) {
  std::vector<TileRec> rec;
  std::vector<int> rb_base(bv.size());
  int nrb = 0;
  for (size_t v = 0; v < bv.size(); ++v) {
    rb_base[v] = nrb;
    nrb += bv[v].nbt;
    for (int J = 0; J < bv[v].nbt; ++J)
      for (int I = 0; I <= J; ++I)
        rec.push_back(TileRec{(int32_t)v, I, J, (int32_t)(bv[v].vec_off / ST), bv[v].kp, -1, bv[v].part_off});
  }
  const int64_t ntile = (int64_t)rec.size();
  if (ntile >= INT32_MAX) return set_err(ctx, PPRVIZ_E_INVALID_ARG, "too many layout tiles");
  std::vector<std::vector<int>> runs_of(nrb);
  int nruns = 0, cur = -1, prev_v = -1, prev_J = -1;
  int64_t b = 0;  // CTA of position p: first(b) <= p < first(b + 1)
  for (int64_t p = 0; p < ntile; ++p) {
    while (b + 1 < (int64_t)G && (b + 1) * ntile / G <= p) ++b;
    TileRec &r = rec[p];
    const bool chunk_start = (b * ntile / G) == p;
    if (r.I == r.J) {  // diagonal: its column sums are not taken
      cur = -1;
      continue;
    }
    if (cur < 0 || chunk_start || r.v != prev_v || r.J != prev_J) {
      cur = nruns++;
      runs_of[rb_base[r.v] + r.J].push_back(cur);
    }
    r.run = cur;
    prev_v = r.v;
    prev_J = r.J;
  }
  std::vector<int2> blocks;
  std::vector<int> run_ptr(1, 0), run_idx;
  for (size_t v = 0; v < bv.size(); ++v)
    for (int R = 0; R < bv[v].nbt; ++R) {
      blocks.push_back(make_int2((int)v, R));
      for (int q : runs_of[rb_base[v] + R]) run_idx.push_back(q);
      run_ptr.push_back((int)run_idx.size());
    }
  if (run_idx.empty()) run_idx.push_back(0);  // keep the device pointer valid
  const size_t o_blocks = 0, o_ptr = (sizeof(int2) * blocks.size() + 255) & ~(size_t)255;
  const size_t o_idx = (o_ptr + sizeof(int) * run_ptr.size() + 255) & ~(size_t)255;
  const size_t bytes = o_idx + sizeof(int) * run_idx.size();
  PPRVIZ_TRY(ws_ensure(ctx, WS_TREC, sizeof(TileRec) * rec.size()));
  PPRVIZ_TRY(ws_ensure(ctx, WS_TROWS, bytes));
  unsigned char *d = static_cast<unsigned char *>(ctx->ws[WS_TROWS].p);
  PPRVIZ_CUDA(ctx, cudaMemcpyAsync(ctx->ws[WS_TREC].p, rec.data(), sizeof(TileRec) * rec.size(),
                                   cudaMemcpyHostToDevice, ctx->stream));
  PPRVIZ_CUDA(ctx, cudaMemcpyAsync(d + o_blocks, blocks.data(), sizeof(int2) * blocks.size(), cudaMemcpyHostToDevice,
                                   ctx->stream));
  PPRVIZ_CUDA(ctx, cudaMemcpyAsync(d + o_ptr, run_ptr.data(), sizeof(int) * run_ptr.size(), cudaMemcpyHostToDevice,
                                   ctx->stream));
  PPRVIZ_CUDA(ctx, cudaMemcpyAsync(d + o_idx, run_idx.data(), sizeof(int) * run_idx.size(), cudaMemcpyHostToDevice,
                                   ctx->stream));
  PPRVIZ_CUDA(ctx, cudaStreamSynchronize(ctx->stream));  // the host vectors are released on return
  pt->recs = ctx->ws[WS_TREC].as<TileRec>();
  pt->ntile = (int)ntile;
  pt->blocks = reinterpret_cast<const int2 *>(d + o_blocks);
  pt->run_ptr = reinterpret_cast<const int *>(d + o_ptr);
  pt->run_idx = reinterpret_cast<const int *>(d + o_idx);
  pt->nblocks = (int)blocks.size();
  pt->nruns = nruns;
  return PPRVIZ_OK;
}

// L2 bytes of each pass matrix kept resident across updates (evict_last):
// the two matrices together stay well inside the 126 MB L2 next to the
// partial sums and coordinates; the rest of each matrix streams from HBM
constexpr double kPinBytes = 32.0 * 1024 * 1024;

// One layout update of all views in the tables: L^Y pass over W1 from X into
// Bv, apply pass over M from Bv into X, each followed by its reduce.
int pass_pair(pprviz_ctx *ctx, unsigned grid, const PassTables &pt, const CUtensorMap *maps, const BatchView *views_d,
              float2 *X, float2 *Bv, float2 *Part, float2 *RunPart, int *perr) {
  const unsigned nb = (unsigned)pt.nblocks;
  const int npin = (int)(kPinBytes / spipe::TILE_BYTES / grid);  // tiles per CTA
  { PPRVIZ_PROF(ctx, PPRVIZ_K_LY); PPRVIZ_CUDA(ctx, launch_dependent(ctx, k_sympass_pipe<0>, grid, spipe::THREADS, spipe::SMEM, pt.ntile, npin, pt.recs, maps, (const float2 *)X, Part, RunPart, perr)); }
  PPRVIZ_LAUNCHED(ctx);
  { PPRVIZ_PROF(ctx, PPRVIZ_K_OTHER); PPRVIZ_CUDA(ctx, launch_dependent(ctx, k_reduce_rows, nb, 1024, 0, pt.blocks, views_d, pt.run_ptr, pt.run_idx, (const float2 *)Part, (const float2 *)RunPart, Bv)); }
  PPRVIZ_LAUNCHED(ctx);
  { PPRVIZ_PROF(ctx, PPRVIZ_K_APPLY); PPRVIZ_CUDA(ctx, launch_dependent(ctx, k_sympass_pipe<1>, grid, spipe::THREADS, spipe::SMEM, pt.ntile, npin, pt.recs, maps, (const float2 *)Bv, Part, RunPart, perr)); }
  PPRVIZ_LAUNCHED(ctx);
  { PPRVIZ_PROF(ctx, PPRVIZ_K_OTHER); PPRVIZ_CUDA(ctx, launch_dependent(ctx, k_reduce_rows, nb, 1024, 0, pt.blocks, views_d, pt.run_ptr, pt.run_idx, (const float2 *)Part, (const float2 *)RunPart, X)); }
  PPRVIZ_LAUNCHED(ctx);
  return PPRVIZ_OK;
}

// Tensor maps of the two pass matrices of every view (maps[2 v] = 1/Delta_s,
// maps[2 v + 1] = M) into the device slot WS_TMAP.
int upload_maps(pprviz_ctx *ctx, const std::vector<BatchView> &bv, const float *W1, const float *M,
                const CUtensorMap **maps_d) {
  std::vector<CUtensorMap> maps(2 * bv.size());
  for (size_t v = 0; v < bv.size(); ++v) {
    PPRVIZ_TRY(tile_map(ctx, W1 + bv[v].mat_off, bv[v].kp, &maps[2 * v]));
    PPRVIZ_TRY(tile_map(ctx, M + bv[v].mat_off, bv[v].kp, &maps[2 * v + 1]));
  }
  PPRVIZ_TRY(ws_ensure(ctx, WS_TMAP, sizeof(CUtensorMap) * maps.size()));
  CUtensorMap *d = reinterpret_cast<CUtensorMap *>(ctx->ws[WS_TMAP].p);
  PPRVIZ_CUDA(ctx, cudaMemcpyAsync(d, maps.data(), sizeof(CUtensorMap) * maps.size(), cudaMemcpyHostToDevice,
                                   ctx->stream));
  // the host vector is released on return: wait for the copy
  PPRVIZ_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  *maps_d = d;
  return PPRVIZ_OK;
}

// All updates of one view in one cooperative launch (k_layout_resident).
// *done = false (and nothing launched) where its rows do not fit.
int resident_updates(pprviz_ctx *ctx, int32_t k, int32_t kp, int iters, const float *W1, const float *M, float2 *X,
                     float2 *B, int *err, bool *done) {
  *done = false;
  int nsm = 0, smax = 0, coop = 0;
  PPRVIZ_CUDA(ctx, cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device));
  PPRVIZ_CUDA(ctx, cudaDeviceGetAttribute(&smax, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device));
  PPRVIZ_CUDA(ctx, cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, ctx->device));
  const int32_t kq = (k + 3) / 4 * 4;
  const unsigned threads = (unsigned)((kq / 4 + 31) / 32 * 32);
  // rows per CTA: as few as the SMs allow, but at least 4 (fewer CTAs wait on
  // each other for less work)
  const int nrows = std::max(4, (k + nsm - 1) / nsm);
  const int NR = nrows <= 4 ? 4 : nrows <= 8 ? 8 : 16;
  const size_t smem = sizeof(float) * (2 * (size_t)nrows * kq + (threads / 32) * 2 * NR);
  const unsigned grid = (unsigned)((k + nrows - 1) / nrows);
  if (!coop || threads > 512 || nrows > resident::NRMAX || smem + 1024 > (size_t)smax) return PPRVIZ_OK;
  if (2 * (int64_t)iters * grid >= (int64_t)resident::GAVE_UP) return PPRVIZ_OK;  // the barrier word counts arrivals
  PPRVIZ_TRY(ws_ensure(ctx, WS_BTAB, 64));
  uint32_t *bar = ctx->ws[WS_BTAB].as<uint32_t>();
  PPRVIZ_CUDA(ctx, cudaMemsetAsync(bar, 0, sizeof(uint32_t), ctx->stream));
  const uint64_t limit_ns = 2000000000ull;  // bounded waits: 2 s
  auto kernel = NR == 4 ? k_layout_resident<4> : NR == 8 ? k_layout_resident<8> : k_layout_resident<16>;
  PPRVIZ_CUDA(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = ctx->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const int withhold = grid > 1 && ctx->expire_here() ? 1 : 0;
  PPRVIZ_PROF(ctx, PPRVIZ_K_LY);
  const cudaError_t e =
      cudaLaunchKernelEx(&cfg, kernel, k, kp, kq, nrows, iters, W1, M, X, B, bar, err, limit_ns, withhold);
  if (e == cudaErrorCooperativeLaunchTooLarge) {  // not all CTAs fit at once: the pipeline takes it
    cudaGetLastError();
    return PPRVIZ_OK;
  }
  PPRVIZ_CUDA(ctx, e);
  PPRVIZ_LAUNCHED(ctx);
  *done = true;
  return PPRVIZ_OK;
}

template <typename T, typename TI, typename TO>
int layout_typed(pprviz_ctx *ctx, const TI *pdist, int32_t k, const TI *x0, int32_t iters, TO *x_out,
                 double *stress_h) {
  using V2 = typename T2<T>::type;
  const int32_t kp = (k + ST - 1) / ST * ST;  // whole symmetric tiles (and NB pivot blocks)
  const int nbt = kp / ST;
  PPRVIZ_TRY(ws_ensure(ctx, WS_W1, sizeof(T) * (size_t)kp * kp));
  PPRVIZ_TRY(ws_ensure(ctx, WS_M, sizeof(T) * (size_t)kp * kp));
  PPRVIZ_TRY(ws_ensure(ctx, WS_PIV, sizeof(T) * spd_inverse_work(kp)));
  PPRVIZ_TRY(ws_ensure(ctx, WS_X, sizeof(V2) * (size_t)kp * 2));            // X and b
  constexpr bool F64 = std::is_same<T, double>::value;
  const int pbt = F64 ? kp / ST64 : nbt;                                    // row blocks of a pass
  PPRVIZ_TRY(ws_ensure(ctx, WS_B, sizeof(V2) * (size_t)pbt * kp));          // partial sums
  PPRVIZ_TRY(ws_ensure(ctx, WS_E, sizeof(V2) * (size_t)k + 64));
  PPRVIZ_TRY(ws_ensure(ctx, WS_RHS, sizeof(double) * (size_t)(kp / 32) * kp));  // build row partials
  PPRVIZ_TRY(ws_ensure(ctx, WS_FLAG, 64));
  T *W1 = ctx->ws[WS_W1].as<T>(), *A = ctx->ws[WS_M].as<T>();
  T *work = ctx->ws[WS_PIV].as<T>();
  V2 *X = ctx->ws[WS_X].as<V2>(), *Bv = X + kp, *Part = ctx->ws[WS_B].as<V2>();
  PPRVIZ_CUDA(ctx, cudaMemsetAsync(Bv, 0, sizeof(V2) * (size_t)kp, ctx->stream));
  double *rowpart = ctx->ws[WS_RHS].as<double>();
  int *flag = ctx->ws[WS_FLAG].as<int>();
  // status words, read once after the updates: [0] a bad distance, [1] an
  // expired wait of the passes, [2] of the inverse
  PPRVIZ_CUDA(ctx, cudaMemsetAsync(flag, 0, 3 * sizeof(int), ctx->stream));
  { PPRVIZ_PROF(ctx, PPRVIZ_K_FACTOR); k_build_sym<TI, T><<<dim3(kp / 32, kp / 32), dim3(32, 8), 0, ctx->stream>>>(k, kp, pdist, W1, A, rowpart, flag); }
  PPRVIZ_LAUNCHED(ctx);
  { PPRVIZ_PROF(ctx, PPRVIZ_K_FACTOR); k_build_diag<T><<<(unsigned)((k + 255) / 256), 256, 0, ctx->stream>>>(k, kp, rowpart, A); }
  PPRVIZ_LAUNCHED(ctx);
  if (iters > 0) {
    if constexpr (std::is_same<T, float>::value) PPRVIZ_TRY(spd_inverse_f32(ctx, kp, A, work, flag + 2));
    else PPRVIZ_TRY(spd_inverse_f64(ctx, kp, A, work));
  }
  { PPRVIZ_PROF(ctx, PPRVIZ_K_OTHER); k_load_x<TI, T><<<(unsigned)((kp + 255) / 256), 256, 0, ctx->stream>>>(k, kp, x0, X); }
  PPRVIZ_LAUNCHED(ctx);
  // the view descriptor (FP32), or the upper tile triangle in row order and the
  // row-block counters of the fused reduce, zero between passes (FP64)
  const BatchView one{0, 0, 0, kp, nbt, k};
  if constexpr (std::is_same<T, float>::value) {
    int *perr = flag + 1;
    bool done = false;
    if (iters > 0) PPRVIZ_TRY(resident_updates(ctx, k, kp, iters, W1, A, X, Bv, perr, &done));
    if (!done && iters > 0) {
      PPRVIZ_TRY(ws_ensure(ctx, WS_BTAB, sizeof(BatchView)));
      BatchView *view_d = reinterpret_cast<BatchView *>(ctx->ws[WS_BTAB].p);
      PPRVIZ_CUDA(ctx, cudaMemcpyAsync(view_d, &one, sizeof(BatchView), cudaMemcpyHostToDevice, ctx->stream));
      unsigned pgrid = 0;
      PPRVIZ_TRY(sympass_pipe_grid(ctx, (size_t)nbt * (nbt + 1) / 2, &pgrid));
      const std::vector<BatchView> one_v{one};
      const CUtensorMap *maps = nullptr;
      PPRVIZ_TRY(upload_maps(ctx, one_v, W1, A, &maps));
      PassTables pt;
      PPRVIZ_TRY(upload_pass_tables(ctx, one_v, pgrid, &pt));
      PPRVIZ_TRY(ws_ensure(ctx, WS_RUNP, sizeof(V2) * ((size_t)pt.nruns * spipe::CWARPS * ST + 1)));
      V2 *RunPart = ctx->ws[WS_RUNP].as<V2>();
      for (int it = 0; it < iters; ++it) PPRVIZ_TRY(pass_pair(ctx, pgrid, pt, maps, view_d, X, Bv, Part, RunPart, perr));
    }
  } else {
    std::vector<int2> tiles;
    for (int I = 0; I < pbt; ++I)
      for (int J = I; J < pbt; ++J) tiles.push_back(make_int2(I, J));
    const size_t cnt_off = (sizeof(int2) * tiles.size() + 255) & ~(size_t)255;
    PPRVIZ_TRY(ws_ensure(ctx, WS_BTAB, cnt_off + sizeof(int) * (size_t)pbt));
    int2 *tiles_d = ctx->ws[WS_BTAB].as<int2>();
    int *cnt = reinterpret_cast<int *>(static_cast<unsigned char *>(ctx->ws[WS_BTAB].p) + cnt_off);
    PPRVIZ_CUDA(ctx, cudaMemcpyAsync(tiles_d, tiles.data(), sizeof(int2) * tiles.size(), cudaMemcpyHostToDevice,
                                     ctx->stream));
    PPRVIZ_CUDA(ctx, cudaMemsetAsync(cnt, 0, sizeof(int) * (size_t)pbt, ctx->stream));
    PPRVIZ_CUDA(ctx, cudaStreamSynchronize(ctx->stream));  // the host table is released below
    const unsigned ntile = (unsigned)tiles.size();
    for (int it = 0; it < iters; ++it) {
      { PPRVIZ_PROF(ctx, PPRVIZ_K_LY); PPRVIZ_CUDA(ctx, launch_dependent(ctx, k_sympass64<0>, ntile, 256, 0, kp, pbt, (const int2 *)tiles_d, (const double *)W1, (const double2 *)X, Part, cnt, Bv)); }
      PPRVIZ_LAUNCHED(ctx);
      { PPRVIZ_PROF(ctx, PPRVIZ_K_APPLY); PPRVIZ_CUDA(ctx, launch_dependent(ctx, k_sympass64<1>, ntile, 256, 0, kp, pbt, (const int2 *)tiles_d, (const double *)A, (const double2 *)Bv, Part, cnt, X)); }
      PPRVIZ_LAUNCHED(ctx);
    }
  }
  int hf[3] = {0, 0, 0};
  PPRVIZ_CUDA(ctx, cudaMemcpyAsync(hf, flag, sizeof(hf), cudaMemcpyDeviceToHost, ctx->stream));
  PPRVIZ_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  if (hf[0]) return set_err(ctx, PPRVIZ_E_INVALID_ARG, "pdist has a non-finite or non-positive off-diagonal entry");
  if (hf[2]) return set_err(ctx, PPRVIZ_E_TIMEOUT, "tensor-core trailing update: a bounded wait expired");
  if (hf[1]) return set_err(ctx, PPRVIZ_E_TIMEOUT, "layout pass: a bounded wait expired");
  V2 *Xc = ctx->ws[WS_E].as<V2>();
  { PPRVIZ_PROF(ctx, PPRVIZ_K_OTHER); k_finish<T, TO><<<1, 1024, 0, ctx->stream>>>(k, X, x_out, Xc); }
  PPRVIZ_LAUNCHED(ctx);
  ctx->stats.layout_iters = iters;
  // algorithmic bytes: each pass reads the upper triangle of one k x k matrix
  const double half = 0.5 * (double)k * ((double)k + 1.0) * sizeof(T);
  ctx->stats.bytes_ly = half * iters;
  ctx->stats.bytes_apply = half * iters;
  if (stress_h) {
    const unsigned eb = energy_blocks(k);
    PPRVIZ_TRY(ws_ensure(ctx, WS_OUT1, sizeof(double) * (eb + 1)));
    double *ep = ctx->ws[WS_OUT1].as<double>();
    // stress of the final layout on the input pdist (Eq. (7)), in the path's arithmetic
    const T *Dt = (const T *)pdist;
    if (!std::is_same<T, TI>::value) {
      T *Dw = W1;  // k*k fits in the kp*kp 1/Delta buffer, which is no longer needed
      const int64_t cnt = (int64_t)k * k;
      { PPRVIZ_PROF(ctx, PPRVIZ_K_OTHER); k_convert<TI, T><<<(unsigned)((cnt + 255) / 256), 256, 0, ctx->stream>>>(cnt, pdist, Dw); }
      PPRVIZ_LAUNCHED(ctx);
      Dt = Dw;
    }
    { PPRVIZ_PROF(ctx, PPRVIZ_K_ENERGY); k_energy<T, false, false><<<eb, ETHREADS, 0, ctx->stream>>>(k, Dt, Xc, T(1), ep, nullptr, nullptr, flag); }
    PPRVIZ_LAUNCHED(ctx);
    { PPRVIZ_PROF(ctx, PPRVIZ_K_ENERGY); k_reduce_energy<<<1, 256, 0, ctx->stream>>>((int)eb, ep, ep + eb); }
    PPRVIZ_LAUNCHED(ctx);
    PPRVIZ_CUDA(ctx, cudaMemcpyAsync(stress_h, ep + eb, sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    PPRVIZ_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  }
  return PPRVIZ_OK;
}

}  // namespace

int layout_run(pprviz_ctx *ctx, const void *pdist_d, int32_t k, const void *x0_d, int32_t iters,
               int precision, bool io64, void *x_out_d, double *stress_h) {
  if (precision == PPRVIZ_FP64) {
    if (io64)
      return layout_typed<double, double, double>(ctx, (const double *)pdist_d, k, (const double *)x0_d, iters,
                                                  (double *)x_out_d, stress_h);
    return layout_typed<double, float, float>(ctx, (const float *)pdist_d, k, (const float *)x0_d, iters,
                                              (float *)x_out_d, stress_h);
  }
  if (io64)
    return layout_typed<float, double, double>(ctx, (const double *)pdist_d, k, (const double *)x0_d, iters,
                                               (double *)x_out_d, stress_h);
  return layout_typed<float, float, float>(ctx, (const float *)pdist_d, k, (const float *)x0_d, iters,
                                           (float *)x_out_d, stress_h);
}

// Many views, FP32: each view's 1/Delta_s and (L^w + J/k)^-1 are built and
// inverted into slices of two batched matrices, then every update runs as two
// launches over all views together (L^Y pass, apply pass, each with its fused
// partial-sum reduce).
int layout_batch_run(pprviz_ctx *ctx, int32_t nviews, const int64_t *k_h, const float *pdist_d,
                     const float *x0_d, int32_t iters, float *x_out_d, double *stress_h) {
  using V2 = float2;
  std::vector<BatchView> bv((size_t)nviews);
  int64_t mat = 0, vec = 0, part = 0, maxkp = 0;
  size_t ntile = 0;
  for (int32_t v = 0; v < nviews; ++v) {
    const int32_t k = (int32_t)k_h[v];
    const int32_t kp = (k + ST - 1) / ST * ST, nbt = kp / ST;
    bv[v] = BatchView{mat, vec, part, kp, nbt, k};
    mat += (int64_t)kp * kp;
    vec += kp;
    part += (int64_t)nbt * kp;
    maxkp = std::max<int64_t>(maxkp, kp);
    ntile += (size_t)nbt * (nbt + 1) / 2;
  }
  PPRVIZ_TRY(ws_ensure(ctx, WS_BW1, sizeof(float) * (size_t)mat));
  PPRVIZ_TRY(ws_ensure(ctx, WS_BM, sizeof(float) * (size_t)mat));
  PPRVIZ_TRY(ws_ensure(ctx, WS_BX, sizeof(V2) * (size_t)vec * 2));
  PPRVIZ_TRY(ws_ensure(ctx, WS_BPART, sizeof(V2) * (size_t)part));
  PPRVIZ_TRY(ws_ensure(ctx, WS_BTAB, sizeof(BatchView) * (size_t)nviews));
  PPRVIZ_TRY(ws_ensure(ctx, WS_RHS, sizeof(double) * (size_t)(maxkp / 32) * maxkp));
  PPRVIZ_TRY(ws_ensure(ctx, WS_FLAG, 64));
  float *W1 = ctx->ws[WS_BW1].as<float>(), *M = ctx->ws[WS_BM].as<float>();
  V2 *X = ctx->ws[WS_BX].as<V2>(), *Bv = X + vec, *Part = ctx->ws[WS_BPART].as<V2>();
  BatchView *views_d = reinterpret_cast<BatchView *>(ctx->ws[WS_BTAB].p);
  double *rowpart = ctx->ws[WS_RHS].as<double>();
  int *flag = ctx->ws[WS_FLAG].as<int>();
  PPRVIZ_CUDA(ctx, cudaMemcpyAsync(views_d, bv.data(), sizeof(BatchView) * bv.size(), cudaMemcpyHostToDevice,
                                   ctx->stream));
  PPRVIZ_CUDA(ctx, cudaMemsetAsync(flag, 0, sizeof(int), ctx->stream));
  int64_t sq = 0, xo = 0;
  std::vector<int32_t> kps((size_t)nviews);
  std::vector<float *> mats((size_t)nviews);
  for (int32_t v = 0; v < nviews; ++v) {
    const int32_t k = bv[v].k, kp = bv[v].kp;
    const float *Dv = pdist_d + sq;
    { PPRVIZ_PROF(ctx, PPRVIZ_K_FACTOR); k_build_sym<float, float><<<dim3(kp / 32, kp / 32), dim3(32, 8), 0, ctx->stream>>>(k, kp, Dv, W1 + bv[v].mat_off, M + bv[v].mat_off, rowpart, flag); }
    PPRVIZ_LAUNCHED(ctx);
    { PPRVIZ_PROF(ctx, PPRVIZ_K_FACTOR); k_build_diag<float><<<(unsigned)((k + 255) / 256), 256, 0, ctx->stream>>>(k, kp, rowpart, M + bv[v].mat_off); }
    PPRVIZ_LAUNCHED(ctx);
    { PPRVIZ_PROF(ctx, PPRVIZ_K_OTHER); k_load_x<float, float><<<(unsigned)((kp + 255) / 256), 256, 0, ctx->stream>>>(k, kp, x0_d + 2 * xo, X + bv[v].vec_off); }
    PPRVIZ_LAUNCHED(ctx);
    kps[v] = kp;
    mats[v] = M + bv[v].mat_off;
    sq += (int64_t)k * k;
    xo += k;
  }
  // every view's (L^w + J/k)^-1 together, pivot step by pivot step
  if (iters > 0) {
    PPRVIZ_TRY(ws_ensure(ctx, WS_FACB, sizeof(float) * spd_inverse_batch_work(nviews, kps.data())));
    PPRVIZ_TRY(spd_inverse_batch_f32(ctx, nviews, kps.data(), mats.data(), ctx->ws[WS_FACB].as<float>()));
  }
  int hf = 0;
  PPRVIZ_CUDA(ctx, cudaMemcpyAsync(&hf, flag, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
  PPRVIZ_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  if (hf) return set_err(ctx, PPRVIZ_E_INVALID_ARG, "a view's pdist has a non-finite or non-positive entry");
  unsigned pgrid = 0;
  PPRVIZ_TRY(sympass_pipe_grid(ctx, ntile, &pgrid));
  const CUtensorMap *maps = nullptr;
  PPRVIZ_TRY(upload_maps(ctx, bv, W1, M, &maps));
  PassTables pt;
  PPRVIZ_TRY(upload_pass_tables(ctx, bv, pgrid, &pt));
  PPRVIZ_TRY(ws_ensure(ctx, WS_RUNP, sizeof(V2) * ((size_t)pt.nruns * spipe::CWARPS * ST + 1)));
  V2 *RunPart = ctx->ws[WS_RUNP].as<V2>();
  int *perr = flag + 1;
  PPRVIZ_CUDA(ctx, cudaMemsetAsync(perr, 0, sizeof(int), ctx->stream));
  // The updates of a batch are launches only (no host decision between them):
  // they are recorded once into a CUDA graph and the graph is launched. With
  // kernel timing on, or if recording or instantiating fails, the same
  // launches go to the stream directly (timing events mark points of the
  // stream, which a recorded graph does not have).
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t gexec = nullptr;
  bool graphed = false;
  if (iters > 1 && !ctx->profiling && cudaStreamBeginCapture(ctx->stream, cudaStreamCaptureModeRelaxed) == cudaSuccess) {
    int st = PPRVIZ_OK;
    ctx->capturing = true;
    for (int it = 0; it < iters && st == PPRVIZ_OK; ++it)
      st = pass_pair(ctx, pgrid, pt, maps, views_d, X, Bv, Part, RunPart, perr);
    ctx->capturing = false;
    const cudaError_t ec = cudaStreamEndCapture(ctx->stream, &graph);
    if (st == PPRVIZ_OK && ec == cudaSuccess && graph && cudaGraphInstantiate(&gexec, graph, 0) == cudaSuccess &&
        cudaGraphLaunch(gexec, ctx->stream) == cudaSuccess)
      graphed = true;
    if (!graphed) {
      cudaGetLastError();
      ctx->err.clear();
      if (gexec) cudaGraphExecDestroy(gexec);
      if (graph) cudaGraphDestroy(graph);
      gexec = nullptr;
      graph = nullptr;
    }
  } else {
    cudaGetLastError();
  }
  ctx->stats.graph_launched = graphed ? 1 : 0;
  if (!graphed)
    for (int it = 0; it < iters; ++it) PPRVIZ_TRY(pass_pair(ctx, pgrid, pt, maps, views_d, X, Bv, Part, RunPart, perr));
  if (graphed) {
    // the graph has run before the objects go (the wait below is the call's own)
    const cudaError_t es = cudaStreamSynchronize(ctx->stream);
    cudaGraphExecDestroy(gexec);
    cudaGraphDestroy(graph);
    if (es != cudaSuccess) return cuda_err(ctx, es, "layout updates (CUDA graph)");
  }
  if (iters > 0) {
    int herr = 0;
    PPRVIZ_CUDA(ctx, cudaMemcpyAsync(&herr, perr, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    PPRVIZ_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    if (herr) return set_err(ctx, PPRVIZ_E_TIMEOUT, "layout pass: tile copy wait expired");
  }
  ctx->stats.layout_iters = iters;
  double half = 0.0;
  for (int32_t v = 0; v < nviews; ++v) half += 0.5 * (double)bv[v].k * ((double)bv[v].k + 1.0) * sizeof(float);
  ctx->stats.bytes_ly = half * iters;
  ctx->stats.bytes_apply = half * iters;
  // centre and emit each view; stress per view on its input pdist
  int64_t maxk = 0;
  for (int32_t v = 0; v < nviews; ++v) maxk = std::max<int64_t>(maxk, bv[v].k);
  const unsigned eb_max = energy_blocks(maxk);
  PPRVIZ_TRY(ws_ensure(ctx, WS_E, sizeof(V2) * (size_t)maxk + 64));
  PPRVIZ_TRY(ws_ensure(ctx, WS_OUT1, sizeof(double) * ((size_t)eb_max + 1) * nviews));
  V2 *Xc = ctx->ws[WS_E].as<V2>();
  double *ep = ctx->ws[WS_OUT1].as<double>();
  sq = 0;
  xo = 0;
  for (int32_t v = 0; v < nviews; ++v) {
    const int32_t k = bv[v].k;
    const unsigned eb = energy_blocks(k);
    double *epv = ep + (size_t)v * (eb_max + 1);
    { PPRVIZ_PROF(ctx, PPRVIZ_K_OTHER); k_finish<float, float><<<1, 1024, 0, ctx->stream>>>(k, X + bv[v].vec_off, x_out_d + 2 * xo, Xc); }
    PPRVIZ_LAUNCHED(ctx);
    if (stress_h) {
      { PPRVIZ_PROF(ctx, PPRVIZ_K_ENERGY); k_energy<float, false, false><<<eb, ETHREADS, 0, ctx->stream>>>(k, pdist_d + sq, Xc, 1.0f, epv, nullptr, nullptr, flag); }
      PPRVIZ_LAUNCHED(ctx);
      { PPRVIZ_PROF(ctx, PPRVIZ_K_ENERGY); k_reduce_energy<<<1, 256, 0, ctx->stream>>>((int)eb, epv, epv + eb_max); }
      PPRVIZ_LAUNCHED(ctx);
    }
    sq += (int64_t)k * k;
    xo += k;
  }
  if (stress_h) {
    std::vector<double> eh((size_t)(eb_max + 1) * nviews);
    PPRVIZ_CUDA(ctx, cudaMemcpyAsync(eh.data(), ep, sizeof(double) * eh.size(), cudaMemcpyDeviceToHost, ctx->stream));
    PPRVIZ_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    for (int32_t v = 0; v < nviews; ++v) stress_h[v] = eh[(size_t)v * (eb_max + 1) + eb_max];
  }
  return PPRVIZ_OK;
}

template <typename T>
static int energy_typed(pprviz_ctx *ctx, const T *pdist, int32_t k, const T *x, double scale, double *e_h,
                        T *gx, T *gD) {
  using V2 = typename T2<T>::type;
  const unsigned eb = energy_blocks(k);
  PPRVIZ_TRY(ws_ensure(ctx, WS_E, sizeof(V2) * (size_t)k + 64));
  // block partials, then the energy and the status word (read back together)
  PPRVIZ_TRY(ws_ensure(ctx, WS_OUT1, sizeof(double) * (eb + 2)));
  V2 *X = ctx->ws[WS_E].as<V2>();
  double *ep = ctx->ws[WS_OUT1].as<double>();
  int *flag = reinterpret_cast<int *>(ep + eb + 1);
  PPRVIZ_CUDA(ctx, cudaMemsetAsync(flag, 0, sizeof(int), ctx->stream));
  { PPRVIZ_PROF(ctx, PPRVIZ_K_OTHER); k_load_x<T, T><<<(unsigned)((k + 255) / 256), 256, 0, ctx->stream>>>(k, k, x, X); }
  PPRVIZ_LAUNCHED(ctx);
  const T s = (T)scale;
  {
    PPRVIZ_PROF(ctx, PPRVIZ_K_ENERGY);
    if (gx && gD) k_energy<T, true, true><<<eb, ETHREADS, 0, ctx->stream>>>(k, pdist, X, s, ep, gx, gD, flag);
    else if (gx) k_energy<T, true, false><<<eb, ETHREADS, 0, ctx->stream>>>(k, pdist, X, s, ep, gx, gD, flag);
    else if (gD) k_energy<T, false, true><<<eb, ETHREADS, 0, ctx->stream>>>(k, pdist, X, s, ep, gx, gD, flag);
    else k_energy<T, false, false><<<eb, ETHREADS, 0, ctx->stream>>>(k, pdist, X, s, ep, gx, gD, flag);
  }
  PPRVIZ_LAUNCHED(ctx);
  { PPRVIZ_PROF(ctx, PPRVIZ_K_ENERGY); k_reduce_energy<<<1, 256, 0, ctx->stream>>>((int)eb, ep, ep + eb); }
  PPRVIZ_LAUNCHED(ctx);
  struct { double e; int flag, pad; } h = {0.0, 0, 0};
  PPRVIZ_CUDA(ctx, cudaMemcpyAsync(&h, ep + eb, sizeof(h), cudaMemcpyDeviceToHost, ctx->stream));
  PPRVIZ_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  if (h.flag) return set_err(ctx, PPRVIZ_E_INVALID_ARG, "pdist has a non-positive off-diagonal entry");
  if (e_h) *e_h = h.e;
  return PPRVIZ_OK;
}

int energy_run(pprviz_ctx *ctx, const void *pdist_d, int32_t k, const void *x_d, double scale, bool f64,
               double *e_h, void *grad_x_d, void *grad_pdist_d) {
  if (f64)
    return energy_typed<double>(ctx, (const double *)pdist_d, k, (const double *)x_d, scale, e_h,
                                (double *)grad_x_d, (double *)grad_pdist_d);
  return energy_typed<float>(ctx, (const float *)pdist_d, k, (const float *)x_d, scale, e_h, (float *)grad_x_d,
                             (float *)grad_pdist_d);
}

// ---------------------------------------------------------------------------
// Allocation-free energy entry point (pprviz_energy_noalloc).
//
// Some callers may not allocate device memory at the time they need the
// energy: code that owns every byte of the device through its own pool or a
// framework allocator (a cudaMalloc there fails or fragments the pool), code
// running under a hard memory cap, or code that only enqueues work on a stream
// it was handed. For them the scratch of the energy pass (the staged
// coordinates, one FP64 partial per block and a status word) lives in the
// fixed device array below, which every GPU that loads the library holds
// until the process exits. The caller provides inputs and outputs.
// ---------------------------------------------------------------------------
constexpr int kNoAllocMaxK = 65536;
constexpr int kNoAllocBlocks = EBLOCKS;
constexpr size_t kNoAllocXBytes = sizeof(float2) * kNoAllocMaxK;             // 512 KiB
constexpr size_t kNoAllocEBytes = sizeof(double) * (kNoAllocBlocks + 1);     // ~5 KiB
constexpr size_t kNoAllocBytes = kNoAllocXBytes + kNoAllocEBytes + 256;       // + status word

static __device__ __align__(256) unsigned char g_energy_scratch[kNoAllocBytes];

}  // namespace pprviz

#include <mutex>

namespace {

// Device address of g_energy_scratch, looked up once per device. In host code
// the array's name is only a host-side stand-in for the device symbol, so the
// kernels get this address instead.
std::mutex g_noalloc_mu;
void *g_noalloc_addr[256] = {nullptr};

cudaError_t noalloc_scratch(void **out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 256) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_addr[dev]) {
    void *p = nullptr;
    e = cudaGetSymbolAddress(&p, pprviz::g_energy_scratch);
    if (e != cudaSuccess) return e;
    g_noalloc_addr[dev] = p;
  }
  *out = g_noalloc_addr[dev];
  return cudaSuccess;
}

}  // namespace

extern "C" int pprviz_energy_noalloc(const float *pdist, int32_t k, const float *x, double grad_scale, double *e_out,
                                     float *grad_x, float *grad_pdist, void *cuda_stream) {
  using namespace pprviz;
  if (!pdist || !x) return PPRVIZ_E_INVALID_ARG;
  if (k < 1 || k > kNoAllocMaxK) return PPRVIZ_E_INVALID_ARG;
  cudaStream_t stream = (cudaStream_t)cuda_stream;
  void *base = nullptr;
  if (noalloc_scratch(&base) != cudaSuccess) {
    cudaGetLastError();
    return PPRVIZ_E_CUDA;
  }
  float2 *X = reinterpret_cast<float2 *>(base);
  double *eparts = reinterpret_cast<double *>(static_cast<unsigned char *>(base) + kNoAllocXBytes);
  int *flag = reinterpret_cast<int *>(static_cast<unsigned char *>(base) + kNoAllocXBytes + kNoAllocEBytes);
  const unsigned eb = energy_blocks(k);
  // the status word keeps the previous call's value: clear it first
  if (cudaMemsetAsync(flag, 0, sizeof(int), stream) != cudaSuccess) return PPRVIZ_E_CUDA;
  k_load_x<float, float><<<(unsigned)((k + 255) / 256), 256, 0, stream>>>(k, k, x, X);
  const float s = (float)grad_scale;
  if (grad_x && grad_pdist)
    k_energy<float, true, true><<<eb, ETHREADS, 0, stream>>>(k, pdist, X, s, eparts, grad_x, grad_pdist, flag);
  else if (grad_x)
    k_energy<float, true, false><<<eb, ETHREADS, 0, stream>>>(k, pdist, X, s, eparts, grad_x, grad_pdist, flag);
  else if (grad_pdist)
    k_energy<float, false, true><<<eb, ETHREADS, 0, stream>>>(k, pdist, X, s, eparts, grad_x, grad_pdist, flag);
  else
    k_energy<float, false, false><<<eb, ETHREADS, 0, stream>>>(k, pdist, X, s, eparts, grad_x, grad_pdist, flag);
  k_reduce_energy<<<1, 256, 0, stream>>>((int)eb, eparts, eparts + eb);
  if (cudaGetLastError() != cudaSuccess) return PPRVIZ_E_CUDA;
  double e = 0.0;
  int hf = 0;
  if (cudaMemcpyAsync(&e, eparts + eb, sizeof(double), cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
      cudaMemcpyAsync(&hf, flag, sizeof(int), cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
      cudaStreamSynchronize(stream) != cudaSuccess) {
    cudaGetLastError();
    return PPRVIZ_E_CUDA;
  }
  if (hf) return PPRVIZ_E_INVALID_ARG;
  if (e_out) *e_out = e;
  return PPRVIZ_OK;
}
