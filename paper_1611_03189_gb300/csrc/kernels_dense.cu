// Batched variable-size dense kernels of the factorization.
//
//   k_gemm       C = alpha op(A) op(B) + beta C over a list of tasks, one tile
//                per CTA.
//   k_sum        dst = beta dst + alpha sum_s op(src_s), sources summed in list
//                order: block gathers, merges and the deterministic Schur
//                scatter of Sec. 3.2 (several super nodes of one wave updating
//                the same neighbour block).
//   k_chol_inv   A = L L^T and L^-1, one CTA per matrix (pivot blocks A_ss and
//                the small Gram matrices of the CholQR of L^-1 U); FP64 from 97
//                unknowns on a cluster of four (k_chol_cluster).
//   k_trunc      truncation of the well-separated block (Sec. 3.2 eq.
//                local_compression, Sec. 6 GC basis), one CTA per super node:
//                cyclic Jacobi eigen-solves of the Gram matrix A_sw A_sw^T.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cfloat>

#include "hs_internal.h"
#include "trunc_common.cuh"

namespace hs {

namespace {

template <typename T>
struct Lim;
template <>
struct Lim<double> {
  static __device__ __forceinline__ double eps() { return 2.220446049250313e-16; }
  static __device__ __forceinline__ double tiny() { return 1e-290; }
};
template <>
struct Lim<float> {
  static __device__ __forceinline__ float eps() { return 1.1920929e-07f; }
  static __device__ __forceinline__ float tiny() { return 1e-35f; }
};

// the task of CTA b: the last one whose first tile is <= b.  A warp probes 32
// places at a time (4096 tasks: three dependent loads instead of twelve)
__device__ __forceinline__ int find_task(const int *tile_start, int ntasks, int b) {
  const int lane = threadIdx.x & 31;
  int lo = 0, len = ntasks;
  while (len > 1) {
    const int step = (len + 31) / 32;
    const int at = lane * step;
    const unsigned below = __ballot_sync(0xffffffffu, at < len && tile_start[lo + min(at, len - 1)] <= b);
    const int c = __popc(below) - 1;   // tile_start[lo] <= b
    lo += c * step;
    len = min(step, len - c * step);
  }
  return lo;
}

// ---------------------------------------------------------------------------
// batched GEMM: one tile of TM x TN outputs per CTA, RM x RN adjacent ones per
// thread, operands staged through shared memory GK rows at a time, the next
// rows loaded while the current ones are used.  An output is the sum over k in
// order, whatever the tile, so a task gets the same bits in any launch.
//
// Symmetric products (task.sym) run the tiles on and below the diagonal and
// write each value to both places; operands with a triangle of zeros
// (task.kmode) limit a tile's k to the part that is not zero.  Both leave the
// results as they are and take about half of the factorization's products'
// work away.
//
// Tile sizes.  FP32: 64 x 64, 4 x 4 a thread (bound by the FMA rate when the
// tiles fill the GPU); 32 x 32 when they do not, or when most of a 64 x 64
// tile would be padding.  FP64: its rate (1/64 of FP32's) bounds any tile, so
// the tiles are small to spread a wave's few large products over the SMs:
// 32 x 32, or 16 x 16 below 8 tiles an SM (a 320^3 product: 25 tiles of 64 x 64
// keep 25 SMs busy for 330 us; 400 of 16 x 16 take about 60).
// ---------------------------------------------------------------------------
template <typename T, int TM, int RM, int GK>
__global__ void __launch_bounds__((TM / RM) * (TM / RM)) k_gemm(const GemmTask<T> *__restrict__ tasks,
                                                                const int *__restrict__ tile_start, int ntasks) {
  constexpr int TX = TM / RM, NT = TX * TX, E = TM * GK / NT;
  constexpr int LD = TM + 16 / (int)sizeof(T);
  __shared__ __align__(16) T As[2][GK][LD];
  __shared__ __align__(16) T Bs[2][GK][LD];
  const int ti = find_task(tile_start, ntasks, blockIdx.x);
  const GemmTask<T> t = tasks[ti];
  const int local = blockIdx.x - tile_start[ti];
  int tr, tc;
  if (t.sym) {
    tr = (int)((sqrtf(8.f * (float)local + 1.f) - 1.f) * 0.5f);
    while (tr * (tr + 1) / 2 > local) --tr;
    while ((tr + 1) * (tr + 2) / 2 <= local) ++tr;
    tc = local - tr * (tr + 1) / 2;
  } else {
    const int tiles_n = (t.N + TM - 1) / TM;
    tr = local / tiles_n;
    tc = local % tiles_n;
  }
  const int row0 = tr * TM, col0 = tc * TM;
  int k_lo = 0, k_hi = t.K;
  if (t.kmode & GEMM_A_LOW) k_hi = min(k_hi, row0 + TM);
  if (t.kmode & GEMM_A_UP) k_lo = max(k_lo, row0);
  if (t.kmode & GEMM_B_UP) k_hi = min(k_hi, col0 + TM);
  if (t.kmode & GEMM_B_LOW) k_lo = max(k_lo, col0);
  const int tid = threadIdx.x;
  const int tx = tid % TX, ty = tid / TX;
  T acc[RM][RM];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RM; ++j) acc[i][j] = T(0);
  T ra[E], rb[E];
  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < E; ++q) {
      const int e = tid + NT * q;
      {
        const int i = t.ta == 0 ? e / GK : e % TM, k = t.ta == 0 ? e % GK : e / TM;
        const int gi = row0 + i, gk = k0 + k;
        ra[q] = gi < t.M && gk < k_hi ? (t.ta == 0 ? t.A[(int64_t)gi * t.lda + gk] : t.A[(int64_t)gk * t.lda + gi])
                                      : T(0);
      }
      {
        const int j = t.tb == 0 ? e % TM : e / GK, k = t.tb == 0 ? e / TM : e % GK;
        const int gj = col0 + j, gk = k0 + k;
        rb[q] = gj < t.N && gk < k_hi ? (t.tb == 0 ? t.B[(int64_t)gk * t.ldb + gj] : t.B[(int64_t)gj * t.ldb + gk])
                                      : T(0);
      }
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int q = 0; q < E; ++q) {
      const int e = tid + NT * q;
      if (t.ta == 0)
        As[buf][e % GK][e / GK] = ra[q];
      else
        As[buf][e / TM][e % TM] = ra[q];
      if (t.tb == 0)
        Bs[buf][e / TM][e % TM] = rb[q];
      else
        Bs[buf][e % GK][e / GK] = rb[q];
    }
  };
  if (k_lo < k_hi) {
    load(k_lo);
    store(0);
  }
  __syncthreads();
  int buf = 0;
  for (int k0 = k_lo; k0 < k_hi; k0 += GK) {
    const bool more = k0 + GK < k_hi;
    if (more) load(k0 + GK);
#pragma unroll
    for (int kk = 0; kk < GK; ++kk) {
      T a[RM], b[RM];
#pragma unroll
      for (int i = 0; i < RM; ++i) a[i] = As[buf][kk][ty * RM + i];
#pragma unroll
      for (int j = 0; j < RM; ++j) b[j] = Bs[buf][kk][tx * RM + j];
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RM; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    if (more) store(buf ^ 1);   // (read last before the barrier of the pass before)
    __syncthreads();
    buf ^= 1;
  }
#pragma unroll
  for (int i = 0; i < RM; ++i) {
    const int r = row0 + ty * RM + i;
    if (r >= t.M) continue;
#pragma unroll
    for (int j = 0; j < RM; ++j) {
      const int c = col0 + tx * RM + j;
      if (c >= t.N) continue;
      T *p = t.C + (int64_t)r * t.ldc + c;
      T v = t.alpha * acc[i][j];
      if (t.beta != T(0)) v = fma(t.beta, *p, v);
      *p = v;
      if (t.sym && tr != tc) t.C[(int64_t)c * t.ldc + r] = v;
    }
  }
}

// ---------------------------------------------------------------------------
// batched deterministic accumulate / copy
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) k_sum(const SumTask<T> *__restrict__ tasks,
                                             const SumSrc<T> *__restrict__ srcs,
                                             const int *__restrict__ tile_start, int ntasks) {
  __shared__ T sm[SUM_TILE][SUM_TILE + 1];
  const int ti = find_task(tile_start, ntasks, blockIdx.x);
  const SumTask<T> t = tasks[ti];
  const int local = blockIdx.x - tile_start[ti];
  const int tiles_c = (t.cols + SUM_TILE - 1) / SUM_TILE;
  const int i0 = (local / tiles_c) * SUM_TILE;
  const int j0 = (local % tiles_c) * SUM_TILE;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8
  T acc[4] = {T(0), T(0), T(0), T(0)};
  for (int s = 0; s < t.nsrc; ++s) {
    const SumSrc<T> src = srcs[t.first + s];
    if (!src.trans) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int i = i0 + ty + 8 * r, j = j0 + tx;
        if (i < t.rows && j < t.cols) acc[r] += src.ptr[(int64_t)i * src.ld + j];
      }
    } else {
      __syncthreads();
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int jj = ty + 8 * r, ii = tx;
        T v = T(0);
        if (i0 + ii < t.rows && j0 + jj < t.cols) v = src.ptr[(int64_t)(j0 + jj) * src.ld + i0 + ii];
        sm[jj][ii] = v;
      }
      __syncthreads();
#pragma unroll
      for (int r = 0; r < 4; ++r) acc[r] += sm[tx][ty + 8 * r];
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int i = i0 + ty + 8 * r, j = j0 + tx;
    if (i < t.rows && j < t.cols) {
      T *p = t.dst + (int64_t)i * t.ld + j;
      T v = t.alpha * acc[r];
      if (t.beta != T(0)) v = fma(t.beta, *p, v);
      *p = v;
    }
  }
}

// ---------------------------------------------------------------------------
// Cholesky and inverse of the factor, one CTA per matrix, in shared memory.
//
// Block columns of 16.  Step b, with j0 = 16 b, L_b its diagonal block, D_b = L_b^-1:
//   panel   P_i = L_ib = W_ib L_b^-T for the rows i below, and the finished block
//           row X_b,0:j0 = -L_b^-1 R_b of the inverse, by substitution, one thread
//           per row or column;
//   update  W_i,c -= P_i P_c^T (c > b, the trailing block) and
//           R_i,c += P_i X_b,c (c <= b, X_bb = D_b): the sums R_i = sum_p L_ip X_p
//           of the inverse's rows grow in place of the columns of L that are no
//           longer needed, so both halves are one rank-16 update of whole rows,
//           in 32 x 16 tiles per warp, 4 x 4 outputs a lane, 16-byte loads along
//           k (P) or along the row (X).
// The only serial chain is the 16 x 16 diagonal block: one warp factors it in
// registers, half its lanes the rows, half D_b's columns.  Warp 0 updates
// the next diagonal block first and factors it while the other warps finish
// the update.  Two barriers per 16 columns.
// What bounds it: the diagonal chain up to m of about 100, the CUDA cores' FMA
// rate above (FP64: throughout).  Twelve matrices a launch, m = 48 / 128 / 224:
// 16.5 / 45 / 115 us in FP32 (column by column, two barriers a column, 49 / 207 /
// 564), 74 / 225 us at 48 / 128 in FP64 (182 / 816).
// Errors of the inverse against one of higher precision, over sizes 8 to 224 and
// conditions 1e1 to 1e5, are below those of the elimination column by column
// (||X A X^T - I|| 0.83 times its value, geometric mean).
// ---------------------------------------------------------------------------
constexpr int kCholNb = 16;

// row strides in elements: odd multiples of 16 bytes, so that 8 consecutive
// rows' 16-byte pieces fall into different banks
template <typename T>
__host__ __device__ constexpr int chol_ps() {
  return kCholNb + 16 / (int)sizeof(T);
}
template <typename T>
__host__ __device__ inline int chol_ld(int m) {
  constexpr int v = 16 / (int)sizeof(T);
  const int q = (m + v - 1) / v;
  return v * (q | 1);
}
template <typename T>
__host__ __device__ inline size_t chol_smem_bytes(int m) {
  return sizeof(T) * (size_t)m * (chol_ld<T>(m) + chol_ps<T>());
}

// v[0 .. 16 / sizeof(T)) = 16 bytes at p
__device__ __forceinline__ void ld16(const float *p, float *v) {
  const float4 q = *reinterpret_cast<const float4 *>(p);
  v[0] = q.x;
  v[1] = q.y;
  v[2] = q.z;
  v[3] = q.w;
}
__device__ __forceinline__ void ld16(const double *p, double *v) {
  const double2 q = *reinterpret_cast<const double2 *>(p);
  v[0] = q.x;
  v[1] = q.y;
}
__device__ __forceinline__ void st16(float *p, const float *v) {
  *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void st16(double *p, const double *v) {
  *reinterpret_cast<double2 *>(p) = make_double2(v[0], v[1]);
}
// d^-1/2 (CUDA's: rounded correctly, and within one unit in the last place)
__device__ __forceinline__ float inv_sqrt(float d) { return __frsqrt_rn(d); }
__device__ __forceinline__ double inv_sqrt(double d) { return rsqrt(d); }

// One warp: the diagonal block at row j0, column j0c of W (jb <= 16 columns, j0 the
// first in the matrix) becomes D = L^-1, with zeros above the diagonal; L goes to
// Lt, transposed (L_ij at Lt[16 j + i], i > j; 1 / L_jj at Lt[17 j]; rows from jb
// on those of the identity).  *fail = first failing pivot + 1.
template <typename T>
__device__ __forceinline__ void chol_diag(T *W, int ld, int j0, int j0c, int jb, T *Lt, int *fail) {
  // lanes 0 .. 15: row i of A, becoming L's; lanes 16 .. 31: column i of D.  Both
  // are scaled by the pivot's inverse root and updated by L's column j.
  const int lane = threadIdx.x & 31, i = lane & 15;
  const bool inverse = lane >= 16;
  T r[kCholNb];
#pragma unroll
  for (int c = 0; c < kCholNb; ++c)
    r[c] = !inverse && i < jb && c <= i ? W[(size_t)(j0 + i) * ld + j0c + c] : (c == i ? T(1) : T(0));
  int bad = 0;
#pragma unroll
  for (int j = 0; j < kCholNb; ++j) {
    T d = __shfl_sync(0xffffffffu, r[j], j);
    if (!(d > T(0)) || !isfinite(d)) {
      if (!bad) bad = j0 + j + 1;
      d = T(1);
    }
    const T is = inv_sqrt(d);
    r[j] *= is;   // L_ij, D_ji
    if (!inverse && i >= j) Lt[kCholNb * j + i] = i == j ? is : r[j];
#pragma unroll
    for (int c = j + 1; c < kCholNb; ++c) r[c] = fma(-r[j], __shfl_sync(0xffffffffu, r[j], c), r[c]);
  }
  __syncwarp();
  if (inverse && i < jb) {
#pragma unroll
    for (int c = 0; c < kCholNb; ++c)
      if (c < jb) W[(size_t)(j0 + c) * ld + j0c + i] = r[c];
  }
  if (bad && lane == 0) *fail = bad;
  __syncwarp();
}

// v <- L_b^-1 v by substitution (Lt: chol_diag's).  (The product with D_b instead
// has an error larger by the block's condition number: at a condition of 1e5 the
// inverse's error was up to 2.3 times that of the substitution.)
template <typename T>
__device__ __forceinline__ void chol_solve(const T *Lt, T (&v)[kCholNb]) {
  constexpr int V = 16 / (int)sizeof(T);
#pragma unroll
  for (int k = 0; k < kCholNb; ++k) {
    T l[kCholNb];
#pragma unroll
    for (int j = k / V * V; j < kCholNb; j += V) ld16(Lt + kCholNb * k + j, l + j);
    v[k] *= l[k];
#pragma unroll
    for (int j = k + 1; j < kCholNb; ++j) v[j] = fma(-l[j], v[k], v[j]);
  }
}

// Matrices up to this size update the trailing block term by term, larger ones add
// up 16 terms before they take them off.  The sums have 0.4 to 0.9 times the error
// above it, but up to 1.6 times below 64 at a graded spectrum of condition 1e5,
// where the terms are larger than what is left.
constexpr int kCholInOrder = 96;

struct NoShift {
  __device__ __forceinline__ operator int() const { return 0; }
};

// Rank-16 update of the tile at rows i0 .. i0 + 31, columns c0 .. c0 + 15,
// which W holds from its column c0 + shift on (a constant 0 in one CTA: a
// variable there costs registers and a tenth of the kernel).
// kind 0: W -= P_i P_c^T; 1: W += P_i X_b; 2: W = P_i X_b (X_b: rows j0 ..)
template <typename T, typename Shift>
__device__ __forceinline__ void chol_tile(T *W, int ld, const T *P, int i0, int c0, Shift shift, int j0, int m, int kind) {
  constexpr int V = 16 / (int)sizeof(T), PS = chol_ps<T>();
  const int lane = threadIdx.x & 31;
  const int ib = i0 + (lane & 7), cg = c0 + 4 * (lane >> 3), cb = cg + shift;
  // in order: the tile's own values first, then one term after another, as an
  // elimination column by column takes them off
  const bool in_order = kind == 0 && m <= kCholInOrder;
  T acc[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; c += V) {
      const int i = ib + 8 * r;
      if (in_order && i < m && cb + c < ld) {
        ld16(W + (size_t)i * ld + cb + c, &acc[r][c]);
      } else {
#pragma unroll
        for (int u = 0; u < V; ++u) acc[r][c + u] = T(0);
      }
    }
  const T *pa[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) pa[r] = P + (size_t)min(ib + 8 * r, m - 1) * PS;
  if (kind == 0) {
    const T *pb[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) pb[c] = P + (size_t)min(cg + c, m - 1) * PS;
#pragma unroll
    for (int k = 0; k < kCholNb; k += V) {
      T a[4][V], b[4][V];
#pragma unroll
      for (int r = 0; r < 4; ++r) ld16(pa[r] + k, a[r]);
#pragma unroll
      for (int c = 0; c < 4; ++c) ld16(pb[c] + k, b[c]);
#pragma unroll
      for (int u = 0; u < V; ++u)
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[r][c] = fma(-a[r][u], b[c][u], acc[r][c]);
    }
  } else {
    const T *xb = W + (size_t)j0 * ld + cb;
#pragma unroll
    for (int k = 0; k < kCholNb; k += V) {
      T a[4][V], b[V][4];
#pragma unroll
      for (int r = 0; r < 4; ++r) ld16(pa[r] + k, a[r]);
#pragma unroll
      for (int u = 0; u < V; ++u)
#pragma unroll
        for (int c = 0; c < 4; c += V) ld16(xb + (size_t)(k + u) * ld + c, &b[u][c]);
#pragma unroll
      for (int u = 0; u < V; ++u)
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[r][c] = fma(a[r][u], b[u][c], acc[r][c]);
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int i = ib + 8 * r;
    if (i >= m) continue;
#pragma unroll
    for (int c = 0; c < 4; c += V) {
      if (cb + c >= ld) continue;   // the last trailing columns; ld is a multiple of V
      T *p = W + (size_t)i * ld + cb + c;
      if (kind != 2 && !in_order) {
        T w[V];
        ld16(p, w);
#pragma unroll
        for (int u = 0; u < V; ++u) acc[r][c + u] += w[u];
      }
      st16(p, &acc[r][c]);
    }
  }
}

template <typename T, int NT>
__global__ void __launch_bounds__(NT) k_chol_inv(const CholTask<T> *__restrict__ tasks, int *__restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(16) T s_l[kCholNb * kCholNb];
  __shared__ int s_fail;
  constexpr int V = 16 / (int)sizeof(T), PS = chol_ps<T>(), NW = NT / 32;
  const CholTask<T> t = tasks[blockIdx.x];
  const int m = t.m, ld = chol_ld<T>(m);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (m == 0) {
    if (tid == 0) status[t.status_idx] = 0;
    return;
  }
  T *W = reinterpret_cast<T *>(smem_raw);
  T *P = W + (size_t)m * ld;
  if (tid == 0) s_fail = 0;
  for (int i = warp; i < m; i += NW)
    for (int c = lane; c < ld; c += 32) W[(size_t)i * ld + c] = c <= i ? t.A[(int64_t)i * t.lda + c] : T(0);
  __syncthreads();
  if (warp == 0) chol_diag<T>(W, ld, 0, 0, min(kCholNb, m), s_l, &s_fail);
  for (int j0 = 0; j0 < m; j0 += kCholNb) {
    __syncthreads();   // D_b, L_b and the update of the step before are complete
    if (s_fail) break;
    const int j1 = min(j0 + kCholNb, m), jb = j1 - j0, rest = m - j1;
    for (int q = tid; q < rest + j0; q += NT) {
      T v[kCholNb];
      if (q < rest) {
        // row j1 + q of the panel (a full block: jb = 16)
        const T *w = W + (size_t)(j1 + q) * ld + j0;
#pragma unroll
        for (int k = 0; k < kCholNb; k += V) ld16(w + k, v + k);
        chol_solve<T>(s_l, v);
#pragma unroll
        for (int k = 0; k < kCholNb; k += V) st16(P + (size_t)(j1 + q) * PS + k, v + k);
      } else {
        // column q - rest of the inverse's block row
        T *w = W + (size_t)j0 * ld + (q - rest);
#pragma unroll
        for (int k = 0; k < kCholNb; ++k) v[k] = k < jb ? -w[(size_t)k * ld] : T(0);
        chol_solve<T>(s_l, v);
#pragma unroll
        for (int k = 0; k < kCholNb; ++k)
          if (k < jb) w[(size_t)k * ld] = v[k];
      }
    }
    __syncthreads();
    if (rest == 0) break;
    if (warp == 0) {
      chol_tile<T>(W, ld, P, j1, j1, NoShift(), j0, m, 0);
      __syncwarp();
      chol_diag<T>(W, ld, j1, j1, min(kCholNb, m - j1), s_l, &s_fail);
    } else {
      // all other tiles, dealt out to the other warps in turn
      const int nic = j1 / kCholNb, nct = (rest + kCholNb - 1) / kCholNb;
      int turn = 1;
      for (int rt = 0; rt * 32 < rest; ++rt) {
        const int ntr = min(2 * (rt + 1), nct);
        for (int ct = 0; ct < nic + ntr; ++ct) {
          if (rt == 0 && ct == nic) continue;   // warp 0's
          if (turn == warp) {
            if (ct < nic)
              chol_tile<T>(W, ld, P, j1 + 32 * rt, kCholNb * ct, NoShift(), j0, m, ct == nic - 1 ? 2 : 1);
            else
              chol_tile<T>(W, ld, P, j1 + 32 * rt, j1 + kCholNb * (ct - nic), NoShift(), j0, m, 0);
          }
          turn = turn + 1 == NW ? 1 : turn + 1;
        }
      }
    }
  }
  __syncthreads();
  const int st = s_fail;
  if (st == 0)
    for (int i = warp; i < m; i += NW)
      for (int c = lane; c < m; c += 32) t.Linv[(int64_t)i * t.ldl + c] = c <= i ? W[(size_t)i * ld + c] : T(0);
  if (tid == 0) status[t.status_idx] = st;
}

// The same factorization by a cluster of kCholC CTAs, for FP64 matrices above
// kCholClusterMin, where one SM's FP64 rate (2 FMAs a cycle) bounds it.
// Blocks of 16 columns are dealt out cyclically and stay with their CTA, first
// as trailing columns, then as the inverse's.  A step needs D_b and the panel
// P_b alone from elsewhere: their owner writes them into every CTA's shared
// memory, so a step has one cluster barrier.  The owner of block b + 1 updates
// that block first, and its diagonal block is inverted beside its other tiles.
// Every element's arithmetic is k_chol_inv's, so a smaller matrix in a launch with
// such a one keeps its bits.
constexpr int kCholC = 4, kCholClusterMin = 96, kCholClThreads = 256;

__host__ __device__ inline int chol_cl_ld(int m) {
  const int nblk = (m + kCholNb - 1) / kCholNb;
  return kCholNb * ((nblk + kCholC - 1) / kCholC) + 2;
}
template <typename T>
__host__ __device__ inline size_t chol_cl_smem_bytes(int m) {
  return sizeof(T) * ((size_t)m * (chol_cl_ld(m) + 2 * chol_ps<T>()) + 2 * kCholNb * kCholNb);
}

template <typename T>
__global__ void __cluster_dims__(kCholC, 1, 1) __launch_bounds__(kCholClThreads)
    k_chol_cluster(const CholTask<T> *__restrict__ tasks, int *__restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(16) T s_l[kCholNb * kCholNb];
  __shared__ int s_fail, s_failed[2];   // found here; published with L_b (step parity)
  constexpr int V = 16 / (int)sizeof(T), PS = chol_ps<T>(), NT = kCholClThreads, NW = NT / 32;
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  const int rank = (int)cluster.block_rank();
  const CholTask<T> t = tasks[blockIdx.x / kCholC];
  const int m = t.m, ld = chol_cl_ld(m), nblk = (m + kCholNb - 1) / kCholNb;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  T *W = reinterpret_cast<T *>(smem_raw);          // own block q: block rank + kCholC q, from column 16 q on
  T *Pb = W + (size_t)m * ld, *Lb = Pb + 2 * (size_t)m * PS;   // two buffers each (step parity)
  if (m == 0) {
    if (tid == 0 && rank == 0) status[t.status_idx] = 0;
    return;
  }
  if (tid == 0) s_fail = 0;
  for (int i = warp; i < m; i += NW)
    for (int c = lane; c < ld; c += 32) {
      const int g = kCholNb * (rank + kCholC * (c / kCholNb)) + c % kCholNb;
      W[(size_t)i * ld + c] = g <= i ? t.A[(int64_t)i * t.lda + g] : T(0);
    }
  cluster.sync();   // (every CTA runs before any writes to it)
  // L_b and its panel to every CTA
  auto publish = [&](int b) {
    const int j0 = b * kCholNb, j1 = min(j0 + kCholNb, m), lc = kCholNb * (b / kCholC), par = b & 1;
    for (int q = tid; q < kCholNb * kCholNb; q += NT)
      if (q % kCholNb >= q / kCholNb)
        for (int r = 0; r < kCholC; ++r) cluster.map_shared_rank(Lb, r)[par * kCholNb * kCholNb + q] = s_l[q];
    for (int i = j1 + tid; i < m; i += NT) {
      const T *w = W + (size_t)i * ld + lc;
      T v[kCholNb];
#pragma unroll
      for (int k = 0; k < kCholNb; k += V) ld16(w + k, v + k);
      chol_solve<T>(s_l, v);
      for (int r = 0; r < kCholC; ++r) {
        T *P = cluster.map_shared_rank(Pb, r) + ((size_t)par * m + i) * PS;
#pragma unroll
        for (int k = 0; k < kCholNb; k += V) st16(P + k, v + k);
      }
    }
    if (tid < kCholC) cluster.map_shared_rank(s_failed, tid)[par] = s_fail;
  };
  if (rank == 0) {
    if (warp == 0) chol_diag<T>(W, ld, 0, 0, min(kCholNb, m), s_l, &s_fail);
    __syncthreads();
    publish(0);
  }
  int fail = 0;
  for (int b = 0; b < nblk; ++b) {
    cluster.sync();   // L_b, P_b are here; every CTA is done with step b - 1
    fail = s_failed[b & 1];
    if (fail) break;
    const int j0 = b * kCholNb, j1 = min(j0 + kCholNb, m), jb = j1 - j0, rest = m - j1;
    const T *P = Pb + (size_t)(b & 1) * m * PS, *Lt = Lb + (b & 1) * kCholNb * kCholNb;
    // row block b of the inverse, own columns (blocks before b)
    const int nq = b > rank ? (b - rank + kCholC - 1) / kCholC : 0;   // own blocks before b
    for (int c = tid; c < kCholNb * nq; c += NT) {
      T *w = W + (size_t)j0 * ld + c;
      T v[kCholNb];
#pragma unroll
      for (int k = 0; k < kCholNb; ++k) v[k] = k < jb ? -w[(size_t)k * ld] : T(0);
      chol_solve<T>(Lt, v);
#pragma unroll
      for (int k = 0; k < kCholNb; ++k)
        if (k < jb) w[(size_t)k * ld] = v[k];
    }
    if (rest == 0) break;
    __syncthreads();
    const int nrt = (rest + 31) / 32, nown = rank < nblk ? (nblk - rank + kCholC - 1) / kCholC : 0;
    const bool next = (b + 1) % kCholC == rank;
    const int qn = next ? (b + 1) / kCholC : -1;
    if (next) {
      for (int rt = warp; rt < nrt; rt += NW)
        chol_tile<T>(W, ld, P, j1 + 32 * rt, j1, kCholNb * qn - j1, j0, m, 0);
      __syncthreads();
      if (warp == 0)
        chol_diag<T>(W, ld, j1, kCholNb * qn, min(kCholNb, m - j1), s_l, &s_fail);
    }
    // the other own tiles (the owner of the next block's warp 0 has its diagonal block)
    if (!next || warp != 0) {
      const int w0 = next ? 1 : 0;
      int turn = w0;
      for (int q = 0; q < nown; ++q) {
        if (q == qn) continue;
        const int blk = rank + kCholC * q, c0 = kCholNb * blk;
        for (int rt = 0; rt < nrt; ++rt) {
          const int i0 = j1 + 32 * rt;
          if (blk > b && i0 + 31 < c0) continue;   // above the diagonal
          if (turn == warp)
            chol_tile<T>(W, ld, P, i0, c0, kCholNb * q - c0, j0, m, blk > b ? 0 : blk == b ? 2 : 1);
          turn = turn + 1 == NW ? w0 : turn + 1;
        }
      }
    }
    if (next) {
      __syncthreads();
      publish(b + 1);
    }
  }
  __syncthreads();
  if (fail == 0)
    for (int i = warp; i < m; i += NW)
      for (int c = lane; c < ld; c += 32) {
        const int g = kCholNb * (rank + kCholC * (c / kCholNb)) + c % kCholNb;
        if (c < ld - 2 && g < m) t.Linv[(int64_t)i * t.ldl + g] = g <= i ? W[(size_t)i * ld + c] : T(0);
      }
  if (tid == 0 && rank == 0) status[t.status_idx] = fail;
}

// ---------------------------------------------------------------------------
// truncation: cyclic Jacobi on the Gram matrix (round-robin pair ordering)
// ---------------------------------------------------------------------------
constexpr int TRUNC_THREADS = 256;

template <typename T>
struct JacobiShared {
  int *pp, *qq;
  T *cs, *sn;
  int *flag;
};

template <typename T>
__device__ double block_sum(double v, double *red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0) {
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
    red[32] = s;
  }
  __syncthreads();
  s = red[32];
  __syncthreads();
  return s;
}

// Eigen-decomposition A = V diag(A') V^T of the symmetric m x m matrix A (ld
// m), in place: on exit diag(A) holds the eigenvalues.  V is filled when
// want_v.  Returns the number of sweeps.
template <typename T>
__device__ int jacobi_eig(T *A, T *V, int m, bool want_v, JacobiShared<T> sh, int max_sweeps) {
  const int tid = threadIdx.x, nt = blockDim.x;
  if (want_v)
    for (int64_t e = tid; e < (int64_t)m * m; e += nt) V[e] = (e / m == e % m) ? T(1) : T(0);
  if (m < 2) {
    __syncthreads();
    return 0;
  }
  // scale for the absolute floor of the rotation test
  T scale = T(0);
  for (int i = 0; i < m; ++i) scale = fmax(scale, fabs(A[i * m + i]));
  // entries below eps * scale move no eigenvalue by more than the rounding of
  // the whole computation: treat them as converged (otherwise rounding noise
  // in the near-null space keeps every sweep busy)
  const T floor_abs = Lim<T>::eps() * scale + Lim<T>::tiny();
  const int mp = m + (m & 1);
  const int np = mp / 2;
  int sweep = 0;
  for (; sweep < max_sweeps; ++sweep) {
    if (tid == 0) *sh.flag = 0;
    __syncthreads();
    for (int r = 0; r < mp - 1; ++r) {
      for (int i = tid; i < np; i += nt) {
        int a, b;
        if (i == 0) {
          a = r;
          b = mp - 1;
        } else {
          a = (r + i) % (mp - 1);
          b = (r - i + (mp - 1)) % (mp - 1);
        }
        if (a > b) {
          const int x = a;
          a = b;
          b = x;
        }
        T c = T(1), s = T(0);
        if (b < m) {
          const T app = A[a * m + a], aqq = A[b * m + b], apq = A[a * m + b];
          if (fabs(apq) > Lim<T>::eps() * sqrt(fabs(app * aqq)) && fabs(apq) > floor_abs) {
            const T th = (aqq - app) / (T(2) * apq);
            const T ath = fabs(th);
            const T root = (ath > T(1)) ? ath * sqrt(T(1) + (T(1) / ath) * (T(1) / ath))
                                        : sqrt(T(1) + th * th);
            T tt = T(1) / (ath + root);
            if (th < T(0)) tt = -tt;
            c = T(1) / sqrt(T(1) + tt * tt);
            s = tt * c;
            *sh.flag = 1;
          }
        }
        sh.pp[i] = a;
        sh.qq[i] = b;
        sh.cs[i] = c;
        sh.sn[i] = s;
      }
      __syncthreads();
      // A <- J^T A J, 2 x 2 blocks of (pair i rows) x (pair j cols)
      for (int w = tid; w < np * np; w += nt) {
        const int i = w / np, j = w - (w / np) * np;
        const T si = sh.sn[i], sj = sh.sn[j];
        if (si == T(0) && sj == T(0)) continue;
        const T ci = sh.cs[i], cj = sh.cs[j];
        const int a = sh.pp[i], b = sh.qq[i], c = sh.pp[j], d = sh.qq[j];
        const bool bv = b < m, dv = d < m;
        const T x00 = A[a * m + c];
        const T x01 = dv ? A[a * m + d] : T(0);
        const T x10 = bv ? A[b * m + c] : T(0);
        const T x11 = (bv && dv) ? A[b * m + d] : T(0);
        // right: columns (c, d) <- (cj col_c - sj col_d, sj col_c + cj col_d)
        const T y00 = cj * x00 - sj * x01, y01 = sj * x00 + cj * x01;
        const T y10 = cj * x10 - sj * x11, y11 = sj * x10 + cj * x11;
        // left: rows (a, b) <- (ci row_a - si row_b, si row_a + ci row_b)
        T z00 = ci * y00 - si * y10, z01 = ci * y01 - si * y11;
        T z10 = si * y00 + ci * y10, z11 = si * y01 + ci * y11;
        if (i == j && si != T(0)) {
          z01 = T(0);
          z10 = T(0);
        }
        A[a * m + c] = z00;
        if (dv) A[a * m + d] = z01;
        if (bv) A[b * m + c] = z10;
        if (bv && dv) A[b * m + d] = z11;
      }
      if (want_v) {
        for (int w = tid; w < m * np; w += nt) {
          const int row = w / np, j = w - (w / np) * np;
          const T sj = sh.sn[j];
          if (sj == T(0)) continue;
          const T cj = sh.cs[j];
          const int c = sh.pp[j], d = sh.qq[j];
          const T v0 = V[row * m + c], v1 = V[row * m + d];
          V[row * m + c] = cj * v0 - sj * v1;
          V[row * m + d] = sj * v0 + cj * v1;
        }
      }
      __syncthreads();
    }
    const int any = *sh.flag;
    __syncthreads();
    if (!any) break;
  }
  return sweep;
}

// Selects the columns of V whose eigenvalues (diag of A) exceed thr, in
// descending order, writing them to U columns col0 .. col0+k-1.  Returns k.
template <typename T>
__device__ int select_columns(const T *A, const T *V, int m, double thr, T *U, int col0,
                              double *red) {
  int cnt = 0;
  for (int i = threadIdx.x; i < m; i += blockDim.x)
    if ((double)A[i * m + i] > thr) ++cnt;
  const int k = (int)(block_sum<T>((double)cnt, red) + 0.5);
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    const T di = A[i * m + i];
    if (!((double)di > thr)) continue;
    int rank = 0;
    for (int j = 0; j < m; ++j) {
      const T dj = A[j * m + j];
      if (dj > di || (dj == di && j < i)) ++rank;
    }
    if (col0 + rank >= m) continue;
    for (int r = 0; r < m; ++r) U[(int64_t)r * m + col0 + rank] = V[(int64_t)r * m + i];
  }
  __syncthreads();
  return k;
}

template <typename T>
__global__ void __launch_bounds__(TRUNC_THREADS) k_trunc(const TruncTask<T> *__restrict__ tasks,
                                                        int *__restrict__ kout, int variant) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[33];
  __shared__ int flag;
  __shared__ double s_gR[kMaxK1 * 2 * kMaxPhi], s_gW[kMaxK1 * kMaxK1 + kMaxK1];
  __shared__ int s_gk;
  __shared__ T s_c[kMaxK1 * kMaxK1];
  const TruncTask<T> t = tasks[blockIdx.x];
  const double eps = t.eps;
  const int m = t.m;
  const int mp = m + (m & 1);
  const int np = mp / 2 > 0 ? mp / 2 : 1;
  unsigned char *p = smem_raw;
  T *A = reinterpret_cast<T *>(p);
  p += sizeof(T) * (size_t)m * m;
  T *V = reinterpret_cast<T *>(p);
  p += sizeof(T) * (size_t)m * m;
  JacobiShared<T> sh;
  sh.cs = reinterpret_cast<T *>(p);
  p += sizeof(T) * np;
  sh.sn = reinterpret_cast<T *>(p);
  p += sizeof(T) * np;
  sh.pp = reinterpret_cast<int *>(p);
  p += sizeof(int) * np;
  sh.qq = reinterpret_cast<int *>(p);
  sh.flag = &flag;
  const int tid = threadIdx.x, nt = blockDim.x;
  if (m == 0) {
    if (tid == 0) kout[t.k_idx] = 0;
    return;
  }
  if (variant == HS_LORASP && eps == 0.0) {
    // no truncation: complete basis U = I
    for (int64_t e = tid; e < (int64_t)m * m; e += nt) t.U[e] = (e / m == e % m) ? T(1) : T(0);
    if (tid == 0) kout[t.k_idx] = m;
    return;
  }
  // ---- GC basis U_1 (Sec. 6: orth[phi_s, A_sw phi_w]; Appendix B: its
  // dominant left singular vectors), scratch in A and V (2 m^2 T >= m doubles)
  int k1 = 0;
  if (variant != HS_LORASP)
    k1 = gc_basis_dev<T>(t.phi, t.a, t.np, m, variant == HS_GC_PROJ, t.eps1, t.U, (double *)A, red, s_gR, s_gW,
                         &s_gk);
  // ---- ||A_sw||_2^2 = lambda_max(G), of G scaled near 1 (as J below)
  const Pow2<T> f = gram_scale(t.G, m, red);
  for (int64_t e = tid; e < (int64_t)m * m; e += nt) A[e] = f(t.G[e]);
  __syncthreads();
  const int max_sweeps = 40;
  double thr;
  if (variant == HS_LORASP) {
    jacobi_eig<T>(A, V, m, true, sh, max_sweeps);
    double lmax = 0.0;
    for (int i = 0; i < m; ++i) lmax = fmax(lmax, (double)A[i * m + i]);
    thr = eps * eps * lmax;
    const int k = select_columns<T>(A, V, m, thr, t.U, 0, red);
    if (tid == 0) kout[t.k_idx] = min(k, t.cap);   // the columns come in descending order
    return;
  }
  if (eps == 0.0) {
    // no truncation: complete the GC basis to all of R^m (Householder QR of U_1;
    // scratch k1 m <= 2 m^2 T in A and V)
    // (nothing to complete when U_1 already spans R^m)
    if (k1 < m) {
      if (k1 <= 2)
        gc_complete<T>(t.U, m, k1, (double *)A, red);
      else
        gc_complete_n<T>(t.U, m, k1, (double *)A, s_gW, red);
    }
    if (tid == 0) kout[t.k_idx] = m;
    return;
  }
  double lmax = 0.0;
  jacobi_eig<T>(A, V, m, false, sh, max_sweeps);
  for (int i = 0; i < m; ++i) lmax = fmax(lmax, (double)A[i * m + i]);
  __syncthreads();
  // ---- matrix whose leading eigenvectors give U_2: (I - U1 U1^T) G (I - U1 U1^T)
  // X = G U1 (m x k1) in V's columns 0..k1-1 (scratch, ld m), all in T
  for (int w = tid; w < m * k1; w += nt) {
    const int i = w / k1, a = w % k1;
    T s = T(0);
    for (int j = 0; j < m; ++j) s = fma(t.G[(int64_t)i * m + j], t.U[(int64_t)j * m + a], s);
    V[i * m + a] = s;
  }
  __syncthreads();
  // c = U1^T G U1 (k1 x k1, ld kMaxK1)
  for (int a = 0; a < k1; ++a)
    for (int b = 0; b < k1; ++b) {
      double s = 0.0;
      for (int i = tid; i < m; i += nt) s += (double)(t.U[(int64_t)i * m + a] * V[i * m + b]);
      const T cab = (T)block_sum<T>(s, red);
      if (tid == 0) s_c[a * kMaxK1 + b] = cab;
    }
  __syncthreads();
  if (k1 <= 2) {
    // one or two basis vectors (one preserved vector): c in registers
    T c[2][2];
    for (int a = 0; a < 2; ++a)
      for (int b = 0; b < 2; ++b) c[a][b] = (a < k1 && b < k1) ? s_c[a * kMaxK1 + b] : T(0);
    for (int64_t e = tid; e < (int64_t)m * m; e += nt) {
      const int i = (int)(e / m), j = (int)(e % m);
      T v = t.G[e];
      for (int a = 0; a < k1; ++a) {
        const T ui = t.U[(int64_t)i * m + a], uj = t.U[(int64_t)j * m + a];
        v = fma(-ui, V[j * m + a], fma(-V[i * m + a], uj, v));
        for (int b = 0; b < k1; ++b) v = fma(ui * c[a][b], t.U[(int64_t)j * m + b], v);
      }
      A[e] = f(v);
    }
  } else {
    for (int64_t e = tid; e < (int64_t)m * m; e += nt) {
      const int i = (int)(e / m), j = (int)(e % m);
      T v = t.G[e];
      for (int a = 0; a < k1; ++a) {
        const T ui = t.U[(int64_t)i * m + a], uj = t.U[(int64_t)j * m + a];
        v = fma(-ui, V[j * m + a], fma(-V[i * m + a], uj, v));
        for (int b = 0; b < k1; ++b) v = fma(ui * s_c[a * kMaxK1 + b], t.U[(int64_t)j * m + b], v);
      }
      A[e] = f(v);
    }
  }
  thr = eps * eps * lmax;
  __syncthreads();
  jacobi_eig<T>(A, V, m, true, sh, max_sweeps);
  const int k2 = select_columns<T>(A, V, m, thr, t.U, k1, red);
  int k = k1 + min(k2, max(t.cap - k1, 0));
  if (k > m) k = m;
  if (tid == 0) kout[t.k_idx] = k;
}

// ---------------------------------------------------------------------------
// CSR value movement
// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_scatter_values(const double *__restrict__ val, const int64_t *__restrict__ dest,
                                 int64_t nnz, T *__restrict__ pool) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t d = dest[e];
    if (d >= 0) pool[d] = (T)val[e];
  }
}

__global__ void k_gather_values(const double *__restrict__ val, const int32_t *__restrict__ src,
                                int64_t nnz, double *__restrict__ out) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz;
       e += (int64_t)gridDim.x * blockDim.x)
    out[e] = val[src[e]];
}

template <typename T>
size_t trunc_small_arrays(int m) {
  const int mp = m + (m & 1);
  const int np = mp / 2 > 0 ? mp / 2 : 1;
  return 2 * sizeof(T) * np + 2 * sizeof(int) * np + 64;
}

}  // namespace

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
template <typename T>
int gemm_tile_class(const GemmTask<T> *tasks, int n) {
  double tiles = 0, work[2] = {0, 0};
  for (int q = 0; q < n; ++q)
    for (int c = 0; c < 2; ++c) {
      const int tm = gemm_tile<T>(c);
      const double w = gemm_tiles(tasks[q], tm);
      if (c == 0) tiles += w;
      work[c] += w * tm * tm * (tasks[q].K + 16.0);
    }
  if (sizeof(T) == 8) return tiles < 152 * 8 ? 1 : 0;
  return tiles < 152 * 2 || work[1] * 1.5 < work[0] ? 1 : 0;
}

template <typename T>
void launch_gemm(const GemmTask<T> *d_tasks, const int *d_tile_start, int ntasks, int total_tiles, int tile_class,
                 cudaStream_t st) {
  if (ntasks == 0 || total_tiles == 0) return;
  if constexpr (sizeof(T) == 4) {
    if (tile_class == 0)
      k_gemm<T, 64, 4, 16><<<total_tiles, 256, 0, st>>>(d_tasks, d_tile_start, ntasks);
    else
      k_gemm<T, 32, 2, 32><<<total_tiles, 256, 0, st>>>(d_tasks, d_tile_start, ntasks);
  } else {
    if (tile_class == 0)
      k_gemm<T, 32, 2, 16><<<total_tiles, 256, 0, st>>>(d_tasks, d_tile_start, ntasks);
    else
      k_gemm<T, 16, 1, 32><<<total_tiles, 256, 0, st>>>(d_tasks, d_tile_start, ntasks);
  }
  count_launch();
  HS_CUDA(cudaGetLastError());
}

template <typename T>
void launch_sum(const SumTask<T> *d_tasks, const SumSrc<T> *d_srcs, const int *d_tile_start,
                int ntasks, int total_tiles, cudaStream_t st) {
  if (ntasks == 0 || total_tiles == 0) return;
  k_sum<T><<<total_tiles, 256, 0, st>>>(d_tasks, d_srcs, d_tile_start, ntasks);
  count_launch();
  HS_CUDA(cudaGetLastError());
}

// first failing pivot over the diagonal blocks of a blocked Cholesky
static __global__ void k_status_merge(const StatusMerge *__restrict__ t, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int r = 0;
  for (int b = 0; b < t[i].nblk && !r; ++b)
    if (t[i].bs[b]) r = b * t[i].nb + t[i].bs[b];
  *t[i].out = r;
}

template <typename T>
int chol_smem_cap() {
  return sizeof(T) == 8 ? 256 : 224;
}

template <typename T, int NT>
static void launch_chol_nt(const CholTask<T> *d_tasks, int ntasks, int *d_status, int max_m, cudaStream_t st) {
  const size_t sm = chol_smem_bytes<T>(max_m);
  check_dynamic_smem(sm, allow_max_dynamic_smem<&k_chol_inv<T, NT>>(), "k_chol_inv");
  k_chol_inv<T, NT><<<ntasks, NT, sm, st>>>(d_tasks, d_status);
}

// FP64 above kCholClusterMin: k_chol_cluster (m = 150 to 160: twice as fast as
// one CTA, 0.31 ms; its limit of 256 also spares nodes up to there the blocked
// path).  Below, the diagonal blocks' serial chain is what counts.
// Threads by the largest matrix of the launch: the update's tiles (about
// m^2 / 1024 a step) keep that many warps busy; a matrix's arithmetic does not
// depend on them.
template <typename T>
void launch_chol_inv(const CholTask<T> *d_tasks, int ntasks, int *d_status, int max_m,
                     cudaStream_t st) {
  if (ntasks == 0) return;
  if (max_m <= 48) {
    launch_chol_nt<T, 128>(d_tasks, ntasks, d_status, max_m, st);
  } else if constexpr (sizeof(T) == 8) {
    if (max_m <= kCholClusterMin) {
      launch_chol_nt<T, 256>(d_tasks, ntasks, d_status, max_m, st);
    } else {
      const size_t sm = chol_cl_smem_bytes<T>(max_m);
      check_dynamic_smem(sm, allow_max_dynamic_smem<&k_chol_cluster<T>>(), "k_chol_cluster");
      k_chol_cluster<T><<<ntasks * kCholC, kCholClThreads, sm, st>>>(d_tasks, d_status);
    }
  } else if (max_m <= 112) {
    launch_chol_nt<T, 256>(d_tasks, ntasks, d_status, max_m, st);
  } else {
    launch_chol_nt<T, 512>(d_tasks, ntasks, d_status, max_m, st);
  }
  count_launch();
  HS_CUDA(cudaGetLastError());
}

template <typename T>
void launch_trunc(const TruncTask<T> *d_tasks, int ntasks, int *d_k, int variant, int max_m, cudaStream_t st) {
  if (ntasks == 0) return;
  const size_t sm = 2 * sizeof(T) * (size_t)max_m * max_m + trunc_small_arrays<T>(max_m);
  check_dynamic_smem(sm, allow_max_dynamic_smem<&k_trunc<T>>(), "k_trunc");
  k_trunc<T><<<ntasks, TRUNC_THREADS, sm, st>>>(d_tasks, d_k, variant);
  count_launch();
  HS_CUDA(cudaGetLastError());
}

template <typename T>
void launch_scatter_values(const double *val, const int64_t *dest, int64_t nnz, T *pool,
                           cudaStream_t st) {
  if (nnz == 0) return;
  const int grid = (int)std::min<int64_t>((nnz + 255) / 256, 152 * 16);
  k_scatter_values<T><<<grid, 256, 0, st>>>(val, dest, nnz, pool);
  count_launch();
  HS_CUDA(cudaGetLastError());
}

void launch_gather_values(const double *val, const int32_t *src, int64_t nnz, double *out,
                          cudaStream_t st) {
  if (nnz == 0) return;
  const int grid = (int)std::min<int64_t>((nnz + 255) / 256, 152 * 16);
  k_gather_values<<<grid, 256, 0, st>>>(val, src, nnz, out);
  count_launch();
  HS_CUDA(cudaGetLastError());
}

// D^-1/2 of each row (the reciprocal square root of its diagonal entry); a
// row whose diagonal entry is missing or not positive sets *flag
static __global__ void k_diag_scale(const int32_t *__restrict__ rp, const int32_t *__restrict__ ci,
                                    const double *__restrict__ va, int64_t n, double *__restrict__ ds,
                                    int *flag) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double d = 0.0;
    for (int e = rp[i]; e < rp[i + 1]; ++e)
      if (ci[e] == i) d += va[e];
    if (d > 0.0) {
      ds[i] = 1.0 / sqrt(d);
    } else {
      ds[i] = 1.0;
      atomicExch(flag, 1);
    }
  }
}

// out = D^-1/2 A D^-1/2 entry by entry
static __global__ void k_scale_values(const int32_t *__restrict__ rp, const int32_t *__restrict__ ci,
                                      const double *__restrict__ va, int64_t n, const double *__restrict__ ds,
                                      double *__restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double di = ds[i];
    for (int e = rp[i]; e < rp[i + 1]; ++e) out[e] = va[e] * di * ds[ci[e]];
  }
}

void launch_diag_scale(const int32_t *rp, const int32_t *ci, const double *val, int64_t n, double *ds,
                       double *val_scaled, int *flag, cudaStream_t st) {
  if (n == 0) return;
  const int grid = (int)std::min<int64_t>((n + 255) / 256, 152 * 16);
  k_diag_scale<<<grid, 256, 0, st>>>(rp, ci, val, n, ds, flag);
  k_scale_values<<<grid, 256, 0, st>>>(rp, ci, val, n, ds, val_scaled);
  count_launch(2);
  HS_CUDA(cudaGetLastError());
}

// preserved vectors of the scaled system: out = D^1/2 raw, n x np row-major
template <typename T>
static __global__ void k_phi_scale(const T *__restrict__ raw, const double *__restrict__ ds, int64_t n, int np,
                                   T *__restrict__ out) {
  const int64_t tot = n * np;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x)
    out[e] = (T)((double)raw[e] / ds[e / np]);
}

template <typename T>
void launch_phi_scale(const T *raw, const double *ds, int64_t n, int np, T *out, cudaStream_t st) {
  if (n == 0) return;
  const int grid = (int)std::min<int64_t>((n * np + 255) / 256, 152 * 16);
  k_phi_scale<T><<<grid, 256, 0, st>>>(raw, ds, n, np, out);
  count_launch();
  HS_CUDA(cudaGetLastError());
}

// one CTA per task, a grid-stride loop over its elements
static __global__ void k_convert_list(const ConvTask *__restrict__ t, int n) {
  const ConvTask c = t[blockIdx.x];
  if (c.widen) {
    const float *s = (const float *)c.src;
    double *d = (double *)c.dst;
    for (int64_t e = threadIdx.x; e < c.n; e += blockDim.x) d[e] = (double)s[e];
  } else {
    const double *s = (const double *)c.src;
    float *d = (float *)c.dst;
    for (int64_t e = threadIdx.x; e < c.n; e += blockDim.x) d[e] = (float)s[e];
  }
}

void launch_convert_list(const ConvTask *d_tasks, int ntasks, cudaStream_t st) {
  if (ntasks == 0) return;
  k_convert_list<<<ntasks, 256, 0, st>>>(d_tasks, ntasks);
  count_launch();
  HS_CUDA(cudaGetLastError());
}

void launch_status_merge(const StatusMerge *d_tasks, int ntasks, cudaStream_t st) {
  if (ntasks == 0) return;
  k_status_merge<<<(ntasks + 127) / 128, 128, 0, st>>>(d_tasks, ntasks);
  count_launch();
  HS_CUDA(cudaGetLastError());
}

#define HS_INST(T)                                                                            \
  template int gemm_tile_class<T>(const GemmTask<T> *, int);                                  \
  template void launch_gemm<T>(const GemmTask<T> *, const int *, int, int, int, cudaStream_t); \
  template void launch_sum<T>(const SumTask<T> *, const SumSrc<T> *, const int *, int, int,   \
                              cudaStream_t);                                                  \
  template void launch_chol_inv<T>(const CholTask<T> *, int, int *, int, cudaStream_t);       \
  template int chol_smem_cap<T>();                                                            \
  template void launch_trunc<T>(const TruncTask<T> *, int, int *, int, int, cudaStream_t);    \
  template void launch_phi_scale<T>(const T *, const double *, int64_t, int, T *, cudaStream_t); \
  template void launch_scatter_values<T>(const double *, const int64_t *, int64_t, T *,       \
                                         cudaStream_t);
HS_INST(double)
HS_INST(float)
#undef HS_INST

}  // namespace hs
