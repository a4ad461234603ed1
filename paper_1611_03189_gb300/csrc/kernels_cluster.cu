// Householder tridiagonalisation of a super node's Gram matrix J on chip
// (Sec. 3.2: the eigen-solve behind the rank decision sigma_i > eps ||A_sw|| and
// the basis U_2; Sec. 6 for the projected J of GC): in one CTA (tri_cta) or, for
// matrices beyond one CTA's shared memory, in one thread-block cluster.
//
// The whole n x n matrix stays in shared memory for all steps; with C CTAs each
// holds a slab of ceil(n / C) columns (all rows).  J is symmetric, so every
// product is a column walk: a few threads own a column, consecutive threads on
// consecutive words.  Step k:
//   1. column k (= row k), with the pending update of step k - 1, and the
//      reflector I - tau v v^T of x = J[k+1.., k];
//   2. one walk of the own columns: the pending update of step k - 1 and
//      p_i = tau sum_j J_ji v_j;
//   3. K = tau (p.v) / 2, w = p - K v; (v, w) are the next pending update
//      J -= v w^T + w v^T.
// What bounds it is the latency of a step: shared-memory loads of the walk and
// the barriers (three a step in one CTA; in a cluster one cluster barrier and the
// distributed reads of column k and p besides).  The reflector's scalars are
// kept off the FP64 pipe in FP32 factors (see reflector() below), and by one
// warp in FP64 ones: every thread computing them in FP64, at 1/64 of the FP32
// rate, took more than half of each step.
// Outputs: d, e (FP64) and tau, reflector k in row k of A (v[0] = 1 implicit,
// v[1..] at A[k][k+2..]), the trailing 2 x 2 block in A.  Where a node is worked
// on and every reduction order depend on n alone, so a node gets the same bits
// in any batch.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cstdlib>
#include <mutex>

#include "hs_internal.h"

namespace cg = cooperative_groups;

namespace hs {

namespace {

constexpr int kClThreads = 512;

// The reflector of x with |x|^2 = xn2 and first entry alpha: beta = -sign(alpha)
// |x| = (beta, lo), tau = (beta - alpha) / beta, v = x * scale beyond the first
// entry, scale = 1 / (alpha - beta); tau = 0 when x has no tail.
// FP32: the square root and both quotients are corrected by their residuals
// (exact through fused multiply-adds, |beta| kept as s + lo), which gives tau and
// scale as if computed in higher precision and rounded, with no FP64 at all.
__device__ __forceinline__ void reflector(float xn2, float alpha, float &scale, float &tau, float &beta, float &lo) {
  if (!(fmaf(-alpha, alpha, xn2) > 0.f)) {
    scale = tau = lo = 0.f;
    beta = alpha;
    return;
  }
  const float a = fabsf(alpha);
  const float s = sqrtf(xn2), inv = 1.f / s;
  const float sl = 0.5f * fmaf(-s, s, xn2) * inv;
  const float sum = a + s, suml = (a - (sum - s)) + sl;   // a <= s
  const float r = 1.f / sum;
  const float sc = fmaf(r, fmaf(-sum, r, 1.f) - r * suml, r);
  const float q = a * inv;
  tau = 1.f + fmaf(inv, fmaf(-q, s, a) - q * sl, q);
  scale = copysignf(sc, alpha);
  beta = -copysignf(s, alpha);
  lo = alpha < 0.f || (alpha == 0.f && signbit(alpha)) ? sl : -sl;
}
__device__ __forceinline__ void reflector(double xn2, double alpha, double &scale, double &tau, double &beta,
                                          double &lo) {
  lo = 0.0;
  if (!(fma(-alpha, alpha, xn2) > 0.0)) {
    scale = tau = 0.0;
    beta = alpha;
    return;
  }
  const double a = fabs(alpha), s = sqrt(xn2);
  scale = copysign(1.0 / (a + s), alpha);
  tau = 1.0 + a / s;
  beta = -copysign(s, alpha);
}

// warp partials of a block sum into red[warp]; complete after a barrier
template <typename T>
__device__ __forceinline__ void put_partial(T v, T *red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
}
// their total, by a fixed tree over NW (a power of two) partials
template <typename T, int NW>
__device__ __forceinline__ T partial_total(const T *red) {
  T r[NW];
#pragma unroll
  for (int q = 0; q < NW; ++q) r[q] = red[q];
#pragma unroll
  for (int h = NW / 2; h > 0; h /= 2)
#pragma unroll
    for (int q = 0; q < h; ++q) r[q] += r[q + h];
  return r[0];
}

// threads per owned column in the cluster kernel (1 .. 8)
__host__ __device__ inline int cl_tpc(int R, int nt) {
  const int q = R > 0 ? nt / R : 1;
  return q < 1 ? 1 : q > 8 ? 8 : q;
}

// One-CTA kernel: 16 columns per warp, two threads (lanes l and l + 16) per
// column on alternate rows, so a row stride of 16 (mod 32) words keeps the two
// rows' columns in different banks (FP64: any stride does)
template <typename T>
__host__ __device__ inline int cta_ld(int m) {
  return sizeof(T) == 4 ? ((m + 15) / 32) * 32 + 16 : m | 1;
}
__host__ __device__ inline int cta_threads(int m) { return m <= 64 ? 128 : m <= 128 ? 256 : 512; }

template <typename T>
__host__ __device__ inline size_t cl_smem_bytes(int m, int C) {
  if (C == 1) return sizeof(T) * ((size_t)m * cta_ld<T>(m) + 4 * (size_t)m + 48) + 64;
  const int R = (m + C - 1) / C;
  return sizeof(T) * ((size_t)R * m + 4 * (size_t)m + (size_t)R * (2 + cl_tpc(R, kClThreads)) + 48) + 64;
}

// (v, w) of the pending update and v of the current step, per row
template <typename T>
struct Pack {
  T vp, wp, v, pad;
};

template <typename T, int NT>
__global__ void __launch_bounds__(NT) k_tri_cta(const GridTri<T> *__restrict__ tasks) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int NW = NT / 32;
  __shared__ T red0[NW], red1[NW];
  __shared__ T s_alpha, s_dk, s_p, s_r[4];
  const GridTri<T> t = tasks[blockIdx.x];
  const int m = t.m, ld = cta_ld<T>(m);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int i = 16 * warp + (lane & 15), half = lane >> 4;   // own column, rows k + 1 + half (mod 2)
  T *W = reinterpret_cast<T *>(smem_raw);   // m x ld
  // m * ld * sizeof(T) is a multiple of 16: ld of 16 words (FP32); FP64 rounds up
  Pack<T> *pk = reinterpret_cast<Pack<T> *>(smem_raw + ((sizeof(T) * (size_t)m * ld + 15) & ~(size_t)15));
  for (int r = warp; r < m; r += NW)
    for (int c = lane; c < m; c += 32) W[(size_t)r * ld + c] = t.A[(int64_t)r * t.ld + c];
  T vpi = T(0), wpi = T(0), vk = T(0), wk = T(0);   // pending update: own column, and row k
  __syncthreads();
  for (int k = 0; k + 2 < m; ++k) {
    // row k (columns >= k) with the pending update, and the norm of its tail
    T a = T(0);
    if (i >= k && i < m) a = fma(-vk, wpi, fma(-wk, vpi, W[(size_t)k * ld + i]));
    if (half == 0) {
      if (i == k + 1) s_alpha = a;
      if (i == k) s_dk = a;
    }
    put_partial<T>(half == 0 && i > k ? a * a : T(0), red0);
    __syncthreads();
    T scale, tau, beta, lo;
    if constexpr (sizeof(T) == 4) {
      reflector(partial_total<T, NW>(red0), s_alpha, scale, tau, beta, lo);
    } else {
      if (warp == 0) {
        reflector(partial_total<T, NW>(red0), s_alpha, scale, tau, beta, lo);
        if (lane == 0) {
          s_r[0] = scale;
          s_r[1] = tau;
          s_r[2] = beta;
        }
      }
      __syncthreads();
      scale = s_r[0];
      tau = s_r[1];
      beta = s_r[2];
      lo = T(0);
    }
    const T vi = i == k + 1 ? T(1) : i > k + 1 ? a * scale : T(0);
    if (half == 0 && i < m) {
      pk[i] = Pack<T>{vpi, wpi, vi, T(0)};
      if (i >= k + 2) t.A[(int64_t)k * t.ld + i] = vi;   // reflector k in row k
    }
    if (tid == 0) {
      t.d[k] = (double)s_dk;
      t.e[k] = (double)beta + (double)lo;
      t.tau[k] = tau;
    }
    __syncthreads();
    // one walk of each trailing column i > k (tau = 0 gives p = w = 0)
    T p = T(0);
    if (i > k && i < m) {
      T *col = W + i;
      T s[4] = {T(0), T(0), T(0), T(0)};
      int j = k + 1 + half;
      for (; j + 6 < m; j += 8) {
        T x[4];
        Pack<T> f[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          f[u] = pk[j + 2 * u];
          x[u] = col[(size_t)(j + 2 * u) * ld];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          x[u] = fma(-f[u].vp, wpi, fma(-f[u].wp, vpi, x[u]));
          col[(size_t)(j + 2 * u) * ld] = x[u];
          s[u] = fma(x[u], f[u].v, s[u]);
        }
      }
      for (; j < m; j += 2) {
        const Pack<T> f = pk[j];
        const T x = fma(-f.vp, wpi, fma(-f.wp, vpi, col[(size_t)j * ld]));
        col[(size_t)j * ld] = x;
        s[0] = fma(x, f.v, s[0]);
      }
      p = (s[0] + s[1]) + (s[2] + s[3]);
    }
    p += __shfl_xor_sync(0xffffffffu, p, 16);
    p *= tau;
    if (half == 0 && i == k + 1) s_p = p;
    put_partial<T>(half == 0 ? p * vi : T(0), red1);
    __syncthreads();
    T K;
    if constexpr (sizeof(T) == 4) {
      K = T(0.5) * tau * partial_total<T, NW>(red1);
    } else {
      if (warp == 0) {
        const T tot = partial_total<T, NW>(red1);
        if (lane == 0) s_r[3] = T(0.5) * tau * tot;
      }
      __syncthreads();
      K = s_r[3];
    }
    vpi = vi;
    wpi = fma(-K, vi, p);
    vk = T(1);            // v of row k + 1
    wk = fma(-K, T(1), s_p);
  }
  // the last pending update on the trailing 2 x 2 block, which is written out
  __syncthreads();
  if (half == 0 && i < m) pk[i] = Pack<T>{vpi, wpi, T(0), T(0)};
  __syncthreads();
  if (half == 0 && i < m && i >= m - 2)
    for (int j = max(m - 2, 0); j <= i; ++j)
      t.A[(int64_t)i * t.ld + j] = fma(-vpi, pk[j].wp, fma(-wpi, pk[j].vp, W[(size_t)i * ld + j]));
}

template <typename T, int C>
__global__ void __launch_bounds__(kClThreads) k_tri_cluster(const GridTri<T> *__restrict__ tasks) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int nt = kClThreads, NW = nt / 32;
  cg::cluster_group cluster = cg::this_cluster();
  const int crank = (int)cluster.block_rank();
  const GridTri<T> t = tasks[blockIdx.x / C];
  const int m = t.m;
  const int R = (m + C - 1) / C;
  const int c0 = crank * R, c1 = min(m, c0 + R);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tpc = cl_tpc(R, nt);               // threads per column
  const int ci = tid % R, part = tid / R;      // own column c0 + ci, rows j = part (mod tpc)
  struct P2 {
    T vp, wp;
  };
  P2 *pend = reinterpret_cast<P2 *>(smem_raw); // pending update of the previous step
  T *x = reinterpret_cast<T *>(pend + m);      // column k of J, rows k..
  T *v = x + m;                                // this step's reflector
  T *pseg = v + m;                             // p on the own columns, two buffers (step parity)
  T *psum = pseg + 2 * (size_t)R;              // tpc partial sums per own column
  T *red0 = psum + (size_t)R * tpc;            // two reduction buffers
  T *red1 = red0 + NW;
  T *pvpart = red1 + NW;                       // this CTA's share of p.v, two buffers
  T *s_r = pvpart + 2;                         // FP64: the reflector's scalars
  T *slab = s_r + 4;                           // columns c0 .. c1-1 of J, all rows: slab[j R + (i - c0)]

  for (int j = warp; j < m; j += NW)
    for (int q = lane; q < R; q += 32) slab[(size_t)j * R + q] = c0 + q < c1 ? t.A[(int64_t)j * t.ld + c0 + q] : T(0);
  for (int j = tid; j < m; j += nt) pend[j] = P2{T(0), T(0)};
  cluster.sync();

  // One cluster barrier per step: p and the share of p.v are double-buffered, so
  // a CTA that runs ahead never overwrites what a slower one still reads, and the
  // column a step reads is not written in that step.
  for (int k = 0; k + 2 < m; ++k) {
    const int owner = k / R;
    const T *ocol = cluster.map_shared_rank(slab, owner) + (k - owner * R);
    const P2 pk = pend[k];
    T s2t = T(0);
    for (int j = k + tid; j < m; j += nt) {
      const P2 pj = pend[j];
      const T a = fma(-pj.vp, pk.wp, fma(-pj.wp, pk.vp, ocol[(size_t)j * R]));
      x[j] = a;
      if (j > k) s2t = fma(a, a, s2t);
    }
    put_partial<T>(s2t, red0);
    __syncthreads();
    T scale, tau, beta, lo;
    if constexpr (sizeof(T) == 4) {
      reflector(partial_total<T, NW>(red0), x[k + 1], scale, tau, beta, lo);
    } else {
      if (warp == 0) {
        reflector(partial_total<T, NW>(red0), x[k + 1], scale, tau, beta, lo);
        if (lane == 0) {
          s_r[0] = scale;
          s_r[1] = tau;
          s_r[2] = beta;
        }
      }
      __syncthreads();
      scale = s_r[0];
      tau = s_r[1];
      beta = s_r[2];
      lo = T(0);
    }
    for (int j = k + 1 + tid; j < m; j += nt) {
      const T vj = (j == k + 1) ? T(1) : x[j] * scale;
      v[j] = vj;
      if (crank == owner && j >= k + 2) t.A[(int64_t)k * t.ld + j] = vj;   // reflector k in row k
    }
    if (crank == owner && tid == 0) {
      t.d[k] = (double)x[k];
      t.e[k] = (double)beta + (double)lo;
      t.tau[k] = tau;
    }
    __syncthreads();
    // the own columns i > k: pending update of rows j > k, then
    // p_i = tau sum_j J_ji v_j (rows split over tpc threads per column)
    T *pcur = pseg + (k & 1) * R;
    const int i = c0 + ci;
    if (part < tpc && i < c1 && i > k) {
      const P2 own = pend[i];
      T s[4] = {T(0), T(0), T(0), T(0)};
      int j = k + 1 + part;
      for (; j + 3 * tpc < m; j += 4 * tpc) {
        T y[4];
        P2 f[4];
        T vj[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          f[u] = pend[j + u * tpc];
          vj[u] = v[j + u * tpc];
          y[u] = slab[(size_t)(j + u * tpc) * R + ci];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          y[u] = fma(-f[u].vp, own.wp, fma(-f[u].wp, own.vp, y[u]));
          slab[(size_t)(j + u * tpc) * R + ci] = y[u];
          s[u] = fma(y[u], vj[u], s[u]);
        }
      }
      for (; j < m; j += tpc) {
        const P2 f = pend[j];
        const T y = fma(-f.vp, own.wp, fma(-f.wp, own.vp, slab[(size_t)j * R + ci]));
        slab[(size_t)j * R + ci] = y;
        s[0] = fma(y, v[j], s[0]);
      }
      psum[part * R + ci] = (s[0] + s[1]) + (s[2] + s[3]);
    }
    __syncthreads();
    T pvt = T(0);
    if (part == 0 && i < c1 && i > k) {
      T acc = T(0);
      for (int q = 0; q < tpc; ++q) acc += psum[q * R + ci];
      const T p = tau * acc;
      pcur[ci] = p;
      pvt = p * v[i];
    }
    put_partial<T>(pvt, red1);
    __syncthreads();
    if (warp == 0) {
      const T tot = partial_total<T, NW>(red1);
      if (lane == 0) pvpart[k & 1] = tot;
    }
    cluster.sync();   // every CTA's p and share of p.v are visible; every walk of step k is done
    T pv = T(0);
    if (sizeof(T) == 4 || warp == 0)
      for (int c = 0; c < C; ++c) pv += cluster.map_shared_rank(pvpart, c)[k & 1];
    T K = T(0.5) * tau * pv;
    if constexpr (sizeof(T) == 8) {
      if (tid == 0) s_r[3] = K;
      __syncthreads();
      K = s_r[3];
    }
    for (int j = k + 1 + tid; j < m; j += nt) {
      const int oj = j / R;
      const T pj = cluster.map_shared_rank(pseg, oj)[(k & 1) * R + j - oj * R];
      pend[j] = P2{v[j], fma(-K, v[j], pj)};   // the next pending update
    }
    __syncthreads();
  }
  // the last pending update on the trailing 2 x 2 block, lower triangle,
  // written out by the owners of its columns
  for (int j = max(c0, m - 2) + tid; j < c1; j += nt)
    for (int i = j; i < m; ++i)
      t.A[(int64_t)i * t.ld + j] =
          fma(-pend[i].vp, pend[j].wp, fma(-pend[i].wp, pend[j].vp, slab[(size_t)i * R + (j - c0)]));
  // no CTA may leave while others still read its shared memory
  cluster.sync();
}

template <typename T, int C>
void cluster_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *attr, int clusters, size_t sm, cudaStream_t st) {
  cfg = {};
  cfg.gridDim = dim3((unsigned)(clusters * C), 1, 1);
  cfg.blockDim = dim3(kClThreads, 1, 1);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
}

template <typename T, int C>
void launch_cluster_c(const GridTri<T> *d_tasks, int ntasks, int m_max, cudaStream_t st) {
  const size_t sm = cl_smem_bytes<T>(m_max, C);
  check_dynamic_smem(sm, allow_max_dynamic_smem<&k_tri_cluster<T, C>>(), "k_tri_cluster");
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  cluster_config<T, C>(cfg, attr, ntasks, sm, st);
  HS_CUDA(cudaLaunchKernelEx(&cfg, k_tri_cluster<T, C>, d_tasks));
  count_launch();
}

template <typename T, int NT>
void launch_cta_nt(const GridTri<T> *d_tasks, int ntasks, int m_max, cudaStream_t st) {
  const size_t sm = cl_smem_bytes<T>(m_max, 1);
  check_dynamic_smem(sm, allow_max_dynamic_smem<&k_tri_cta<T, NT>>(), "k_tri_cta");
  k_tri_cta<T, NT><<<ntasks, NT, sm, st>>>(d_tasks);
  count_launch();
}

// usable dynamic shared memory of a CTA if a cluster of C such CTAs can be
// resident at all, else 0 (16 CTAs need the non-portable size allowed)
template <typename T, int C>
size_t cluster_room() {
  if (C > 8 && cudaFuncSetAttribute(k_tri_cluster<T, C>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
                   cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  const size_t sm = (size_t)allow_max_dynamic_smem<&k_tri_cluster<T, C>>();
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  cluster_config<T, C>(cfg, attr, 1, sm, nullptr);
  int n = 0;
  const cudaError_t e = cudaOccupancyMaxActiveClusters(&n, k_tri_cluster<T, C>, &cfg);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n > 0 ? sm : 0;
}

// Largest m that one CTA (q = 0) or a cluster of 2, 4, 8 or 16 CTAs (q = 1 ..
// 4) takes, 0 if such a cluster cannot be resident; once per device.
template <typename T>
int tri_max_m(int q) {
  static std::mutex mu;
  static int table[64][kTriClasses];
  static bool ready[64] = {false};
  int dev = 0;
  HS_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) fail(HS_ERR_CUDA, "device ordinal out of range");
  std::lock_guard<std::mutex> lk(mu);
  if (!ready[dev]) {
    const size_t room[kTriClasses] = {(size_t)allow_max_dynamic_smem<&k_tri_cta<T, 512>>(), cluster_room<T, 2>(),
                                      cluster_room<T, 4>(), cluster_room<T, 8>(), cluster_room<T, 16>()};
    for (int c = 0; c < kTriClasses; ++c) {
      const int C = 1 << c;
      int mm = 0;
      // (one CTA: 16 columns per warp; a cluster: at most one owned column per thread)
      while (cl_smem_bytes<T>(mm + 1, C) <= room[c] && (c == 0 ? mm + 1 <= 256 : (mm + C) / C <= kClThreads)) ++mm;
      table[dev][c] = mm;
    }
    ready[dev] = true;
  }
  return table[dev][q];
}

}  // namespace

// FP32: one CTA while it fits, then 4 CTAs (a step is bound by its barriers and
// distributed reads, which cost 2 CTAs as much), then 8, then 16.
// FP64: the arithmetic itself (3 n^2 FMAs a step at 1/64 of the FP32 rate)
// outgrows the barriers from about n = 112 on, so 8 CTAs share it from there.
// HS_TRI_CLUSTER=1 (environment) keeps to one CTA, =2 takes the smallest
// cluster that fits.
static int tri_mode() {
  static const int mode = [] {
    const char *e = std::getenv("HS_TRI_CLUSTER");
    return e && (e[0] == '1' || e[0] == '2') ? e[0] - '0' : 0;
  }();
  return mode;
}
template <typename T>
int tri_class(int m) {
  const int mode = tri_mode();
  if (mode == 1) return m <= tri_max_m<T>(0) ? 0 : -1;
  int first = 0;
  if (mode == 0) {
    if (sizeof(T) == 8 && m > 112)
      first = 3;
    else if (m > tri_max_m<T>(0))
      first = 2;
  }
  for (int q = first; q < kTriClasses; ++q)
    if (m <= tri_max_m<T>(q)) return q;
  return -1;
}

template <typename T>
int tri_onchip_max() {
  int mm = 0;
  for (int q = 0; q < (tri_mode() == 1 ? 1 : kTriClasses); ++q) mm = std::max(mm, tri_max_m<T>(q));
  return mm;
}

template <typename T>
void launch_tri_onchip(const GridTri<T> *d_tasks, int ntasks, int q, int m_max, cudaStream_t st) {
  if (ntasks == 0) return;
  switch (q) {
    case 0: {
      const int nt = cta_threads(m_max);
      if (nt == 128) launch_cta_nt<T, 128>(d_tasks, ntasks, m_max, st);
      else if (nt == 256) launch_cta_nt<T, 256>(d_tasks, ntasks, m_max, st);
      else launch_cta_nt<T, 512>(d_tasks, ntasks, m_max, st);
      break;
    }
    case 1: launch_cluster_c<T, 2>(d_tasks, ntasks, m_max, st); break;
    case 2: launch_cluster_c<T, 4>(d_tasks, ntasks, m_max, st); break;
    case 3: launch_cluster_c<T, 8>(d_tasks, ntasks, m_max, st); break;
    case 4: launch_cluster_c<T, 16>(d_tasks, ntasks, m_max, st); break;
    default: fail(HS_ERR_INVALID, "internal: class of the tridiagonalisation");
  }
  HS_CUDA(cudaGetLastError());
}

template int tri_class<double>(int);
template int tri_class<float>(int);
template int tri_onchip_max<double>();
template int tri_onchip_max<float>();
template void launch_tri_onchip<double>(const GridTri<double> *, int, int, int, cudaStream_t);
template void launch_tri_onchip<float>(const GridTri<float> *, int, int, int, cudaStream_t);

}  // namespace hs
