// Householder tridiagonalisation of a super node's Gram matrix J on chip
// (Sec. 3.2: the eigen-solve behind the rank decision sigma_i > eps ||A_sw|| and
// the basis U_2; Sec. 6 for the projected J of GC): in one CTA (tri_cta) or, for
// matrices beyond one CTA's shared memory, in one thread-block cluster.
//
// The whole n x n matrix stays in shared memory for all steps; with C CTAs each
// holds every C-th column (all rows).  J is symmetric, so every product is a
// column walk.  Step k:
//   1. column k (= row k), with the pending update of step k - 1, and the
//      reflector I - tau v v^T of x = J[k+1.., k];
//   2. one walk of the own columns: the pending update of step k - 1 and
//      p_i = tau sum_j J_ji v_j;
//   3. K = tau (p.v) / 2, w = p - K v; (v, w) are the next pending update
//      J -= v w^T + w v^T.
// What bounds it is the latency of a step: the walk's shared-memory loads and
// the barriers (three a step; in a cluster one cluster barrier and the reads of
// column k and p from the other CTAs besides).  Measured: about 1 us a step in
// one CTA, 3.4 us in 16 CTAs at n = 900 (8.0 us when every CTA read column k from
// the CTA that holds it).  The reflector's scalars are kept off the FP64 pipe in
// FP32 factors (reflector.h; the off-diagonal entries' FP64 roots are taken
// together at the end), and computed by one warp in FP64 ones:
// every thread computing them in FP64, at 1/64 of the FP32 rate, took more than
// half of each step.
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
#include "reflector.h"

namespace cg = cooperative_groups;

namespace hs {

namespace {

constexpr int kClThreads = 512;

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

// cluster kernel: neighbouring columns per warp and pass (FP64 is bound by its
// FMAs, which fewer columns spread better over the warps), and the row stride
// in words: the slots rounded up to twice an odd number
template <typename T>
constexpr int kClSlots = sizeof(T) == 4 ? 4 : 2;
__host__ __device__ inline int cl_ld(int R) { return R + (6 - R % 4) % 4; }

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
  return sizeof(T) * ((size_t)cl_ld(R) * m + 3 * (size_t)m + 2 * (size_t)R) + 64;
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
    // row k (columns >= k) with the pending update, and the norm of its tail beyond k + 1
    T a = T(0);
    if (i >= k && i < m) a = fma(-vk, wpi, fma(-wk, vpi, W[(size_t)k * ld + i]));
    if (half == 0) {
      if (i == k + 1) s_alpha = a;
      if (i == k) s_dk = a;
    }
    put_partial<T>(half == 0 && i > k + 1 ? a * a : T(0), red0);
    __syncthreads();
    T scale, tau, xn2;
    if constexpr (sizeof(T) == 4) {
      reflector(partial_total<T, NW>(red0), s_alpha, scale, tau, xn2);
    } else {
      if (warp == 0) {
        reflector(partial_total<T, NW>(red0), s_alpha, scale, tau, xn2);
        if (lane == 0) {
          s_r[0] = scale;
          s_r[1] = tau;
          s_r[2] = xn2;
        }
      }
      __syncthreads();
      scale = s_r[0];
      tau = s_r[1];
      xn2 = s_r[2];
    }
    const T vi = i == k + 1 ? T(1) : i > k + 1 ? a * scale : T(0);
    if (half == 0 && i < m) {
      pk[i] = Pack<T>{vpi, wpi, vi, T(0)};
      if (i >= k + 2) t.A[(int64_t)k * t.ld + i] = vi;   // reflector k in row k
    }
    if (tid == 0) {
      t.d[k] = (double)s_dk;
      t.e[k] = beta_code(tau, xn2, s_alpha);
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
  for (int k = tid; k + 2 < m; k += NT) t.e[k] = beta_of(t.e[k], t.tau[k] != T(0));
  if (half == 0 && i < m) pk[i] = Pack<T>{vpi, wpi, T(0), T(0)};
  __syncthreads();
  if (half == 0 && i < m && i >= m - 2)
    for (int j = max(m - 2, 0); j <= i; ++j)
      t.A[(int64_t)i * t.ld + j] = fma(-vpi, pk[j].wp, fma(-wpi, pk[j].vp, W[(size_t)i * ld + j]));
}

template <typename T>
struct alignas(2 * sizeof(T)) Pair {
  T x, y;
};

// Columns are dealt out cyclically (column i is slot i / C of CTA i % C), so
// every CTA keeps its share of the trailing matrix to the end.  A warp takes
// kClSlots neighbouring slots at a time and its lanes the rows: one pass
// applies the pending update and accumulates p = J v, whose sum over the rows
// stays in the warp.  The loads of the pending update's and v's rows then serve
// kClSlots columns, and the row stride (twice an odd number) spreads a warp's
// rows over the banks.
template <typename T, int C>
__global__ void __launch_bounds__(kClThreads) k_tri_cluster(const GridTri<T> *__restrict__ tasks) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int nt = kClThreads, NW = nt / 32, S = kClSlots<T>;
  __shared__ T red0[NW], red1[NW], s_x[2], s_r[4];
  cg::cluster_group cluster = cg::this_cluster();
  const int crank = (int)cluster.block_rank();
  const GridTri<T> t = tasks[blockIdx.x / C];
  const int m = t.m;
  const int R = (m + C - 1) / C, ld = cl_ld(R);
  const int ns = crank < m ? (m - 1 - crank) / C + 1 : 0;   // own columns
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  T *slab = reinterpret_cast<T *>(smem_raw);                // slot s of row j at slab[j ld + s]
  Pair<T> *pend = reinterpret_cast<Pair<T> *>(slab + (size_t)m * ld);   // (v, w) of the pending update
  T *v = reinterpret_cast<T *>(pend + m);                   // this step's reflector
  T *pseg = v + m;                                          // p on the own columns, two buffers (step parity)

  for (int q = warp; q < m; q += NW)
    for (int s = lane; s < ld; s += 32)
      slab[(size_t)q * ld + s] = s < ns ? t.A[(int64_t)q * t.ld + s * C + crank] : T(0);
  for (int j = tid; j < m; j += nt) pend[j] = Pair<T>{T(0), T(0)};
  cluster.sync();

  // One cluster barrier per step: p is double-buffered, so a CTA that runs ahead
  // never overwrites what a slower one still reads, and the row a step reads is
  // not written from that step on.
  T tau = T(0);
  for (int k = 0; k + 1 < m; ++k) {
    // rows j = k + tid (+ nt): the pending update of step k - 1, and column k
    // with it applied.  p and the column are read from all CTAs together, the
    // column as row k of J: one CTA holds the column itself, and all C reading
    // it there word by word took most of a step (8 us at n = 900, C = 16).
    T col[2], pj[2], vj[2];
    T pk = T(0);
    // block sum over the rows (a warp without any has nothing to add up)
    auto put_rows = [&](T x, T *red) {
      if (k + warp * 32 < m) put_partial<T>(x, red);
      else if (lane == 0) red[warp] = T(0);
    };
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int j = k + tid + u * nt;
      col[u] = j < m ? cluster.map_shared_rank(slab, j & (C - 1))[(size_t)k * ld + j / C] : T(0);
      pj[u] = vj[u] = T(0);
      if (k > 0 && j < m) {
        pj[u] = cluster.map_shared_rank(pseg, j & (C - 1))[((k - 1) & 1) * R + j / C];
        vj[u] = v[j];
      }
    }
    if (k > 0) {
      pk = cluster.map_shared_rank(pseg, k & (C - 1))[((k - 1) & 1) * R + k / C];
      put_rows(fma(pj[0], vj[0], pj[1] * vj[1]), red1);
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
      pk -= K;                                    // w of row k, where v is 1
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int j = k + tid + u * nt;
        if (j < m) {
          pj[u] = fma(-K, vj[u], pj[u]);          // w of row j
          pend[j] = Pair<T>{vj[u], pj[u]};
          col[u] = fma(-vj[u], pk, col[u] - pj[u]);
        }
      }
    }
    if (k + 2 >= m) {                             // the trailing 2 x 2 block, lower triangle
      __syncthreads();
      for (int j = max(m - 2, 0); j < m; ++j)
        if ((j & (C - 1)) == crank && j + tid < m) {
          const int i = j + tid;
          const Pair<T> f = pend[i], o = pend[j];
          t.A[(int64_t)i * t.ld + j] = fma(-f.x, o.y, fma(-f.y, o.x, slab[(size_t)i * ld + j / C]));
        }
      break;
    }
    if (tid < 2) s_x[tid] = col[0];               // entries k and k + 1
    put_rows(fma(col[1], col[1], tid > 1 ? col[0] * col[0] : T(0)), red0);
    __syncthreads();
    T scale, xn2;
    if constexpr (sizeof(T) == 4) {
      reflector(partial_total<T, NW>(red0), s_x[1], scale, tau, xn2);
    } else {
      if (warp == 0) {
        reflector(partial_total<T, NW>(red0), s_x[1], scale, tau, xn2);
        if (lane == 0) {
          s_r[0] = scale;
          s_r[1] = tau;
          s_r[2] = xn2;
        }
      }
      __syncthreads();
      scale = s_r[0];
      tau = s_r[1];
      xn2 = s_r[2];
    }
    const bool owner = (k & (C - 1)) == crank;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int j = k + tid + u * nt;
      if (j > k && j < m) {
        const T x = j == k + 1 ? T(1) : col[u] * scale;
        v[j] = x;
        if (owner && j >= k + 2) t.A[(int64_t)k * t.ld + j] = x;   // reflector k in row k
      }
    }
    if (owner && tid == 0) {
      t.d[k] = (double)col[0];
      t.e[k] = beta_code(tau, xn2, s_x[1]);
      t.tau[k] = tau;
    }
    __syncthreads();
    // the own columns i > k: pending update of rows j > k, then p_i = tau sum_j J_ji v_j
    T *pcur = pseg + (k & 1) * R;
    const int live = k >= crank ? (k - crank) / C + 1 : 0;         // first slot with i > k
    for (int g = live / S + warp; g * S < ns; g += NW) {
      const int s0 = g * S;
      Pair<T> own[S];
      bool on[S];
      T acc[S];
#pragma unroll
      for (int u = 0; u < S; ++u) {
        on[u] = s0 + u >= live && s0 + u < ns;
        own[u] = on[u] ? pend[(s0 + u) * C + crank] : Pair<T>{T(0), T(0)};
        acc[u] = T(0);
      }
#pragma unroll 4
      for (int j = k + 1 + lane; j < m; j += 32) {
        const Pair<T> f = pend[j];
        const T vv = v[j];
        Pair<T> *row = reinterpret_cast<Pair<T> *>(slab + (size_t)j * ld + s0);
#pragma unroll
        for (int u = 0; u < S; u += 2) {
          if (!on[u] && !on[u + 1]) continue;
          Pair<T> y = row[u / 2];
          y.x = fma(-f.x, own[u].y, fma(-f.y, own[u].x, y.x));
          y.y = fma(-f.x, own[u + 1].y, fma(-f.y, own[u + 1].x, y.y));
          row[u / 2] = y;
          acc[u] = fma(y.x, vv, acc[u]);
          acc[u + 1] = fma(y.y, vv, acc[u + 1]);
        }
      }
      // sums over the lanes, half of the columns handed over at each step
      int mine = 0;
#pragma unroll
      for (int w = S / 2, o = 16; w > 0; w /= 2, o /= 2) {
        const bool up = lane & o;
#pragma unroll
        for (int u = 0; u < w; ++u) {
          const T keep = up ? acc[u + w] : acc[u], give = up ? acc[u] : acc[u + w];
          acc[u] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
        if (up) mine += w;
      }
#pragma unroll
      for (int o = 16 / S; o > 0; o >>= 1) acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
      if ((lane & (32 / S - 1)) == 0 && s0 + mine >= live && s0 + mine < ns) pcur[s0 + mine] = tau * acc[0];
    }
    cluster.sync();   // every CTA's p is visible; every walk of step k is done
  }
  // (the barrier also makes thread 0's words visible)
  __syncthreads();
  for (int k = crank + C * tid; k + 2 < m; k += C * nt) t.e[k] = beta_of(t.e[k], t.tau[k] != T(0));
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

// Largest m that one CTA (class 0) or a cluster of 2, 4, 8 or 16 CTAs (classes 1 ..
// 4) takes, 0 if such a cluster cannot be resident; once per device.
template <typename T>
const int (&tri_max_m())[kTriClasses] {
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
      // (one CTA: 16 columns per warp; a cluster: two rows per thread)
      while (cl_smem_bytes<T>(mm + 1, C) <= room[c] && mm + 1 <= (c == 0 ? 256 : 2 * kClThreads)) ++mm;
      table[dev][c] = mm;
    }
    ready[dev] = true;
  }
  return table[dev];
}

}  // namespace

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
  return tri_pick(tri_max_m<T>(), m, sizeof(T) == 8, tri_mode());
}

template <typename T>
int tri_onchip_max() {
  return tri_pick_max(tri_max_m<T>(), tri_mode());
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
