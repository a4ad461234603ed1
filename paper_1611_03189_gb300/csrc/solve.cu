// Solve phase: the apply z = A_H^-1 r (Appendix A, Algorithm 2) and FP64
// preconditioned conjugate gradients around it.
//
// Workspace layout: one vector per level, level L first (the unknowns in
// cluster order), then the red nodes made at level L, ..., then the root; each
// unknown holds nrhs consecutive doubles.  A super node's unknowns at a level
// are the concatenation of its two children's, so super node and red nodes of
// a level share the same memory.
//
// With B_s = M_ss A_sN (made by the factorization), Algorithm 2's steps of a
// wave become one launch each way (in elimination order, then in reverse):
//   k_fwd:  t_s = M_ss phi_s, phi_r = P_ss phi_s           (restriction)
//           phi_n -= sum_s B_s[:, n]^T phi_s               (forward substitution:
//                                                           A_ns M_ss = B_s[:, n]^T)
//   k_bwd:  x_s = t_s + P_ss^T x_r - B_s x_N               (backward substitution
//                                                           and prolongation:
//                                                           M_ss (phi_s - A_sN x_N))
// and the root solve (k_copy, k_root) between them.  The form with A_sN needs
// two dependent launches each way and reads M_ss twice.  What bounds an
// application is the chain of dependent launches at the top levels and the
// latency of the loads inside each, so both are kept short: at 512 x 512 (59
// waves, FP32, one right-hand side) 120 launches and 0.60 ms an application
// against 181 and 1.5 ms with the form above, one warp per row; at 300 x 217
// (FP64, five right-hand sides) 1.59 ms against 4.43; at 40^3 (FP32, sixteen)
// a four-iteration solve takes 15.6 ms against 34.0.
// t_s goes to the wave's scratch (every row of the wave reads phi_s), and the
// next wave's launch moves it into the place of phi_s, which nothing reads any
// more; the scratch is two buffers used in turn.
// A launch is a list of items, one CTA each (apply_prepare): 32 rows of
// [M_ss; P_ss], 32 unknowns of a target n or of x_s, or up to 8 nodes' t_s to
// move.  Rows are walked by warps, four rows sharing each load of x; columns
// (P_ss^T, B_s^T) by the CTA's 8 warps together, 32 adjacent columns each.
// What an item does and the order of every sum depend on the node alone, so
// results depend neither on scheduling nor on the number of right-hand sides.
#include <algorithm>
#include <cmath>
#include <vector>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <string>
#include <type_traits>

#include "handle.h"

namespace hs {

namespace {

constexpr int AW = 8;         // warps per CTA in the apply kernels
constexpr int AT = AW * 32;
constexpr int AR = kApplyRows / AW;   // rows of an item per warp

// NR consecutive values of one unknown; VEC: 16-byte loads (every column of
// the chunk in use, unknown stride and first column multiples of 16 bytes)
template <typename T, int NR, bool VEC>
__device__ __forceinline__ void load_x(const T *x, int nr, T (&v)[NR]) {
  if constexpr (VEC) {
    constexpr int W = 16 / (int)sizeof(T);
#pragma unroll
    for (int i = 0; i < NR / W; ++i) {
      if constexpr (sizeof(T) == 4) {
        const float4 q = reinterpret_cast<const float4 *>(x)[i];
        v[4 * i] = q.x;
        v[4 * i + 1] = q.y;
        v[4 * i + 2] = q.z;
        v[4 * i + 3] = q.w;
      } else {
        const double2 q = reinterpret_cast<const double2 *>(x)[i];
        v[2 * i] = q.x;
        v[2 * i + 1] = q.y;
      }
    }
  } else {
#pragma unroll
    for (int j = 0; j < NR; ++j) v[j] = j < nr ? x[j] : T(0);
  }
}

// Programmatic dependent launch.  Each wave's launch may start while the one
// before it still runs: it reads its item and its first record entries, asks for
// the rest of them to come to L2 (none of which any launch of the solve writes),
// and only then waits for the launch before.  That takes the two longest loads
// of a step, descriptor and records from HBM, off the chain of dependent
// launches: 692 -> 591 us an iteration at 512 x 512 (FP32, one right-hand side),
// the 64 x 64 FP64 solve 829 -> 725 us, GMRES at 256 x 256 5.00 -> 4.62 ms.  FP64
// passes of 8 or more right-hand sides keep to plain launches (300 x 217, five:
// 1.59 ms against 1.66: they are bound by the FP64 rate, and CTAs that wait take
// slots).  DEP is false there and inside the persistent kernel.
template <typename T, int NR>
__host__ __device__ constexpr bool early_start() {
  return sizeof(T) == 4 || NR < 8;
}
__device__ __forceinline__ void dep_launch() { asm volatile("griddepcontrol.launch_dependents;"); }
template <bool DEP>
__device__ __forceinline__ void dep_wait() {
  if constexpr (DEP) asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// av[u][r] = a[r][c0 + 32 u + lane] (0 from len on)
template <typename T, int R>
__device__ __forceinline__ void load_chunk(const T *const (&a)[R], int c0, int len, int lane, T (&av)[4][R]) {
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int c = c0 + 32 * u + lane;
#pragma unroll
    for (int r = 0; r < R; ++r) av[u][r] = c < len ? __ldg(a[r] + c) : T(0);
  }
}

// acc[r][j] += sum_c a[r][c] x[c*stride + j] for c = lane, lane + 32, ... < len:
// R rows share every load of x, and 4 R row elements per lane are in flight;
// av holds the first chunk
template <typename T, int NR, int R, bool VEC>
__device__ __forceinline__ void rows_dot(const T *const (&a)[R], const T *x, int len, int64_t stride, int nr,
                                         int lane, T (&av)[4][R], T (&acc)[R][NR]) {
  for (int c0 = 0; c0 < len; c0 += 128) {
    if (c0 > 0) load_chunk<T, R>(a, c0, len, lane, av);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (c0 + 32 * u < len) {
        const int c = min(c0 + 32 * u + lane, len - 1);
        T xv[NR];
        load_x<T, NR, VEC>(x + (int64_t)c * stride, nr, xv);
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
          for (int j = 0; j < NR; ++j) acc[r][j] = fma(av[u][r], xv[j], acc[r][j]);
      }
  }
}

// Warp sums of V values (a power of two).  While a lane holds two values or
// more it exchanges half of them with its partner and keeps the other half,
// so V sums cost about V shuffles instead of 5 V.  Every value is summed over
// the lanes in the order of the plain butterfly (partners 16, 8, 4, 2, 1
// lanes away), whatever V is, so a right-hand side's bits do not depend on
// how many share the pass.  Afterwards lane l holds values
// [warp_sum_first<V>(l), + warp_sum_count<V>()) in v[0..).
template <typename T, int V>
__device__ __forceinline__ void warp_sums(T (&v)[V], int lane) {
  static_assert((V & (V - 1)) == 0, "V must be a power of two");
#pragma unroll
  for (int s = 0; s < 5; ++s) {
    const int o = 16 >> s;
    const int n = V >> s;
    if (n >= 2) {
      const bool up = lane & o;
#pragma unroll
      for (int i = 0; i < n / 2; ++i) {
        const T give = up ? v[i] : v[i + n / 2];
        const T keep = up ? v[i + n / 2] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
      }
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    }
  }
}
template <int V>
__device__ __forceinline__ int warp_sum_first(int lane) {
  return V >= 32 ? lane * (V / 32) : lane / (32 / V);
}
template <int V>
__host__ __device__ __forceinline__ constexpr int warp_sum_count() {
  return V >= 32 ? V / 32 : 1;
}
// one lane of those that hold the same value
template <int V>
__device__ __forceinline__ bool warp_sum_writer(int lane) {
  return V >= 32 || lane % (32 / (V >= 32 ? 32 : V)) == 0;
}

// av[u] = A[q*ld] for q = q0 + AW u (0 from len on)
template <typename T>
__device__ __forceinline__ void load_cols(const T *A, int64_t ld, int q0, int len, bool active, T (&av)[4]) {
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int q = q0 + AW * u;
    av[u] = active && q < len ? __ldg(A + q * ld) : T(0);
  }
}

// acc[j] += sum_q A[q*ld] x[q*stride + j] over q = warp, warp + AW, ... < len:
// a CTA's warps share the walk down 32 adjacent columns (lane: one column);
// av holds the first entries
template <typename T, int NR, bool VEC>
__device__ __forceinline__ void cols_dot(const T *A, int64_t ld, const T *x, int len, int64_t stride, int nr, int warp,
                                         bool active, T (&av)[4], T (&acc)[NR]) {
  for (int q0 = warp; q0 < len; q0 += 4 * AW) {
    if (q0 > warp) load_cols<T>(A, ld, q0, len, active, av);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int q = q0 + AW * u;
      if (q < len) {
        T xv[NR];
        load_x<T, NR, VEC>(x + (int64_t)q * stride, nr, xv);
#pragma unroll
        for (int j = 0; j < NR; ++j) acc[j] = fma(av[u], xv[j], acc[j]);
      }
    }
  }
}

// Shared memory of one item: the warps' partial sums of a column walk and the
// row sums of the same 32 unknowns.
template <typename T, int NR>
struct ItemSmem {
  T part[AW][NR][32];
  T rows[32][NR];
};

// rows per pass of a warp: its accumulators stay within 64 registers
template <typename T, int NR>
__host__ __device__ constexpr int rows_per_pass() {
  return NR * AR * (int)sizeof(T) <= 256 ? AR : NR * 2 * (int)sizeof(T) <= 256 ? 2 : 1;
}

// One item of the forward step of a wave.
template <typename T, int NR, bool VEC, bool DEP>
__device__ __forceinline__ void fwd_item(const ApplyItem &it, const ApplyNode *__restrict__ nodes,
                                         const ApplyContrib *__restrict__ cb, T *ws, T *tcur, const T *tprev, int nrhs,
                                         int j0, ItemSmem<T, NR> &sm) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nr = min(NR, nrhs - j0);
  if (it.kind == ApplyItem::ROWS) {
    // t_s = M_ss phi_s and phi_r = P_ss phi_s, rows i0 .. i0 + 31 of [M; P]
    constexpr int R = rows_per_pass<T, NR>();
    const int total = it.m + it.k;
    const T *x = ws + it.x * nrhs + j0;
    const int w0 = it.i0 + warp * AR, w1 = min(w0 + AR, total);
    auto row_ptr = [&](int row) {
      row = min(row, total - 1);
      return row < it.m ? (const T *)it.A + (int64_t)row * it.m : (const T *)it.P + (int64_t)(row - it.m) * it.m;
    };
    const T *a[R];
    T av[4][R];
#pragma unroll
    for (int r = 0; r < R; ++r) a[r] = row_ptr(w0 + r);
    if (w0 < w1) {
      load_chunk<T, R>(a, 0, it.m, lane, av);
      if constexpr (DEP) {
        // the rest of the rows, one line (128 bytes) per lane and turn
        constexpr int LE = 128 / (int)sizeof(T);
        const int lines = it.m > 128 ? (it.m - 128 + LE - 1) / LE : 0;
        for (int q = lane; q < AR * lines; q += 32) prefetch_l2(row_ptr(w0 + q % AR) + 128 + (q / AR) * LE);
      }
    }
    dep_wait<DEP>();
#pragma unroll 1
    for (int r0 = w0; r0 < w1; r0 += R) {
      T acc[R][NR];
      if (r0 > w0) {
#pragma unroll
        for (int r = 0; r < R; ++r) a[r] = row_ptr(r0 + r);
        load_chunk<T, R>(a, 0, it.m, lane, av);
      }
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int j = 0; j < NR; ++j) acc[r][j] = T(0);
      rows_dot<T, NR, R, VEC>(a, x, it.m, nrhs, nr, lane, av, acc);
      constexpr int V = R * NR;
      T(&v)[V] = reinterpret_cast<T(&)[V]>(acc);
      warp_sums<T, V>(v, lane);
      if (warp_sum_writer<V>(lane)) {
#pragma unroll
        for (int i = 0; i < warp_sum_count<V>(); ++i) {
          const int idx = warp_sum_first<V>(lane) + i;
          const int row = r0 + idx / NR, j = idx % NR;
          if (row < total && j < nr) {
            T *o = row < it.m ? tcur + (it.t + row) * nrhs + j0 : ws + (it.r + row - it.m) * nrhs + j0;
            o[j] = v[i];
          }
        }
      }
    }
  } else if (it.kind == ApplyItem::TARGET) {
    // phi_n -= sum_s B_s[:, n]^T phi_s, unknowns i0 .. i0 + 31 of n
    const int i = it.i0 + lane;
    const bool active = i < it.m;
    T acc[NR];
#pragma unroll
    for (int j = 0; j < NR; ++j) acc[j] = T(0);
    ApplyContrib ac = cb[it.first];
    T av[4];
    load_cols<T>((const T *)ac.A + i, ac.ld, warp, ac.m, active, av);
    dep_wait<DEP>();
    for (int c = 0; c < it.count; ++c) {
      if (c > 0) {
        ac = cb[it.first + c];
        load_cols<T>((const T *)ac.A + i, ac.ld, warp, ac.m, active, av);
      }
      cols_dot<T, NR, VEC>((const T *)ac.A + i, ac.ld, ws + ac.x * nrhs + j0, ac.m, nrhs, nr, warp, active, av, acc);
    }
#pragma unroll
    for (int j = 0; j < NR; ++j) sm.part[warp][j][lane] = acc[j];
    __syncthreads();
    for (int e = threadIdx.x; e < 32 * nr; e += AT) {
      const int l = e & 31, j = e >> 5;
      T s = T(0);
#pragma unroll
      for (int w = 0; w < AW; ++w) s += sm.part[w][j][l];
      if (it.i0 + l < it.m) ws[(it.x + it.i0 + l) * nrhs + j0 + j] -= s;
    }
    __syncthreads();
  } else {
    // t_s of the previous wave into the place of its phi_s, one node per warp
    dep_wait<DEP>();
    if (warp < it.count) {
      const ApplyNode &nd = nodes[it.first + warp];
      const int64_t src = nd.toff * nrhs, dst = nd.xs * nrhs;
      const int m = nd.m;
      for (int e = lane; e < m * nr; e += 32) {
        const int64_t o = (int64_t)(e / nr) * nrhs + j0 + e % nr;
        ws[dst + o] = tprev[src + o];
      }
    }
  }
}

// One item of the backward step: x_s = t_s + P_ss^T x_r - B_s x_N for the
// unknowns i0 .. i0 + 31 of s, in place of t_s (tsrc: the last wave's t_s)
template <typename T, int NR, bool VEC, bool DEP>
__device__ __forceinline__ void bwd_item(const ApplyItem &it, const ApplyNbr *__restrict__ nb, T *ws, const T *tsrc,
                                         int nrhs, int j0, ItemSmem<T, NR> &sm) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nr = min(NR, nrhs - j0);
  const int i = it.i0 + lane;
  T acc[NR];
#pragma unroll
  for (int j = 0; j < NR; ++j) acc[j] = T(0);
  const T *P = (const T *)it.P + i;
  T av[4];
  load_cols<T>(P, it.m, warp, it.k, i < it.m, av);
  if constexpr (DEP) {
    // what the first loads leave: lines of P_ss's rows, and of the rows of B_s
    for (int q = 4 * AW + (int)threadIdx.x; q < it.k; q += AT)
      prefetch_l2((const T *)it.P + (int64_t)q * it.m + it.i0);
    constexpr int LE = 128 / (int)sizeof(T);
    if (it.count > 0) {
      const int lines = (it.dN + LE - 1) / LE, rows = min(kApplyRows, it.m - it.i0);
      for (int q = threadIdx.x; q < rows * lines; q += AT)
        prefetch_l2((const T *)it.A + (int64_t)(it.i0 + q / lines) * it.dN + (q % lines) * LE);
    }
  }
  dep_wait<DEP>();
  if (it.k > 0) cols_dot<T, NR, VEC>(P, it.m, ws + it.r * nrhs + j0, it.k, nrhs, nr, warp, i < it.m, av, acc);
#pragma unroll
  for (int j = 0; j < NR; ++j) sm.part[warp][j][lane] = acc[j];
  if (it.count > 0) {
    constexpr int R = rows_per_pass<T, NR>();
#pragma unroll 1
    for (int q = 0; q < AR; q += R) {
      const int r0 = warp * AR + q;   // row inside the item
      const T *a[R];
      T ra[R][NR];
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int j = 0; j < NR; ++j) ra[r][j] = T(0);
      for (int b = 0; b < it.count; ++b) {
        const ApplyNbr n = nb[it.first + b];
#pragma unroll
        for (int r = 0; r < R; ++r)
          a[r] = (const T *)it.A + (int64_t)min(it.i0 + r0 + r, it.m - 1) * it.dN + n.col;
        T bv[4][R];
        load_chunk<T, R>(a, 0, n.size, lane, bv);
        rows_dot<T, NR, R, VEC>(a, ws + n.x * nrhs + j0, n.size, nrhs, nr, lane, bv, ra);
      }
      constexpr int V = R * NR;
      T(&v)[V] = reinterpret_cast<T(&)[V]>(ra);
      warp_sums<T, V>(v, lane);
      if (warp_sum_writer<V>(lane))
#pragma unroll
        for (int u = 0; u < warp_sum_count<V>(); ++u) {
          const int idx = warp_sum_first<V>(lane) + u;
          sm.rows[r0 + idx / NR][idx % NR] = v[u];
        }
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < 32 * nr; e += AT) {
    const int l = e & 31, j = e >> 5;
    if (it.i0 + l < it.m) {
      T s = T(0);
#pragma unroll
      for (int w = 0; w < AW; ++w) s += sm.part[w][j][l];
      T *o = ws + (it.x + it.i0 + l) * nrhs + j0 + j;
      const T t = tsrc ? tsrc[(it.t + it.i0 + l) * nrhs + j0 + j] : *o;
      s += t;
      if (it.count > 0) s -= sm.rows[l][j];
      *o = s;
    }
  }
  __syncthreads();
}

template <typename T, int NR, bool VEC>
__global__ void __launch_bounds__(AT) k_fwd(const ApplyItem *__restrict__ items, const ApplyNode *__restrict__ nodes,
                                            const ApplyContrib *__restrict__ cb, T *ws, T *tcur, const T *tprev,
                                            int nrhs, int j0) {
  __shared__ ItemSmem<T, NR> sm;
  if constexpr (early_start<T, NR>()) dep_launch();
  fwd_item<T, NR, VEC, early_start<T, NR>()>(items[blockIdx.x], nodes, cb, ws, tcur, tprev, nrhs, j0, sm);
}

template <typename T, int NR, bool VEC>
__global__ void __launch_bounds__(AT) k_bwd(const ApplyItem *__restrict__ items, const ApplyNbr *__restrict__ nb,
                                            T *ws, const T *tsrc, int nrhs, int j0) {
  __shared__ ItemSmem<T, NR> sm;
  if constexpr (early_start<T, NR>()) dep_launch();
  bwd_item<T, NR, VEC, early_start<T, NR>()>(items[blockIdx.x], nb, ws, tsrc, nrhs, j0, sm);
}

template <typename T>
__global__ void k_copy(const T *__restrict__ src, T *__restrict__ dst, int64_t n) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    dst[e] = src[e];
}

// root: x = A_root^-1 phi (phi copied to tb first), one warp per row
template <typename T, int NR, bool VEC>
__device__ __forceinline__ void root_warp(const T *__restrict__ Ainv, int m, int64_t off, int w, int lane, T *ws,
                                          const T *tb, int nrhs, int j0) {
  const int nr = min(NR, nrhs - j0);
  const T *a[1] = {Ainv + (int64_t)w * m};
  T acc[1][NR];
#pragma unroll
  for (int j = 0; j < NR; ++j) acc[0][j] = T(0);
  T av[4][1];
  load_chunk<T, 1>(a, 0, m, lane, av);
  rows_dot<T, NR, 1, VEC>(a, tb + j0, m, nrhs, nr, lane, av, acc);
  warp_sums<T, NR>(acc[0], lane);
  if (warp_sum_writer<NR>(lane)) {
    const int j = warp_sum_first<NR>(lane);
    if (j < nr) ws[(off + w) * nrhs + j0 + j] = acc[0][0];
  }
}

template <typename T, int NR, bool VEC>
__global__ void __launch_bounds__(AT) k_root(const T *__restrict__ Ainv, int m, int64_t off, T *ws, const T *tb,
                                             int nrhs, int j0) {
  const int w = blockIdx.x * AW + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (w < m) root_warp<T, NR, VEC>(Ainv, m, off, w, lane, ws, tb, nrhs, j0);
}

// ---------------------------------------------------------------------------
// Persistent apply: the whole of Algorithm 2 for one chunk of right-hand sides
// in ONE cooperative launch.  The per-step launches above cost a launch
// latency per dependent step (two per wave); here every CTA of a grid sized
// to be resident walks the step list (forward step per wave; root copy and
// solve; backward step per wave in reverse), the CTAs of the grid sharing each
// step's items, with a grid-wide barrier between dependent steps.  The barrier
// is one arrival counter; its wait is bounded (clock cycles) and a wait that
// runs out sets *err and ends the kernel (the host reports HS_ERR_TIMEOUT).
// The steps and their arithmetic are those of the per-step kernels, so the
// result is the same bit for bit.
// ---------------------------------------------------------------------------
enum { AS_FWD = 0, AS_COPY = 1, AS_ROOT = 2, AS_BWD = 3 };

struct ApplyStepDev {
  int kind;
  int wave;          // index into the waves (forward, backward)
};

// Grid barrier number `round` (0, 1, ...): one counter that only grows; CTA
// thread 0 adds 1 with release semantics and waits, with acquire loads, until
// all CTAs of this and every earlier round have arrived.  The counter is
// cleared on the stream before each launch.
__device__ __forceinline__ unsigned atom_add_release_gpu(unsigned *p, unsigned v) {
  unsigned old;
  asm volatile("atom.add.release.gpu.global.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
  return old;
}
__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// hs_test_wait_probe's switch for the persistent apply, per device
__device__ int g_apply_probe = 0;

__device__ bool grid_barrier(unsigned *bar, unsigned round, int *err, long long limit) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    const unsigned target = (round + 1u) * gridDim.x;
    atom_add_release_gpu(bar, 1u);
    const long long t0 = clock64();
    while (ld_acquire_gpu(bar) < target) {
      if (clock64() - t0 > limit) {
        atomicExch(err, 1);
        ok = 0;
        break;
      }
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// tb0, tb1: the wave scratch of even and odd waves
template <typename T, int NR, bool VEC>
__global__ void __launch_bounds__(AT) k_apply_persistent(
    const ApplyStepDev *__restrict__ steps, int nsteps, const WaveApply *__restrict__ waves, int nwaves,
    const ApplyItem *__restrict__ items, const ApplyNode *__restrict__ nodes, const ApplyNbr *__restrict__ nbrs,
    const ApplyContrib *__restrict__ cb, const T *__restrict__ root_inv, int root_m, int64_t root_off, T *ws, T *tb0,
    T *tb1, int nrhs, int j0, unsigned *bar, int *err, long long limit) {
  __shared__ ItemSmem<T, NR> sm;
  const int lane = threadIdx.x & 31;
  const int gw = blockIdx.x * AW + (threadIdx.x >> 5), gwarps = gridDim.x * AW;
  // test of the time-out path: a barrier round no launch can complete (the
  // switch is read at run time, so recorded graphs follow it too)
  if (g_apply_probe && !grid_barrier(bar, 1u << 20, err, limit)) return;
  T *troot = (nwaves & 1) ? tb1 : tb0;   // not the last wave's scratch
  for (int si = 0; si < nsteps; ++si) {
    const ApplyStepDev st = steps[si];
    if (st.kind == AS_COPY) {
      const int64_t n = (int64_t)root_m * nrhs;
      for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        troot[e] = ws[root_off * nrhs + e];
    } else if (st.kind == AS_ROOT) {
      for (int w = gw; w < root_m; w += gwarps)
        root_warp<T, NR, VEC>(root_inv, root_m, root_off, w, lane, ws, troot, nrhs, j0);
    } else {
      const WaveApply wa = waves[st.wave];
      T *tc = (st.wave & 1) ? tb1 : tb0, *tp = (st.wave & 1) ? tb0 : tb1;
      if (st.kind == AS_FWD) {
        for (int i = blockIdx.x; i < wa.f_count; i += gridDim.x)
          fwd_item<T, NR, VEC, false>(items[wa.f_first + i], nodes, cb, ws, tc, tp, nrhs, j0, sm);
      } else {
        const T *ts = st.wave == nwaves - 1 ? tc : nullptr;
        for (int i = blockIdx.x; i < wa.b_count; i += gridDim.x)
          bwd_item<T, NR, VEC, false>(items[wa.b_first + i], nbrs, ws, ts, nrhs, j0, sm);
      }
    }
    if (si + 1 < nsteps && !grid_barrier(bar, (unsigned)si, err, limit)) return;
  }
}

// user layout (column-major, ld, FP64) <-> workspace layout (unknown-major, cluster order, T)
// ds (optional): D^-1/2 per cluster-order unknown of a scaled factorization
// (A_H^-1 = D^-1/2 A'_H^-1 D^-1/2), applied on the way in and on the way out
template <typename T>
__global__ void k_gather_in(const double *__restrict__ r, int64_t ld, const int32_t *__restrict__ perm,
                            int64_t n, int nrhs, int nrhs_p, T *__restrict__ out, const double *__restrict__ ds) {
  const int64_t total = n * nrhs_p;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p = e / nrhs_p;
    const int j = (int)(e - p * nrhs_p);
    const double v = j < nrhs ? r[(int64_t)perm[p] + j * ld] : 0.0;
    out[e] = (T)(ds ? v * ds[p] : v);
  }
}

template <typename T>
__global__ void k_scatter_out(const T *__restrict__ in, const int32_t *__restrict__ perm, int64_t n, int nrhs,
                              int nrhs_p, double *__restrict__ z, int64_t ld, const double *__restrict__ ds) {
  const int64_t total = n * nrhs;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p = e / nrhs;
    const int j = (int)(e - p * nrhs);
    const double v = (double)in[p * nrhs_p + j];
    z[(int64_t)perm[p] + j * ld] = ds ? v * ds[p] : v;
  }
}

// element-wise precision change between the FP64 PCG vectors (n x np,
// unknown-major) and the workspace, times ds[unknown] when scaling
template <typename A, typename B>
__global__ void k_convert(const A *__restrict__ a, B *__restrict__ b, int64_t n, int np,
                          const double *__restrict__ ds) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    b[e] = ds ? (B)((double)a[e] * ds[e / np]) : (B)a[e];
}

// ---------------------------------------------------------------------------
// PCG kernels.  Vectors are n x NP (row-major, NP = right-hand sides rounded up
// to a power of two <= 32).  Every reduction visits the rows of one right-hand
// side in an order that depends on n alone: thread t of block b takes rows
// b*PT + t + k*gridDim*PT in turn, blocks reduce in a fixed tree, and the last
// block to finish adds the block partials in a fixed order.  So a right-hand
// side gets the same bits whether it is solved alone or batched with others
// (the apply and the SpMV are column-wise already).
// ---------------------------------------------------------------------------
constexpr int PT = 256;

struct PcgScal {       // per-rhs scalars, each an array of NP doubles
  double *bnorm2, *rz, *alpha, *beta, *pq, *rr, *tol2;   // tol2: rtol^2 ||b||^2
};
struct PcgFlags {
  int *active, *iters, *counter, *done;
};

// block sums of v[j] -> part[block*NP + j], in a fixed order
template <int NP>
__device__ void block_partial(const double (&v)[NP], double *part) {
  __shared__ double wsum[PT / 32][NP];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    double s = v[j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) wsum[warp][j] = s;
  }
  __syncthreads();
  if (threadIdx.x < NP) {
    double s = 0.0;
    for (int w = 0; w < PT / 32; ++w) s += wsum[w][threadIdx.x];
    part[blockIdx.x * NP + threadIdx.x] = s;
  }
}

// Returns true in the last block to finish; sums[j] = the total of the block
// partials.  Warp j (then j + 8, ...) adds right-hand side j's: lane l takes
// blocks l, l + 32, ... in turn, then the lanes in the butterfly's order (an
// order that depends on the grid alone, so on n alone).  One thread per
// right-hand side adding the partials one after another made this the longest
// part of each of the three vector kernels at n = 262144: 57 to 66 us a kernel,
// of which the vectors themselves need about 2 us; the 512 x 512 FP32 solve is
// 1.19 times faster with the sums spread over the lanes (and the vector passes
// around an application fused into these kernels).
template <int NP>
__device__ bool finish_sum(const double *part, int *counter, double *sums) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = (atomicAdd(counter, 1) == (int)gridDim.x - 1);
  __syncthreads();
  if (!last) return false;
  __threadfence();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nb = (int)gridDim.x;
  for (int j = warp; j < NP; j += PT / 32) {
    double s = 0.0;
#pragma unroll 8
    for (int b = lane; b < nb; b += 32) s += __ldcg(part + (int64_t)b * NP + j);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) sums[j] = s;
  }
  __syncthreads();
  if (threadIdx.x == 0) *counter = 0;
  return true;
}

// out[j] = u_j . w_j
template <int NP>
__global__ void __launch_bounds__(PT) k_dot(const double *__restrict__ u, const double *__restrict__ w, int64_t n,
                                            double *part, PcgFlags fl, double *out) {
  __shared__ double sums[NP];
  double v[NP];
#pragma unroll
  for (int j = 0; j < NP; ++j) v[j] = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)PT + threadIdx.x; i < n; i += (int64_t)gridDim.x * PT)
#pragma unroll
    for (int j = 0; j < NP; ++j) v[j] = fma(u[i * NP + j], w[i * NP + j], v[j]);
  block_partial<NP>(v, part);
  if (!finish_sum<NP>(part, fl.counter, sums)) return;
  if (threadIdx.x < NP) out[threadIdx.x] = sums[threadIdx.x];
}

// The start of a solve in one pass: the right-hand sides from the caller's
// layout (cluster order, padded to NP), r = b, x = p = 0, the apply's workspace
// from r (factor precision, times ds when scaling), ||b||^2 and the counters
template <typename T, int NP>
__global__ void __launch_bounds__(PT) k_start(const double *__restrict__ b, int64_t ld,
                                              const int32_t *__restrict__ perm, int64_t n, int nrhs,
                                              const double *__restrict__ ds, double *__restrict__ B,
                                              double *__restrict__ R, double *__restrict__ X, double *__restrict__ P,
                                              T *__restrict__ ws, double *part, PcgScal sc, PcgFlags fl, double rtol2) {
  __shared__ double sums[NP];
  double v[NP];
#pragma unroll
  for (int j = 0; j < NP; ++j) v[j] = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)PT + threadIdx.x; i < n; i += (int64_t)gridDim.x * PT) {
    const int64_t src = perm[i];
    const double d = ds ? ds[i] : 1.0;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      const double r = j < nrhs ? b[src + j * ld] : 0.0;
      B[i * NP + j] = r;
      R[i * NP + j] = r;
      X[i * NP + j] = 0.0;
      P[i * NP + j] = 0.0;
      ws[i * NP + j] = (T)(ds ? r * d : r);
      v[j] = fma(r, r, v[j]);
    }
  }
  block_partial<NP>(v, part);
  if (!finish_sum<NP>(part, fl.counter, sums)) return;
  const int j = threadIdx.x;
  if (j < NP) {
    sc.bnorm2[j] = sums[j];
    sc.tol2[j] = rtol2 * sums[j];
    sc.rz[j] = 0.0;   // beta = 0 in the first iteration
    fl.active[j] = sums[j] > 0.0 ? 1 : 0;
    fl.iters[j] = 0;
  }
}

// z from the apply's workspace (factor precision, times ds when scaling),
// r . z and beta in one pass
template <typename T, int NP>
__global__ void __launch_bounds__(PT) k_zdot(const T *__restrict__ ws, const double *__restrict__ ds,
                                             const double *__restrict__ r, int64_t n, double *__restrict__ z,
                                             double *part, PcgScal sc, PcgFlags fl) {
  __shared__ double sums[NP];
  double v[NP];
#pragma unroll
  for (int j = 0; j < NP; ++j) v[j] = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)PT + threadIdx.x; i < n; i += (int64_t)gridDim.x * PT) {
    const double d = ds ? ds[i] : 1.0;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      const double w = (double)ws[i * NP + j];
      const double zv = ds ? w * d : w;
      z[i * NP + j] = zv;
      v[j] = fma(r[i * NP + j], zv, v[j]);
    }
  }
  block_partial<NP>(v, part);
  if (!finish_sum<NP>(part, fl.counter, sums)) return;
  const int j = threadIdx.x;
  if (j < NP) {
    sc.beta[j] = (fl.active[j] && sc.rz[j] != 0.0) ? sums[j] / sc.rz[j] : 0.0;
    sc.rz[j] = sums[j];
  }
}

// p_new = z + beta p_old ; q = A p_new ; partial p_new . q ; alpha = rz / (p.q)
template <int NP>
__global__ void __launch_bounds__(PT) k_spmv_p(const int32_t *__restrict__ rp, const int32_t *__restrict__ ci,
                                               const double *__restrict__ va, int64_t n,
                                               const double *__restrict__ z, const double *__restrict__ pold,
                                               double *__restrict__ pnew, double *__restrict__ q,
                                               double *part, PcgScal sc, PcgFlags fl) {
  __shared__ double sums[NP];
  double beta[NP], v[NP];
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    beta[j] = sc.beta[j];
    v[j] = 0.0;
  }
  for (int64_t i = blockIdx.x * (int64_t)PT + threadIdx.x; i < n; i += (int64_t)gridDim.x * PT) {
    double acc[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) acc[j] = 0.0;
    for (int k = rp[i]; k < rp[i + 1]; ++k) {
      const double a = va[k];
      const int64_t c = (int64_t)ci[k] * NP;
#pragma unroll
      for (int j = 0; j < NP; ++j) acc[j] = fma(a, fma(beta[j], pold[c + j], z[c + j]), acc[j]);
    }
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      const double pn = fma(beta[j], pold[i * NP + j], z[i * NP + j]);
      pnew[i * NP + j] = pn;
      q[i * NP + j] = acc[j];
      v[j] = fma(pn, acc[j], v[j]);
    }
  }
  block_partial<NP>(v, part);
  if (!finish_sum<NP>(part, fl.counter, sums)) return;
  const int j = threadIdx.x;
  if (j < NP) {
    sc.pq[j] = sums[j];
    sc.alpha[j] = (fl.active[j] && sums[j] != 0.0) ? sc.rz[j] / sums[j] : 0.0;
  }
}

// x += alpha p ; r -= alpha q, also into the apply's workspace (factor
// precision, times ds when scaling) ; partial ||r||^2 ; convergence per rhs
template <typename T, int NP>
__global__ void __launch_bounds__(PT) k_update(double *__restrict__ x, double *__restrict__ r,
                                               const double *__restrict__ p, const double *__restrict__ q, int64_t n,
                                               const double *__restrict__ ds, T *__restrict__ ws, double *part,
                                               PcgScal sc, PcgFlags fl) {
  __shared__ double sums[NP];
  double alpha[NP], v[NP];
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    alpha[j] = sc.alpha[j];
    v[j] = 0.0;
  }
  for (int64_t i = blockIdx.x * (int64_t)PT + threadIdx.x; i < n; i += (int64_t)gridDim.x * PT) {
    const double d = ds ? ds[i] : 1.0;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      const int64_t e = i * NP + j;
      const double xv = fma(alpha[j], p[e], x[e]);
      const double rv = fma(-alpha[j], q[e], r[e]);
      x[e] = xv;
      r[e] = rv;
      ws[e] = (T)(ds ? rv * d : rv);
      v[j] = fma(rv, rv, v[j]);
    }
  }
  block_partial<NP>(v, part);
  if (!finish_sum<NP>(part, fl.counter, sums)) return;
  const int j = threadIdx.x;
  if (j < NP) {
    sc.rr[j] = sums[j];
    if (fl.active[j]) {
      fl.iters[j] += 1;
      if (sums[j] <= sc.tol2[j]) fl.active[j] = 0;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int any = 0;
    for (int i = 0; i < NP; ++i) any |= fl.active[i];
    *fl.done = any ? 0 : 1;
  }
}

// calls f(std::integral_constant<int, NP>{}) for the power of two np <= 32
template <typename F>
void with_np(int np, F &&f) {
  switch (np) {
    case 1: f(std::integral_constant<int, 1>{}); break;
    case 2: f(std::integral_constant<int, 2>{}); break;
    case 4: f(std::integral_constant<int, 4>{}); break;
    case 8: f(std::integral_constant<int, 8>{}); break;
    case 16: f(std::integral_constant<int, 16>{}); break;
    case 32: f(std::integral_constant<int, 32>{}); break;
    default: fail(HS_ERR_INVALID, "right-hand-side block must be a power of two <= 32");
  }
}

// q = b - A x
__global__ void k_residual(const int32_t *__restrict__ rp, const int32_t *__restrict__ ci,
                           const double *__restrict__ va, int64_t n, int nrhs_p,
                           const double *__restrict__ x, const double *__restrict__ b,
                           double *__restrict__ q) {
  const int64_t total = n * nrhs_p;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / nrhs_p;
    const int j = (int)(e - i * nrhs_p);
    double acc = 0.0;
    for (int k = rp[i]; k < rp[i + 1]; ++k) acc = fma(va[k], x[(int64_t)ci[k] * nrhs_p + j], acc);
    q[e] = b[e] - acc;
  }
}

int grid_for(int64_t total) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((total + 255) / 256, 152 * 8));
}

// grid of the PCG reduction kernels: a function of n only (see above)
int rgrid_for(int64_t n) { return (int)std::max<int64_t>(1, std::min<int64_t>((n + PT - 1) / PT, 152 * 4)); }

// A launch of k_fwd or k_bwd, which with `early` may start before the one
// before it ends (dep_wait)
template <typename... P, typename... A>
void launch_step(bool early, void (*kernel)(P...), int grid, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3(AT, 1, 1);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = early ? 1 : 0;
  HS_CUDA(cudaLaunchKernelEx(&cfg, kernel, args...));
  count_launch();
}

// One pass of Algorithm 2 over right-hand sides [j0, j0 + NR) of the
// workspace ws (layout [unknown][nrhs]); tb0 and tb1 are the scratch of even and
// odd waves.
template <typename T, int NR, bool VEC>
void apply_waves_nr(const FactorHandle &h, T *ws, T *tb0, T *tb1, int nrhs, int j0, cudaStream_t st) {
  const int nw = (int)h.waves.size();
  auto buf = [&](int w) { return (w & 1) ? tb1 : tb0; };
  for (int w = 0; w < nw; ++w) {
    const WaveApply &wa = h.waves[w];
    if (!wa.f_count) continue;
    launch_step(early_start<T, NR>(), k_fwd<T, NR, VEC>, wa.f_count, st, (const ApplyItem *)(h.d_items + wa.f_first),
                 (const ApplyNode *)h.d_nodes, (const ApplyContrib *)h.d_contribs, ws, buf(w), (const T *)buf(w + 1),
                 nrhs, j0);
  }
  if (h.root_m > 0) {
    const int64_t cnt = (int64_t)h.root_m * nrhs;
    T *tr = buf(nw);   // the other buffer holds the last wave's t_s
    k_copy<T><<<(int)std::min<int64_t>((cnt + 255) / 256, 1024), 256, 0, st>>>(ws + h.root_off * nrhs, tr, cnt);
    k_root<T, NR, VEC><<<(h.root_m + AW - 1) / AW, AT, 0, st>>>((const T *)h.root_inv, h.root_m, h.root_off, ws, tr,
                                                                nrhs, j0);
    count_launch(2);
  }
  for (int w = nw - 1; w >= 0; --w) {
    const WaveApply &wa = h.waves[w];
    if (!wa.b_count) continue;
    launch_step(early_start<T, NR>(), k_bwd<T, NR, VEC>, wa.b_count, st, (const ApplyItem *)(h.d_items + wa.b_first),
                 (const ApplyNbr *)h.d_nbrs, ws, w == nw - 1 ? (const T *)buf(w) : (const T *)nullptr, nrhs, j0);
  }
  HS_CUDA(cudaGetLastError());
}

// The persistent apply is opt-in (HS_APPLY_PERSISTENT=1): on the 512 x 512
// workload its grid barriers cost more than the graph's launch gaps.
// HS_APPLY_PERSISTENT_BPS (1..4) sets the CTAs per SM.
bool persistent_apply_enabled() {
  static const bool on = [] {
    const char *e = std::getenv("HS_APPLY_PERSISTENT");
    return e && e[0] == '1';
  }();
  return on;
}
int persistent_apply_bps() {
  static const int v = [] {
    const char *e = std::getenv("HS_APPLY_PERSISTENT_BPS");
    const int b = e ? std::atoi(e) : 0;
    return b >= 1 && b <= 4 ? b : 0;
  }();
  return v;
}

// One chunk of right-hand sides [j0, j0 + NR) through the persistent kernel.
// The grid is the number of CTAs that can be resident at once (at most four
// per SM), launched cooperatively so that they are; the barrier words are
// cleared on the stream first.
template <typename T, int NR, bool VEC>
void apply_persistent_nr(const FactorHandle &h, T *ws, T *tb0, T *tb1, int nrhs, int j0, cudaStream_t st) {
  static int blocks_per_sm[64] = {0};
  static std::mutex mu;
  int dev = 0;
  HS_CUDA(cudaGetDevice(&dev));
  int bps = 0, nsm = 0;
  {
    std::lock_guard<std::mutex> lk(mu);
    if (dev < 0 || dev >= 64) fail(HS_ERR_CUDA, "device ordinal out of range");
    if (!blocks_per_sm[dev]) {
      int b = 0;
      HS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_apply_persistent<T, NR, VEC>, AT, 0));
      blocks_per_sm[dev] = std::max(1, std::min(b, persistent_apply_bps() ? persistent_apply_bps() : 4));
    }
    bps = blocks_per_sm[dev];
  }
  HS_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  HS_CUDA(cudaMemsetAsync(h.d_apply_bar, 0, sizeof(unsigned), st));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(nsm * bps), 1, 1);
  cfg.blockDim = dim3(AT, 1, 1);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  // about one second of SM clocks per barrier unless hs_opts.timeout_cycles says otherwise
  const long long limit = h.timeout_cycles > 0 ? (long long)h.timeout_cycles : 2000000000LL;
  HS_CUDA(cudaLaunchKernelEx(&cfg, k_apply_persistent<T, NR, VEC>, (const ApplyStepDev *)h.d_apply_steps,
                             h.apply_nsteps, (const WaveApply *)h.d_waves, (int)h.waves.size(),
                             (const ApplyItem *)h.d_items, (const ApplyNode *)h.d_nodes, (const ApplyNbr *)h.d_nbrs,
                             (const ApplyContrib *)h.d_contribs, (const T *)h.root_inv, h.root_m, h.root_off, ws, tb0,
                             tb1, nrhs, j0, h.d_apply_bar, h.d_apply_err, limit));
  count_launch();
}

template <typename T, int NR, bool VEC>
void apply_chunk_v(const FactorHandle &h, T *ws, T *tb0, T *tb1, int nrhs, int j0, cudaStream_t st) {
  if (persistent_apply_enabled() && h.d_apply_steps && h.apply_nsteps > 0)
    apply_persistent_nr<T, NR, VEC>(h, ws, tb0, tb1, nrhs, j0, st);
  else
    apply_waves_nr<T, NR, VEC>(h, ws, tb0, tb1, nrhs, j0, st);
}

// 16-byte loads of the right-hand sides of an unknown when the chunk is full
// and every unknown's values start on a 16-byte boundary (the workspace and
// both scratch buffers do)
template <typename T, int NR>
void apply_chunk_nr(const FactorHandle &h, T *ws, T *tb0, T *tb1, int nrhs, int j0, cudaStream_t st) {
  constexpr int W = 16 / (int)sizeof(T);
  if constexpr (NR % W == 0) {
    const bool aligned = (((uintptr_t)ws | (uintptr_t)tb0 | (uintptr_t)tb1) & 15) == 0;
    if (aligned && nrhs - j0 >= NR && nrhs % W == 0 && j0 % W == 0) {
      apply_chunk_v<T, NR, true>(h, ws, tb0, tb1, nrhs, j0, st);
      return;
    }
  }
  apply_chunk_v<T, NR, false>(h, ws, tb0, tb1, nrhs, j0, st);
}

// The whole apply on a workspace whose level-L part holds the right-hand
// sides, in chunks of at most 16 of them (register accumulators).  The red
// nodes' parts need no clearing: the restriction that makes a red node's
// vector is the first to write it.
template <typename T>
void apply_chunks(const FactorHandle &h, T *ws, T *tb, T *tb2, int nrhs, cudaStream_t st) {
  for (int j0 = 0; j0 < nrhs;) {
    const int rem = nrhs - j0;
    if (rem > 8) {
      apply_chunk_nr<T, 16>(h, ws, tb, tb2, nrhs, j0, st);
      j0 += 16;
    } else if (rem > 4) {
      apply_chunk_nr<T, 8>(h, ws, tb, tb2, nrhs, j0, st);
      j0 += 8;
    } else if (rem > 2) {
      apply_chunk_nr<T, 4>(h, ws, tb, tb2, nrhs, j0, st);
      j0 += 4;
    } else if (rem == 2) {
      apply_chunk_nr<T, 2>(h, ws, tb, tb2, nrhs, j0, st);
      j0 += 2;
    } else {
      apply_chunk_nr<T, 1>(h, ws, tb, tb2, nrhs, j0, st);
      j0 += 1;
    }
  }
}

// apply on the handle's workspace d_ws, launched directly
void apply_ws_direct(const FactorHandle &h, int nrhs, cudaStream_t st) {
  if (h.prec == HS_PREC_F64) {
    double *tb = (double *)h.d_t;
    apply_chunks<double>(h, (double *)h.d_ws, tb, tb + h.t_cap * h.nrhs_cap, nrhs, st);
  } else {
    float *tb = (float *)h.d_t;
    apply_chunks<float>(h, (float *)h.d_ws, tb, tb + h.t_cap * h.nrhs_cap, nrhs, st);
  }
}

// ---------------------------------------------------------------------------
// CUDA graphs.  One apply is two dependent launches per wave (about 120 at
// the 512 x 512 workload), each too short to hide its launch latency, so
// the launch sequence is recorded once per factorization and right-hand-side
// count and replayed with one cudaGraphLaunch.  Recording happens on a private
// stream of the handle in thread-local capture mode (other threads keep
// working); the graph is then launched on the caller's stream.  Graphs hold
// the handle's device pointers, so they are dropped whenever the schedule or
// the solve buffers change.  HS_APPLY_GRAPH=0 in the environment selects
// direct launches instead.
// ---------------------------------------------------------------------------
bool graphs_enabled() {
  static const bool on = [] {
    const char *e = std::getenv("HS_APPLY_GRAPH");
    return !(e && e[0] == '0');
  }();
  return on;
}

constexpr int kDirectIters = 8;

template <typename F>
const GraphEntry &graph_for(FactorHandle &h, int key, F &&record) {
  for (const GraphEntry &g : h.graphs)
    if (g.key == key) return g;
  if (!h.cap_stream) HS_CUDA(cudaStreamCreateWithFlags(&h.cap_stream, cudaStreamNonBlocking));
  cudaGraph_t graph = nullptr;
  HS_CUDA(cudaStreamBeginCapture(h.cap_stream, cudaStreamCaptureModeThreadLocal));
  try {
    CountPause pause;   // launches are counted when the graph runs
    record(h.cap_stream);
  } catch (...) {
    cudaStreamEndCapture(h.cap_stream, &graph);
    if (graph) cudaGraphDestroy(graph);
    throw;
  }
  HS_CUDA(cudaStreamEndCapture(h.cap_stream, &graph));
  size_t nn = 0;
  cudaError_t e = cudaGraphGetNodes(graph, nullptr, &nn);
  std::vector<cudaGraphNode_t> nodes(nn);
  if (e == cudaSuccess && nn) e = cudaGraphGetNodes(graph, nodes.data(), &nn);
  int kernels = 0;
  for (size_t i = 0; e == cudaSuccess && i < nn; ++i) {
    cudaGraphNodeType t;
    e = cudaGraphNodeGetType(nodes[i], &t);
    kernels += (e == cudaSuccess && t == cudaGraphNodeTypeKernel) ? 1 : 0;
  }
  cudaGraphExec_t exec = nullptr;
  if (e == cudaSuccess) e = cudaGraphInstantiate(&exec, graph, 0);
  cudaGraphDestroy(graph);
  HS_CUDA(e);
  h.graphs.push_back(GraphEntry{key, exec, kernels});
  return h.graphs.back();
}

void run_graph(const GraphEntry &g, cudaStream_t st) {
  HS_CUDA(cudaGraphLaunch(g.exec, st));
  count_launch(g.kernels);
}

// The first apply after a factorization is launched directly: recording and
// instantiating some 120 launches takes longer than issuing them once.
void apply_ws(FactorHandle &h, int nrhs, cudaStream_t st) {
  if (!graphs_enabled() || !h.applied) {
    h.applied = true;
    apply_ws_direct(h, nrhs, st);
    return;
  }
  run_graph(graph_for(h, nrhs, [&](cudaStream_t cs) { apply_ws_direct(h, nrhs, cs); }), st);
}

void ensure_buffers(FactorHandle &h, int nrhs_cap, cudaStream_t st) {
  // a multiple of 4, so that the second buffer starts on a 16-byte boundary
  const int64_t tneed0 = (std::max<int64_t>(std::max<int64_t>(h.tmax, h.root_m), 1) + 3) & ~(int64_t)3;
  if (h.nrhs_cap >= nrhs_cap && h.d_ws && h.ws_cap >= h.ws_size && h.t_cap >= tneed0) return;
  nrhs_cap = std::max(nrhs_cap, h.nrhs_cap);
  h.drop_graphs();   // they hold the old buffers
  h.alloc.put(h.d_ws, st);
  h.alloc.put(h.d_t, st);
  h.alloc.put(h.d_pcg, st);
  h.alloc.put(h.d_part, st);
  h.alloc.put(h.d_scal, st);
  h.alloc.put(h.d_iflags, st);
  h.d_ws = h.d_t = h.d_pcg = h.d_part = h.d_scal = nullptr;
  h.d_iflags = nullptr;
  h.nrhs_cap = 0;   // until every buffer below exists (an allocation may fail)
  const int64_t n = h.plan.n;
  const size_t es = h.prec == HS_PREC_F64 ? sizeof(double) : sizeof(float);
  h.alloc.get(&h.d_ws, es * std::max<int64_t>(h.ws_size, 1) * nrhs_cap, st);
  const int64_t tneed = tneed0;
  h.alloc.get(&h.d_t, es * 2 * tneed * nrhs_cap, st);
  h.ws_cap = std::max<int64_t>(h.ws_size, 1);
  h.t_cap = tneed;
  h.alloc.get(&h.d_pcg, sizeof(double) * 7 * n * nrhs_cap, st);
  h.part_blocks = 152 * 8;
  h.alloc.get(&h.d_part, sizeof(double) * h.part_blocks * 32, st);
  h.alloc.get(&h.d_scal, sizeof(double) * 7 * 32, st);
  h.alloc.get(&h.d_iflags, sizeof(int) * (2 * 32 + 2), st);
  HS_CUDA(cudaMemsetAsync(h.d_iflags, 0, sizeof(int) * (2 * 32 + 2), st));
  if (!h.h_done) HS_CUDA(cudaMallocHost(&h.h_done, sizeof(int)));
  h.nrhs_cap = nrhs_cap;
}

}  // namespace

void apply_prepare(FactorHandle &h, cudaStream_t st) {
  // the items of every wave (one CTA each), longest chains first
  const int nw = (int)h.waves.size();
  std::vector<ApplyItem> items;
  size_t cnt = 0;
  for (const ApplyNode &nd : h.nodes) cnt += (size_t)(2 * nd.m + nd.k) / kApplyRows + 3;
  items.reserve(cnt + h.targets.size() * 2);
  for (int w = 0; w < nw; ++w) {
    WaveApply &wa = h.waves[w];
    wa.f_first = (int)items.size();
    for (int t = wa.tgt_first; t < wa.tgt_first + wa.tgt_count; ++t) {
      const ApplyTarget &tg = h.targets[t];
      for (int i = 0; i < tg.size; i += kApplyRows) {
        ApplyItem it{};
        it.kind = ApplyItem::TARGET;
        it.x = tg.x;
        it.m = tg.size;
        it.i0 = i;
        it.first = tg.first;
        it.count = tg.count;
        items.push_back(it);
      }
    }
    auto node_item = [](const ApplyNode &nd, int i) {
      ApplyItem it{};
      it.P = nd.P;
      it.x = nd.xs;
      it.r = nd.xr;
      it.t = nd.toff;
      it.m = nd.m;
      it.k = nd.k;
      it.i0 = i;
      return it;
    };
    for (int q = wa.node_first; q < wa.node_first + wa.node_count; ++q) {
      const ApplyNode &nd = h.nodes[q];
      for (int i = 0; i < nd.m + nd.k; i += kApplyRows) {
        ApplyItem it = node_item(nd, i);
        it.kind = ApplyItem::ROWS;
        it.A = nd.M;
        items.push_back(it);
      }
    }
    if (w > 0)
      for (int q = 0; q < h.waves[w - 1].node_count; q += AW) {
        ApplyItem it{};
        it.kind = ApplyItem::MOVE;
        it.first = h.waves[w - 1].node_first + q;
        it.count = std::min(AW, h.waves[w - 1].node_count - q);
        items.push_back(it);
      }
    wa.f_count = (int)items.size() - wa.f_first;
    wa.b_first = (int)items.size();
    for (int q = wa.node_first; q < wa.node_first + wa.node_count; ++q) {
      const ApplyNode &nd = h.nodes[q];
      for (int i = 0; i < nd.m; i += kApplyRows) {
        ApplyItem it = node_item(nd, i);
        it.A = nd.B;
        it.dN = nd.dN;
        it.first = nd.nb_first;
        it.count = nd.dN > 0 ? nd.nb_count : 0;
        items.push_back(it);
      }
    }
    wa.b_count = (int)items.size() - wa.b_first;
  }
  if (items.size() > h.items_cap) {
    h.alloc.put(h.d_items, st);
    h.d_items = nullptr;
    h.items_cap = 0;
    h.alloc.get(&h.d_items, sizeof(ApplyItem) * items.size(), st);
    h.items_cap = items.size();
  }
  if (!items.empty())
    HS_CUDA(cudaMemcpyAsync(h.d_items, items.data(), sizeof(ApplyItem) * items.size(), cudaMemcpyHostToDevice, st));
  // the step list of Algorithm 2, in the order of the per-step launches
  std::vector<ApplyStepDev> steps;
  for (int w = 0; w < nw; ++w)
    if (h.waves[w].f_count) steps.push_back(ApplyStepDev{AS_FWD, w});
  if (h.root_m > 0) {
    steps.push_back(ApplyStepDev{AS_COPY, 0});
    steps.push_back(ApplyStepDev{AS_ROOT, 0});
  }
  for (int w = nw - 1; w >= 0; --w)
    if (h.waves[w].b_count) steps.push_back(ApplyStepDev{AS_BWD, w});
  h.alloc.put(h.d_apply_steps, st);
  h.alloc.put(h.d_waves, st);
  h.d_apply_steps = nullptr;
  h.d_waves = nullptr;
  h.apply_nsteps = (int)steps.size();
  if (steps.empty()) return;
  h.alloc.get(&h.d_apply_steps, sizeof(ApplyStepDev) * steps.size(), st);
  HS_CUDA(cudaMemcpyAsync(h.d_apply_steps, steps.data(), sizeof(ApplyStepDev) * steps.size(), cudaMemcpyHostToDevice,
                          st));
  h.alloc.get(&h.d_waves, sizeof(WaveApply) * std::max<size_t>(h.waves.size(), 1), st);
  if (!h.waves.empty())
    HS_CUDA(cudaMemcpyAsync(h.d_waves, h.waves.data(), sizeof(WaveApply) * h.waves.size(), cudaMemcpyHostToDevice,
                            st));
  if (!h.d_apply_bar) {
    h.alloc.get(&h.d_apply_bar, 2 * sizeof(unsigned) + sizeof(int), st);
    HS_CUDA(cudaMemsetAsync(h.d_apply_bar, 0, 2 * sizeof(unsigned) + sizeof(int), st));
    h.d_apply_err = (int *)(h.d_apply_bar + 2);
  }
}

void set_apply_probe(bool on) {
  const int v = on ? 1 : 0;
  HS_CUDA(cudaMemcpyToSymbol(g_apply_probe, &v, sizeof(int)));
}

int apply_error(FactorHandle &h) {
  if (!h.d_apply_err) return 0;
  int e = 0;
  HS_CUDA(cudaMemcpy(&e, h.d_apply_err, sizeof(int), cudaMemcpyDeviceToHost));
  if (e) HS_CUDA(cudaMemset(h.d_apply_err, 0, sizeof(int)));   // reported once
  return e;
}

void apply_solve(FactorHandle &h, const double *r, double *z, int nrhs, int64_t ld, cudaStream_t st) {
  ensure_buffers(h, std::max(nrhs, h.nrhs_cap), st);
  const int64_t n = h.plan.n;
  if (h.prec == HS_PREC_F64) {
    k_gather_in<double><<<grid_for(n * nrhs), 256, 0, st>>>(r, ld, h.d_perm, n, nrhs, nrhs, (double *)h.d_ws,
                                                            h.d_dscale);
    apply_ws(h, nrhs, st);
    k_scatter_out<double><<<grid_for(n * nrhs), 256, 0, st>>>((const double *)h.d_ws, h.d_perm, n, nrhs, nrhs, z, ld,
                                                              h.d_dscale);
  } else {
    k_gather_in<float><<<grid_for(n * nrhs), 256, 0, st>>>(r, ld, h.d_perm, n, nrhs, nrhs, (float *)h.d_ws,
                                                           h.d_dscale);
    apply_ws(h, nrhs, st);
    k_scatter_out<float><<<grid_for(n * nrhs), 256, 0, st>>>((const float *)h.d_ws, h.d_perm, n, nrhs, nrhs, z, ld,
                                                             h.d_dscale);
  }
  count_launch(2);
  HS_CUDA(cudaGetLastError());
}

namespace {

// z = A_H^-1 r on the FP64 PCG vectors (layout n x np): through the workspace
// in the factor precision
void apply_pcg(FactorHandle &h, const double *R, double *Z, int np, cudaStream_t st, bool direct) {
  const int64_t tot = h.plan.n * np;
  if (h.prec == HS_PREC_F64 && !h.scale) {
    HS_CUDA(cudaMemcpyAsync(h.d_ws, R, sizeof(double) * tot, cudaMemcpyDeviceToDevice, st));
  } else if (h.prec == HS_PREC_F64) {
    k_convert<double, double><<<grid_for(tot), 256, 0, st>>>(R, (double *)h.d_ws, tot, np, h.d_dscale);
    count_launch();
  } else {
    k_convert<double, float><<<grid_for(tot), 256, 0, st>>>(R, (float *)h.d_ws, tot, np, h.d_dscale);
    count_launch();
  }
  if (direct)
    apply_ws_direct(h, np, st);
  else
    apply_ws(h, np, st);
  if (h.prec == HS_PREC_F64 && !h.scale) {
    HS_CUDA(cudaMemcpyAsync(Z, h.d_ws, sizeof(double) * tot, cudaMemcpyDeviceToDevice, st));
  } else if (h.prec == HS_PREC_F64) {
    k_convert<double, double><<<grid_for(tot), 256, 0, st>>>((const double *)h.d_ws, Z, tot, np, h.d_dscale);
    count_launch();
  } else {
    k_convert<float, double><<<grid_for(tot), 256, 0, st>>>((const float *)h.d_ws, Z, tot, np, h.d_dscale);
    count_launch();
  }
}

}  // namespace

int pcg_solve(FactorHandle &h, const double *b, double *x, int nrhs, int64_t ld, double rtol,
              int maxit, int *iters, double *relres, cudaStream_t st) {
  int np = 1;
  while (np < nrhs) np <<= 1;
  ensure_buffers(h, std::max(np, h.nrhs_cap), st);
  const int64_t n = h.plan.n;
  const int64_t tot = n * np;
  double *X = h.d_pcg, *R = X + tot, *P0 = R + tot, *P1 = P0 + tot, *Q = P1 + tot, *B = Q + tot, *Z = B + tot;
  PcgScal sc{h.d_scal,      h.d_scal + 32,  h.d_scal + 64, h.d_scal + 96,
             h.d_scal + 128, h.d_scal + 160, h.d_scal + 192};
  PcgFlags fl{h.d_iflags, h.d_iflags + 32, h.d_iflags + 64, h.d_iflags + 65};
  const int g = rgrid_for(n);
  const double rtol2 = rtol * rtol;
  auto with_t = [&](auto &&f) {
    if (h.prec == HS_PREC_F64)
      f((double *)h.d_ws);
    else
      f((float *)h.d_ws);
  };
  with_t([&](auto *ws) {
    using T = std::remove_pointer_t<decltype(ws)>;
    with_np(np, [&](auto c) {
      constexpr int NP = decltype(c)::value;
      k_start<T, NP><<<g, PT, 0, st>>>(b, ld, h.d_perm, n, nrhs, h.d_dscale, B, R, X, P0, ws, h.d_part, sc, fl,
                                       rtol2);
    });
  });
  count_launch();
  HS_CUDA(cudaGetLastError());
  // One iteration: z = A_H^-1 r (r is in the workspace already), beta, p_new =
  // z + beta p_old, q = A p_new, alpha, x and r updates.  Right-hand sides that
  // have converged get alpha = beta = 0 and stay as they are.  Recorded as a
  // graph per direction buffer pair; nothing of one call (its tolerance,
  // buffers or iteration limit) is in it.
  auto body = [&, np](cudaStream_t cs, double *pold, double *pnew) {
    apply_ws_direct(h, np, cs);
    with_t([&](auto *ws) {
      using T = std::remove_pointer_t<decltype(ws)>;
      with_np(np, [&](auto c) {
        constexpr int NP = decltype(c)::value;
        k_zdot<T, NP><<<g, PT, 0, cs>>>(ws, h.d_dscale, R, n, Z, h.d_part, sc, fl);
        k_spmv_p<NP><<<g, PT, 0, cs>>>(h.d_rowptr, h.d_col, h.d_val, n, Z, pold, pnew, Q, h.d_part, sc, fl);
        k_update<T, NP><<<g, PT, 0, cs>>>(X, R, pnew, Q, n, h.d_dscale, ws, h.d_part, sc, fl);
      });
    });
    count_launch(3);
    HS_CUDA(cudaGetLastError());
  };
  for (int it = 0;;) {
    // after an odd number of iterations the latest direction is in P1
    double *pold = (it & 1) ? P1 : P0, *pnew = (it & 1) ? P0 : P1;
    // a factorization's first iterations are launched directly: two recordings
    // of some 120 launches only pay from a few replays on (24 systems factored
    // and solved once each: 103 ms with graphs from the start, 93 without)
    const bool direct = h.pcg_direct < kDirectIters;
    if (direct) ++h.pcg_direct;
    if (graphs_enabled() && !direct) {
      const int key = kPcgGraphKey + 2 * np + (it & 1);
      run_graph(graph_for(h, key, [&](cudaStream_t cs) { body(cs, pold, pnew); }), st);
    } else {
      body(st, pold, pnew);
    }
    ++it;
    HS_CUDA(cudaMemcpyAsync(h.h_done, fl.done, sizeof(int), cudaMemcpyDeviceToHost, st));
    HS_CUDA(cudaStreamSynchronize(st));
    if (*h.h_done || it >= maxit) break;
  }
  // true relative residual
  k_residual<<<grid_for(tot), 256, 0, st>>>(h.d_rowptr, h.d_col, h.d_val, n, np, X, B, Q);
  count_launch();
  double *rr_d = h.d_scal + 5 * 32;
  with_np(np, [&](auto c) {
    constexpr int NP = decltype(c)::value;
    k_dot<NP><<<g, PT, 0, st>>>(Q, Q, n, h.d_part, fl, rr_d);
  });
  count_launch();
  k_scatter_out<double><<<grid_for(n * nrhs), 256, 0, st>>>(X, h.d_perm, n, nrhs, np, x, ld, nullptr);
  count_launch();
  HS_CUDA(cudaGetLastError());
  std::vector<double> hs(6 * 32);
  std::vector<int> hi(2 * 32 + 2);
  HS_CUDA(cudaMemcpyAsync(hs.data(), h.d_scal, sizeof(double) * 6 * 32, cudaMemcpyDeviceToHost, st));
  HS_CUDA(cudaMemcpyAsync(hi.data(), h.d_iflags, sizeof(int) * (2 * 32 + 2), cudaMemcpyDeviceToHost, st));
  HS_CUDA(cudaStreamSynchronize(st));
  if (apply_error(h)) fail(HS_ERR_TIMEOUT, "a grid barrier of the persistent apply ran out");
  bool all = true;
  for (int j = 0; j < nrhs; ++j) {
    iters[j] = hi[32 + j];
    const double bn = hs[j];
    relres[j] = bn > 0 ? std::sqrt(hs[160 + j] / bn) : 0.0;
    all = all && hi[j] == 0;
  }
  return all ? HS_OK : HS_ERR_NO_CONVERGENCE;
}

// ---------------------------------------------------------------------------
// GMRES (hs_gmres): the outer solver of the paper's experiments (Sec. 7,
// Tables 2-5), right-preconditioned by A_H^-1, x_0 = 0, FP64.  Arnoldi on
// A A_H^-1 with classical Gram-Schmidt applied twice (two fused passes instead
// of the j + 1 dependent reductions of modified Gram-Schmidt); the Hessenberg
// least-squares problem by Givens rotations on the host, which reads one
// column of dot products per step.  Flexible form: the preconditioned vectors
// z_j = A_H^-1 v_j are kept and a cycle ends with x += Z y.  With an FP32
// factor each application of A_H^-1 rounds differently; x = A_H^-1 (V y)
// would then miss the Arnoldi relation A Z = V H by that rounding (a true
// residual near 1e-6 where the estimate says 1e-10), while A Z y stays exact.
// Reductions run in an order fixed by n alone.
// ---------------------------------------------------------------------------
namespace {

constexpr int GT = 256;

int gm_blocks(int64_t n) { return (int)std::max<int64_t>(1, std::min<int64_t>((n + 4095) / 4096, 128)); }

// part[i * gridDim.x + b] = block b's share of V_i . w, i = blockIdx.y < nv
__global__ void __launch_bounds__(GT) k_gm_dots(const double *__restrict__ V, int64_t n,
                                                const double *__restrict__ w, double *__restrict__ part) {
  __shared__ double ws[GT / 32];
  const double *v = V + (int64_t)blockIdx.y * n;
  double s = 0.0;
  for (int64_t k = blockIdx.x * (int64_t)GT + threadIdx.x; k < n; k += (int64_t)gridDim.x * GT)
    s = fma(v[k], w[k], s);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int q = 0; q < GT / 32; ++q) t += ws[q];
    part[(int64_t)blockIdx.y * gridDim.x + blockIdx.x] = t;
  }
}

// h[i] = sum over b of part[i * nb + b], one warp per i
__global__ void k_gm_sum(const double *__restrict__ part, int nb, int nv, double *__restrict__ h) {
  const int i = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (i >= nv) return;
  double s = 0.0;
  for (int b = lane; b < nb; b += 32) s += part[(int64_t)i * nb + b];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) h[i] = s;
}

// w -= sum_{i < nv} h_i V_i
__global__ void k_gm_sub(const double *__restrict__ V, int64_t n, int nv, const double *__restrict__ h,
                         double *__restrict__ w) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    double s = w[k];
    for (int i = 0; i < nv; ++i) s = fma(-h[i], V[(int64_t)i * n + k], s);
    w[k] = s;
  }
}

// u = sum_{i < nv} y_i V_i
__global__ void k_gm_comb(const double *__restrict__ V, int64_t n, int nv, const double *__restrict__ y,
                          double *__restrict__ u) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int i = 0; i < nv; ++i) s = fma(y[i], V[(int64_t)i * n + k], s);
    u[k] = s;
  }
}

// v = a w ; x += z
__global__ void k_gm_scale(const double *__restrict__ w, int64_t n, double a, double *__restrict__ v) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    v[k] = a * w[k];
}
__global__ void k_gm_add(double *__restrict__ x, const double *__restrict__ z, int64_t n) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    x[k] += z[k];
}

// y = A x (permuted CSR)
__global__ void k_spmv(const int32_t *__restrict__ rp, const int32_t *__restrict__ ci, const double *__restrict__ va,
                       int64_t n, const double *__restrict__ x, double *__restrict__ y) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double acc = 0.0;
    for (int k = rp[i]; k < rp[i + 1]; ++k) acc = fma(va[k], x[ci[k]], acc);
    y[i] = acc;
  }
}

// out[0 .. nv) = V_i . w for i < nv (device), through part
void gm_dots(const double *V, int64_t n, int nv, const double *w, double *part, double *out, cudaStream_t st) {
  const int nb = gm_blocks(n);
  k_gm_dots<<<dim3(nb, nv), GT, 0, st>>>(V, n, w, part);
  k_gm_sum<<<(nv * 32 + 255) / 256, 256, 0, st>>>(part, nb, nv, out);
  count_launch(2);
}

}  // namespace

int gmres_solve(FactorHandle &h, const double *b, double *x, double rtol, int maxit, int restart, int *iters,
                double *relres, cudaStream_t st) {
  ensure_buffers(h, std::max(1, h.nrhs_cap), st);
  const int64_t n = h.plan.n;
  const int mr = std::max(1, (restart > 0 && restart < maxit) ? restart : maxit);
  // V (mr + 1 vectors), Z (mr), w, u, X, B, R; part (mr + 1) x blocks; h1, h2,
  // |w|^2; y
  const int nb = gm_blocks(n);
  const size_t need = (size_t)(2 * mr + 6) * n + (size_t)(mr + 1) * nb + 2 * (size_t)(mr + 1) + 2 + (size_t)(mr + 1);
  if (h.gm_cap < need) {
    h.alloc.put(h.d_gm, st);
    h.d_gm = nullptr;
    h.gm_cap = 0;
    h.alloc.get(&h.d_gm, sizeof(double) * need, st);
    h.gm_cap = need;
  }
  double *V = h.d_gm, *Zm = V + (size_t)(mr + 1) * n, *W = Zm + (size_t)mr * n, *U = W + n, *X = U + n, *B = X + n,
         *R = B + n;
  double *part = R + n, *hd = part + (size_t)(mr + 1) * nb, *yd = hd + 2 * (size_t)(mr + 1) + 2;
  const int g = grid_for(n);
  k_gather_in<double><<<g, 256, 0, st>>>(b, n, h.d_perm, n, 1, 1, B, nullptr);
  count_launch();
  HS_CUDA(cudaMemsetAsync(X, 0, sizeof(double) * n, st));
  std::vector<double> hh(2 * (size_t)(mr + 1) + 2);
  auto read = [&](int cnt) {
    HS_CUDA(cudaMemcpyAsync(hh.data(), hd, sizeof(double) * cnt, cudaMemcpyDeviceToHost, st));
    HS_CUDA(cudaStreamSynchronize(st));
  };
  gm_dots(B, n, 1, B, part, hd, st);
  read(1);
  const double bnorm = std::sqrt(hh[0]);
  int total = 0;
  bool converged = bnorm == 0.0;
  // Hessenberg (column-major, ld mr + 1), Givens rotations, rotated rhs
  std::vector<double> H((size_t)(mr + 1) * mr), cs(mr), sn(mr), gv(mr + 1), y(mr);
  while (!converged && total < maxit) {
    // r = b - A x; v_0 = r / |r|
    if (total == 0) {
      HS_CUDA(cudaMemcpyAsync(R, B, sizeof(double) * n, cudaMemcpyDeviceToDevice, st));
    } else {
      k_residual<<<g, 256, 0, st>>>(h.d_rowptr, h.d_col, h.d_val, n, 1, X, B, R);
      count_launch();
    }
    gm_dots(R, n, 1, R, part, hd, st);
    read(1);
    const double beta = std::sqrt(hh[0]);
    if (beta < rtol * bnorm) {
      converged = true;
      break;
    }
    k_gm_scale<<<g, 256, 0, st>>>(R, n, 1.0 / beta, V);
    count_launch();
    std::fill(gv.begin(), gv.end(), 0.0);
    gv[0] = beta;
    int j = 0;
    for (; j < mr && total < maxit; ++j) {
      // z_j = A_H^-1 v_j ; w = A z_j
      double *zj = Zm + (size_t)j * n;
      apply_pcg(h, V + (size_t)j * n, zj, 1, st, !graphs_enabled());
      k_spmv<<<g, 256, 0, st>>>(h.d_rowptr, h.d_col, h.d_val, n, zj, W);
      count_launch();
      // two passes of classical Gram-Schmidt, then |w|^2
      double *h1 = hd, *h2 = hd + (mr + 1);
      gm_dots(V, n, j + 1, W, part, h1, st);
      k_gm_sub<<<g, 256, 0, st>>>(V, n, j + 1, h1, W);
      gm_dots(V, n, j + 1, W, part, h2, st);
      k_gm_sub<<<g, 256, 0, st>>>(V, n, j + 1, h2, W);
      gm_dots(W, n, 1, W, part, hd + 2 * (mr + 1), st);
      count_launch(2);
      HS_CUDA(cudaGetLastError());
      HS_CUDA(cudaMemcpyAsync(hh.data(), hd, sizeof(double) * (2 * (mr + 1) + 1), cudaMemcpyDeviceToHost, st));
      HS_CUDA(cudaStreamSynchronize(st));
      double *col = &H[(size_t)j * (mr + 1)];
      for (int i = 0; i <= j; ++i) col[i] = hh[i] + hh[(mr + 1) + i];
      const double hn = std::sqrt(hh[2 * (mr + 1)]);
      col[j + 1] = hn;
      ++total;
      // previous rotations, then the one that zeroes col[j + 1]
      for (int i = 0; i < j; ++i) {
        const double a = col[i], c = col[i + 1];
        col[i] = cs[i] * a + sn[i] * c;
        col[i + 1] = -sn[i] * a + cs[i] * c;
      }
      const double den = std::hypot(col[j], col[j + 1]);
      cs[j] = den > 0.0 ? col[j] / den : 1.0;
      sn[j] = den > 0.0 ? col[j + 1] / den : 0.0;
      col[j] = den;
      col[j + 1] = 0.0;
      gv[j + 1] = -sn[j] * gv[j];
      gv[j] = cs[j] * gv[j];
      if (std::fabs(gv[j + 1]) < rtol * bnorm || hn == 0.0) {
        converged = true;
        ++j;
        break;
      }
      if (j + 1 < mr && total < maxit) {
        k_gm_scale<<<g, 256, 0, st>>>(W, n, 1.0 / hn, V + (size_t)(j + 1) * n);
        count_launch();
      }
    }
    // y = R^-1 g (upper triangular, j columns); x += Z y
    const int k = j;
    for (int i = k - 1; i >= 0; --i) {
      double s = gv[i];
      for (int c = i + 1; c < k; ++c) s -= H[(size_t)c * (mr + 1) + i] * y[c];
      const double d = H[(size_t)i * (mr + 1) + i];
      y[i] = d != 0.0 ? s / d : 0.0;
    }
    HS_CUDA(cudaMemcpyAsync(yd, y.data(), sizeof(double) * k, cudaMemcpyHostToDevice, st));
    k_gm_comb<<<g, 256, 0, st>>>(Zm, n, k, yd, U);
    count_launch();
    k_gm_add<<<g, 256, 0, st>>>(X, U, n);
    count_launch();
    HS_CUDA(cudaGetLastError());
  }
  // true relative residual, x back to the original order
  k_residual<<<g, 256, 0, st>>>(h.d_rowptr, h.d_col, h.d_val, n, 1, X, B, R);
  count_launch();
  gm_dots(R, n, 1, R, part, hd, st);
  read(1);
  k_scatter_out<double><<<g, 256, 0, st>>>(X, h.d_perm, n, 1, 1, x, n, nullptr);
  count_launch();
  HS_CUDA(cudaGetLastError());
  HS_CUDA(cudaStreamSynchronize(st));
  if (apply_error(h)) fail(HS_ERR_TIMEOUT, "a grid barrier of the persistent apply ran out");
  *iters = total;
  *relres = bnorm > 0.0 ? std::sqrt(hh[0]) / bnorm : 0.0;
  return converged ? HS_OK : HS_ERR_NO_CONVERGENCE;
}

// ---------------------------------------------------------------------------
// Allocation-free apply (hs_apply_static).  Some callers cannot allocate device
// memory when they solve: a service that fixes its device-memory footprint at
// start-up, or code running where a cudaMalloc could block behind other work
// or is not permitted.  For them
// the apply workspace comes from one file-scope device array instead of the
// handle's lazily grown buffers.  The array is shared by every call on a
// device and keeps the previous call's contents; calls that overlap on the
// GPU race on it.
// ---------------------------------------------------------------------------
constexpr size_t kStaticApplyBytes = size_t(16) << 20;   // 16 MiB per device
static __device__ __align__(256) unsigned char g_static_apply_ws[kStaticApplyBytes];

namespace {

std::mutex g_static_mu;
void *g_static_ptr[64] = {nullptr};

// Device address of the array for the current device.  Outside a stream
// capture it is looked up on every call (with the device current), so a
// device reset or a new primary context never leaves a stale address behind;
// while `st` is capturing, the address cached by the last call outside a
// capture is used, and a device that has none yet is an error.
void *static_ws_for_current_device(cudaStream_t st) {
  int dev = 0;
  HS_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) fail(HS_ERR_CUDA, "device ordinal out of range for the static apply buffer");
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  const cudaError_t ce = cudaStreamIsCapturing(st, &cs);
  const bool capturing = ce != cudaSuccess || cs != cudaStreamCaptureStatusNone;
  if (ce != cudaSuccess) cudaGetLastError();   // a query error is not sticky; clear it
  std::lock_guard<std::mutex> lk(g_static_mu);
  if (!capturing) {
    void *ptr = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&ptr, g_static_apply_ws);
    if (e != cudaSuccess || !ptr)
      fail(HS_ERR_CUDA, std::string("cudaGetSymbolAddress of the static apply buffer: ") + cudaGetErrorString(e));
    g_static_ptr[dev] = ptr;
  } else if (!g_static_ptr[dev]) {
    fail(HS_ERR_INVALID, "hs_apply_static: the first call on a device must come before any stream capture");
  }
  return g_static_ptr[dev];
}

template <typename T>
void apply_static_t(FactorHandle &h, const double *r, double *z, int nrhs, int64_t ld, cudaStream_t st) {
  const int64_t n = h.plan.n;
  const int64_t tcap = std::max<int64_t>(std::max<int64_t>(h.tmax, h.root_m), 1);
  // layout: workspace (ws_size x nrhs), t (tcap x nrhs), second t (tcap x nrhs), 256-byte aligned parts
  auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
  const size_t ws_b = up(sizeof(T) * (size_t)h.ws_size * nrhs);
  const size_t t_b = up(sizeof(T) * (size_t)tcap * nrhs);
  const size_t need = ws_b + 2 * t_b;
  if (need > kStaticApplyBytes)
    fail(HS_ERR_CAPACITY, "hs_apply_static needs " + std::to_string(need) + " bytes of workspace for this factor and " +
                              std::to_string(nrhs) + " right-hand sides; the static buffer holds " +
                              std::to_string(kStaticApplyBytes) + " bytes");
  unsigned char *base = (unsigned char *)static_ws_for_current_device(st);
  T *ws = (T *)base, *tb = (T *)(base + ws_b), *tb2 = (T *)(base + ws_b + t_b);
  k_gather_in<T><<<grid_for(n * nrhs), 256, 0, st>>>(r, ld, h.d_perm, n, nrhs, nrhs, ws, h.d_dscale);
  count_launch();
  apply_chunks<T>(h, ws, tb, tb2, nrhs, st);
  k_scatter_out<T><<<grid_for(n * nrhs), 256, 0, st>>>(ws, h.d_perm, n, nrhs, nrhs, z, ld, h.d_dscale);
  count_launch();
  HS_CUDA(cudaGetLastError());
}

}  // namespace

void apply_static(FactorHandle &h, const double *r, double *z, int nrhs, int64_t ld, cudaStream_t st) {
  if (h.prec == HS_PREC_F64)
    apply_static_t<double>(h, r, z, nrhs, ld, st);
  else
    apply_static_t<float>(h, r, z, nrhs, ld, st);
}

FactorHandle::~FactorHandle() {
  drop_graphs();
  if (cap_stream) cudaStreamDestroy(cap_stream);
  if (h_done) cudaFreeHost(h_done);
  alloc.put(d_src, stream);
  alloc.put(d_leaf_dest, stream);
  alloc.put(d_phi0, stream);
  alloc.put(d_phi_raw, stream);
  alloc.put(d_apply_steps, stream);
  alloc.put(d_waves, stream);
  alloc.put(d_apply_bar, stream);
  alloc.put(d_items, stream);
  alloc.put(d_dscale, stream);
  alloc.put(d_val_f, stream);
  alloc.put(d_flag, stream);
  alloc.put(d_rowptr, stream);
  alloc.put(d_col, stream);
  alloc.put(d_val, stream);
  alloc.put(d_perm, stream);
  alloc.put(d_nodes, stream);
  alloc.put(d_nbrs, stream);
  alloc.put(d_contribs, stream);
  alloc.put(d_ws, stream);
  alloc.put(d_t, stream);
  alloc.put(d_pcg, stream);
  alloc.put(d_gm, stream);
  alloc.put(d_part, stream);
  alloc.put(d_scal, stream);
  alloc.put(d_iflags, stream);
}

}  // namespace hs
