// Truncation of super nodes above the shared-memory Jacobi limit: symmetric
// eigen-decomposition of the Gram matrix by Householder tridiagonalisation,
// Sturm-sequence multisection and inverse iteration.  Per wave, one launch of
// each kernel for all its nodes:
//   1. k_trunc_prep (one CTA per node): GC basis U_1 = orth[phi_s, A_sw phi_w]
//      (Sec. 6; Appendix B: its dominant left singular vectors), J = G (LoRaSp)
//      or (I - U1 U1^T) G (I - U1 U1^T) (GC), and with C = U1^T G U1 the
//      coupling X = (I - U1 U1^T) G U1 of the two blocks of G; J, X and C times
//      a power of two that brings G's largest diagonal entry near 1.
//   2. J = Q T Q^T (kernels_cluster.cu, or the step kernels below), and
//      Z = Q^T X (k_qmul).
//   3. k_rank (one CTA per node): ||A_sw||_2^2 = lambda_max(G), from T (LoRaSp)
//      or from the inertia of G - sigma I in the basis [U_1, its complement]
//      (GC); the rank k2 = #{lambda(T) > eps^2 lambda_max(G)} by one Sturm count
//      in FP64 (Sec. 3.2, strict).
//   4. k_eigval: the k2 largest eigenvalues of T, 8 or 32 lanes each.
//   5. k_invit: their eigenvectors by inverse iteration on T (tridiagonal LU
//      with partial pivoting, three steps, modified Gram-Schmidt inside
//      clusters of eigenvalues closer than 10 u ||T||), one lane each.
//   6. k_qmul: U_2 = Q Y by the stored reflectors, a few columns per warp.
// The host re-orthonormalises [U_1, U_2] afterwards (CholQR2), which keeps its
// span.  What a kernel does for a node depends on the node alone, so it gets
// the same bits in any batch.
//
// All of it is bound by chains of dependent steps (a division per row of T, a
// reduction per reflector), not by arithmetic or bandwidth, so the kernels cut
// the number of steps (many points of a section at once), spread the
// eigenvalues over the SMs, and keep the chains in registers and shared
// memory.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cstdlib>

#include "hs_internal.h"
#include "trunc_common.cuh"

namespace hs {

namespace {

// Block-wide sum in T (red: 33 T of shared memory); every thread gets the total.
// Reductions inside the per-step loops stay in the factor precision: on this
// GPU FP64 instructions issue at a small fraction of the FP32 rate.
template <typename T>
__device__ T bsum_t(T v, T *red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    T s = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : T(0);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) red[32] = s;
  }
  __syncthreads();
  const T r = red[32];
  __syncthreads();
  return r;
}

template <typename R>
__device__ __forceinline__ R unit_round();
template <>
__device__ __forceinline__ double unit_round<double>() { return 2.220446049250313e-16; }
template <>
__device__ __forceinline__ float unit_round<float>() { return 1.1920929e-07f; }

__device__ __forceinline__ float hash_unit(uint32_t a, uint32_t b) {
  uint32_t x = a * 0x9E3779B9u ^ (b + 0x7F4A7C15u);
  x ^= x >> 16;
  x *= 0x85EBCA6Bu;
  x ^= x >> 13;
  x *= 0xC2B2AE35u;
  x ^= x >> 16;
  return (float)(x >> 8) * (2.0f / 16777216.0f) - 1.0f;
}


// Sign and magnitude tests of the Sturm pivots, in FP64 by the high word
// (comparisons issue on the FP64 pipe too): pivmin's low word is zero
// (sturm_pivmin), so the comparison of the high words is that of the values
__device__ __forceinline__ bool pivot_tiny(float q, float pivmin) { return fabs(q) < pivmin; }
__device__ __forceinline__ bool pivot_tiny(double q, double pivmin) {
  return (__double2hiint(q) & 0x7fffffff) < __double2hiint(pivmin);
}
__device__ __forceinline__ bool pivot_pos(float q) { return q > 0.f; }
__device__ __forceinline__ bool pivot_pos(double q) { return __double2hiint(q) >= 0; }   // (not zero: not tiny)

// number of eigenvalues above sigma of the tridiagonal with diagonal d and
// squared sub-diagonal e2 (e2[i] couples i - 1 and i; e2[0] unused)
template <typename R>
__device__ __forceinline__ int count_above(const R *d, const R *e2, int m, R sigma, R pivmin) {
  R q = d[0] - sigma;
  if (pivot_tiny(q, pivmin)) q = -pivmin;
  int c = pivot_pos(q);
#pragma unroll 4
  for (int i = 1; i < m; ++i) {
    q = (d[i] - sigma) - e2[i] / q;
    if (pivot_tiny(q, pivmin)) q = -pivmin;
    c += pivot_pos(q);
  }
  return c;
}

// positive eigenvalues of the symmetric k x k matrix S (ld N)
template <typename R, int N>
__device__ __forceinline__ int count_positive(R (&S)[N][N], int k) {
  if constexpr (N == 1) {
    return S[0][0] > R(0);
  } else if constexpr (N == 2) {
    if (k == 0) return 0;
    if (k == 1) return S[0][0] > R(0);
    const R det = S[0][0] * S[1][1] - S[1][0] * S[1][0];
    if (det < R(0)) return 1;
    return S[0][0] + S[1][1] > R(0) ? 2 : 0;
  } else {
    // cyclic Jacobi
    for (int sweep = 0; sweep < 16; ++sweep)
      for (int p = 0; p < k; ++p)
        for (int q = p + 1; q < k; ++q) {
          const R apq = S[q][p];
          if (fabs(apq) <= R(1e-30)) continue;
          const R th = (S[q][q] - S[p][p]) / (R(2) * apq);
          R tt = R(1) / (fabs(th) + sqrt(R(1) + th * th));
          if (th < R(0)) tt = -tt;
          const R c = R(1) / sqrt(R(1) + tt * tt), sn = tt * c;
          for (int l = 0; l < k; ++l) {
            const R slp = S[l][p], slq = S[l][q];
            S[l][p] = c * slp - sn * slq;
            S[l][q] = sn * slp + c * slq;
          }
          for (int l = 0; l < k; ++l) {
            const R spl = S[p][l], sql = S[q][l];
            S[p][l] = c * spl - sn * sql;
            S[q][l] = sn * spl + c * sql;
          }
        }
    int pos = 0;
    for (int p = 0; p < k; ++p) pos += S[p][p] > R(0);
    return pos;
  }
}

// Eigenvalues above sigma > 0 of G = [[C, X^T], [X, J]] (basis [U_1, its
// complement]), J = Q T Q^T, Z = Q^T X (column a at Z + a ldz).  Haynsworth
// inertia of [[T - sigma I, Z], [Z^T, C - sigma I]]: those of T - sigma I, plus
// those of C - sigma I - Z^T (T - sigma I)^-1 Z.  (T carries k1 more zero
// eigenvalues than the complement's block, which no sigma > 0 counts.)  With
// T - sigma I = L D L^T and W = L^-1 Z, the product is W^T D^-1 W: one forward
// sweep with register accumulators.  The FP32 sweep and the FP64 one differ
// in precision only.
template <typename R, int KB>
__device__ __forceinline__ int count_above_gc(const R *d, const R *e, const R *e2, int m, const R *Z, int ldz, int k1,
                                              const R *C, R sigma, R pivmin) {
  R w[KB], g[KB][KB];
#pragma unroll
  for (int a = 0; a < KB; ++a) {
    w[a] = R(0);
#pragma unroll
    for (int b = 0; b < KB; ++b) g[a][b] = R(0);
  }
  int c = 0;
  R l = R(0), inv = R(0);
#pragma unroll 2
  for (int i = 0; i < m; ++i) {
    R q = (d[i] - sigma) - e2[i] * inv;   // e2[0] = 0
    if (pivot_tiny(q, pivmin)) q = -pivmin;
    c += pivot_pos(q);
    inv = R(1) / q;
#pragma unroll
    for (int a = 0; a < KB; ++a)
      if (KB <= 2 || a < k1) w[a] = (KB == 1 || a < k1 ? Z[(size_t)a * ldz + i] : R(0)) - l * w[a];
#pragma unroll
    for (int a = 0; a < KB; ++a)
#pragma unroll
      for (int b = 0; b <= a; ++b)
        if (KB <= 2 || a < k1) g[a][b] = fma(w[a] * inv, w[b], g[a][b]);
    l = e[i] * inv;                        // e[m - 1] = 0
  }
  R S[KB][KB];
#pragma unroll
  for (int a = 0; a < KB; ++a)
#pragma unroll
    for (int b = 0; b <= a; ++b) {
      const R v = (a < k1 && b < k1 ? R(0.5) * (C[a * kMaxK1 + b] + C[b * kMaxK1 + a]) : R(0)) - g[a][b] -
                  (a == b ? sigma : R(0));
      S[a][b] = v;
      S[b][a] = v;
    }
  return c + count_positive<R, KB>(S, k1);
}

// several preserved vectors (k1 > 2) in a call of its own, off the register
// allocation of the one-vector path
template <typename R>
__device__ __noinline__ int count_above_gc_wide(const R *d, const R *e, const R *e2, int m, const R *Z, int ldz,
                                                int k1, const R *C, R sigma, R pivmin) {
  return count_above_gc<R, kMaxK1>(d, e, e2, m, Z, ldz, k1, C, sigma, pivmin);
}

// smallest pivot of a Sturm recurrence (FP64: its low word cleared, for pivot_tiny)
__device__ __forceinline__ float sturm_pivmin(float emax2) { return fmaxf(1e-30f * fmaxf(1.f, emax2), 1e-35f); }
__device__ __forceinline__ double sturm_pivmin(double emax2) {
  return __hiloint2double(__double2hiint(1e-30 * fmax(1.0, emax2)), 0);
}

// The multisection of one value by the lanes of a warp group: `above(sigma)`
// is true below the wanted eigenvalue and false above it.  With closed ends
// the L points include lo and hi, whose counts confirm the bracket (returns -1
// when the value lies below lo, 1 above hi); else they divide (lo, hi) into
// L + 1 parts.
template <typename R, int L, typename F>
__device__ __forceinline__ int section(R &lo, R &hi, int lane, bool closed, F &&above) {
  const int l = lane % L;
  const R h = hi - lo;
  const R p0 = closed ? lo + h * R(l) / R(L - 1) : lo + h * R(l + 1) / R(L + 1);
  const unsigned ball = __ballot_sync(0xffffffffu, above(p0));
  const unsigned mine = L == 32 ? ball : (ball >> (lane / L * L)) & ((1u << (L & 31)) - 1u);
  const int n = __popc(mine);   // points below the value
  if (closed) {
    if (n == 0) return -1;
    if (n == L) return 1;
    const R a = lo + h * R(n - 1) / R(L - 1), b = lo + h * R(n) / R(L - 1);
    lo = a;
    hi = b;
  } else {
    const R a = n > 0 ? lo + h * R(n) / R(L + 1) : lo, b = n < L ? lo + h * R(n + 1) / R(L + 1) : hi;
    lo = a;
    hi = b;
  }
  return 0;
}

// J = G - U1 X^T - X U1^T + U1 c U1^T (the Gram matrix projected off span U_1),
// X = G U1 in Y's columns and U1 in U's (column a at + a m), c in shared memory
// (ld kMaxK1), times f; one warp per row.  KB >= k1 sizes the per-row registers.
template <typename T, int KB>
__device__ void build_projected_gram(const T *G, const T *U, const T *Y, const T *s_c, T *A, int m, int k1,
                                     const Pow2<T> &f) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = blockDim.x >> 5;
  for (int i = warp; i < m; i += nw) {
    T ui[KB], xi[KB], cu[KB];
#pragma unroll
    for (int a = 0; a < KB; ++a) {
      ui[a] = a < k1 ? U[(size_t)a * m + i] : T(0);
      xi[a] = a < k1 ? Y[(size_t)a * m + i] : T(0);
    }
#pragma unroll
    for (int bb = 0; bb < KB; ++bb) {
      T su = T(0);
#pragma unroll
      for (int a = 0; a < KB; ++a)
        if (a < k1) su = fma(ui[a], s_c[a * kMaxK1 + bb], su);
      cu[bb] = su;
    }
    for (int j = lane; j < m; j += 32) {
      T v = G[(int64_t)i * m + j];
#pragma unroll
      for (int a = 0; a < KB; ++a)
        if (a < k1) {
          const T uj = U[(size_t)a * m + j];
          v = fma(-ui[a], Y[(size_t)a * m + j], fma(-xi[a], uj, v));
          v = fma(cu[a], uj, v);
        }
      A[(int64_t)i * m + j] = f(v);
    }
  }
}

// k1 > 2 (several preserved vectors) in a call of its own, off the register
// allocation of the one-vector path
template <typename T>
__device__ __noinline__ void build_projected_gram_wide(const T *G, const T *U, const T *Y, const T *s_c, T *A,
                                                       int m, int k1, const Pow2<T> &f) {
  build_projected_gram<T, kMaxK1>(G, U, Y, s_c, A, m, k1, f);
}

// U_1, J, X and C of one node, or the complete basis (eps = 0)
template <typename T, int NT>
__global__ void __launch_bounds__(NT) k_trunc_prep(const TruncTask<T> *__restrict__ tasks, int *__restrict__ kout,
                                                  int variant) {
  __shared__ double red[33];
  __shared__ double s_gR[kMaxK1 * 2 * kMaxPhi], s_gW[kMaxK1 * kMaxK1 + kMaxK1];
  __shared__ int s_gk;
  __shared__ T s_c[kMaxK1 * kMaxK1];   // C = U1^T G U1, ld kMaxK1
  __shared__ T redt[34];
  const TruncTask<T> t = tasks[blockIdx.x];
  const int m = t.m;
  const int tid = threadIdx.x, nt = blockDim.x;
  const BigLayout<T> L = big_layout<T>(t.work, m);
  T *A = L.A, *Y = L.Y;
  const bool gc = variant != HS_LORASP;
  if (!gc) {
    if (t.eps == 0.0) {
      // no truncation: the complete basis U = I
      for (int64_t q = tid; q < (int64_t)m * m; q += nt) t.U[q] = (q / m == q % m) ? T(1) : T(0);
      if (tid == 0) kout[t.k_idx] = m;
      return;
    }
    const Pow2<T> f = gram_scale(t.G, m, red);
    for (int64_t q = tid; q < (int64_t)m * m; q += nt) A[q] = f(t.G[q]);
    if (tid == 0) L.sc_int[0] = 0;
    return;
  }
  // GC basis (scratch: m doubles in LS)
  const int k1 = gc_basis_dev<T>(t.phi, t.a, t.np, m, variant == HS_GC_PROJ, t.eps1, t.U, (double *)L.LS, red, s_gR,
                                 s_gW, &s_gk);
  if (t.eps == 0.0) {
    // no truncation: complete the GC basis to all of R^m (Householder QR of
    // U_1; scratch k1 m doubles); nothing to complete when it spans R^m
    if (k1 < m) {
      if (k1 <= 2)
        gc_complete<T>(t.U, m, k1, (double *)L.LS, red);
      else
        gc_complete_n<T>(t.U, m, k1, (double *)L.LS, s_gW, red);
    }
    if (tid == 0) kout[t.k_idx] = m;
    return;
  }
  // U1's columns side by side (in U they are m apart, a sector a word: each of
  // the loops over G below reads them once per row)
  T *Uc = L.LS + (size_t)kMaxK1 * m;   // (X takes the first kMaxK1 columns of LS)
  for (int64_t q = tid; q < (int64_t)m * k1; q += nt) Uc[q] = t.U[(q % m) * m + q / m];
  __syncthreads();
  // G U1 in Y's first columns, C = U1^T G U1; one warp per row of G
  {
    const int warp = tid >> 5, lane = tid & 31, nw = nt >> 5;
    for (int i = warp; i < m; i += nw)
      for (int a = 0; a < k1; ++a) {
        T s = T(0);
        for (int j = lane; j < m; j += 32) s = fma(t.G[(int64_t)i * m + j], Uc[(size_t)a * m + j], s);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) Y[(size_t)a * m + i] = s;
      }
  }
  __syncthreads();
  for (int q = tid; q < kMaxK1 * kMaxK1; q += nt) s_c[q] = T(0);
  __syncthreads();
  for (int a = 0; a < k1; ++a)
    for (int bb = 0; bb < k1; ++bb) {
      T s = T(0);
      for (int i = tid; i < m; i += nt) s = fma(Uc[(size_t)a * m + i], Y[(size_t)bb * m + i], s);
      const T cab = bsum_t<T>(s, redt);
      if (tid == 0) s_c[a * kMaxK1 + bb] = cab;
    }
  __syncthreads();
  const Pow2<T> f = gram_scale(t.G, m, red);
  if (k1 <= 2)
    build_projected_gram<T, 2>(t.G, Uc, Y, s_c, A, m, k1, f);
  else
    build_projected_gram_wide<T>(t.G, Uc, Y, s_c, A, m, k1, f);
  // X = G U1 - U1 C (the scratch in LS is no longer in use)
  T *X = L.LS;
  for (int64_t q = tid; q < (int64_t)m * k1; q += nt) {
    const int a = (int)(q / m), i = (int)(q % m);
    T x = Y[(size_t)a * m + i];
    for (int b = 0; b < k1; ++b) x = fma(-Uc[(size_t)b * m + i], s_c[b * kMaxK1 + a], x);
    X[(size_t)a * m + i] = f(x);
  }
  if (tid == 0) L.sc_int[0] = k1;
  for (int q = tid; q < kMaxK1 * kMaxK1; q += nt) L.sc_c[q] = (double)f(s_c[q]);
}

// ---------------------------------------------------------------------------
// lambda_max(G) and the rank of one node per CTA.
// lambda_max: FP32 factors section its bracket by 256 points a round (three
// rounds to 4 u); the FP64 factor starts from such an FP32 value and confirms
// and refines it by one warp's sections in FP64, whose rate (1/64 of FP32's)
// makes more points a round cost more than they save.  The bracket is
// [largest diagonal entry, Gershgorin bound of T + trace C].
// Rank: the FP64 Sturm count at eps^2 lambda_max runs from both ends of T at
// once (two threads) and meets in the middle row, whose pivot takes both
// neighbours' quotients: the same inertia in half the dependent divisions.
// ---------------------------------------------------------------------------
constexpr int kRankThreads = 256;

// dynamic shared memory: d, e2 (FP64), d, e, e2, Z in T, and for the FP64
// factor also in FP32; Z stays in global memory when it does not fit, and all of
// it when the rest does not (0 bytes).  The places decide which recurrences a node
// runs, so they depend on the node alone, not on what else is in the launch.
struct RankPlace {
  int zcols;      // columns of Z in shared memory (room for 2 np, or none)
  size_t bytes;
};
template <typename T>
__host__ __device__ inline RankPlace rank_place(int m, int np, bool gc, size_t limit) {
  const size_t mm = (size_t)m + 1;
  const size_t base = (2 * sizeof(double) + 3 * sizeof(float) + (sizeof(T) == 8 ? sizeof(double) : 0)) * mm + 64;
  const size_t col = (sizeof(float) + (sizeof(T) == 8 ? sizeof(double) : 0)) * mm;
  const int z = gc ? 2 * np : 0;
  if (base + col * z <= limit) return RankPlace{z, base + col * z};
  return RankPlace{0, base <= limit ? base : 0};
}

template <typename T>
__global__ void __launch_bounds__(kRankThreads) k_rank(const TruncTask<T> *__restrict__ tasks, int *__restrict__ kout,
                                                      int variant, size_t limit) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double s_red[3 * kRankThreads / 32];
  __shared__ float s_cf[kMaxK1 * kMaxK1];
  __shared__ T s_ct[kMaxK1 * kMaxK1];
  __shared__ double s_half[2], s_lmax;
  __shared__ int s_cnt[2];
  const TruncTask<T> t = tasks[blockIdx.x];
  const int m = t.m;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const BigLayout<T> L = big_layout<T>(t.work, m);
  const bool gc = variant != HS_LORASP;
  const int k1 = gc ? L.sc_int[0] : 0;
  const RankPlace place = rank_place<T>(m, t.np, gc, limit);
  const int zcols = place.zcols;
  const bool in_smem = place.bytes > 0;
  const size_t mm = (size_t)m + 1;
  // (nodes beyond shared memory keep these vectors in Y, which is free until
  // the eigenvectors go there)
  double *d = in_smem ? (double *)smem_raw : (double *)(((uintptr_t)L.Y + 15) & ~(uintptr_t)15), *e2 = d + mm;
  unsigned char *p = (unsigned char *)(e2 + mm);
  double *ed = nullptr, *zd = nullptr;   // FP64 factor: e and Z
  if constexpr (sizeof(T) == 8) {
    ed = (double *)p;
    zd = ed + mm;
    p = (unsigned char *)(zd + (size_t)zcols * mm);
  }
  float *df = (float *)p, *ef = df + mm, *e2f = ef + mm, *zf = e2f + mm;
  const bool zs = zcols >= k1;           // Z in shared memory
  // T: the tridiagonalisation left d, e for k < m - 2 and the trailing 2 x 2 block in A
  double dmax = -1e300, emax = 0.0, glo = 1e300, ghi = -1e300;
  auto dat = [&](int i) {
    return i + 2 < m ? L.d[i] : (double)L.A[(int64_t)i * m + i];
  };
  auto eat = [&](int i) {   // e_i couples i and i + 1
    return i + 2 < m ? L.e[i] : i + 2 == m ? (double)L.A[(int64_t)(m - 1) * m + m - 2] : 0.0;
  };
  for (int i = tid; i < m; i += kRankThreads) {
    // FP32 factors work on the FP32 rounding of T throughout, the count in FP64
    const double di = dat(i), ei = eat(i), em = i > 0 ? eat(i - 1) : 0.0;
    d[i] = di;
    e2[i] = em * em;
    const double r = fabs(em) + fabs(ei);
    glo = fmin(glo, di - r);
    ghi = fmax(ghi, di + r);
    dmax = fmax(dmax, di);
    emax = fmax(emax, em * em);
    L.dt[i] = (T)di;
    L.et[i] = (T)ei;
    if (sizeof(T) == 8) ed[i] = ei;
  }
  for (int o = 16; o > 0; o >>= 1) {
    glo = fmin(glo, __shfl_xor_sync(0xffffffffu, glo, o));
    ghi = fmax(ghi, __shfl_xor_sync(0xffffffffu, ghi, o));
    dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    emax = fmax(emax, __shfl_xor_sync(0xffffffffu, emax, o));
  }
  constexpr int NW = kRankThreads / 32;
  __shared__ double s_emax[NW];
  if (lane == 0) {
    s_red[warp] = glo;
    s_red[NW + warp] = ghi;
    s_red[2 * NW + warp] = dmax;
    s_emax[warp] = emax;
  }
  __syncthreads();
  for (int q = 0; q < NW; ++q) {
    glo = fmin(glo, s_red[q]);
    ghi = fmax(ghi, s_red[NW + q]);
    dmax = fmax(dmax, s_red[2 * NW + q]);
    emax = fmax(emax, s_emax[q]);
  }
  const double tnorm = fmax(fabs(glo), fabs(ghi));
  // the bracket of lambda_max(G): C's diagonal bounds it below, its trace above
  double ctr = 0.0, cmax = 0.0;
  for (int a = 0; a < k1; ++a) {
    const double c = L.sc_c[a * kMaxK1 + a];
    ctr += fmax(c, 0.0);
    cmax = fmax(cmax, c);
  }
  const double hi0 = (fmax(ghi, 0.0) + ctr) * (1.0 + 1e-4) + (sizeof(T) == 8 ? 1e-290 : 1e-30);
  const double lo0 = fmax(fmax(dmax, cmax), 0.0) * (1.0 - 1e-4);
  for (int i = tid; i < m; i += kRankThreads) {
    const float e1 = (float)eat(i), e0 = i > 0 ? (float)eat(i - 1) : 0.f;
    df[i] = (float)d[i];
    ef[i] = e1;
    e2f[i] = e0 * e0;
    if (zs)
      for (int a = 0; a < k1; ++a) {
        const T z = L.LS[(size_t)a * m + i];
        zf[(size_t)a * mm + i] = (float)z;
        if (sizeof(T) == 8) zd[(size_t)a * mm + i] = (double)z;
      }
  }
  for (int q = tid; q < kMaxK1 * kMaxK1; q += kRankThreads) {
    s_cf[q] = (float)L.sc_c[q];
    s_ct[q] = (T)L.sc_c[q];
  }
  __syncthreads();
  const float pivf = sturm_pivmin((float)emax);
  double lmax;   // (of G as k_trunc_prep scales it)
  const bool wide_global = gc && !zs;   // many preserved vectors on a huge node
  {
    float lo = (float)lo0, hi = (float)hi0 * 1.000001f + 1e-37f;
    if (!wide_global || sizeof(T) == 4) {
      for (int round = 0; round < 8 && hi - lo > 4.f * unit_round<float>() * hi; ++round) {
        const float h = hi - lo;
        const float sig = lo + h * (float)(tid + 1) * (1.f / (kRankThreads + 1));
        int c;
        if (k1 == 0)
          c = count_above<float>(df, e2f, m, sig, pivf);
        else if (wide_global)
          c = count_above_gc_wide<float>(df, ef, e2f, m, (const float *)(const void *)L.LS, m, k1, s_cf, sig, pivf);
        else if (k1 == 1)
          c = count_above_gc<float, 1>(df, ef, e2f, m, zf, (int)mm, k1, s_cf, sig, pivf);
        else if (k1 == 2)
          c = count_above_gc<float, 2>(df, ef, e2f, m, zf, (int)mm, k1, s_cf, sig, pivf);
        else
          c = count_above_gc_wide<float>(df, ef, e2f, m, zf, (int)mm, k1, s_cf, sig, pivf);
        const int n = __syncthreads_count(c >= 1);
        const float a = n > 0 ? lo + h * (float)n * (1.f / (kRankThreads + 1)) : lo;
        const float b = n < kRankThreads ? lo + h * (float)(n + 1) * (1.f / (kRankThreads + 1)) : hi;
        lo = a;
        hi = b;
      }
    }
    lmax = (double)(0.5f * (lo + hi));
    if constexpr (sizeof(T) == 8) {
      if (warp == 0) {
        const double piv = sturm_pivmin(emax);
        auto above = [&](double sig) {
          if (k1 == 0) return count_above<double>(d, e2, m, sig, piv) >= 1;
          const double *z = zs ? zd : (const double *)L.LS;
          const int ldz = zs ? (int)mm : m;
          return (k1 == 1   ? count_above_gc<double, 1>(d, ed, e2, m, z, ldz, k1, s_ct, sig, piv)
                  : k1 == 2 ? count_above_gc<double, 2>(d, ed, e2, m, z, ldz, k1, s_ct, sig, piv)
                            : count_above_gc_wide<double>(d, ed, e2, m, z, ldz, k1, s_ct, sig, piv)) >= 1;
        };
        double l = lmax * (1.0 - 7.6e-6), h = lmax * (1.0 + 7.6e-6);   // 64 u of FP32
        const int miss = wide_global ? 2 : section<double, 32>(l, h, lane, true, above);
        if (miss != 0) {
          const double was_l = lmax * (1.0 - 7.6e-6), was_h = lmax * (1.0 + 7.6e-6);
          l = miss == 1 ? was_h : lo0;
          h = miss == -1 ? was_l : hi0;
        }
        for (int round = 0; round < 40 && h - l > 4.0 * unit_round<double>() * h; ++round) {
          const double pl = l, ph = h;
          section<double, 32>(l, h, lane, false, above);
          if (!(l > pl || h < ph)) break;
        }
        if (lane == 0) s_lmax = 0.5 * (l + h);
      }
      __syncthreads();
      lmax = s_lmax;
    }
  }
  const double thr = t.eps * t.eps * lmax;
  // the Sturm count in FP64 from both ends, middle row h
  const double piv = sturm_pivmin(emax);
  const int h = m / 2;
  if (tid == 0) {
    int c = 0;
    double q = 0.0;
    for (int i = 0; i < h; ++i) {
      q = d[i] - thr - (i > 0 ? e2[i] / q : 0.0);
      if (fabs(q) < piv) q = -piv;
      c += q < 0.0;
    }
    s_half[0] = h > 0 ? e2[h] / q : 0.0;
    s_cnt[0] = c;
  } else if (tid == 32) {
    int c = 0;
    double q = 0.0;
    for (int i = m - 1; i > h; --i) {
      q = d[i] - thr - (i + 1 < m ? e2[i + 1] / q : 0.0);
      if (fabs(q) < piv) q = -piv;
      c += q < 0.0;
    }
    s_half[1] = h + 1 < m ? e2[h + 1] / q : 0.0;
    s_cnt[1] = c;
  }
  __syncthreads();
  if (tid == 0) {
    double q = d[h] - thr - s_half[0] - s_half[1];
    if (fabs(q) < piv) q = -piv;
    int k2 = m - (s_cnt[0] + s_cnt[1] + (q < 0.0 ? 1 : 0));
    k2 = max(0, min(k2, min(m - k1, t.cap - k1)));   // max_rank_ratio: the largest eigenvalues are kept
    L.sc_int[1] = k2;
    L.sc_b[0] = thr;
    L.sc_b[1] = ghi + unit_round<T>() * tnorm * 2.0 * m + (sizeof(T) == 8 ? 1e-290 : 1e-30);
    L.sc_b[2] = emax;
    *L.sc_tnorm = tnorm;
    kout[t.k_idx] = k1 + k2;
  }
}

// ---------------------------------------------------------------------------
// The k2 largest eigenvalues of T (shifts of the inverse iteration), `lanes`
// of a warp sectioning each: 8 below m = 128, where a wave has many nodes and
// the work counts, 32 from there on, where the rounds do.  FP64, bound by its
// issue rate, takes 8 throughout.  The bracket is
// (eps^2 lambda_max, Gershgorin bound).  The FP64 factor places them in FP32
// first and confirms and refines that bracket in FP64.
// ---------------------------------------------------------------------------
constexpr int kEigThreads = 128;
template <typename T>
__host__ __device__ inline int eig_lanes(int m) { return sizeof(T) == 8 || m < 128 ? 8 : 32; }

template <typename T>
__host__ __device__ inline size_t eigval_smem_bytes(int m) {
  return 2 * sizeof(float) * (size_t)m + (sizeof(T) == 8 ? 2 * sizeof(double) * (size_t)m : 0) + 16;
}

template <typename Task>
__device__ __forceinline__ int task_of(const Task *tasks, int ntasks, int b) {
  int lo = 0, hi = ntasks - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tasks[mid].blk0 <= b)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

template <typename T, int LN>
__device__ void eigvals(const EigTask<T> &t, int first, const double *d, const double *e2, const float *df,
                        const float *e2f) {
  const int m = t.m, k2 = t.sc[1];
  const int lane = threadIdx.x & 31;
  const int jj = first + (int)threadIdx.x / LN;
  const int j = min(jj, k2 - 1);
  const double thr = t.sb[0], hi0 = t.sb[1], emax = t.sb[2], tnorm = *t.tnorm;
  const float pivf = sturm_pivmin((float)emax);
  float lo = (float)thr, hi = (float)hi0;
  const float tol = 4.f * unit_round<float>() * (float)tnorm;
  for (int round = 0; round < 12 && __any_sync(0xffffffffu, hi - lo > tol); ++round)
    section<float, LN>(lo, hi, lane, false,
                       [&](float s) { return count_above<float>(df, e2f, m, s, pivf) > j; });
  if constexpr (sizeof(T) == 4) {
    if (jj < k2 && lane % LN == 0) t.lam[jj] = 0.5f * (lo + hi);
  } else {
    const double piv = sturm_pivmin(emax);
    auto above = [&](double s) { return count_above<double>(d, e2, m, s, piv) > j; };
    const double mid = 0.5 * ((double)lo + (double)hi), w = 64.0 * 1.2e-7 * tnorm;
    double l = mid - w, h = mid + w;
    const int miss = section<double, LN>(l, h, lane, true, above);
    if (miss != 0) {
      l = miss == 1 ? mid + w : fmin(thr, mid - 2.0 * w);
      h = miss == -1 ? mid - w : hi0;
    }
    const double told = 4.0 * unit_round<double>() * tnorm;
    for (int round = 0; round < 40 && __any_sync(0xffffffffu, h - l > told); ++round)
      section<double, LN>(l, h, lane, false, above);
    if (jj < k2 && lane % LN == 0) t.lam[jj] = 0.5 * (l + h);
  }
}

template <typename T>
__global__ void __launch_bounds__(kEigThreads) k_eigval(const EigTask<T> *__restrict__ tasks, int ntasks) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const EigTask<T> t = tasks[task_of(tasks, ntasks, blockIdx.x)];
  const int m = t.m;
  const int lanes = eig_lanes<T>(m);
  const int first = (blockIdx.x - t.blk0) * (kEigThreads / lanes);
  if (first >= t.sc[1]) return;
  double *d = (double *)smem_raw, *e2 = d + m;
  float *df = sizeof(T) == 8 ? (float *)(e2 + m) : (float *)smem_raw;
  float *e2f = df + m;
  for (int i = threadIdx.x; i < m; i += kEigThreads) {
    const T di = t.dt[i], ei = i > 0 ? t.et[i - 1] : T(0);
    df[i] = (float)di;
    e2f[i] = (float)ei * (float)ei;
    if (sizeof(T) == 8) {
      d[i] = (double)di;
      e2[i] = (double)ei * (double)ei;
    }
  }
  __syncthreads();
  if (lanes == 8)
    eigvals<T, 8>(t, first, d, e2, df, e2f);
  else
    eigvals<T, 32>(t, first, d, e2, df, e2f);
}

// ---------------------------------------------------------------------------
// Inverse iteration for the selected eigenvalues, one lane each: LU of
// T - lam I with partial pivoting (rows i, i+1 interchanged when the
// sub-diagonal dominates), three solves from a fixed pseudo-random start,
// modified Gram-Schmidt against the vectors already found of the same cluster
// of eigenvalues closer than 10 u ||T|| (those could come out nearly
// parallel; the lane of a cluster's first eigenvalue takes them all in turn, and
// the warp orthogonalises together).
// Only the span of the selected vectors matters and the host
// re-orthonormalises them, which tolerates the overlap u ||T|| / gap that
// inverse iteration leaves between vectors of distinct eigenvalues.
// One warp per CTA; a lane's LU (pivots, two super-diagonals,
// multipliers), vector and interchange flags sit in shared memory, element i
// of lane s at i * st + s with st odd, so that neither the lanes' sweeps nor
// the write-out of whole vectors conflict.  A sweep carries its two last
// values in registers: one fused multiply-add (forward) or two and a quotient
// (backward) per row on the dependent chain.
// ---------------------------------------------------------------------------
template <typename T>
__host__ __device__ inline size_t invit_smem_bytes(int m, int slots, bool with_t) {
  return ((5 * sizeof(T) + 1) * (size_t)(slots | 1) + (with_t ? 2 * sizeof(T) : 0)) * (size_t)m + 16;
}

template <typename T>
__global__ void __launch_bounds__(32) k_invit(const EigTask<T> *__restrict__ tasks, int ntasks, int spc,
                                              int with_t) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const EigTask<T> t = tasks[task_of(tasks, ntasks, blockIdx.x)];
  const int m = t.m, k2 = t.sc[1];
  const int lane = threadIdx.x;
  const int q0 = (blockIdx.x - t.blk0) * spc;
  if (q0 >= k2) return;
  const int st = spc | 1;
  const size_t sm = (size_t)m * st;
  T *u0 = (T *)smem_raw + (with_t ? 2 * (size_t)m : 0), *u1 = u0 + sm, *u2 = u1 + sm, *lm = u2 + sm, *y = lm + sm;
  unsigned char *fl = (unsigned char *)(y + sm);
  const T *dt = t.dt, *et = t.et;   // staged when they fit beside the slots
  if (with_t) {
    T *ds = (T *)smem_raw, *es = ds + m;
    for (int i = lane; i < m; i += 32) {
      ds[i] = t.dt[i];
      es[i] = t.et[i];
    }
    dt = ds;
    et = es;
  }
  __syncwarp();
  const T tnorm = (T)*t.tnorm;
  const T ortol = T(10) * unit_round<T>() * tnorm;
  const T small = unit_round<T>() * tnorm + T(sizeof(T) == 8 ? 1e-290 : 1e-30);
  const int q = q0 + lane;
  // lane of a cluster's first eigenvalue: vectors q .. q + nrun - 1
  int nrun = 0;
  if (lane < spc && q < k2 && (q == 0 || t.lam[q - 1] - t.lam[q] >= ortol)) {
    nrun = 1;
    while (q + nrun < k2 && t.lam[q + nrun - 1] - t.lam[q + nrun] < ortol) ++nrun;
  }
  for (int run = 0; __any_sync(0xffffffffu, run < nrun); ++run) {
    const bool on = run < nrun;
    if (on) {
      const T lam = t.lam[q + run];
      const uint32_t seed = (uint32_t)((q + run) * 7919 + 17);
      T a = dt[0] - lam, c = m > 1 ? et[0] : T(0);
      for (int i = 0; i + 1 < m; ++i) {
        const T b = et[i];
        const T an = dt[i + 1] - lam;
        const T cn = i + 2 < m ? et[i + 1] : T(0);
        const size_t o = (size_t)i * st + lane;
        const bool swap = fabs(a) < fabs(b);
        T piv = swap ? b : (a == T(0) ? small : a);
        const T mult = (swap ? a : b) / piv;
        u0[o] = fabs(piv) < small ? copysign(small, piv) : piv;
        u1[o] = swap ? an : c;
        u2[o] = swap ? cn : T(0);
        lm[o] = mult;
        fl[o] = swap;
        const T na = swap ? c - mult * an : an - mult * c;
        c = swap ? -mult * cn : cn;
        a = na;
      }
      u0[(size_t)(m - 1) * st + lane] = fabs(a) < small ? copysign(small, a) : a;
      for (int i = 0; i < m; ++i) y[(size_t)i * st + lane] = (T)hash_unit(seed, (uint32_t)i);
    }
    T scale = T(1);
    for (int it = 0; it < 3; ++it) {
      T big = T(0);
      if (on) {
        T cur = y[lane] * scale;
#pragma unroll 4
        for (int i = 0; i + 1 < m; ++i) {
          const size_t o = (size_t)i * st + lane;
          const T yn = y[o + st] * scale;
          const T l = lm[o];
          const bool swap = fl[o];
          y[o] = swap ? yn : cur;
          cur = swap ? fma(-l, yn, cur) : fma(-l, cur, yn);
        }
        T y1 = cur / u0[(size_t)(m - 1) * st + lane], y2 = T(0);
        y[(size_t)(m - 1) * st + lane] = y1;
        big = fabs(y1);
#pragma unroll 4
        for (int i = m - 2; i >= 0; --i) {
          const size_t o = (size_t)i * st + lane;
          const T s = fma(-u1[o], y1, fma(-u2[o], y2, y[o])) / u0[o];
          y[o] = s;
          y2 = y1;
          y1 = s;
          big = fmax(big, fabs(s));
        }
      }
      if (run > 0) {
        // the whole warp orthogonalises one lane's vector after another
        // against the cluster's vectors so far (a lane alone walks both with
        // uncoalesced loads: most of the kernel's time at m = 1340)
        __syncwarp();
        for (int s = 0; s < spc; ++s) {
          if (!__shfl_sync(0xffffffffu, (int)on, s)) continue;
          const T *prev = t.Y + (size_t)(q0 + s) * m;
          for (int pass = 0; pass < 2; ++pass)
            for (int p = 0; p < run; ++p) {
              const T *v = prev + (size_t)p * m;
              T dot = T(0);
              for (int i = lane; i < m; i += 32) dot = fma(v[i], y[(size_t)i * st + s], dot);
              for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
              for (int i = lane; i < m; i += 32) y[(size_t)i * st + s] = fma(-dot, v[i], y[(size_t)i * st + s]);
            }
          T bg = T(0);
          for (int i = lane; i < m; i += 32) bg = fmax(bg, fabs(y[(size_t)i * st + s]));
          for (int o = 16; o > 0; o >>= 1) bg = fmax(bg, __shfl_xor_sync(0xffffffffu, bg, o));
          if (lane == s) big = bg;
        }
        __syncwarp();
      }
      if (on) {
        // norm, scaling by the largest entry first to keep the sum in range;
        // the next sweep applies the factor as it reads
        const T sc = big > T(0) ? T(1) / big : T(0);
        T n0 = T(0), n1 = T(0);
#pragma unroll 2
        for (int i = 0; i + 1 < m; i += 2) {
          const T v0 = y[(size_t)i * st + lane] * sc, v1 = y[(size_t)(i + 1) * st + lane] * sc;
          n0 = fma(v0, v0, n0);
          n1 = fma(v1, v1, n1);
        }
        if (m & 1) {
          const T v0 = y[(size_t)(m - 1) * st + lane] * sc;
          n0 = fma(v0, v0, n0);
        }
        const T nrm = sqrt(n0 + n1);
        scale = nrm > T(0) ? sc / nrm : T(0);
      }
    }
    if (on)
      for (int i = 0; i < m; ++i) y[(size_t)i * st + lane] *= scale;
    __syncwarp();
    // whole vectors, consecutive lanes on consecutive entries
    for (int s = 0; s < spc; ++s) {
      if (!__shfl_sync(0xffffffffu, (int)on, s)) continue;
      T *out = t.Y + (size_t)(q0 + s + run) * m;
      for (int i = lane; i < m; i += 32) out[i] = y[(size_t)i * st + s];
    }
    __syncwarp();   // the vectors are read back by the next of a cluster
  }
}

// ---------------------------------------------------------------------------
// Products with Q = H_0 ... H_{m-3} (I - tau_k v_k v_k^T, v_k = 1 at row k + 1,
// its tail in row k of A): forward (Z = Q^T X, in place) or backward (U_2 = Q Y,
// into U's columns from k1 on).  A warp keeps its columns in registers (row
// lane + 32 e in register e, e < E) and applies the reflectors one after the
// other: products over the rows above, one warp sum for all its columns, one
// update, no barrier; the next reflector's row is loaded meanwhile.  Four warps
// per CTA.  A node's E, columns per warp and sums depend on m alone.
// (One CTA per 16 columns with block sums took three barriers a reflector.)
// ---------------------------------------------------------------------------
constexpr int kQmWarps = 4;
// (E = 48, 64: FP32 only, whose three rows of E registers fit; a CTA per 16
// columns with block sums, which FP64 keeps there, took 3.2 ms for the four
// largest nodes of a 40^3 grid, m = 1340)
__host__ __device__ inline int qmul_e(int m) {
  return m <= 64 ? 2 : m <= 128 ? 4 : m <= 256 ? 8 : m <= 512 ? 16 : m <= 1024 ? 32 : m <= 1536 ? 48 : 64;
}
template <typename T>
__host__ __device__ constexpr int qmul_cols(int E) {
  return sizeof(T) == 4 ? (E <= 8 ? 4 : E == 16 ? 2 : 1) : (E <= 4 ? 4 : E == 8 ? 2 : 1);
}

template <typename T, int E, int C>
__device__ void qmul_warp(const QmulTask<T> &t, int j0, int nc, T *stage, int sld) {
  const int m = t.m, lane = threadIdx.x & 31;
  T yv[C][E];
#pragma unroll
  for (int c = 0; c < C; ++c)
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int i = lane + 32 * e;
      yv[c][e] = i < m && c < nc ? t.cols[(size_t)(j0 + c) * m + i] : T(0);
    }
  const int steps = m - 2;
  auto load = [&](int s, T (&v)[E], T &tau) {
    const int k = t.fwd ? s : m - 3 - s;
    tau = t.tau[k];
    const T *row = t.A + (size_t)k * m;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int i = lane + 32 * e;
      v[e] = i > k + 1 && i < m ? __ldg(row + i) : (i == k + 1 ? T(1) : T(0));
    }
  };
  T v[E], tau;
  if (steps > 0) load(0, v, tau);
  for (int s = 0; s < steps; ++s) {
    T vn[E], taun = T(0);
    if (s + 1 < steps) load(s + 1, vn, taun);
    T dot[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
      dot[c] = T(0);
#pragma unroll
      for (int e = 0; e < E; ++e) dot[c] = fma(v[e], yv[c][e], dot[c]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int c = 0; c < C; ++c) dot[c] += __shfl_xor_sync(0xffffffffu, dot[c], o);
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const T f = tau * dot[c];
#pragma unroll
      for (int e = 0; e < E; ++e) yv[c][e] = fma(-f, v[e], yv[c][e]);
    }
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = vn[e];
    tau = taun;
  }
  if (t.fwd) {
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int i = lane + 32 * e;
        if (i < m && c < nc) t.cols[(size_t)(j0 + c) * m + i] = yv[c][e];
      }
  } else {
    // through shared memory: U's rows take the CTA's adjacent columns together
    const int c0 = (threadIdx.x >> 5) * C;
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int i = lane + 32 * e;
        if (i < m && c < nc) stage[(size_t)i * sld + c0 + c] = yv[c][e];
      }
  }
}

// EM: the largest E of the launch (its registers); a node runs its own E
template <typename T, int EM>
__global__ void __launch_bounds__(kQmWarps * 32) k_qmul(const QmulTask<T> *__restrict__ tasks, int ntasks) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const QmulTask<T> t = tasks[task_of(tasks, ntasks, blockIdx.x)];
  const int m = t.m, E = qmul_e(m);
  const int k1 = t.sc[0];
  const int ncol = t.fwd ? k1 : t.sc[1];
  const int C = qmul_cols<T>(E);
  const int per = kQmWarps * C;
  const int jc = (blockIdx.x - t.blk0) * per;   // the CTA's first column
  if (jc >= ncol) return;
  T *stage = (T *)smem_raw;
  const int sld = per + 1;
  const int j0 = jc + (threadIdx.x >> 5) * C;
  const int nc = min(C, ncol - j0);
  if (nc > 0) {
    if (E == 2)
      qmul_warp<T, 2, qmul_cols<T>(2)>(t, j0, nc, stage, sld);
    if constexpr (EM >= 4)
      if (E == 4) qmul_warp<T, 4, qmul_cols<T>(4)>(t, j0, nc, stage, sld);
    if constexpr (EM >= 8)
      if (E == 8) qmul_warp<T, 8, qmul_cols<T>(8)>(t, j0, nc, stage, sld);
    if constexpr (EM >= 16)
      if (E == 16) qmul_warp<T, 16, qmul_cols<T>(16)>(t, j0, nc, stage, sld);
    if constexpr (EM >= 32)
      if (E == 32) qmul_warp<T, 32, qmul_cols<T>(32)>(t, j0, nc, stage, sld);
    if constexpr (EM >= 48)
      if (E == 48) qmul_warp<T, 48, qmul_cols<T>(48)>(t, j0, nc, stage, sld);
    if constexpr (EM >= 64)
      if (E == 64) qmul_warp<T, 64, qmul_cols<T>(64)>(t, j0, nc, stage, sld);
  }
  if (t.fwd) return;
  __syncthreads();
  const int w = min(per, ncol - jc);
  for (int q = threadIdx.x; q < m * w; q += kQmWarps * 32) {
    const int i = q / w, c = q % w;
    t.U[(int64_t)i * m + k1 + jc + c] = stage[(size_t)i * sld + c];
  }
}

// ---------------------------------------------------------------------------
// Multi-CTA tridiagonalisation of very large nodes.  One CTA per node cannot
// use more than one SM, and its traffic grows as m^3: here each step is spread
// over ceil(m / kTriRows) CTAs per node, one warp per row.  Step k:
//   phase 0 (k_tri_update): rows i >= k get the rank-2 update of step k - 1,
//     A_ij -= v_i w_j + w_i v_j (w = p - K v, K = tau p.v / 2 from the CTAs'
//     partials in block order); then x_i = A_ik for i > k and d_k = A_kk, with
//     per-CTA partials of |x|^2 beyond x's first entry.
//   phase 1 (k_tri_symv): every CTA forms the reflector of x from the partials
//     (same arithmetic in every CTA), v_i for its rows, p_i = tau sum_j A_ij v_j,
//     and per-CTA partials of p.v; v is also kept in row k of A for the later
//     products with Q (as the one-CTA path stores it).
// Reductions run in a fixed order, so results do not depend on scheduling.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ int tri_task(const GridTri<T> *tasks, int ntasks, int b) {
  int lo = 0, hi = ntasks - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tasks[mid].blk0 <= b)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

// fixed-order sum of n partials by one warp (every lane gets it)
template <typename T>
__device__ __forceinline__ T warp_sum_parts(const T *part, int n, int lane) {
  T s = T(0);
  for (int c = lane; c < n; c += 32) s += part[c];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

template <typename T>
__global__ void __launch_bounds__(kTriRows * 32) k_tri_update(const GridTri<T> *__restrict__ tasks, int ntasks,
                                                               int k) {
  __shared__ T sK;
  __shared__ T wpart[kTriRows];
  const GridTri<T> t = tasks[tri_task(tasks, ntasks, blockIdx.x)];
  const int m = t.m;
  if (k > t.kend) return;
  const int rb = blockIdx.x - t.blk0;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = rb * kTriRows + warp;
  if (k >= 1) {
    if (warp == 0) {
      const T s = warp_sum_parts<T>(t.ppv, t.nblk, lane);
      if (lane == 0) sK = T(0.5) * t.tau[k - 1] * s;
    }
    __syncthreads();
  }
  T part = T(0);
  if (i >= k && i < m) {
    T *row = t.A + (int64_t)i * m;
    if (k >= 1) {
      const T K = sK;
      const T vi = t.V[i];
      const T wi = fma(-K, vi, t.P[i]);
      const T *V = t.V, *P = t.P;
      auto upd = [&](T a, int j) {
        const T vj = V[j];
        return fma(-vi, fma(-K, vj, P[j]), fma(-wi, vj, a));
      };
      // four independent row elements in flight per lane (the step is a
      // stream over the trailing rows)
      int j = k + lane;
      for (; j + 96 < m; j += 128) {
        const T a0 = row[j], a1 = row[j + 32], a2 = row[j + 64], a3 = row[j + 96];
        row[j] = upd(a0, j);
        row[j + 32] = upd(a1, j + 32);
        row[j + 64] = upd(a2, j + 64);
        row[j + 96] = upd(a3, j + 96);
      }
      for (; j < m; j += 32) row[j] = upd(row[j], j);
      __syncwarp();
    }
    if (k <= m - 3 && lane == 0) {
      const T x = row[k];
      if (i == k) {
        t.d[k] = (double)x;
      } else {
        t.X[i] = x;
        if (i > k + 1) part = x * x;
      }
    }
  }
  if (lane == 0) wpart[warp] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    T s = T(0);
    for (int w = 0; w < kTriRows; ++w) s += wpart[w];
    t.px[rb] = s;
  }
}

template <typename T>
__global__ void __launch_bounds__(kTriRows * 32) k_tri_symv(const GridTri<T> *__restrict__ tasks, int ntasks,
                                                             int k) {
  __shared__ double s_scale, s_tau;
  __shared__ T wpart[kTriRows];
  const GridTri<T> t = tasks[tri_task(tasks, ntasks, blockIdx.x)];
  const int m = t.m;
  if (k >= t.kend) return;
  const int rb = blockIdx.x - t.blk0;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == 0) {
    // the reflector of x = A[k+1.., k] (as in the cluster tridiagonalisation)
    const double tail2 = (double)warp_sum_parts<T>(t.px, t.nblk, lane);
    if (lane == 0) {
      const double alpha = (double)t.X[k + 1];
      double tau = 0.0, beta = alpha, scale = 0.0;
      if (tail2 > (sizeof(T) == 8 ? 1e-290 : 1e-30)) {   // (as in reflector.h)
        beta = -copysign(sqrt(fma(alpha, alpha, tail2)), alpha);
        tau = (beta - alpha) / beta;
        scale = 1.0 / (alpha - beta);
      }
      s_scale = scale;
      s_tau = tau;
      if (rb == 0) {
        t.e[k] = beta;
        t.tau[k] = (T)tau;
      }
    }
  }
  __syncthreads();
  const T scale_t = (T)s_scale, tau_t = (T)s_tau;
  const int i = rb * kTriRows + warp;
  T pv = T(0);
  if (i >= k + 1 && i < m) {
    const T vi = (i == k + 1) ? T(1) : t.X[i] * scale_t;
    T p = T(0);
    if (s_tau != 0.0) {
      const T *row = t.A + (int64_t)i * m;
      const T *X = t.X;
      auto vj = [&](int j) { return j == k + 1 ? T(1) : X[j] * scale_t; };
      T a0 = T(0), a1 = T(0), a2 = T(0), a3 = T(0);
      int j = k + 1 + lane;
      for (; j + 96 < m; j += 128) {
        a0 = fma(row[j], vj(j), a0);
        a1 = fma(row[j + 32], vj(j + 32), a1);
        a2 = fma(row[j + 64], vj(j + 64), a2);
        a3 = fma(row[j + 96], vj(j + 96), a3);
      }
      for (; j < m; j += 32) a0 = fma(row[j], vj(j), a0);
      T acc = (a0 + a1) + (a2 + a3);
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      p = tau_t * acc;
    }
    if (lane == 0) {
      t.V[i] = vi;
      t.P[i] = p;
      pv = p * vi;
      if (i >= k + 2) t.A[(int64_t)k * m + i] = vi;   // reflector k kept in row k
    }
  }
  if (lane == 0) wpart[warp] = pv;
  __syncthreads();
  if (threadIdx.x == 0) {
    T s = T(0);
    for (int w = 0; w < kTriRows; ++w) s += wpart[w];
    t.ppv[rb] = s;
  }
}

// The same products for nodes too large for a warp's registers (m > kQmulMax), one CTA
// per batch of columns held in shared memory: for each reflector the block forms all the batch's dot
// products (fixed-order reduction), then updates the columns.
constexpr int RT = 256;
constexpr int RNB = 16;   // most columns per task

template <typename T>
__global__ void __launch_bounds__(RT) k_refl(const ReflTask<T> *__restrict__ tasks, int nb) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ T red[RT / 32][RNB];
  __shared__ T tot[RNB];
  const ReflTask<T> t = tasks[blockIdx.x];
  const int m = t.m;
  const int k1 = t.sc[0];
  const int ncol = t.fwd ? k1 : t.sc[1];
  if (t.j0 >= ncol) return;
  const int nc = min(nb, ncol - t.j0);
  T *Ys = (T *)smem_raw;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int64_t q = tid; q < (int64_t)nc * m; q += RT) Ys[q] = t.cols[(size_t)t.j0 * m + q];
  __syncthreads();
  for (int kk = 0; kk + 2 < m; ++kk) {
    const int k = t.fwd ? kk : m - 3 - kk;
    const T tk = t.tau[k];
    if (tk == T(0)) continue;
    const int n1 = m - k - 1;
    const T *vrow = t.A + (int64_t)k * m + k + 1;   // v[0] = 1 implicit
    T s[RNB];
#pragma unroll
    for (int c = 0; c < RNB; ++c) s[c] = T(0);
    for (int i = tid; i < n1; i += RT) {
      const T vi = i == 0 ? T(1) : vrow[i];
#pragma unroll
      for (int c = 0; c < RNB; ++c)
        if (c < nc) s[c] = fma(vi, Ys[(size_t)c * m + k + 1 + i], s[c]);
    }
#pragma unroll
    for (int c = 0; c < RNB; ++c) {
      T x = s[c];
      for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      if (lane == 0) red[warp][c] = x;
    }
    __syncthreads();
    if (tid < nc) {
      T x = T(0);
      for (int w = 0; w < RT / 32; ++w) x += red[w][tid];
      tot[tid] = tk * x;
    }
    __syncthreads();
    for (int i = tid; i < n1; i += RT) {
      const T vi = i == 0 ? T(1) : vrow[i];
      for (int c = 0; c < nc; ++c) Ys[(size_t)c * m + k + 1 + i] -= tot[c] * vi;
    }
    __syncthreads();
  }
  if (t.fwd) {
    for (int64_t q = tid; q < (int64_t)nc * m; q += RT) t.cols[(size_t)t.j0 * m + q] = Ys[q];
  } else {
    for (int64_t q = tid; q < (int64_t)m * nc; q += RT) {
      const int i = (int)(q / nc), c = (int)(q % nc);
      t.U[(int64_t)i * m + k1 + t.j0 + c] = Ys[(size_t)c * m + i];
    }
  }
}

}  // namespace

template <typename T>
size_t trunc_big_work_elems(int m) {
  // A, Y (2 m^2 T), LS (32 m T), the vectors and SC
  const size_t bytes = sizeof(T) * (2 * (size_t)m * m + 32 * (size_t)m) + 16 + big_vec_bytes<T>(m) + 16 + kBigScBytes + 64;
  return (bytes + sizeof(T) - 1) / sizeof(T);
}

// 256 threads per node up to m = 256, 1024 above (a function of m alone)
template <typename T>
void launch_trunc_prep(const TruncTask<T> *d_tasks, int ntasks, int *d_k, int variant, int max_m, cudaStream_t st) {
  if (ntasks == 0) return;
  if (max_m <= kTruncPrepMid)
    k_trunc_prep<T, 256><<<ntasks, 256, 0, st>>>(d_tasks, d_k, variant);
  else
    k_trunc_prep<T, 1024><<<ntasks, 1024, 0, st>>>(d_tasks, d_k, variant);
  count_launch();
  HS_CUDA(cudaGetLastError());
}

template <typename T>
size_t rank_bytes(int m, int np, int variant) {
  return rank_place<T>(m, np, variant != HS_LORASP, (size_t)allow_max_dynamic_smem<&k_rank<T>>()).bytes;
}

template <typename T>
void launch_rank(const TruncTask<T> *d_tasks, int ntasks, int *d_k, int variant, size_t bytes, cudaStream_t st) {
  if (ntasks == 0) return;
  const size_t limit = (size_t)allow_max_dynamic_smem<&k_rank<T>>();
  k_rank<T><<<ntasks, kRankThreads, bytes, st>>>(d_tasks, d_k, variant, limit);
  count_launch();
  HS_CUDA(cudaGetLastError());
}

template <typename T>
int eigval_blocks(int m) {
  const int per = kEigThreads / eig_lanes<T>(m);
  return (m + per - 1) / per;
}

template <typename T>
void launch_eigval(const EigTask<T> *d_tasks, int ntasks, int total_blocks, int m_max, cudaStream_t st) {
  if (ntasks == 0 || total_blocks == 0) return;
  const size_t sm = eigval_smem_bytes<T>(m_max);
  check_dynamic_smem(sm, allow_max_dynamic_smem<&k_eigval<T>>(), "k_eigval");
  k_eigval<T><<<total_blocks, kEigThreads, sm, st>>>(d_tasks, ntasks);
  count_launch();
  HS_CUDA(cudaGetLastError());
}

template <typename T>
int invit_slots(int m) {
  const size_t budget = 200 * 1024;
  int spc = 32;
  while (spc > 1 && invit_smem_bytes<T>(std::max(m, 1), spc, true) > budget) --spc;
  return spc;
}

template <typename T>
void launch_invit(const EigTask<T> *d_tasks, int ntasks, int total_blocks, int spc, int m_max, cudaStream_t st) {
  if (ntasks == 0 || total_blocks == 0) return;
  const int limit = allow_max_dynamic_smem<&k_invit<T>>();
  const bool with_t = invit_smem_bytes<T>(m_max, spc, true) <= (size_t)limit;
  const size_t sm = invit_smem_bytes<T>(m_max, spc, with_t);
  check_dynamic_smem(sm, limit, "k_invit");
  k_invit<T><<<total_blocks, 32, sm, st>>>(d_tasks, ntasks, spc, with_t ? 1 : 0);
  count_launch();
  HS_CUDA(cudaGetLastError());
}

template <typename T>
int qmul_blocks(int m, int ncol) {
  const int per = kQmWarps * qmul_cols<T>(qmul_e(m));
  return (ncol + per - 1) / per;
}

template <typename T, int EM>
static void launch_qmul_e(const QmulTask<T> *d_tasks, int ntasks, int total_blocks, size_t sm, cudaStream_t st) {
  check_dynamic_smem(sm, allow_max_dynamic_smem<&k_qmul<T, EM>>(), "k_qmul");
  k_qmul<T, EM><<<total_blocks, kQmWarps * 32, sm, st>>>(d_tasks, ntasks);
}

template <typename T>
void launch_qmul(const QmulTask<T> *d_tasks, int ntasks, int total_blocks, int m_max, bool fwd, cudaStream_t st) {
  if (ntasks == 0 || total_blocks == 0) return;
  const int E = qmul_e(m_max);
  // the staged columns: the larger of m (4 C(E) + 1) over the classes up to E
  size_t sm = 0;
  if (!fwd)
    for (int e : {2, 4, 8, 16, 32, 48, 64})
      if (e <= E) sm = std::max(sm, sizeof(T) * (size_t)std::min(m_max, 32 * e) * (kQmWarps * qmul_cols<T>(e) + 1));
  switch (E) {
    case 2: launch_qmul_e<T, 2>(d_tasks, ntasks, total_blocks, sm, st); break;
    case 4: launch_qmul_e<T, 4>(d_tasks, ntasks, total_blocks, sm, st); break;
    case 8: launch_qmul_e<T, 8>(d_tasks, ntasks, total_blocks, sm, st); break;
    case 16: launch_qmul_e<T, 16>(d_tasks, ntasks, total_blocks, sm, st); break;
    case 32: launch_qmul_e<T, 32>(d_tasks, ntasks, total_blocks, sm, st); break;
    default:
      if constexpr (sizeof(T) == 4) {
        if (E == 48) launch_qmul_e<T, 48>(d_tasks, ntasks, total_blocks, sm, st);
        else launch_qmul_e<T, 64>(d_tasks, ntasks, total_blocks, sm, st);
      } else {
        fail(HS_ERR_INVALID, "internal: size of the products with Q");
      }
  }
  count_launch();
  HS_CUDA(cudaGetLastError());
}

template <typename T>
void launch_tri_step(const GridTri<T> *d_tasks, int ntasks, int total_blocks, int k, int phase, cudaStream_t st) {
  if (ntasks == 0 || total_blocks == 0) return;
  if (phase == 0)
    k_tri_update<T><<<total_blocks, kTriRows * 32, 0, st>>>(d_tasks, ntasks, k);
  else
    k_tri_symv<T><<<total_blocks, kTriRows * 32, 0, st>>>(d_tasks, ntasks, k);
  count_launch();
  HS_CUDA(cudaGetLastError());
}

template <typename T>
int refl_batch(int m) {
  const size_t budget = 200 * 1024;
  const int nb = (int)(budget / (sizeof(T) * (size_t)std::max(m, 1)));
  return std::max(1, std::min(nb, RNB));
}

template <typename T>
void launch_refl(const ReflTask<T> *d_tasks, int ntasks, int nb, int m_max, cudaStream_t st) {
  if (ntasks == 0) return;
  const size_t sm = sizeof(T) * (size_t)nb * m_max;
  check_dynamic_smem(sm, allow_max_dynamic_smem<&k_refl<T>>(), "k_refl");
  k_refl<T><<<ntasks, RT, sm, st>>>(d_tasks, nb);
  count_launch();
  HS_CUDA(cudaGetLastError());
}


#define HS_INST(T)                                                                                             \
  template void launch_trunc_prep<T>(const TruncTask<T> *, int, int *, int, int, cudaStream_t);                \
  template size_t rank_bytes<T>(int, int, int);                                                                \
  template void launch_rank<T>(const TruncTask<T> *, int, int *, int, size_t, cudaStream_t);                   \
  template int eigval_blocks<T>(int);                                                                          \
  template void launch_eigval<T>(const EigTask<T> *, int, int, int, cudaStream_t);                             \
  template int invit_slots<T>(int);                                                                            \
  template void launch_invit<T>(const EigTask<T> *, int, int, int, int, cudaStream_t);                         \
  template int qmul_blocks<T>(int, int);                                                                       \
  template void launch_qmul<T>(const QmulTask<T> *, int, int, int, bool, cudaStream_t);                        \
  template void launch_tri_step<T>(const GridTri<T> *, int, int, int, int, cudaStream_t);                      \
  template int refl_batch<T>(int);                                                                             \
  template void launch_refl<T>(const ReflTask<T> *, int, int, int, cudaStream_t);                              \
  template size_t trunc_big_work_elems<T>(int);
HS_INST(double)
HS_INST(float)
#undef HS_INST

}  // namespace hs
