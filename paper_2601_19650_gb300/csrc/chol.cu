// FP64 Cholesky factorisation and lower-triangular solve for CholeskyQR2.
//
// The backward sweep decomposes S^[i] = R Q^[i] on the leg chi_{i-1} (Eq.
// (tt_cbc_qr_decomp); Eq. (cbc_tree_qr) on trees).  With S of m rows and n >= m columns
// the GPU path forms G = S S^H, factors G = C C^H, and solves Q = C^{-1} S; doing it
// twice (CholeskyQR2) restores orthonormality to FP64 round-off.
//
// Cholesky: one thread-block cluster per matrix with the rows in shared memory
// (chol_cluster_kernel), a CTA per matrix for larger batches (chol1_kernel); for matrices
// that no cluster holds, a group of CTAs that wait on each other works in 32-wide column
// blocks on global memory (chol_kernel): per block, CTA 0 factors the diagonal block in shared
// memory, every other row of the panel is solved by one warp (shuffles carry the solved
// entries), and the trailing lower triangle is updated from a shared-memory copy of the panel;
// bounded grid barriers separate the phases.
// Triangular solve: where there is enough of it, by matrix products with inverted diagonal
// blocks (trsm_products); else columns of S are independent, so each warp owns one column and
// runs the forward substitution in 32-row groups without any inter-CTA synchronisation.
// Divisions use Newton reciprocals (rcp64): long dependent chains of FP64 divisions are
// slow on this part.
#include <cooperative_groups.h>

#include <algorithm>

#include "df.cuh"
#include "kernels.cuh"
#include "planner.h"

namespace cbc {
namespace {

constexpr int NB = 32, TPB = 256;

template <typename T>
__device__ __forceinline__ T ldg_cg(const T* p);
template <>
__device__ __forceinline__ double ldg_cg<double>(const double* p) { return __ldcg(p); }
template <>
__device__ __forceinline__ zdbl ldg_cg<zdbl>(const zdbl* p) {
  double2 v = __ldcg(reinterpret_cast<const double2*>(p));
  return {v.x, v.y};
}

template <typename T>
__device__ __forceinline__ T shfl(T v, int src);
template <>
__device__ __forceinline__ double shfl<double>(double v, int src) {
  return __shfl_sync(0xffffffffu, v, src);
}
template <>
__device__ __forceinline__ zdbl shfl<zdbl>(zdbl v, int src) {
  return {__shfl_sync(0xffffffffu, v.re, src), __shfl_sync(0xffffffffu, v.im, src)};
}

template <typename T>
struct CholArgs {
  T* G;
  int m;
  int* status;
  GridBarrier* bar;
  int P;  // CTAs per matrix; CTA b works on matrix b / P (G + (b / P) m^2, bar + b / P)
};

// G (row-major m x m, Hermitian, lower triangle read) -> C (lower triangle), G = C C^H
// PSMEM: the panel of the trailing update is copied to shared memory (m up to ~440
// complex); else the update reads it from global memory (L2).
template <typename T, bool PSMEM>
__global__ void __launch_bounds__(TPB) chol_kernel(CholArgs<T> a) {
  using O = ops<T>;
  extern __shared__ unsigned char sm_raw[];
  T* pan = reinterpret_cast<T*>(sm_raw);  // panel rows [b0, m) x NB, or the diag block
  __shared__ double s_rd[NB];             // reciprocals of the diagonal of the block
  __shared__ int s_bad;
  const int m = a.m, P = a.P, cta = blockIdx.x % P;
  a.G += (int64_t)(blockIdx.x / P) * m * m;
  a.bar += blockIdx.x / P;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int b0 = 0; b0 < m; b0 += NB) {
    const int nb = min(NB, m - b0);
    // (1) diagonal block on CTA 0
    if (cta == 0) {
      T* blk = pan;  // nb x NB
      for (int t = threadIdx.x; t < nb * NB; t += blockDim.x) {
        int i = t / NB, l = t % NB;
        blk[t] = (l <= i && l < nb) ? ldg_cg(a.G + (int64_t)(b0 + i) * m + b0 + l) : O::zero();
      }
      if (threadIdx.x == 0) s_bad = 0;
      __syncthreads();
      for (int jj = 0; jj < nb; ++jj) {
        const double piv = O::real(blk[jj * NB + jj]);
        if (!(piv > 0.0) || !isfinite(piv)) {
          if (threadIdx.x == 0) s_bad = 1;
          break;
        }
        const double rc = rsqrt64(piv);  // 1 / sqrt(piv)
        const double rp = rc * rc;        // 1 / piv
        // trailing update with the unscaled column (divide by piv), then scale column
        for (int t = threadIdx.x; t < nb * nb; t += blockDim.x) {
          int i = t / nb, l = t % nb;
          if (i > jj && l > jj && l <= i)
            blk[i * NB + l] = blk[i * NB + l] -
                              O::scale(rp, blk[i * NB + jj] * O::conj(blk[l * NB + jj]));
        }
        __syncthreads();
        for (int i = jj + threadIdx.x; i < nb; i += blockDim.x)
          blk[i * NB + jj] = (i == jj) ? O::make(piv * rc, 0.0) : O::scale(rc, blk[i * NB + jj]);
        __syncthreads();
      }
      __syncthreads();
      if (s_bad) {
        if (threadIdx.x == 0) set_status(a.status, CBC_ERR_NOT_POSITIVE_DEFINITE);
      } else {
        for (int t = threadIdx.x; t < nb * nb; t += blockDim.x) {
          int i = t / nb, l = t % nb;
          if (l <= i) a.G[(int64_t)(b0 + i) * m + b0 + l] = blk[i * NB + l];
        }
      }
      __threadfence();
    }
    if (!grid_sync(a.bar, a.status, (unsigned)P)) return;
    if (*((volatile int*)a.status) != 0) return;
    // (2) panel rows below: x C_bb^H = g, one warp per row (lane l holds entry l)
    {
      T* cbb = pan;  // nb x NB copy of the factored block
      for (int t = threadIdx.x; t < nb * NB; t += blockDim.x) {
        int i = t / NB, l = t % NB;
        cbb[t] = (l <= i && l < nb) ? ldg_cg(a.G + (int64_t)(b0 + i) * m + b0 + l) : O::zero();
      }
      for (int i = threadIdx.x; i < nb; i += blockDim.x)
        s_rd[i] = rcp64(O::real(ldg_cg(a.G + (int64_t)(b0 + i) * m + b0 + i)));
      __syncthreads();
      for (int r = b0 + nb + cta * nw + warp; r < m; r += P * nw) {
        T* row = a.G + (int64_t)r * m + b0;
        T acc = (lane < nb) ? ldg_cg(row + lane) : O::zero();
        T x = O::zero();
        for (int t = 0; t < nb; ++t) {
          const T xt = shfl(O::scale(s_rd[t], acc), t);  // lane t is final at step t
          if (lane == t) x = xt;
          if (lane > t && lane < nb) acc = acc - xt * O::conj(cbb[lane * NB + t]);
        }
        if (lane < nb) row[lane] = x;
      }
    }
    if (!grid_sync(a.bar, a.status, (unsigned)P)) return;
    // (3) trailing update of the lower triangle from a shared copy of the panel
    const int r0 = b0 + nb;
    if (r0 < m) {
      const int rows = m - r0;
      if (PSMEM) {
        for (int t = threadIdx.x; t < rows * NB; t += blockDim.x) {
          int i = t / NB, l = t % NB;
          pan[t] = (l < nb) ? ldg_cg(a.G + (int64_t)(r0 + i) * m + b0 + l) : O::zero();
        }
        __syncthreads();
      }
      const int64_t nt = (int64_t)rows * (rows + 1) / 2;
      for (int64_t t = (int64_t)cta * blockDim.x + threadIdx.x; t < nt; t += (int64_t)P * blockDim.x) {
        // t -> (i, c) with c <= i in the packed lower triangle
        const int i = tri_row(t);
        const int c = (int)(t - (int64_t)i * (i + 1) / 2);
        T sacc = O::zero();
        if (PSMEM) {
#pragma unroll 8
          for (int l = 0; l < NB; ++l) sacc = O::fma(pan[i * NB + l], O::conj(pan[c * NB + l]), sacc);
        } else {
          const T* pi = a.G + (int64_t)(r0 + i) * m + b0;
          const T* pc = a.G + (int64_t)(r0 + c) * m + b0;
          for (int l = 0; l < nb; ++l) sacc = O::fma(ldg_cg(pi + l), O::conj(ldg_cg(pc + l)), sacc);
        }
        T* g = a.G + (int64_t)(r0 + i) * m + r0 + c;
        *g = ldg_cg(g) - sacc;
      }
    }
    if (!grid_sync(a.bar, a.status, (unsigned)P)) return;
  }
}

// offset of own row t (r = q + P t) in rank q's packed triangle: sum_{u<t} (q + P u + 1)
__device__ __forceinline__ int tri_off(int q, int P, int t) {
  return t * (q + 1) + P * (t * (t - 1) / 2);
}

// One CTA per matrix of a batch (blockIdx.x), the lower triangle packed in shared memory
// ((i, l) at i (i + 1) / 2 + l): right-looking, one column per step, no grid barriers.
// For batches, where the matrices themselves fill the SMs.
template <typename T>
__global__ void __launch_bounds__(TPB) chol1_kernel(T* G, int m, int* status) {
  using O = ops<T>;
  extern __shared__ unsigned char sm_raw[];
  T* L = reinterpret_cast<T*>(sm_raw);
  __shared__ double s_rc;
  __shared__ int s_bad;
  G += (int64_t)blockIdx.x * m * m;
  const int64_t tri = (int64_t)m * (m + 1) / 2;
  for (int64_t t = threadIdx.x; t < tri; t += blockDim.x) {
    const int i = tri_row(t);
    L[t] = G[(int64_t)i * m + (t - (int64_t)i * (i + 1) / 2)];
  }
  if (threadIdx.x == 0) s_bad = 0;
  __syncthreads();
  for (int j = 0; j < m; ++j) {
    const int64_t dj = (int64_t)j * (j + 1) / 2 + j;
    if (threadIdx.x == 0) {
      const double piv = O::real(L[dj]);
      if (!(piv > 0.0) || !isfinite(piv)) {
        s_bad = 1;
      } else {
        const double rc = rsqrt64(piv);  // 1 / sqrt(piv)
        L[dj] = O::make(piv * rc, 0.0);
        s_rc = rc;
      }
    }
    __syncthreads();
    if (s_bad) break;
    const double rc = s_rc;
    for (int i = j + 1 + threadIdx.x; i < m; i += blockDim.x) {
      T* x = L + (int64_t)i * (i + 1) / 2 + j;
      *x = O::scale(rc, *x);
    }
    __syncthreads();
    // trailing lower triangle (i, l), j < l <= i: L[i][l] -= L[i][j] conj(L[l][j])
    const int r = m - j - 1;
    const int64_t nt = (int64_t)r * (r + 1) / 2;
    for (int64_t t = threadIdx.x; t < nt; t += blockDim.x) {
      const int ii = tri_row(t);
      const int i = j + 1 + ii, l = j + 1 + (int)(t - (int64_t)ii * (ii + 1) / 2);
      const int64_t bi = (int64_t)i * (i + 1) / 2, bl = (int64_t)l * (l + 1) / 2;
      L[bi + l] = O::fma(O::scale(-1.0, L[bi + j]), O::conj(L[bl + j]), L[bi + l]);
    }
    __syncthreads();
  }
  if (s_bad) {
    if (threadIdx.x == 0) set_status(status, CBC_ERR_NOT_POSITIVE_DEFINITE);
    return;
  }
  for (int64_t t = threadIdx.x; t < tri; t += blockDim.x) {
    const int i = tri_row(t);
    G[(int64_t)i * m + (t - (int64_t)i * (i + 1) / 2)] = L[t];
  }
}

// One thread-block cluster of P CTAs (a power of two) per matrix, the lower triangle of each
// CTA's rows r = rank + P t packed in shared memory; right-looking, two columns per step.  A
// CTA sets its rows' entries of the next two columns aside while it updates them; after the
// step's one cluster barrier every CTA reads both columns from their owners (distributed
// shared memory) and updates the second by the first itself.  The updates need 1 / pivot only,
// A[r][c] -= (A[r][j] / pivot) conj(A[c][j]); the roots and the scaled columns come from one
// warp beside them.  Bound by that chain (~64 clocks per dependent FP64 operation).  Column
// blocks of 32 with three barriers through global memory each / one column per step / this:
// m = 128 complex 466 / 260 / 206 us (64 218 / 101 / 72).
constexpr int CHT = 128;
template <typename T>
__global__ void __launch_bounds__(CHT) chol_cluster_kernel(T* G, int m, int rows_cap, int nr_cap,
                                                           int* status) {
  using O = ops<T>;
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const int P = (int)cluster.num_blocks(), lp = 31 - __clz(P), pm = P - 1;
  const int cta = (int)cluster.block_rank();
  G += (int64_t)(blockIdx.x >> lp) * m * m;
  extern __shared__ unsigned char sm_raw[];
  T* rows = reinterpret_cast<T*>(sm_raw);
  T* set = rows + rows_cap;      // [2][nr_cap][2] own rows' entries of these two columns and the next
  T* col0 = set + 4 * nr_cap;    // [m] the columns
  T* col1 = col0 + m;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = CHT / 32;
  const int nr = (m - cta + pm) >> lp;
  for (int t = warp; t < nr; t += nw) {
    const int r = cta + (t << lp);
    T* dst = rows + tri_off(cta, P, t);
    for (int c = lane; c <= r; c += 32) {
      const T x = G[(int64_t)r * m + c];
      dst[c] = x;
      if (c < 2) set[2 * t + c] = x;
    }
  }
  // not positive or not finite, on the bits
  auto no_pivot = [](double p) {
    return (unsigned)__double2hiint(p) >= 0x7ff00000u || __double_as_longlong(p) == 0ll;
  };
  // 1 / pivot rounded up by one unit, so that a row that repeats an earlier one ends in a pivot
  // that is not positive
  // (below 2^-1019, where it would overflow, of 2^100 pivot)
  auto tiny = [](double p) { return __double2hiint(p) < 0x00400000; };
  auto inv_pivot = [&](double p) {
    return __longlong_as_double(__double_as_longlong(rcp64(tiny(p) ? 0x1p100 * p : p)) + 1ll);
  };
  // -x / pivot
  auto over = [&](double p, double rp, T x) {
    return O::scale(-rp, tiny(p) ? O::scale(0x1p100, x) : x);
  };
  bool bad = false;
  for (int j = 0; j < m && !bad; j += 2) {
    const T* now = set + ((j >> 1) & 1) * 2 * nr_cap;
    T* next = set + (((j >> 1) & 1) ^ 1) * 2 * nr_cap;
    const bool two = j + 1 < m;
    cluster.sync();
    for (int c = j + tid; c < m; c += CHT) {
      const T* src = cluster.map_shared_rank(now, c & pm) + 2 * (c >> lp);
      col0[c] = src[0];
      if (c > j) col1[c] = src[1];
    }
    __syncthreads();
    const double p0 = O::real(col0[j]);
    if (no_pivot(p0)) {
      bad = true;  // in every CTA
      break;
    }
    const double rp0 = inv_pivot(p0);
    if (two) {
      const T a1 = over(p0, rp0, O::conj(col0[j + 1]));
      for (int c = j + 1 + tid; c < m; c += CHT) col1[c] = O::fma(a1, col0[c], col1[c]);
    }
    __syncthreads();
    const double p1 = two ? O::real(col1[j + 1]) : 1.0;
    if (no_pivot(p1)) {
      bad = true;
      break;
    }
    if (warp == nw - 1) {  // the scaled columns
      const double rc0 = rsqrt64_short(p0), rc1 = rsqrt64_short(p1);
      for (int t = ((j > cta) ? (j - cta + pm) >> lp : 0) + lane; t < nr; t += 32) {
        const int r = cta + (t << lp);
        T* row = rows + tri_off(cta, P, t) + j;
        row[0] = (r == j) ? O::make(p0 * rc0, 0.0) : O::scale(rc0, col0[r]);
        if (r > j) row[1] = (r == j + 1) ? O::make(p1 * rc1, 0.0) : O::scale(rc1, col1[r]);
      }
    }
    const double rp1 = inv_pivot(p1);
    const int t0 = (j + 2 > cta) ? (j + 2 - cta + pm) >> lp : 0;  // first own row beyond j + 1
    // (by the other warps alone where there are few rows)
    const int uw = nr <= 16 ? nw - 1 : nw;
    for (int t = warp < uw ? t0 + warp : nr; t < nr; t += uw) {
      const int r = cta + (t << lp);
      T* row = rows + tri_off(cta, P, t);
      const T f0 = over(p0, rp0, col0[r]), f1 = over(p1, rp1, col1[r]);
      for (int c = j + 2 + lane; c <= r; c += 32) {
        const T x = O::fma(f1, O::conj(col1[c]), O::fma(f0, O::conj(col0[c]), row[c]));
        row[c] = x;
        if (c < j + 4) next[2 * t + c - j - 2] = x;
      }
    }
  }
  cluster.sync();  // no CTA leaves while another still reads its columns
  if (bad) {
    if (tid == 0) set_status(status, CBC_ERR_NOT_POSITIVE_DEFINITE);
    return;
  }
  for (int t = warp; t < nr; t += nw) {
    const int r = cta + (t << lp);
    const T* src = rows + tri_off(cta, P, t);
    for (int c = lane; c <= r; c += 32) G[(int64_t)r * m + c] = src[c];
  }
}

// S (m x n) <- C^{-1} S, C lower triangular (row-major m x m).  One warp per column.
template <typename T, bool CSMEM>
__global__ void trsm_cols_kernel(const T* C, T* S, int m, int n) {
  using O = ops<T>;
  C += (int64_t)blockIdx.y * m * m;  // problem blockIdx.y of a batch
  S += (int64_t)blockIdx.y * m * n;
  extern __shared__ unsigned char sm_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  T* cl = reinterpret_cast<T*>(sm_raw);  // packed lower triangle (CSMEM)
  double* rd = reinterpret_cast<double*>(cl + (CSMEM ? (size_t)m * (m + 1) / 2 : 0));
  T* xs = reinterpret_cast<T*>(rd + m);
  if (CSMEM) {
    const int64_t tot = (int64_t)m * (m + 1) / 2;
    for (int64_t t = threadIdx.x; t < tot; t += blockDim.x) {
      const int i = tri_row(t);
      const int l = (int)(t - (int64_t)i * (i + 1) / 2);
      cl[t] = C[(int64_t)i * m + l];
    }
  }
  for (int i = threadIdx.x; i < m; i += blockDim.x) rd[i] = rcp64(O::real(C[(int64_t)i * m + i]));
  __syncthreads();
  const int c = blockIdx.x * nw + warp;
  if (c >= n) return;
  T* x = xs + (size_t)warp * m;
  auto cel = [&](int i, int l) -> T {
    return CSMEM ? cl[(int64_t)i * (i + 1) / 2 + l] : C[(int64_t)i * m + l];
  };
  for (int b0 = 0; b0 < m; b0 += 32) {
    const int i = b0 + lane;
    const bool live = i < m;
    T acc = live ? S[(int64_t)i * n + c] : O::zero();
    for (int l = 0; l < b0; ++l) acc = acc - (live ? cel(i, l) : O::zero()) * x[l];
    const int gb = min(32, m - b0);
    for (int t = 0; t < gb; ++t) {
      const T xt = shfl(O::scale(rd[b0 + t], acc), t);
      if (lane == t) x[i] = xt;
      if (lane > t && live) acc = acc - cel(i, b0 + t) * xt;
    }
    __syncwarp();
  }
  for (int i = lane; i < m; i += 32) S[(int64_t)i * n + c] = x[i];
}

// The same solve in double-float arithmetic (the mixed path): the factor's lower
// triangle D and the reciprocal pivots R come as double-float pairs (converted once per
// solve by to_df_kernel), and the accumulation and the solution stay double-float; FP64
// only to read S and to write the result.
template <typename T, bool CSMEM>
__global__ void trsm_cols_df_kernel(const typename dfof<T>::type* D, const df1* R, T* S, int m,
                                    int n) {
  using O = ops<T>;
  using E = typename dfof<T>::type;
  D += (int64_t)blockIdx.y * m * m;
  R += (int64_t)blockIdx.y * m;
  S += (int64_t)blockIdx.y * m * n;
  extern __shared__ unsigned char sm_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  E* cl = reinterpret_cast<E*>(sm_raw);  // packed lower triangle (CSMEM)
  df1* rd = reinterpret_cast<df1*>(cl + (CSMEM ? (size_t)m * (m + 1) / 2 : 0));
  E* xs = reinterpret_cast<E*>(rd + m);
  if (CSMEM) {
    const int64_t tot = (int64_t)m * (m + 1) / 2;
    for (int64_t t = threadIdx.x; t < tot; t += blockDim.x) {
      const int i = tri_row(t);
      cl[t] = D[(int64_t)i * m + (int)(t - (int64_t)i * (i + 1) / 2)];
    }
  }
  for (int i = threadIdx.x; i < m; i += blockDim.x) rd[i] = R[i];
  __syncthreads();
  const int c = blockIdx.x * nw + warp;
  if (c >= n) return;
  E* x = xs + (size_t)warp * m;
  auto cel = [&](int i, int l) -> E {
    return CSMEM ? cl[(int64_t)i * (i + 1) / 2 + l] : D[(int64_t)i * m + l];
  };
  const df1 z1{0.f, 0.f};
  for (int b0 = 0; b0 < m; b0 += 32) {
    const int i = b0 + lane;
    const bool live = i < m;
    E acc = live ? to_df(S[(int64_t)i * n + c]) : E{};
    if (live)
      for (int l = 0; l < b0; ++l) acc = dff(df_neg(cel(i, l)), x[l], acc);
    const int gb = min(32, m - b0);
    for (int t = 0; t < gb; ++t) {
      E xt;
      if constexpr (O::cplx)
        xt = E{df_fma(acc.re, rd[b0 + t], z1), df_fma(acc.im, rd[b0 + t], z1)};
      else
        xt = df_fma(acc, rd[b0 + t], z1);
      xt = df_shfl_idx(xt, t);
      if (lane == t) x[i] = xt;
      if (lane > t && live) acc = dff(df_neg(cel(i, b0 + t)), xt, acc);
    }
    __syncwarp();
  }
  for (int i = lane; i < m; i += 32) S[(int64_t)i * n + c] = from_df(x[i]);
}

// The lower triangle of C (row-major m x m) and the reciprocals of its (real) pivots as
// double-float pairs, for trsm_cols_df_kernel; nb factors, m*m (and m) elements apart.
template <typename T>
__global__ void to_df_kernel(const T* C, typename dfof<T>::type* D, df1* R, int m) {
  using O = ops<T>;
  C += (int64_t)blockIdx.y * m * m;
  D += (int64_t)blockIdx.y * m * m;
  R += (int64_t)blockIdx.y * m;
  const int64_t tot = (int64_t)m * m;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < tot;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(t / m), l = (int)(t % m);
    if (l <= i) D[t] = to_df(C[t]);
  }
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x)
    R[i] = df_make(rcp64(O::real(C[(int64_t)i * m + i])));
}

// ---- triangular solve by matrix products -----------------------------------------------
// Blocks of TRB rows, X_b = C_bb^-1 (S_b - C_b,<b X_<b), with the inverses of the diagonal
// blocks and every product on the tensor cores (8 slices, an error below that of FP64 sums).
// A product with an inverse leaves a residual of the block's condition number times rounding,
// substitution one of rounding, so each block is corrected once: X_b += C_bb^-1 (S_b - C_bb
// X_b).  Bound by the chain of products; warp-per-column substitution / this, 64 of 128 x 256
// complex: 2360 / 700 us.
// (S comes with rows of unit norm: a slice has one exponent per column, and rows far smaller
// than others would be lost in the products with the inverses.)
constexpr int TRB = 64, TRH = 32;

// The diagonal blocks of C (lower triangular, m x m, nb of them) as TRB x TRB matrices with
// zeros above the diagonal (D; rows beyond m: unit rows), and the inverses of their two TRH x
// TRH diagonal halves (Inv); both zeroed before.  One CTA per half (blockIdx.x: block and half,
// blockIdx.y: matrix), four lanes per column of the inverse: x_r = -(1 / L_rr) sum_{i <= l < r}
// L[r][l] x_l.
template <typename T>
__global__ void __launch_bounds__(128) trsm_inv_kernel(const T* C, int m, T* D, T* Inv,
                                                       int64_t bs) {
  using O = ops<T>;
  __shared__ T g[TRH][TRH + 1];
  __shared__ double rl[TRH];
  const int blk = blockIdx.x >> 1, half = blockIdx.x & 1;
  const int r0 = blk * TRB + half * TRH;
  C += (int64_t)blockIdx.y * m * m;
  D += blockIdx.y * bs + (int64_t)blk * TRB * TRB + half * TRH * TRB;  // its rows
  Inv += blockIdx.y * bs + (int64_t)blk * TRB * TRB + half * TRH * (TRB + 1);
  for (int e = threadIdx.x; e < TRH * TRH; e += blockDim.x) {
    const int i = e / TRH, l = e % TRH, r = r0 + i;
    T x = (i == l) ? O::one() : O::zero();
    if (r < m) x = l <= i ? C[(int64_t)r * m + r0 + l] : O::zero();
    g[i][l] = x;
    D[(int64_t)i * TRB + half * TRH + l] = x;
    if (half == 1 && r < m) D[(int64_t)i * TRB + l] = C[(int64_t)r * m + r0 - TRH + l];
  }
  __syncthreads();
  if (threadIdx.x < TRH) rl[threadIdx.x] = rcp64(O::real(g[threadIdx.x][threadIdx.x]));
  __syncthreads();
  const int i = threadIdx.x >> 2, sub = threadIdx.x & 3;  // column i, terms l = sub (mod 4)
  T x[TRH / 4];                                           // x_l, l = sub + 4 q
#pragma unroll
  for (int q = 0; q < TRH / 4; ++q) x[q] = (sub + 4 * q == i) ? O::make(rl[i], 0.0) : O::zero();
#pragma unroll
  for (int r = 1; r < TRH; ++r) {
    T acc = O::zero();
#pragma unroll
    for (int q = 0; q < TRH / 4; ++q)
      if (4 * q < r) {
        const int l = sub + 4 * q;
        if (l < r) acc = O::fma(g[r][l], x[q], acc);
      }
    acc = acc + shfl_xor(acc, 1);
    acc = acc + shfl_xor(acc, 2);
    if (r > i && (r & 3) == sub) x[r >> 2] = O::scale(-rl[r], acc);
  }
#pragma unroll
  for (int q = 0; q < TRH / 4; ++q) Inv[(int64_t)(sub + 4 * q) * TRB + i] = x[q];
}

size_t al256(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace

template <typename T>
cudaError_t cholesky_lower(T* G, int m, int* status, void* bar, int num_sms, cudaStream_t s,
                           int nb, bool steady) {
  // the rows in the shared memory of one cluster per matrix: as many CTAs (and FP64 units) as
  // the batch leaves idle, 4 rows each at least; where that is one, a kernel without a cluster.
  // (`steady`: the earlier choice, the column blocks below, one CTA per matrix from 8 matrices on.
  // A change of the order of these sums by 1e-16 has moved mixed results on 64-bit data by 2e-9.)
  const size_t tri_bytes = (size_t)m * (m + 1) / 2 * sizeof(T);
  if (!steady) {
    const void* kc = (const void*)chol_cluster_kernel<T>;
    cudaError_t err = allow_max_smem(kc);
    if (err != cudaSuccess) return err;
    int want = 1;
    while (want < 16 && want * 4 < m && 2 * want * nb <= num_sms) want *= 2;
    if (want == 1 && nb > 1 && tri_bytes <= 200 * 1024) {
      err = allow_max_smem((const void*)chol1_kernel<T>);
      if (err != cudaSuccess) return err;
      note_launches(CBC_K_CHOLQR, 1);
      chol1_kernel<T><<<nb, TPB, tri_bytes, s>>>(G, m, status);
      return cudaGetLastError();
    }
    for (int P = want; P <= 16; P *= 2) {
      int rows_cap = 0, nr_cap = (m + P - 1) / P;
      for (int q = 0; q < P && q < m; ++q) {
        const int nr = (m - q + P - 1) / P;
        rows_cap = std::max(rows_cap, nr * (q + 1) + P * (nr * (nr - 1) / 2));
      }
      const size_t smem = ((size_t)rows_cap + 4 * nr_cap + 2 * m) * sizeof(T);
      if (smem > 220 * 1024 || cluster_ctas(kc, P, CHT, smem) != P) continue;
      note_launches(CBC_K_CHOLQR, 1);
      void* args[] = {&G, &m, &rows_cap, &nr_cap, &status};
      return launch_cluster(kc, P, nb * P, CHT, smem, args, s);
    }
  }
  if (steady && nb >= 8 && tri_bytes <= 200 * 1024) {
    cudaError_t err = allow_max_smem((const void*)chol1_kernel<T>);
    if (err != cudaSuccess) return err;
    note_launches(CBC_K_CHOLQR, 1);
    chol1_kernel<T><<<nb, TPB, tri_bytes, s>>>(G, m, status);
    return cudaGetLastError();
  }
  // larger matrices: column blocks with the matrix in global memory, one cluster of up to 16
  // CTAs per matrix when it fits (concurrent with other streams' work), else a cooperative
  // launch over more SMs per matrix
  cudaError_t err = cudaMemsetAsync(bar, 0, sizeof(GridBarrier) * nb, s);
  if (err != cudaSuccess) return err;
  // the panel in shared memory when it fits, else read from global memory
  const bool psmem = (size_t)std::max(m, NB) * NB * sizeof(T) <= 200 * 1024;
  const size_t shm = (size_t)(psmem ? std::max(m, NB) : NB) * NB * sizeof(T);
  const void* kch = psmem ? (const void*)chol_kernel<T, true> : (const void*)chol_kernel<T, false>;
  if (shm > 48 * 1024) {
    err = allow_max_smem(kch);
    if (err != cudaSuccess) return err;
  }
  note_launches(CBC_K_CHOLQR, 1);
  int P = std::max(1, std::min(16, (m * m) / 256));
  if (cluster_ctas(kch, P, TPB, shm) == P) {
    CholArgs<T> a{G, m, status, (GridBarrier*)bar, P};
    void* args[] = {&a};
    return launch_cluster(kch, P, nb * P, TPB, shm, args, s);
  }
  P = std::max(1, std::min(num_sms, (m * m) / 256));
  for (int b = 0; b < nb; ++b) {
    CholArgs<T> a{G + (int64_t)b * m * m, m, status, (GridBarrier*)bar + b, P};
    void* args[] = {&a};
    err = cudaLaunchCooperativeKernel(kch, dim3(P), dim3(TPB), args, shm, s);
    if (err != cudaSuccess) return err;
  }
  return cudaSuccess;
}

size_t trsm_products_bytes(int m, int n, bool cplx, int nb, bool df) {
  // Each block is a chain of four products (~75 us where they are small), so the line is work
  // per block.  Both solves of a CholeskyQR2, substitution / products in us: 128 x 256 complex,
  // 16 of them 1350 / 550, one 231 / 465; 64 of 64 x 128 complex 718 / 410; complex 400 x 800
  // 2586 / 1370, 256 x 512 694 / 806; real 600 x 1200 1265 / 1720.  Double-float substitution
  // takes about half as long.
  const double line = df ? 1.2e8 : 6e7;
  if ((double)m * m * n * nb * (cplx ? 4 : 1) < line * ((m + TRB - 1) / TRB)) return 0;
  const size_t ts = cplx ? sizeof(zdbl) : sizeof(double);
  const size_t nblk = (m + TRB - 1) / TRB;
  if (nb * nblk > TC_MAX_PROBLEMS) return 0;  // (the blocks' inverses are one call)
  size_t g = gemm_tc_workspace_bytes(TRH, TRH, TRH, cplx, 8, (int)(nb * nblk));
  g = std::max(g, gemm_tc_workspace_bytes(std::min(TRB, m), n, m, cplx, 8, nb));
  return 256 + al256(2 * nb * nblk * TRB * TRB * ts) + al256(nb * nblk * TRH * TRH * ts) +
         al256((size_t)nb * TRB * n * ts) + g;
}

template <typename T>
cudaError_t trsm_products(const T* C, T* S, int m, int n, int* status, void* ws, cudaStream_t s,
                          int nb) {
  const int nblk = (m + TRB - 1) / TRB;
  const int64_t sq = TRB * TRB, bs = nblk * sq, hf = TRH * TRH, mn = (int64_t)m * n;
  char* w = static_cast<char*>(ws);
  auto take = [&](size_t bytes) {
    char* p = w;
    w += al256(bytes);
    return p;
  };
  TcWide set;
  // Not read: S has finite rows of unit norm and C is the factor of its Gram, which a row with Inf
  // or NaN would have failed (the call then returns that status whatever the solve makes of it).
  set.wide = reinterpret_cast<int*>(take(4));
  T* D = reinterpret_cast<T*>(take(2 * nb * bs * sizeof(T)));
  T* Inv = D + nb * bs;
  T* tmp = reinterpret_cast<T*>(take(sizeof(T) * nb * nblk * hf));
  T* X = reinterpret_cast<T*>(take(sizeof(T) * (size_t)nb * TRB * n));
  void* gw = w;
  cudaError_t e = cudaMemsetAsync(D, 0, 2 * nb * bs * sizeof(T), s);
  if (e != cudaSuccess) return e;
  note_launches(CBC_K_CHOLQR, 1);
  trsm_inv_kernel<T><<<dim3(2 * nblk, nb), 128, 0, s>>>(C, m, D, Inv, bs);
  // dst = A B (acc 0), dst - A B (-1) or base + A B (1)
  auto mul = [&](int M, int N, int K, const T* A, int64_t lda, int64_t abs, const T* B,
                 int64_t ldb, int64_t bbs, T* dst, int64_t ldc, int64_t cbs, int cnt, int acc,
                 const T* base) {
    if (e != cudaSuccess) return;
    TcWide o = set;
    o.acc = acc;
    o.base = base;
    o.base_bs = (int64_t)TRB * n;  // (X)
    e = gemm_tc<T>(M, N, K, A, View::rowmajor(lda, abs), false, B, View::rowmajor(ldb, bbs), false,
                   dst, View::rowmajor(ldc, cbs), 8, gw, status, s, cnt, o);
  };
  // the inverse of a block from its halves': Inv21 = -Inv22 (C21 Inv11)
  mul(TRH, TRH, TRH, D + TRH * TRB, TRB, sq, Inv, TRB, sq, tmp, TRH, hf, nb * nblk, 0, nullptr);
  mul(TRH, TRH, TRH, Inv + TRH * (TRB + 1), TRB, sq, tmp, TRH, hf, Inv + TRH * TRB, TRB, sq,
      nb * nblk, -1, nullptr);
  for (int q = 0; q < nblk; ++q) {
    const int r0 = q * TRB, h = std::min(TRB, m - r0);
    T* Sb = S + (int64_t)r0 * n;
    const T *Db = D + q * sq, *Ib = Inv + q * sq;
    if (q > 0)
      mul(h, n, r0, C + (int64_t)r0 * m, m, (int64_t)m * m, S, n, mn, Sb, n, mn, nb, -1, nullptr);
    mul(h, n, h, Ib, TRB, bs, Sb, n, mn, X, n, (int64_t)TRB * n, nb, 0, nullptr);
    mul(h, n, h, Db, TRB, bs, X, n, (int64_t)TRB * n, Sb, n, mn, nb, -1, nullptr);
    mul(h, n, h, Ib, TRB, bs, Sb, n, mn, Sb, n, mn, nb, 1, X);
  }
  return e;
}

template <typename T>
cudaError_t trsm_lower_left(const T* C, T* S, int m, int n, int* status, void* bar, int num_sms,
                            cudaStream_t s, int nb, void* dfbuf) {
  (void)status;
  (void)bar;
  (void)num_sms;
  if (dfbuf) {  // double-float solve: the factor converted once, then one warp per column
    using E = typename dfof<T>::type;
    E* D = static_cast<E*>(dfbuf);
    df1* R = reinterpret_cast<df1*>(D + (size_t)nb * m * m);
    note_launches(CBC_K_CHOLQR, 2);
    to_df_kernel<T><<<dim3(std::max(1, std::min(64, (m * m + 255) / 256)), nb), 256, 0, s>>>(C, D, R, m);
    const int nw = nb >= 8 ? 8 : 4;
    const size_t tri = (size_t)m * (m + 1) / 2 * sizeof(E);
    const size_t rest = (size_t)m * sizeof(df1) + (size_t)nw * m * sizeof(E);
    const dim3 grid((n + nw - 1) / nw, nb);
    cudaError_t err;
    if (tri + rest <= 200 * 1024) {
      err = allow_max_smem((const void*)trsm_cols_df_kernel<T, true>);
      if (err != cudaSuccess) return err;
      trsm_cols_df_kernel<T, true><<<grid, 32 * nw, tri + rest, s>>>(D, R, S, m, n);
    } else {
      if (rest > 48 * 1024) {
        err = allow_max_smem((const void*)trsm_cols_df_kernel<T, false>);
        if (err != cudaSuccess) return err;
      }
      trsm_cols_df_kernel<T, false><<<grid, 32 * nw, rest, s>>>(D, R, S, m, n);
    }
    return cudaGetLastError();
  }
  // warps (columns) per CTA sharing one staged triangle: two per SM sub-partition when a
  // batch provides the CTAs, else one (more CTAs for a lone solve)
  const int nw = nb >= 8 ? 8 : 4;
  const size_t tri = (size_t)m * (m + 1) / 2 * sizeof(T);
  const size_t rest = (size_t)m * sizeof(double) + (size_t)nw * m * sizeof(T);
  note_launches(CBC_K_CHOLQR, 1);
  const dim3 grid((n + nw - 1) / nw, nb);
  cudaError_t err;
  if (tri + rest <= 200 * 1024) {
    err = allow_max_smem((const void*)trsm_cols_kernel<T, true>);
    if (err != cudaSuccess) return err;
    trsm_cols_kernel<T, true><<<grid, 32 * nw, tri + rest, s>>>(C, S, m, n);
  } else {
    if (rest > 48 * 1024) {
      err = allow_max_smem((const void*)trsm_cols_kernel<T, false>);
      if (err != cudaSuccess) return err;
    }
    trsm_cols_kernel<T, false><<<grid, 32 * nw, rest, s>>>(C, S, m, n);
  }
  return cudaGetLastError();
}

template cudaError_t cholesky_lower<double>(double*, int, int*, void*, int, cudaStream_t, int, bool);
template cudaError_t cholesky_lower<zdbl>(zdbl*, int, int*, void*, int, cudaStream_t, int, bool);
template cudaError_t trsm_products<double>(const double*, double*, int, int, int*, void*,
                                           cudaStream_t, int);
template cudaError_t trsm_products<zdbl>(const zdbl*, zdbl*, int, int, int*, void*, cudaStream_t,
                                         int);
template cudaError_t trsm_lower_left<double>(const double*, double*, int, int, int*, void*, int,
                                             cudaStream_t, int, void*);
template cudaError_t trsm_lower_left<zdbl>(const zdbl*, zdbl*, int, int, int*, void*, int,
                                           cudaStream_t, int, void*);

}  // namespace cbc
