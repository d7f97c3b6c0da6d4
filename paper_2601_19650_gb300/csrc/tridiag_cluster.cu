// Householder reduction of the truncation Gram matrices to real symmetric tridiagonal
// form (the first stage of the eigensolver behind the compression of Sec. III A), one
// thread-block cluster per matrix.
//
// Layout: the P CTAs of a cluster (a power of two) own the rows r = rank + P t of the matrix
// and keep only their lower triangle (columns 0 .. r) in shared memory, packed row after row.
//
// Column k (H_k = I - tau v v^H, H^H x = beta e_1, beta real; x = A[k+1:, k]):
//   1. every CTA holds x.  One warp computes beta, tau and 1 / (alpha - beta) (the same data in
//      the same order, so identical values in every CTA: no broadcast needed) while the others
//      apply the rank-2 update of column k-1, A -= v w^H + w v^H, to the stored rows;
//   2. each CTA's share of A v: each stored entry A[r][c] (c <= r) contributes A[r][c] v_c to
//      row r and, below the diagonal, conj(A[r][c]) v_r to row c.  The entries of column k+1
//      are set aside, and v goes into column k of the rows, which is no longer needed;
//   3. cluster barrier, the only one of the column (the exchange buffers alternate);
//   4. every CTA adds the P shares in one fixed order and reads column k+1 (distributed
//      shared memory), forms w = tau A v - (|tau|^2 / 2)(v^H A v) v (v^H A v is real) and
//      the next x = A[:, k+1] - v conj(w_{k+1}) - w by itself.
// Nothing goes to global memory before the end: a store in flight holds up the release of
// every cluster barrier.  The reduction is a chain of m columns of reductions, exchanges and
// the CTA's share of the arithmetic, which in turn needs several independent rows per warp to
// cover its dependent operations.  Two barriers,
// one row at a time and the update behind the scalars / this, double-float: 64 of m = 256 complex
// 7.9 / 7.2 ms, 8 of 512 real 6.9 / 6.0, 64 of 64 complex 0.60 / 0.38; FP64: 2 of 512 real 10.1
// / 7.0.  (16 of m = 256 complex: issue slots of the busy SMs 37%, FP32 pipe 29%.)
// DF (the mixed path): the rows and every per-element quantity as double-float pairs, so all
// O(m) and O(m^2) work per column runs in FP32 arithmetic with error-free transformations;
// FP64 only for the handful of Householder scalars.  Otherwise FP64 throughout.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "df.cuh"
#include "isum.cuh"
#include "kernels.cuh"
#include "planner.h"

namespace cg = cooperative_groups;

namespace cbc {
namespace {

constexpr int TCL_G = 4;  // consecutive own rows that a warp works on side by side

template <typename T>
struct TriClArgs {
  const T* A;      // nb matrices m x m (row-major, Hermitian; lower triangle read)
  int m;
  double* d;       // per-matrix outputs, workspaces wb bytes apart:
  double* e;       //   diagonal, off-diagonal (beta_j), tau_j, and the reflectors
  T* tau;          //   V (row j: [j+1] = 1, [c] = v_c for c > j + 1)
  T* V;
  int64_t a_bs;    // elements between consecutive matrices A
  size_t wb;       // bytes between consecutive workspaces
  int rows_cap;    // stored elements of the largest share of rows
  int nr_cap;      // rows of the largest share
};

template <typename P>
__device__ __forceinline__ P* shift_bytes(P* p, size_t bytes) {
  return reinterpret_cast<P*>(reinterpret_cast<char*>(p) + bytes);
}

// Element type of the stored rows and of every per-element quantity (v, w, A v and its
// shares), and the arithmetic on them: FP64 (T itself), or double-float pairs on the
// mixed path, where every per-element operation and every reduction runs on the FP32
// pipes and FP64 is left to the few scalars of each Householder step.  (Sums renormalised
// only after a few products take 7% less time and give 15 to 35% larger errors: not used.)
template <typename T, bool DF>
struct RowArith;
template <typename T>
struct RowArith<T, false> {
  using O = ops<T>;
  using E = T;
  using R = double;  // real quantities
  __device__ static __forceinline__ E cvt(T x) { return x; }
  __device__ static __forceinline__ R rcvt(double x) { return x; }
  __device__ static __forceinline__ E make(R re, R im) { return O::make(re, im); }
  __device__ static __forceinline__ R re(E a) { return O::real(a); }
  __device__ static __forceinline__ R im(E a) { return O::imag(a); }
  __device__ static __forceinline__ T back(E x) { return x; }
  __device__ static __forceinline__ E mac(E a, E b, E c) { return O::fma(a, b, c); }
  __device__ static __forceinline__ E cj(E a) { return O::conj(a); }
  __device__ static __forceinline__ E zero() { return O::zero(); }
  __device__ static __forceinline__ E one() { return O::one(); }
  __device__ static __forceinline__ E add(E a, E b) { return a + b; }
  __device__ static __forceinline__ E neg(E a) { return O::scale(-1.0, a); }
  __device__ static __forceinline__ E rscale(R a, E b, E c) {  // c + a b, a real
    if constexpr (O::cplx)
      return zdbl{::fma(a, b.re, c.re), ::fma(a, b.im, c.im)};
    else
      return ::fma(a, b, c);
  }
  __device__ static __forceinline__ E shfl(E a, int o) { return shfl_xor(a, o); }
  __device__ static __forceinline__ R rzero() { return 0.0; }
  __device__ static __forceinline__ R radd(R a, R b) { return a + b; }
  __device__ static __forceinline__ R rmul(R a, R b) { return a * b; }
  // c + Re(conj(a) b)
  __device__ static __forceinline__ R redot(E a, E b, R c) {
    if constexpr (O::cplx)
      return ::fma(a.im, b.im, ::fma(a.re, b.re, c));
    else
      return ::fma(a, b, c);
  }
  __device__ static __forceinline__ double rback(R a) { return a; }
  __device__ static __forceinline__ R rshfl(R a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
};
template <typename T>
struct RowArith<T, true> {
  using O = ops<T>;
  using E = typename dfof<T>::type;
  using R = df1;
  __device__ static __forceinline__ E cvt(T x) { return to_df(x); }
  __device__ static __forceinline__ R rcvt(double x) { return df_make(x); }
  __device__ static __forceinline__ E make(R re, R im) {
    if constexpr (O::cplx)
      return {re, im};
    else
      return re;
  }
  __device__ static __forceinline__ R re(E a) {
    if constexpr (O::cplx)
      return a.re;
    else
      return a;
  }
  __device__ static __forceinline__ R im(E a) {
    if constexpr (O::cplx)
      return a.im;
    else
      return R{};
  }
  __device__ static __forceinline__ T back(E x) { return from_df(x); }
  __device__ static __forceinline__ E mac(E a, E b, E c) { return dff(a, b, c); }
  __device__ static __forceinline__ E cj(E a) { return dfconj(a); }
  __device__ static __forceinline__ E zero() { return E{}; }
  __device__ static __forceinline__ E one() {
    E x{};
    if constexpr (O::cplx) x.re.h = 1.f; else x.h = 1.f;
    return x;
  }
  __device__ static __forceinline__ E add(E a, E b) { return df_add(a, b); }
  __device__ static __forceinline__ E neg(E a) { return df_neg(a); }
  __device__ static __forceinline__ E rscale(R a, E b, E c) {
    if constexpr (O::cplx)
      return {df_fma(a, b.re, c.re), df_fma(a, b.im, c.im)};
    else
      return df_fma(a, b, c);
  }
  __device__ static __forceinline__ E shfl(E a, int o) { return df_shfl_xor(a, o); }
  __device__ static __forceinline__ R rzero() { return R{}; }
  __device__ static __forceinline__ R radd(R a, R b) { return df_add(a, b); }
  __device__ static __forceinline__ R rmul(R a, R b) { return df_fma(a, b, R{}); }
  __device__ static __forceinline__ R redot(E a, E b, R c) {
    if constexpr (O::cplx)
      return df_fma(a.im, b.im, df_fma(a.re, b.re, c));
    else
      return df_fma(a, b, c);
  }
  __device__ static __forceinline__ double rback(R a) { return from_df(a); }
  __device__ static __forceinline__ R rshfl(R a, int o) { return df_shfl_xor(a, o); }
};

// offset of own row t (r = q + P t) in rank q's packed triangle: sum_{u<t} (q + P u + 1)
__device__ __forceinline__ int row_off(int q, int P, int t) {
  return t * (q + 1) + P * (t * (t - 1) / 2);
}

// The sums of TCL_G = 4 values over the 32 lanes, row 2 (lane / 16) + (lane / 8) % 2 in every
// lane: two levels pass on half of the rows each, so 6 additions instead of 20
template <typename AR>
__device__ __forceinline__ typename AR::E rows_sum(typename AR::E (&r)[TCL_G], int lane) {
  static_assert(TCL_G == 4, "two halving levels");
  const bool h16 = lane & 16, h8 = lane & 8;
  const typename AR::E a = AR::add(h16 ? r[2] : r[0], AR::shfl(h16 ? r[0] : r[2], 16));
  const typename AR::E b = AR::add(h16 ? r[3] : r[1], AR::shfl(h16 ? r[1] : r[3], 16));
  typename AR::E x = AR::add(h8 ? b : a, AR::shfl(h8 ? a : b, 8));
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) x = AR::add(x, AR::shfl(x, o));
  return x;
}

template <typename T, bool DF, int TH>
__global__ void __launch_bounds__(TH) tridiag_cluster_kernel(TriClArgs<T> a0) {
  using O = ops<T>;
  using AR = RowArith<T, DF>;
  using E = typename AR::E;
  using R = typename AR::R;
  constexpr int NW = TH / 32;
  cg::cluster_group cluster = cg::this_cluster();
  const int P = (int)cluster.num_blocks();  // a power of two
  const int lp = 31 - __clz(P), pm = P - 1;
  const int cta = (int)cluster.block_rank();
  const int inst = blockIdx.x >> lp;
  const int m = a0.m;
  const T* A = a0.A + (int64_t)inst * a0.a_bs;
  const size_t off = (size_t)inst * a0.wb;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  E* rows = reinterpret_cast<E*>(smem_raw);
  E* vbuf = rows + a0.rows_cap;          // [2][m] x, then v, of this column; v of the one before
  E* wE = vbuf + 2 * m;                  // w of the one before (tau A v before that)
  E* ppE = wE + m;                       // [2][m] this CTA's share of A v (read by the others)
  E* colE = ppE + 2 * m;                 // [2][nr_cap] own rows' entries of the next column
  E* rpE = colE + 2 * a0.nr_cap;         // row sums of own rows
  E* wpartE = rpE + a0.nr_cap;           // [warp][m] column sums
  T* s_tau = reinterpret_cast<T*>(wpartE + (size_t)NW * m);  // tau, d and e of every column
  double* s_d = reinterpret_cast<double*>(s_tau + m);
  double* s_e = s_d + m;
  __shared__ WarpSum s_norm[NW], s_dot[NW];
  __shared__ E s_tyE;
  __shared__ R s_sc[5];  // tau (re, im), 1 / (alpha - beta) (re, im), -|tau|^2 / 2

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nr = (m - cta + pm) >> lp;   // own rows r = cta + P t, t < nr
  for (int t = 0; t < nr; ++t) {
    const int r = cta + (t << lp);
    const T* src = A + (int64_t)r * m;
    E* dst = rows + row_off(cta, P, t);
    for (int c = tid; c <= r; c += TH) dst[c] = AR::cvt(src[c]);
  }
  R part = AR::rzero();
  for (int c = tid; c < m; c += TH) {  // the first column
    const E x = AR::cvt(A[(int64_t)c * m]);
    vbuf[c] = x;
    if (c >= 2) part = AR::redot(x, x, part);
  }

  for (int k = 0;; ++k) {
    E* vE = vbuf + (k & 1) * m;            // x of column k
    E* vp = vbuf + ((k & 1) ^ 1) * m;      // v of column k - 1
    {
      const WarpSum s = warp_isum(AR::rback(part));
      if (lane == 0) s_norm[warp] = s;
    }
    __syncthreads();
    if (k == m - 1) {
      if (tid == 0) s_d[k] = O::real(AR::back(vE[k]));
      break;
    }
    const int t0 = (k + 1 > cta) ? (k + 1 - cta + pm) >> lp : 0;  // first own row beyond k
    const int c_first = (k + 1) & ~31, g_first = t0 / TCL_G;
    // 1. a warp takes TCL_G own rows at a time, lanes over columns (from a multiple of 32)
    if (warp == 0) {
      // the Householder scalars in FP64, lanes 0 and 1 (2 and 3) holding the real and the
      // imaginary part of one quantity each: an FP64 instruction costs the same for one lane
      // as for 32
      const double xn2 = block_isum<NW>(s_norm);
      const E al = vE[k + 1], xk = vE[k];
      const double in = AR::rback(lane == 0 ? AR::re(al) : (lane == 1 ? AR::im(al) : AR::re(xk)));
      const double ar = __shfl_sync(0xffffffffu, in, 0);
      const double ai = O::cplx ? __shfl_sync(0xffffffffu, in, 1) : 0.0;
      double out = 0.0, beta = ar;  // xn2 = 0 and alpha real: the identity
      const double n2 = O::cplx ? fma(ar, ar, fma(ai, ai, xn2)) : fma(ar, ar, xn2);
      const bool rest = __double_as_longlong(xn2) != 0ll ||
                        (__double_as_longlong(ai) & 0x7fffffffffffffffll) != 0ll;
      if (rest && __double_as_longlong(n2) != 0ll) {
        const double rn = rsqrt64_short(n2);  // 1 / ||x||
        const double nrm = n2 * rn;
        const bool pos = __double2hiint(ar) >= 0;
        beta = pos ? -nrm : nrm;
        const double ib = pos ? -rn : rn;  // 1 / beta
        const double zr = ar - beta;       // alpha - beta = (zr, ai)
        const double den = O::cplx ? fma(zr, zr, ai * ai) : zr * zr;
        const double iden = rcp64(den);
        // tau = -(alpha - beta) / beta, 1 / (alpha - beta) = conj(alpha - beta) / den
        const double z = (lane & 1) ? ai : zr;
        const double f = lane < 2 ? -ib : ((lane & 1) ? -iden : iden);
        out = lane < 4 ? z * f : -0.5 * (den * (rn * rn));
      }
      if (lane < 5) s_sc[lane] = AR::rcvt(out);
      if (O::cplx || lane == 0) {
        if (lane < 2) reinterpret_cast<double*>(s_tau + k)[lane] = out;
      }
      if (lane == 2) {
        s_d[k] = in;
        s_e[k] = beta;
      }
    } else if (k > 0 && (DF || (warp & 3))) {
      // FP64: not by the warps that share warp 0's FP64 unit
      const int wi = DF ? warp - 1 : warp - 1 - (warp >> 2), wn = DF ? NW - 1 : NW - NW / 4;
      for (int gq = g_first + wi; gq * TCL_G < nr; gq += wn) {
        E nv[TCL_G], nw[TCL_G];
        E* row[TCL_G];
        int rr[TCL_G], rmax = -1;
#pragma unroll
        for (int i = 0; i < TCL_G; ++i) {
          const int t = gq * TCL_G + i;
          const bool ok = t >= t0 && t < nr;
          rr[i] = ok ? cta + (t << lp) : -1;
          rmax = max(rmax, rr[i]);
          row[i] = rows + row_off(cta, P, ok ? t : 0);
          nv[i] = ok ? AR::neg(vp[rr[i]]) : AR::zero();
          nw[i] = ok ? AR::neg(wE[rr[i]]) : AR::zero();
        }
        for (int base = c_first; base <= rmax; base += 32) {
          const int c = base + lane;
          const bool in = c > k && c < m;
          const E pv = in ? AR::cj(vp[c]) : AR::zero(), pw = in ? AR::cj(wE[c]) : AR::zero();
          E x[TCL_G];
#pragma unroll
          for (int i = 0; i < TCL_G; ++i) x[i] = (in && c <= rr[i]) ? row[i][c] : AR::zero();
#pragma unroll
          for (int i = 0; i < TCL_G; ++i)
            x[i] = AR::mac(nw[i], pv, AR::mac(nv[i], pw, x[i]));
#pragma unroll
          for (int i = 0; i < TCL_G; ++i)
            if (in && c <= rr[i]) row[i][c] = x[i];
        }
      }
    }
    __syncthreads();
    const E tauE = AR::make(s_sc[0], s_sc[1]);
    {
      const E sc = AR::make(s_sc[2], s_sc[3]);  // zero where the reflector is the identity
      for (int c = k + 1 + tid; c < m; c += TH)
        vE[c] = (c == k + 1) ? AR::one() : AR::mac(vE[c], sc, AR::zero());
    }
    __syncthreads();

    // 2. this CTA's share of A v
    E* pp = ppE + (k & 1) * m;
    E* colx = colE + (k & 1) * a0.nr_cap;
    E* wpart = wpartE + (size_t)warp * m;
    bool first = true;
    for (int gq = g_first + warp; first || gq * TCL_G < nr; gq += NW) {
      E racc[TCL_G], vr[TCL_G];
      E* row[TCL_G];
      int rr[TCL_G], rmax = -1;
#pragma unroll
      for (int i = 0; i < TCL_G; ++i) {
        const int t = gq * TCL_G + i;
        const bool ok = t >= t0 && t < nr;
        rr[i] = ok ? cta + (t << lp) : -1;
        rmax = max(rmax, rr[i]);
        row[i] = rows + row_off(cta, P, ok ? t : 0);
        racc[i] = AR::zero();
        vr[i] = ok ? vE[rr[i]] : AR::zero();
      }
      for (int base = c_first; base < m; base += 32) {
        const int c = base + lane;
        const bool in = c > k && c < m;
        E acc = AR::zero();
        if (base <= rmax) {
          const E vc = in ? vE[c] : AR::zero();
          E x[TCL_G];
#pragma unroll
          for (int i = 0; i < TCL_G; ++i) x[i] = (in && c <= rr[i]) ? row[i][c] : AR::zero();
#pragma unroll
          for (int i = 0; i < TCL_G; ++i) {
            if (c == k + 1 && rr[i] >= 0) colx[gq * TCL_G + i] = x[i];
            racc[i] = AR::mac(x[i], vc, racc[i]);  // A[r][c] v_c -> row r
            // conj(A[r][c]) v_r -> row c, below the diagonal
            acc = AR::mac(AR::cj(x[i]), c < rr[i] ? vr[i] : AR::zero(), acc);
          }
        }
        if (in) {
          wpart[c] = first ? acc : AR::add(wpart[c], acc);
        }
      }
      first = false;
      const E sum = rows_sum<AR>(racc, lane);
      const int t = gq * TCL_G + ((lane >> 4) & 1) * 2 + ((lane >> 3) & 1);
      if ((lane & 7) == 0 && t >= t0 && t < nr) {
        rpE[t] = sum;
        rows[row_off(cta, P, t) + k] = vE[cta + (t << lp)];
      }
    }
    __syncthreads();
    for (int c = k + 1 + tid; c < m; c += TH) {
      E sum = ((c & pm) == cta) ? rpE[c >> lp] : AR::zero();
#pragma unroll
      for (int w = 0; w < NW; ++w) sum = AR::add(sum, wpartE[(size_t)w * m + c]);
      pp[c] = sum;
    }
    // 3. every share and column k+1 are ready; the buffers of column k-1 are free again
    cluster.sync();

    // 4. A v from the P shares in a fixed order; w; x of the next column, in the buffer of the
    // last v
    R dp = AR::rzero();
    for (int c = k + 1 + tid; c < m; c += TH) {
      const E col = cluster.map_shared_rank(colx, c & pm)[c >> lp];
      E y = AR::zero();
      for (int q0 = 0; q0 < P; q0 += 8) {  // eight remote reads in flight
        E sh[8];
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (q0 + q < P) sh[q] = cluster.map_shared_rank(pp, q0 + q)[c];
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (q0 + q < P) y = AR::add(y, sh[q]);
      }
      const E ty = AR::mac(tauE, y, AR::zero());
      wE[c] = ty;
      vp[c] = col;
      if (c == k + 1) s_tyE = ty;
      dp = AR::redot(vE[c], y, dp);
    }
    {
      const WarpSum s = warp_isum(AR::rback(dp));
      if (lane == 0) s_dot[warp] = s;
    }
    __syncthreads();
    const R coef = AR::rmul(s_sc[4], AR::rcvt(block_isum<NW>(s_dot)));
    const E nwk = AR::neg(AR::cj(AR::rscale(coef, AR::one(), s_tyE)));  // v_{k+1} = 1
    part = AR::rzero();
    for (int c = k + 1 + tid; c < m; c += TH) {
      const E v = vE[c];
      const E w = AR::rscale(coef, v, wE[c]);
      wE[c] = w;
      const E x = AR::add(AR::mac(v, nwk, vp[c]), AR::neg(w));
      vp[c] = x;
      if (c >= k + 3) part = AR::redot(x, x, part);
    }
  }
  cluster.sync();  // no CTA leaves while another still reads its shares
  // the reflectors, by the rows' owners: v_k at column k of the rows beyond k
  T* V = shift_bytes(a0.V, off);
  for (int t = warp; t < nr; t += NW) {
    const int r = cta + (t << lp);
    const E* row = rows + row_off(cta, P, t);
    for (int k = lane; k < r; k += 32) V[(int64_t)k * m + r] = AR::back(row[k]);
  }
  if (cta == 0) {
    double* d = shift_bytes(a0.d, off);
    double* e = shift_bytes(a0.e, off);
    T* tau = shift_bytes(a0.tau, off);
    for (int k = tid; k < m; k += TH) {
      d[k] = s_d[k];
      if (k < m - 1) {
        e[k] = s_e[k];
        tau[k] = s_tau[k];
      }
    }
  }
}

template <typename T>
void cluster_shape(int m, int P, int* rows_cap, int* nr_cap) {
  int rc = 0, nc = 0;
  for (int q = 0; q < P; ++q) {
    const int nr = (m - q + P - 1) / P;
    const int cnt = nr * (q + 1) + P * (nr * (nr - 1) / 2);
    rc = std::max(rc, cnt);
    nc = std::max(nc, nr);
  }
  *rows_cap = rc;
  *nr_cap = nc;
}

template <typename T>
size_t cluster_smem(int m, int P, int threads) {
  int rc, nc;
  cluster_shape<T>(m, P, &rc, &nc);
  // a double-float element has the size of its FP64 one
  return ((size_t)rc + (size_t)(6 + threads / 32) * m + (size_t)3 * nc) * sizeof(T) +
         (size_t)2 * m * sizeof(double);
}

template <typename T, int TH>
const void* cluster_kernel(bool df) {
  return df ? (const void*)tridiag_cluster_kernel<T, true, TH>
            : (const void*)tridiag_cluster_kernel<T, false, TH>;
}
template <typename T>
const void* cluster_kernel(bool df, int threads) {
  return threads == 256 ? cluster_kernel<T, 256>(df) : cluster_kernel<T, 128>(df);
}

}  // namespace

template <typename T>
TriClusterShape tridiag_cluster_shape(int m, int nb, bool df) {
  static_assert(sizeof(typename dfof<T>::type) == sizeof(T), "double-float element size");
  // Double-float: the fewest CTAs (at least 4) that hold the matrix, since every CTA repeats
  // the O(m) work of a column; 8 warps where m gives them rows (4 warps cost 8 of m = 512
  // real 23% more, 8 warps cost 64 of 64 complex 21% more).  FP64: as many SMs' FP64 units as the
  // batch leaves idle (2 of m = 512 real on 8 / 16 CTAs 8220 / 6960 us; 4 of 256 complex on 4 /
  // 8 / 16 7010 / 5210 / 5290).
  const int lead = m > 256 || !df ? 256 : 128;
  int low = 4;
  if (!df)
    while (low < (m >= 400 ? 16 : 8) && 2 * low * nb <= num_sms()) low *= 2;
  for (int threads : {lead, 384 - lead}) {
    const void* k = cluster_kernel<T>(df, threads);
    if (allow_max_smem(k) != cudaSuccess) return {};
    for (int P : {4, 8, 16}) {
      if (P < low) continue;
      const size_t smem = cluster_smem<T>(m, P, threads);
      if (smem > 222 * 1024) continue;
      if (cluster_ctas(k, P, threads, smem) == P) return {P, threads};
    }
  }
  return {};
}

template <typename T>
cudaError_t tridiag_cluster(const T* A, int m, double* d, double* e, T* tau, T* V, int64_t a_bs,
                            size_t wb, int nb, const TriClusterShape& sh, bool df,
                            cudaStream_t s) {
  TriClArgs<T> a{A, m, d, e, tau, V, a_bs, wb, 0, 0};
  cluster_shape<T>(m, sh.ctas, &a.rows_cap, &a.nr_cap);
  void* args[] = {&a};
  return launch_cluster(cluster_kernel<T>(df, sh.threads), sh.ctas, nb * sh.ctas, sh.threads,
                        cluster_smem<T>(m, sh.ctas, sh.threads), args, s);
}

template TriClusterShape tridiag_cluster_shape<double>(int, int, bool);
template TriClusterShape tridiag_cluster_shape<zdbl>(int, int, bool);
template cudaError_t tridiag_cluster<double>(const double*, int, double*, double*, double*,
                                             double*, int64_t, size_t, int,
                                             const TriClusterShape&, bool, cudaStream_t);
template cudaError_t tridiag_cluster<zdbl>(const zdbl*, int, double*, double*, zdbl*, zdbl*,
                                           int64_t, size_t, int, const TriClusterShape&, bool,
                                           cudaStream_t);

}  // namespace cbc
