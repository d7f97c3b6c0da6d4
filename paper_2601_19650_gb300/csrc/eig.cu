// FP64 Hermitian eigensolver for the truncation of Sec. III A / III B.
//
// The paper names an SVD as one way to compress the fused leg (Sec. III A).  The GPU path
// reaches the same truncation through the Gram matrix K = M M^H (or M^H M): its
// eigenvectors are the singular vectors of M and its eigenvalues the squared singular
// values, so keeping the k largest eigenpairs keeps the same subspace as the truncated
// SVD.  Stages:
//   1. Householder reduction to a real symmetric tridiagonal T = Q^H K Q by one group
//      of CTAs that wait on each other (a thread-block cluster per matrix of a batch, else a
//      cooperative launch); rows of K are dealt round-robin to the CTAs so the shrinking
//      trailing block stays balanced.  FP64 work is spread over several SMs because one
//      GB300 SM retires only ~2 DFMA per clock.
//   2. Estimates of all eigenvalues of T by single-precision Sturm-count multisection,
//      one warp per eigenvalue (a dependent chain of FP64 divisions per Sturm step is
//      slow on this part; the estimates only need to separate the eigenvalues).
//   3. Eigenvectors of T for the candidates (the kmax largest) by FP64 inverse
//      iteration seeded with those estimates (one LU, four solves); eigenvalues =
//      Rayleigh quotients.  (The rank rule runs on the host, on weights measured on the
//      factor.)
//   4. Back transformation u = H_0 H_1 ... H_{m-2} x.
#include <float.h>

#include <algorithm>
#include <type_traits>

#include "df.cuh"
#include "isum.cuh"
#include "kernels.cuh"
#include "planner.h"

namespace cbc {
namespace {

constexpr int TPB = 256;

// p moved by `bytes` (the per-instance stride of a batched workspace)
template <typename P>
__host__ __device__ __forceinline__ P* byte_shift(P* p, size_t bytes) {
  return reinterpret_cast<P*>(reinterpret_cast<uintptr_t>(p) + bytes);
}

template <typename T>
__device__ __forceinline__ T ldcg(const T* p);
template <>
__device__ __forceinline__ double ldcg<double>(const double* p) {
  return __ldcg(p);
}
template <>
__device__ __forceinline__ zdbl ldcg<zdbl>(const zdbl* p) {
  double2 v = __ldcg(reinterpret_cast<const double2*>(p));
  return {v.x, v.y};
}

__device__ __forceinline__ double block_sum(double v, double* sh) {
  v = warp_sum(v);
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 32) {
    t = (threadIdx.x < (blockDim.x >> 5)) ? sh[threadIdx.x] : 0.0;
    t = warp_sum(t);
    if (threadIdx.x == 0) sh[0] = t;
  }
  __syncthreads();
  t = sh[0];
  __syncthreads();
  return t;
}

template <typename T>
struct TriArgs {
  T* A;
  int m;
  double* d;
  double* e;
  T* tau;
  T* V;     // (m-1) x m: row j = v_j (entries j+1 .. m-1, v_j[j+1] = 1)
  T* vbuf;  // 2 x m
  T* p;     // m
  double* dot;  // 2 x 2 (re, im) accumulators, double buffered
  GridBarrier* bar;
  int* status;
};

// Householder vector of column j (zlarfg convention: H = I - tau v v^H, H^H x = beta e_1,
// beta real), computed by the CTA that owns row j from its own (current) row.
template <typename T>
__device__ void householder_col(const TriArgs<T>& a, int j, double* sh) {
  using O = ops<T>;
  const int m = a.m;
  const T* row = a.A + (int64_t)j * m;
  // x_c = A[c][j] = conj(A[j][c]) for c > j
  double xn2 = 0.0;
  for (int c = j + 2 + threadIdx.x; c < m; c += blockDim.x) xn2 += O::abs2(row[c]);
  xn2 = block_sum(xn2, sh);
  T alpha = O::conj(row[j + 1]);
  double ar = O::real(alpha), ai = O::imag(alpha);
  T tau;
  double beta;
  T scale;
  bool trivial = (xn2 == 0.0 && ai == 0.0);
  if (trivial) {
    tau = O::zero();
    beta = ar;
    scale = O::zero();
  } else {
    double nrm = sqrt(ar * ar + ai * ai + xn2);
    beta = (ar >= 0.0) ? -nrm : nrm;
    const double ib = rcp64(beta);
    tau = O::make((beta - ar) * ib, -ai * ib);
    // scale = 1 / (alpha - beta)
    double zr = ar - beta, zi = ai;
    const double iden = rcp64(zr * zr + zi * zi);
    scale = O::make(zr * iden, -zi * iden);
  }
  T* vb = a.vbuf + (j & 1) * m;
  T* vs = a.V + (int64_t)j * m;
  for (int c = j + 1 + threadIdx.x; c < m; c += blockDim.x) {
    T v;
    if (c == j + 1)
      v = O::one();
    else
      v = trivial ? O::zero() : O::conj(row[c]) * scale;
    vb[c] = v;
    vs[c] = v;
  }
  if (threadIdx.x == 0) {
    a.tau[j] = tau;
    a.e[j] = beta;
    a.d[j] = O::real(row[j]);
    a.dot[(j & 1) * 2 + 0] = 0.0;
    a.dot[(j & 1) * 2 + 1] = 0.0;
  }
  __threadfence();
}

template <typename T>
__global__ void __launch_bounds__(TPB) tridiag_kernel(TriArgs<T> a) {
  using O = ops<T>;
  __shared__ double sh[64];
  const int m = a.m;
  const int P = gridDim.x, cta = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  if (m == 1) {
    if (cta == 0 && threadIdx.x == 0) a.d[0] = O::real(a.A[0]);
    return;
  }
  if (cta == 0) householder_col(a, 0, sh);
  if (!grid_sync(a.bar, a.status)) return;
  for (int j = 0; j < m - 1; ++j) {
    const T* v = a.vbuf + (j & 1) * m;
    const T tau = ldcg(a.tau + j);
    // ---- phase B: p_r = tau * sum_{c>j} A[r][c] v_c for own rows r > j
    // own rows: r = cta + P*t; the t-th own row goes to warp t % nw
    double dre = 0.0, dim = 0.0;
    int t0 = (j + 1 - cta + P - 1) / P;  // first t with cta + P t > j
    if (t0 < 0) t0 = 0;
    for (int t = t0 + warp; cta + P * t < m; t += nw) {
      int r = cta + P * t;
      const T* row = a.A + (int64_t)r * m;
      T acc = O::zero();
      for (int c = j + 1 + lane; c < m; c += 32) acc = O::fma(row[c], ldcg(v + c), acc);
      if constexpr (O::cplx) {
        acc = zdbl{warp_sum(O::real(acc)), warp_sum(O::imag(acc))};
      } else {
        acc = warp_sum(acc);
      }
      T pr = tau * acc;
      if (lane == 0) {
        a.p[r] = pr;
        T vd = O::conj(ldcg(v + r)) * pr;
        dre += O::real(vd);
        dim += O::imag(vd);
      }
    }
    dre = block_sum(dre, sh);
    if constexpr (O::cplx) dim = block_sum(dim, sh);
    if (threadIdx.x == 0) {
      atomicAdd(a.dot + (j & 1) * 2 + 0, dre);
      if constexpr (O::cplx) atomicAdd(a.dot + (j & 1) * 2 + 1, dim);
    }
    if (!grid_sync(a.bar, a.status)) return;
    // ---- phase C: A22 -= v w^H + w v^H, w = p - (conj(tau)/2) (v^H p) v
    T s = O::make(__ldcg(a.dot + (j & 1) * 2 + 0), __ldcg(a.dot + (j & 1) * 2 + 1));
    T coef = O::scale(-0.5, O::conj(tau) * s);
    for (int t = t0 + warp; cta + P * t < m; t += nw) {
      int r = cta + P * t;
      T* row = a.A + (int64_t)r * m;
      T vr = ldcg(v + r);
      T wr = O::fma(coef, vr, ldcg(a.p + r));
      for (int c = j + 1 + lane; c < m; c += 32) {
        T vc = ldcg(v + c);
        T wc = O::fma(coef, vc, ldcg(a.p + c));
        T upd = O::fma(vr, O::conj(wc), wr * O::conj(vc));
        row[c] = row[c] - upd;
      }
    }
    __syncthreads();
    if (j + 1 < m - 1) {
      if ((j + 1) % P == cta) householder_col(a, j + 1, sh);
    } else if ((m - 1) % P == cta && threadIdx.x == 0) {
      a.d[m - 1] = O::real(a.A[(int64_t)(m - 1) * m + (m - 1)]);
    }
    if (!grid_sync(a.bar, a.status)) return;
  }
}

// ---- tridiagonalisation of a lone matrix with the rows in shared memory ----------------
// For m <= 1024 with every CTA's rows r = cta + P t in its shared memory.  The reduction is
// a chain of m columns, and what bounds it is that chain: one exchange between the CTAs
// through L2 (~1600 clocks) and, on this part, ~64 clocks for every dependent FP64 operation
// and for every FP64 instruction of a warp.  So per column:
//   * one exchange.  Every CTA publishes A u for its own rows together with their entries of
//     the next column; every CTA then forms w and the next column x by itself, with the same
//     operations in the same order, so no Householder vector travels.  Both go out as plain
//     data into buffers filled with the all-ones bit pattern before the launch, each entry
//     written once with a relaxed store and polled until it differs from that pattern: no
//     fence, counter or atomic on the chain.  Every wait is bounded.
//   * the reflector unscaled, u = x - beta e_1 and H = I - gamma u u^H: only beta stands
//     between the norm and A u; gamma and the scaled vector for the back transformation are
//     formed while the exchange is under way.  u^H A u is real, so w = gamma A u + c u with a
//     real c = -|gamma|^2 (u^H A u) / 2.
//   * both sums over the block in integers: the terms are aligned to the largest one and
//     added exactly (no FP64 instruction, and the same value in every CTA);
//   * the rank-2 update of the rows while one warp computes beta.
// Two exchanges per column and FP64 sums / this: m = 256 complex 2.93 / 1.40 ms, 64 0.55 /
// 0.26 ms, 512 real 5.29 / 3.00 ms, 1000 real 13.7 / 9.0 ms.
template <typename T>
struct Tri2Args {
  const T* A;
  int m;
  double* d;
  double* e;
  T* tau;
  T* V;    // m x m; row j: [j+1, m) = v_j
  T* X;    // m x m pairs; row j: [j+1, m) = (A u_j, column j+1 before its update by u_j);
           // sentinel-filled before the launch
  int* status;
};

constexpr long long kSentinel = -1LL;  // all bits set: a NaN that arithmetic never yields
constexpr long long kWaitCycles = 4000000000LL;
constexpr int kLoneMaxM = 1024;

__device__ __forceinline__ double pub_value(double x) {
  return (__double_as_longlong(x) == kSentinel) ? __longlong_as_double(0x7ff8000000000000LL) : x;
}
__device__ __forceinline__ void st_pub(double* p, double v) {
  asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(p), "d"(pub_value(v)) : "memory");
}
__device__ __forceinline__ void st_pub(zdbl* p, zdbl v) {
  asm volatile("st.relaxed.gpu.global.v2.f64 [%0], {%1, %2};" ::"l"(p), "d"(pub_value(v.re)),
               "d"(pub_value(v.im))
               : "memory");
}
__device__ __forceinline__ bool ld_pub(const double* p, double* v) {
  double x;
  asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(x) : "l"(p) : "memory");
  *v = x;
  return __double_as_longlong(x) != kSentinel;
}
__device__ __forceinline__ bool ld_pub(const zdbl* p, zdbl* v) {
  double x, y;
  asm volatile("ld.relaxed.gpu.global.v2.f64 {%0, %1}, [%2];" : "=d"(x), "=d"(y) : "l"(p) : "memory");
  *v = zdbl{x, y};
  return __double_as_longlong(x) != kSentinel && __double_as_longlong(y) != kSentinel;
}

// N pairs of published values at p[i] (skipped where p[i] is NULL), all loads in flight
// together; false when the wait ran out or another CTA has reported an error
template <typename T, int N>
__device__ __forceinline__ bool wait_pairs(const T* const (&p)[N], T (&y)[N], T (&z)[N],
                                           int* status) {
  bool all = true;
#pragma unroll
  for (int i = 0; i < N; ++i)
    if (p[i]) {
      const bool a = ld_pub(p[i], &y[i]), b = ld_pub(p[i] + 1, &z[i]);
      all = all && a && b;
    }
  if (all) return true;
  const long long t0 = clock64();
  while (true) {
    all = true;
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (p[i]) {
        const bool a = ld_pub(p[i], &y[i]), b = ld_pub(p[i] + 1, &z[i]);
        all = all && a && b;
      }
    if (all) return true;
    if (*((volatile int*)status) != 0) return false;
    if (clock64() - t0 > kWaitCycles) {
      set_status(status, CBC_ERR_TIMEOUT);
      return false;
    }
  }
}

// the sum of x over the warp's lanes: every lane for a real x; for a complex one lane 0 holds
// the real part and lane 16 the imaginary part (one FP64 addition per level either way)
__device__ __forceinline__ double warp_sum_parts(double x) { return warp_sum(x); }
__device__ __forceinline__ double warp_sum_parts(zdbl x) {
  const bool up = threadIdx.x & 16;
  double v = (up ? x.im : x.re) + __shfl_xor_sync(0xffffffffu, up ? x.re : x.im, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// NE: columns per thread (m <= 256 NE)
template <typename T, int NE>
__global__ void __launch_bounds__(TPB) tridiag_lone_kernel(Tri2Args<T> a) {
  using O = ops<T>;
  constexpr int NW = TPB / 32, NC = O::cplx ? 2 : 1;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  __shared__ WarpSum s_norm[NW], s_dot[NW];
  __shared__ double s_acc[NW][NW][NC];
  __shared__ double s_beta, s_ib;
  __shared__ T s_typ;
  const int P = gridDim.x, cta = blockIdx.x, m = a.m;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nr = (m - cta + P - 1) / P;  // own rows r = cta + P t
  T* rows = reinterpret_cast<T*>(sm_raw);
  T* ubuf = rows + (size_t)((m + P - 1) / P) * m;  // u of this column and of the one before
  T* wsm = ubuf + 2 * (size_t)m;                   // w of the one before
  for (int t = 0; t < nr; ++t)
    for (int c = tid; c < m; c += TPB) rows[(size_t)t * m + c] = a.A[(int64_t)(cta + P * t) * m + c];
  T x[NE];  // column k of the current matrix at rows c = tid + 256 i
#pragma unroll
  for (int i = 0; i < NE; ++i) {
    const int c = tid + TPB * i;
    x[i] = c < m ? a.A[(int64_t)c * m] : O::zero();
  }
  for (int k = 0;; ++k) {
    T* u = ubuf + (size_t)(k & 1) * m;
    const T* up = ubuf + (size_t)((k & 1) ^ 1) * m;
    double part = 0.0;
#pragma unroll
    for (int i = 0; i < NE; ++i) {
      const int c = tid + TPB * i;
      if (c >= k && c < m) {
        u[c] = x[i];
        if (c == k && cta == 0) a.d[k] = O::real(x[i]);
        if (c >= k + 2) {
          if constexpr (O::cplx)
            part = fma(x[i].re, x[i].re, fma(x[i].im, x[i].im, part));
          else
            part = fma(x[i], x[i], part);
        }
      }
    }
    if (k == m - 1) break;
    {
      const WarpSum s = warp_isum(part);
      if (lane == 0) s_norm[warp] = s;
    }
    __syncthreads();
    const int t0 = (k + 1 > cta) ? (k + 1 - cta + P - 1) / P : 0;  // first own row beyond k
    if (warp == 0) {  // beta, and u's first entry alpha - beta
      const double xn2 = block_isum<NW>(s_norm);
      const T alpha = u[k + 1];
      const double ar = O::real(alpha), ai = O::imag(alpha);
      // xn2 = 0 and alpha real: H is the identity (tests on the bits: an FP64 comparison costs
      // as much as an addition)
      double beta = ar, ib = 0.0, z = 0.0;
      const double n2 = O::cplx ? fma(ar, ar, fma(ai, ai, xn2)) : fma(ar, ar, xn2);
      const bool rest = __double_as_longlong(xn2) != 0ll ||
                        (__double_as_longlong(ai) & 0x7fffffffffffffffll) != 0ll;
      if (rest && __double_as_longlong(n2) != 0ll) {
        const double rn = rsqrt64_short(n2);  // 1 / ||x||
        const bool pos = __double2hiint(ar) >= 0;
        const double nrm = n2 * rn;
        beta = pos ? -nrm : nrm;
        ib = pos ? -rn : rn;
        z = ar - beta;
      }
      __syncwarp();
      if (lane == 0) {
        u[k + 1] = O::make(z, rest ? ai : 0.0);
        s_beta = beta;
        s_ib = ib;
      }
    } else if (k > 0 && (warp & 3)) {
      // meanwhile the update of column k-1, A -= u w^H + w u^H, by the warps that don't share
      // warp 0's FP64 unit
      for (int t = t0; t < nr; ++t) {
        T* row = rows + (size_t)t * m;
        const int r = cta + P * t;
        const T nu = O::scale(-1.0, up[r]), nw = O::scale(-1.0, wsm[r]);
        for (int c = k + 1 + (warp - 1 - (warp >> 2)) * 32 + lane; c < m; c += 6 * 32)
          row[c] = O::fma(nw, O::conj(up[c]), O::fma(nu, O::conj(wsm[c]), row[c]));
      }
    }
    __syncthreads();
    // A u for the own rows: S warps per row
    const int live = nr - t0;
    T* xg = a.X + (int64_t)k * m * 2;
    int S = NW;
    while (S > 1 && (S * live > NW || 32 * S >= 2 * (m - k - 1))) S >>= 1;
    for (int l0 = 0; l0 < live; l0 += NW / S) {
      const int li = l0 + warp / S, seg = warp % S;
      if (li < live) {
        const T* row = rows + (size_t)(t0 + li) * m;
        T acc = O::zero();
        for (int c = k + 1 + seg * 32 + lane; c < m; c += S * 32) acc = O::fma(row[c], u[c], acc);
        const double v = warp_sum_parts(acc);
        const int r = cta + P * (t0 + li);
        if (seg == 0 && lane == 1) st_pub(xg + 2 * r + 1, row[k + 1]);
        if ((lane & 15) == 0 && lane < 16 * NC) {
          if (S == 1)
            st_pub(reinterpret_cast<double*>(xg + 2 * r) + (lane >> 4), v);
          else
            s_acc[li][seg][lane >> 4] = v;
        }
      }
    }
    if (S > 1) {  // (then S live <= NW: all rows were done in one round)
      __syncthreads();
      if (tid < live * NC) {
        const int li = tid / NC, q = tid % NC;
        double v = s_acc[li][0][q];
        for (int s = 1; s < S; ++s) v += s_acc[li][s][q];
        st_pub(reinterpret_cast<double*>(xg + 2 * (cta + P * (t0 + li))) + q, v);
      }
    }
    // while the others' rows arrive: gamma = -1 / (beta conj(alpha - beta)), tau and the
    // scaled reflector of the own rows for the back transformation
    const T up0 = u[k + 1];
    const double zr = O::real(up0), zi = O::imag(up0), ib = s_ib;
    T gamma = O::zero(), scale = O::zero();
    if (ib != 0.0) {
      const double iden = rcp64(O::cplx ? fma(zr, zr, zi * zi) : zr * zr);
      const double f = -ib * iden;
      gamma = O::make(zr * f, zi * f);
      scale = O::make(zr * iden, -zi * iden);  // 1 / (alpha - beta)
    }
    if (tid >= TPB - 32) {
      for (int t = t0 + lane; t < nr; t += 32) {
        const int r = cta + P * t;
        a.V[(int64_t)k * m + r] = (r == k + 1) ? O::one() : u[r] * scale;
      }
      if (cta == 0 && lane == 31) {
        a.tau[k] = O::make(-zr * ib, -zi * ib);
        a.e[k] = s_beta;
      }
    }
    T ty[NE], col[NE];
    double dp = 0.0;
    bool ok;
    {
      const T* src[NE];
#pragma unroll
      for (int i = 0; i < NE; ++i) {
        const int c = tid + TPB * i;
        src[i] = (c > k && c < m) ? xg + 2 * c : nullptr;
        ty[i] = col[i] = O::zero();
      }
      ok = wait_pairs<T, NE>(src, ty, col, a.status);
#pragma unroll
      for (int i = 0; i < NE; ++i) {
        const int c = tid + TPB * i;
        if (src[i]) {
          const T uc = u[c], y = ty[i];
          if constexpr (O::cplx)
            dp = fma(uc.re, y.re, fma(uc.im, y.im, dp));
          else
            dp = fma(uc, y, dp);
          ty[i] = gamma * y;
          if (c == k + 1) s_typ = ty[i];
        }
      }
    }
    {
      const WarpSum s = warp_isum(dp);
      if (lane == 0) s_dot[warp] = s;
    }
    if (!__syncthreads_and(ok)) return;
    const double dot = block_isum<NW>(s_dot);
    const double gr = O::real(gamma), gi = O::imag(gamma);
    const double cf = O::cplx ? -0.5 * fma(gr, gr * dot, gi * (gi * dot)) : -0.5 * (gr * (gr * dot));
    // w = gamma A u + c u, and column k+1 after the update: x - u conj(w_{k+1}) - w conj(u_{k+1})
    const T nwc = O::conj(s_typ + O::scale(cf, up0)), nuc = O::conj(up0);
#pragma unroll
    for (int i = 0; i < NE; ++i) {
      const int c = tid + TPB * i;
      if (c > k && c < m) {
        const T uc = u[c];
        T w;
        if constexpr (O::cplx)
          w = zdbl{fma(cf, uc.re, ty[i].re), fma(cf, uc.im, ty[i].im)};
        else
          w = fma(cf, uc, ty[i]);
        wsm[c] = w;
        x[i] = O::fma(-w, nuc, O::fma(-uc, nwc, col[i]));
      }
    }
  }
}

// ---- eigenvalues of T: single-precision multisection, one warp per eigenvalue --------
// The values only seed the shifts of the FP64 inverse iteration below, whose Rayleigh
// quotients are the eigenvalues used for the rank rule.  T is scaled by a power of two to
// entries below 1, so any norm fits FP32.
__device__ __forceinline__ int sturm32(const float* dd, const float* e2, int m, float x,
                                       float pivmin) {
  int cnt = 0;
  float q = dd[0] - x;
  if (q < 0.f) cnt++;
  for (int i = 1; i < m; ++i) {
    if (fabsf(q) < pivmin) q = -pivmin;
    q = (dd[i] - x) - __fdividef(e2[i - 1], q);
    if (q < 0.f) cnt++;
  }
  return cnt;
}

// lam32: eigenvalues / *scale, descending; lam[j] for j >= kmax (the estimates that the
// caller gets; the first kmax come from the inverse iteration)
__global__ void bisect32_kernel(const double* d, const double* e, int m, int kmax, float* lam32,
                                double* scale, double* lam, size_t wb) {
  extern __shared__ float shf[];
  d = byte_shift(d, blockIdx.y * wb);  // matrix blockIdx.y of a batch
  e = byte_shift(e, blockIdx.y * wb);
  lam32 = byte_shift(lam32, blockIdx.y * wb);
  scale = byte_shift(scale, blockIdx.y * wb);
  lam += (size_t)blockIdx.y * m;
  float* dd = shf;
  float* e2 = shf + m;
  __shared__ int s_exp;
  __shared__ double s_lo[32], s_hi[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (threadIdx.x == 0) s_exp = 0;
  __syncthreads();
  auto field = [](double x) { return ((unsigned)__double2hiint(x) >> 20) & 0x7ffu; };
  unsigned ex = 0;
  for (int i = threadIdx.x; i < m; i += blockDim.x)
    ex = max(ex, max(field(d[i]), i < m - 1 ? field(e[i]) : 0u));
  ex = __reduce_max_sync(0xffffffffu, ex);
  if (lane == 0) atomicMax(&s_exp, (int)ex);
  __syncthreads();
  const int E = min(s_exp, 2044);
  const double inv = __hiloint2double((2045 - E) << 20, 0), sc = __hiloint2double((E + 1) << 20, 0);
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    dd[i] = (float)(d[i] * inv);
    const double ei = (i < m - 1) ? e[i] * inv : 0.0;
    e2[i] = (float)(ei * ei);
  }
  // Gershgorin's bounds and the squares are formed in FP64 and rounded once: the estimates are
  // points of the grid that the bounds span, to FP32 accuracy, and move with them
  double glo = DBL_MAX, ghi = -DBL_MAX;
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    double r = 0.0;
    if (i > 0) r += fabs(e[i - 1] * inv);
    if (i < m - 1) r += fabs(e[i] * inv);
    glo = fmin(glo, d[i] * inv - r);
    ghi = fmax(ghi, d[i] * inv + r);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    glo = fmin(glo, __shfl_xor_sync(0xffffffffu, glo, o));
    ghi = fmax(ghi, __shfl_xor_sync(0xffffffffu, ghi, o));
  }
  if (lane == 0) {
    s_lo[warp] = glo;
    s_hi[warp] = ghi;
  }
  __syncthreads();
  for (int w = 0; w < nw; ++w) {
    glo = fmin(glo, s_lo[w]);
    ghi = fmax(ghi, s_hi[w]);
  }
  const double span = fmax(fabs(glo), fabs(ghi));
  float lo = (float)(glo - 1e-6 * span) - FLT_MIN, hi = (float)(ghi + 1e-6 * span) + FLT_MIN;
  __syncthreads();
  if (blockIdx.x == 0 && threadIdx.x == 0) *scale = sc;
  const int jj = blockIdx.x * nw + warp;  // descending index
  if (jj >= m) return;
  const int target = m - 1 - jj;
  for (int round = 0; round < 12; ++round) {
    const float x = lo + (hi - lo) * (float)(lane + 1) * (1.f / 33.f);
    const int cnt = sturm32(dd, e2, m, x, FLT_MIN);
    const unsigned bits = __ballot_sync(0xffffffffu, cnt <= target);
    const int nle = __popc(bits);
    const float xl = __shfl_sync(0xffffffffu, x, max(nle - 1, 0));
    const float xh = __shfl_sync(0xffffffffu, x, min(nle, 31));
    if (nle > 0) lo = xl;
    if (nle < 32) hi = xh;
    if (hi - lo <= 2e-7f * fmaxf(fabsf(lo), fabsf(hi)) + FLT_MIN) break;
  }
  if (lane == 0) {
    const float v = 0.5f * (lo + hi);
    lam32[jj] = v;
    if (jj >= kmax) lam[jj] = (double)v * sc;
  }
}

// ---- eigenvectors of T by FP64 inverse iteration ----------------------------------
// One LU of T - sigma I and four solves per candidate, in T's scaled units.  The chain of
// dependent FP64 operations (~64 clocks each, and as many for every FP64 instruction a warp
// issues) is the cost, so
//   * the elimination runs from both ends of T to the middle, one lane per half, which
//     halves the chain: the two halves meet in a 2 x 2 system;
//   * partial pivoting without a branch: 7 FP64 operations per row and factorisation, 4 per
//     row and solve (pivots kept as reciprocals, U scaled by them);
//   * no normalisation between the solves: T has entries below 1 and a pivot is at least
//     2^-52 of its span, so four solves grow a vector by
//     less than 2^250;
//   * norms, Rayleigh quotients and orthogonalisation by all lanes of the warp.
// A candidate whose single-precision eigenvalue is separated from its neighbours by more
// than 1e-4 of the spectral radius stands alone; a run of closer candidates is a cluster
// that one warp iterates as a block, orthonormalising after every solve.
// One thread per candidate from the top, and the clusters in a kernel behind / this: 128
// candidates of m = 256 0.52 / 0.19 ms, 64 such matrices 2.7 / 1.0 ms; 1024 of m = 2048 31 /
// 5.9 ms.
__device__ __forceinline__ uint32_t hash32(uint32_t x) {
  x ^= x >> 16;
  x *= 0x7feb352dU;
  x ^= x >> 15;
  x *= 0x846ca68bU;
  x ^= x >> 16;
  return x;
}

struct InvArgs {
  const double* d;
  const double* e;
  const float* lam32;   // descending, in scaled units
  const double* scale;
  int m;
  int kmax;             // candidates j < kmax
  double* X;            // m x kmax (row i, column j)
  double* lam;          // [m] per matrix: lam[j], j < kmax, Rayleigh quotients
  size_t wb;            // workspace bytes between the matrices of a batch (blockIdx.y)
  int per;              // lone candidates per warp
  int cper;             // members of a cluster iterated together
  int nclu;             // the first nclu CTAs of a matrix take its clusters, round robin
  int staged;           // scaled d and e in shared memory
};

constexpr int kInvMax = 16;  // members per warp: two lanes each

// The state of one warp: member t on lanes 2t (rows 0, 1, ... of T) and 2t + 1 (rows m-1,
// m-2, ...).  Row p of a half is element [p * ld + lane] of the arrays.  Lanes without a member
// (act false, n = 1: no rows to walk) take part in the shuffles and touch no shared column:
// the solves work in place, so only the lane that owns a column may read or write it.
struct Inv {
  double *f, *r, *u1, *u2, *b;  // multipliers (last bit: rows swapped), 1/pivot, U's
                                // superdiagonals / pivot, the vector
  const double *d, *e;
  double inv;                   // factor from d, e to scaled units (1 if they are scaled)
  int m, h, n, ld, lane;        // h rows in the upper half, n in this lane's
  bool act, top, swap;
  double r1, f1, a2, r2;        // the factored 2 x 2 system in the middle

  __device__ double D(int p) const { return d[top ? p : m - 1 - p] * inv; }
  // the coupling of row p of the half to its next one (of the last row: to the other half)
  __device__ double E(int p) const { return e[top ? p : m - 2 - p] * inv; }
  __device__ double* at(int i, int t) const {  // element i of member t's vector
    return b + (i < h ? (size_t)i * ld + 2 * t : (size_t)(m - 1 - i) * ld + 2 * t + 1);
  }
  static __device__ bool less_abs(double x, double y) {  // |x| < |y| on the bits
    return (__double_as_longlong(x) & 0x7fffffffffffffffll) <
           (__double_as_longlong(y) & 0x7fffffffffffffffll);
  }
  static __device__ double guard(double x, double tiny) {
    return less_abs(x, tiny) ? __hiloint2double(__double2hiint(tiny) | (__double2hiint(x) & 0x80000000),
                                                __double2loint(tiny))
                             : x;
  }

  __device__ void factor(double sigma, double tiny) {
    double dc = D(0) - sigma, uc = m > 1 ? E(0) : 0.0;
    for (int p = 0; p < n - 1; ++p) {
      const double li = E(p), dn = D(p + 1) - sigma, un = E(p + 1);
      const bool sw = less_abs(dc, li);
      const double rp = rcp64(guard(sw ? li : dc, tiny));
      const double num = sw ? dc : li, A = sw ? dn : uc, B = sw ? un : 0.0, C = sw ? uc : dn;
      double mult = num * rp;
      mult = __longlong_as_double((__double_as_longlong(mult) & ~1ll) | (sw ? 1ll : 0ll));
      const size_t o = (size_t)p * ld + lane;
      f[o] = mult;
      r[o] = rp;
      u1[o] = A * rp;
      u2[o] = B * rp;
      dc = fma(-mult, A, C);
      const double g = -mult * un;
      uc = sw ? g : un;
    }
    // the last rows of both halves: dT x_T + uT x_B = b_T, uB x_T + dB x_B = b_B
    const double dp = __shfl_xor_sync(0xffffffffu, dc, 1), upn = __shfl_xor_sync(0xffffffffu, uc, 1);
    const double dT = top ? dc : dp, uT = top ? uc : upn, dB = top ? dp : dc, uB = top ? upn : uc;
    swap = less_abs(dT, uB);
    a2 = swap ? dB : uT;
    r1 = rcp64(guard(swap ? uB : dT, tiny));
    f1 = (swap ? dT : uB) * r1;
    r2 = rcp64(guard(fma(-f1, a2, swap ? uT : dB), tiny));
  }

  __device__ void solve() {
    double carry = act ? b[lane] : 0.0;
    int p = 0;
    for (; p + 4 <= n - 1; p += 4) {  // four rows' operands in flight
      double fl[4], nx[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        fl[q] = f[(size_t)(p + q) * ld + lane];
        nx[q] = b[(size_t)(p + q + 1) * ld + lane];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const bool sw = __double_as_longlong(fl[q]) & 1;
        const double y = sw ? nx[q] : carry;
        carry = fma(-fl[q], y, sw ? carry : nx[q]);
        b[(size_t)(p + q) * ld + lane] = y;
      }
    }
    for (; p < n - 1; ++p) {
      const double fl = f[(size_t)p * ld + lane], nx = b[(size_t)(p + 1) * ld + lane];
      const bool sw = __double_as_longlong(fl) & 1;
      const double y = sw ? nx : carry;
      carry = fma(-fl, y, sw ? carry : nx);
      b[(size_t)p * ld + lane] = y;
    }
    const double cp = __shfl_xor_sync(0xffffffffu, carry, 1);
    const double bT = top ? carry : cp, bB = top ? cp : carry;
    const double c1 = swap ? bB : bT, c2 = swap ? bT : bB;
    const double xB = fma(-f1, c1, c2) * r2;
    const double xT = fma(-a2, xB, c1) * r1;
    double x1 = top ? xT : xB, x2 = top ? xB : xT;
    if (act) b[(size_t)(n - 1) * ld + lane] = x1;
    p = n - 2;
    for (; p >= 3; p -= 4) {
      double y[4], v1[4], v2[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const size_t o = (size_t)(p - q) * ld + lane;
        y[q] = b[o] * r[o];
        v1[q] = u1[o];
        v2[q] = u2[o];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const double x = fma(-v1[q], x1, fma(-v2[q], x2, y[q]));
        b[(size_t)(p - q) * ld + lane] = x;
        x2 = x1;
        x1 = x;
      }
    }
    for (; p >= 0; --p) {
      const size_t o = (size_t)p * ld + lane;
      const double x = fma(-u1[o], x1, fma(-u2[o], x2, b[o] * r[o]));
      b[o] = x;
      x2 = x1;
      x1 = x;
    }
  }

  // ---- by the whole warp, over the elements of one member's vector ----
  __device__ void start(int t, int j) {
    const int ln = threadIdx.x & 31;
    for (int i = ln; i < m; i += 32) {
      const uint32_t hsh = hash32((uint32_t)(i * 7919 + j * 104729 + 17));
      *at(i, t) = ((double)(hsh & 0xffffff) / 16777216.0) - 0.5;
    }
  }
  __device__ double norm2(int t) const {
    double s = 0.0;
    for (int i = threadIdx.x & 31; i < m; i += 32) {
      const double x = *at(i, t);
      s = fma(x, x, s);
    }
    return warp_sum(s);
  }
  __device__ void scale_by(int t, double f) {
    for (int i = threadIdx.x & 31; i < m; i += 32) *at(i, t) *= f;
  }
  // Rayleigh quotient of member t's vector (in T's own units) and the unit vector as column j
  __device__ void finish(const InvArgs& a, int t, int j, double sc) {
    const int ln = threadIdx.x & 31;
    double s = 0.0, q = 0.0;
    for (int i = ln; i < m; i += 32) {
      const double x = *at(i, t);
      double tx = (d[i] * inv) * x;
      if (i + 1 < m) tx = fma(2.0 * inv * e[i], *at(i + 1, t), tx);
      q = fma(x, tx, q);
      s = fma(x, x, s);
    }
    s = warp_sum(s);
    q = warp_sum(q);
    const double rn = (s > 0.0) ? rsqrt64_short(s) : 0.0;
    for (int i = ln; i < m; i += 32) a.X[(size_t)i * a.kmax + j] = *at(i, t) * rn;
    if (ln == 0) a.lam[j] = (q * rn * rn) * sc;
  }
};

// Each solve shrinks the components along eigenvectors at distance delta by about
// |lambda - sigma| / delta with |lambda - sigma| ~ 1e-7 span (single-precision shifts);
// four solves reach FP64 accuracy for delta >= 1e-4 span.  Candidates closer than that
// to a neighbour form a cluster.
__device__ __forceinline__ bool close_pair(const float* lam32, int j, double ortol) {
  return (double)lam32[j] - (double)lam32[j + 1] <= ortol;  // descending
}

// One cluster [jj, cend) by the warp, cper members at a time, iterated as a block (block
// inverse iteration): every member solves with its own shift (shifts at least 1e-10 span
// apart), then the block is orthonormalised (modified Gram-Schmidt) against the cluster's
// finished columns and within itself, four times.  The vectors then span the invariant
// subspace of the cluster's eigenvalues (any basis of it is a valid set of eigenvectors
// when they are not resolved individually).
__device__ void invit_cluster(const InvArgs& a, Inv& w, int jj, int cend, double span, double tiny,
                              double sc) {
  const int m = a.m, K = a.kmax, ln = threadIdx.x & 31;
  for (int j0 = jj; j0 < cend; j0 += a.cper) {
    const int nact = min(a.cper, cend - j0);
    const int j = j0 + min(w.lane >> 1, nact - 1);
    double sigma = (double)a.lam32[jj];
    for (int q = jj + 1; q <= j; ++q) sigma = fmin((double)a.lam32[q], sigma - 1e-10 * span);
    w.factor(sigma, tiny);
    for (int t = 0; t < nact; ++t) w.start(t, j0 + t);
    __syncwarp();
    for (int it = 0; it < 4; ++it) {
      w.solve();
      __syncwarp();
      for (int t = 0; t < nact; ++t) {
        const double s = w.norm2(t);
        w.scale_by(t, s > 0.0 ? rsqrt64_short(s) : 0.0);
      }
      __syncwarp();
      for (int t = 0; t < nact; ++t) {
        for (int q = jj; q < j0 + t; ++q) {  // the finished columns, then the block's earlier ones
          const bool fin = q < j0;
          double dv = 0.0;
          for (int i = ln; i < m; i += 32)
            dv = fma(fin ? a.X[(size_t)i * K + q] : *w.at(i, q - j0), *w.at(i, t), dv);
          dv = warp_sum(dv);
          for (int i = ln; i < m; i += 32) {
            double* x = w.at(i, t);
            *x = fma(-dv, fin ? a.X[(size_t)i * K + q] : *w.at(i, q - j0), *x);
          }
        }
        const double s = w.norm2(t);
        w.scale_by(t, s > 0.0 ? rsqrt64_short(s) : 0.0);
        __syncwarp();
      }
    }
    for (int t = 0; t < nact; ++t) w.finish(a, t, j0 + t, sc);
    __syncwarp();
  }
}

__global__ void __launch_bounds__(32) invit_kernel(InvArgs a) {
  extern __shared__ double shd[];
  {
    const size_t off = blockIdx.y * a.wb;
    a.d = byte_shift(a.d, off);
    a.e = byte_shift(a.e, off);
    a.lam32 = byte_shift(a.lam32, off);
    a.scale = byte_shift(a.scale, off);
    a.X = byte_shift(a.X, off);
    a.lam += (size_t)blockIdx.y * a.m;
  }
  const int m = a.m, K = a.kmax, ln = threadIdx.x;
  const double sc = *a.scale;  // a power of two
  const double inv = __hiloint2double((2046 << 20) - __double2hiint(sc), 0);
  const bool clusters = (int)blockIdx.x < a.nclu;
  const int per = clusters ? a.cper : a.per;
  Inv w;
  w.m = m;
  w.h = (m + 1) / 2;
  w.ld = 2 * per + (per >= 8 ? 1 : 0);  // odd rows where the whole warp walks a column
  w.act = ln < 2 * per;
  w.lane = w.act ? ln : (ln & 1);
  w.top = !(w.lane & 1);
  w.n = !w.act ? 1 : (w.top ? w.h : m - w.h);
  const size_t sz = (size_t)w.h * w.ld;
  w.f = shd;
  w.r = w.f + sz;
  w.u1 = w.r + sz;
  w.u2 = w.u1 + sz;
  w.b = w.u2 + sz;
  w.d = a.d;
  w.e = a.e;
  w.inv = inv;
  if (a.staged) {
    double* sd = w.b + sz;
    double* se = sd + m;
    for (int i = ln; i < m; i += 32) {
      sd[i] = a.d[i] * inv;
      se[i] = (i < m - 1) ? a.e[i] * inv : 0.0;
    }
    w.d = sd;
    w.e = se;
    w.inv = 1.0;
    __syncwarp();
  }
  if (m == 1) {
    if (ln == 0 && blockIdx.x == gridDim.x - 1) {
      a.X[0] = 1.0;
      a.lam[0] = a.d[0];
    }
    return;
  }
  const double span = fmax(fabs((double)a.lam32[0]), fabs((double)a.lam32[m - 1])) + DBL_MIN;
  const double ortol = 1e-4 * span;
  const double tiny = 2.220446049250313e-16 * span;
  if (clusters) {
    // clusters blockIdx.x, blockIdx.x + nclu, ... in order (a run of two or more candidates
    // whose neighbours are close)
    int cidx = -1;
    for (int jj = 0; jj + 1 < K;) {
      if (!close_pair(a.lam32, jj, ortol)) {
        ++jj;
        continue;
      }
      int cend = jj + 2;
      while (cend < K && close_pair(a.lam32, cend - 1, ortol)) ++cend;
      ++cidx;
      if (cidx % a.nclu == (int)blockIdx.x) invit_cluster(a, w, jj, cend, span, tiny, sc);
      jj = cend;
    }
    return;
  }
  // candidates j0 .. j0 + per - 1, the lone ones among them
  const int j0 = ((int)blockIdx.x - a.nclu) * per;
  const int nact = min(per, K - j0);
  auto lone = [&](int j) {
    return !((j > 0 && close_pair(a.lam32, j - 1, ortol)) ||
             (j + 1 < K && close_pair(a.lam32, j, ortol)));
  };
  bool any = false;
  for (int t = 0; t < nact; ++t) any = any || lone(j0 + t);
  if (!any) return;
  const int j = j0 + min(w.lane >> 1, nact - 1);
  w.factor((double)a.lam32[j], tiny);
  for (int t = 0; t < nact; ++t) w.start(t, j0 + t);
  __syncwarp();
  for (int it = 0; it < 4; ++it) w.solve();
  __syncwarp();
  for (int t = 0; t < nact; ++t)
    if (lone(j0 + t)) w.finish(a, t, j0 + t, sc);
}

// ---- back transformation: U[:, jj] = H_0 ... H_{m-2} X[:, jj] ------------------------
// One CTA of four warps per kept eigenvector (one warp per SM sub-partition, since a
// warp alone reaches only its own partition's FP64 unit).  Each reflector application
// is a dot product over the rows (per-warp partial sums combined through shared
// memory) and an axpy; the rows are split across the 128 threads.
template <typename T>
__global__ void __launch_bounds__(128) backtransform_kernel(const T* V, const T* tau,
                                                            const double* X, int m, int kmax,
                                                            T* U, size_t wb) {
  using O = ops<T>;
  extern __shared__ unsigned char smem_raw[];
  T* u = reinterpret_cast<T*>(smem_raw);
  __shared__ T part[2][4];
  // matrix blockIdx.y of a batch
  V = byte_shift(V, blockIdx.y * wb);
  tau = byte_shift(tau, blockIdx.y * wb);
  X = byte_shift(X, blockIdx.y * wb);
  U += (size_t)blockIdx.y * m * kmax;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int jj = blockIdx.x;
  for (int i = tid; i < m; i += 128) u[i] = O::make(X[(int64_t)i * kmax + jj], 0.0);
  __syncthreads();
  int par = 0;
  for (int j = m - 2; j >= 0; --j) {
    const T* vj = V + (int64_t)j * m;
    const T t = tau[j];
    T sacc = O::zero();
    // each thread owns rows r = tid (mod 128) for the whole loop, so u needs no barrier
    for (int r = tid; r < m; r += 128)
      if (r > j) sacc = O::fma(O::conj(vj[r]), u[r], sacc);
    if constexpr (O::cplx) {
      sacc = zdbl{warp_sum(O::real(sacc)), warp_sum(O::imag(sacc))};
    } else {
      sacc = warp_sum(sacc);
    }
    if (lane == 0) part[par][warp] = sacc;
    __syncthreads();
    const T tot = (part[par][0] + part[par][1]) + (part[par][2] + part[par][3]);
    const T ts = t * tot;
    for (int r = tid; r < m; r += 128)
      if (r > j) u[r] = u[r] - vj[r] * ts;
    par ^= 1;  // the next partial sums go to the other buffer: one barrier per reflector
  }
  __syncthreads();
  for (int i = tid; i < m; i += 128) U[(int64_t)i * kmax + jj] = u[i];
}

// Same back transformation with the lanes on the eigenvectors: a CTA takes 32 vectors
// (one per lane, held in shared memory as u[row][lane]) and 8 warps split the rows.
// Per reflector every lane sums conj(v_r) u_r over its warp's rows, the 8 partial sums
// meet in shared memory (one barrier), and every lane updates its rows.  No shuffle
// reductions and no half-empty warps: about a quarter of the FP64 instructions of the
// one-vector-per-CTA form.  u needs m * 32 elements of shared memory.
constexpr int BT_WARPS = 8;

// DF (mixed path, batches): u and the staged v as double-float pairs, the two O(m) loops
// per reflector in FP32 (the partial sums and tau * sum stay FP64).
template <typename T, bool DF>
__global__ void __launch_bounds__(32 * BT_WARPS) backtransform32_kernel(
    const T* V, const T* tau, const double* X, int m, int kmax, T* U, size_t wb) {
  using O = ops<T>;
  using D = typename dfof<T>::type;
  using E = typename std::conditional<DF, D, T>::type;  // element type of u and v in smem
  extern __shared__ unsigned char smem_raw[];
  E* u = reinterpret_cast<E*>(smem_raw);  // [m][32]
  E* vs = u + (size_t)m * 32;             // [3][m]: v_j in slot j % 3 (staged one ahead)
  // per-warp partial dots (double-float in the DF variant: the cross-warp sum and the
  // tau scaling then stay on the FP32 pipes, which every active warp repeats per reflector)
  __shared__ E part[2][BT_WARPS][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // matrix blockIdx.y of a batch
  V = byte_shift(V, blockIdx.y * wb);
  tau = byte_shift(tau, blockIdx.y * wb);
  X = byte_shift(X, blockIdx.y * wb);
  U += (size_t)blockIdx.y * m * kmax;
  const int c0 = blockIdx.x * 32;
  const int col = c0 + lane;
  const bool live = col < kmax;
  const int rb = (m + BT_WARPS - 1) / BT_WARPS;
  const int r0 = warp * rb, r1 = min(m, r0 + rb);
  auto to_e = [](const T& x) -> E {
    if constexpr (DF)
      return to_df(x);
    else
      return x;
  };
  for (int r = r0; r < r1; ++r)
    u[(size_t)r * 32 + lane] = to_e(O::make(live ? X[(int64_t)r * kmax + col] : 0.0, 0.0));
  if (m >= 2) {  // v_{m-2}: rows > m - 2
    const T* vg = V + (int64_t)(m - 2) * m;
    E* v0 = vs + (size_t)((m - 2) % 3) * m;
    for (int q = m - 1 + (int)threadIdx.x; q < m; q += blockDim.x) v0[q] = to_e(vg[q]);
  }
  __syncthreads();
  int par = 0;
  for (int j = m - 2; j >= 0; --j) {
    const E* v = vs + (size_t)(j % 3) * m;
    // partial dot over this warp's rows r > j, four independent accumulators
    const int rs = max(r0, j + 1);
    E psum;
    if constexpr (DF) {
      const D z = to_df(O::zero());
      D a0 = z, a1 = z, a2 = z, a3 = z;
      int r = rs;
      for (; r + 3 < r1; r += 4) {
        a0 = dff(dfconj(v[r]), u[(size_t)r * 32 + lane], a0);
        a1 = dff(dfconj(v[r + 1]), u[(size_t)(r + 1) * 32 + lane], a1);
        a2 = dff(dfconj(v[r + 2]), u[(size_t)(r + 2) * 32 + lane], a2);
        a3 = dff(dfconj(v[r + 3]), u[(size_t)(r + 3) * 32 + lane], a3);
      }
      for (; r < r1; ++r) a0 = dff(dfconj(v[r]), u[(size_t)r * 32 + lane], a0);
      psum = df_add(df_add(a0, a1), df_add(a2, a3));
    } else {
      T a0 = O::zero(), a1 = O::zero(), a2 = O::zero(), a3 = O::zero();
      int r = rs;
      for (; r + 3 < r1; r += 4) {
        a0 = O::fma(O::conj(v[r]), u[(size_t)r * 32 + lane], a0);
        a1 = O::fma(O::conj(v[r + 1]), u[(size_t)(r + 1) * 32 + lane], a1);
        a2 = O::fma(O::conj(v[r + 2]), u[(size_t)(r + 2) * 32 + lane], a2);
        a3 = O::fma(O::conj(v[r + 3]), u[(size_t)(r + 3) * 32 + lane], a3);
      }
      for (; r < r1; ++r) a0 = O::fma(O::conj(v[r]), u[(size_t)r * 32 + lane], a0);
      psum = (a0 + a1) + (a2 + a3);
    }
    part[par][warp][lane] = psum;
    // stage the next reflector's vector (rows > j - 1).  Its slot last held v_{j+2},
    // whose readers all finished before the barrier this warp passed last.
    if (j >= 1) {
      const T* vg = V + (int64_t)(j - 1) * m;
      E* vn = vs + (size_t)((j - 1) % 3) * m;
      for (int q = j + threadIdx.x; q < m; q += blockDim.x) vn[q] = to_e(vg[q]);
    }
    __syncthreads();
    if (rs < r1) {
      if constexpr (DF) {
        D tot = part[par][0][lane];
#pragma unroll
        for (int w = 1; w < BT_WARPS; ++w) tot = df_add(tot, part[par][w][lane]);
        const D ncf = df_neg(dff(to_df(tau[j]), tot, to_df(O::zero())));
        for (int q = rs; q < r1; ++q) u[(size_t)q * 32 + lane] = dff(v[q], ncf, u[(size_t)q * 32 + lane]);
      } else {
        T tot = part[par][0][lane];
#pragma unroll
        for (int w = 1; w < BT_WARPS; ++w) tot = tot + part[par][w][lane];
        const T cf = tau[j] * tot;
        for (int q = rs; q < r1; ++q) u[(size_t)q * 32 + lane] = u[(size_t)q * 32 + lane] - v[q] * cf;
      }
    }
    par ^= 1;
  }
  __syncthreads();
  if (live)
    for (int r = r0; r < r1; ++r) {
      if constexpr (DF)
        U[(int64_t)r * kmax + col] = from_df(u[(size_t)r * 32 + lane]);
      else
        U[(int64_t)r * kmax + col] = u[(size_t)r * 32 + lane];
    }
}

// ---- back transformation by matrix products -----------------------------------------
// Blocks of BT_NB reflectors in the compact WY form H_j0 .. H_{j0+b-1} = I - V T V^H (V: one
// column per reflector, T upper triangular), applied from the last block to the first,
// U <- U - (V T)(V^H U), with the products on the tensor cores (8 slices: an error below that
// of FP64 sums; U's columns may span any range here, since what counts is their norm).  One
// reflector at a time the transformation is a chain of m dot products, each ~3000 clocks of
// FP64 reductions, and FP64 work of 8 m^2 kmax flops on its pipes.
// One at a time / products, with the rest of the eigensolver behind the reduction: m = 2048
// complex, 1024 vectors 73.9 / 10.6 ms; 64 matrices of m = 256, 128 vectors 4.0 / 2.6 ms.
constexpr int BT_NB = 64, BT_HALF = 32;

// U = X (real) as nb matrices of n elements, X wb bytes apart
template <typename T>
__global__ void widen_x_kernel(const double* X, int64_t n, T* U, size_t wb) {
  X = byte_shift(X, blockIdx.y * wb);
  U += (int64_t)blockIdx.y * n;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    U[i] = ops<T>::make(X[i], 0.0);
}

// NaN into U (n elements) of every matrix blockIdx.y whose flag is set (an Inf or NaN among its
// V, T or X, which the slices don't carry)
template <typename T>
__global__ void poison_kernel(const int* flag, T* U, int64_t n) {
  if (!flag[blockIdx.y]) return;
  U += blockIdx.y * n;
  const double nan = __longlong_as_double(0x7ff8000000000000LL);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    U[i] = ops<T>::make(nan, ops<T>::cplx ? nan : 0.0);
}

// T of BT_HALF reflectors from G = V^H V (BT_HALF x BT_HALF, leading dimension BT_NB):
// T^-1 = diag(1 / tau) + the strict upper triangle of G, so column i of T is x_i = tau_i,
// x_r = -tau_r sum_{r < l <= i} G[r][l] x_l.  One CTA per half block (blockIdx.x: block and
// half, blockIdx.y: matrix), four lanes per column that share each sum.
template <typename T>
__global__ void __launch_bounds__(128) wy_t_kernel(const T* G, const T* tau, int m, T* Tm,
                                                   size_t wb, int64_t bs) {
  using O = ops<T>;
  __shared__ T g[BT_HALF][BT_HALF + 1];
  __shared__ T tt[BT_HALF];
  const int blk = blockIdx.x >> 1, half = blockIdx.x & 1;
  const int64_t at = blockIdx.y * bs + (int64_t)blk * BT_NB * BT_NB + half * BT_HALF * (BT_NB + 1);
  tau = byte_shift(tau, blockIdx.y * wb);
  G += at;
  Tm += at;
  for (int i = threadIdx.x; i < BT_HALF * BT_HALF; i += blockDim.x)
    g[i / BT_HALF][i % BT_HALF] = G[(int64_t)(i / BT_HALF) * BT_NB + i % BT_HALF];
  if (threadIdx.x < BT_HALF) {
    const int j = blk * BT_NB + half * BT_HALF + threadIdx.x;
    tt[threadIdx.x] = j < m - 1 ? tau[j] : O::zero();
  }
  __syncthreads();
  const int i = threadIdx.x >> 2, sub = threadIdx.x & 3;  // column i, terms l = sub (mod 4)
  T x[BT_HALF / 4];                                       // x_l, l = sub + 4 q
#pragma unroll
  for (int q = 0; q < BT_HALF / 4; ++q) x[q] = (sub + 4 * q == i) ? tt[i] : O::zero();
#pragma unroll
  for (int r = BT_HALF - 1; r >= 0; --r) {
    T acc = O::zero();
#pragma unroll
    for (int q = 0; q < BT_HALF / 4; ++q)
      if (4 * q + 3 > r) {
        const int l = sub + 4 * q;
        if (l > r) acc = O::fma(g[r][l], x[q], acc);
      }
    acc = acc + shfl_xor(acc, 1);
    acc = acc + shfl_xor(acc, 2);
    if (r < i && (r & 3) == sub) x[r >> 2] = O::scale(-1.0, tt[r] * acc);
  }
#pragma unroll
  for (int q = 0; q < BT_HALF / 4; ++q) Tm[(int64_t)(sub + 4 * q) * BT_NB + i] = x[q];
}

// Initial contents of a batch of eigensolver workspaces in one launch: up to 6 segments
// of 64-bit words per instance (instance blockIdx.y, workspaces wb bytes apart).
struct WsInit {
  unsigned long long* seg[6];
  int64_t words[6];
  unsigned long long val[6];
  int nseg;
  size_t wb;
};

__global__ void ws_init_kernel(WsInit a) {
  const size_t off = blockIdx.y * a.wb;
  for (int g = 0; g < a.nseg; ++g) {
    unsigned long long* p = byte_shift(a.seg[g], off);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < a.words[g];
         i += (int64_t)gridDim.x * blockDim.x)
      p[i] = a.val[g];
  }
}

}  // namespace

// workspace layout (all 256-byte aligned)
static size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

size_t eig_workspace_bytes(int m, int kmax, bool cplx) {
  size_t ts = cplx ? sizeof(zdbl) : sizeof(double);
  size_t b = 0;
  b += align256(sizeof(double) * m);                 // d
  b += align256(sizeof(double) * m);                 // e
  b += align256(sizeof(float) * m);                  // lam32
  b += align256(ts * m);                             // tau
  b += align256(ts * (size_t)m * m);                 // V
  b += align256(ts * 2 * m);                         // vbuf
  b += align256(ts * 2 * m);                         // p (two buffers)
  b += align256(sizeof(double) * 4);                 // dot
  b += align256(sizeof(double));                     // scale of T
  b += align256(sizeof(GridBarrier));                // barrier
  b += align256(sizeof(double) * (size_t)m * kmax);  // X
  b += align256(2 * ts * (size_t)m * m);             // exchange of the lone reduction
  return b;
}

// Where the products pay: they cost ~12 launches and ~70 us per block of 64 reflectors before
// the work counts, one reflector at a time costs ~1.9 us each.  One at a time / products, the
// eigensolver behind the reduction in us: lone m = 128 complex, 64 vectors 340 / 362; 256, 128
// vectors 722 / 588; 512 real, 256 vectors 1250 / 997; 64 matrices of m = 32 195 / 238, of 64
// 769 / 334; 5 of m = 97 real 214 / 344.
static bool bt_products(int m, int kmax, int nb) {
  return m >= 48 && (double)m * m * kmax * nb >= 4e6;
}

static size_t bt_gemm_bytes(int m, int kmax, bool cplx, int nb) {
  const int nblk = (m + BT_NB - 1) / BT_NB;
  const int rep = nb > 1 ? nb : nblk;  // the products on V alone: a block of all matrices, or
                                       // all blocks of a lone one
  size_t b = 0;
  auto need = [&](int M, int N, int K, int n) {
    b = std::max(b, gemm_tc_workspace_bytes(M, N, K, cplx, 8, n));
  };
  need(BT_NB, BT_NB, m, rep);                      // V^H V
  need(BT_HALF, BT_HALF, BT_HALF, nb * nblk);      // T
  need(m, BT_NB, BT_NB, rep);                      // V T
  need(BT_NB, kmax, m, nb);                        // V^H U
  need(m, kmax, BT_NB, nb);                        // (V T)(V^H U)
  return b;
}

size_t eig_bt_bytes(int m, int kmax, bool cplx, int nb) {
  if (!bt_products(m, kmax, nb)) return 0;
  const size_t ts = cplx ? sizeof(zdbl) : sizeof(double);
  const size_t nblk = (m + BT_NB - 1) / BT_NB;
  if (nb * nblk > TC_MAX_PROBLEMS) return 0;  // (the blocks' T are one call)
  return align256(sizeof(int) * nb) + align256(2 * nb * nblk * BT_NB * BT_NB * ts) +
         align256(nb * nblk * BT_HALF * BT_HALF * ts) + align256((size_t)nb * BT_NB * kmax * ts) +
         bt_gemm_bytes(m, kmax, cplx, nb);
}

// U = H_0 .. H_{m-2} X.  V (rows v_j, zero up to the diagonal), tau, X and Y (room for m rows
// more than m columns each) lie in the matrices' workspaces, wb bytes apart.
template <typename T>
static cudaError_t backtransform_products(const T* V, const T* tau, const double* X, T* Y, int m,
                                          int kmax, T* U, size_t wb, void* bt, int* status,
                                          cudaStream_t s, int nb) {
  const int nblk = (m + BT_NB - 1) / BT_NB;
  const int64_t we = (int64_t)(wb / sizeof(T)), sq = BT_NB * BT_NB, tbs = nblk * sq;
  char* w = static_cast<char*>(bt);
  auto take = [&](size_t bytes) {
    char* p = w;
    w += align256(bytes);
    return p;
  };
  int* flag = reinterpret_cast<int*>(take(sizeof(int) * nb));  // one per matrix
  T* G = reinterpret_cast<T*>(take(2 * nb * tbs * sizeof(T)));
  T* Tm = G + nb * tbs;
  T* tmp = reinterpret_cast<T*>(take(sizeof(T) * nb * nblk * BT_HALF * BT_HALF));
  T* W = reinterpret_cast<T*>(take(sizeof(T) * (size_t)nb * BT_NB * kmax));
  void* ws = w;
  TcWide opt;
  opt.wide = flag;
  TcWide sub = opt;
  sub.acc = -1;
  cudaError_t e = cudaMemsetAsync(bt, 0, (char*)(G + 2 * nb * tbs) - (char*)bt, s);  // flag, G, T
  // (n problems: one per matrix, all blocks of all matrices, or blocks of a lone one)
  auto mul = [&](int M, int N, int K, const T* A, View va, int64_t abs, bool ca, const T* B,
                 View vb, int64_t bbs, T* C, int64_t ldc, int64_t cbs, int n, TcWide o) {
    if (e != cudaSuccess) return;
    o.per = n / nb;
    va.bs = abs;
    vb.bs = bbs;
    e = gemm_tc<T>(M, N, K, A, va, ca, B, vb, false, C, View::rowmajor(ldc, cbs), 8, ws, status, s,
                   n, o);
  };
  const int64_t n = (int64_t)m * kmax;
  note_launches(CBC_K_EIG, 3);
  widen_x_kernel<T><<<dim3((unsigned)std::min<int64_t>(256, (n + 255) / 256), nb), 256, 0, s>>>(
      X, n, U, wb);
  // G = V^H V per block.  V's rows beyond m are not there: the last block has m - j0 of them
  const int full = m / BT_NB;  // blocks of BT_NB rows
  for (int q = 0; q < nblk; ++q) {
    const int j0 = q * BT_NB, b = std::min(BT_NB, m - j0);
    const bool all = nb == 1 && q == 0 && full > 1;  // a lone matrix: every full block at once
    const int64_t vbs = nb > 1 ? we : (int64_t)BT_NB * m, gbs = nb > 1 ? tbs : sq;
    const int c0 = all ? 0 : j0;  // v_j starts at column j + 1
    const T* Vb = V + (int64_t)j0 * m + c0;
    mul(b, b, m - c0, Vb, View::rowmajor(m), vbs, true, Vb, View::transposed(m), vbs,
        G + q * sq, BT_NB, gbs, nb > 1 ? nb : (all ? full : 1), opt);
    if (all) q = full - 1;
  }
  if (e != cudaSuccess) return e;
  wy_t_kernel<T><<<dim3(2 * nblk, nb), 128, 0, s>>>(G, tau, m, Tm, wb, tbs);
  // the halves of a block: T12 = -T1 (V1^H V2) T2
  const int64_t hf = BT_HALF * BT_HALF;
  mul(BT_HALF, BT_HALF, BT_HALF, G + BT_HALF, View::rowmajor(BT_NB), sq, false,
      Tm + BT_HALF * (BT_NB + 1), View::rowmajor(BT_NB), sq, tmp, BT_HALF, hf, nb * nblk, opt);
  mul(BT_HALF, BT_HALF, BT_HALF, Tm, View::rowmajor(BT_NB), sq, false, tmp,
      View::rowmajor(BT_HALF), hf, Tm + BT_HALF, BT_NB, sq, nb * nblk, sub);
  // Y = V T per block, m x BT_NB each
  const int64_t ybs = (int64_t)BT_NB * m;
  for (int q = 0; q < nblk; ++q) {
    const int j0 = q * BT_NB, b = std::min(BT_NB, m - j0);
    const bool all = nb == 1 && q == 0 && full > 1;
    const int c0 = all ? 0 : j0;
    mul(m - c0, BT_NB, b, V + (int64_t)j0 * m + c0, View::transposed(m), nb > 1 ? we : ybs, false,
        Tm + q * sq, View::rowmajor(BT_NB), nb > 1 ? tbs : sq, Y + q * ybs + (int64_t)c0 * BT_NB,
        BT_NB, nb > 1 ? we : ybs, nb > 1 ? nb : (all ? full : 1), opt);
    if (all) q = full - 1;
  }
  for (int q = nblk - 1; q >= 0; --q) {
    const int j0 = q * BT_NB, b = std::min(BT_NB, m - j0), r = m - j0;
    const T* Vb = V + (int64_t)j0 * m + j0;
    T* Ub = U + (int64_t)j0 * kmax;
    mul(b, kmax, r, Vb, View::rowmajor(m), we, true, Ub, View::rowmajor(kmax), n, W, kmax,
        (int64_t)BT_NB * kmax, nb, opt);
    mul(r, kmax, b, Y + q * ybs + (int64_t)j0 * BT_NB, View::rowmajor(BT_NB), we, false, W,
        View::rowmajor(kmax), (int64_t)BT_NB * kmax, Ub, kmax, n, nb, sub);
  }
  if (e != cudaSuccess) return e;
  poison_kernel<T><<<dim3((unsigned)std::min<int64_t>(256, (n + 255) / 256), nb), 256, 0, s>>>(
      flag, U, n);
  return cudaGetLastError();
}

template <typename T>
cudaError_t heev_top(T* A, int m, int kmax, double* lam, T* U, void* work, int* status,
                     int num_sms, cudaStream_t s, int nb, bool prefer_cluster, bool df, void* bt) {
  char* w = static_cast<char*>(work);
  auto take = [&](size_t bytes) {
    char* p = w;
    w += align256(bytes);
    return p;
  };
  const size_t ts = sizeof(T);
  const size_t wb = eig_workspace_bytes(m, kmax, ops<T>::cplx);  // per matrix
  double* d = (double*)take(sizeof(double) * m);
  double* e = (double*)take(sizeof(double) * m);
  float* lam32 = (float*)take(sizeof(float) * m);
  T* tau = (T*)take(ts * m);
  T* V = (T*)take(ts * (size_t)m * m);
  T* vbuf = (T*)take(ts * 2 * m);
  T* p = (T*)take(ts * 2 * m);
  double* dot = (double*)take(sizeof(double) * 4);
  double* scale = (double*)take(sizeof(double));
  GridBarrier* bar = (GridBarrier*)take(sizeof(GridBarrier));
  double* X = (double*)take(sizeof(double) * (size_t)m * kmax);
  T* Xg = (T*)take(2 * ts * (size_t)m * m);

  cudaError_t err = cudaSuccess;
  // algorithmic FP64 flops: Householder tridiagonalisation (16/3) m^3 complex,
  // (4/3) m^3 real; back transformation of kmax vectors 8 m^2 kmax complex, 2 m^2 kmax real
  const double cm = ops<T>::cplx ? 4.0 : 1.0;
  const double fl_tri = cm * (4.0 / 3.0) * m * (double)m * m * nb;
  const double fl_rest = cm * 2.0 * m * (double)m * kmax * nb;
  // 1. tridiagonalisation.  A batch or an instance that runs next to others (prefer_cluster):
  // one thread-block cluster per matrix (tridiag_cluster.cu), co-scheduled and, unlike a
  // cooperative launch, concurrent with other streams' work.  Else, and where no cluster
  // holds the matrix, a cooperative launch per matrix, with the rows in shared memory up to
  // kLoneMaxM and in global memory beyond.
  df = df && nb > 1;  // a lone reduction runs in FP64
  TriClusterShape cl;
  if ((nb > 1 || prefer_cluster) && m >= 2) cl = tridiag_cluster_shape<T>(m, nb, df);
  // rows per CTA: more CTAs shorten the work on the rows but lengthen the exchange, which
  // every CTA polls (m = 256 real: 2 rows 1.31 ms, 4 rows 1.00, 6 1.09; complex, with four
  // times the work, 1.40, 1.45 and 1.64 ms)
  const int R = std::max(ops<T>::cplx ? 2 : 4, (m + num_sms - 1) / num_sms);
  const int Pl = (m + R - 1) / R;
  const size_t shl = ((size_t)R + 3) * m * ts;
  const bool lone = cl.ctas == 0 && m <= kLoneMaxM && shl <= 200 * 1024;
  const void* kl = m <= TPB ? (const void*)tridiag_lone_kernel<T, 1>
                   : m <= 2 * TPB ? (const void*)tridiag_lone_kernel<T, 2>
                                  : (const void*)tridiag_lone_kernel<T, 4>;
  const bool products = bt && bt_products(m, kmax, nb);
  {
    // barrier, tau and e[0] start at zero; the exchange buffers of the lone reduction as
    // all-ones bit patterns (the "not yet written" mark)
    WsInit wi{};
    auto add = [&](void* p, size_t bytes, unsigned long long v) {
      wi.seg[wi.nseg] = static_cast<unsigned long long*>(p);
      wi.words[wi.nseg] = (int64_t)(bytes / 8);
      wi.val[wi.nseg] = v;
      ++wi.nseg;
    };
    add(bar, sizeof(GridBarrier), 0ull);
    add(tau, ts * m, 0ull);
    add(e, sizeof(double), 0ull);
    if (products) add(V, ts * (size_t)m * m, 0ull);  // v_j is zero up to column j
    if (lone) {
      add(Xg, ts * (size_t)m * m * 2, ~0ull);
    }
    wi.wb = wb;
    note_launches(CBC_K_AUX, 1);
    ws_init_kernel<<<dim3((unsigned)std::min<int64_t>(64, ((int64_t)m * m * (ts / 8) + 255) / 256), nb), 256, 0, s>>>(wi);
    err = cudaGetLastError();
    if (err == cudaSuccess && lone) err = allow_max_smem(kl);
    if (err != cudaSuccess) return err;
  }
  {
  KTimer tt(CBC_K_TRIDIAG, s, cl.ctas > 0 ? 1 : nb, fl_tri);
  if (cl.ctas > 0) {
    err = tridiag_cluster<T>(A, m, d, e, tau, V, (int64_t)m * m, wb, nb, cl, df, s);
  } else {
    for (int b = 0; b < nb && err == cudaSuccess; ++b) {
      const size_t off = (size_t)b * wb;
      T* Ab = A + (int64_t)b * m * m;
      if (lone) {
        Tri2Args<T> ta{Ab, m, byte_shift(d, off), byte_shift(e, off), byte_shift(tau, off),
                       byte_shift(V, off), byte_shift(Xg, off), status};
        void* args[] = {&ta};
        err = cudaLaunchCooperativeKernel(kl, dim3(Pl), dim3(TPB), args, shl, s);
      } else {
        TriArgs<T> ta{Ab, m, byte_shift(d, off), byte_shift(e, off), byte_shift(tau, off),
                      byte_shift(V, off), byte_shift(vbuf, off), byte_shift(p, off),
                      byte_shift(dot, off), byte_shift(bar, off), status};
        void* args[] = {&ta};
        err = cudaLaunchCooperativeKernel((const void*)tridiag_kernel<T>,
                                          dim3(std::max(1, std::min(num_sms, m / 4))), dim3(TPB),
                                          args, 0, s);
      }
    }
  }
  }
  if (err != cudaSuccess) return err;
  KTimer te(CBC_K_EIG, s, 3, fl_rest);
  // 2. eigenvalue estimates
  const int wpb = 8;
  bisect32_kernel<<<dim3((m + wpb - 1) / wpb, nb), 32 * wpb, 2 * sizeof(float) * m, s>>>(
      d, e, m, kmax, lam32, scale, lam, wb);
  // 3. eigenvectors of T for the candidates, FP64: as few per warp as gives every SM one warp
  // (a warp costs the same for one member as for 16), and at most what shared memory holds
  {
    const size_t room = 216 * 1024, half = (size_t)(m + 1) / 2;
    auto bytes = [&](int per) {
      return 5 * half * (size_t)(2 * per + (per >= 8 ? 1 : 0)) * sizeof(double);
    };
    int cper = kInvMax;
    while (cper > 1 && bytes(cper) > room) --cper;
    const int nclu = kmax >= 2 ? std::min(4, kmax / 2) : 0;
    const int sms = std::max(1, num_sms - nclu * nb);
    const int per = (int)std::min<int64_t>(
        cper, std::max<int64_t>(1, ((int64_t)nb * kmax + sms - 1) / sms));
    size_t sh = std::max(bytes(per), nclu > 0 ? bytes(cper) : 0);
    const bool staged = sh + 2 * (size_t)m * sizeof(double) <= 226 * 1024;
    if (staged) sh += 2 * (size_t)m * sizeof(double);
    err = allow_max_smem((const void*)invit_kernel);
    if (err != cudaSuccess) return err;
    InvArgs ia{d, e, lam32, scale, m, kmax, X, lam, wb, per, cper, nclu, staged ? 1 : 0};
    invit_kernel<<<dim3(nclu + (kmax + per - 1) / per, nb), 32, sh, s>>>(ia);
    err = cudaGetLastError();
    if (err != cudaSuccess) return err;
  }
  // 4. back transformation: by matrix products where there is room for them (the exchange
  // buffer of the reduction holds V T)
  if (products)
    return backtransform_products<T>(V, tau, X, Xg, m, kmax, U, wb, bt, status, s, nb);
  // else 32 vectors per CTA (fewer FP64 instructions) when u fits in
  // shared memory and the batch gives enough CTAs to spread the FP64 work over the SMs;
  // else one vector per CTA
  const size_t shm32 = ((size_t)m * 32 + 3 * (size_t)m) * ts;
  if (shm32 <= 200 * 1024 && (size_t)nb * ((kmax + 31) / 32) * 2 >= (size_t)num_sms) {
    const void* kbt = df ? (const void*)backtransform32_kernel<T, true>
                         : (const void*)backtransform32_kernel<T, false>;
    err = allow_max_smem(kbt);
    if (err != cudaSuccess) return err;
    if (df)
      backtransform32_kernel<T, true><<<dim3((kmax + 31) / 32, nb), 32 * BT_WARPS, shm32, s>>>(
          V, tau, X, m, kmax, U, wb);
    else
      backtransform32_kernel<T, false><<<dim3((kmax + 31) / 32, nb), 32 * BT_WARPS, shm32, s>>>(
          V, tau, X, m, kmax, U, wb);
    return cudaGetLastError();
  }
  size_t shm = (size_t)m * ts;
  if (shm > 48 * 1024) {
    err = allow_max_smem((const void*)backtransform_kernel<T>);
    if (err != cudaSuccess) return err;
  }
  backtransform_kernel<T><<<dim3(kmax, nb), 128, shm, s>>>(V, tau, X, m, kmax, U, wb);
  return cudaGetLastError();
}

template cudaError_t heev_top<double>(double*, int, int, double*, double*, void*, int*, int,
                                      cudaStream_t, int, bool, bool, void*);
template cudaError_t heev_top<zdbl>(zdbl*, int, int, double*, zdbl*, void*, int*, int,
                                    cudaStream_t, int, bool, bool, void*);

}  // namespace cbc
