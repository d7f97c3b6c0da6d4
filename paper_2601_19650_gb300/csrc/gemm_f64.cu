// FP64 SIMT strided GEMM: the products of the plain-FP64 CBC path that the tensor cores do
// not take (gemm_f64_split in gemm_tc.cu): short K, operands that split_guard.cuh turns down,
// and callers without room for slices.
//
// It works on leg views of the node tensors (kernels.cuh: View).  On GB300 the FP64 pipe delivers
// about 2 DFMA per clock per SM, so this kernel is FP64-throughput bound by design: a
// 64x64 (32x32) output tile per CTA, 16-deep K slices staged in shared memory, 4x4 (2x2)
// outputs per thread, and a K split (FP64 atomics into a zeroed C) when the output tiles
// alone cannot occupy every SM.
#include <algorithm>

#include "kernels.cuh"
#include "planner.h"
#include "split_guard.cuh"

namespace cbc {
namespace {

constexpr int BK = 16, NT = 256;

template <typename T>
struct GemmArgs {
  int M, N, K, splits, kchunk;
  const T* A;
  View va;
  const T* B;
  View vb;
  T* C;
  View vc;
  const int* guard;  // not NULL: only the problems that the split turns down
  int tiles_n, tiles_m, total;  // tiles of one (problem, split); of the launch
};

// R x R outputs per thread, 16 R x 16 R per CTA
template <typename T, bool CA, bool CB, bool ATOMIC, int R>
__global__ void __launch_bounds__(NT) gemm_f64_kernel(GemmArgs<T> g) {
  using O = ops<T>;
  constexpr int BM = 16 * R, BN = 16 * R;
  if (g.guard && g.total == g.tiles_m * g.tiles_n * g.splits && split_holds(g.guard)) return;
  __shared__ T As[BK][BM + 1];
  __shared__ T Bs[BK][BN + 1];
  __shared__ int64_t a_row[BM];
  __shared__ int64_t b_col[BN];

  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  for (int tile = blockIdx.x; tile < g.total; tile += gridDim.x) {
    const int bn = tile % g.tiles_n * BN, bm = tile / g.tiles_n % g.tiles_m * BM;
    const int z = tile / (g.tiles_n * g.tiles_m);
    const int batch = z / g.splits;
    if (g.guard && split_holds(g.guard + batch * GUARD_WORDS)) continue;
    const int split = z % g.splits;
    const int kbeg = split * g.kchunk;
    const int kend = min(g.K, kbeg + g.kchunk);

    const T* A = g.A + (int64_t)batch * g.va.bs;
    const T* B = g.B + (int64_t)batch * g.vb.bs;
    T* C = g.C + (int64_t)batch * g.vc.bs;

    for (int i = tid; i < BM; i += NT) a_row[i] = (bm + i < g.M) ? g.va.roff(bm + i) : -1;
    for (int i = tid; i < BN; i += NT) b_col[i] = (bn + i < g.N) ? g.vb.coff(bn + i) : -1;
    __syncthreads();

    T acc[R][R];
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int j = 0; j < R; ++j) acc[i][j] = O::zero();

    for (int k0 = kbeg; k0 < kend; k0 += BK) {
      // A tile: BM x BK, consecutive threads walk K (the contiguous leg of most views)
#pragma unroll
      for (int q = 0; q < (BM * BK) / NT; ++q) {
        int idx = tid + q * NT;
        int kk = idx % BK, mm = idx / BK;
        int k = k0 + kk;
        T v = O::zero();
        int64_t ro = a_row[mm];
        if (ro >= 0 && k < kend) {
          v = A[ro + g.va.coff(k)];
          if (CA) v = O::conj(v);
        }
        As[kk][mm] = v;
      }
      // B tile: BK x BN, consecutive threads walk N
#pragma unroll
      for (int q = 0; q < (BN * BK) / NT; ++q) {
        int idx = tid + q * NT;
        int nn = idx % BN, kk = idx / BN;
        int k = k0 + kk;
        T v = O::zero();
        int64_t co = b_col[nn];
        if (co >= 0 && k < kend) {
          v = B[g.vb.roff(k) + co];
          if (CB) v = O::conj(v);
        }
        Bs[kk][nn] = v;
      }
      __syncthreads();
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) {
        T a[R], b[R];
#pragma unroll
        for (int i = 0; i < R; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
        for (int j = 0; j < R; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
          for (int j = 0; j < R; ++j) acc[i][j] = O::fma(a[i], b[j], acc[i][j]);
      }
      __syncthreads();
    }

#pragma unroll
    for (int i = 0; i < R; ++i) {
      int r = bm + ty + 16 * i;
      if (r >= g.M) continue;
      int64_t ro = g.vc.roff(r);
#pragma unroll
      for (int j = 0; j < R; ++j) {
        int c = bn + tx + 16 * j;
        if (c >= g.N) continue;
        T* dst = C + ro + g.vc.coff(c);
        if (ATOMIC) {
          if constexpr (O::cplx) {
            double* d = reinterpret_cast<double*>(dst);
            atomicAdd(d, O::real(acc[i][j]));
            atomicAdd(d + 1, O::imag(acc[i][j]));
          } else {
            atomicAdd(reinterpret_cast<double*>(dst), O::real(acc[i][j]));
          }
        } else {
          *dst = acc[i][j];
        }
      }
    }
  }
}

template <typename T>
__global__ void zero_view_kernel(T* C, View vc, int M, int N, int batch, const int* guard) {
  if (guard && batch == 1 && split_holds(guard)) return;
  int64_t total = (int64_t)M * N * batch;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    int c = (int)(t % N);
    int64_t rb = t / N;
    int r = (int)(rb % M);
    int b = (int)(rb / M);
    if (guard && batch > 1 && split_holds(guard + b * GUARD_WORDS)) continue;
    C[(int64_t)b * vc.bs + vc.roff(r) + vc.coff(c)] = ops<T>::zero();
  }
}

int g_num_sms = 0;

// How a product is dealt to the CTAs.  Behind a split product (guard) tiles of 32 x 32 where
// those of 64 x 64 leave SMs idle: the same sums in the same order, and what the slicing cost is
// won back.  A product that the split turns down, cbc_gemm in all, on the SIMT kernel at once /
// behind the split, us: real 256 x 256 x 64 104 / 77, 64 x 64 x 8192 181 / 166 (without a split
// of K 9700), complex 64 x 128 x 256 565 / 214, 501 x 777 x 1030 4257 / 3141.
struct SimtShape {
  int edge, tiles, splits, kchunk;
};
SimtShape simt_shape(int M, int N, int K, int batch, bool guard) {
  if (g_num_sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
    if (g_num_sms <= 0) g_num_sms = 148;
  }
  const int target = 2 * g_num_sms;
  auto count = [&](int e) { return ((M + e - 1) / e) * ((N + e - 1) / e) * batch; };
  SimtShape s;
  s.edge = guard && count(64) < target ? 32 : 64;
  s.tiles = count(s.edge);
  const int ksteps = (K + BK - 1) / BK;
  // (by the 64 x 64 tiles in either case: partial sums as long as without a split product before)
  const int tiles64 = count(64);
  s.splits = 1;
  if (tiles64 < target && ksteps >= 16) {
    s.splits = (target + tiles64 - 1) / tiles64;
    s.splits = min(s.splits, ksteps / 8);
    s.splits = max(s.splits, 1);
  }
  s.kchunk = ((ksteps + s.splits - 1) / s.splits) * BK;
  s.splits = max(1, (K + s.kchunk - 1) / max(s.kchunk, 1));
  return s;
}

}  // namespace

template <typename T>
cudaError_t gemm_f64(int M, int N, int K, int batch, const T* A, const View& va, bool conjA,
                     const T* B, const View& vb, bool conjB, T* C, const View& vc,
                     cudaStream_t s, const int* guard) {
  if (M <= 0 || N <= 0 || batch <= 0) return cudaSuccess;
  const SimtShape sh = simt_shape(M, N, K, batch, guard != nullptr);
  const int edge = sh.edge, tiles = sh.tiles, splits = sh.splits;
  if (K <= 0) {  // empty contraction: C = 0
    note_launches(CBC_K_GEMM_F64, 1);
    zero_view_kernel<T><<<256, 256, 0, s>>>(C, vc, M, N, batch, nullptr);
    return cudaGetLastError();
  }
  GemmArgs<T> g{M,  N, K,  splits, sh.kchunk, A, va, B, vb, C, vc, guard,
                (N + edge - 1) / edge, (M + edge - 1) / edge, tiles * splits};
  // a product that usually does not run (guard) is launched as one resident wave
  const int grid = guard ? std::min(g.total, 2 * g_num_sms) : g.total;
  note_launches(CBC_K_GEMM_F64, splits > 1 ? 2 : 1);
  if (splits > 1) {
    int zb = (int)std::min<int64_t>(guard ? g_num_sms : 4096, ((int64_t)M * N * batch + 255) / 256);
    zero_view_kernel<T><<<zb, 256, 0, s>>>(C, vc, M, N, batch, guard);
  }
#define CBC_GEMM_LAUNCH(CA, CB)                                                     \
  if (edge == 32 && splits > 1)                                                     \
    gemm_f64_kernel<T, CA, CB, true, 2><<<grid, NT, 0, s>>>(g);                     \
  else if (edge == 32)                                                              \
    gemm_f64_kernel<T, CA, CB, false, 2><<<grid, NT, 0, s>>>(g);                    \
  else if (splits > 1)                                                              \
    gemm_f64_kernel<T, CA, CB, true, 4><<<grid, NT, 0, s>>>(g);                     \
  else                                                                              \
    gemm_f64_kernel<T, CA, CB, false, 4><<<grid, NT, 0, s>>>(g);
  if (conjA && conjB) {
    CBC_GEMM_LAUNCH(true, true)
  } else if (conjA) {
    CBC_GEMM_LAUNCH(true, false)
  } else if (conjB) {
    CBC_GEMM_LAUNCH(false, true)
  } else {
    CBC_GEMM_LAUNCH(false, false)
  }
#undef CBC_GEMM_LAUNCH
  return cudaGetLastError();
}

template cudaError_t gemm_f64<double>(int, int, int, int, const double*, const View&, bool,
                                      const double*, const View&, bool, double*, const View&,
                                      cudaStream_t, const int*);
template cudaError_t gemm_f64<zdbl>(int, int, int, int, const zdbl*, const View&, bool,
                                    const zdbl*, const View&, bool, zdbl*, const View&,
                                    cudaStream_t, const int*);

}  // namespace cbc
