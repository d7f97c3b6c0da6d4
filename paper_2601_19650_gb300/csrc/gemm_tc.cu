// Split-precision tensor-core GEMM for sm_103a (tcgen05 + TMA + TMEM).
//
// The contractions and Gram products of the CBC sweeps (Sec. III A/B) are dense, so
// the mixed path runs them on the 5th-generation tensor cores.  The CBC truncation is
// sensitive to rounding in the forward sweep (a subspace choice at every bond), so
// plain bf16/TF32 products are not accurate enough; instead every operand element is
// written exactly as a short sum of bf16 integers ("slices") on a fixed-point grid:
//
//   row (or column) exponent e with max|x| < 2^e,  x = 2^(e-7) * sum_s 2^(-8s) q_s,
//   q_s integers in [-128, 128] (exact in bf16), s = 0 .. S-1, round to nearest.
//
// A product a.b then is 2^(ea+eb-14) * sum_{s,t} 2^(-8(s+t)) (q^a_s . q^b_t).  The
// terms with s+t < S are kept; for each level g = s+t the tensor cores accumulate
// sum_{s+t=g} q^a_s . q^b_t in FP32 over a K chunk short enough (<= 1024 / S products
// of magnitude <= 2^14 per element) that every partial sum is an integer below 2^24,
// hence exact.  The epilogue warps read the S level sums of a chunk from TMEM,
// convert them to integers and fold them into one int64 per output element,
// I += sum_g C_g << 8(S-1-g); the final value is 2^(ea+eb-14-8(S-1)) * I in FP64.
// With S slices an operand keeps ~8S-1 bits relative to its row maximum.  2 to 5 slices
// serve the mixed path; 8 serve the FP64 path (gemm_f64_split at the end of this file), with
// x = 2^(e-6) sum_s 2^(-8s) q_s and the level sums in two int64 per output element.
//
// Complex operands use the real 2x2 embedding: A' = [re, im] interleaved along K
// (M x 2K) and B' = [[br, bi], [-bi, br]] blocks (2K x 2N), so C' = A' B' holds
// [Re C, Im C] interleaved along N: the 4 real products of a complex product in one
// real GEMM.
//
// Kernel: persistent, one CTA per SM (cta_group::1) looping over 128 x BN output tiles of
// all the problems of a call (a lockstep group of CBC instances is one call).  Warp 0
// issues TMA loads of 64-wide K atoms (32-wide for 8 slices; S slices of A and of B per
// atom, 128B or 64B swizzle, two smem stages), warp 1 issues tcgen05.mma (one elected thread;
// one MMA per slice of A, against all the slices of B it meets side by side) into S TMEM
// accumulators per K chunk, double buffered across chunks and tiles so the epilogue of one chunk
// overlaps the MMAs of the next, and 4 epilogue warps per 16 columns drain TMEM (tcgen05.ld) into
// int64 registers and write FP64, assembled with integer operations.  Every wait is bounded (clock64); a timeout raises CBC_ERR_TIMEOUT in the
// status word, all roles leave their loops, and TMEM is freed before the CTA exits.
#include <cooperative_groups.h>
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

#include "kernels.cuh"
#include "planner.h"
#include "split_guard.cuh"

namespace cbc {
namespace tc {

constexpr int BM = 128;          // rows of the output tile (TMEM lanes)
constexpr int KA = 64;           // K is padded to this many bf16 elements
// bf16 elements per K atom of a smem stage: one 128-byte swizzle row, or one of 64 bytes
// for 8 slices, of which two stages of 128-byte rows do not fit in shared memory
__host__ __device__ constexpr int ka(int S) { return S > 5 ? 32 : 64; }
// an operand element is x = 2^(e - head) (q_0 + q_1 2^-8 + ...): 8 slices keep one bit less
// so that the digit word and its bias fit in 64 bits
__host__ __device__ constexpr int head(int S) { return S > 5 ? 6 : 7; }
constexpr int NSTAGE = 2;
// warps: 0 TMA, 1 MMA, then 4 epilogue warps (one per TMEM lane quarter) per group of 16
// accumulator columns: a tile's last sums leave through integer chains that one warp per
// scheduler cannot hide (64-wide tiles, chosen for long K, keep 32 per warp and their
// registers)
__host__ __device__ constexpr int epi_cols(int BN) { return BN == 64 ? 32 : 16; }
__host__ __device__ constexpr int epi_warps(int BN) { return (BN / epi_cols(BN)) * 4; }
__host__ __device__ constexpr int nthreads(int BN) { return 64 + 32 * epi_warps(BN); }
int g_sms = 0;
constexpr long long WAIT_CYCLES = 4000000000LL;  // ~2 s at 2 GHz

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait on an mbarrier phase.  Returns false (and raises the abort flag) on
// timeout or when another role already aborted.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                          int* status) {
  long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (*abort_flag) return false;
    if (clock64() - t0 > WAIT_CYCLES) {
      *abort_flag = 1;
      set_status(status, CBC_ERR_TIMEOUT);
      return false;
    }
  }
  return true;
}

__device__ __forceinline__ void tma_load_3d(const CUtensorMap* map, uint64_t* bar, void* dst, int c0,
                                            int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(smem_u32(dst)),
      "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}

// UMMA shared-memory descriptor: K-major tile of ROWB-byte rows with the swizzle of that
// width, 8-row core groups back to back.
template <int ROWB>
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  static_assert(ROWB == 128 || ROWB == 64, "swizzle width");
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;               // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(8 * ROWB >> 4) << 32; // stride byte offset
  d |= (uint64_t)1 << 46;               // descriptor version of the tcgen05 family
  d |= (uint64_t)(ROWB == 128 ? 2 : 4) << 61;  // 128-byte or 64-byte swizzle
  return d;
}

// instruction descriptor: D f32, A and B bf16, both K-major, M x N
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc,
                                          uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
      "%11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
      "%11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, "
      "%28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

template <int CW>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&r)[CW]) {
  if constexpr (CW == 32)
    tmem_ld32(taddr, r);
  else
    tmem_ld16(taddr, r);
}

struct TcArgs {
  int M, N2;             // real-embedded output rows / columns
  int atoms_total;       // K2_pad / ka(S)
  int atoms_per_split;   // multiple of atoms_per_chunk
  int atoms_per_chunk;
  const int* expA;       // [M_pad]
  const int* expB;       // [N_pad] (one per complex column when cplx)
  int cplx;
  int atomic;
  char* C;               // FP64 output (double or zdbl) through the view
  View vc;               // vc.bs: elements between the outputs of consecutive problems
  int* status;
  int* guard;            // not NULL: the words of split_guard.cuh (gemm_f64_split)
  int guard_k;           // terms of the real sums
  int check_atoms;       // atoms of the magnitudes' product, check_step apart
  int check_step;
  int acc;               // 1 or -1: base + A B or base - A B instead of A B
  const char* base;      // rows and columns as C's (C itself when it is split along K)
  int64_t base_shift;    // base's bytes from problem to problem less C's
  int splits;            // K splits per problem
  int Mp, N2p;           // packed rows of one problem in the A and B planes
  int ebsB;              // entries of expB per problem
  int tiles_m, tiles_n;  // output tiles of one (problem, split)
  int total_tiles;       // tiles_m * tiles_n * splits * problems
};

// (n + sticky) 2^e with n normalised (bit 63 set) and sticky != 0 for bits that fell off below
// it, rounded to a double (to nearest, ties to even) in integer operations: the epilogue keeps
// off the narrow FP64 pipe of this part.  Adding the 53-bit significand to the exponent field
// less one carries into the exponent both for its leading bit and when rounding overflows.
__device__ __forceinline__ double round_ldexp(unsigned long long n, bool sticky, int e, bool neg) {
  const unsigned long long r = n + 0x3ffull + (((n >> 11) & 1ull) | (sticky ? 1ull : 0ull));
  const unsigned long long mant = (r >> 11) | (r < n ? 1ull << 53 : 0ull);
  const int E = 63 + e + 1023;  // exponent field of n 2^e
  if (E <= 0 || E >= 2046) {
    const double v = ldexp((double)mant, e + 11);
    return neg ? -v : v;
  }
  return __longlong_as_double((long long)(((unsigned long long)(E - 1) << 52) + mant +
                                          (neg ? 1ull << 63 : 0ull)));
}
// ldexp((double)a, e)
__device__ __forceinline__ double i64_ldexp(long long a, int e) {
  if (a == 0) return 0.0;
  const unsigned long long m = a < 0 ? 0ull - (unsigned long long)a : (unsigned long long)a;
  const int lz = __clzll((long long)m);
  return round_ldexp(m << lz, false, e - lz, a < 0);
}
// ldexp(hi 2^32 + lo, e) with one rounding
__device__ __forceinline__ double i96_ldexp(long long hi, long long lo, int e) {
  hi += lo >> 32;
  unsigned long long h = (unsigned long long)hi;
  unsigned long long l = (unsigned long long)lo << 32;  // its low half, left aligned
  const bool neg = hi < 0;
  if (neg) {  // -(h 2^64 + l)
    l = 0ull - l;
    h = ~h + (l == 0ull ? 1ull : 0ull);
  }
  if (h == 0ull) {
    if (l == 0ull) return 0.0;
    const int lz = __clzll((long long)l);
    return round_ldexp(l << lz, false, e - 32 - lz, neg);
  }
  const int lz = __clzll((long long)h);
  const unsigned long long n = (h << lz) | (lz ? l >> (64 - lz) : 0ull);
  return round_ldexp(n, (l << lz) != 0ull, e + 32 - lz, neg);
}

template <int S, int BN>
__global__ void __launch_bounds__(nthreads(BN), 1)
    gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                   TcArgs a) {
  constexpr int KAS = ka(S);
  constexpr int A_BYTES = BM * KAS * 2;
  constexpr int B_BYTES = BN * KAS * 2;
  constexpr int STAGE_BYTES = S * (A_BYTES + B_BYTES);
  constexpr uint32_t TMEM_COLS = 512;
  static_assert(2 * S * BN <= (int)TMEM_COLS, "TMEM budget");  // hence S BN <= 256, the widest MMA
  static_assert(BN % 16 == 0, "MMA width");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + NSTAGE * STAGE_BYTES);
  uint64_t* empty = full + NSTAGE;
  uint64_t* tfull = empty + NSTAGE;
  uint64_t* tempty = tfull + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // Persistent: CTA b takes tiles b, b + gridDim.x, ...  A tile index runs over the
  // 128-row blocks fastest (neighbouring CTAs share the B tile), then the column
  // blocks, then (problem, K split).  The smem ring and the two TMEM buffers carry on
  // across tiles, so one tile's epilogue overlaps the next tile's loads and MMAs.
  struct Tile {
    int m0, n0, prob, a_begin, n_atoms, n_chunks;
    bool check;
  };
  // FP64 products (a.guard): nothing runs for a problem with Inf or NaN, and the tiles of the
  // others begin with a chunk of their own, the product of the magnitudes, whose entries the
  // epilogue holds against the line of split_guard.cuh
  auto tile_of = [&](int t) {
    Tile q;
    const int mt = t % a.tiles_m, r = t / a.tiles_m;
    const int nt = r % a.tiles_n, z = r / a.tiles_n;
    q.m0 = mt * BM;
    q.n0 = nt * BN;
    q.prob = z / a.splits;
    q.a_begin = (z % a.splits) * a.atoms_per_split;
    q.n_atoms = max(0, min(a.atoms_total, q.a_begin + a.atoms_per_split) - q.a_begin);
    q.check = false;
    if (S > 5 && a.guard) {
      if (a.guard[(int64_t)q.prob * GUARD_WORDS + GUARD_BAD])
        q.n_atoms = 0;  // (no role has anything to do in the tile)
      else
        q.check = q.a_begin == 0;
    }
    q.n_chunks = (q.n_atoms + a.atoms_per_chunk - 1) / a.atoms_per_chunk;
    return q;
  };

  if (threadIdx.x == 0) {
    for (int i = 0; i < NSTAGE; ++i) {
      mbar_init(full + i, 1);
      mbar_init(empty + i, 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(tfull + i, 1);
      mbar_init(tempty + i, epi_warps(BN));
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(&tmB) : "memory");
      int jg = 0;  // atoms loaded by this CTA so far (position in the smem ring)
      bool run = true;
      for (int t = blockIdx.x; t < a.total_tiles && run; t += gridDim.x) {
        const Tile q = tile_of(t);
        if (S > 5 && q.check) {
          // up to S atoms at once, in the places of the slices
          for (int j = 0; j < a.check_atoms; j += S, ++jg) {
            const int stage = jg % NSTAGE, use = jg / NSTAGE;
            if (!mbar_wait(empty + stage, (use & 1) ^ 1, abort_flag, a.status)) {
              run = false;
              break;
            }
            uint8_t* sA = smem + stage * STAGE_BYTES;
            uint8_t* sB = sA + S * A_BYTES;
            const int n = min(S, a.check_atoms - j);
            mbar_expect_tx(full + stage, n * (A_BYTES + B_BYTES));
            for (int s = 0; s < n; ++s) {
              const int k = (j + s) * a.check_step * KAS;
              tma_load_3d(&tmA, full + stage, sA + s * A_BYTES, k, q.prob * a.Mp + q.m0, S);
              tma_load_3d(&tmB, full + stage, sB + s * B_BYTES, k, q.prob * a.N2p + q.n0, S);
            }
          }
          if (!run) break;
        }
        for (int j = 0; j < q.n_atoms; ++j, ++jg) {
          const int stage = jg % NSTAGE, use = jg / NSTAGE;
          if (!mbar_wait(empty + stage, (use & 1) ^ 1, abort_flag, a.status)) {
            run = false;
            break;
          }
          uint8_t* sA = smem + stage * STAGE_BYTES;
          uint8_t* sB = sA + S * A_BYTES;
          mbar_expect_tx(full + stage, STAGE_BYTES);
          const int k = (q.a_begin + j) * KAS;
#pragma unroll
          for (int s = 0; s < S; ++s) {
            tma_load_3d(&tmA, full + stage, sA + s * A_BYTES, k, q.prob * a.Mp + q.m0, s);
            tma_load_3d(&tmB, full + stage, sB + s * B_BYTES, k, q.prob * a.N2p + q.n0, s);
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    if (lane == 0) {
      int jg = 0, cg = 0;  // atoms consumed, chunks issued (TMEM buffer cg & 1)
      bool run = true;
      for (int t = blockIdx.x; t < a.total_tiles && run; t += gridDim.x) {
        const Tile q = tile_of(t);
        if (S > 5 && q.check) {
          const int buf = cg & 1, use = cg >> 1;
          if (!mbar_wait(tempty + buf, (use & 1) ^ 1, abort_flag, a.status)) break;
          tc_fence_after();
          for (int j = 0; j < a.check_atoms; j += S, ++jg) {
            const int stage = jg % NSTAGE, su = jg / NSTAGE;
            if (!mbar_wait(full + stage, su & 1, abort_flag, a.status)) {
              run = false;
              break;
            }
            tc_fence_after();
            const uint32_t sA = smem_u32(smem + stage * STAGE_BYTES);
            const uint32_t sB = sA + S * A_BYTES;
            const int n = min(S, a.check_atoms - j);
            for (int s = 0; s < n; ++s)
#pragma unroll
              for (int kk = 0; kk < KAS / 16; ++kk)
                umma_bf16(tmem_base + (uint32_t)(buf * S * BN),
                          sdesc<2 * KAS>(sA + s * A_BYTES + kk * 32),
                          sdesc<2 * KAS>(sB + s * B_BYTES + kk * 32), idesc_bf16(BM, BN),
                          (j + s + kk == 0) ? 0u : 1u);
            umma_commit(empty + stage);
          }
          if (!run) break;
          umma_commit(tfull + buf);
          ++cg;
        }
        int j = 0;
        for (int c = 0; c < q.n_chunks; ++c, ++cg) {
          const int buf = cg & 1, use = cg >> 1;
          if (!mbar_wait(tempty + buf, (use & 1) ^ 1, abort_flag, a.status)) {
            run = false;
            break;
          }
          tc_fence_after();
          const int j_end = min(q.n_atoms, j + a.atoms_per_chunk);
          bool first = true;
          for (; j < j_end; ++j, ++jg) {
            const int stage = jg % NSTAGE, su = jg / NSTAGE;
            if (!mbar_wait(full + stage, su & 1, abort_flag, a.status)) {
              run = false;
              break;
            }
            tc_fence_after();
            const uint32_t sA = smem_u32(smem + stage * STAGE_BYTES);
            const uint32_t sB = sA + S * A_BYTES;
            // One MMA per slice of A: the slices 0 .. S-1-s of B lie back to back in shared
            // memory and the accumulators of the levels s .. S-1 they belong to (slice t of
            // B: level s + t) back to back in TMEM, so they are one operand of (S-s) BN
            // columns.  Issued one pair of slices at a time the MMAs were bound by reading
            // A's 4 KB from shared memory again for every BN columns (8192 x 4096 x 1024
            // complex, S = 5: 5.1 ms; stacked 3.3 ms: 39 GB of slices from L2 by the tiles' shapes,
            // tensor pipe busy 59% of the time).  s = 0 covers every level, so its first MMA of a
            // chunk clears them all.
#pragma unroll
            for (int kk = 0; kk < KAS / 16; ++kk) {
#pragma unroll
              for (int s = 0; s < S; ++s) {
                const uint32_t d = tmem_base + (uint32_t)((buf * S + s) * BN);
                const uint64_t ad = sdesc<2 * KAS>(sA + s * A_BYTES + kk * 32);
                const uint64_t bd = sdesc<2 * KAS>(sB + kk * 32);
                umma_bf16(d, ad, bd, idesc_bf16(BM, (S - s) * BN),
                          (first && s == 0 && kk == 0) ? 0u : 1u);
              }
            }
            first = false;
            umma_commit(empty + stage);  // smem stage free once these MMAs complete
          }
          if (!run) break;
          umma_commit(tfull + buf);      // chunk sums ready in TMEM
        }
      }
    }
  } else {
    // ---------------- epilogue (warps 2 ..) ----------------
    // warp w may read TMEM lanes 32*(w%4) .. +31; warps 2-5 take accumulator columns
    // 0 .. CW-1, warps 6-9 the next CW columns, and so on
    constexpr int CW = epi_cols(BN);
    const int ew = warp - 2;
    const int quarter = warp & 3;
    const int colg = ew >> 2;
    int cg = 0;  // chunks drained (TMEM buffer cg & 1)
    bool run = true;
    for (int t = blockIdx.x; t < a.total_tiles && run; t += gridDim.x) {
      const Tile q = tile_of(t);
      const int row = q.m0 + quarter * 32 + lane;
      if (S > 5 && q.check) {
        const int buf = cg & 1, use = cg >> 1;
        if (!mbar_wait(tfull + buf, use & 1, abort_flag, a.status)) break;
        tc_fence_after();
        uint32_t r[CW];
        tmem_ld<CW>(tmem_base + ((uint32_t)(quarter * 32) << 16) +
                        (uint32_t)(buf * S * BN + colg * CW), r);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty + buf);
        ++cg;
        const int mycol = q.n0 + colg * CW + lane;
        const bool colok =
            lane < CW && mycol < a.N2 &&
            a.expB[(int64_t)q.prob * a.ebsB + (a.cplx ? mycol >> 1 : mycol)] != GUARD_ZERO_ROW;
        const unsigned cols = __ballot_sync(0xffffffffu, colok);
        const bool rowok = row < a.M && a.expA[q.prob * a.Mp + row] != GUARD_ZERO_ROW;
        const float line = 0x1p14f * guard_line(a.guard_k);
        bool below = false;
#pragma unroll
        for (int i = 0; i < CW; ++i)
          below = below || ((cols >> i & 1u) && __uint_as_float(r[i]) < line);
        if (below && rowok) a.guard[(int64_t)q.prob * GUARD_WORDS + GUARD_FAIL] = 1;
      }
      // 8 slices span 2 x 32 bits more than one int64 holds: levels 0-3 and 4-7 apart
      constexpr int NACC = S > 5 ? 2 : 1;
      constexpr int LV = S / NACC;  // levels per accumulator
      long long acc[NACC][CW];
#pragma unroll
      for (int i = 0; i < NACC * CW; ++i) acc[i / CW][i % CW] = 0;
      for (int c = 0; c < q.n_chunks; ++c, ++cg) {
        const int buf = cg & 1, use = cg >> 1;
        if (!mbar_wait(tfull + buf, use & 1, abort_flag, a.status)) {
          run = false;
          break;
        }
        tc_fence_after();
#pragma unroll
        for (int g = 0; g < S; ++g) {
          const int shift = 8 * (LV - 1 - g % LV);
          uint32_t r[CW];
          tmem_ld<CW>(tmem_base + ((uint32_t)(quarter * 32) << 16) +
                        (uint32_t)((buf * S + g) * BN + colg * CW),
                    r);
#pragma unroll
          for (int i = 0; i < CW; ++i) {
            long long qv = (long long)__float2int_rn(__uint_as_float(r[i]));
            acc[g / LV][i] += qv << shift;
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty + buf);
      }
      if (!run) break;
      if (q.n_chunks > 0) {
        // the CW columns of this warp are shared by its lanes (the lanes are rows): lane i
        // finds column i's offset and exponent once, the loop takes them by shuffle
        const int* expB = a.expB + (int64_t)q.prob * a.ebsB;
        char* Cp = a.C + (int64_t)q.prob * a.vc.bs * (a.cplx ? 16 : 8);
        const int mycol = q.n0 + colg * CW + lane;
        const int myn = a.cplx ? (mycol >> 1) : mycol;
        const bool myok = lane < CW && mycol < a.N2;
        const long long mycoff = myok ? (long long)a.vc.coff(myn) : 0;
        const int myexp = myok ? expB[myn] : 0;
        const bool rowok = row < a.M;
        const int ea = rowok ? a.expA[q.prob * a.Mp + row] : 0;
        const int bias = -2 * head(S) - 8 * (S - 1);
        const int64_t ro = rowok ? a.vc.roff(row) : 0;
        const bool pair =
            a.cplx && !a.atomic && !a.acc && (reinterpret_cast<uintptr_t>(a.C) & 15) == 0;
        auto value = [&](int i, int e) {
          if constexpr (NACC == 2)
            return i96_ldexp(acc[0][i], acc[1][i], e);
          else
            return i64_ldexp(acc[0][i], e);
        };
        auto put = [&](double* dst, double v) {
          if (a.atomic)
            atomicAdd(dst, a.acc < 0 ? -v : v);
          else if (a.acc)
            *dst = *reinterpret_cast<const double*>(a.base + (reinterpret_cast<char*>(dst) - a.C) +
                                                    q.prob * a.base_shift) +
                   (a.acc < 0 ? -v : v);
          else
            *dst = v;
        };
#pragma unroll
        for (int i = 0; i < CW; i += 2) {
          // a complex element, in one store where C is 16-byte aligned, or two real ones
          const long long co = __shfl_sync(0xffffffffu, mycoff, i);
          const long long co1 = __shfl_sync(0xffffffffu, mycoff, i + 1);
          const int e0 = ea + bias + __shfl_sync(0xffffffffu, myexp, i);
          const int e1 = ea + bias + __shfl_sync(0xffffffffu, myexp, i + 1);
          const int col = q.n0 + colg * CW + i;
          if (rowok && col < a.N2) {
            const double v0 = value(i, e0), v1 = value(i + 1, e1);
            if (a.cplx) {
              double* dst = reinterpret_cast<double*>(Cp + 16 * (ro + co));
              if (pair) {
                *reinterpret_cast<double2*>(dst) = make_double2(v0, v1);
              } else {
                put(dst, v0);
                put(dst + 1, v1);
              }
            } else {
              put(reinterpret_cast<double*>(Cp + 8 * (ro + co)), v0);
              if (col + 1 < a.N2) put(reinterpret_cast<double*>(Cp + 8 * (ro + co1)), v1);
            }
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                 "r"(TMEM_COLS));
  }
}

// ---------------- operand slicing ----------------
// Logical rows are the rows of A, or the columns of B for the B^T side.  One launch cuts
// both operands: a CTA takes 32 logical rows and a share of K, the CTAs of a cluster share
// those rows' K range.  The elements are copied to shared memory once, along whichever index
// is contiguous in memory and all at once (up to `keep` tiles; a longer share is copied a
// second time, from L2), the rows' exponents are combined through the cluster's shared
// memory, and the slices leave coalesced along K to the [S][rows][K2_pad] planes.  16 B are read
// and 4 S (A) or 8 S (B) B written per complex element; 4096 x 4096 x 1024 with 5 slices keeps
// issue slots 54% and DRAM 38% busy: between the arithmetic on digits and the wait for the one
// copy in, three CTAs of an SM at a time.  Rows of padding are not written:
// they reach only rows and columns of the accumulators that the epilogue skips.
constexpr int PACK_ROWS = 32;
// tiles held in shared memory: more cover a longer share in one copy, fewer leave room for
// other CTAs on the SM
constexpr int PACK_KEEP = 4;
constexpr int PACK_CLUSTER = 8;  // most CTAs that share the K range of one row block

// exponent of |x| (biased-exponent field) without FP64 arithmetic: max|x| < 2^e with
// e = field - 1022 for normal numbers; 0 maps to a floor value
__device__ __forceinline__ int expo_bits(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
  if (b == 0ull) return -2000;
  const int f = (int)(b >> 52);
  if (f == 0x7ff) return 0x40000000;  // Inf or NaN
  if (f == 0) return -1021 - (__clzll((long long)b) - 12);  // subnormal: roughly
  return f - 1022;
}

// Balanced base-256 digits of t = x 2^(head-e) (|t| < 2^head): N = t 256^(S-1) rounded to the
// nearest integer (ties to even: of the 14 bits that 5 slices drop, all but the first are zero
// in one entry of 2^14), then t = sum_s q_s 256^-s up to 0.5 256^-(S-1) with q_1 .. q_{S-1}
// the balanced remainders of N by 256 (in [-128, 127]) and q_0 the remaining quotient
// (|q_0| <= 128).  N is taken straight from the bit pattern of x (the mantissa plus what
// rounds it, shifted): integer operations only, since a scaling and an FP64-to-integer conversion
// per value would run on the narrow FP64 pipe of this part.
// Returned is N + sum_{i<S-1} 128 256^i: its byte i is q_{S-1-i} + 128 for i < S-1, and its
// bits from 8 (S-1) up are q_0.
// Rows of subnormals below 2^LOW_ROW are scaled by 2^LOW_SHIFT before they are cut (5 slices or
// fewer; exact)
constexpr int LOW_ROW = -1021, LOW_SHIFT = 100;
template <int S>
constexpr long long DIGIT_BIAS =
    (long long)(0x8080808080808080ull & ((1ull << (8 * (S - 1))) - 1ull));
template <int S>
__device__ __forceinline__ long long digit_word(double x, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ffu);
  const unsigned long long mant = (b & 0xfffffffffffffull) | (ex ? (1ull << 52) : 0ull);
  // N = mant 2^-sh; the largest exponent of a row, ex = e + 1022, has the smallest sh: -9 for 8
  // slices, 14 and more for up to 5 (rows below LOW_ROW come scaled)
  constexpr int MIN_SH = 53 - head(S) - 8 * (S - 1);
  const int sh = MIN_SH + e + 1022 - (ex ? ex : 1);
  unsigned long long n;
  if (MIN_SH < 1 && sh <= 0)
    n = mant << -sh;
  else
    n = sh < 64 ? (mant + ((1ull << (sh - 1)) - 1ull) + ((mant >> sh) & 1ull)) >> sh : 0ull;
  const long long N = (b >> 63) ? -(long long)n : (long long)n;
  return N + DIGIT_BIAS<S>;
}
// the word of -x from x's
template <int S>
__device__ __forceinline__ long long negated_word(long long w) {
  return 2 * DIGIT_BIAS<S> - w;
}

// digit q_s as the bits of a float (exact; its upper half is the bf16): 2^23 + 128 + q is
// formed by placing the byte in the mantissa of 2^23
template <int S>
__device__ __forceinline__ uint32_t digit_f32(long long w, int s) {
  uint32_t u;
  if (s == 0) {
    u = 0x4b000000u + (uint32_t)((int)(w >> (8 * (S - 1))) + 128);
  } else {
    const int byte = S - 1 - s;
    u = __byte_perm(byte < 4 ? (uint32_t)w : (uint32_t)(w >> 32), 0x4b000000u, 0x7540 + (byte & 3));
  }
  return __float_as_uint(__uint_as_float(u) - 8388736.0f);
}
__device__ __forceinline__ uint32_t bf16_pair(uint32_t flo, uint32_t fhi) {
  return __byte_perm(flo, fhi, 0x7632);
}

// floor(2^7 |x| / 2^e) as the bits of a float, from the digit word (8 slices: x 2^(62-e) as an
// integer; the complement of a negative one, so at most one less)
__device__ __forceinline__ uint32_t leading7(long long w) {
  const int h = (int)((w - DIGIT_BIAS<8>) >> 32);
  return __float_as_uint(__uint_as_float(0x4b000000u + ((uint32_t)(h ^ (h >> 31)) >> 23)) -
                         8388608.0f);
}
template <typename T>
struct PackSide {
  const T* src;
  View v;              // of the operand as a matrix: rows x K for A, K x columns for B
  int conj, rows, rowlanes;
  __nv_bfloat16* out;  // planes; problem p at row block p
  int* expo;           // exponents of the logical rows, ebs per problem
  int ebs, rows_pad;   // packed rows of one problem in a plane
};
template <typename T>
struct PackArgs {
  PackSide<T> a, b;
  int blocks_a;        // row blocks of A (then those of B)
  int K, K2p, tiles_per_cta, keep;
  size_t plane_a, plane_b;
  int* status;
  int* wide;           // 8 slices: word (problem / per) is set when an operand holds Inf or NaN,
  int per;
  int* guard;          // or the problem's word of split_guard.cuh is, and the magnitudes'
                       // leading bits go to one plane more
};

// one element to shared memory, zero if !in; complex ones in one copy where the operand is
// 16-byte aligned (a caller's need not be), else in two
__device__ __forceinline__ void copy_async(double* dst, const double* src, bool in, bool) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(smem_u32(dst)), "l"(src),
               "r"(in ? 8 : 0)
               : "memory");
}
__device__ __forceinline__ void copy_async(zdbl* dst, const zdbl* src, bool in, bool al16) {
  if (al16) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src),
                 "r"(in ? 16 : 0)
                 : "memory");
  } else {
    copy_async(&dst->re, &src->re, in, false);
    copy_async(&dst->im, &src->im, in, false);
  }
}

template <typename T, bool SIDE_B, int S, int ROWS>
__device__ __forceinline__ void pack_rows(const PackArgs<T>& g, const PackSide<T>& o, size_t plane,
                                          int block, T* tiles, int* s_max, int* s_exp, int* s_low) {
  using O = ops<T>;
  constexpr bool CPLX = O::cplx;
  constexpr int KT = CPLX ? 32 : 64;  // logical K of a tile: one 64-wide packed atom
  constexpr int LD = KT + 1;
  constexpr int NQ = ROWS * KT / 256, RQ = ROWS / 8;
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  const int nranks = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r0 = block * ROWS;
  const T* src = o.src + (int64_t)blockIdx.z * o.v.bs;
  const int ntiles = g.K2p / KA;
  const int t_begin = rank * g.tiles_per_cta;
  const int t_end = min(ntiles, t_begin + g.tiles_per_cta);
  auto off_r = [&](int r) -> int64_t { return SIDE_B ? o.v.coff(r) : o.v.roff(r); };
  // (the two divisions of a two-level index only where it has two levels)
  const bool flat = (SIDE_B ? o.v.r_in : o.v.c_in) == 0x7fffffff;
  const int64_t ks = SIDE_B ? o.v.rs_in : o.v.cs_in;
  auto off_k = [&](int k) -> int64_t {
    return flat ? k * ks : (SIDE_B ? o.v.roff(k) : o.v.coff(k));
  };
  // element q of this thread in a tile.  Rows on the lanes: row = lane mod ROWS, the lanes
  // beyond on the next k; K on the lanes: k = lane + 32 (q / RQ), row = warp + 8 (q mod RQ)
  const bool rl = o.rowlanes != 0, al16 = (reinterpret_cast<uintptr_t>(o.src) & 15) == 0;
  int64_t ro[RQ];
#pragma unroll
  for (int q = 0; q < RQ; ++q) {
    const int r = r0 + (rl ? lane % ROWS : warp + 8 * q);
    ro[q] = r < o.rows ? off_r(r) : -1;
  }
  // tiles [t, min(t + keep, t_end)) into shared memory
  auto load_tiles = [&](int t) {
    const int te = min(t + g.keep, t_end);
    for (int i = t; i < te; ++i) {
      T* dst = tiles + (i - t) * ROWS * LD;
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const int kk = rl ? lane / ROWS + (32 / ROWS) * (warp + 8 * q) : lane + 32 * (q / RQ);
        const int k = i * KT + kk;
        const int64_t rr = ro[q % RQ];
        const bool in = rr >= 0 && k < g.K;
        copy_async(dst + (rl ? lane % ROWS : warp + 8 * (q % RQ)) * LD + kk, in ? src + rr + off_k(k) : src,
                   in, al16);
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
  };
  // largest exponents of rows warp + 8 q
  int best[RQ];
#pragma unroll
  for (int q = 0; q < RQ; ++q) best[q] = -2000;
  for (int t = t_begin; t < t_end; t += g.keep) {
    if (t > t_begin) __syncthreads();
    load_tiles(t);
    __syncthreads();
    const int n = min(g.keep, t_end - t);
    for (int i = 0; i < n; ++i)
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const T x = tiles[(i * ROWS + warp + 8 * (q % RQ)) * LD + lane + 32 * (q / RQ)];
        best[q % RQ] = max(best[q % RQ], max(expo_bits(O::real(x)), expo_bits(O::imag(x))));
      }
  }
#pragma unroll
  for (int q = 0; q < RQ; ++q) {
    const int b = __reduce_max_sync(0xffffffffu, best[q]);
    if (lane == 0) s_max[warp + 8 * q] = b;
  }
  __syncthreads();
  if (nranks > 1) cluster.sync();
  bool low = false;
  if (tid < ROWS) {
    int b = s_max[tid];
    for (int q = 0; q < nranks; ++q)
      if (q != rank) b = max(b, cluster.map_shared_rank(s_max, q)[tid]);
    if (b >= 0x40000000) {  // Inf or NaN in the row
      if constexpr (S > 5) {
        if (g.guard)
          g.guard[(int64_t)blockIdx.z * GUARD_WORDS + GUARD_BAD] = 1;
        else
          g.wide[blockIdx.z / g.per] = 1;
      } else {
        set_status(g.status, CBC_ERR_NUMERICAL);
      }
    }
    const bool zero = b < -1100;  // an all-zero (or padding) row
    b = zero ? 0 : b;
    low = S <= 5 && b < LOW_ROW;
    s_low[tid] = low;
    s_exp[tid] = low ? b + LOW_SHIFT : b;
    if (rank == 0 && r0 + tid < o.rows)
      o.expo[(int64_t)blockIdx.z * o.ebs + r0 + tid] = S > 5 && g.guard && zero ? GUARD_ZERO_ROW : b;
  }
  const bool any_low = __syncthreads_or(low);
  uint32_t* out = reinterpret_cast<uint32_t*>(o.out + (size_t)blockIdx.z * o.rows_pad * g.K2p);
  const size_t pl = plane / 2, ld = (size_t)g.K2p / 2;  // in words of two bf16
  const bool held = t_end - t_begin <= g.keep;  // the whole share is still there
  for (int t = t_begin; t < t_end; ++t) {
    const int i = (t - t_begin) % g.keep;
    const T* tile = tiles + i * ROWS * LD;
    if (!held && i == 0) {
      __syncthreads();
      load_tiles(t);
      __syncthreads();
    }
    if (any_low)
      for (int q = 0; q < NQ; ++q) {
        const int lr = warp + 8 * (q % RQ);
        T* x = tiles + (i * ROWS + lr) * LD + lane + 32 * (q / RQ);
        if (s_low[lr]) *x = O::scale(0x1p100, *x);
      }
    __syncwarp();
#pragma unroll 1
    for (int q = 0; q < RQ; ++q) {
      const int lr = warp + 8 * q;
      if (r0 + lr >= o.rows) continue;
      const int e = s_exp[lr];
      if constexpr (!CPLX) {
        const long long w0 = digit_word<S>(tile[lr * LD + 2 * lane], e);
        const long long w1 = digit_word<S>(tile[lr * LD + 2 * lane + 1], e);
        uint32_t* d = out + (size_t)(r0 + lr) * ld + t * 32 + lane;
        if (S > 5 && g.guard) d[S * pl] = bf16_pair(leading7(w0), leading7(w1));
#pragma unroll
        for (int sl = 0; sl < S; ++sl)
          d[sl * pl] = bf16_pair(digit_f32<S>(w0, sl), digit_f32<S>(w1, sl));
      } else {
        T x = tile[lr * LD + lane];
        if (o.conj) x = O::conj(x);
        const long long wr = digit_word<S>(O::real(x), e), wi = digit_word<S>(O::imag(x), e);
        // -x has digits of its own (a digit of -128 carries), and products that leave out the
        // last levels depend on them
        const long long wn = negated_word<S>(wi);
        uint32_t* d = out + (size_t)(SIDE_B ? 2 : 1) * (r0 + lr) * ld + t * 32 + lane;
        if (S > 5 && g.guard) {
          const uint32_t ar = leading7(wr), ai = leading7(wi);
          d[S * pl] = bf16_pair(ar, ai);
          if (SIDE_B) d[S * pl + ld] = bf16_pair(ai, ar);
        }
#pragma unroll
        for (int sl = 0; sl < S; ++sl) {
          const uint32_t fr = digit_f32<S>(wr, sl), fi = digit_f32<S>(wi, sl);
          if (!SIDE_B) {
            d[sl * pl] = bf16_pair(fr, fi);
          } else {  // rows 2n: [br, -bi] and 2n + 1: [bi, br]
            d[sl * pl] = bf16_pair(fr, digit_f32<S>(wn, sl));
            d[sl * pl + ld] = bf16_pair(fi, fr);
          }
        }
      }
    }
  }
  if (nranks > 1) cluster.sync();  // no CTA leaves while another still reads its row maxima
}

template <typename T, int S, int ROWS>
__global__ void __launch_bounds__(256) pack_kernel(PackArgs<T> g) {
  extern __shared__ __align__(16) unsigned char pack_smem[];
  __shared__ int s_max[ROWS], s_exp[ROWS], s_low[ROWS];
  T* tiles = reinterpret_cast<T*>(pack_smem);
  const int block = blockIdx.x / (int)cooperative_groups::this_cluster().num_blocks();
  if (block < g.blocks_a)
    pack_rows<T, false, S, ROWS>(g, g.a, g.plane_a, block, tiles, s_max, s_exp, s_low);
  else
    pack_rows<T, true, S, ROWS>(g, g.b, g.plane_b, block - g.blocks_a, tiles, s_max, s_exp, s_low);
}

// strides of the logical (row, k) indices at the origin, to pick the read pattern
template <bool SIDE_B>
bool rows_contiguous(const View& v) {
  const int64_t sr = SIDE_B ? (v.coff(1) - v.coff(0)) : (v.roff(1) - v.roff(0));
  const int64_t sk = SIDE_B ? (v.roff(1) - v.roff(0)) : (v.coff(1) - v.coff(0));
  return sr == 1 && sk != 1;
}

template <typename T, int S, int ROWS>
cudaError_t launch_pack(PackArgs<T> g, int cs, int nb, cudaStream_t s) {
  constexpr int KT = ops<T>::cplx ? 32 : 64;
  cudaError_t e = allow_max_smem((const void*)pack_kernel<T, S, ROWS>);
  if (e != cudaSuccess) return e;
  g.blocks_a = (g.a.rows + ROWS - 1) / ROWS;
  const int blocks = g.blocks_a + (g.b.rows + ROWS - 1) / ROWS;
  g.keep = std::min(PACK_KEEP * PACK_ROWS / ROWS, g.tiles_per_cta);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)cs * blocks, 1, nb);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = (size_t)g.keep * ROWS * (KT + 1) * sizeof(T);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cs;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  note_launches(CBC_K_AUX, 1);
  return cudaLaunchKernelEx(&cfg, pack_kernel<T, S, ROWS>, g);
}

template <typename T, int S>
cudaError_t pack_slices(PackArgs<T> g, int nb, cudaStream_t s) {
  const int tiles = g.K2p / KA;
  // as many CTAs along K as keep their share in shared memory, up to PACK_CLUSTER
  int cs = 1;
  while (cs < PACK_CLUSTER && cs * PACK_KEEP < tiles) cs *= 2;
  g.tiles_per_cta = (tiles + cs - 1) / cs;
  const int64_t ctas =
      (int64_t)cs * nb *
      ((g.a.rows + PACK_ROWS - 1) / PACK_ROWS + (g.b.rows + PACK_ROWS - 1) / PACK_ROWS);
  if (ctas < 2 * g_sms) return launch_pack<T, S, PACK_ROWS / 2>(g, cs, nb, s);
  return launch_pack<T, S, PACK_ROWS>(g, cs, nb, s);
}

// both operands of nb problems (sources v.bs elements apart) into their planes
template <typename T>
cudaError_t pack_operands(const PackArgs<T>& g, int S, int nb, cudaStream_t s) {
  switch (S) {
    case 2: return pack_slices<T, 2>(g, nb, s);
    case 3: return pack_slices<T, 3>(g, nb, s);
    case 4: return pack_slices<T, 4>(g, nb, s);
    case 8: return pack_slices<T, 8>(g, nb, s);
    default: return pack_slices<T, 5>(g, nb, s);
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

bool make_map(CUtensorMap* m, void* base, int K2_pad, int64_t rows_pad, int S, int planes,
              int box_rows) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {(cuuint64_t)K2_pad, (cuuint64_t)rows_pad, (cuuint64_t)planes};
  cuuint64_t strides[2] = {(cuuint64_t)K2_pad * 2, (cuuint64_t)rows_pad * K2_pad * 2};
  cuuint32_t box[3] = {(cuuint32_t)ka(S), (cuuint32_t)box_rows, 1};
  cuuint32_t es[3] = {1, 1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE,
                  ka(S) == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

constexpr int CHECK_ATOMS = 16;  // of 32 entries, of the magnitudes' product
int atoms_per_chunk_for(int S) { return std::max(1, (1024 / S) / ka(S)); }
size_t a256(size_t x) { return (x + 255) & ~size_t(255); }

struct Geo {
  int Mp, N2, N2p, K2, K2p;
};
Geo geometry(int M, int N, int K, bool cplx, int S) {
  Geo g;
  g.Mp = (M + BM - 1) / BM * BM;
  g.N2 = cplx ? 2 * N : N;
  // a multiple of 64 so that complex B^T planes hold whole 32-row slicing tiles
  g.N2p = (g.N2 + 63) / 64 * 64;
  g.K2 = cplx ? 2 * K : K;
  g.K2p = (g.K2 + KA - 1) / KA * KA;
  return g;
}

// Tile widths a slice count can use: two sets of S accumulators of BN columns fit the
// 512 TMEM columns of an SM (2 S BN <= 512) and two smem stages of S (128 + BN) x 64 bf16
// fit the 227 KB opt-in shared memory.  S = 5: 32 or 48; S = 4: 32 or 64; S <= 3: 64;
// S = 8: 32.
int bn_candidates(int S, int (&out)[2]) {
  if (S == 8) {
    out[0] = 32;
    return 1;
  }
  if (S == 5) {
    out[0] = 32;
    out[1] = 48;
    return 2;
  }
  if (S == 4) {
    out[0] = 32;
    out[1] = 64;
    return 2;
  }
  out[0] = 64;
  return 1;
}

template <int S, int BN>
constexpr size_t smem_bytes() {
  return (size_t)NSTAGE * S * (BM + BN) * ka(S) * 2 + 1024 + 256;
}

template <int S, int BN>
cudaError_t launch_bn(const CUtensorMap& ma, const CUtensorMap& mb, const TcArgs& args, dim3 grid,
                      cudaStream_t s) {
  static_assert(smem_bytes<S, BN>() <= 232448, "shared memory");
  static std::once_flag once;
  static cudaError_t attr = cudaSuccess;
  std::call_once(once, [] {
    attr = cudaFuncSetAttribute(gemm_tc_kernel<S, BN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)smem_bytes<S, BN>());
  });
  if (attr != cudaSuccess) return attr;
  gemm_tc_kernel<S, BN><<<grid, nthreads(BN), smem_bytes<S, BN>(), s>>>(ma, mb, args);
  return cudaGetLastError();
}

cudaError_t launch(int S, int BN, const CUtensorMap& ma, const CUtensorMap& mb, const TcArgs& args,
                   dim3 grid, cudaStream_t s) {
  switch (S * 1000 + BN) {
    case 2064: return launch_bn<2, 64>(ma, mb, args, grid, s);
    case 3064: return launch_bn<3, 64>(ma, mb, args, grid, s);
    case 4032: return launch_bn<4, 32>(ma, mb, args, grid, s);
    case 4064: return launch_bn<4, 64>(ma, mb, args, grid, s);
    case 5032: return launch_bn<5, 32>(ma, mb, args, grid, s);
    case 5048: return launch_bn<5, 48>(ma, mb, args, grid, s);
    case 8032: return launch_bn<8, 32>(ma, mb, args, grid, s);
    default: return cudaErrorInvalidValue;
  }
}

// Autotuned tile width per problem shape: the first call of a shape runs every candidate
// width on its own operands, times each with CUDA events on its stream and keeps the
// fastest for every later call of that shape (process-wide, all threads).
struct TuneKey {
  int S, Mp, N2p, K2p, nb, cplx;
  bool operator<(const TuneKey& o) const {
    return std::tie(S, Mp, N2p, K2p, nb, cplx) < std::tie(o.S, o.Mp, o.N2p, o.K2p, o.nb, o.cplx);
  }
};
std::mutex g_tune_mu;
std::map<TuneKey, int> g_tuned;

}  // namespace tc

namespace {
// The SIMT kernel walks K at ~1 us (real) or ~4 us (complex) per 16 terms whatever M and N
// are, the split costs ~15 us of launches more.  cbc_gemm in all, SIMT / split / SIMT behind the
// split (operands graded against each other), us:
//   real     256 x 256 x 64 104 / 63 / 77; 1000 x 1000 x 28 101 / 62 / 137,
//            x 1000 2117 / 139 / 2006
//   complex  16 x 16 x 16 102 / 51 / 75, 1000 x 1000 x 8 164 / 90 / 200, x 24 297 / 90 / 321,
//            128 x 2048 x 128 565 / 79 / 337
// So a product that is turned down costs up to a third more where K is short and the tiles fill
// the GPU, up to 8% more at other sizes that fill it, and less elsewhere (the smaller tiles).
constexpr int SPLIT_MIN_K_REAL = 28, SPLIT_MIN_K_CPLX = 8;
constexpr size_t SPLIT_MAX_BYTES = size_t(16) << 30;
}  // namespace

size_t gemm_tc_workspace_bytes(int M, int N, int K, bool cplx, int S, int nb) {
  using namespace tc;
  if (M < BM && N > M) std::swap(M, N);
  Geo g = geometry(M, N, K, cplx, S);
  const size_t b = (size_t)std::max(nb, 1);
  return a256(b * S * g.Mp * g.K2p * 2) + a256(b * S * g.N2p * g.K2p * 2) +
         a256(b * sizeof(int) * g.Mp) + a256(b * sizeof(int) * g.N2p) + 1024;
}

static View transpose_view(const View& v) {
  View t;
  t.r_in = v.c_in;
  t.rs_out = v.cs_out;
  t.rs_in = v.cs_in;
  t.c_in = v.r_in;
  t.cs_out = v.rs_out;
  t.cs_in = v.rs_in;
  t.bs = v.bs;
  return t;
}

template <typename T>
cudaError_t gemm_tc(int M, int N, int K, const T* A, const View& va, bool conjA, const T* B,
                    const View& vb, bool conjB, T* C, const View& vc, int S, void* ws,
                    int* status, cudaStream_t s, int nb, const TcWide& opt) {
  using namespace tc;
  if (M <= 0 || N <= 0 || nb <= 0) return cudaSuccess;
  if ((S < 2 || S > 5) && !(S == 8 && (opt.wide || opt.guard))) return cudaErrorInvalidValue;
  // keep the long dimension on the 128-row side: C^T = B^T A^T
  if (M < BM && N > M) {
    return gemm_tc<T>(N, M, K, B, transpose_view(vb), conjB, A, transpose_view(va), conjA, C,
                      transpose_view(vc), S, ws, status, s, nb, opt);
  }
  constexpr bool CPLX = ops<T>::cplx;
  if (g_sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
  }
  Geo g = geometry(M, N, K, CPLX, S);
  char* w = static_cast<char*>(ws);
  w = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(w) + 255) & ~uintptr_t(255));
  const size_t b = (size_t)nb;
  const int planes1 = S + (opt.guard ? 1 : 0);  // of one problem: the magnitudes behind the slices
  const size_t planes = b * planes1;
  __nv_bfloat16* sa = reinterpret_cast<__nv_bfloat16*>(w);
  w += a256(planes * g.Mp * g.K2p * 2);
  __nv_bfloat16* sb = reinterpret_cast<__nv_bfloat16*>(w);
  w += a256(planes * g.N2p * g.K2p * 2);
  int* ea = reinterpret_cast<int*>(w);
  w += a256(b * sizeof(int) * g.Mp);
  int* eb = reinterpret_cast<int*>(w);
  if (K <= 0) return cudaErrorInvalidValue;
  // slices of A (rows) and of B (columns, embedded); problem p owns row block p
  PackArgs<T> pk{};
  pk.a = {A, va, conjA ? 1 : 0, M, rows_contiguous<false>(va) ? 1 : 0, sa, ea, g.Mp, g.Mp};
  pk.b = {B, vb, conjB ? 1 : 0, N, rows_contiguous<true>(vb) ? 1 : 0, sb, eb,
          CPLX ? g.N2p / 2 : g.N2p, g.N2p};
  pk.K = K;
  pk.K2p = g.K2p;
  pk.plane_a = b * g.Mp * g.K2p;
  pk.plane_b = b * g.N2p * g.K2p;
  pk.status = status;
  pk.wide = opt.wide;
  pk.per = opt.per;
  pk.guard = opt.guard;
  cudaError_t pe = pack_operands<T>(pk, S, nb, s);
  if (pe != cudaSuccess) return pe;
  CUtensorMap ma;
  if (!make_map(&ma, sa, g.K2p, nb * g.Mp, S, planes1, BM)) return cudaErrorInvalidValue;
  const int atoms = g.K2p / ka(S);
  const int apc = atoms_per_chunk_for(S);
  const int chunks = (atoms + apc - 1) / apc;
  // one launch with tile width BN; a partial last column tile reads the next problem's
  // rows (or the zero fill past the planes) for columns the epilogue never writes
  auto run_bn = [&](int BN) -> cudaError_t {
    CUtensorMap mb;
    if (!make_map(&mb, sb, g.K2p, nb * g.N2p, S, planes1, BN)) return cudaErrorInvalidValue;
    const int tiles_n = (g.N2p + BN - 1) / BN;
    const int tiles = (g.Mp / BM) * tiles_n * nb;
    int splits = 1;
    if (tiles < g_sms && chunks > 1 && !opt.base) splits = std::min(chunks, std::max(1, g_sms / tiles));
    const int chunks_per_split = (chunks + splits - 1) / splits;
    splits = (chunks + chunks_per_split - 1) / chunks_per_split;
    TcArgs args;
    args.M = M;
    args.N2 = g.N2;
    args.atoms_total = atoms;
    args.atoms_per_chunk = apc;
    args.atoms_per_split = chunks_per_split * apc;
    args.expA = ea;
    args.expB = eb;
    args.cplx = CPLX ? 1 : 0;
    args.atomic = splits > 1 ? 1 : 0;
    args.C = reinterpret_cast<char*>(C);
    args.vc = vc;
    args.status = status;
    args.guard = opt.guard;
    // of a long K at most CHECK_ATOMS atoms of the magnitudes, evenly apart: a part of the sum is
    // below it too, and the line rises with the square root of K only
    args.check_step = (atoms + CHECK_ATOMS - 1) / CHECK_ATOMS;
    args.check_atoms = (atoms + args.check_step - 1) / args.check_step;
    args.guard_k = g.K2;
    args.acc = opt.acc;
    args.base = opt.base ? static_cast<const char*>(opt.base) : args.C;
    args.base_shift = opt.base ? (opt.base_bs - vc.bs) * (int64_t)sizeof(T) : 0;
    args.splits = splits;
    args.Mp = g.Mp;
    args.N2p = g.N2p;
    args.ebsB = CPLX ? g.N2p / 2 : g.N2p;
    if (splits > 1 && !opt.acc) {
      // the split partial sums are added into a zeroed C
      cudaError_t e = gemm_f64<T>(M, N, 0, nb, A, va, false, B, vb, false, C, vc, s);
      if (e != cudaSuccess) return e;
    }
    args.tiles_m = g.Mp / BM;
    args.tiles_n = tiles_n;
    args.total_tiles = args.tiles_m * args.tiles_n * splits * nb;
    dim3 grid(std::min(args.total_tiles, g_sms));
    note_launches(S == 8 ? CBC_K_GEMM_F64 : CBC_K_GEMM_TC, 1);
    if (S != 8)
      note_flops(CBC_K_TC_ISSUED,
               2.0 * g.Mp * ((double)tiles_n * BN) * g.K2p * (S * (S + 1) / 2) * nb);
    return launch(S, BN, ma, mb, args, grid, s);
  };
  int cand[2] = {64, 64};
  const int ncand = bn_candidates(S, cand);
  const TuneKey key{S, g.Mp, g.N2p, g.K2p, nb, CPLX ? 1 : 0};
  int BN = -1;
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    auto it = g_tuned.find(key);
    if (it != g_tuned.end()) BN = it->second;
  }
  if (BN > 0 || ncand == 1) return run_bn(BN > 0 ? BN : cand[0]);
  // first call of this shape: every candidate computes the same exact sums, so the
  // output of the last one stands; the fastest is kept for later calls
  cudaEvent_t ev[3];
  for (int c = 0; c <= ncand; ++c) cudaEventCreate(&ev[c]);
  cudaError_t e = cudaEventRecord(ev[0], s);
  for (int c = 0; c < ncand && e == cudaSuccess; ++c) {
    e = run_bn(cand[c]);
    if (e == cudaSuccess) e = cudaEventRecord(ev[c + 1], s);
  }
  if (e == cudaSuccess) e = cudaEventSynchronize(ev[ncand]);
  if (e == cudaSuccess) {
    int best = cand[0];
    float best_ms = 0.0f;
    for (int c = 0; c < ncand; ++c) {
      float ms = 0.0f;
      cudaEventElapsedTime(&ms, ev[c], ev[c + 1]);
      if (c == 0 || ms < best_ms) {
        best_ms = ms;
        best = cand[c];
      }
    }
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tuned.emplace(key, best);
  }
  for (int c = 0; c <= ncand; ++c) cudaEventDestroy(ev[c]);
  return e;
}

// ---- FP64 products on the tensor cores -------------------------------------------------
// 8 slices hold 62 bits of an entry relative to its row's (column's) maximum; the kept products
// of slices are summed exactly and rounded once to 53 bits (once more per K split).  Whether
// that is as accurate as an FP64 sum every tile finds out for its entries (split_guard.cuh);
// where it is not, the SIMT kernel behind does the problem (again).  Largest error
// in units of 2^-53 |A| |B|, SIMT kernel / split: Gaussian 64 x 64 x 28 2.4 / 0.5, complex
// 501 x 777 x 1030 1.3 / 0.07; positive entries 300 x 300 x 100 8.2 / 1.0; half of the entries
// zero 1.9 / 0.4; rows and columns scaled by 2^-30 to 2^30 2.4 / 0.2.
size_t gemm_f64_split_bytes(int M, int N, int K, bool cplx, int nb) {
  if (K < (cplx ? SPLIT_MIN_K_CPLX : SPLIT_MIN_K_REAL)) return 0;
  const size_t b = gemm_tc_workspace_bytes(M, N, K, cplx, 9, nb) +  // (8 slices, the magnitudes)
                   tc::a256(sizeof(int) * GUARD_WORDS * nb);
  return b <= SPLIT_MAX_BYTES ? b : 0;
}

template <typename T>
cudaError_t gemm_f64_split(int M, int N, int K, int nb, const T* A, const View& va, bool conjA,
                           const T* B, const View& vb, bool conjB, T* C, const View& vc, void* ws,
                           int* status, cudaStream_t s) {
  TcWide opt;
  opt.guard = static_cast<int*>(ws);
  const size_t gb = tc::a256(sizeof(int) * GUARD_WORDS * nb);
  cudaError_t e = cudaMemsetAsync(ws, 0, gb, s);
  if (e != cudaSuccess) return e;
  e = gemm_tc<T>(M, N, K, A, va, conjA, B, vb, conjB, C, vc, 8, static_cast<char*>(ws) + gb,
                 status, s, nb, opt);
  if (e != cudaSuccess) return e;
  return gemm_f64<T>(M, N, K, nb, A, va, conjA, B, vb, conjB, C, vc, s, opt.guard);
}

template cudaError_t gemm_f64_split<double>(int, int, int, int, const double*, const View&, bool,
                                            const double*, const View&, bool, double*,
                                            const View&, void*, int*, cudaStream_t);
template cudaError_t gemm_f64_split<zdbl>(int, int, int, int, const zdbl*, const View&, bool,
                                          const zdbl*, const View&, bool, zdbl*, const View&,
                                          void*, int*, cudaStream_t);
template cudaError_t gemm_tc<double>(int, int, int, const double*, const View&, bool,
                                     const double*, const View&, bool, double*, const View&, int,
                                     void*, int*, cudaStream_t, int, const TcWide&);
template cudaError_t gemm_tc<zdbl>(int, int, int, const zdbl*, const View&, bool, const zdbl*,
                                   const View&, bool, zdbl*, const View&, int, void*, int*,
                                   cudaStream_t, int, const TcWide&);

}  // namespace cbc
