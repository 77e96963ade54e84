// ttm_tc.cuh -- float64-accurate GEMM on the fifth-generation tensor cores (tcgen05) by
// exact slicing of the operands into bf16 integers (the Ozaki scheme: Ozaki, Ogita, Oishi &
// Rump 2012, error-free splitting of a matrix product into exactly computed partial products).
//
// C = A B with A (M x K) and B (K x N) in float64. Every row r of A is scaled by a power of
// two 2^e_r so that its entries lie in (-1, 1) (every column of B likewise, 2^f_c), and each
// scaled entry x is written as a sum of S signed integer digits,
//     x = sum_t s_t 2^(-6 - 7 t),   |s_t| <= 64,   t = 0 .. S-1,
// every digit exact in bf16. A product of two digits is an integer of magnitude <= 2^12, so
// a K-sum of up to 1024 of them is an integer below 2^24: the tensor core's float32
// accumulator holds it exactly. The partial products of digit levels t + u = l share the
// weight 2^(-12 - 7 l); each level l < S accumulates in its own TMEM accumulator (levels up
// to 3 exactly, the higher ones with a float32 rounding far below float64 resolution of the
// result), and the epilogue combines the levels in float64:
//     C_rc = 2^(e_r + f_c) sum_l 2^(-12 - 7 l) acc_l,
// over the S (S + 1) / 2 digit pairs with t + u < S. With S = 8 the digits carry 55 bits, so
// the result is as accurate as a float64 GEMM. An optional power-of-two scale per K index
// (A diag(2^-q) times diag(2^q) B, mathematically the identity) lets graded operands keep
// relative accuracy per column (W = Theta V with column norms spanning many decades).
//
// Kernels: oz_prep_kernel (row / column exponents and digits, written in the tcgen05
// shared-memory layout: K-major, no swizzle, 8 x 16-byte core matrices, so that one
// bulk copy per operand moves a stage), oz_gemm_kernel (one CTA per 128 x 64 output tile: a TMA
// producer warp with cp.async.bulk, one thread issuing tcgen05.mma kind::f16 into eight
// TMEM accumulators, four epilogue warps reading them with tcgen05.ld).
//
// Bound at 1024^3 by the operand traffic (96 KB per K chunk and CTA through L2), at small sizes by one
// tile's chain. Measured (GB300): exponents and digits in one integer launch instead of five float64
// ones, one instruction per four digits of B, and an epilogue of three float64 instructions per
// output instead of eight take a 1500 x 1024 x 2000 product from 1100 to 550 us and a 320^3 one from
// about 110 to 45 us.
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

#include "ttm_common.cuh"
#include "ttm_gemm.cuh"

namespace ttm {

constexpr int kOzMaxS = 8;        // digits per operand (and TMEM accumulators)
constexpr int kOzTM = 128;        // rows of an output tile (UMMA M)
constexpr int kOzTN = 64;         // columns of an output tile (UMMA N)
constexpr int kOzKC = 32;         // K of one pipeline stage
constexpr int kOzKB = 1024;       // K summed exactly in one accumulator block
constexpr int kOzATile = kOzTM * kOzKC * 2;  // bytes of one A digit tile (8 KB)
constexpr int kOzBTile = kOzTN * kOzKC * 2;  // bytes of one B digit tile (4 KB)
constexpr int kOzStages = 2;
constexpr int kOzThreads = 192;   // warps 0-3 epilogue, warp 4 TMA producer, warp 5 MMA issuer
constexpr int kOzExpNone = -100000;  // exponent of an all-zero row or column
constexpr int kOzExpNaN = 100000;    // a row or column with a NaN or an infinity: its outputs are NaN

__host__ __device__ constexpr int oz_stage_bytes(int S) { return S * (kOzATile + kOzBTile); }
__host__ __device__ constexpr int oz_smem_bytes(int S) { return kOzStages * oz_stage_bytes(S) + 256; }
// TMEM columns of the S accumulators (a power of two, at least 32)
__host__ __device__ constexpr uint32_t oz_tmem_cols(int S) {
  return S * kOzTN <= 32 ? 32u : S * kOzTN <= 64 ? 64u : S * kOzTN <= 128 ? 128u : S * kOzTN <= 256 ? 256u : 512u;
}

// One GEMM of a launch: the float64 problem (from a functor, as for dgemm_kernel) and where
// its digits live.
struct OzWs {
  unsigned char* a;   // digits of A: [row tiles of 128][K chunks of 32] blocks of S x 8 KB
  unsigned char* b;   // digits of B^T: [column tiles of 64][K chunks of 32] blocks of S x 4 KB
  int* ea;            // row exponents of A (M entries)
  int* eb;            // column exponents of B (N entries)
  long a_stride, b_stride, e_stride;  // bytes / ints per (z, batch) problem
  int S;
  int* err;           // set to TTM_ERR_TIMEOUT when a bounded wait gives up
  int kscale_buf;     // buffer id of per-K power-of-two exponents q_k (ints in a double
                      // buffer: A diag(2^-q) times diag(2^q) B), -1 = none
};

// Per-column binary exponents q_j of a column-major m x n matrix (frexp of the column's
// largest magnitude; 0 for a zero column), written as ints into a double buffer: the K scale
// that makes W diag(2^-q) have columns of magnitude near 1. One warp per column.
struct ColExpArgs {
  Tables t;
  int bw, bq;
  Dim m, n;
};
__global__ void colexp_kernel(ColExpArgs a) {
  pdl_begin();
  const int z = blockIdx.y;
  const int j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  const int n = a.n.eval(a.t, z);
  if (j >= n) return;
  const int m = a.m.eval(a.t, z);
  const double* w = bufp(a.t, z, a.bw) + (long)j * m;
  double mx = 0.0;
  for (int r = lane; r < m; r += 32) mx = fmax(mx, fabs(w[r]));
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) {
    int e = 0;
    if (mx > 0.0) frexp(mx, &e);
    reinterpret_cast<int*>(bufp(a.t, z, a.bq))[j] = e;
  }
}

// ---------------------------------------------------------------- operand views
// Operand X (0 = A as R = M rows, 1 = B viewed transposed as R = N rows), both with K columns.
template <class F>
struct OzArgs {
  F f;
  int nbatch;
  OzWs w;
  double* fl;     // nullptr, or per-product flop accumulators (stride fl_stride)
  int fl_stride;
};

// Layout of the digits: one contiguous block per (row tile, K chunk of 32) with all S digits, so that
// a stage is one bulk copy per operand. Core matrices are 8 rows of 16 bytes (8 k).
//   A (tiles of 128 rows): [digit][K group of 8][row group of 8], leading byte offset 2048 between K
//     neighbours, stride byte offset 128 between row groups;
//   B (tiles of 64 rows): [K group][digit][row group], leading byte offset S 1024, stride byte offset
//     128 across the row groups of all digits: consecutive digits of B are one operand of up to
//     256 rows, and their products with one digit of A land in consecutive accumulators.
__device__ __forceinline__ long oz_off_a(int r, int k, int nkc, int S) {
  const long tile = (long)(r / kOzTM) * nkc + k / kOzKC;
  return tile * S * kOzATile + (((k % kOzKC) >> 3) * (kOzTM / 8) + ((r % kOzTM) >> 3)) * 128 + (r & 7) * 16;
}
__device__ __forceinline__ long oz_off_b(int r, int k, int nkc, int S) {
  const long tile = (long)(r / kOzTN) * nkc + k / kOzKC;
  return tile * S * kOzBTile + (((k % kOzKC) >> 3) * S * (kOzTN / 8) + ((r % kOzTN) >> 3)) * 128 + (r & 7) * 16;
}

// x 2^sh as a 64-bit integer, rounded to nearest (|x| 2^sh < 2^62), by integer arithmetic.
__device__ __forceinline__ long long oz_fixed(long long bits, int sh) {
  const int ef = (int)((bits >> 52) & 0x7ff);
  const long long m = (bits & 0xfffffffffffffll) | (ef != 0 ? 0x10000000000000ll : 0ll);
  const int s = max(ef, 1) - 1075 + sh;  // x 2^sh = +-m 2^s
  long long v;
  if (s >= 0) v = m << min(s, 62);  // (beyond 9 for subnormal numbers only)
  else if (s < -54) v = 0;
  else v = ((m >> (-s - 1)) + 1) >> 1;
  return bits < 0 ? -v : v;
}

// Exponents and digits of both operands over their padded extents (zeros outside the matrix).
// Exponent of row r: the largest frexp exponent of X_rk 2^(-+q_k), kOzExpNone for a zero row.
// Digits: x 2^(6 + 7 (S - 1) - e_r) rounded to an integer, split into balanced base-128 digits from
// the low end. Everything is integer arithmetic on the bit patterns (a float64 instruction takes
// 64 clocks of a sub-partition: slicing by rint and multiplication spent 24 of them per element).
// Grid: x = 16-row groups of A, then of B; z = problems. 256 threads: a thread takes 8 consecutive k
// of one row, which is one 16-byte store per digit; the second pass over K finds its data in L1.
constexpr int kOzPrepRows = 16;
template <class F>
__global__ void __launch_bounds__(256) oz_prep_kernel(OzArgs<F> a, int mpad, int npad, int kpad) {
  pdl_begin();
  const int zb = blockIdx.z, z = zb / a.nbatch, b = zb % a.nbatch;
  const GemmDesc g = a.f(z, b);
  if (g.M <= 0 || g.N <= 0) return;  // nothing of this problem is multiplied
  const int na = mpad / kOzPrepRows;
  const int which = (int)blockIdx.x < na ? 0 : 1;
  const int r0 = ((int)blockIdx.x - (which ? na : 0)) * kOzPrepRows;
  const int R = which == 0 ? g.M : g.N, K = g.K;
  const int TR = which == 0 ? kOzTM : kOzTN;
  // row tiles that no output tile reads
  if (r0 >= (R + TR - 1) / TR * TR) return;
  const double* p = which == 0 ? g.A.p : g.B.p;
  const long rs = which == 0 ? g.A.rs : g.B.cs, ks = which == 0 ? g.A.cs : g.B.rs;
  const int* q = a.w.kscale_buf >= 0 ? reinterpret_cast<const int*>(bufp(a.f.t, z, a.w.kscale_buf)) : nullptr;
  const int rl = threadIdx.x & 15, kg = threadIdx.x >> 4, r = r0 + rl;  // row, group of 8 k
  const int kend = (K + kOzKC - 1) / kOzKC * kOzKC;
  __shared__ int s_e[kOzPrepRows];
  if (threadIdx.x < kOzPrepRows) s_e[threadIdx.x] = kOzExpNone;
  __syncthreads();
  int e = kOzExpNone;
  if (r < R)
    for (int k0 = kg * 8; k0 < K; k0 += 128)
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int k = k0 + u;
        if (k < K) {
          const unsigned long long x = (unsigned long long)__double_as_longlong(p[(long)r * rs + (long)k * ks]) << 1;
          const int ef = (int)(x >> 53);
          const int qq = q ? (which == 0 ? -q[k] : q[k]) : 0;
          if (ef != 0) e = max(e, ef == 0x7ff ? kOzExpNaN : ef - 1022 + qq);
          else if (x != 0) e = max(e, 63 - __clzll((long long)x) - 1074 + qq);  // subnormal
        }
      }
  if (e != kOzExpNone) atomicMax(&s_e[rl], e);
  __syncthreads();
  e = s_e[rl];
  if (kg == 0 && r < R) ((which == 0 ? a.w.ea : a.w.eb) + (long)zb * a.w.e_stride)[r] = e;
  unsigned char* base = which == 0 ? a.w.a + zb * a.w.a_stride : a.w.b + zb * a.w.b_stride;
  const int S = a.w.S, nkc = kpad / kOzKC;
  for (int k0 = kg * 8; k0 < kend; k0 += 128) {
    long long v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = k0 + u;
      v[u] = 0;
      if (r < R && k < K && e != kOzExpNone) {
        const int qq = q ? (which == 0 ? -q[k] : q[k]) : 0;
        v[u] = oz_fixed(__double_as_longlong(p[(long)r * rs + (long)k * ks]), 7 * S - 1 - e + qq);
      }
    }
    const long off0 = which == 0 ? oz_off_a(r, k0, nkc, S) : oz_off_b(r, k0, nkc, S);
    const long plane = which == 0 ? kOzATile : (kOzTN / 8) * 128;  // between digits
    for (int t = S - 1; t >= 0; --t) {
      unsigned w[4];
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        unsigned pr = 0;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const int u = 2 * h + c;
          int d;
          if (t > 0) {
            d = (int)(v[u] & 127);
            if (d >= 64) d -= 128;
            v[u] = (v[u] - d) >> 7;
          } else {
            d = (int)v[u];  // at most 64 in magnitude
          }
          pr |= (__float_as_uint((float)d) >> 16) << (16 * c);  // a small integer is exact in bf16
        }
        w[h] = pr;
      }
      *reinterpret_cast<uint4*>(base + off0 + t * plane) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
}

// ---------------------------------------------------------------- PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint64_t globaltimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Waits for the phase with the given parity to complete; gives up after limit_ns and
// returns false (the caller records TTM_ERR_TIMEOUT and winds down without trapping).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint64_t limit_ns) {
  uint32_t done = 0;
  const uint64_t t0 = globaltimer_ns();
  while (true) {
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    if (globaltimer_ns() - t0 > limit_ns) return false;
  }
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
// Shared-memory matrix descriptor of tcgen05.mma: start address, leading byte offset (between
// core matrices along K) and stride byte offset (between core matrices along M / N), all in
// 16-byte units; version 1 at bits 46-47; no swizzle.
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}
// Instruction descriptor of kind::f16: bf16 A and B (K-major), float32 accumulator, M x N.
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
// 32 lanes x 16 consecutive float32 columns of TMEM into 16 registers per thread.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

constexpr uint64_t kOzWaitNs = 2000000000ull;  // 2 s: far beyond any legitimate wait

// ---------------------------------------------------------------- the GEMM
// Grid: (N tiles of 64, M tiles of 128, problems). Dynamic shared memory: oz_smem_bytes(S).
template <class F>
__global__ void __launch_bounds__(kOzThreads, 1) oz_gemm_kernel(OzArgs<F> a, int mpad, int npad, int kpad) {
  pdl_begin();
  extern __shared__ __align__(1024) unsigned char smem[];
  const int zb = blockIdx.z, z = zb / a.nbatch, b = zb % a.nbatch;
  const GemmDesc g = a.f(z, b);
  const int m0 = blockIdx.y * kOzTM, n0 = blockIdx.x * kOzTN;
  if (g.M <= 0 || g.N <= 0 || m0 >= g.M || n0 >= g.N) return;   // CTA-uniform exit
  if (m0 == 0 && n0 == 0 && threadIdx.x == 0) gemm_count_flops(a.fl, a.fl_stride, z, g);
  if (g.upper && m0 > n0 + kOzTN - 1) return;
  const int S = a.w.S;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nkc = (g.K + kOzKC - 1) / kOzKC;            // K chunks of this problem
  const int nkcp = kpad / kOzKC;
  const int stage_bytes = oz_stage_bytes(S);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kOzStages * stage_bytes);
  // bars: full[2], empty[2], acc_full, acc_empty; then the TMEM address
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 8);
  __shared__ int s_abort;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kOzStages; ++s) {
      mbar_init(smem_u32(&bars[s]), 1);
      mbar_init(smem_u32(&bars[2 + s]), 1);
    }
    mbar_init(smem_u32(&bars[4]), 1);
    mbar_init(smem_u32(&bars[5]), 128);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  const uint32_t tcols = oz_tmem_cols(S);
  __syncwarp();     // warp 0 reconverges after thread 0's barrier set-up (alloc is warp-collective)
  if (warp == 0) {  // TMEM: S accumulators of 64 float32 columns
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(tcols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int nkb = (nkc + (kOzKB / kOzKC) - 1) / (kOzKB / kOzKC);  // exact accumulation blocks

  if (warp == 4) {
    // ---------------- TMA producer: all S digit tiles of A and of B for one K chunk per stage
    if (lane == 0) {
      const unsigned char* Ab = a.w.a + zb * a.w.a_stride;
      const unsigned char* Bb = a.w.b + zb * a.w.b_stride;
      for (int kc = 0; kc < nkc; ++kc) {
        const int s = kc % kOzStages;
        if (kc >= kOzStages && !mbar_wait(smem_u32(&bars[2 + s]), ((kc / kOzStages) - 1) & 1, kOzWaitNs)) {
          atomicExch(&s_abort, 1);
          break;
        }
        if (s_abort) break;
        const uint32_t full = smem_u32(&bars[s]);
        mbar_expect_tx(full, (uint32_t)stage_bytes);
        unsigned char* st = smem + s * stage_bytes;
        const long ta = (long)blockIdx.y * nkcp + kc, tb = (long)blockIdx.x * nkcp + kc;
        bulk_g2s(smem_u32(st), Ab + ta * S * kOzATile, (uint32_t)(S * kOzATile), full);
        bulk_g2s(smem_u32(st + S * kOzATile), Bb + tb * S * kOzBTile, (uint32_t)(S * kOzBTile), full);
      }
    }
  } else if (warp == 5) {
    // ---------------- MMA issuer: every digit pair (t, u) with t + u < S, two K steps of 16. Up to
    // four digits of B are one instruction (N up to 256): A is read from shared memory 12 times
    // instead of 36 per K step, which leaves the tensor pipe and not the shared memory as the bound.
    if (lane == 0) {
      int kc = 0;
      for (int kb = 0; kb < nkb && !s_abort; ++kb) {
        if (kb > 0 && !mbar_wait(smem_u32(&bars[5]), (kb - 1) & 1, kOzWaitNs)) {  // epilogue drained
          atomicExch(&s_abort, 1);
          break;
        }
        tc_fence_after();
        const int kc_end = min(nkc, (kb + 1) * (kOzKB / kOzKC));
        bool first = true;
        for (; kc < kc_end; ++kc) {
          const int s = kc % kOzStages;
          if (!mbar_wait(smem_u32(&bars[s]), (kc / kOzStages) & 1, kOzWaitNs)) {
            atomicExch(&s_abort, 1);
            break;
          }
          tc_fence_after();
          const uint32_t st = smem_u32(smem + s * stage_bytes);
          for (int ks = 0; ks < kOzKC / 16; ++ks) {
            for (int t = 0; t < S; ++t) {
              const uint64_t ad = umma_desc(st + t * kOzATile + ks * 2 * (kOzTM / 8) * 128, (kOzTM / 8) * 128, 128);
              for (int u = 0; u + t < S; u += 4) {
                const int nu = min(4, S - t - u);
                const uint64_t bd =
                    umma_desc(st + S * kOzATile + (ks * 2 * S + u) * (kOzTN / 8) * 128, S * (kOzTN / 8) * 128, 128);
                // the first step of a block starts every accumulator afresh
                umma_bf16(tmem + (uint32_t)((t + u) * kOzTN), ad, bd, umma_idesc_bf16(kOzTM, nu * kOzTN),
                          first ? (t == 0 ? 0u : 1u) : 1u);
              }
            }
            // level l receives its first product from t = 0 (u = l), which zeroes it
            first = false;
          }
          umma_commit(smem_u32(&bars[2 + s]));  // the stage is free once these MMAs are done
        }
        umma_commit(smem_u32(&bars[4]));        // block done: accumulators ready
      }
    }
  } else {
    // ---------------- epilogue: warps 0-3, thread = tile row (TMEM lane)
    const int row = warp * 32 + lane;
    const int gr = m0 + row;
    const int* eA = a.w.ea + (long)zb * a.w.e_stride;
    const int* eB = a.w.eb + (long)zb * a.w.e_stride;
    const int er = gr < g.M ? eA[gr] : kOzExpNone;
    // Levels 0..3 and 4..7 are combined as 64-bit integers (every accumulator holds an integer of at
    // most 2^25), so an output takes three float64 instructions instead of one per level.
    double acc[kOzTN];
    bool ok = true;
    for (int kb = 0; kb < nkb; ++kb) {
      // one lane waits, the warp reconverges before the warp-collective tcgen05.ld
      int got = lane == 0 ? (mbar_wait(smem_u32(&bars[4]), kb & 1, kOzWaitNs) ? 1 : 0) : 0;
      got = __shfl_sync(0xffffffffu, got, 0);
      __syncwarp();
      if (!got) {
        if (lane == 0) atomicExch(&s_abort, 1);
        ok = false;
        break;
      }
      tc_fence_after();
#pragma unroll
      for (int h = 0; h < kOzTN / 16; ++h) {
        long long hi[16], lo[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) hi[j] = lo[j] = 0;
        for (int l = 0; l < S; ++l) {
          float v[16];
          tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(l * kOzTN + h * 16), v);
          if (l < 4) {
#pragma unroll
            for (int j = 0; j < 16; ++j) hi[j] += (long long)__float2int_rn(v[j]) << (21 - 7 * l);
          } else {
#pragma unroll
            for (int j = 0; j < 16; ++j) lo[j] += (long long)__float2int_rn(v[j]) << (49 - 7 * l);
          }
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          // exact: |hi|, |lo| < 2^50; hi 2^-33 + lo 2^-61
          const double dh = __longlong_as_double(0x4338000000000000ll + hi[j]) - 6755399441055744.0;
          const double dl = __longlong_as_double(0x4338000000000000ll + lo[j]) - 6755399441055744.0;
          const double s = fma(dl, 1.0 / 268435456.0, dh);
          acc[h * 16 + j] = kb == 0 ? s : acc[h * 16 + j] + s;
        }
      }
      tc_fence_before();
      __syncwarp();
      mbar_arrive(smem_u32(&bars[5]));
    }
    if (ok && gr < g.M) {
#pragma unroll
      for (int j = 0; j < kOzTN; ++j) {  // fully unrolled: acc stays in registers
        const int gc = n0 + j;
        if (gc < g.N) {
          const int ec = eB[gc];
          double v = 0.0;
          if (er == kOzExpNaN || ec == kOzExpNaN) {
            v = __longlong_as_double(0x7ff8000000000000ll);
          } else if (er != kOzExpNone && ec != kOzExpNone) {
            const int sh = er + ec - 33, hw = __double2hiint(acc[j]), ef = (hw >> 20) & 0x7ff;
            if (ef + sh > 0 && ef + sh < 2047 && ef != 0)
              v = __hiloint2double(hw + (sh << 20), __double2loint(acc[j]));
            else
              v = ldexp(acc[j], sh);
          }
          double* c = g.C.p + (long)gr * g.C.rs + (long)gc * g.C.cs;
          if (g.alpha != 1.0) v *= g.alpha;
          if (g.beta != 0.0) v = fma(g.beta, *c, v);
          *c = v;
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (s_abort && threadIdx.x == 0 && a.w.err) atomicExch(a.w.err, (int)TTM_ERR_TIMEOUT);
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tcols) : "memory");
  }
}

// ---------------------------------------------------------------- host side
inline long oz_cdiv(long a, long b) { return (a + b - 1) / b; }

// Kernel of launch_tc_gemm that last reported an error (for the error message).
inline const char*& tc_failed_step() {
  static thread_local const char* step = "";
  return step;
}

// Digit workspace of one launch of nprob problems with the given upper bounds.
inline size_t tc_ws_bytes(long nprob, int M_ub, int N_ub, int K_ub, int S) {
  const long mpad = oz_cdiv(M_ub, kOzTM) * kOzTM, npad = oz_cdiv(N_ub, kOzTN) * kOzTN;
  const long kpad = oz_cdiv(K_ub > 0 ? K_ub : 1, kOzKC) * kOzKC;
  const long e_ints = mpad > npad ? mpad : npad;
  return (size_t)(nprob * S * (mpad + npad) * kpad * 2 + 2 * nprob * e_ints * (long)sizeof(int) + 256);
}

// Exponents, digits and the tensor-core product of every (z, batch) problem of the functor.
// ws: tc_ws_bytes(nz * nbatch, ...) bytes of device memory; err: int set on a timeout.
template <class F>
cudaError_t launch_tc_gemm(cudaStream_t st, const F& f, int nz, int nbatch, int M_ub, int N_ub, int K_ub, int kscale_buf,
                    int S, unsigned char* ws, int* err, double* fl = nullptr, int fl_stride = 0) {
  const long mpad = oz_cdiv(M_ub, kOzTM) * kOzTM, npad = oz_cdiv(N_ub, kOzTN) * kOzTN;
  const long kpad = oz_cdiv(K_ub > 0 ? K_ub : 1, kOzKC) * kOzKC;
  const long nprob = (long)nz * nbatch;
  const long a_bytes = S * mpad * kpad * 2, b_bytes = S * npad * kpad * 2;
  const long e_ints = mpad > npad ? mpad : npad;
  OzWs w;
  w.a = ws;
  w.b = ws + nprob * a_bytes;
  w.ea = reinterpret_cast<int*>(ws + nprob * (a_bytes + b_bytes));
  w.eb = w.ea + nprob * e_ints;
  w.a_stride = a_bytes;
  w.b_stride = b_bytes;
  w.e_stride = e_ints;
  w.S = S;
  w.err = err;
  w.kscale_buf = kscale_buf;
  OzArgs<F> oa{f, nbatch, w, fl, fl_stride};
  // every launch is checked at once: the caller gets the first failing step
  const char*& step = tc_failed_step();
  step = "oz_prep_kernel";
  cudaError_t e = launch_pdl(oz_prep_kernel<F>, dim3((unsigned)((mpad + npad) / kOzPrepRows), 1, (unsigned)nprob),
                             dim3(256), 0, st, oa, (int)mpad, (int)npad, (int)kpad);
  if (e != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(oz_gemm_kernel<F>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                oz_smem_bytes(kOzMaxS))) != cudaSuccess)
    return e;
  step = "oz_gemm_kernel";
  return launch_pdl(oz_gemm_kernel<F>, dim3((unsigned)(npad / kOzTN), (unsigned)(mpad / kOzTM), (unsigned)nprob),
                    dim3(kOzThreads), oz_smem_bytes(S), st, oa, (int)mpad, (int)npad, (int)kpad);
}

}  // namespace ttm
