// ttm_pre.cuh -- the Swap SVD (Fig. 1C, Eq. eps) by a preconditioned float32 Jacobi and float64
// Newton steps on the reduced problem; the default for Swap matrices of at most 1024 rows and 2048
// columns (Engine::pre_fits), as long as the distributed kernels' CTAs for all products of a batch are
// resident together: up to 57 products with Swaps of 256 x 256, 25 of 384 x 384, 9 of 512 x 512, 2 of
// 1024 x 1024 on 152 SMs. What does not fit takes the general pipeline (Engine::swap).
//
// Theta is m x n, p = min(m, n):
//   1. Theta^T = Q1 R1 in float64 (ttm_qrd.cuh); L = R1^T is m x p, Q1 stays as reflectors;
//   2. L = Q2 R2 in float32 (each column of L keeps its relative accuracy); X = R2^T has graded
//      columns and is nearly orthogonal column by column (the preconditioning of Drmac & Veselic
//      2008: two QR factorisations act as a step of the QR iteration), so that
//   3. the one-sided Jacobi on X converges in 4 .. 10 sweeps instead of the 27 of three passes on
//      Theta itself (measured on the Swaps of 1D, 2D and 3D fields and of random trains), and V, the
//      right singular vectors of L, are its normalised columns: no V is accumulated;
//   4. W = L V in float64 and two to four Newton steps for [W; V] (below);
//   5. order by column norm, Eq. eps and cap; new left carriage W[:, top k], new right carriage
//      (Q1 V[:, top k])^T through the reflectors.
//
// Newton steps. V has float32 errors, so a small column of W = L V carries up to 1e-6 of the largest
// singular vector, far above itself when the spectrum spans many decades; couplings G_ij between
// two small columns are then dominated by that part, and the plain step of ttm_newton.cuh cannot
// be used (its float32 passes on W remove the part first). Here G = W^T W is eliminated in
// descending order, U = the upper factor of G = L_G U: row i of U holds the couplings of column i
// after the larger ones are taken out, G'_ij = U_ij (i < j) and d_i = U_ii, each with float64
// accuracy relative to its own size. The step uses G' and d in the formula of ttm_newton.cuh,
//   S_ij = (E_ij (d_i + d_j) / 2 - G'_ij) / (d_i - d_j),  X = I - E / 2 + S,  E = V^T V - I,
// with the same filters. Measured: corrections 1e-3, 1e-7, 0 for successive steps.
//
// Where it is slow: a spectrum of many decades whose L is not graded by columns (the right parts of a chain
// of square Gaussian cores, say) loses everything below 6e-8 of its largest singular value in step 2; the
// rotations among those columns are then of order 1, four Newton steps do not converge, and the Swap takes
// the float64 Jacobi from V = I. A left-canonical Gaussian train times a constant at chi = 256, L = 18,
// eps = 1e-18: 33 of 153 Swaps, 4.2 s per product, against 0.96 s with f32_passes = 3; at eps = 1e-14, where
// that tail is dropped, 4 Swaps and 0.85 s. Fields and random products need it for none or one Swap.
//
// Bound by latencies: the chains of the two QRs (about 1.3 and 0.7 us per column), of the inner rounds
// of the Jacobi and of the elimination. Measured per product (GB300) against three float32 passes
// with V, three to five Newton steps and a saved state: 2D field, d = 4, chi = 64 332 -> 153 ms; 3D
// field, d = 8, chi = 96 503 -> 205 ms; random L = 10 61 -> 21 ms; chi = 160, L = 18 1616 -> 825 ms
// (129, 131, 8.6 and 486 ms with what was made faster in these kernels and their launches since).
#pragma once
#include <cooperative_groups.h>
#include "ttm_common.cuh"
#include "ttm_newton.cuh"
#include "ttm_pjac.cuh"
#include "ttm_qrd.cuh"
#include "ttm_svd.cuh"

namespace cg = cooperative_groups;

namespace ttm {

constexpr int kPreMax = 1024;       // largest p and m
constexpr int kPreSweeps = 30;      // sweep limit (the Newton steps and the fallback finish what is left)
constexpr double kPreTol = 4 * 5.96e-8;  // times sqrt(p): couplings below are not rotated
constexpr float kPreBig = 1e-3f;    // a sweep without a coupling above this is the last: the couplings
                                    // it leaves are of the order of its largest one squared. (With 1e-2
                                    // 5 of 2300 Swaps of fields and random trains, p to 768, needed the
                                    // float64 Jacobi, with 1e-3 none of 8600, at the same time per product.
                                    // At chi = 512, p to 1024, five of 435 do with 1e-3, from the Newton
                                    // steps: see pre_x_kernel.)
constexpr float kPreRidge = 1e-15f; // added to the diagonal of R2 (max |R1| = 1): no column of X vanishes

// Binary exponent that W leaves out: the squares of its columns stay in the float64 range whatever the
// norm of Theta. 0 for a Theta of ordinary size.
__device__ __forceinline__ int pre_exp(double absmax) {  // integer arithmetic: it lies on the chain of a Swap
  const int hi = __double2hiint(absmax), e = (hi >> 20) - 1022;  // as frexp
  const bool ordinary = (e <= 256 && e >= -256) || hi == 0 || e > 1024;  // (zero, infinite)
  return ordinary ? 0 : max(-1000, min(1000, e));
}
__device__ __forceinline__ double pre_pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }  // |e| <= 1000

// G = W^T W (batch 0, K = m) and M = V^T V (batch 1, K = p), upper triangles.
struct PreGramFn {
  Tables t;
  int bw, bv, bg, bm;
  Dim m, p;
  int step, only;  // only: -1 both, else that batch index for b = 0
  __device__ GemmDesc operator()(int z, int b0) const {
    const int b = only >= 0 ? only : b0;
    const int M = m.eval(t, z), P = p.eval(t, z), ld = b == 0 ? M : P;
    const double* A = bufp(t, z, b == 0 ? bw : bv);
    GemmDesc g;
    g.M = pre_active(t, z, step) ? P : 0;
    g.N = P;
    g.K = ld;
    g.A = MatRef{A, ld, 1};
    g.B = MatRef{A, 1, ld};
    g.C = OutRef{bufp(t, z, b == 0 ? bg : bm), 1, P};
    g.alpha = 1.0; g.beta = 0.0; g.upper = 1;
    return g;
  }
};
// W' = W X (batch 0) and V' = V X (batch 1).
struct PreApplyFn {
  Tables t;
  int bw, bv, bx, bwo, bvo;
  Dim m, p;
  int step, only;
  __device__ GemmDesc operator()(int z, int b0) const {
    const int b = only >= 0 ? only : b0;
    const int M = m.eval(t, z), P = p.eval(t, z), rows = b == 0 ? M : P;
    GemmDesc g;
    g.M = pre_active(t, z, step) ? rows : 0;
    g.N = P;
    g.K = P;
    g.A = MatRef{bufp(t, z, b == 0 ? bw : bv), 1, rows};
    g.B = MatRef{bufp(t, z, bx), 1, P};
    g.C = OutRef{bufp(t, z, b == 0 ? bwo : bvo), 1, rows};
    g.alpha = 1.0; g.beta = 0.0; g.upper = 0;
    return g;
  }
};
// W = L V 2^-e, all column-major (L m x p, V p x p).
struct PreProductFn {
  Tables t;
  int bl, bv, bw;
  Dim m, p;
  __device__ GemmDesc operator()(int z, int) const {
    const int M = m.eval(t, z), P = p.eval(t, z);
    GemmDesc g;
    g.M = M; g.N = P; g.K = P;
    g.A = MatRef{bufp(t, z, bl), 1, M};
    g.B = MatRef{bufp(t, z, bv), 1, P};
    g.C = OutRef{bufp(t, z, bw), 1, M};
    g.alpha = pre_pow2(-*pre_exp_slot(t, z)); g.beta = 0.0; g.upper = 0;
    return g;
  }
};

// ---------------------------------------------------------------- norms, order, Eq. eps
// Squared column norms: of X (float, times the scale that the second QR took out and W does not) or of W
// (in the buffer where the Newton steps left it). One warp per column. l1: the sums of the magnitudes instead,
// which say whether a column vanishes or is not finite whatever its size.
struct PreNormArgs {
  Tables t;
  int bw, bw2;      // W's two buffers; float: bw = X
  int bnrm;
  Dim m, p;
  int l1;
};
template <typename T>
__global__ void pre_norm_kernel(PreNormArgs a) {
  pdl_begin();
  const int z = blockIdx.y, lane = threadIdx.x & 31;
  const int j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int p = a.p.eval(a.t, z);
  if (j >= p) return;
  double s = 0.0;
  if constexpr (sizeof(T) == 4) {
    const float* x = reinterpret_cast<const float*>(bufp(a.t, z, a.bw)) + (long)j * p;
    for (int r = lane; r < p; r += 32) {
      const double v = x[r];
      s = fma(v, v, s);
    }
    s = warp_sum(s);
    const double mx = a.t.pre[z * kPreSlots + PR_ABSMAX];
    s = ldexp(s, 2 * (qd_scale_exp(mx) - pre_exp(mx)));
  } else {
    const int m = a.m.eval(a.t, z);
    const double* x = bufp(a.t, z, pre_where(a.t, z) ? a.bw2 : a.bw) + (long)j * m;
    if (a.l1)
      for (int r = lane; r < m; r += 32) s += fabs(x[r]);
    else
      for (int r = lane; r < m; r += 32) s = fma(x[r], x[r], s);
    s = warp_sum(s);
  }
  if (lane == 0) bufp(a.t, z, a.bnrm)[j] = s;
}

// Descending order of the squared norms (bitonic, ties by index, a NaN last), the rank of Eq. eps
// (strict) with the cap, and the statistics of the truncation. One CTA per product; the keys are
// compared as integers, since a float64 comparison takes 64 clocks of a sub-partition. Block: a power
// of two of at least max(32, p) threads (1024 threads on p = 16 took 9 us, most of it in the scans).
struct PreOrderArgs {
  Tables t;
  int bnrm, bsort, bperm;
  Dim m, n, p;
  int inew;
  double eps;
  int cap;
  int wslot;
  int record;       // 0: provisional rank; 1: final; 2: final, without Newton steps (their state is left)
  int ikeep;
  int* svd_log;
  int svd_stride;
  int sort;         // 0: the columns stay in their order (nothing is truncated)
};
__global__ void __launch_bounds__(1024) pre_order_kernel(PreOrderArgs a) {
  pdl_begin();
  const int z = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int p = a.p.eval(a.t, z);
  __shared__ long long key[kPreMax];
  __shared__ short idx[kPreMax];
  __shared__ double wsum[32], s_total, s_tail;
  __shared__ int kbest, s_k;
  int np = 32;
  while (np < p) np <<= 1;
  const double* nr = bufp(a.t, z, a.bnrm);
  int ex = 0;
  if (a.record == 0) ex = pre_exp(a.t.pre[z * kPreSlots + PR_ABSMAX]);
  if (a.record == 1) ex = *pre_exp_slot(a.t, z);
  int nan_seen = 0;
  if (tid < np) {
    long long k = -2;  // padding, after everything
    if (tid < p) {
      const double v = nr[tid];
      const long long b = __double_as_longlong(v);
      nan_seen = (b & 0x7fffffffffffffffll) >= 0x7ff0000000000000ll;
      k = nan_seen ? -1 : b;
    }
    key[tid] = k;
    idx[tid] = (short)tid;
  }
  if (tid == 0) kbest = p;
  nan_seen = __syncthreads_or(nan_seen);
  if (a.sort)
  for (int size = 2; size <= np; size <<= 1)
    for (int st = size >> 1; st > 0; st >>= 1) {
      if (tid < np / 2) {
        const int lo = 2 * tid - (tid & (st - 1)), hi = lo + st;
        const bool desc = (lo & size) == 0;
        const long long ka = key[lo], kb = key[hi];
        const short ia = idx[lo], ib = idx[hi];
        const bool a_first = ka > kb || (ka == kb && ia < ib);
        if (a_first != desc) {
          key[lo] = kb;
          key[hi] = ka;
          idx[lo] = ib;
          idx[hi] = ia;
        }
      }
      __syncthreads();
    }
  // suffix sums, from the small end
  const double v = (tid < p && key[tid] > 0) ? __longlong_as_double(key[tid]) : 0.0;
  double s = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double u = __shfl_down_sync(0xffffffffu, s, o);
    if (lane + o < 32) s += u;
  }
  if (lane == 0) wsum[warp] = s;
  __syncthreads();
  if (warp == 0) {
    const int nw = blockDim.x >> 5;
    double q = lane < nw ? wsum[lane] : 0.0;
    for (int o = 1; o < nw; o <<= 1) {
      const double u = __shfl_down_sync(0xffffffffu, q, o);
      if (lane + o < 32) q += u;
    }
    const double e = __shfl_down_sync(0xffffffffu, q, 1);
    wsum[lane] = lane < 31 ? e : 0.0;  // sum of the warps behind
    if (lane == 0) s_total = q;
  }
  __syncthreads();
  const double total = s_total;
  const double tail = s + wsum[warp];  // sum of this and the smaller ones
  if (tid < p) {
    bufp(a.t, z, a.bsort)[tid] = v;
    reinterpret_cast<int*>(bufp(a.t, z, a.bperm))[tid] = idx[tid];
    if (tid >= 1 && a.eps > 0.0 && tail < a.eps * total) atomicMin(&kbest, tid);
  }
  __syncthreads();
  if (tid == 0) {
    int k = kbest;
    if (nan_seen) atomicExch(&a.t.istat[z * a.t.nis + IS_STATUS], (int)TTM_ERR_NONFINITE);
    if (!(total > 0.0)) k = 1;
    if (a.cap > 0 && k > a.cap) k = a.cap;
    if (a.ikeep >= 0 && a.t.istat[z * a.t.nis + IS_ROUND] == 0) k = bondv(a.t, z, a.ikeep);
    k = max(1, min(k, p));
    s_k = k;
    s_tail = 0.0;
  }
  __syncthreads();
  if (tid == s_k && tid < p) s_tail = tail;
  __syncthreads();
  if (tid == 0) {
    const int k = s_k;
    a.t.bond[z * a.t.nbd + a.inew] = k;
    double* st = a.t.stat + z * a.t.ns;
    int* is = a.t.istat + z * a.t.nis;
    double* pr = a.t.pre + z * kPreSlots;
    if (!a.record) {
      for (int q = 0; q < 3; ++q) pr[PR_RES + q] = 0.0;
      pr[PR_ITRACE] = total > 0.0 ? 1.0 / total : 0.0;
      *pre_exp_slot(a.t, z) = ex;
      return;
    }
    const double w = ex == 0 ? s_tail : ldexp(s_tail, 2 * ex);
    st[ST_WSUM] += w;
    st[ST_WSQRT] += sqrt(w);
    if (a.wslot >= 0) st[a.wslot] = w;
    if (k > is[IS_MAX_BOND]) is[IS_MAX_BOND] = k;
    const bool s2 = pre_active(a.t, z, 2), s3 = pre_active(a.t, z, 3);
    const double res = pr[PR_RES + (s3 ? 2 : s2 ? 1 : 0)];
    const bool bad = a.record == 1 && pre_failed(a.t, z);
    pr[PR_ABSMAX] = 0.0;  // for the next Swap
    is[IS_FALLBACK] = 0;
    if (bad) is[IS_NEWTON_BAD] += 1;
    else if (a.record == 1 && res > st[ST_NEWTON_RES]) st[ST_NEWTON_RES] = res;
    if (a.svd_log) {
      int* rec = a.svd_log + (long)z * a.svd_stride;
      rec[SR_M] = a.m.eval(a.t, z);
      rec[SR_N] = a.n.eval(a.t, z);
      rec[SR_K] = k;
      rec[SR_FALLBACK] = bad ? 1 : 0;
    }
  }
}

// V[:, j] = X[:, perm j] / |X[:, perm j]| in float64: one warp per column.
struct PreVArgs {
  Tables t;
  int bx, bperm, bv;
  Dim p;
};
__global__ void pre_v_kernel(PreVArgs a) {
  pdl_begin();
  const int z = blockIdx.y, lane = threadIdx.x & 31;
  const int j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int p = a.p.eval(a.t, z);
  if (j >= p) return;
  const int pj = max(0, min(reinterpret_cast<const int*>(bufp(a.t, z, a.bperm))[j], p - 1));
  const float* x = reinterpret_cast<const float*>(bufp(a.t, z, a.bx)) + (long)pj * p;
  double* v = bufp(a.t, z, a.bv) + (long)j * p;
  double s = 0.0;
  for (int r = lane; r < p; r += 32) {
    const double e = x[r];
    s = fma(e, e, s);
  }
  s = warp_sum(s);
  const double inv = s > 0.0 ? rsqrt(s) : 0.0;
  for (int r = lane; r < p; r += 32) v[r] = s > 0.0 ? (double)x[r] * inv : (r == pj ? 1.0 : 0.0);
}

// ---------------------------------------------------------------- transport inside a cluster
// A cluster of G CTAs hands a block of columns on through distributed shared memory: it stays where its
// owner holds it, the owner's release-arrival on one mbarrier per receiver says that it is final, and
// the receivers read it there. Slot of block c: c mod 32 (a multiple of G, so that the CTAs that use
// a slot are the same on every turn, and the chain cannot run 32 blocks ahead of a CTA, since every
// CTA owns one in G); phase: c / 32.
constexpr int kQdSlots = 32;
constexpr int kElimCluster = 16;      // largest cluster of the elimination
constexpr int kElimClusterMax = 384;  // largest p on a cluster
__device__ __forceinline__ uint32_t qc_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t qc_map(uint32_t addr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void qc_init(uint64_t* bars, int tid) {
  if (tid < kQdSlots) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(qc_smem(bars + tid)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void qc_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Block c is final in this CTA (its writers have been joined with the calling warp): tells the CTAs
// that hold a block from c on. nc: blocks of the matrix.
__device__ __forceinline__ void qc_publish(uint64_t* bars, int c, int nc, int G, int b, int lane) {
  if (lane < G && lane != b) {
    const int last = lane < nc ? lane + (nc - 1 - lane) / G * G : -1;
    if (last >= c)
      asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(
                       qc_map(qc_smem(bars + (c & (kQdSlots - 1))), lane))
                   : "memory");
  }
}
__device__ __forceinline__ bool qc_wait(uint64_t* bars, int c) {
  const uint32_t bar = qc_smem(bars + (c & (kQdSlots - 1))), parity = (uint32_t)(c / kQdSlots) & 1;
  for (int polls = 0; polls < kQdPolls; ++polls) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}
__device__ __forceinline__ double qc_ld(uint32_t addr, double) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr) : "memory");
  return v;
}
// ---------------------------------------------------------------- elimination of G
// U of G = L_G U without pivoting (the columns come in descending order): U_ij for i <= j, stored
// at [j + i p]. A pivot that cancelled to rounding level counts as zero and eliminates nothing.
// Distributed like the QR: blocks of columns are dealt out to G CTAs and handed on through the
// cluster's shared memory, or past kElimClusterMax through the polled exchange buffer.
struct PreElimArgs {
  Tables t;
  int bg, bu;
  Dim p;
  int step;
  int G, blocks_ub, ld_ub;
  unsigned long long* ex;
  unsigned long long* ex_next;
  long ex_stride, clear_n;
};
// 1 / d for a positive d: float32 seed and one step of Householder's third-order iteration (as the tau of
// ttm_qrd.cuh); 0 for a pivot d that is not positive or
// below 2^-46 of g0, its column's squared norm (by the high words).
__device__ __forceinline__ double pre_pivot_inv(double d, double g0) {
  const int dh = __double2hiint(d), gh = __double2hiint(g0);
  if (!(dh > 0 && dh < 0x7ff00000 && dh > gh - (46 << 20))) return 0.0;
  const int e = (dh >> 20) - 1023;
  if (e <= -900 || e >= 900) return 1.0 / d;
  const int sh = dh - (e << 20), lo = __double2loint(d);
  const unsigned u =
      __float_as_uint(__fdividef(1.f, __uint_as_float(((unsigned)(sh - 0x38000000) << 3) | ((unsigned)lo >> 29))));
  const double q0 = __hiloint2double((int)(u >> 3) + 0x38000000, (int)(u << 29));
  const double r = fma(-__hiloint2double(sh, lo), q0, 1.0);
  const double q = fma(q0 * r, 1.0 + r, q0);
  return __hiloint2double(__double2hiint(q) - (e << 20), __double2loint(q));
}

// One block of kElB columns at a time: a hand-over costs some 1500 clk whatever it carries. The columns
// of a block are eliminated among themselves by four warps (one per sub-partition: a float64
// instruction occupies its sub-partition for 64 clk), with the next block's update before them on the
// chain; all other updates are off it. The reciprocals travel in two rows of the block's last columns that
// lie above the diagonal. Mean over the calls of a product of 1D fields (L = 20, chi = 48 capped at 64, p to
// 128) 19.9 us against 26.4 with one column per hand-over, of an L = 18, chi = 160 product (p to 320)
// 296 us against 369; what bounds it is the chain: at p = 320, 3100 clk of a block's 7600 are the update of
// the next one at the float64 rate, 2900 its own columns.
constexpr int kElB = 4;
constexpr int kElimSmem = 216 * 1024;  // blocks of one CTA
template <bool CL>
__global__ void __launch_bounds__(kQdThreads, 3) pre_elim_kernel(PreElimArgs a) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char qd_raw[];
  const int G = a.G, z = blockIdx.x / G, b = blockIdx.x % G;
  const int p = a.p.eval(a.t, z);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (long e = (long)b * kQdThreads + tid; e < a.clear_n; e += (long)G * kQdThreads)
    a.ex_next[z * a.ex_stride + e] = kQdEmpty;
  const int nb = (p + kElB - 1) / kElB, nl = b < nb ? (nb - b + G - 1) / G : 0;  // blocks, in all and here
  if (!pre_active(a.t, z, a.step)) return;  // alike in all CTAs of the product
  if (!CL && nl == 0) return;
  const int ld = a.ld_ub;
  double* cols = reinterpret_cast<double*>(qd_raw);  // [blocks_ub][kElB][ld], a block from its first row down
  double* xs = cols + (long)a.blocks_ub * kElB * ld;  // [kElB][ld]
  __shared__ int s_abort;
  __shared__ __align__(8) uint64_t bars[CL ? kQdSlots : 1];
  if (tid == 0) s_abort = 0;
  if constexpr (CL) qc_init(bars, tid);
  const double* Gm = bufp(a.t, z, a.bg);
  double* U = bufp(a.t, z, a.bu);
  for (int e = tid; e < nl * p * kElB; e += kQdThreads) {
    const int u = e % kElB, l = e / (kElB * p), i = e / kElB - l * p;
    const int c = (b + G * l) * kElB + u;
    if (i >= c - u) cols[(l * kElB + u) * ld + i] = (c < p && i >= c) ? Gm[c + (long)i * p] : 0.0;  // row c of the upper triangle
  }
  unsigned long long* ex = a.ex + z * a.ex_stride;
  // Warps 0 to 3: eliminates block blk (local l) within itself and hands it on. gl: lane u's squared
  // norm of column u.
  auto factor = [&](int blk, int l, double gl) {
    double* ac = cols + l * kElB * ld;
    const int cb = blk * kElB;
    const bool next = blk + 1 < nb && G > 1;
    double inv[kElB];
#pragma unroll
    for (int k = 0; k < kElB; ++k) {
      asm volatile("bar.sync 2, 128;" ::: "memory");
      inv[k] = 0.0;
      if (cb + k >= p) continue;
      inv[k] = pre_pivot_inv(ac[k * ld + cb + k], __shfl_sync(0xffffffffu, gl, k));
      double fl = 0.0;
      if (lane > k && lane < kElB && cb + lane < p) fl = ac[k * ld + cb + lane] * inv[k];
      double f[kElB];
#pragma unroll
      for (int u = k + 1; u < kElB; ++u) f[u] = __shfl_sync(0xffffffffu, fl, u);
      for (int i = cb + tid; i < p; i += 128) {
        const double x = ac[k * ld + i];
#pragma unroll
        for (int u = k + 1; u < kElB; ++u) ac[u * ld + i] = fma(-f[u], x, ac[u * ld + i]);
        if (!CL && next) {
          double y = x;
          if (k >= 2 && i < cb + 2) y = i == cb ? inv[2 * k - 4] : inv[2 * k - 3];
          qd_st(ex + (long)(cb + k) * p + i, QdBits<double>::to(y));
        }
      }
    }
    if (tid < 2 && cb + tid < p) {
      ac[2 * ld + cb + tid] = tid == 0 ? inv[0] : inv[1];
      ac[3 * ld + cb + tid] = tid == 0 ? inv[2] : inv[3];
    }
    if (CL && next) {
      asm volatile("bar.sync 2, 128;" ::: "memory");
      if (warp == 0) qc_publish(bars, blk, nb, G, b, lane);
    }
  };
  // The 16 factors of the update of block c0 / kElB by the block at x (first column jb), one per lane.
  auto factors = [&](const double* x, int jb, int c0) {
    const int k = lane & 3, c = c0 + (lane >> 2);
    return lane < 16 && c < p ? x[k * ld + c] * x[(2 + (k >> 1)) * ld + jb + (k & 1)] : 0.0;
  };
  auto update = [&](const double* x, double* ac, const double (&f)[16], int i) {
    const double x0 = x[i], x1 = x[ld + i], x2 = x[2 * ld + i], x3 = x[3 * ld + i];
#pragma unroll
    for (int u = 0; u < kElB; ++u)
      ac[u * ld + i] = fma(-f[4 * u + 3], x3, fma(-f[4 * u + 2], x2, fma(-f[4 * u + 1], x1, fma(-f[4 * u], x0, ac[u * ld + i]))));
  };
  __syncthreads();
  if constexpr (CL) qc_sync();
  if (b == 0 && nl > 0 && warp < 4) factor(0, 0, lane < kElB && lane < p ? Gm[lane * (long)(p + 1)] : 0.0);
  __syncthreads();
  int lj = 0, jr = 0;
  for (int blk = 0; blk < nb; ++blk) {
    if (nl == 0 || b + G * (nl - 1) < blk) break;  // no block from blk on is held here
    const bool mine = jr == b;
    const int jb = blk * kElB, cb = jb + kElB;
    const int nr = jr + 1 == G ? 0 : jr + 1, nlj = jr + 1 == G ? lj + 1 : lj;
    const bool chain = nr == b && blk + 1 < nb;
    const double* x = mine ? cols + lj * kElB * ld : xs;
    double gl = 0.0;
    if (chain && lane < kElB && cb + lane < p) gl = Gm[(cb + lane) * (long)(p + 1)];
    if (!mine) {
      const int k0 = 2 * (tid >> 7);  // two columns per half of the threads
      if (CL) {
        if (!qc_wait(bars, blk)) s_abort = 1;
        const uint32_t rem = qc_map(qc_smem(cols + (lj * kElB + k0) * ld), jr);
        for (int i = jb + (tid & 127); i < p; i += 128) {
          const double y0 = qc_ld(rem + (uint32_t)(i * 8), 0.0), y1 = qc_ld(rem + (uint32_t)((ld + i) * 8), 0.0);
          xs[k0 * ld + i] = y0;
          xs[(k0 + 1) * ld + i] = y1;
        }
      } else {
        const unsigned long long* s0 = ex + (long)(jb + k0) * p;
        for (int i = jb + (tid & 127); i < p; i += 256) {
          unsigned long long bits[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int r = i + 128 * (u >> 1);
            bits[u] = r < p ? qd_ld(s0 + (u & 1) * (long)p + r) : 0;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int r = i + 128 * (u >> 1);
            if (r >= p) continue;
            for (int polls = 0; bits[u] == kQdEmpty && polls < kQdPolls; ++polls) bits[u] = qd_ld(s0 + (u & 1) * (long)p + r);
            if (bits[u] == kQdEmpty) s_abort = 1;
            xs[(k0 + (u & 1)) * ld + r] = QdBits<double>::from(bits[u]);
          }
        }
      }
      __syncthreads();
    }
    if (chain) {
      if (warp < 4) {
        const double fl = factors(x, jb, cb);
        double f[16];
#pragma unroll
        for (int t = 0; t < 16; ++t) f[t] = __shfl_sync(0xffffffffu, fl, t);
        for (int i = cb + tid; i < p; i += 128) update(x, cols + nlj * kElB * ld, f, i);
        factor(blk + 1, nlj, gl);
      }
      __syncthreads();
    }
    if (mine) {  // rows jb.. of U; zeros for a pivot that does not count
      for (int k = 0; k < kElB && jb + k < p; ++k) {
        const bool counts = x[(2 + (k >> 1)) * ld + jb + (k & 1)] != 0.0;
        for (int i = jb + k + tid; i < p; i += kQdThreads) U[i + (long)(jb + k) * p] = counts ? x[k * ld + i] : 0.0;
      }
    }
    // the other blocks, in chunks of 32 rows dealt out to the warps
    int t = warp;
    for (int l = chain ? nlj + 1 : lj + (b > jr ? 0 : 1); l < nl; ++l) {
      const int c0 = (b + G * l) * kElB, n = (p - c0 + 31) >> 5;
      if (t < n) {
        const double fl = factors(x, jb, c0);
        double f[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) f[u] = __shfl_sync(0xffffffffu, fl, u);
        for (; t < n; t += 8) {
          const int i = c0 + 32 * t + lane;
          if (i < p) update(x, cols + l * kElB * ld, f, i);
        }
      }
      t -= n;
    }
    lj = nlj;
    jr = nr;
    __syncthreads();
    if (s_abort) {
      if (tid == 0) atomicExch(&a.t.istat[z * a.t.nis + IS_STATUS], (int)TTM_ERR_TIMEOUT);
      break;
    }
  }
  if constexpr (CL) qc_sync();  // no CTA leaves while another may still read its columns
}

// X of a Newton step from M and the eliminated G (U), with the filters of ttm_newton.cuh.
struct PreXArgs {
  Tables t;
  int bu, bm, bx;
  Dim p;
  int bsort, ikprov;
  int step, islot_frozen;
};
__global__ void __launch_bounds__(256) pre_x_kernel(PreXArgs a) {
  pdl_begin();
  const int z = blockIdx.z;
  const int p = a.p.eval(a.t, z);
  const int i = blockIdx.x * 32 + (threadIdx.x & 31), j = blockIdx.y * 8 + (threadIdx.x >> 5);
  if (blockIdx.x * 32 >= p || blockIdx.y * 8 >= p || !pre_active(a.t, z, a.step)) return;
  double smax = 0.0;
  int frozen = 0;
  if (i < p && j < p) {
    const double* U = bufp(a.t, z, a.bu);
    const double* M = bufp(a.t, z, a.bm);
    const int lo = min(i, j), hi = max(i, j);
    const double e = M[lo + (long)hi * p] - (i == j ? 1.0 : 0.0);
    double x;
    if (i == j) {
      x = 1.0 - 0.5 * e;
      smax = 0.5 * fabs(e);
    } else {
      // The first two steps take the couplings after elimination. From then on what the small columns
      // carry of the large ones is at rounding level for most Swaps, and G itself serves. Not where two
      // small columns were still rotated by 1e-3 or more: that rotation hands on what the other one carried,
      // the next corrections stay at that size, and the Swap ends in the float64 Jacobi (five of 435 at
      // chi = 512, 0.6 s each; none with an elimination in steps 2 and 3 too, two more launches per Swap).
      const double g = a.step < 2 ? U[hi + (long)lo * p] : U[lo + (long)hi * p];
      const double di = U[i + (long)i * p], dj = U[j + (long)j * p];
      const double dmax = fmax(di, dj);
      const int kp = bondv(a.t, z, a.ikprov);
      const double dcut = bufp(a.t, z, a.bsort)[max(0, min(kp, p) - 1)];
      const double itr = a.t.pre[z * kPreSlots + PR_ITRACE];
      const double num = 0.5 * e * (di + dj) - g, den = di - dj;
      double s = 0.0;
      const double nt = num * itr;
      // |num| > kNewtonFloor sqrt(dmax trace), squared and divided by trace^2
      if (dmax >= kNewtonRelevance * dcut && nt * nt > kNewtonFloor * kNewtonFloor * (dmax * itr)) {
        if (fabs(num) <= kNewtonMaxS * fabs(den)) s = num / den;
        else frozen = i < j ? 1 : 0;
      }
      smax = fmax(fabs(s), 0.5 * fabs(e));
      x = s - 0.5 * e;
    }
    bufp(a.t, z, a.bx)[i + (long)j * p] = x;
  }
  if (a.step == 0) return;
  // the largest correction (non-negative doubles order like their bit patterns; a NaN is above all)
  long long mb = __double_as_longlong(smax) & 0x7fffffffffffffffll;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const long long u = __shfl_xor_sync(0xffffffffu, mb, o);
    mb = u > mb ? u : mb;
    frozen += __shfl_xor_sync(0xffffffffu, frozen, o);
  }
  __shared__ long long s_max[8];
  __shared__ int s_frz[8];
  if ((threadIdx.x & 31) == 0) {
    s_max[threadIdx.x >> 5] = mb;
    s_frz[threadIdx.x >> 5] = frozen;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int f = 0;
    for (int q = 0; q < 8; ++q) {
      mb = s_max[q] > mb ? s_max[q] : mb;
      f += s_frz[q];
    }
    if (mb > 0)
      atomicMax(reinterpret_cast<unsigned long long*>(&a.t.pre[z * kPreSlots + PR_RES + a.step - 1]),
                (unsigned long long)mb);
    if (a.step == 1 && f > 0) atomicAdd(&a.t.istat[z * a.t.nis + a.islot_frozen], f);
  }
}

// IS_FALLBACK for the products whose last Newton step did not converge, with W = L and V = I for the
// float64 Jacobi that follows. One launch, empty for the others.
struct PreRescueArgs {
  Tables t;
  int bl, bw, bv;
  Dim m, p;
};
__global__ void pre_rescue_kernel(PreRescueArgs a) {
  pdl_begin();
  const int z = blockIdx.y;
  const bool bad = pre_failed(a.t, z);
  if (blockIdx.x == 0 && threadIdx.x == 0) a.t.istat[z * a.t.nis + IS_FALLBACK] = bad ? 1 : 0;
  if (!bad) return;
  const int m = a.m.eval(a.t, z), p = a.p.eval(a.t, z);
  const double* L = bufp(a.t, z, a.bl);
  const double inv = pre_pow2(-*pre_exp_slot(a.t, z));
  double* W = bufp(a.t, z, a.bw);
  for (long e = (long)blockIdx.x * blockDim.x + threadIdx.x; e < (long)m * p; e += (long)gridDim.x * blockDim.x)
    W[e] = L[e] * inv;
}

// New left carriage, row-major [m][k]: column perm[j] of W, times 2^e where W leaves it out (scaled). 32 x 32
// tiles through shared memory.
struct PreLeftArgs {
  Tables t;
  int bw, bw2, bperm, bout;
  Dim m;
  int ik;
  int scaled;
};
__global__ void __launch_bounds__(256) pre_left_kernel(PreLeftArgs a) {
  pdl_begin();
  const int z = blockIdx.z;
  const int m = a.m.eval(a.t, z), k = bondv(a.t, z, a.ik);
  const int r0 = blockIdx.x * 32, j0 = blockIdx.y * 32;
  if (r0 >= m || j0 >= k) return;
  __shared__ double tile[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int ex = a.scaled ? *pre_exp_slot(a.t, z) : 0;
  const double* W = bufp(a.t, z, pre_where(a.t, z) ? a.bw2 : a.bw);
  const int* perm = reinterpret_cast<const int*>(bufp(a.t, z, a.bperm));
  for (int q = ty; q < 32; q += 8)
    if (j0 + q < k && r0 + tx < m) tile[q][tx] = W[(long)perm[j0 + q] * m + r0 + tx];
  __syncthreads();
  double* out = bufp(a.t, z, a.bout);
  for (int q = ty; q < 32; q += 8)
    if (r0 + q < m && j0 + tx < k) {
      const double v = tile[tx][q];
      out[(long)(r0 + q) * k + j0 + tx] = ex == 0 ? v : v * pre_pow2(ex);
    }
}

}  // namespace ttm
