// ttm_pre.cuh -- the Swap SVD (Fig. 1C, Eq. eps) by a preconditioned float32 Jacobi and float64
// Newton steps on the reduced problem; the default for Swap matrices of at most 1024 rows and
// 1024 columns of the smaller side.
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
// Bound by latencies: the chains of the two QRs (about 1.3 and 0.7 us per column), of the inner rounds
// of the Jacobi and of the elimination. Measured per product (GB300) against three float32 passes
// with V, three to five Newton steps and a saved state: 2D field, d = 4, chi = 64 332 -> 153 ms; 3D
// field, d = 8, chi = 96 503 -> 205 ms; random L = 10 61 -> 21 ms; chi = 160, L = 18 1616 -> 825 ms.
#pragma once
#include <cooperative_groups.h>
#include "ttm_common.cuh"
#include "ttm_jres.cuh"
#include "ttm_newton.cuh"
#include "ttm_qrd.cuh"
#include "ttm_svd.cuh"

namespace cg = cooperative_groups;

namespace ttm {

constexpr int kPreMax = 1024;       // largest p and m
constexpr int kPreSweeps = 30;      // sweep limit (the Newton steps and the fallback finish what is left)
constexpr double kPreTol = 4 * 5.96e-8;  // times sqrt(p): couplings below are not rotated
constexpr float kPreBig = 1e-3f;    // a sweep without a coupling above this is the last: the couplings
                                    // it leaves are of the order of its largest one squared. (With 1e-2
                                    // 5 of 2300 Swaps needed the float64 Jacobi, with 1e-3 none of 8600, at
                                    // the same time per product.)
constexpr float kPreRidge = 1e-15f; // added to the diagonal of R2 (max |R1| = 1): no column of X vanishes

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
// W = L V, all column-major (L m x p, V p x p).
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
    g.alpha = 1.0; g.beta = 0.0; g.upper = 0;
    return g;
  }
};

// ---------------------------------------------------------------- float32 Jacobi without V
// Blocks of 16 columns in a round-robin tournament, one CTA of 16 warps per block pair: a warp
// keeps one column of the first block in registers and meets the 16 columns of the second block,
// staged in shared memory, in 16 inner rounds (the schedule of ttm_jres.cuh). Squared norms are
// formed when a column is staged and carried through the rotations (a' = a - t g, b' = b + t g;
// formed again when b' or a' lost more than 90 %), so a visit costs one dot product and one warp
// reduction. The CTAs of a product meet at a cluster barrier (up to 8 CTAs) or at a counter in
// global memory; products of a batch do not wait for each other.
// Bound by the latency of an inner round (load, dot, reduction, rotation, CTA barrier).
__device__ __forceinline__ int pj_ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
constexpr int kPjB = 16;
constexpr int kPjThreads = kPjB * 32;
constexpr int kPjPolls = 1 << 22;
struct PreJacArgs {
  Tables t;
  int bx;             // X: p x p float column-major (in/out)
  Dim p;
  int G;              // CTAs per product (half the padded number of blocks, upper bound)
  int ngroup;         // groups of G CTAs in the launch
  int cluster;        // 1: a group is one cluster
  int max_sweeps;
  int* counters;      // [nz][stride]: large couplings per sweep, then at [kPjBarrier] the barrier
  int stride;
  float tol, big;
  int flop_slot, sweep_slot;
  int* svd_log;
  int svd_stride, svd_field;
};
constexpr int kPjBarrier = 39;  // kPreSweeps < kPjBarrier < the counters' stride

template <int R>
__global__ void __launch_bounds__(kPjThreads, 1) jacobi_pre_kernel(PreJacArgs a) {
  extern __shared__ __align__(16) unsigned char pj_raw[];
  constexpr int B = kPjB, MR = 32 * R;
  constexpr int VW = JrVec<float, R>::VW;
  float* sc = reinterpret_cast<float*>(pj_raw);  // [2B][MR]
  __shared__ float nrm[2 * B];
  __shared__ int s_big, s_stop;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int i = blockIdx.x % a.G;
  unsigned long long visits = 0, rots = 0;
  for (int z = blockIdx.x / a.G; z < a.t.nz; z += a.ngroup) {
    const int p = a.p.eval(a.t, z);
    const int nb = (p + B - 1) / B, nbp = nb + (nb & 1), half = nbp / 2;
    int* cnt = a.counters + (long)z * a.stride;
    const bool here = i < half;
    if (!here && !a.cluster) continue;
    float* X = reinterpret_cast<float*>(bufp(a.t, z, a.bx));
    const bool vec = (p % VW) == 0;
    int barriers = 0, sweep = 0;
    if (threadIdx.x == 0) {
      s_big = 0;
      s_stop = 0;
    }
    __syncthreads();
    for (; sweep < a.max_sweeps; ++sweep) {
      int rot_any = 0;
      for (int r = 0; r < nbp - 1; ++r) {
        if (here) {
          int P, Q;
          jr_pair(nbp, r, i, P, Q);
          const int gp = P * B + w, gq = Q * B + w;
          float x[R], y[R];
          auto stage = [&](int g, float (&v)[R]) {
            if (g < p) {
              const float* col = X + (long)g * p;
              if (vec) {
                using V = typename JrVecT<float, VW>::type;
#pragma unroll
                for (int q = 0; q < R / VW; ++q) {
                  const int row = 32 * VW * q + VW * lane;
                  V u{};
                  if (row < p) u = __ldcg(reinterpret_cast<const V*>(col + row));
                  const float* e = reinterpret_cast<const float*>(&u);
#pragma unroll
                  for (int s = 0; s < VW; ++s) v[VW * q + s] = e[s];
                }
              } else {
#pragma unroll
                for (int q = 0; q < R; ++q) {
                  const int row = 32 * VW * (q / VW) + VW * lane + q % VW;
                  v[q] = row < p ? __ldcg(col + row) : 0.f;
                }
              }
            } else {
#pragma unroll
              for (int q = 0; q < R; ++q) v[q] = 0.f;
            }
          };
          auto unstage = [&](int g, const float (&v)[R]) {
            if (g >= p) return;
            float* col = X + (long)g * p;
            if (vec) {
              using V = typename JrVecT<float, VW>::type;
#pragma unroll
              for (int q = 0; q < R / VW; ++q) {
                const int row = 32 * VW * q + VW * lane;
                V u;
                float* e = reinterpret_cast<float*>(&u);
#pragma unroll
                for (int s = 0; s < VW; ++s) e[s] = v[VW * q + s];
                if (row < p) *reinterpret_cast<V*>(col + row) = u;
              }
            } else {
#pragma unroll
              for (int q = 0; q < R; ++q) {
                const int row = 32 * VW * (q / VW) + VW * lane + q % VW;
                if (row < p) col[row] = v[q];
              }
            }
          };
          auto norm2 = [&](const float (&v)[R]) {
            float s0 = 0.f, s1 = 0.f;
#pragma unroll
            for (int q = 0; q < R; ++q) {
              if (q & 1) s1 = fmaf(v[q], v[q], s1);
              else s0 = fmaf(v[q], v[q], s0);
            }
            return jr_sum(s0 + s1);
          };
          // rotates (x, na) against (y, nb2) if their coupling is above tol
          auto visit = [&](float& na, float& nb2) -> bool {
            constexpr int NA = R >= 4 ? 4 : R;
            float g[NA];
#pragma unroll
            for (int u = 0; u < NA; ++u) g[u] = 0.f;
#pragma unroll
            for (int q = 0; q < R; ++q) g[q % NA] = fmaf(x[q], y[q], g[q % NA]);
#pragma unroll
            for (int u = 1; u < NA; ++u) g[0] += g[u];
            const float g2 = jr_sum(g[0]);
            const float cpl = fabsf(g2) * rsqrtf(na) * rsqrtf(nb2);
            if (!(cpl > a.tol)) return false;  // also a padding column (0 inf = NaN)
            if (cpl > a.big) rot_any = 1;
            float c, s;
            if (!jr_rot<float>(na, nb2, g2, c, s)) return false;
            const float tg = __fdividef(s, c) * g2;
#pragma unroll
            for (int q = 0; q < R; ++q) {
              const float xp = x[q], yq = y[q];
              x[q] = c * xp - s * yq;
              y[q] = fmaf(s, xp, c * yq);
            }
            const float na1 = na - tg, nb1 = nb2 + tg;
            na = na1 < 0.1f * na ? norm2(x) : na1;
            nb2 = nb1 < 0.1f * nb2 ? norm2(y) : nb1;
            return true;
          };
          stage(gp, x);
          stage(gq, y);
          float na = norm2(x);
          {
            const float nq = norm2(y);
            if (lane == 0) nrm[B + w] = nq;
          }
          jr_store<float, R>(sc + (B + w) * MR, lane, y);
          if (r == 0) {  // the pairs inside each block
            jr_store<float, R>(sc + w * MR, lane, x);
            if (lane == 0) nrm[w] = na;
            __syncthreads();
            for (int s = 0; s < B - 1; ++s) {
              const int hb = w < B / 2 ? 0 : B, iw = w % (B / 2);
              int cp, cq;
              jr_pair(B, s, iw, cp, cq);
              cp += hb;
              cq += hb;
              jr_load<float, R>(sc + cp * MR, lane, x);
              jr_load<float, R>(sc + cq * MR, lane, y);
              float n1 = nrm[cp], n2 = nrm[cq];
              if (lane == 0) ++visits;
              if (visit(n1, n2)) {
                jr_store<float, R>(sc + cp * MR, lane, x);
                jr_store<float, R>(sc + cq * MR, lane, y);
                __syncwarp();
                if (lane == 0) {
                  nrm[cp] = n1;
                  nrm[cq] = n2;
                  ++rots;
                }
              }
              __syncthreads();
            }
            jr_load<float, R>(sc + w * MR, lane, x);
            na = nrm[w];
          }
          __syncthreads();
          for (int s = 0; s < B; ++s) {
            const int q = B + (w + s) % B;
            jr_load<float, R>(sc + q * MR, lane, y);
            float nq = nrm[q];
            __syncwarp();
            if (lane == 0) ++visits;
            if (visit(na, nq)) {
              jr_store<float, R>(sc + q * MR, lane, y);
              if (lane == 0) {
                nrm[q] = nq;
                ++rots;
              }
            }
            __syncthreads();
          }
          unstage(gp, x);
          jr_load<float, R>(sc + (B + w) * MR, lane, y);
          unstage(gq, y);
        }
        // the product's CTAs exchange columns
        const bool last = r == nbp - 2;
        if (last && rot_any && lane == 0) atomicOr(&s_big, 1);
        if (half > 1 || last) {
          __syncthreads();
          if (last && threadIdx.x == 0 && s_big) {
            atomicAdd(&cnt[sweep], 1);
            s_big = 0;
          }
        }
        if (a.cluster) {
          asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
        } else if (half > 1) {
          ++barriers;
          if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(&cnt[kPjBarrier], 1);
            int polls = 0;
            while (pj_ld_acquire(&cnt[kPjBarrier]) < barriers * half && ++polls < kPjPolls) {}
            if (polls >= kPjPolls) {
              s_stop = 1;
              atomicExch(&a.t.istat[z * a.t.nis + IS_STATUS], (int)TTM_ERR_TIMEOUT);
            }
          }
          __syncthreads();
          if (s_stop) break;
        } else if (last) {
          __threadfence();
          __syncthreads();
        }
      }
      if (s_stop || __ldcg(&cnt[sweep]) == 0) break;
    }
    if (i == 0 && threadIdx.x == 0) {
      const int used = min(sweep + 1, a.max_sweeps);
      int* is = a.t.istat + z * a.t.nis;
      if (used > is[IS_SWEEPS_MAX]) is[IS_SWEEPS_MAX] = used;
      a.t.stat[z * a.t.ns + a.sweep_slot] += used;
      if (a.svd_log) a.svd_log[(long)z * a.svd_stride + a.svd_field] = used;
    }
    // 2 p flops per visit, 6 p per rotation
    if (lane == 0 && visits) atomicAdd(&a.t.stat[a.flop_slot], 2.0 * p * (double)visits + 6.0 * p * (double)rots);
    visits = rots = 0;
    __syncthreads();
  }
}

// ---------------------------------------------------------------- norms, order, Eq. eps
// Squared column norms: of X (float, times the scale that the second QR took out) or of W (in the
// buffer where the Newton steps left it). One warp per column.
struct PreNormArgs {
  Tables t;
  int bw, bw2;      // W's two buffers; float: bw = X
  int bnrm;
  Dim m, p;
};
template <typename T>
__global__ void pre_norm_kernel(PreNormArgs a) {
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
    s = ldexp(s, 2 * qd_scale_exp(a.t.pre[z * kPreSlots + PR_ABSMAX]));
  } else {
    const int m = a.m.eval(a.t, z);
    const double* x = bufp(a.t, z, pre_where(a.t, z) ? a.bw2 : a.bw) + (long)j * m;
    for (int r = lane; r < m; r += 32) s = fma(x[r], x[r], s);
    s = warp_sum(s);
  }
  if (lane == 0) bufp(a.t, z, a.bnrm)[j] = s;
}

// Descending order of the squared norms (bitonic, ties by index, a NaN last), the rank of Eq. eps
// (strict) with the cap, and the statistics of the truncation. One CTA per product; the keys are
// compared as integers, since a float64 comparison takes 64 clocks of a sub-partition.
struct PreOrderArgs {
  Tables t;
  int bnrm, bsort, bperm;
  Dim m, n, p;
  int inew;
  double eps;
  int cap;
  int wslot, record;
  int ikeep;
  int* svd_log;
  int svd_stride;
};
__global__ void __launch_bounds__(1024) pre_order_kernel(PreOrderArgs a) {
  const int z = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int p = a.p.eval(a.t, z);
  __shared__ long long key[kPreMax];
  __shared__ short idx[kPreMax];
  __shared__ double wsum[32], s_total, s_tail;
  __shared__ int kbest, s_k;
  int np = 32;
  while (np < p) np <<= 1;
  const double* nr = bufp(a.t, z, a.bnrm);
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
    double q = wsum[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
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
      return;
    }
    const double w = s_tail;
    st[ST_WSUM] += w;
    st[ST_WSQRT] += sqrt(w);
    if (a.wslot >= 0) st[a.wslot] = w;
    if (k > is[IS_MAX_BOND]) is[IS_MAX_BOND] = k;
    const bool s2 = pre_active(a.t, z, 2), s3 = pre_active(a.t, z, 3);
    const double res = pr[PR_RES + (s3 ? 2 : s2 ? 1 : 0)];
    const bool bad = pre_failed(a.t, z);
    pr[PR_ABSMAX] = 0.0;  // for the next Swap
    is[IS_FALLBACK] = 0;
    if (bad) is[IS_NEWTON_BAD] += 1;
    else if (res > st[ST_NEWTON_RES]) st[ST_NEWTON_RES] = res;
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

// ---------------------------------------------------------------- elimination of G
// U of G = L_G U without pivoting (the columns come in descending order): U_ij for i <= j, stored
// at [j + i p]. A pivot that cancelled to rounding level counts as zero and eliminates nothing.
// Distributed like the QR (columns dealt out to G CTAs, column j polled from the exchange buffer);
// a step is one reciprocal and one update, no reduction.
struct PreElimArgs {
  Tables t;
  int bg, bu;
  Dim p;
  int step;
  int G, cols_ub, ld_ub;
  unsigned long long* ex;
  unsigned long long* ex_next;
  long ex_stride, clear_n;
};
// 1 / d for a positive d: float32 seed and one cubic step; 0 for a pivot d that is not positive or
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

__global__ void __launch_bounds__(kQdThreads) pre_elim_kernel(PreElimArgs a) {
  extern __shared__ __align__(16) unsigned char qd_raw[];
  const int G = a.G, z = blockIdx.x / G, b = blockIdx.x % G;
  const int p = a.p.eval(a.t, z);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (long e = (long)b * kQdThreads + tid; e < a.clear_n; e += (long)G * kQdThreads)
    a.ex_next[z * a.ex_stride + e] = kQdEmpty;
  const int nl = b < p ? (p - b + G - 1) / G : 0;
  if (nl == 0 || !pre_active(a.t, z, a.step)) return;  // the second alike in all CTAs of the product
  double* cols = reinterpret_cast<double*>(qd_raw);     // [cols_ub][ld], column c from row c down
  const int ld = a.ld_ub;
  double* xs = cols + (long)a.cols_ub * ld;             // [ld]
  __shared__ int s_abort;
  if (tid == 0) s_abort = 0;
  const double* Gm = bufp(a.t, z, a.bg);
  double* U = bufp(a.t, z, a.bu);
  for (int e = tid; e < nl * p; e += kQdThreads) {
    const int l = e / p, i = e - l * p, c = b + G * l;
    if (i >= c) cols[l * ld + i] = Gm[c + (long)i * p];  // row c of the upper triangle
  }
  unsigned long long* ex = a.ex + z * a.ex_stride;
  __syncthreads();
  if (G > 1 && b == 0)
    for (int i = tid; i < p; i += kQdThreads) qd_st(ex + i, QdBits<double>::to(cols[i]));
  int lj = 0, jr = 0;
  for (int j = 0; j < p; ++j) {
    if (b + G * (nl - 1) < j) break;  // no column from j on is held here
    const bool mine = jr == b;
    const int nxt = j + 1;
    const int nr = jr + 1 == G ? 0 : jr + 1, nlj = jr + 1 == G ? lj + 1 : lj;
    const int lc = (nr == b && nxt < p) ? nlj : -1;
    const double* x = mine ? cols + lj * ld : xs;
    const int base = j & ~31;
    const double g0 = __ldg(Gm + j + (long)j * p);
    if (!mine) {
      constexpr int NB = 4;
      for (int i0 = base + tid; i0 < p; i0 += kQdThreads * NB) {
        unsigned long long bits[NB];
#pragma unroll
        for (int u = 0; u < NB; ++u) {
          const int i = i0 + kQdThreads * u;
          bits[u] = (i >= j && i < p) ? qd_ld(ex + (long)j * p + i) : 0;
        }
#pragma unroll
        for (int u = 0; u < NB; ++u) {
          const int i = i0 + kQdThreads * u;
          if (i >= p) break;
          for (int polls = 0; bits[u] == kQdEmpty && polls < kQdPolls; ++polls) bits[u] = qd_ld(ex + (long)j * p + i);
          if (bits[u] == kQdEmpty) s_abort = 1;
          xs[i] = QdBits<double>::from(bits[u]);
        }
      }
    }
    __syncthreads();
    if (s_abort) {
      if (tid == 0) atomicExch(&a.t.istat[z * a.t.nis + IS_STATUS], (int)TTM_ERR_TIMEOUT);
      return;
    }
    const double inv = (warp < 4 || !(lc >= 0)) ? pre_pivot_inv(x[j], g0) : 0.0;
    if (lc >= 0) {  // the chain: column j + 1 by one warp per sub-partition, published at once
      if (warp < 4) {
        double* ac = cols + lc * ld;
        const double f = x[nxt] * inv;
        for (int i = base + tid; i < p; i += 128)
          if (i > j) {
            const double y = fma(-f, x[i], ac[i]);
            ac[i] = y;
            if (G > 1) qd_st(ex + (long)nxt * p + i, QdBits<double>::to(y));
          }
      }
      __syncthreads();
    }
    if (mine)  // row j of U; zeros for a pivot that does not count
      for (int i = j + tid; i < p; i += kQdThreads) U[i + (long)j * p] = pre_pivot_inv(x[j], g0) != 0.0 ? x[i] : 0.0;
    const int l0 = lj + (b > jr ? 0 : 1);
    if (l0 + warp < nl) {
      const double iv = lc >= 0 ? pre_pivot_inv(x[j], g0) : inv;
      for (int l = l0 + warp; l < nl; l += 8) {
        if (l == lc) continue;
        double* ac = cols + l * ld;
        const int c = b + G * l;
        const double f = x[c] * iv;
        for (int i = (c & ~31) + lane; i < p; i += 32)
          if (i >= c) ac[i] = fma(-f, x[i], ac[i]);
      }
    }
    lj = nlj;
    jr = nr;
    __syncthreads();
  }
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
      const double g = U[hi + (long)lo * p], di = U[i + (long)i * p], dj = U[j + (long)j * p];
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
  const int z = blockIdx.y;
  const bool bad = pre_failed(a.t, z);
  if (blockIdx.x == 0 && threadIdx.x == 0) a.t.istat[z * a.t.nis + IS_FALLBACK] = bad ? 1 : 0;
  if (!bad) return;
  const int m = a.m.eval(a.t, z), p = a.p.eval(a.t, z);
  const double* L = bufp(a.t, z, a.bl);
  double* W = bufp(a.t, z, a.bw);
  for (long e = (long)blockIdx.x * blockDim.x + threadIdx.x; e < (long)m * p; e += (long)gridDim.x * blockDim.x)
    W[e] = L[e];
}

// New left carriage, row-major [m][k]: column perm[j] of W. 32 x 32 tiles through shared memory.
struct PreLeftArgs {
  Tables t;
  int bw, bw2, bperm, bout;
  Dim m;
  int ik;
};
__global__ void __launch_bounds__(256) pre_left_kernel(PreLeftArgs a) {
  const int z = blockIdx.z;
  const int m = a.m.eval(a.t, z), k = bondv(a.t, z, a.ik);
  const int r0 = blockIdx.x * 32, j0 = blockIdx.y * 32;
  if (r0 >= m || j0 >= k) return;
  __shared__ double tile[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const double* W = bufp(a.t, z, pre_where(a.t, z) ? a.bw2 : a.bw);
  const int* perm = reinterpret_cast<const int*>(bufp(a.t, z, a.bperm));
  for (int q = ty; q < 32; q += 8)
    if (j0 + q < k && r0 + tx < m) tile[q][tx] = W[(long)perm[j0 + q] * m + r0 + tx];
  __syncthreads();
  double* out = bufp(a.t, z, a.bout);
  for (int q = ty; q < 32; q += 8)
    if (r0 + q < m && j0 + tx < k) out[(long)(r0 + q) * k + j0 + tx] = tile[tx][q];
}

}  // namespace ttm
