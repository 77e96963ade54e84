// ttm_gemm.cuh -- float64 GEMM for the contractions of the sweep.
//
// C = alpha * A * B + beta * C for every (product z, batch index b) of a launch.
// Each operand is a strided view (element (i, j) at p[i*rs + j*cs]), so the leg
// permutations of the Swap (Fig. 1C) and the "same physical index" selection of
// the Contract (Eq. contract) are expressed purely by strides: no permuted copy
// is ever materialised. A functor F maps (z, b) to the problem, reading the bond
// table, so sizes are the realised ones.
//
// Bound: the float64 pipe (2 DFMA per clock and SM, about 1.1 TFLOP/s for the whole GPU), not
// memory; one 64 x 64 x 256 tile is 0.26 ms of one SM's pipe, so what decides the time of the
// sweep's GEMMs (16 .. 1024 on a side) is over how many SMs the work is spread. Tiles of 16 x 16
// or 32 x 32 outputs, K panels of 32 prefetched into registers, 256 threads in four groups that
// split the panel's K (so one CTA alone fills the four sub-partitions), and, where the tiles are
// fewer than the SMs can hold, up to 8 CTAs of a cluster that split K and add their partial tiles
// through distributed shared memory in a fixed order. Measured against 64 x 64 tiles without a
// split (GB300): the GEMMs of a 256 x 256 Swap 133 -> 19 us each, the overlap of two L = 30 trains
// of bonds 512 and 300 22.6 -> 6.2 ms (1.07 TFLOP/s), a gradient at L = 20, d = 4, chi = 64
// 172 -> 33 ms; 2048 x 2048 x 1024 runs at 1.23 TFLOP/s.
#pragma once
#include <cooperative_groups.h>
#include "ttm_common.cuh"

namespace cg = cooperative_groups;

namespace ttm {

struct MatRef {
  const double* p;
  long rs, cs;
};
struct OutRef {
  double* p;
  long rs, cs;
};
struct GemmDesc {
  int M, N, K;
  MatRef A, B;
  OutRef C;
  double alpha, beta;
  int upper;  // 1: only the output tiles that meet the upper triangle (symmetric results)
};

constexpr int kDgK = 32;        // K panel
constexpr int kDgThreads = 256;
constexpr int kDgMaxSplit = 8;  // CTAs of a cluster that split K

// Realised flops of one problem (2 M N K; M (M + 1) K for a symmetric Gram whose upper
// triangle is formed), added by one thread of the problem's first tile when fl is set: a
// predicated-off problem (M = 0) adds nothing.
__device__ __forceinline__ void gemm_count_flops(double* fl, int fl_stride, int z, const GemmDesc& g) {
  if (fl == nullptr) return;
  const double f = g.upper ? (double)g.M * (g.N + 1) * g.K : 2.0 * g.M * g.N * g.K;
  atomicAdd(fl + (long)z * fl_stride, f);
}

// Realised shape of a launch's GEMMs (per product and batch index), for the flop count.
struct GemmShape {
  Dim M, N, K;
  int nbatch;
  int sym;  // 1: symmetric result, only the upper triangle is counted
};

// Grid: x = (M tile * n_tiles + N tile) * split + K part (the parts of a tile are one cluster),
// z = problems.
template <class F, int DT>
__global__ void __launch_bounds__(kDgThreads) dgemm_kernel(F f, int nbatch, int n_tiles, int split, double* fl,
                                                           int fl_stride) {
  pdl_begin();
  const int z = blockIdx.z / nbatch, bi = blockIdx.z % nbatch;
  const GemmDesc g = f(z, bi);
  const int rank = blockIdx.x % split, tile = blockIdx.x / split;
  const int m0 = tile / n_tiles * DT, n0 = tile % n_tiles * DT;
  if (g.M <= 0 || g.N <= 0 || m0 >= g.M || n0 >= g.N) return;  // uniform over the cluster
  if (m0 == 0 && n0 == 0 && rank == 0 && threadIdx.x == 0) gemm_count_flops(fl, fl_stride, z, g);
  if (g.upper && m0 > n0) return;
  constexpr int MI = DT / 8;                 // rows and columns per thread
  constexpr int LD = DT + 1;
  constexpr int PER = DT * kDgK / kDgThreads;  // panel elements per thread and operand
  constexpr int OUT = DT * DT / kDgThreads;    // outputs per thread in the final sum
  constexpr int kPanels = 2 * kDgK * LD, kPart = 4 * DT * DT;
  __shared__ double sm[kPanels > kPart ? kPanels : kPart];
  double* As = sm;                // [kDgK][LD]
  double* Bs = sm + kDgK * LD;    // [kDgK][LD]
  const int tid = threadIdx.x;
  const int grp = tid >> 6, tx = tid & 7, ty = (tid >> 3) & 7;
  // consecutive threads follow the unit stride of the operand when it has one
  const bool a_kfast = (g.A.cs == 1), b_kfast = (g.B.cs != 1);
  int per = (g.K + split - 1) / split;
  per = (per + kDgK - 1) / kDgK * kDgK;
  const int kbeg = rank * per, kend = min(g.K, kbeg + per);
  double ra[PER], rb[PER];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int e = tid + u * kDgThreads;
      const int mm = a_kfast ? e / kDgK : e % DT, ka = k0 + (a_kfast ? e % kDgK : e / DT);
      const int nn = b_kfast ? e / kDgK : e % DT, kb = k0 + (b_kfast ? e % kDgK : e / DT);
      ra[u] = (m0 + mm < g.M && ka < kend) ? g.A.p[(long)(m0 + mm) * g.A.rs + (long)ka * g.A.cs] : 0.0;
      rb[u] = (n0 + nn < g.N && kb < kend) ? g.B.p[(long)kb * g.B.rs + (long)(n0 + nn) * g.B.cs] : 0.0;
    }
  };
  double acc[MI][MI];
#pragma unroll
  for (int i = 0; i < MI; ++i)
#pragma unroll
    for (int j = 0; j < MI; ++j) acc[i][j] = 0.0;
  if (kbeg < kend) fetch(kbeg);
  for (int k0 = kbeg; k0 < kend; k0 += kDgK) {
    __syncthreads();
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int e = tid + u * kDgThreads;
      As[(a_kfast ? e % kDgK : e / DT) * LD + (a_kfast ? e / kDgK : e % DT)] = ra[u];
      Bs[(b_kfast ? e % kDgK : e / DT) * LD + (b_kfast ? e / kDgK : e % DT)] = rb[u];
    }
    __syncthreads();
    if (k0 + kDgK < kend) fetch(k0 + kDgK);
#pragma unroll
    for (int q = 0; q < kDgK / 4; ++q) {
      const int kk = q * 4 + grp;
      double a[MI], b[MI];
#pragma unroll
      for (int i = 0; i < MI; ++i) a[i] = As[kk * LD + ty + 8 * i];
#pragma unroll
      for (int j = 0; j < MI; ++j) b[j] = Bs[kk * LD + tx + 8 * j];
#pragma unroll
      for (int i = 0; i < MI; ++i)
#pragma unroll
        for (int j = 0; j < MI; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
  }
  __syncthreads();
  double* part = sm;  // [4][DT][DT]
#pragma unroll
  for (int i = 0; i < MI; ++i)
#pragma unroll
    for (int j = 0; j < MI; ++j) part[grp * DT * DT + (ty + 8 * i) * DT + tx + 8 * j] = acc[i][j];
  __syncthreads();
  const bool c_rfast = (g.C.rs == 1);
  auto put = [&](int e, double v) {  // e = row * DT + column
    const int gm = m0 + e / DT, gn = n0 + e % DT;
    if (gm >= g.M || gn >= g.N) return;
    double* c = g.C.p + (long)gm * g.C.rs + (long)gn * g.C.cs;
    v *= g.alpha;
    if (g.beta != 0.0) v = fma(g.beta, *c, v);
    *c = v;
  };
  auto slot = [&](int o) { return c_rfast ? (o % DT) * DT + o / DT : o; };  // writes along C's unit stride
  if (split == 1) {
#pragma unroll
    for (int u = 0; u < OUT; ++u) {
      const int e = slot(tid + u * kDgThreads);
      put(e, (part[e] + part[DT * DT + e]) + (part[2 * DT * DT + e] + part[3 * DT * DT + e]));
    }
    return;
  }
#pragma unroll
  for (int u = 0; u < OUT; ++u) {
    const int e = tid + u * kDgThreads;
    part[e] = (part[e] + part[DT * DT + e]) + (part[2 * DT * DT + e] + part[3 * DT * DT + e]);
  }
  cg::cluster_group cl = cg::this_cluster();
  cl.sync();
  for (int o = rank * kDgThreads + tid; o < DT * DT; o += split * kDgThreads) {
    const int e = slot(o);
    double v = 0.0;
    for (int q = 0; q < split; ++q) v += cl.map_shared_rank(part, q)[e];
    put(e, v);
  }
  cl.sync();  // the partial tile is read by the other CTAs of the cluster until here
}

// Launches the float64 product of nprob = (products x batch) problems with these upper bounds.
template <class F>
cudaError_t launch_dgemm(cudaStream_t st, const F& f, int nprob, int nbatch, int M_ub, int N_ub, int K_ub, int num_sms,
                         double* fl = nullptr, int fl_stride = 0) {
  auto cdiv = [](long a, long b) { return (a + b - 1) / b; };
  const long t32 = cdiv(M_ub, 32) * cdiv(N_ub, 32) * nprob;
  const bool big = t32 >= 8L * num_sms;
  const long DT = big ? 32 : 16;
  const long tiles = cdiv(M_ub, DT) * cdiv(N_ub, DT);
  const int n_tiles = (int)cdiv(N_ub, DT);
  int split = 1;
  while (split < kDgMaxSplit && tiles * nprob * split * 2 <= 4L * num_sms && K_ub >= 2 * kDgK * split * 2) split *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(tiles * split), 1, (unsigned)nprob);
  cfg.blockDim = dim3(kDgThreads);
  cfg.stream = st;
  cudaLaunchAttribute at[2] = {pdl_attr(), cluster_attr((unsigned)split)};
  cfg.attrs = at;
  cfg.numAttrs = split > 1 ? 2 : 1;
  if (big) return cudaLaunchKernelEx(&cfg, dgemm_kernel<F, 32>, f, nbatch, n_tiles, split, fl, fl_stride);
  return cudaLaunchKernelEx(&cfg, dgemm_kernel<F, 16>, f, nbatch, n_tiles, split, fl, fl_stride);
}

// ---------------------------------------------------------------------------
// Problem functors. All cores are row-major [Dl][d][Dr].

// Swap, two-site contraction with the physical legs permuted (Fig. 1C):
//   Theta[(l,t),(s,r)] = sum_m X[l,s,m] Y[m,t,r],
// stored column-major with m_rows = Dl*d rows (row = l*d + t, col = s*Dr + r),
// which is the layout the one-sided Jacobi SVD works on. Batch b = s*d + t.
// keep_legs = 1 forms the plain two-site tensor Theta[(l,s),(t,r)] instead (the SVD
// sweep of the final rounding, where the legs stay in place).
struct ThetaFn {
  Tables t;
  int bx, by, bth;  // buffers: X, Y, Theta workspace
  int il, im, ir;   // bond ids: left of X, shared, right of Y
  int d;
  int keep_legs;    // 0: permuted legs (Swap); 1: legs in place
  __device__ GemmDesc operator()(int z, int b) const {
    const int s = b / d, tt = b % d;
    const int Dl = bondv(t, z, il), Dm = bondv(t, z, im), Dr = bondv(t, z, ir);
    const double* X = bufp(t, z, bx);
    const double* Y = bufp(t, z, by);
    double* T = bufp(t, z, bth);
    const long mrows = (long)Dl * d;
    const int row_leg = keep_legs ? s : tt, col_leg = keep_legs ? tt : s;
    GemmDesc g;
    g.M = Dl; g.N = Dr; g.K = Dm;
    g.A = MatRef{X + (long)s * Dm, (long)d * Dm, 1};
    g.B = MatRef{Y + (long)tt * Dr, (long)d * Dr, 1};
    g.C = OutRef{T + row_leg + (long)col_leg * Dr * mrows, d, mrows};
    g.alpha = 1.0; g.beta = 0.0; g.upper = 0;
    return g;
  }
};

// Contract (Eq. contract): Pi[l, e, r] = sum_a K[l, e, a] M[a, e, r]; batch b = e.
// The COPY tensor makes sigma = omega = eta, so only the d diagonal products are formed.
struct ContractFn {
  Tables t;
  int bk, bm, bo;
  int il, ia, ir;
  int d;
  __device__ GemmDesc operator()(int z, int e) const {
    const int Dl = bondv(t, z, il), Da = bondv(t, z, ia), Dr = bondv(t, z, ir);
    GemmDesc g;
    g.M = Dl; g.N = Dr; g.K = Da;
    g.A = MatRef{bufp(t, z, bk) + (long)e * Da, (long)d * Da, 1};
    g.B = MatRef{bufp(t, z, bm) + (long)e * Dr, (long)d * Dr, 1};
    g.C = OutRef{bufp(t, z, bo) + (long)e * Dr, (long)d * Dr, 1};
    g.alpha = 1.0; g.beta = 0.0; g.upper = 0;
    return g;
  }
};

// Gauge move, second half: Next'[k, (s, r)] = sum_c R[k, c] Next[c, (s, r)].
// R is row-major k x n (n = bond between the two carriages before the move).
struct RMergeFn {
  Tables t;
  int br, bn, bo;
  int ik, in, irr;
  int d;
  __device__ GemmDesc operator()(int z, int) const {
    const int k = bondv(t, z, ik), n = bondv(t, z, in), Drr = bondv(t, z, irr);
    GemmDesc g;
    g.M = k; g.N = d * Drr; g.K = n;
    g.A = MatRef{bufp(t, z, br), n, 1};
    g.B = MatRef{bufp(t, z, bn), (long)d * Drr, 1};
    g.C = OutRef{bufp(t, z, bo), (long)d * Drr, 1};
    g.alpha = 1.0; g.beta = 0.0; g.upper = 0;
    return g;
  }
};

// W = Theta V0 with both column-major (Theta m x n, V0 n x n, W m x n).
struct ThetaVFn {
  Tables t;
  int bth, bv, bw;
  Dim m, n;
  __device__ GemmDesc operator()(int z, int) const {
    const int M = m.eval(t, z), N = n.eval(t, z);
    GemmDesc g;
    g.M = M; g.N = N; g.K = N;
    g.A = MatRef{bufp(t, z, bth), 1, M};
    g.B = MatRef{bufp(t, z, bv), 1, N};
    g.C = OutRef{bufp(t, z, bw), 1, M};
    g.alpha = 1.0; g.beta = 0.0; g.upper = 0;
    return g;
  }
};

// Gram matrix G = W^T W of a column-major m x n matrix (n x n column-major; the tiles of
// the upper triangle only: G is symmetric and its readers take G[min(i,j) + max(i,j) n]).
struct GramFn {
  Tables t;
  int bw, bg;
  Dim m, n;
  __device__ GemmDesc operator()(int z, int) const {
    const int M = m.eval(t, z), N = n.eval(t, z);
    const double* W = bufp(t, z, bw);
    GemmDesc g;
    g.M = N; g.N = N; g.K = M;
    g.A = MatRef{W, M, 1};
    g.B = MatRef{W, 1, M};
    g.C = OutRef{bufp(t, z, bg), 1, N};
    g.alpha = 1.0; g.beta = 0.0; g.upper = 1;
    return g;
  }
};

// Right-to-left rounding: Prev'[(l, s), j] = sum_c Prev[(l, s), c] Wk[c, j],
// Wk column-major (rows = c, ld = wrows), j < k.
struct LMergeFn {
  Tables t;
  int bp, bw, bo;
  int il, ic, ik;
  Dim wrows;
  int d;
  __device__ GemmDesc operator()(int z, int) const {
    const int Dl = bondv(t, z, il), c = bondv(t, z, ic), k = bondv(t, z, ik);
    const long ld = wrows.eval(t, z);
    GemmDesc g;
    g.M = Dl * d; g.N = k; g.K = c;
    g.A = MatRef{bufp(t, z, bp), c, 1};
    g.B = MatRef{bufp(t, z, bw), 1, ld};
    g.C = OutRef{bufp(t, z, bo), k, 1};
    g.alpha = 1.0; g.beta = 0.0; g.upper = 0;
    return g;
  }
};

}  // namespace ttm
