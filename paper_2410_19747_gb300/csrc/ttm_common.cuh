// ttm_common.cuh -- shared device-side data model of the TTM engine.
//
// Every product of a batch owns a row of three tables in device memory:
//   buf  [z][nb]   : pointers to its carriage buffers and workspaces,
//   bond [z][nbd]  : the current value of every bond id (written by the kernels
//                    that create bonds: QR moves, Swap truncations),
//   stat [z][ns]   : float64 statistics (discarded weights, norms, flop counters),
//   istat[z][nis]  : int32 statistics (max bond, Jacobi sweeps, status flags).
// The host walks a static schedule and passes only ids; the kernels read the
// realised bond values, so the whole sweep needs no host synchronisation and can
// be captured in a CUDA graph. Grids are sized by host-side upper bounds and
// blocks beyond the realised sizes exit early. gridDim.z (or a loop) runs over
// the products of a batch.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "ttm.h"

namespace ttm {

struct Tables {
  double** buf;
  int* bond;
  double* stat;
  int* istat;
  int nb, nbd, ns, nis;
  int nz;  // products in this launch
  double* pre;  // [z][kPreSlots] state of the preconditioned Swap SVD (ttm_pre.cuh), or nullptr
};
// pre slots: last correction of Newton steps 1, 2, 3; 1 / ||Theta||_F^2; max |R1|; W and its norms are
// those of Theta times 2^-PR_EXP (an int in the slot's first word)
enum { PR_RES = 0, PR_ITRACE = 3, PR_ABSMAX = 4, PR_EXP = 5, kPreSlots = 8 };

__device__ __forceinline__ int bondv(const Tables& t, int z, int id) {
  return id < 0 ? 1 : t.bond[z * t.nbd + id];
}
__device__ __forceinline__ double* bufp(const Tables& t, int z, int id) {
  return t.buf[z * t.nb + id];
}

// istat slots
enum { IS_STATUS = 0, IS_MAX_BOND = 1, IS_SWEEPS_MAX = 2, IS_NONCONV = 3, IS_NFROZEN = 4, IS_NEWTON_BAD = 5,
       IS_ROUND = 6, IS_CAST_EXP = 7, IS_FALLBACK = 8, IS_NEWTON_MORE = 9, IS_NFIXED = 10 };
// stat slots (the per-truncation weights follow from ST_NFIXED)
enum { ST_WSUM = 0, ST_WSQRT = 1, ST_NEWTON_RES = 2, ST_JFLOPS32 = 3, ST_NEWTON_CUR = 4, ST_TRACE = 5,
       ST_JFLOPS = 6, ST_JSWEEPS32 = 7, ST_GFLOPS = 8, ST_NFIXED = 9 };

// Per-SVD diagnostic record (the report's svd_trace): m, n, k, float32 sweeps of passes
// 0, 1, 2, fallback flag.
constexpr int kSvdRec = 8;
enum { SR_M = 0, SR_N = 1, SR_K = 2, SR_SW0 = 3, SR_FALLBACK = 6 };

// Largest correction max(|S_ij|, |E_ij| / 2) of the last Newton step of an SVD for which it
// counts as converged: the error left after a step is of the order of its correction squared,
// so 1e-7 leaves couplings and an orthogonality defect near 1e-14.
constexpr double kNewtonConverged = 1e-7;
// The preconditioned Swap SVD takes another step while its last correction is above this: the
// steps are short there, and the result is then final to rounding also where singular values cluster.
constexpr double kPreConverged = 1e-9;

// Which of the four Newton steps of the preconditioned Swap SVD a product takes: steps 0 and 1
// always, 2 and 3 while the last correction is above kPreConverged.
__device__ __forceinline__ bool pre_active(const Tables& t, int z, int step) {
  if (step < 2) return true;
  const double* r = t.pre + z * kPreSlots + PR_RES;
  const bool s2 = !(r[0] <= kPreConverged);
  return step == 2 ? s2 : s2 && !(r[1] <= kPreConverged);
}
// 1: its W and V are in the second pair of buffers (after an odd number of steps)
__device__ __forceinline__ int pre_where(const Tables& t, int z) {
  return pre_active(t, z, 2) && !pre_active(t, z, 3) ? 1 : 0;
}
__device__ __forceinline__ bool pre_failed(const Tables& t, int z) {
  return !(t.pre[z * kPreSlots + PR_RES + 2] <= kNewtonConverged);
}

__device__ __forceinline__ int* pre_exp_slot(const Tables& t, int z) {
  return reinterpret_cast<int*>(t.pre + z * kPreSlots + PR_EXP);
}

// A dimension written as mul * bond[id] (id < 0 means the constant mul).
struct Dim {
  int mul, id;
  __device__ __forceinline__ int eval(const Tables& t, int z) const { return mul * bondv(t, z, id); }
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---------------------------------------------------------------- dependent launches
// A plain launch behind another in a stream starts 2.7 us later than a programmatic dependent one (4.1
// against 1.4 us per launch of a small kernel, 1.0 against 0.8 inside a graph), and a product is some 500
// to 8000 small launches in a row. Every kernel launched this way calls pdl_begin() before anything
// else, in all threads: it waits until all earlier work of the stream is done and visible, and
// then lets the next kernel be set up. No read-only (__ldg, __restrict__) loads in these kernels:
// their operands are still being written when their blocks are set up.
__device__ __forceinline__ void pdl_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
inline cudaLaunchAttribute pdl_attr() {
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  return at;
}
inline cudaLaunchAttribute cluster_attr(unsigned x) {
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = x;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  return at;
}
inline cudaError_t launch_pdl_c(const void* fn, dim3 grid, dim3 block, size_t smem, cudaStream_t st, void** kargs,
                                unsigned cluster = 1) {
  cudaLaunchAttribute at[2] = {pdl_attr(), cluster_attr(cluster)};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelExC(&cfg, fn, kargs);
}
template <class... P, class... A>
cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, const A&... args) {
  cudaLaunchAttribute at[1] = {pdl_attr()};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

}  // namespace ttm
