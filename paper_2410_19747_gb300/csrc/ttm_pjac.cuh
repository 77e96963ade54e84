// ttm_pjac.cuh -- the float32 one-sided Jacobi of the preconditioned Swap SVD (ttm_pre.cuh).
#pragma once
#include "ttm_common.cuh"
#include "ttm_jres.cuh"

namespace ttm {

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

// Pairs of float32 operations in one instruction, from eight rows per lane on, where the issue slots
// of the dots and rotations show (d = 8, chi = 96, p to 768: 50.8 ms of Jacobi per product against
// 54.0); with fewer rows the packing costs what it saves.
constexpr int kPjPacked = 8;
__device__ __forceinline__ unsigned long long pj_pack(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void pj_unpack(unsigned long long v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ unsigned long long pj_fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ unsigned long long pj_mul2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// Sum over this lane's rows of a b.
template <int R>
__device__ __forceinline__ float pj_dot(const float (&a)[R], const float (&b)[R]) {
  if constexpr (R < kPjPacked) {
    constexpr int NA = R >= 4 ? 4 : R;
    float s[NA];
#pragma unroll
    for (int u = 0; u < NA; ++u) s[u] = 0.f;
#pragma unroll
    for (int q = 0; q < R; ++q) s[q % NA] = fmaf(a[q], b[q], s[q % NA]);
    float t = s[0];
#pragma unroll
    for (int u = 1; u < NA; ++u) t += s[u];
    return t;
  } else {
    constexpr int NA = 4;
    unsigned long long s[NA];
#pragma unroll
    for (int u = 0; u < NA; ++u) s[u] = 0;
#pragma unroll
    for (int q = 0; q < R / 2; ++q)
      s[q % NA] = pj_fma2(pj_pack(a[2 * q], a[2 * q + 1]), pj_pack(b[2 * q], b[2 * q + 1]), s[q % NA]);
    float t = 0.f;
#pragma unroll
    for (int u = 0; u < NA; ++u) {
      float lo, hi;
      pj_unpack(s[u], lo, hi);
      t += lo + hi;
    }
    return t;
  }
}
// (x, y) <- (c x - s y, s x + c y)
template <int R>
__device__ __forceinline__ void pj_rotate(float (&x)[R], float (&y)[R], float c, float s) {
  if constexpr (R < kPjPacked) {
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const float xp = x[q], yq = y[q];
      x[q] = c * xp - s * yq;
      y[q] = fmaf(s, xp, c * yq);
    }
  } else {
    const unsigned long long c2 = pj_pack(c, c), s2 = pj_pack(s, s), m2 = pj_pack(-s, -s);
#pragma unroll
    for (int q = 0; q < R / 2; ++q) {
      const unsigned long long xp = pj_pack(x[2 * q], x[2 * q + 1]), yp = pj_pack(y[2 * q], y[2 * q + 1]);
      pj_unpack(pj_fma2(m2, yp, pj_mul2(c2, xp)), x[2 * q], x[2 * q + 1]);
      pj_unpack(pj_fma2(s2, xp, pj_mul2(c2, yp)), y[2 * q], y[2 * q + 1]);
    }
  }
}

template <int R>
__global__ void __launch_bounds__(kPjThreads, 1) jacobi_pre_kernel(PreJacArgs a) {
  pdl_begin();
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
          auto norm2 = [&](const float (&v)[R]) { return jr_sum(pj_dot<R>(v, v)); };
          // rotates (x, na) against (y, nb2) if their coupling is above tol
          auto visit = [&](float& na, float& nb2) -> bool {
            const float g2 = jr_sum(pj_dot<R>(x, y));
            const float cpl = fabsf(g2) * rsqrtf(na) * rsqrtf(nb2);
            if (!(cpl > a.tol)) return false;  // also a padding column (0 inf = NaN)
            if (cpl > a.big) rot_any = 1;
            float c, s;
            if (!jr_rot<float>(na, nb2, g2, c, s)) return false;
            const float tg = __fdividef(s, c) * g2;
            pj_rotate<R>(x, y, c, s);
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

}  // namespace ttm
