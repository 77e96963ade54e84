// ttm_qrd.cuh -- Householder QR with the columns resident in shared memory, distributed over the
// CTAs of a product, and the application of its reflectors.
//
// A (M x N) = Q R with k = min(M, N). Reflector j is kept as H = I - tau v v^T with v = x - beta e_j
// (x: column j from row j down, beta = -sign(x_j) ||x||, tau = 2 / v^T v = 1 / (||x|| (||x|| + |x_j|));
// Golub & Van Loan, Alg. 5.1.1, without the division by v_j). Serves the gauge moves (a carriage,
// float64) and the Swap SVD (Theta^T in float64; its triangular factor again in float32).
//
// What bounds it: a chain of k dependent steps, and in it the float64 pipe, on which one warp
// instruction takes 64 clocks of its sub-partition whatever its lanes do (measured; a warp sum is
// 600 clocks, a division 450, a square root 700). So the chain has one reduction per step and as few
// float64 instructions as possible:
//   - column j travels as it is; whoever receives it forms x.x and x.a for its next column in one
//     joint sum (4 warps, one per sub-partition) and derives beta, tau and v.a = x.a - beta a_j;
//   - ||x|| and 1 / (||x||^2 + |x_j| ||x||) come from a float32 seed and one step of Householder's
//     third-order iteration (Householder 1970, ch. 4; 10 instructions instead of a square root and two
//     divisions). For r near 1 / sqrt(g) and e = 1 - g r^2 it is r (1 + e / 2 + 3 e^2 / 8), for q near 1 / D
//     and f = 1 - D q it is q (1 + f + f^2): from 2^-20 to rounding. Exponents beyond 900 take CUDA's own;
//   - columns are dealt out cyclically to G CTAs and stay in shared memory; the owner of column
//     j + 1 updates and publishes it before its other columns. Receivers poll the data itself (the
//     exchange buffer is filled with a NaN pattern that arithmetic does not produce), so a step
//     costs one one-way trip through L2 (about 1000 clocks) and no flag or grid barrier.
// The other columns are updated by one warp each, four per pass when there are that many (their
// sums share a reduce-scatter of 6 instead of 4 x 5 additions). Every wait is bounded.
#pragma once
#include "ttm_common.cuh"

namespace ttm {

constexpr int kQdThreads = 256;
constexpr int kQdMaxRows = 2048;
constexpr int kQdSmem = 200 * 1024;  // columns of one CTA
constexpr int kQdPolls = 2 << 20;    // bound of a wait (a second or so)
constexpr unsigned long long kQdEmpty = ~0ull;  // exchange element not written yet

struct QrdArgs {
  Tables t;
  int bsrc;          // A: float64 buffer
  int src_rowmajor;  // 1: A row-major (ld N); 0: A column-major (ld M)
  int bv, btau;      // out (bv < 0: none): reflectors, column-major M x k (row j holds v_j), and tau[k]
  int br;            // out: R, row-major k x N (zero below the diagonal), type T
  Dim m, n;
  int ik;            // -1, or bond id that receives k
  int G;             // CTAs per product
  int cols_ub, ld_ub;           // columns held per CTA (upper bound) and their leading dimension
  unsigned long long* ex;       // exchange, ex_stride elements per product, holding kQdEmpty (G > 1)
  unsigned long long* ex_next;  // the buffer of the next launch: its first clear_n elements are emptied
  long ex_stride, clear_n;
  int scaled;        // T = double: max |R| goes to PR_ABSMAX; T = float: A is divided by the power of two
                     // above PR_ABSMAX
  float ridge;       // T = float: diagonal entries of R are moved away from zero by this much
};

template <typename T>
__device__ __forceinline__ T qd_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sums of four values over a warp: the sum of value q ends in the lanes with lane / 8 == q.
template <typename T>
__device__ __forceinline__ T qd_sum4(const T (&s)[4], int lane) {
  const bool hi = lane & 16, h2 = lane & 8;
  T a = hi ? s[2] : s[0], b = hi ? s[3] : s[1];
  a += __shfl_xor_sync(0xffffffffu, hi ? s[0] : s[2], 16);
  b += __shfl_xor_sync(0xffffffffu, hi ? s[1] : s[3], 16);
  T c = h2 ? b : a;
  c += __shfl_xor_sync(0xffffffffu, h2 ? a : b, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  return c;
}

// A float64 column whose squared norm g is below the normal range (but the column is not zero), or finite
// and at least 2^1020 (its tau would leave the range), is scaled by a power of two that brings its largest
// entry near 1 before its scalars are formed; beta, v and tau are then those of the scaled column, and only
// the diagonal entry of R is scaled back. Every other column, a zero, an infinite and a NaN one included,
// stays as it is. mag: the largest qd_mag of the column. The test is made only where qd_scalars has left its
// main branch (as a comparison of its own on the chain it cost 1 to 3 % of a product).
__device__ __forceinline__ bool qd_out_of_range(double g) {  // g >= 0 or a NaN
  return (unsigned)(__double2hiint(g) - 0x00100000) >= (unsigned)(0x7fb00000 - 0x00100000);
}
__device__ __forceinline__ unsigned qd_mag(double x) {  // orders like |x| up to a factor of 1 + 2^-20; 0 for 0 only
  return (__double2hiint(x) & 0x7fffffff) | (__double2loint(x) != 0);
}
__device__ __forceinline__ double qd_rescale(double g, unsigned mag) {
  if (mag == 0 || (__double2hiint(g) & 0x7fffffff) >= 0x7ff00000) return 1.0;
  return __hiloint2double(min(2023, 2046 - (int)(mag >> 20)) << 20, 0);
}

// beta, v_j and tau of a column with squared norm g and leading entry alpha. A column that counts as
// zero has tau = 0; a NaN travels on in beta. rescale(g, alpha): called for a g out of range; may scale the
// column and replace both.
template <class Rescale>
__device__ __forceinline__ void qd_scalars(double g, double alpha, double& beta, double& vj, double& tau, Rescale&& rescale) {
  const int hi = __double2hiint(g), lo = __double2loint(g), ex = (hi >> 20) - 1023;
  bool neg = __double2hiint(alpha) < 0;
  double aa = __hiloint2double(__double2hiint(alpha) & 0x7fffffff, __double2loint(alpha));
  double mu, D;
  if (__builtin_expect(ex > -900 && ex < 900, 1)) {  // (a negative or NaN g is outside)
    const int h = ex >> 1;
    const int gh = hi - ((2 * h) << 20);  // g 2^(-2h) in [1, 4)
    const double gs = __hiloint2double(gh, lo);
    const unsigned s = __float_as_uint(rsqrtf(__uint_as_float(((unsigned)(gh - 0x38000000) << 3) | ((unsigned)lo >> 29))));
    const double r0 = __hiloint2double((int)(s >> 3) + 0x38000000, (int)(s << 29));
    const double m0 = gs * r0;                       // sqrt to float32 accuracy, then one cubic step
    const double e = fma(-m0, r0, 1.0);
    const double ms = fma(m0 * e, fma(e, 0.375, 0.5), m0);
    mu = __hiloint2double(__double2hiint(ms) + (h << 20), __double2loint(ms));
    D = fma(aa, mu, g);                              // mu (mu + |alpha|) = v^T v / 2, in [g, 2 g (1 + u)]
    const int dh = __double2hiint(D), dl = __double2loint(D), de = (dh >> 20) - 1023;
    const int sh = dh - (de << 20);
    const unsigned t =
        __float_as_uint(__fdividef(1.f, __uint_as_float(((unsigned)(sh - 0x38000000) << 3) | ((unsigned)dl >> 29))));
    const double q0 = __hiloint2double((int)(t >> 3) + 0x38000000, (int)(t << 29));
    const double f = fma(-__hiloint2double(sh, dl), q0, 1.0);
    const double q = fma(q0 * f, 1.0 + f, q0);
    tau = __hiloint2double(__double2hiint(q) - (de << 20), __double2loint(q));
  } else {
    if (qd_out_of_range(g)) {
      rescale(g, alpha);
      neg = __double2hiint(alpha) < 0;
      aa = fabs(alpha);
    }
    if (!(g >= 2.2250738585072014e-308)) {  // (the smallest normal number) zero, or a NaN
      beta = g == g ? alpha : g;
      vj = 0.0;
      tau = 0.0;
      return;
    }
    mu = sqrt(g);
    tau = 1.0 / fma(aa, mu, g);
  }
  beta = neg ? mu : -mu;
  const double y = aa + mu;
  vj = neg ? -y : y;
}
template <class Rescale>
__device__ __forceinline__ void qd_scalars(float g, float alpha, float& beta, float& vj, float& tau, Rescale&&) {
  if (g > 1e-36f) {  // below (columns of 1e-18 of max |A|) tau would leave the float range
    float r = rsqrtf(g);
    r = fmaf(r * 0.5f, fmaf(-(g * r), r, 1.f), r);
    const float mu = g * r, y = fabsf(alpha) + mu;
    tau = __fdividef(r, y);
    beta = alpha <= 0.f ? mu : -mu;
    vj = alpha <= 0.f ? -y : y;
  } else {
    beta = g == g ? alpha : g;
    vj = 0.f;
    tau = 0.f;
  }
}

// Binary exponent of the scale that brings max |R1| to [1/2, 1); 0 for a zero or non-finite maximum.
__device__ __forceinline__ int qd_scale_exp(double mx) {
  int e = 0;
  if (mx > 0.0 && mx < 1.7e308) frexp(mx, &e);
  return max(-1000, min(1000, e));
}

template <typename T> struct QdBits;
template <> struct QdBits<double> {
  static __device__ __forceinline__ unsigned long long to(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    return b == kQdEmpty ? 0x7ff8000000000000ull : b;
  }
  static __device__ __forceinline__ double from(unsigned long long b) { return __longlong_as_double((long long)b); }
};
template <> struct QdBits<float> {
  static __device__ __forceinline__ unsigned long long to(float x) { return __float_as_uint(x); }  // high word 0
  static __device__ __forceinline__ float from(unsigned long long b) { return __uint_as_float((unsigned)b); }
};
__device__ __forceinline__ unsigned long long qd_ld(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void qd_st(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// The same for a column in the registers of one warp: its scale and its two sums after it.
struct QdScaled {
  double up, g, d;
};
__device__ __noinline__ QdScaled qd_scaled_sums(double g, double x0, double x1, double x2, double x3, double c0, double c1,
                                                double c2, double c3) {
  const double x[4] = {x0, x1, x2, x3}, c[4] = {c0, c1, c2, c3};
  unsigned mag = 0;
#pragma unroll
  for (int u = 0; u < 4; ++u) mag = max(mag, qd_mag(x[u]));
  QdScaled q{qd_rescale(g, __reduce_max_sync(0xffffffffu, mag)), 0.0, 0.0};
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const double y = x[u] * q.up;
    q.g = fma(y, y, q.g);
    q.d = fma(y, c[u], q.d);
  }
  q.g = qd_sum(q.g);
  q.d = qd_sum(q.d);
  return q;
}

// The joint sums and scalars of a step once more, for a column x that qd_rescale has scaled in place:
// g = x.x and d = x.c from row j down. All threads of the CTA; out of line, so that the step's registers do
// not pay for it.
__device__ __noinline__ void qd_scaled_step(const double* x, const double* c, int j, int M, double* red, double* sc) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (warp < 4) {
    double p0 = 0.0, p1 = 0.0;
    for (int i = (j & ~31) + tid; i < M; i += 128)
      if (i >= j) {
        p0 = fma(x[i], x[i], p0);
        if (c) p1 = fma(x[i], c[i], p1);
      }
    p0 = qd_sum(p0);
    p1 = qd_sum(p1);
    if (lane == 0) {
      red[warp] = p0;
      red[warp + 4] = p1;
    }
  }
  __syncthreads();
  if (tid == 0) {
    double beta, vj, tau;
    qd_scalars((red[0] + red[1]) + (red[2] + red[3]), x[j], beta, vj, tau, [](double&, double&) {});
    sc[0] = beta;
    sc[1] = vj;
    sc[2] = tau;
    if (c) sc[3] = tau * fma(-beta, c[j], (red[4] + red[5]) + (red[6] + red[7]));
  }
  __syncthreads();
}

template <typename T>
__global__ void __launch_bounds__(kQdThreads, 3) qrd_kernel(QrdArgs a) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char qd_raw[];
  const int G = a.G, z = blockIdx.x / G, b = blockIdx.x % G;
  const int M = a.m.eval(a.t, z), N = a.n.eval(a.t, z), k = min(M, N);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ld = a.ld_ub;
  T* cols = reinterpret_cast<T*>(qd_raw);          // [cols_ub][ld]
  T* xs = cols + (long)a.cols_ub * ld;              // [ld] the column received
  __shared__ T red[8];
  __shared__ T s_sc[4];                             // beta, v_j, tau, the chain column's factor
  __shared__ T s_up;
  __shared__ int s_flags;                           // byte 0: a wait ran out, byte 1: the column is to be scaled
  volatile unsigned char* flags = reinterpret_cast<unsigned char*>(&s_flags);
  if (b == 0 && tid == 0 && a.ik >= 0) a.t.bond[z * a.t.nbd + a.ik] = k;
  for (long e = (long)b * kQdThreads + tid; e < a.clear_n; e += (long)G * kQdThreads)
    a.ex_next[z * a.ex_stride + e] = kQdEmpty;
  const int nl = b < N ? (N - b + G - 1) / G : 0;
  if (nl == 0) return;  // nothing of this product here, and no one waits for this CTA
  if (tid == 0) s_flags = 0;
  const double* src = bufp(a.t, z, a.bsrc);
  double scale = 1.0;
  if constexpr (sizeof(T) == 4) {
    if (a.scaled) scale = ldexp(1.0, -qd_scale_exp(a.t.pre[z * kPreSlots + PR_ABSMAX]));
  }
  for (int e = tid; e < nl * M; e += kQdThreads) {
    int l, i;
    if (G == 1 && a.src_rowmajor) {  // consecutive threads along a row
      i = e / nl;
      l = e - i * nl;
    } else {
      l = e / M;
      i = e - l * M;
    }
    const int c = b + G * l;
    const double x = a.src_rowmajor ? src[(long)i * N + c] : src[(long)c * M + i];
    cols[l * ld + i] = sizeof(T) == 4 ? (T)(x * scale) : (T)x;
  }
  unsigned long long* ex = a.ex + z * a.ex_stride;
  T* R = reinterpret_cast<T*>(bufp(a.t, z, a.br));
  double* V = a.bv >= 0 ? bufp(a.t, z, a.bv) : nullptr;
  double* taug = a.bv >= 0 ? bufp(a.t, z, a.btau) : nullptr;
  __syncthreads();
  if (G > 1 && b == 0)
    for (int i = tid; i < M; i += kQdThreads) qd_st(ex + i, QdBits<T>::to(cols[i]));

  // The order in which warps take columns: warp 0 computes the scalars, so it and the warp that
  // shares its sub-partition come last.
  const int rank = warp == 0 ? 7 : warp < 4 ? warp - 1 : warp == 4 ? 6 : warp - 2;
  int lj = 0, jr = 0;  // j / G and j % G
  for (int j = 0; j < k; ++j) {
    if (b + G * (nl - 1) < j) break;  // no column from j on is held here
    const bool mine = jr == b;
    const int nxt = j + 1;
    const int nr = jr + 1 == G ? 0 : jr + 1, nlj = jr + 1 == G ? lj + 1 : lj;
    const int lc = (nr == b && nxt < N) ? nlj : -1;  // local index of column j + 1, if it is here
    const T* x = mine ? cols + lj * ld : xs;
    const int base = j & ~31;
    T* crit = lc >= 0 ? cols + lc * ld : nullptr;
    const unsigned long long* src_x = ex + (long)j * M;
    unsigned long long* dst_x = ex + (long)nxt * M;
    // the other columns right of j: local index from l0 on; up to eight are one per warp, whose dot
    // product with x is formed while warp 0 is at the scalars
    const int l0 = lc >= 0 ? lc + 1 : lj + (b > jr ? 0 : 1);
    const int rest = nl - l0;
    const bool one = rest <= 8, have = one && rank < rest;
    T* am = have ? cols + (l0 + rank) * ld : nullptr;
    T dme = T(0);
    const bool narrow = M - base <= 128;  // warp 0 takes the chain alone, x in the registers of every warp
    T xr[4] = {T(0), T(0), T(0), T(0)};
    if (narrow) {
      if (mine) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = base + lane + 32 * u;
          if (i >= j && i < M) xr[u] = x[i];
        }
      } else if (warp == 0 || have) {
        unsigned long long bits[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = base + lane + 32 * u;
          bits[u] = (i >= j && i < M) ? qd_ld(src_x + i) : 0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = base + lane + 32 * u;
          for (int polls = 0; bits[u] == kQdEmpty && polls < kQdPolls; ++polls) bits[u] = qd_ld(src_x + i);
          if (bits[u] == kQdEmpty) flags[0] = 1;
          xr[u] = QdBits<T>::from(bits[u]);
          if (!one && i < M) xs[i] = xr[u];  // (warp 0)
        }
      }
      if (warp == 0) {
        T p0 = T(0), p1 = T(0), cr[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = base + lane + 32 * u;
          cr[u] = (crit && i < M) ? crit[i] : T(0);
          if (base + 32 * u < M) {
            p0 = fma(xr[u], xr[u], p0);
            if (crit) p1 = fma(xr[u], cr[u], p1);
          }
        }
        const bool hi = lane & 16;
        T s = hi ? p1 : p0;
        s += __shfl_xor_sync(0xffffffffu, hi ? p0 : p1, 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const T g = __shfl_sync(0xffffffffu, s, 0);
        T d = __shfl_sync(0xffffffffu, s, 16);
        T beta, vj, tau;
        qd_scalars(g, __shfl_sync(0xffffffffu, xr[0], j & 31), beta, vj, tau, [&](auto& gr, auto& alpha) {
          const QdScaled q = qd_scaled_sums(gr, xr[0], xr[1], xr[2], xr[3], cr[0], cr[1], cr[2], cr[3]);
          if (q.up == 1.0) return;
          if (lane == 0) {
            s_up = q.up;
            flags[1] = 1;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) xr[u] *= q.up;
          gr = q.g;
          d = q.d;
          alpha *= q.up;
        });
        if (crit) {
          const T cj = __shfl_sync(0xffffffffu, cr[0], j & 31);
          const T f = tau * fma(-beta, cj, d);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = base + lane + 32 * u;
            if (base + 32 * u < M) {
              const T y = fma(-f, xr[u], cr[u]);
              if (i > j && i < M) {
                if (G > 1 && nxt < k) qd_st(dst_x + i, QdBits<T>::to(y));
                crit[i] = y;
              }
            }
          }
          if (lane == 0) R[(long)j * N + nxt] = fma(-f, vj, cj);
        }
        if (lane == 0) {
          s_sc[0] = beta;
          s_sc[1] = vj;
          s_sc[2] = tau;
        }
      } else if (have) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (base + 32 * u < M) {
            const int i = base + lane + 32 * u;
            if (i < M) dme = fma(xr[u], am[i], dme);
          }
        dme = qd_sum(dme);
      }
    } else {
      if (warp < 4) {
        T p0 = T(0), p1 = T(0);
        if (mine) {
          for (int i = base + tid; i < M; i += 128) {
            const T xi = i >= j ? x[i] : T(0);
            p0 = fma(xi, xi, p0);
            if (crit) p1 = fma(xi, crit[i], p1);
          }
        } else {
          // all of this thread's rows are requested before any is waited for
          constexpr int NB = 8;
          for (int i0 = base + tid; i0 < M; i0 += 128 * NB) {
            unsigned long long bits[NB];
#pragma unroll
            for (int u = 0; u < NB; ++u) {
              const int i = i0 + 128 * u;
              bits[u] = (i >= j && i < M) ? qd_ld(src_x + i) : 0;
            }
#pragma unroll
            for (int u = 0; u < NB; ++u) {
              const int i = i0 + 128 * u;
              if (i >= M) break;
              for (int polls = 0; bits[u] == kQdEmpty && polls < kQdPolls; ++polls) bits[u] = qd_ld(src_x + i);
              if (bits[u] == kQdEmpty) flags[0] = 1;
              const T xi = QdBits<T>::from(bits[u]);
              xs[i] = xi;
              p0 = fma(xi, xi, p0);
              if (crit) p1 = fma(xi, crit[i], p1);
            }
          }
        }
        const bool hi = lane & 16;
        T s = hi ? p1 : p0;
        s += __shfl_xor_sync(0xffffffffu, hi ? p0 : p1, 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((lane & 15) == 0) red[warp + (hi ? 4 : 0)] = s;
      }
      __syncthreads();
      if (warp == 0) {
        T s = red[lane & 7];
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        const T g = __shfl_sync(0xffffffffu, s, 0), d = __shfl_sync(0xffffffffu, s, 4);
        T beta, vj, tau;
        qd_scalars(g, x[j], beta, vj, tau, [&](auto& gr, auto&) {  // the step is done again after the barrier
          unsigned mag = 0;
          for (int i = base + lane; i < M; i += 32)
            if (i >= j) mag = max(mag, qd_mag(x[i]));
          const double up = qd_rescale(gr, __reduce_max_sync(0xffffffffu, mag));
          if (up != 1.0 && lane == 0) {
            s_up = up;
            flags[1] = 1;
          }
        });
        const T cj = crit ? crit[j] : T(0);
        const T f = tau * fma(-beta, cj, d);
        if (lane == 0) {
          s_sc[0] = beta;
          s_sc[1] = vj;
          s_sc[2] = tau;
          s_sc[3] = f;
          if (crit) R[(long)j * N + nxt] = fma(-f, vj, cj);
        }
      } else if (have) {
        for (int i = base + lane; i < M; i += 32) dme = fma(i >= j ? x[i] : T(0), am[i], dme);
        dme = qd_sum(dme);
      }
    }
    __syncthreads();
    bool scaled = false;
    if (__builtin_expect(s_flags != 0, 0)) {  // every thread sees it: it was set before the barrier
      if (flags[0]) {
        if (tid == 0) atomicExch(&a.t.istat[z * a.t.nis + IS_STATUS], (int)TTM_ERR_TIMEOUT);
        return;
      }
      if constexpr (sizeof(T) == 8) {
        const double up = s_up;
        scaled = true;
        T* xw = mine ? cols + lj * ld : xs;
        if (mine || !narrow || !one)
          for (int i = j + tid; i < M; i += kQdThreads) xw[i] *= up;
        __syncthreads();
        if (tid == 0) s_flags = 0;
        if (!narrow) {
          qd_scaled_step(x, crit, j, M, red, s_sc);
          if (tid == 0 && crit) R[(long)j * N + nxt] = fma(-s_sc[3], s_sc[1], crit[j]);
        }
        if (have && warp != 0) {
          dme = T(0);
          if (narrow) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int i = base + lane + 32 * u;
              xr[u] *= up;
              if (i < M) dme = fma(xr[u], am[i], dme);
            }
          } else {
            for (int i = base + lane; i < M; i += 32) dme = fma(i >= j ? x[i] : T(0), am[i], dme);
          }
          dme = qd_sum(dme);
        }
      }
    }
    if (!narrow && crit && warp < 4) {
      const T f = s_sc[3];
      for (int i = base + tid; i < M; i += 128)
        if (i > j) {
          const T y = fma(-f, x[i], crit[i]);
          if (G > 1 && nxt < k) qd_st(dst_x + i, QdBits<T>::to(y));
          crit[i] = y;
        }
    }
    if (mine && tid == 0) {
      T rd = s_sc[0];
      if (scaled) rd *= __hiloint2double(0x7fe00000 - __double2hiint(s_up), 0);  // 1 / s_up, a power of two
      if constexpr (sizeof(T) == 4) rd += rd < T(0) ? -a.ridge : a.ridge;
      R[(long)j * N + j] = rd;
      if (V) {
        V[(long)j * M + j] = (double)s_sc[1];
        taug[j] = (double)s_sc[2];
      }
    }
    if (have) {
      const T beta = s_sc[0], vj = s_sc[1], tau = s_sc[2];
      if (warp == 0) {  // (its dot product had to wait)
        if (narrow) {
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = base + lane + 32 * u;
            if (i < M) dme = fma(xr[u], am[i], dme);
          }
        } else {
          for (int i = base + lane; i < M; i += 32) dme = fma(i >= j ? x[i] : T(0), am[i], dme);
        }
        dme = qd_sum(dme);
      }
      const T cj = am[j];
      const T f = tau * fma(-beta, cj, dme);
      if (lane == 0) R[(long)j * N + b + (long)G * (l0 + rank)] = fma(-f, vj, cj);
      if (narrow) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = base + lane + 32 * u;
          if (base + 32 * u < M && i > j && i < M) am[i] = fma(-f, xr[u], am[i]);
        }
      } else {
        for (int i = base + lane; i < M; i += 32)
          if (i > j) am[i] = fma(-f, x[i], am[i]);
      }
    } else if (!one) {
      const T beta = s_sc[0], vj = s_sc[1], tau = s_sc[2];
      for (int q0 = 0; q0 < rest; q0 += 32) {
        // up to four columns of this warp: l0 + q0 + warp + 8 q
        const int cnt = min(32, rest - q0);
        const int lw = l0 + q0 + warp;
        T s[4] = {T(0), T(0), T(0), T(0)};
        T* ac[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) ac[q] = cols + min(lw + 8 * q, nl - 1) * ld;
        for (int i = base + lane; i < M; i += 32) {
          const T xi = i >= j ? x[i] : T(0);
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (warp + 8 * q < cnt) s[q] = fma(xi, ac[q][i], s[q]);
        }
        const int mq = lane >> 3;
        const T dsum = qd_sum4(s, lane);
        const T cj = cols[min(lw + 8 * mq, nl - 1) * ld + j];
        const T f = tau * fma(-beta, cj, dsum);
        T fq[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) fq[q] = __shfl_sync(0xffffffffu, f, 8 * q);
        if ((lane & 7) == 0 && warp + 8 * mq < cnt)
          R[(long)j * N + b + (long)G * (lw + 8 * mq)] = fma(-f, vj, cj);
        for (int i = base + lane; i < M; i += 32) {
          const T xi = x[i];
          if (i > j) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (warp + 8 * q < cnt) ac[q][i] = fma(-fq[q], xi, ac[q][i]);
          }
        }
      }
    }
    lj = nlj;
    jr = nr;
    __syncthreads();
  }
  // zeros of R below the diagonal, the reflectors, and the largest magnitude of R
  double mx = 0.0;
  for (int e = tid; e < nl * k; e += kQdThreads) {
    const int l = e / k, i = e - l * k, c = b + G * l;
    if (i > c) R[(long)i * N + c] = T(0);
    else if (sizeof(T) == 8 && a.scaled) mx = fmax(mx, fabs((double)R[(long)i * N + c]));
  }
  if constexpr (sizeof(T) == 8) {
    if (V)
      for (int e = tid; e < nl * M; e += kQdThreads) {
        const int l = e / M, i = e - l * M, c = b + G * l;
        if (c < k && i > c) V[(long)c * M + i] = cols[l * ld + i];
      }
    if (a.scaled) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      if (lane == 0 && mx > 0.0)
        atomicMax(reinterpret_cast<unsigned long long*>(a.t.pre + z * kPreSlots + PR_ABSMAX),
                  (unsigned long long)__double_as_longlong(mx));
    }
  }
}

// Y = H_0 H_1 .. H_{k-1} Y0 in float64: one column per warp in shared memory, four columns per CTA;
// the reflectors arrive through a ring of shared buffers filled by cp.async three steps ahead. Y0 is
// the first columns of the identity (bvec < 0) or the columns perm[c] of a k x k column-major matrix,
// padded with zeros. What bounds it: the float64 pipe (per step 2 M / 32 + 7 warp instructions of 64
// clocks; the columns are independent, so the launch fills the chip with them).
constexpr int kQaThreads = 128;
constexpr int kQaStages = 4;
struct QrdApplyArgs {
  Tables t;
  int bv, btau;   // reflectors and tau of qrd_kernel<double>
  Dim m, n;       // A was m x n
  int bvec, bvec2, bperm;  // bvec2: the matrix when pre_where() is 1
  int ic;         // bond id: columns of Y
  int bout;
  int out_rows;   // 1: Y row-major (m x columns); 0: Y^T row-major (columns x m)
  int ld_ub;
};

// WPC: warps per column (1: four columns per CTA; 4: one, for launches with fewer columns than the
// chip has sub-partitions). On 256 rows a step takes about 1400 clocks with one warp, 900 with four.
template <int WPC>
__global__ void __launch_bounds__(kQaThreads) qrd_apply_kernel(QrdApplyArgs a) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char qd_raw[];
  constexpr int CPB = 4 / WPC;  // columns per CTA
  __shared__ double red[2][4];
  const int z = blockIdx.y;
  const int M = a.m.eval(a.t, z), N = a.n.eval(a.t, z), k = min(M, N), nc = bondv(a.t, z, a.ic);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c0 = blockIdx.x * CPB, c = WPC == 1 ? c0 + warp : c0;
  const int r0 = WPC == 1 ? lane : threadIdx.x;  // this thread's first row above the step's base
  constexpr int RS = 32 * WPC;                   // and its row stride
  if (c0 >= nc) return;
  const int ld = a.ld_ub;
  double* vs = reinterpret_cast<double*>(qd_raw);                              // [kQaStages][ld]
  double* y = vs + (kQaStages + (WPC == 1 ? warp : 0)) * (long)ld;              // this warp's column
  const double* V = bufp(a.t, z, a.bv);
  const double* tau = bufp(a.t, z, a.btau);
  const bool on = c < nc;
  int j0;
  if (a.bvec < 0) {
    j0 = min(min(c0 + CPB - 1, nc - 1), k - 1);
    for (int i = r0; i < M; i += RS) y[i] = i == c ? 1.0 : 0.0;
  } else {
    j0 = k - 1;
    const int pc = on ? reinterpret_cast<const int*>(bufp(a.t, z, a.bperm))[c] : 0;
    const double* x = bufp(a.t, z, pre_where(a.t, z) ? a.bvec2 : a.bvec) + (long)max(0, min(pc, k - 1)) * k;
    for (int i = r0; i < M; i += RS) y[i] = i < k ? x[i] : 0.0;
  }
  auto fetch = [&](int q) {  // reflector q into its stage; one commit group per call
    if (q >= 0) {
      double* dst = vs + (q & (kQaStages - 1)) * (long)ld;
      const double* src = V + (long)q * M;
      for (int i = (q & ~31) + threadIdx.x; i < M; i += kQaThreads)
        if (i >= q)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst + i)),
                       "l"(src + i)
                       : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int s = 0; s < kQaStages - 1; ++s) fetch(j0 - s);
  for (int j = j0; j >= 0; --j) {
    const double tj = tau[j];
    asm volatile("cp.async.wait_group %0;" ::"n"(kQaStages - 2) : "memory");
    __syncthreads();  // reflector j is here, and its ring slot of step j + 1 is free again
    fetch(j - (kQaStages - 1));
    const double* v = vs + (j & (kQaStages - 1)) * (long)ld;
    double s = 0.0;
    for (int i = (j & ~31) + r0; i < M; i += RS)
      if (i >= j) s = fma(v[i], y[i], s);
    s = qd_sum(s);
    if constexpr (WPC == 4) {
      if (lane == 0) red[j & 1][warp] = s;
      __syncthreads();
      s = (red[j & 1][0] + red[j & 1][1]) + (red[j & 1][2] + red[j & 1][3]);
    }
    const double f = tj * s;
    for (int i = (j & ~31) + r0; i < M; i += RS)
      if (i >= j) y[i] = fma(-f, v[i], y[i]);
    if constexpr (WPC == 1) __syncwarp();
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  if constexpr (WPC == 4) __syncthreads();
  if (!on) return;
  double* out = bufp(a.t, z, a.bout);
  if (a.out_rows)
    for (int i = r0; i < M; i += RS) out[(long)i * nc + c] = y[i];
  else
    for (int i = r0; i < M; i += RS) out[(long)c * M + i] = y[i];
}

}  // namespace ttm
