// Rayleigh-Ritz eigensolve of a symmetric s x s matrix (s <= 96): FP32 Jacobi, then FP64 refinement of
// all eigenvectors at once (Ogita and Aishima, "Iterative refinement for symmetric eigenvalue
// decomposition", 2018), by one cluster of eight CTAs.
//
// What bounds it.  Plain FP64 Jacobi in one CTA (small.cu) spends 16k FP64 operations in each of its
// 62 rounds a sweep at s = 63, 8k clocks of one SM's FP64 pipe, and a serial chain of FP64 divisions
// and square roots before them, over 8 or 9 sweeps.  FP32 rounds have no such pipe to wait for, and one
// refinement step is four s x s x s products (1 M multiply-adds at s = 63) that eight SMs share; it
// squares the error, so two or three steps take FP32's 1e-6 to FP64's rounding.  Microseconds per call,
// one-CTA Jacobi (plain) and this: s = 3 122, 93   8 186, 98   12 239, 107   24 520, 148   63 3,680, 468.  The FP32
// rounds, latency-bound, are about two thirds of it (counters at s = 63: FP64 pipe 17%, integer 21%, the
// warps wait at barriers).
//
// The solver's FP64 phases keep plain Jacobi.  With this kernel in them the mixed + diagonal form on one
// matrix (n = 10^5) needs more than 4,000 iterations from each of five starts 1e-14 apart, where Jacobi
// takes 885 to 3,929; on another both take the same.  Eigenvalues and vectors agree in every iteration
// compared to Jacobi's own rounding (1e-14, entries above 1e-14 to 5e-12 of themselves), so what slows
// that solve is not known.  Random starts of n = 2,000 fail with either kernel (9 of 24 with Jacobi, 3 of
// 24 with this one).
//
// Layout.  Every CTA holds all of A and X in shared memory.  In the FP32 stage every CTA rotates its own
// copy of the matrix (the same operations, so the same rotations) but only its own rows of the
// eigenvector matrix, so the stage needs no exchange.  In the refinement CTA c forms the columns
// J_c = [c nb, (c + 1) nb) of every product and writes its new columns of X into all eight copies.
//
// One step, with R = I - X^T X and S = X^T A X: lambda_j = S_jj / (1 - R_jj) and X <- X + X (R / 2 + K) with
// K antisymmetric, K_ij = N_ij / (lambda_j - lambda_i), N = (S + S^T) / 2 + R (lambda_i + lambda_j) / 2.  The
// halves of S come together through U, so K is antisymmetric to the last bit and rounding of S over a
// small gap only turns vectors, it never takes them off orthonormality (S_ij alone did, by 4e-9 at a
// gap of 1e-7), but for the second order K^T K: steps that no longer converge, over gaps of 1e-10 ||A||,
// are followed by steps of R / 2 alone.  Where N_ij is rounding noise of ||A|| and the gap within 1e-10 ||A|| (repeated
// eigenvalues) K_ij = 0; over any wider gap a coupling counts whatever its size.  Where it is not small
// against the gap (close eigenvalues that FP32 did not separate) the Jacobi angle of the pair, halved,
// takes the quotient's place: the pair turns by a bounded angle, and the quotient applies once it is
// small.  Without convergence in kMaxSteps, or with a non-finite entry, lambda_0 is set to NaN, on which
// the plain Jacobi kernel launched behind this one runs (else it returns at once).
#include <cooperative_groups.h>

#include <algorithm>

#include "common.cuh"

namespace lobpcg {
namespace {

namespace cg = cooperative_groups;

constexpr int kCl = 8;           // CTAs of the cluster
constexpr int kThreads = 1024;
constexpr int kMaxNb = kMaxS / kCl;                                   // columns per CTA
constexpr int kPer = (kMaxS * kMaxNb + kThreads - 1) / kThreads;      // elements per thread
constexpr int kMaxSteps = 18;
constexpr int kMaxSweeps32 = 14;

__device__ __forceinline__ float block_sumf(float v, float* red) {
  v = warp_sum(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  float s = 0.f;
  for (int i = 0; i < kThreads / 32; ++i) s += red[i];
  return s;
}
__device__ __forceinline__ float block_maxf(float v, float* red) {
  // NaN counts as larger than any number
  uint32_t b = __float_as_uint(v) & 0x7fffffffu;
  b = __reduce_max_sync(0xffffffffu, b);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = __uint_as_float(b);
  __syncthreads();
  uint32_t m = 0u;
  for (int i = 0; i < kThreads / 32; ++i) m = max(m, __float_as_uint(red[i]));
  return __uint_as_float(m);
}

// Pair i of round r (circle method over N = M + 1 players, player M fixed): p < q; q may be the dummy.
__device__ __forceinline__ void pair_of(int M, int r, int i, int& p, int& q) {
  int a = i == 0 ? M : r + i, b = i == 0 ? r : r - i;
  if (i && a >= M) a -= M;
  if (b < 0) b += M;
  p = min(a, b), q = max(a, b);
}

// FP32 cyclic Jacobi in parallel order on a (s x s, column-major, ld, full storage); v holds rows
// [0, nb) of this CTA's part of the rotation product as v[col * nb + row].  A round is the rotation of
// every pair, then one pass over the 2 x 2 blocks between pairs (mirrored) and the pairs' columns of v.  A
// thread's blocks are the same in every round, and their rows and columns follow from the round by
// additions, so the pass waits on shared memory twice (rotation and entries together, stores); a round is
// latency-bound: 2.3k clocks at s = 63 with tables and 512 threads.
__device__ void jacobi32(int s, float* a, int ld, float* v, int nb, float tol, float* red, float2* cs) {
  const int N = s + (s & 1), half = N / 2, M = N - 1, nblk = half * (half + 1) / 2, total = nblk + half * nb;
  constexpr int kItems = ((kMaxS / 2) * (kMaxS / 2 + 1) / 2 + kMaxS / 2 * kMaxNb + kThreads - 1) / kThreads;
  int i1[kItems], i2[kItems];  // pairs of a block (i1 <= i2), or the pair and -1 - row of v; i1 = -1: none
#pragma unroll
  for (int k = 0; k < kItems; ++k) {
    const int e = threadIdx.x + k * kThreads;
    i1[k] = -1, i2[k] = 0;
    if (e < nblk) {
      int row = 0, base = 0;  // row-major upper triangle
      while (e >= base + half - row) base += half - row, ++row;
      i1[k] = row, i2[k] = row + e - base;
    } else if (e < total) {
      const int f = e - nblk;
      i1[k] = f / nb, i2[k] = -1 - f % nb;
    }
  }
  float f2 = 0.f;
  for (int e = threadIdx.x; e < s * s; e += kThreads) f2 += a[e % s + (e / s) * ld] * a[e % s + (e / s) * ld];
  const float fro = sqrtf(block_sumf(f2, red));
  for (int sweep = 0; sweep < kMaxSweeps32; ++sweep) {
    float o2 = 0.f;
    for (int e = threadIdx.x; e < s * s; e += kThreads) {
      const int i = e % s, j = e / s;
      if (i != j) o2 += a[i + j * ld] * a[i + j * ld];
    }
    if (sqrtf(block_sumf(o2, red)) <= tol * fro) return;
    for (int r = 0; r < M; ++r) {
      if (threadIdx.x < half) {
        int p, q;
        pair_of(M, r, threadIdx.x, p, q);
        float c = 1.f, sn = 0.f;
        if (q < s) {
          const float apq = a[p + q * ld], app = a[p + p * ld], aqq = a[q + q * ld];
          // couplings below FP32's rounding of the pair stay
          if (apq * apq > 1e-17f * fabsf(app * aqq) && fabsf(apq) > 1e-18f * fro) {
            const float tau = __fdividef(aqq - app, 2.f * apq);
            // 1 / (|tau| + sqrt(1 + tau^2)); beyond 1e15 the square would leave FP32
            const float t = fabsf(tau) > 1e15f ? __fdividef(0.5f, tau)
                                               : copysignf(__fdividef(1.f, fabsf(tau) + sqrtf(1.f + tau * tau)), tau);
            c = rsqrtf(1.f + t * t);
            sn = t * c;
          }
        }
        cs[threadIdx.x] = make_float2(c, sn);
      }
      __syncthreads();
#pragma unroll
      for (int k = 0; k < kItems; ++k) {
        if (i1[k] < 0) continue;
        const float2 r1 = cs[i1[k]];
        int p1, q1;
        pair_of(M, r, i1[k], p1, q1);
        if (i2[k] >= 0) {
          const float2 r2 = cs[i2[k]];
          int p2, q2;
          pair_of(M, r, i2[k], p2, q2);
          const bool v1 = q1 < s, v2 = q2 < s;
          const float x00 = a[p1 + p2 * ld], x01 = v2 ? a[p1 + q2 * ld] : 0.f;
          const float x10 = v1 ? a[q1 + p2 * ld] : 0.f, x11 = v1 && v2 ? a[q1 + q2 * ld] : 0.f;
          const float r00 = r1.x * x00 - r1.y * x10, r01 = r1.x * x01 - r1.y * x11;
          const float r10 = r1.y * x00 + r1.x * x10, r11 = r1.y * x01 + r1.x * x11;
          const float n00 = r2.x * r00 - r2.y * r01, n01 = r2.y * r00 + r2.x * r01;
          const float n10 = r2.x * r10 - r2.y * r11, n11 = r2.y * r10 + r2.x * r11;
          if (i1[k] == i2[k]) {  // the pair's own block: its off-diagonal entry is annihilated
            a[p1 + p1 * ld] = n00;
            if (v1) {
              const float off = r1.y != 0.f ? 0.f : x01;
              a[q1 + q1 * ld] = n11, a[p1 + q1 * ld] = off, a[q1 + p1 * ld] = off;
            }
          } else {
            a[p1 + p2 * ld] = n00, a[p2 + p1 * ld] = n00;
            if (v2) a[p1 + q2 * ld] = n01, a[q2 + p1 * ld] = n01;
            if (v1) a[q1 + p2 * ld] = n10, a[p2 + q1 * ld] = n10;
            if (v1 && v2) a[q1 + q2 * ld] = n11, a[q2 + q1 * ld] = n11;
          }
        } else if (q1 < s) {
          const int j = -1 - i2[k];
          const float vp = v[p1 * nb + j], vq = v[q1 * nb + j];
          v[p1 * nb + j] = r1.x * vp - r1.y * vq;
          v[q1 * nb + j] = r1.y * vp + r1.x * vq;
        }
      }
      __syncthreads();
    }
  }
}

// stop, mstop: a step with ||E||_F^2 and max |E| at most these is the last.
__global__ void __cluster_dims__(kCl, 1, 1) __launch_bounds__(kThreads)
    syev_cluster_kernel(int s, const double* __restrict__ a_in, int upper_only, double* __restrict__ lam,
                        double* __restrict__ U, int* steps_out, float stop, float mstop) {
  extern __shared__ double sm[];
  __shared__ float red[32];
  __shared__ float2 cs[kMaxS / 2];
  __shared__ double lsh[kMaxS];       // lambda, written by its column's CTA
  __shared__ float emax_all[kCl], esum_all[kCl];
  __shared__ int rank_of[kMaxS];
  cg::cluster_group cluster = cg::this_cluster();
  const int me = (int)cluster.block_rank(), tid = threadIdx.x;
  const int ld = s | 1;  // odd stride: columns start in different banks
  const int nb = (s + kCl - 1) / kCl;
  const int j0 = min(s, me * nb), nj = min(s, j0 + nb) - j0, cnt = s * nj;
  double* A = sm;
  double* X = A + s * ld;
  double* Wb = X + s * ld;   // nb columns
  double* Eb = Wb + nb * ld;
  float* a32 = reinterpret_cast<float*>(X);   // until X is written
  float* v32 = reinterpret_cast<float*>(Eb);

  float mx = 0.f;
  for (int e = tid; e < s * s; e += kThreads) {
    const int i = e % s, j = e / s;
    const double v = upper_only ? (i <= j ? a_in[i + j * s] : a_in[j + i * s]) : 0.5 * (a_in[i + j * s] + a_in[j + i * s]);
    A[i + j * ld] = v;
    // the exponent of the largest magnitude (NaN and infinities included)
    mx = fmaxf(mx, (float)((__double2hiint(v) >> 20) & 0x7ff));
  }
  const int ex = (int)block_maxf(mx, red);
  if (ex > 2000 || ex < 46) {  // not finite, zero, huge or tiny: the same in every CTA
    if (me == 0 && tid == 0) lam[0] = __longlong_as_double(0x7ff8000000000000ll);
    return;
  }
  // scaled by a power of two so that FP32 holds it: 1 <= max |a| < 2
  const double down = __longlong_as_double((long long)(2046 - ex) << 52), up = 1.0 / down;
  double f2 = 0.0;
  for (int e = tid; e < s * s; e += kThreads) {
    const int i = e % s, j = e / s;
    const double v = A[i + j * ld] * down;
    A[i + j * ld] = v;
    a32[i + j * ld] = (float)v;
    f2 += (float)v * (float)v;
  }
  for (int e = tid; e < s * nj; e += kThreads) v32[e] = e / nj == j0 + e % nj ? 1.f : 0.f;
  const float fro = sqrtf(block_sumf((float)f2, red));
  jacobi32(s, a32, ld, v32, nj, 1e-6f, red, cs);
  cluster.sync();  // every copy of a32 is done with: X takes its place
  for (int t = 0; t < kCl; ++t) {
    double* Xt = cluster.map_shared_rank(X, t);
    for (int e = tid; e < s * nj; e += kThreads) Xt[j0 + e % nj + (e / nj) * ld] = (double)v32[e];
  }
  cluster.sync();

  const double noise = 1e-15 * fro;  // what the plain solver leaves off the diagonal
  float last = 1.f;
  int step = 0;
  bool good = false, ortho = false;
  for (; step < kMaxSteps; ++step) {
    double R[kPer], S[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int e = tid + k * kThreads;
      if (e >= cnt) break;
      const int i = e % s, jl = e / s;
      const double *xi = X + i * ld, *xj = X + (j0 + jl) * ld, *ai = A + i * ld;
      double g = 0.0, w = 0.0;
#pragma unroll 4
      for (int r = 0; r < s; ++r) {
        const double x = xj[r];
        g = fma(xi[r], x, g);
        w = fma(ai[r], x, w);
      }
      R[k] = (i == j0 + jl ? 1.0 : 0.0) - g;
      Wb[i + jl * ld] = w;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int e = tid + k * kThreads;
      if (e >= cnt) break;
      const int i = e % s, jl = e / s;
      const double *xi = X + i * ld, *wj = Wb + jl * ld;
      double g = 0.0;
#pragma unroll 4
      for (int r = 0; r < s; ++r) g = fma(xi[r], wj[r], g);
      S[k] = g;
      U[i + (j0 + jl) * s] = g;
      if (i == j0 + jl) {
        const double l = g / (1.0 - R[k]);
        for (int t = 0; t < kCl; ++t) cluster.map_shared_rank(lsh, t)[i] = l;
      }
    }
    cluster.sync();  // lambda and S complete
    float em = 0.f, es = 0.f;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int e = tid + k * kThreads;
      if (e >= cnt) break;
      const int i = e % s, j = j0 + e / s;
      double E = 0.5 * R[k];
      if (i != j && !ortho) {
        const double gap = lsh[j] - lsh[i];
        const double num = 0.5 * (S[k] + __ldcg(U + j + i * s)) + (0.5 * (lsh[i] + lsh[j])) * R[k];
        // a small coupling over a normal gap counts whatever its size against ||a||: the Ritz vectors of
        // a graded matrix (P directions) live on it
        if (fabs(num) > 0.2 * fabs(gap)) {
          if (fabs(num) > noise) {
            const double tau = gap / (2.0 * num);
            E += 0.5 * (tau > 0.0 || (tau == 0.0 && i < j) ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
          }
        } else if (fabs(num) > noise || fabs(gap) > 1e5 * noise) {
          E += num / gap;
        }
      }
      Eb[i + (j - j0) * ld] = E;
      em = __uint_as_float(max(__float_as_uint(em), __float_as_uint((float)E) & 0x7fffffffu));
      es += (float)E * (float)E;
    }
    em = block_maxf(em, red);  // its barriers also complete Eb
    es = block_sumf(es, red);
    if (tid < kCl) cluster.map_shared_rank(emax_all, tid)[me] = em, cluster.map_shared_rank(esum_all, tid)[me] = es;
    double xn[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int e = tid + k * kThreads;
      if (e >= cnt) break;
      const int r = e % s, jl = e / s;
      const double* ej = Eb + jl * ld;
      double g = 0.0;
#pragma unroll 4
      for (int i = 0; i < s; ++i) g = fma(X[r + i * ld], ej[i], g);
      xn[k] = X[r + (j0 + jl) * ld] + g;
    }
    cluster.sync();  // every CTA has read X; emax_all and esum_all complete
    float m = 0.f, f2 = 0.f;
    for (int t = 0; t < kCl; ++t) {
      m = __uint_as_float(max(__float_as_uint(m), __float_as_uint(emax_all[t]) & 0x7fffffffu));
      f2 += esum_all[t];
    }
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int e = tid + k * kThreads;
      if (e >= cnt) break;
      const int o = e % s + (j0 + e / s) * ld;
      for (int t = 0; t < kCl; ++t) cluster.map_shared_rank(X, t)[o] = xn[k];
    }
    cluster.sync();
    if (!(m < 0.75f)) break;  // diverging or NaN (the same in every CTA)
    // what a step leaves off the diagonal is of second order, at most 5 ||E||_F^2 ||a||_F
    if (ortho ? m <= 1e-9f : f2 <= stop && m <= mstop) {
      good = true;
      ++step;
      break;
    }
    // no longer falling as squares do: rounding over small gaps, which turns vectors by up to m and takes
    // them off orthonormality by the square of it, K^T K.  Steps of R / 2 alone take that back.
    if (step >= 3 && m <= 1e-5f && m >= 0.1f * last) ortho = true;
    last = m;
  }
  // ascending eigenvalues (ties keep index order); CTA c writes its columns
  for (int i = tid; i < s; i += kThreads) {
    int r = 0;
    for (int j = 0; j < s; ++j) r += lsh[j] < lsh[i] || (lsh[j] == lsh[i] && j < i);
    rank_of[i] = r;
  }
  __syncthreads();
  if (!good) {
    if (me == 0 && tid == 0) lam[0] = __longlong_as_double(0x7ff8000000000000ll);
    return;
  }
  for (int e = tid; e < cnt; e += kThreads) U[e % s + rank_of[j0 + e / s] * s] = X[e % s + (j0 + e / s) * ld];
  for (int j = tid; j < nj; j += kThreads) lam[rank_of[j0 + j]] = lsh[j0 + j] * up;
  if (me == 0 && tid == 0 && steps_out) *steps_out = step;
}

}  // namespace

// Leaves lam[0] = NaN where the refinement did not converge (see above).
void launch_syev_cluster(int s, const double* a, bool upper_only, double* lam, double* U, int* steps_out, double tol,
                         cudaStream_t st) {
  const int ld = s | 1, nb = (s + kCl - 1) / kCl;
  const size_t smem = ((size_t)2 * s * ld + (size_t)2 * nb * ld) * sizeof(double);
  // set once per process; function-local statics initialise thread-safely
  static const bool attr = [&] {
    LB_CUDA(cudaFuncSetAttribute(syev_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (2 * kMaxS + 2 * kMaxNb) * (kMaxS + 1) * 8));
    return true;
  }();
  (void)attr;
  syev_cluster_kernel<<<kCl, kThreads, smem, st>>>(s, a, upper_only ? 1 : 0, lam, U, steps_out, (float)(tol / 5.0),
                                                  tol < 1e-12 ? 1e-9f : 1.f);
  LB_LAUNCH_CHECK();
}

}  // namespace lobpcg
