// FP64 SVD of the truncation step (Sec. IV A, Sec. V step 4): Householder QR, then
// the one-sided Jacobi method on R^T, in this library's kernels (cuSOLVER factorises
// the matrices too large for the shared memory of the GPU's SMs).
//
// One-sided Jacobi (Hestenes): plane rotations of column pairs (a, b) of a
// matrix Y, each chosen so that the rotated pair is orthogonal; repeated over
// all pairs until every pair is orthogonal to the tolerance.  For a pair with
// Gram entries alpha = |y_a|^2, beta = |y_b|^2, gamma = <y_a, y_b>, the angle
// has t = tan(theta) the smaller root of t^2 + 2 zeta t - 1 = 0, zeta =
// (beta - alpha) / (2 gamma), and
//   y_a <- c y_a - s y_b,   y_b <- s y_a + c y_b,   c = 1/sqrt(1+t^2), s = c t,
// after which <y_a, y_b> = 0 in exact arithmetic.  A pair is rotated only when
// |gamma| > tol sqrt(alpha beta), tol = max(sqrt(n), 32) 2^-52 (relative
// orthogonality; the floor keeps tol above the rounding error of the computed
// dot product, which would otherwise restart rotations of pairs with equal
// norms indefinitely).
//
// Working on R^T (A P = Q R, Householder QR of A with its columns in
// descending norm order) instead of A: the singular values of a truncated MPS
// span many orders of magnitude, and on such matrices the method needs several
// times fewer sweeps on R^T than on A; the norm order cuts the sweeps on the
// most graded sectors by a further third.
//
// Parallel order: columns in blocks of kJacB, blocks paired by the circle
// (round-robin) schedule.  With nb' = the number of blocks rounded up to even and
// N = nb' - 1, round r (0 <= r < N) pairs block r with N and (r + k) mod N with
// (r - k) mod N for k = 1 .. nb'/2 - 1; the N rounds of a sweep meet every pair of
// blocks exactly once and the pairs of one round are disjoint.  A pair of blocks
// is a CTA, which takes the pairs of columns across the two blocks in kJacB
// inner rounds of kJacB disjoint pairs, one warp each (in round 0 all pairs of
// the 2 kJacB columns, in the circle schedule); columns >= n are skipped.  One
// launch runs a round of every matrix of the batch; one sweep (a launch per
// round) is a CUDA graph.  A matrix with no rotation in a sweep is converged: in later
// sweeps its CTAs exit after their loads (the loads do not wait for the count of the
// sweep before, which would cost the CTAs still rotating a memory latency a round).
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstdlib>
#include <string>
#include <thread>

#include "fp64.cuh"
#include "kernels.hpp"
#include "launch.hpp"
#include "svd.hpp"

namespace dmrg3s {

namespace {

constexpr int kJacThreads = 128;

// Device table entry of one matrix.
struct JacJob {
  int64_t offA, offY, offV, offTau;   // Y = R^T (n x n, ld n); V1 (n x n) or offV = -1
  int64_t offS, offVT, offU;          // outputs (offU = -1: no left vectors)
  int32_t m, n, col0, pad;            // col0: first column of the matrix in the batch numbering
};

// One pair of column blocks of a round launch (a CTA): pair k of its matrix's N
// rounds.
struct JacPair {
  int64_t offY, offV;
  int32_t n, col0, k, N;
  int32_t job, staged;                // staged: the columns are held in shared memory
  float tol2;                         // the square of the pair tolerance
};

// Sum of v over the CTA (kJacThreads threads), returned to every thread.
template <class T>
__device__ __forceinline__ T cta_sum(T v, T* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  T s = red[0];
  for (int w = 1; w < kJacThreads / 32; ++w) s += red[w];
  return s;
}

// Y = R^T from the upper triangle of the factorised A (R[j][i] = A[j + i m],
// j <= i); V1 = I where the left vectors are wanted.  One CTA per column j.
__global__ void __launch_bounds__(kJacThreads)
jac_init_kernel(const JacJob* __restrict__ jobs, const int* __restrict__ col_job,
                const double* A, double* Y, double* V) {
  grid_next();
  grid_wait();
  const JacJob J = jobs[col_job[blockIdx.x]];
  const int j = blockIdx.x - J.col0;
  double* y = Y + J.offY + (int64_t)j * J.n;
  for (int i = threadIdx.x; i < J.n; i += kJacThreads)
    y[i] = i >= j ? A[J.offA + j + (int64_t)i * J.m] : 0.0;
  if (J.offV >= 0) {
    double* v = V + J.offV + (int64_t)j * J.n;
    for (int i = threadIdx.x; i < J.n; i += kJacThreads) v[i] = i == j ? 1.0 : 0.0;
  }
}

// Squared norm of every column of every A (m rows, ld m).  One CTA per column.
__global__ void __launch_bounds__(kJacThreads)
jac_anorm_kernel(const JacJob* __restrict__ jobs, const int* __restrict__ col_job,
                 const double* A, double* nrm) {
  grid_next();
  grid_wait();
  __shared__ double red[kJacThreads / 32];
  const JacJob J = jobs[col_job[blockIdx.x]];
  const int j = blockIdx.x - J.col0;
  const double* x = A + J.offA + (int64_t)j * J.m;
  double s = 0.0;
  for (int i = threadIdx.x; i < J.m; i += kJacThreads) s = fma(x[i], x[i], s);
  s = cta_sum(s, red);
  if (threadIdx.x == 0) nrm[blockIdx.x] = s;
}

// T = A P: column j of T is column perm[j] of A.  One CTA per column.
__global__ void __launch_bounds__(kJacThreads)
jac_permute_kernel(const JacJob* __restrict__ jobs, const int* __restrict__ col_job,
                   const int* perm, const double* A,
                   double* T) {
  grid_next();
  grid_wait();
  const JacJob J = jobs[col_job[blockIdx.x]];
  const int j = blockIdx.x - J.col0;
  const double* x = A + J.offA + (int64_t)perm[blockIdx.x] * J.m;
  double* t = T + J.offA + (int64_t)j * J.m;
  for (int i = threadIdx.x; i < J.m; i += kJacThreads) t[i] = x[i];
}

// ---- Householder QR of every matrix of the batch ----

// A matrix's columns are dealt round-robin to G CTAs, which hold them in shared
// memory.  Step j: the owner of column j forms its reflector (LAPACK's
// convention: v below the diagonal with v_j = 1 implied, beta on it, H = I - tau v
// v^T) and publishes it in place; every CTA applies it to its later columns,
// the owner of column j + 1 to that one first, so that the next reflector is on
// its way while the others still update (a step waits for one flag, not for a
// barrier).  CTAs of one matrix wait for each other: cooperative launch, a CTA takes
// its share of one divided matrix first and then whole small matrices.
// Bound by the FP64 pipe of the matrix's SMs (two multiply-adds per element of
// the trailing columns and step) and, per step, by ~2 us of the chain norm, square
// root, publication.  Whole SVDs with cuSOLVER's QR before: the 14 sectors (up to 762 x
// 245) of an m = 512 XXZ truncation 22.1 -> 10.9 ms, 60 matrices of 60 x 40 31.0 ->
// 3.5, 762 x 245 alone 11.9 -> 10.1, 1300 x 1100 121 -> 110, 16 x 8 1.09 -> 0.55.
struct QrItem {
  int64_t offA, offTau;
  int32_t m, n, rank, G, job, pad;   // G CTAs, this one has the columns rank, rank + G, ..
};
constexpr int kQrThreads = 512, kQrWarps = kQrThreads / 32;
constexpr size_t kQrSmem = 200 * 1024;
constexpr int kQrUnits = 64;         // partial dot products of a round

// The chain of a step runs on the first four warps, one per sub-partition: with
// more, the reductions' FP64 additions would cost more than the split saves.
constexpr int kQrChain = 128;
__device__ __forceinline__ void chain_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

// Sum over the chain's warps, the same in every thread of it.
__device__ __forceinline__ double chain_sum4(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  chain_sync();
  return (red[0] + red[1]) + (red[2] + red[3]);
}

__device__ __forceinline__ double chain_max4(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  chain_sync();
  return fmax(fmax(red[0], red[1]), fmax(red[2], red[3]));
}

// By the chain's threads: the reflector of column a (rows j .. m - 1, in shared
// memory) into v (v[j] = 1) and, with beta on the diagonal, into the matrix; tau
// into *tau and red[6 + (j & 1)] (a CTA of a matrix of its own forms reflector j + 1
// while its other warps still read tau_j).
__device__ __forceinline__ void qr_reflector(double* a, double* v, int j, int m, double* T,
                                             double* tau, double* red) {
  double s = 0.0;
  for (int i = j + 1 + threadIdx.x; i < m; i += kQrChain) s = fma(a[i], a[i], s);
  s = chain_sum4(s, red);
  const double alpha = a[j];
  double beta = alpha, tv = 0.0, sc = 0.0;
  const double n2 = fma(alpha, alpha, s);
  if (n2 > 1e-290 && n2 < 1e290) {
    if (s != 0.0) {
      const double nr = sqrt_of(n2);
      beta = alpha >= 0.0 ? -nr : nr;
      sc = recip(alpha - beta);         // |alpha - beta| >= |beta|
      tv = (beta - alpha) * recip(beta);
    }
  } else {
    // squares outside the FP64 range (a norm with few digits would give a reflection
    // that is not orthogonal): the column scaled by a power of two of its largest
    // element (Inf and NaN pass through)
    double mx = 0.0;
    for (int i = j + threadIdx.x; i < m; i += kQrChain) mx = fmax(mx, fabs(a[i]));
    chain_sync();
    mx = chain_max4(mx, red);
    if (!(n2 == n2)) mx = n2;
    if (mx != 0.0) {
      const double up = inverse_scale(mx);
      for (int i = j + threadIdx.x; i < m; i += kQrChain) a[i] *= up;
      chain_sync();
      double s1 = 0.0;
      for (int i = j + 1 + threadIdx.x; i < m; i += kQrChain) s1 = fma(a[i], a[i], s1);
      s1 = chain_sum4(s1, red);
      if (s1 != 0.0) {                  // (NaN: every result is NaN)
        const double al = up * alpha, nr = sqrt(fma(al, al, s1));
        const double b = al >= 0.0 ? -nr : nr;
        beta = b / up;
        sc = 1.0 / (al - b);
        tv = (b - al) / b;
      }
    }
  }
  for (int i = j + threadIdx.x; i < m; i += kQrChain) {
    const double x = i == j ? 1.0 : a[i] * sc;
    v[i] = x;
    T[i] = i == j ? beta : x;
  }
  if (threadIdx.x == 0) {
    *tau = tv;
    red[6 + (j & 1)] = tv;
  }
}

__global__ void __launch_bounds__(kQrThreads, 1)
qr_kernel(const QrItem* __restrict__ items, const int* __restrict__ cta_item, double* A, double* tau,
          int* ready, int* err, uint64_t limit_ns) {
  extern __shared__ double sh[];
  __shared__ double red[8];              // a sum's partials, two taus
  __shared__ double part[kQrUnits * kQrWarps];
  __shared__ int s_ok;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int it = cta_item[blockIdx.x]; it < cta_item[blockIdx.x + 1]; ++it) {
    const QrItem Q = items[it];
    const int m = Q.m, n = Q.n, G = Q.G;
    const int nc = Q.rank < n ? (n - Q.rank + G - 1) / G : 0;   // own columns
    double* vb = sh;                                 // two reflectors, then the columns
    double* cols = sh + 2 * m;
    double* T = A + Q.offA;
    for (int q = 0; q < nc; ++q) {
      const double* src = T + (int64_t)(Q.rank + q * G) * m;
      for (int i = tid; i < m; i += kQrThreads) cols[(int64_t)q * m + i] = src[i];
    }
    __syncthreads();
    double t_next = 0.0;
    bool have = false;                               // the next reflector is in place
    const int steps = min(n, m);
    for (int j = 0; j < steps; ++j) {
      double* v = vb + (j & 1) * m;
      double tv;
      if (have) {
        tv = t_next;
      } else if (j % G == Q.rank) {                  // (step 0 only)
        if (tid < kQrChain)
          qr_reflector(cols + (int64_t)(j / G) * m, v, j, m, T + (int64_t)j * m,
                       tau + Q.offTau + j, red);
        __syncthreads();
        tv = red[6 + (j & 1)];
        if (G > 1 && tid == 0) {
          __threadfence();
          asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(ready + Q.job), "r"(j + 1) : "memory");
        }
      } else {
        if (j >= Q.rank + (nc - 1) * G) break;       // no column of this CTA is left
        if (tid == 0) {
          int ok = 1, r;
          uint64_t t0, t;
          asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
          for (;;) {
            asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(r) : "l"(ready + Q.job) : "memory");
            if (r > j) break;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
            if (t - t0 > limit_ns) {
              atomicExch(err, 1);
              ok = 0;
              break;
            }
          }
          s_ok = ok;
        }
        __syncthreads();
        if (!s_ok) return;
        const double* src = T + (int64_t)j * m;
        for (int i = j + tid; i < m; i += kQrThreads) v[i] = i == j ? 1.0 : __ldcg(src + i);
        tv = __ldcg(tau + Q.offTau + j);
        __syncthreads();
      }
      // the next column first, by the whole CTA, and its reflector
      have = j + 1 < steps && (j + 1) % G == Q.rank;
      int q0 = j < Q.rank ? 0 : (j - Q.rank) / G + 1;   // first own column > j
      if (have) {
        if (tid < kQrChain) {
          double* a = cols + (int64_t)q0 * m;
          double s = 0.0;
          for (int i = j + tid; i < m; i += kQrChain) s = fma(v[i], a[i], s);
          s = -tv * chain_sum4(s, red);
          for (int i = j + tid; i < m; i += kQrChain) a[i] = fma(s, v[i], a[i]);
          chain_sync();
          qr_reflector(a, vb + ((j + 1) & 1) * m, j + 1, m, T + (int64_t)(j + 1) * m,
                       tau + Q.offTau + j + 1, red);
        }
        __syncthreads();
        t_next = red[6 + ((j + 1) & 1)];
        if (G > 1 && tid == 0) {
          __threadfence();
          asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(ready + Q.job), "r"(j + 2) : "memory");
        }
        ++q0;
      }
      // the others: w warps a column, in rounds of kQrUnits columns
      for (int qb = q0; qb < nc; qb += kQrUnits) {
        const int k = min(kQrUnits, nc - qb);
        int w = 1;
        while (2 * w * k <= kQrWarps) w *= 2;
        const int len = (((m - j + w - 1) / w) + 31) & ~31;   // rows of a warp
        for (int u = warp; u < k * w; u += kQrWarps) {
          const int c = u / w, part_i = u % w;
          const double* a = cols + (int64_t)(qb + c) * m;
          const int i0 = j + part_i * len, i1 = min(m, i0 + len);
          double s0 = 0.0, s1 = 0.0;
          int i = i0 + lane;
          for (; i + 32 < i1; i += 64) {
            s0 = fma(v[i], a[i], s0);
            s1 = fma(v[i + 32], a[i + 32], s1);
          }
          if (i < i1) s0 = fma(v[i], a[i], s0);
          s0 += s1;
          for (int o = 16; o > 0; o >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, o);
          if (w == 1) {
            const double f = -tv * s0;
            double* aw = cols + (int64_t)(qb + c) * m;
            for (i = i0 + lane; i < i1; i += 32) aw[i] = fma(f, v[i], aw[i]);
          } else if (lane == 0) {
            part[c * kQrWarps + part_i] = s0;
          }
        }
        if (w > 1) {
          __syncthreads();
          for (int u = warp; u < k * w; u += kQrWarps) {
            const int c = u / w, part_i = u % w;
            double s = part[c * kQrWarps];
            for (int x = 1; x < w; ++x) s += part[c * kQrWarps + x];
            const double f = -tv * s;
            double* a = cols + (int64_t)(qb + c) * m;
            const int i0 = j + part_i * len, i1 = min(m, i0 + len);
            for (int i = i0 + lane; i < i1; i += 32) a[i] = fma(f, v[i], a[i]);
          }
        }
      }
      __syncthreads();
    }
    // R above the diagonal (the rest is in place)
    for (int q = 0; q < nc; ++q) {
      const int c = Q.rank + q * G;
      for (int i = tid; i < min(c, m); i += kQrThreads) T[(int64_t)c * m + i] = cols[(int64_t)q * m + i];
    }
    __syncthreads();
  }
}

// U <- Q U for the left vectors: the reflectors in reverse order on every column, a
// warp per column with the column in shared memory (m <= kQrApplyRows) and the
// same rows in the same lanes throughout, so a warp needs nothing from another.
// Bound by the FP64 pipe.  Whole SVDs with left vectors, cuSOLVER's ormqr before: 60
// matrices of 60 x 40 34 -> 4.1 ms, 14 sectors up to 762 x 245 24.1 -> 16.7, 200 x 100
// 6.6 -> 5.2, 762 x 245 alone 16.6 -> 16.2.
struct QrColumns {
  int32_t job, col0;
};
constexpr int kQrApplyWarps = 4;
constexpr int kQrApplyRows = 6400;
constexpr size_t kQrApplySmem = sizeof(double) * kQrApplyWarps * kQrApplyRows;
__global__ void __launch_bounds__(32 * kQrApplyWarps)
qr_apply_kernel(const JacJob* __restrict__ jobs, const QrColumns* __restrict__ items, const double* A,
                const double* tau, double* U, int stride) {
  grid_next();
  grid_wait();
  extern __shared__ double sh[];
  const QrColumns I = items[blockIdx.x];
  const JacJob J = jobs[I.job];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c = I.col0 + warp, m = J.m, n = J.n;
  if (c >= n) return;
  double* ug = U + J.offU + (int64_t)c * m;
  const bool staged = m <= stride;
  double* u = staged ? sh + (int64_t)warp * stride : ug;
  if (staged)
    for (int i = lane; i < m; i += 32) u[i] = ug[i];
  const double* T = A + J.offA;
  double t_next = tau[J.offTau + n - 1];
  for (int j = n - 1; j >= 0; --j) {
    const double t = t_next;
    if (j > 0) t_next = tau[J.offTau + j - 1];
    if (t == 0.0) continue;
    const double* v = T + (int64_t)j * m;
    const int i0 = (j & ~31) + lane;                 // v is 0 above row j, 1 on it
    const double vd = i0 > j ? (i0 < m ? v[i0] : 0.0) : i0 == j ? 1.0 : 0.0;
    double s0 = i0 < m ? vd * u[i0] : 0.0, s1 = 0.0;
    int i = i0 + 32;
#pragma unroll 2
    for (; i + 32 < m; i += 64) {
      s0 = fma(v[i], u[i], s0);
      s1 = fma(v[i + 32], u[i + 32], s1);
    }
    if (i < m) s0 = fma(v[i], u[i], s0);
    s0 += s1;
    for (int o = 16; o > 0; o >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, o);
    const double f = -t * s0;
    if (i0 < m) u[i0] = fma(f, vd, u[i0]);
#pragma unroll 4
    for (i = i0 + 32; i < m; i += 32) u[i] = fma(f, v[i], u[i]);
  }
  if (staged)
    for (int i = lane; i < m; i += 32) ug[i] = u[i];
}

// The batch's matrices dealt to at most `ctas` CTAs so that the longest takes about
// the least time by a model of the kernel (microseconds): FP64 work over the
// matrix's SMs plus a step's chain.  `lib` receives the matrices whose columns do
// not fit the shared memory of the CTAs (cuSOLVER factorises those).
struct QrPlan {
  std::vector<QrItem> items;
  std::vector<int> cta_item{0};
  size_t smem = 0;
};
void plan_qr(const std::vector<JacJob>& tab, int ctas, QrPlan* plan, std::vector<int>* lib) {
  const auto time = [](double m, double n, int G) {
    return n * (G > 1 ? 3.0 : 2.0) + (m * n * n - n * n * n / 3.0) / (3800.0 * G);
  };
  const auto least = [](int64_t m, int64_t n) {       // CTAs whose shared memory holds the columns
    const int64_t fit = (int64_t)(kQrSmem / sizeof(double)) / m - 2;
    return fit < 1 ? (int64_t)0 : (n + fit - 1) / fit;
  };
  std::vector<int> jobs;
  lib->clear();
  int64_t need = 0;
  for (int k = 0; k < (int)tab.size(); ++k) {
    const int64_t g = least(tab[k].m, tab[k].n);
    if (g < 1 || (g > 1 && need + g > ctas - 2)) {
      lib->push_back(k);
    } else {
      if (g > 1) need += g;
      jobs.push_back(k);
    }
  }
  if (jobs.empty()) return;
  // the CTAs of every matrix for a makespan t: the fewest that keep to it
  std::vector<int> G(tab.size(), 1);
  const auto fits = [&](double t) {
    int64_t many = 0;
    double rest = 0.0;
    for (int k : jobs) {
      const double m = tab[k].m, n = tab[k].n;
      int64_t g = least(tab[k].m, tab[k].n);
      if (g == 1 && time(m, n, 1) <= t) {
        rest += time(m, n, 1);
      } else {
        g = std::max<int64_t>(g, 2);
        while (g < tab[k].n && time(m, n, (int)g) > t) ++g;
        many += g;
      }
      G[k] = (int)g;
    }
    return many + (int64_t)std::ceil(rest / t) + (rest > 0.0 ? 1 : 0) <= ctas;
  };
  double t = 20.0;
  while (!fits(t) && t < 1e9) t *= 1.1;
  if (t >= 1e9) {                                    // (the CTAs are few: everything to the library)
    lib->insert(lib->end(), jobs.begin(), jobs.end());
    return;
  }
  std::vector<std::vector<QrItem>> queue;
  std::vector<double> load;
  std::sort(jobs.begin(), jobs.end(), [&](int a, int b) {
    if ((G[a] > 1) != (G[b] > 1)) return G[a] > 1;
    return time(tab[a].m, tab[a].n, 1) > time(tab[b].m, tab[b].n, 1);
  });
  for (int k : jobs) {
    const JacJob& J = tab[k];
    const QrItem q{J.offA, J.offTau, J.m, J.n, 0, G[k], k, 0};
    const size_t own = (size_t)((J.n + G[k] - 1) / G[k]);
    plan->smem = std::max(plan->smem, (2 + own) * J.m * sizeof(double));
    if (G[k] > 1) {
      for (int r = 0; r < G[k]; ++r) {
        queue.push_back({q});
        queue.back()[0].rank = r;
        load.push_back(time(J.m, J.n, G[k]));
      }
      continue;
    }
    // whole matrices: to the least loaded CTA, a new one while there are any
    size_t w = std::min_element(load.begin(), load.end()) - load.begin();
    if ((int)queue.size() < ctas) {
      w = queue.size();
      queue.emplace_back();
      load.push_back(0.0);
    }
    queue[w].push_back(q);
    load[w] += time(J.m, J.n, 1);
  }
  for (const auto& v : queue) {
    plan->items.insert(plan->items.end(), v.begin(), v.end());
    plan->cta_item.push_back((int)plan->items.size());
  }
}

// The rotation of a pair with d = beta - alpha and gamma = g, as p = tan(theta / 2)
// and s = sin(theta) = 2 p / (1 + p^2).  GB300 issues FP64 at 1/64 of its FP32
// rate, and a division or square root in FP64 is a long chain of such
// instructions, so the angle is computed in FP32 from d and 2 g scaled by a
// common power of two; p is that FP32 number and s belongs to it to FP64
// accuracy (an FP32 reciprocal r0 of q = 1 + p^2, then 1 / q = r0 (1 + e + e^2 +
// ..) with e = 1 - q r0 below 2^-22).  The angle carries FP32 rounding (~1e-7
// relative): the rotated pair is orthogonal to ~1e-7 of its former cosine rather
// than exactly, which the next sweep removes; the rotation itself is orthogonal
// to FP64 rounding, so the singular values are unaffected.
__device__ __forceinline__ void jacobi_rotation(double d, double g, double* p, double* p2,
                                                double* s) {
  const int ed = exponent_of(d);
  const int eg = exponent_of(g) + 1;   // of 2 g
  double pp, pp2;
  float pf = 0.f;
  if (ed - eg > 20) {
    // |zeta| > 2^19: theta = gamma / (beta - alpha) to FP32 rounding
    const float t = __fdividef(float_of(g, eg - 1), float_of(d, ed));
    pp = double_of(t, eg - ed - 2);
    pp2 = double_of(t, eg - ed - 1);
  } else {
    // tan(theta) = 2 g / (d +- sqrt(d^2 + 4 g^2)), tan(theta / 2) = t / (1 + sqrt(1 + t^2))
    const int e = max(ed, eg);
    const float df = float_of(d, e), gf = float_of(g, e - 1);
    const float h2 = fmaf(df, df, gf * gf);
    const float t = __fdividef(copysignf(1.0f, df) * gf, fabsf(df) + h2 * rsqrtf(h2));
    const float u2 = fmaf(t, t, 1.0f);
    pf = __fdividef(t, 1.0f + u2 * rsqrtf(u2));
    pp = double_of(pf, 0);
    pp2 = double_of(pf, 1);
  }
  const double r0 = double_of(__fdividef(1.0f, fmaf(pf, pf, 1.0f)), 0);
  const double q = fma(pp, pp, 1.0);
  const double e1 = fma(-q, r0, 1.0);
  const double s0 = pp2 * r0;
  *p = pp;
  *p2 = pp2;
  *s = fma(s0, fma(e1, e1, e1), s0);
}

// (a, b) <- (c a - s b, s a + c b) as three shears: half the roundings of the
// product form, and the error of each is that of a fused multiply-add (the
// singular values of graded 100 to 245-column matrices, against long double: 1.4
// to 2.7e-15 at the largest, 4 to 7e-15 in the product form).
__device__ __forceinline__ void shears(double p, double s, double& a, double& b) {
  a = fma(-p, b, a);
  b = fma(s, a, b);
  a = fma(-p, b, a);
}

// gamma^2 > tol2 alpha beta, for positive alpha and beta, in FP32 on the mantissas
// (the threshold moves by 1e-6 of itself at most).
__device__ __forceinline__ bool needs_rotation(double alpha, double beta, double g, float tol2) {
  const int ea = exponent_of(alpha), eb = exponent_of(beta), eg = exponent_of(g);
  const float fg = float_of(g, eg), f = __fdividef(fg * fg, float_of(alpha, ea) * float_of(beta, eb));
  const int e = 2 * eg - ea - eb;                    // gamma^2 / (alpha beta) = f 2^e, f in (1/4, 4)
  if (eg == 0 || e < -120) return false;
  return e > 100 || f * __uint_as_float((unsigned)(e + 127) << 23) > tol2;
}

// Sum of the lanes' x to FP64 rounding, in every lane, without FP64 additions: the
// significands are shifted to a common exponent (63 bits with the carries of 32
// lanes) and added as integers.  *finite is false when a lane holds Inf or NaN.
__device__ __forceinline__ double warp_sum_fixed(double x, bool* finite) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int e = exponent_of(x);
  const int top = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
  *finite = top < 0x7ff;
  const int sh = top - e;
  unsigned long long m = ((u & 0xfffffffffffffull) | (e > 0 ? 1ull << 52 : 0ull)) << 5;
  m = sh < 64 ? m >> sh : 0ull;
  const long long v = (long long)u < 0 ? -(long long)m : (long long)m;   // x 2^(1080 - top)
  // limbs of 26 bits (the last signed)
  const unsigned s0 = __reduce_add_sync(0xffffffffu, (unsigned)v & 0x3ffffffu);
  const unsigned s1 = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 26) & 0x3ffffffu);
  const int s2 = __reduce_add_sync(0xffffffffu, (int)(v >> 52));
  const long long s = (long long)s0 + ((long long)s1 << 26) + ((long long)s2 << 52);
  const double r = (double)s;
  // times 2^(top - 1080) on the exponent (0 below the normal range)
  const int er = exponent_of(r) + top - 1080;
  return s == 0 || er < 1 ? 0.0
                          : __longlong_as_double((__double_as_longlong(r) & ~(0x7ffll << 52)) |
                                                 (long long)er << 52);
}

// Starts a sweep: the squared norm of every column of every Y (one CTA per
// column), and the sweep counter read by the round kernels.
__global__ void __launch_bounds__(kJacThreads)
jac_sweep_kernel(const JacJob* __restrict__ jobs, const int* __restrict__ col_job,
                 const double* Y, double* nrm, int* sweep) {
  grid_next();
  grid_wait();
  __shared__ double red[kJacThreads / 32];
  const JacJob J = jobs[col_job[blockIdx.x]];
  const double* y = Y + J.offY + (int64_t)(blockIdx.x - J.col0) * J.n;
  double s = 0.0;
  for (int i = threadIdx.x; i < J.n; i += kJacThreads) s = fma(y[i], y[i], s);
  s = cta_sum(s, red);
  if (threadIdx.x == 0) {
    nrm[blockIdx.x] = s;
    if (blockIdx.x == 0) *sweep += 1;
  }
}

// One round r of the current sweep for every matrix: one CTA per pair of
// blocks, one warp per pair of columns.  rot[s * njobs + job] counts the
// rotations of sweep s.  GB300 runs an FP64 warp instruction in ~64 cycles of a
// sub-partition, and the pairs of a truncation are about as many as the chip's
// sub-partitions, so an inner round is priced in FP64 instructions of one warp:
// one dot product (the squared norms are kept through the sweep by the rotation's
// own recurrence, |y_a'|^2 = alpha + s (s (beta - alpha) - 2 c gamma), and formed
// anew at the next sweep's start, so the last sweep, which rotates nothing, tests
// every pair with fresh norms), a reduction in integers, ~11 for the rotation (every
// lane computes the identical one: no exchange) and the norms, and three shears per
// element, four elements' chains interleaved: ~43 at n = 245, where three dot
// products and the product form took ~80.  The columns of a CTA stay in shared
// memory between the inner rounds where they fit, so that only every kJacB-th
// round pays for a launch and for its loads.  ncu: the FP64 pipe 46 % busy on the
// fullest SM, the rest is the chain of shared-memory loads, reduction and rotation.
// Whole factorisations (a launch per round of column pairs / this / this with
// the reduction, test and angle in FP64 and IEEE FP32): 762 x 245 18.1 / 11.9 / 13.2 ms,
// 900 x 600 74 / 41 / 45, 1300 x 1100 (columns in global memory) 213 / 122 / 126;
// the local update of an m = 512 XXZ window 30.6 / 22.7 / 24.3.
constexpr int kJacB = 4;
constexpr int kJacCache = 8;              // elements of a column that a lane keeps in registers
constexpr size_t kJacStage = 64 * 1024;   // shared memory of a CTA: three fit an SM
__global__ void __launch_bounds__(32 * kJacB)
jac_round_kernel(const JacPair* __restrict__ pairs, int njobs, int r, const int* sweep, int* rot,
                 double* nrm, double* Y, double* V) {
  grid_next();
  grid_wait();
  extern __shared__ double cols[];
  __shared__ double s_nrm[2 * kJacB];
  const JacPair P = pairs[blockIdx.x];
  const int sw = *sweep;
  if (r >= P.N || sw < 0 || sw >= kJacobiMaxSweeps) return;
  const int n = P.n, k = P.k, N = P.N;
  // first columns of the two blocks
  const int ca = (k == 0 ? r : (r + k) % N) * kJacB;
  const int cb = (k == 0 ? N : (r - k + N) % N) * kJacB;
  if (r > 0 && (ca >= n || cb >= n)) return;   // the padding block
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int before = sw > 0 ? rot[(sw - 1) * njobs + P.job] : 1;
  const bool vec = P.offV >= 0;
  double* yg = Y + P.offY;
  double* vg = vec ? V + P.offV : nullptr;
  double* ys = cols;
  double* vs = cols + 2 * kJacB * n;
  const auto column = [&](int c) { return c < kJacB ? ca + c : cb + c - kJacB; };
  if (P.staged) {
    for (int h = 0; h < 2; ++h) {
      const int c = warp + h * kJacB;
      const int g = column(c);
      if (g >= n) continue;
      for (int i = lane; i < n; i += 32) ys[c * n + i] = yg[(int64_t)g * n + i];
      if (vec)
        for (int i = lane; i < n; i += 32) vs[c * n + i] = vg[(int64_t)g * n + i];
    }
  }
  if (threadIdx.x < 2 * kJacB) {
    const int g = column(threadIdx.x);
    s_nrm[threadIdx.x] = g < n ? nrm[P.col0 + g] : 0.0;
  }
  if (before == 0) return;   // converged in the previous sweep (the same for the whole CTA)
  __syncthreads();
  const int M = 2 * kJacB - 1;
  const int ne = (n + 31) / 32;
  const int inner = r == 0 ? M : kJacB;
  int nrot = 0;
  for (int q = 0; q < inner; ++q) {
    int a, b;
    if (r > 0) {
      a = warp;
      b = kJacB + ((warp + q) & (kJacB - 1));
    } else {
      a = warp == 0 ? q : (q + warp) % M;
      b = warp == 0 ? M : (q - warp + M) % M;
    }
    const int ga = column(a), gb = column(b);
    if (ga < n && gb < n) {
      double* ya = P.staged ? ys + a * n : yg + (int64_t)ga * n;
      double* yb = P.staged ? ys + b * n : yg + (int64_t)gb * n;
      const double alpha = s_nrm[a], beta = s_nrm[b];
      double ua[kJacCache], ub[kJacCache];
      double gs[2] = {0.0, 0.0};
#pragma unroll
      for (int e = 0; e < kJacCache; ++e) {
        const int i = lane + e * 32;
        ua[e] = i < n ? ya[i] : 0.0;
        ub[e] = i < n ? yb[i] : 0.0;
      }
      // elements in fours (interleaved chains) while whole fours remain, then one
      // by one
#pragma unroll
      for (int e0 = 0; e0 < kJacCache; e0 += 4) {
        if (ne >= e0 + 4) {
#pragma unroll
          for (int e = e0; e < e0 + 4; ++e) gs[e & 1] = fma(ua[e], ub[e], gs[e & 1]);
        } else {
#pragma unroll
          for (int e = e0; e < e0 + 3; ++e)
            if (e < ne) gs[e & 1] = fma(ua[e], ub[e], gs[e & 1]);
        }
      }
      for (int i = lane + kJacCache * 32; i < n; i += 32) gs[0] = fma(ya[i], yb[i], gs[0]);
      bool finite;
      const double g = warp_sum_fixed(gs[0] + gs[1], &finite);
      // zero columns, Inf and NaN leave the pair unrotated (NaN reaches the
      // singular values); a norm cancelled to nothing waits for the next sweep's
      if (finite && __double_as_longlong(alpha) > 0 && __double_as_longlong(beta) > 0 &&
          needs_rotation(alpha, beta, g, P.tol2)) {
        const double d = beta - alpha;
        double p, p2, s;
        jacobi_rotation(d, g, &p, &p2, &s);
        ++nrot;
#pragma unroll
        for (int e0 = 0; e0 < kJacCache; e0 += 4) {
          if (ne >= e0 + 4) {
#pragma unroll
            for (int e = e0; e < e0 + 4; ++e) ua[e] = fma(-p, ub[e], ua[e]);
#pragma unroll
            for (int e = e0; e < e0 + 4; ++e) ub[e] = fma(s, ua[e], ub[e]);
#pragma unroll
            for (int e = e0; e < e0 + 4; ++e) ua[e] = fma(-p, ub[e], ua[e]);
          } else {
#pragma unroll
            for (int e = e0; e < e0 + 3; ++e)
              if (e < ne) shears(p, s, ua[e], ub[e]);
          }
        }
#pragma unroll
        for (int e = 0; e < kJacCache; ++e) {
          const int i = lane + e * 32;
          if (i < n) {
            ya[i] = ua[e];
            yb[i] = ub[e];
          }
        }
        for (int i = lane + kJacCache * 32; i < n; i += 32) {
          double u = ya[i], v = yb[i];
          shears(p, s, u, v);
          ya[i] = u;
          yb[i] = v;
        }
        if (vec) {
          double* va = P.staged ? vs + a * n : vg + (int64_t)ga * n;
          double* vb = P.staged ? vs + b * n : vg + (int64_t)gb * n;
#pragma unroll 4
          for (int i = lane; i < n; i += 32) {
            double u = va[i], v = vb[i];
            shears(p, s, u, v);
            va[i] = u;
            vb[i] = v;
          }
        }
        const double c2 = fma(-p2, s, 2.0);   // 2 cos(theta)
        const double dl = s * fma(s, d, -(c2 * g));
        __syncwarp();
        if (lane == 0) {
          s_nrm[a] = alpha + dl;
          s_nrm[b] = beta - dl;
        }
      }
    }
    __syncthreads();
  }
  if (nrot && lane == 0) atomicAdd(rot + sw * njobs + P.job, nrot);
  if (!__syncthreads_or(nrot)) return;
  if (P.staged) {
    for (int h = 0; h < 2; ++h) {
      const int c = warp + h * kJacB;
      const int g = column(c);
      if (g >= n) continue;
      for (int i = lane; i < n; i += 32) yg[(int64_t)g * n + i] = ys[c * n + i];
      if (vec)
        for (int i = lane; i < n; i += 32) vg[(int64_t)g * n + i] = vs[c * n + i];
    }
  }
  if (threadIdx.x < 2 * kJacB) {
    const int g = column(threadIdx.x);
    if (g < n) nrm[P.col0 + g] = s_nrm[threadIdx.x];
  }
}

__global__ void __launch_bounds__(kJacThreads)
jac_norm_kernel(const JacJob* __restrict__ jobs, const int* __restrict__ col_job,
                const double* Y, double* sig) {
  grid_next();
  grid_wait();
  __shared__ double red[kJacThreads / 32];
  const JacJob J = jobs[col_job[blockIdx.x]];
  const int j = blockIdx.x - J.col0;
  const double* y = Y + J.offY + (int64_t)j * J.n;
  double s = 0.0;
  for (int i = threadIdx.x; i < J.n; i += kJacThreads) s = fma(y[i], y[i], s);
  s = cta_sum(s, red);
  if (threadIdx.x == 0) sig[blockIdx.x] = sqrt(s);
}

// Sort key: NaN above everything, so that it lands in S and is seen.
__device__ __forceinline__ double sig_key(double x) { return x != x ? INFINITY : x; }

// Column j of matrix J goes to position c = its rank (descending sigma, ties
// by index): S[c] = sigma_j, VT row c = P y_j / sigma_j (P: the column order
// of the factorised A P), and, when wanted, U column c = (V1 column j; 0),
// which Q then multiplies.  One CTA per column.
__global__ void __launch_bounds__(kJacThreads)
jac_scatter_kernel(const JacJob* __restrict__ jobs, const int* __restrict__ col_job,
                   const int* perm, const double* Y,
                   const double* V, const double* sig,
                   double* S, double* VT, double* U) {
  grid_next();
  grid_wait();
  __shared__ int red[kJacThreads / 32];
  const JacJob J = jobs[col_job[blockIdx.x]];
  const int j = blockIdx.x - J.col0;
  const int n = J.n;
  const double s = sig[blockIdx.x];
  const double ks = sig_key(s);
  int cnt = 0;
  for (int i = threadIdx.x; i < n; i += kJacThreads) {
    const double o = sig_key(sig[J.col0 + i]);
    cnt += (o > ks || (o == ks && i < j)) ? 1 : 0;
  }
  const int c = cta_sum(cnt, red);
  if (threadIdx.x == 0) S[J.offS + c] = s;
  const double* y = Y + J.offY + (int64_t)j * n;
  const int* pj = perm + J.col0;   // row i of R belongs to column pj[i] of A
  for (int i = threadIdx.x; i < n; i += kJacThreads)
    VT[J.offVT + c + (int64_t)pj[i] * n] = s > 0.0 ? y[i] / s : 0.0;
  if (J.offU >= 0) {
    const double* v = V + J.offV + (int64_t)j * n;
    double* u = U + J.offU + (int64_t)c * J.m;
    for (int i = threadIdx.x; i < J.m; i += kJacThreads) u[i] = i < n ? v[i] : 0.0;
  }
}

dmrg3s_status cuda_ok(Context* c, cudaError_t e, const char* what) {
  if (e == cudaSuccess) return DMRG3S_OK;
  return fail(c, DMRG3S_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

}  // namespace

dmrg3s_status lane_ready(Context* c, SvdLane* w) {
  if (w->ev) return DMRG3S_OK;
  if (cusolverDnCreate(&w->h) != CUSOLVER_STATUS_SUCCESS ||
      cusolverDnCreateParams(&w->p) != CUSOLVER_STATUS_SUCCESS ||
      cudaStreamCreateWithFlags(&w->s, cudaStreamNonBlocking) != cudaSuccess ||
      cudaEventCreateWithFlags(&w->ev, cudaEventDisableTiming) != cudaSuccess) {
    lane_destroy(w);
    return fail(c, DMRG3S_ERR_CUDA, "SVD lane set-up");
  }
  return DMRG3S_OK;
}

void lane_destroy(SvdLane* w) {
  if (w->dwork) cudaFree(w->dwork);
  if (w->p) cusolverDnDestroyParams(w->p);
  if (w->h) cusolverDnDestroy(w->h);
  if (w->ev) cudaEventDestroy(w->ev);
  if (w->s) cudaStreamDestroy(w->s);
  *w = SvdLane();
}

int jacobi_max_sweeps() {
  const char* e = std::getenv("DMRG3S_JACOBI_SWEEPS");
  if (!e) return kJacobiMaxSweeps;
  const int v = std::atoi(e);
  return v < 1 ? 1 : (v > kJacobiMaxSweeps ? kJacobiMaxSweeps : v);
}

dmrg3s_status svd_jacobi(Context* c, std::vector<SvdLane>& lanes, int nlanes,
                         const std::vector<SvdJob>& jobs, double* A, double* S, double* VT,
                         double* U, int* info, cudaStream_t st, std::string* diag,
                         int* sweeps) {
  const int nj = (int)jobs.size();
  if (nj == 0) return DMRG3S_OK;
  if (nlanes < 1 || nlanes > (int)lanes.size()) nlanes = (int)lanes.size();
  if (nlanes < 1) return fail(c, DMRG3S_ERR_ARG, "no SVD lane");
  // ---- tables
  std::vector<JacJob> tab(nj);
  std::vector<JacPair> pairs;
  std::vector<int> col_job;
  int64_t ny = 0, nv = 0, ntau = 0;
  int maxr = 0;
  size_t smem = 0;
  for (int k = 0; k < nj; ++k) {
    const SvdJob& jb = jobs[k];
    if (jb.n < 1 || jb.m < jb.n || jb.m > (1 << 30) || jb.n > kJacobiMaxN)
      return fail(c, DMRG3S_ERR_ARG, "SVD matrix shape (need 1 <= n <= m, n <= 32768)");
    if (jb.offU >= 0 && !U) return fail(c, DMRG3S_ERR_ARG, "SVD left vectors without a buffer");
    JacJob& t = tab[k];
    t.offA = jb.offA;
    t.offY = ny;
    ny += jb.n * jb.n;
    t.offV = jb.offU >= 0 ? nv : -1;
    if (jb.offU >= 0) nv += jb.n * jb.n;
    t.offTau = ntau;
    ntau += jb.n;
    t.offS = jb.offS;
    t.offVT = jb.offVT;
    t.offU = jb.offU;
    t.m = (int32_t)jb.m;
    t.n = (int32_t)jb.n;
    t.col0 = (int32_t)col_job.size();
    t.pad = 0;
    col_job.insert(col_job.end(), t.n, k);
    const double tol = std::max(std::sqrt((double)t.n), 32.0) * DBL_EPSILON;
    const int nb = (t.n + kJacB - 1) / kJacB, nbpad = nb + (nb & 1);
    const size_t bytes = (size_t)2 * kJacB * t.n * sizeof(double) * (t.offV >= 0 ? 2 : 1);
    const bool staged = bytes <= kJacStage;
    if (staged) smem = std::max(smem, bytes);
    maxr = std::max(maxr, nbpad - 1);
    for (int q = 0; q < nbpad / 2; ++q)
      pairs.push_back(JacPair{t.offY, t.offV, t.n, t.col0, q, nbpad - 1, k, staged, (float)(tol * tol)});
  }
  const int ncta = (int)pairs.size(), ncol = (int)col_job.size();
  int64_t na = 0;   // extent of the A buffer used by the jobs
  for (const JacJob& t : tab) na = std::max(na, t.offA + (int64_t)t.m * t.n);
  std::vector<QrColumns> qcols;  // the left vectors' columns by CTA
  int umax = 0;                  // their longest
  for (int k = 0; k < nj; ++k)
    if (tab[k].offU >= 0) {
      for (int q = 0; q < tab[k].n; q += kQrApplyWarps) qcols.push_back(QrColumns{k, q});
      umax = std::max(umax, (int)tab[k].m);
    }
  QrPlan qr;
  std::vector<int> by_lib;       // matrices left to cuSOLVER's QR
  plan_qr(tab, plan_ctas(), &qr, &by_lib);
  // ---- device buffers: doubles [tau | Y | V1 | sigma | column norms | T = A P],
  //      ints [col_job | perm | rot | sweep | qinfo | QR flags | QR error | QR items | left columns]
  const int64_t nd = ntau + ny + nv + 2 * (int64_t)ncol + na;
  const int64_t ni = 2 * (int64_t)ncol + (int64_t)kJacobiMaxSweeps * nj + 1 + 2 * nj + 1 +
                     (int64_t)qr.cta_item.size() + 2 * (int64_t)qcols.size();
  double* dd = nullptr;
  int* di = nullptr;
  JacJob* dt = nullptr;
  JacPair* dp = nullptr;
  QrItem* dq = nullptr;
  dmrg3s_status s = DMRG3S_OK;
  if ((s = cuda_ok(c, cudaMallocAsync((void**)&dd, (size_t)nd * sizeof(double), st), "SVD buffers")) ||
      (s = cuda_ok(c, cudaMallocAsync((void**)&di, (size_t)ni * sizeof(int), st), "SVD buffers")) ||
      (s = cuda_ok(c, cudaMallocAsync((void**)&dt, tab.size() * sizeof(JacJob), st), "SVD buffers")) ||
      (s = cuda_ok(c, cudaMallocAsync((void**)&dp, pairs.size() * sizeof(JacPair), st), "SVD buffers")) ||
      (!qr.items.empty() &&
       (s = cuda_ok(c, cudaMallocAsync((void**)&dq, qr.items.size() * sizeof(QrItem), st), "SVD buffers"))) ||
      (s = cuda_ok(c, cudaFuncSetAttribute(qr_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)kQrSmem), "QR shared memory")) ||
      (s = cuda_ok(c, cudaFuncSetAttribute(jac_round_kernel,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)kJacStage), "Jacobi shared memory"))) {
    if (dd) cudaFreeAsync(dd, st);
    if (di) cudaFreeAsync(di, st);
    if (dt) cudaFreeAsync(dt, st);
    if (dp) cudaFreeAsync(dp, st);
    if (dq) cudaFreeAsync(dq, st);
    return s;
  }
  double* tau = dd;
  double* Y = tau + ntau;
  double* V1 = Y + ny;
  double* sig = V1 + nv;
  double* anrm = sig + ncol;
  double* T = anrm + ncol;
  int* d_col = di;
  int* d_perm = d_col + ncol;
  int* rot = d_perm + ncol;
  int* d_sweep = rot + (int64_t)kJacobiMaxSweeps * nj;
  int* qinfo = d_sweep + 1;
  int* qr_ready = qinfo + nj;
  int* qr_err = qr_ready + nj;
  int* qr_cta = qr_err + 1;
  QrColumns* d_qcols = reinterpret_cast<QrColumns*>(qr_cta + qr.cta_item.size());
  cudaMemcpyAsync(dt, tab.data(), tab.size() * sizeof(JacJob), cudaMemcpyHostToDevice, st);
  cudaMemcpyAsync(dp, pairs.data(), pairs.size() * sizeof(JacPair), cudaMemcpyHostToDevice, st);
  cudaMemcpyAsync(d_col, col_job.data(), col_job.size() * sizeof(int), cudaMemcpyHostToDevice, st);
  cudaMemsetAsync(qr_ready, 0, (size_t)(nj + 1) * sizeof(int), st);
  if (!qcols.empty())
    cudaMemcpyAsync(d_qcols, qcols.data(), qcols.size() * sizeof(QrColumns), cudaMemcpyHostToDevice, st);
  if (!qr.items.empty()) {
    cudaMemcpyAsync(dq, qr.items.data(), qr.items.size() * sizeof(QrItem), cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(qr_cta, qr.cta_item.data(), qr.cta_item.size() * sizeof(int), cudaMemcpyHostToDevice, st);
  }
  cudaMemsetAsync(rot, 0, (size_t)kJacobiMaxSweeps * nj * sizeof(int), st);
  cudaMemsetAsync(d_sweep, 0xff, sizeof(int), st);   // -1: the first sweep advances it to 0
  s = cuda_ok(c, cudaGetLastError(), "SVD tables");
  // ---- columns in descending norm order, T = A P: the Jacobi sweeps on R^T
  // of A P need fewer sweeps than on R^T of A when the column norms are graded
  std::vector<int> perm(ncol);
  if (!s) {
    std::vector<double> hn(ncol);
    launch_chain(jac_anorm_kernel, ncol, kJacThreads, 0, st, dt, d_col, A, anrm);
    count_launch();
    if (!(s = cuda_ok(c, cudaMemcpyAsync(hn.data(), anrm, ncol * sizeof(double),
                                         cudaMemcpyDeviceToHost, st), "column norms")) &&
        !(s = cuda_ok(c, cudaStreamSynchronize(st), "column norms"))) {
      for (const JacJob& t : tab) {
        int* pj = perm.data() + t.col0;
        for (int i = 0; i < t.n; ++i) pj[i] = i;
        const double* nj_ = hn.data() + t.col0;
        std::stable_sort(pj, pj + t.n, [&](int x, int y) { return nj_[x] > nj_[y]; });
      }
      cudaMemcpyAsync(d_perm, perm.data(), ncol * sizeof(int), cudaMemcpyHostToDevice, st);
      launch_chain(jac_permute_kernel, ncol, kJacThreads, 0, st, dt, d_col, d_perm, A, T);
      count_launch();
      s = cuda_ok(c, cudaGetLastError(), "column order");
    }
  }
  // ---- 1. A = Q R: qr_kernel, and cuSOLVER for the matrices too large for it.  A
  // stream with fewer SMs than the plan's CTAs (of a green context, say) refuses the
  // cooperative launch: then cuSOLVER factorises every matrix.
  if (!s && !qr.items.empty()) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeCooperative;
    at.val.cooperative = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = (unsigned)qr.cta_item.size() - 1;
    cfg.blockDim = kQrThreads;
    cfg.dynamicSmemBytes = qr.smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, qr_kernel, (const QrItem*)dq, (const int*)qr_cta, T, tau, qr_ready, qr_err,
                           c->wait_ns) == cudaSuccess) {
      count_launch();
    } else {
      cudaGetLastError();
      by_lib.resize(nj);
      for (int k = 0; k < nj; ++k) by_lib[k] = k;
    }
  }
  // ---- lanes for cuSOLVER's matrices, by the cost m n^2, largest first; created when
  // first used
  std::vector<int> order(by_lib);
  std::sort(order.begin(), order.end(), [&](int a, int b) {
    return (double)tab[a].m * tab[a].n * tab[a].n > (double)tab[b].m * tab[b].n * tab[b].n;
  });
  nlanes = std::min(nlanes, (int)order.size());
  std::vector<std::vector<int>> part(nlanes);
  std::vector<double> load(nlanes, 0.0);
  for (int k : order) {
    const int w = (int)(std::min_element(load.begin(), load.end()) - load.begin());
    part[w].push_back(k);
    load[w] += (double)tab[k].m * tab[k].n * tab[k].n + 1e5;
  }
  for (int w = 0; !s && w < nlanes; ++w) s = lane_ready(c, &lanes[w]);
  size_t dmax = 1, hmax = 1;
  for (int k : order) {
    if (s) break;
    const JacJob& t = tab[k];
    size_t wd = 0, wh = 0;
    if (cusolverDnXgeqrf_bufferSize(lanes[0].h, lanes[0].p, t.m, t.n, CUDA_R_64F, T + t.offA, t.m,
                                    CUDA_R_64F, tau + t.offTau, CUDA_R_64F, &wd,
                                    &wh) != CUSOLVER_STATUS_SUCCESS)
      s = fail(c, DMRG3S_ERR_CUDA, "QR buffer size");
    dmax = std::max(dmax, wd);
    hmax = std::max(hmax, wh);
  }
  for (int w = 0; !s && w < nlanes; ++w) {
    SvdLane& l = lanes[w];
    if (l.dbytes < dmax) {
      if (l.dwork) cudaFree(l.dwork);
      l.dwork = nullptr;
      l.dbytes = 0;
      if (cudaMalloc(&l.dwork, dmax) != cudaSuccess) {
        s = fail(c, DMRG3S_ERR_CUDA, "SVD workspace");
        break;
      }
      l.dbytes = dmax;
    }
    if (l.hwork.size() < hmax) l.hwork.resize(hmax);
  }
  cudaEvent_t ev_in = nullptr;
  if (!s && cudaEventCreateWithFlags(&ev_in, cudaEventDisableTiming) != cudaSuccess)
    s = fail(c, DMRG3S_ERR_CUDA, "SVD event");
  if (!s && nlanes > 0) {
    // on the lanes after the work queued on st, which waits for them
    cudaEventRecord(ev_in, st);
    std::vector<int> bad(nlanes, 0);
    auto run = [&](int w) {
      SvdLane& l = lanes[w];
      cudaSetDevice(c->device);
      cudaStreamWaitEvent(l.s, ev_in, 0);
      cusolverDnSetStream(l.h, l.s);
      for (int k : part[w]) {
        const JacJob& t = tab[k];
        if (cusolverDnXgeqrf(l.h, l.p, t.m, t.n, CUDA_R_64F, T + t.offA, t.m, CUDA_R_64F,
                             tau + t.offTau, CUDA_R_64F, l.dwork, l.dbytes, l.hwork.data(),
                             l.hwork.size(), qinfo + k) != CUSOLVER_STATUS_SUCCESS)
          bad[w] = 1;
      }
      cudaEventRecord(l.ev, l.s);
    };
    std::vector<std::thread> th;
    for (int w = 1; w < nlanes; ++w) th.emplace_back(run, w);
    run(0);
    for (auto& t : th) t.join();
    for (int w = 0; w < nlanes; ++w) {
      if (bad[w] && !s) s = fail(c, DMRG3S_ERR_CUDA, "QR factorisation");
      cudaStreamWaitEvent(st, lanes[w].ev, 0);
    }
  }
  // ---- 2. Y = R^T, V1 = I
  if (!s) {
    launch_chain(jac_init_kernel, ncol, kJacThreads, 0, st, dt, d_col, T, Y, V1);
    count_launch();
    s = cuda_ok(c, cudaGetLastError(), "Jacobi set-up");
  }
  // ---- 3. sweeps: one CUDA graph of (sweep counter, rounds 0 .. maxr-1)
  const PlainLaunches plain;
  cudaStream_t cap = nullptr;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t gexec = nullptr;
  if (!s && cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking) == cudaSuccess &&
      cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
    launch_chain(jac_sweep_kernel, ncol, kJacThreads, 0, cap, dt, d_col, Y, anrm, d_sweep);
    for (int r = 0; r < maxr; ++r)
      launch_chain(jac_round_kernel, ncta, 32 * kJacB, smem, cap, dp, nj, r, d_sweep, rot, anrm, Y, V1);
    if (cudaStreamEndCapture(cap, &graph) != cudaSuccess ||
        cudaGraphInstantiate(&gexec, graph, 0) != cudaSuccess)
      gexec = nullptr;
  }
  cudaGetLastError();   // a failed capture leaves the plain launches below
  std::vector<int> hrot(nj), active(nj, 1);
  int herr = 0;
  std::vector<int> conv(nj, 0);
  Profiler& pr = c->prof;
  const int max_sweeps = jacobi_max_sweeps();
  if (sweeps) *sweeps = 0;
  for (int sw = 0; !s && sw < max_sweeps; ++sw) {
    if (sweeps) *sweeps = sw + 1;
    const int id = pr.on ? pr.begin(kProfJacobi, 0.0, 0.0, st) : -1;
    if (gexec) {
      s = cuda_ok(c, cudaGraphLaunch(gexec, st), "Jacobi sweep");
    } else {
      launch_chain(jac_sweep_kernel, ncol, kJacThreads, 0, st, dt, d_col, Y, anrm, d_sweep);
      for (int r = 0; r < maxr; ++r)
        launch_chain(jac_round_kernel, ncta, 32 * kJacB, smem, st, dp, nj, r, d_sweep, rot, anrm, Y, V1);
      s = cuda_ok(c, cudaGetLastError(), "Jacobi sweep");
    }
    count_launch(maxr + 1);
    if (id >= 0) pr.end(id, st);
    if (s) break;
    if ((s = cuda_ok(c, cudaMemcpyAsync(hrot.data(), rot + (int64_t)sw * nj, nj * sizeof(int),
                                        cudaMemcpyDeviceToHost, st), "Jacobi rotations")) ||
        (sw == 0 && (s = cuda_ok(c, cudaMemcpyAsync(&herr, qr_err, sizeof(int), cudaMemcpyDeviceToHost,
                                                    st), "QR status"))) ||
        (s = cuda_ok(c, cudaStreamSynchronize(st), "Jacobi sweep")))
      break;
    if (herr) {
      s = fail(c, DMRG3S_ERR_TIMEOUT, "the QR factorisation gave up a bounded wait");
      break;
    }
    // algorithmic cost of the sweep: a pair test reads two columns (16n bytes)
    // for a dot product (2n flops); a rotation of a column pair of Y and
    // of V1 takes 6n flops each and writes 16n bytes each (V1 also read)
    double fl = 0.0, by = 0.0;
    bool more = false;
    for (int k = 0; k < nj; ++k) {
      if (!active[k]) continue;
      const double n = tab[k].n, pairs = 0.5 * n * (n - 1.0);
      const bool v = tab[k].offV >= 0;
      fl += pairs * 2.0 * n + hrot[k] * 6.0 * n * (v ? 2.0 : 1.0);
      by += pairs * 16.0 * n + hrot[k] * 16.0 * n * (v ? 3.0 : 1.0);
      if (hrot[k] == 0) {
        active[k] = 0;
        conv[k] = 1;
      } else {
        more = true;
      }
    }
    if (id >= 0) {
      pr.recs[id].flops = fl;
      pr.recs[id].bytes = by;
      pr.recs[id].launches = maxr + 1;
    }
    if (!more) break;
  }
  if (gexec) cudaGraphExecDestroy(gexec);
  if (graph) cudaGraphDestroy(graph);
  if (cap) cudaStreamDestroy(cap);
  // ---- 4. singular values in descending order, VT, (V1; 0) for the left vectors
  if (!s) {
    launch_chain(jac_norm_kernel, ncol, kJacThreads, 0, st, dt, d_col, Y, sig);
    launch_chain(jac_scatter_kernel, ncol, kJacThreads, 0, st, dt, d_col, d_perm, Y, V1, sig, S, VT, U);
    count_launch(2);
    s = cuda_ok(c, cudaGetLastError(), "singular vectors");
  }
  // ---- 5. U = Q (V1; 0)
  if (!s && !qcols.empty()) {
    const int stride = std::min(umax, kQrApplyRows);
    const size_t bytes = (size_t)kQrApplyWarps * stride * sizeof(double);
    // (the limit belongs to the kernel, not to the call: always the same value, or
    // another thread's smaller one could come between it and the launch)
    if (!(s = cuda_ok(c, cudaFuncSetAttribute(qr_apply_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)kQrApplySmem), "left vectors")))
      launch_chain(qr_apply_kernel, (int)qcols.size(), 32 * kQrApplyWarps, bytes, st, dt, d_qcols, T, tau, U,
                   stride);
    count_launch();
    if (!s) s = cuda_ok(c, cudaGetLastError(), "left vectors");
  }
  for (int k = 0; k < nj; ++k) {
    info[k] = conv[k] ? 0 : 1;
    if (!conv[k] && diag && diag->empty())
      *diag = "matrix " + std::to_string(k) + " (" + std::to_string(tab[k].m) + " x " +
              std::to_string(tab[k].n) + ") still had " + std::to_string(hrot[k]) +
              " rotations in sweep " + std::to_string(max_sweeps);
  }
  cudaFreeAsync(dd, st);
  cudaFreeAsync(di, st);
  cudaFreeAsync(dt, st);
  cudaFreeAsync(dp, st);
  if (dq) cudaFreeAsync(dq, st);
  if (ev_in) cudaEventDestroy(ev_in);
  return s;
}

}  // namespace dmrg3s

extern "C" dmrg3s_status dmrg3s_svd(dmrg3s_ctx ctx, int32_t nmat, const int64_t* m,
                                    const int64_t* n, double* A, double* S, double* VT, double* U,
                                    dmrg3s_stream stream) {
  using namespace dmrg3s;
  Context* c = reinterpret_cast<Context*>(ctx);
  if (!c) return DMRG3S_ERR_ARG;
  if (nmat < 0 || (nmat > 0 && (!m || !n || !A || !S || !VT)))
    return fail(c, DMRG3S_ERR_ARG, "dmrg3s_svd: null argument or negative count");
  if (nmat == 0) return DMRG3S_OK;
  dmrg3s_status s = use_device(c);
  if (s) return s;
  std::vector<SvdJob> jobs(nmat);
  int64_t oa = 0, os = 0, ov = 0;
  for (int k = 0; k < nmat; ++k) {
    if (n[k] < 1 || m[k] < n[k]) return fail(c, DMRG3S_ERR_ARG, "dmrg3s_svd: need 1 <= n <= m");
    jobs[k].m = m[k];
    jobs[k].n = n[k];
    jobs[k].offA = oa;
    jobs[k].offU = U ? oa : -1;
    jobs[k].offS = os;
    jobs[k].offVT = ov;
    oa += m[k] * n[k];
    os += n[k];
    ov += n[k] * n[k];
  }
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  std::vector<SvdLane> lanes(1);
  std::vector<int> info(nmat, 0);
  std::string diag;
  s = svd_jacobi(c, lanes, 1, jobs, A, S, VT, U, info.data(), st, &diag);
  if (!s && cudaStreamSynchronize(st) != cudaSuccess)
    s = fail(c, DMRG3S_ERR_CUDA, "dmrg3s_svd: stream synchronisation");
  lane_destroy(&lanes[0]);
  for (int k = 0; !s && k < nmat; ++k)
    if (info[k]) s = fail(c, DMRG3S_ERR_NOT_CONVERGED, "dmrg3s_svd: " + diag);
  return s;
}
