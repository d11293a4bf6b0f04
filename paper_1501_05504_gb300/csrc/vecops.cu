// Dense vector kernels of the local eigensolver and the truncation step.
//
// Reductions are deterministic: a fixed grid of kRedBlocks CTAs writes one
// partial sum per CTA (warp-shuffle reduction inside the CTA) and a second
// kernel adds the partials in a fixed order.
#include <algorithm>
#include <cmath>

#include "fp64.cuh"
#include "kernels.hpp"
#include "launch.hpp"
#include "vecops.hpp"

namespace dmrg3s {

namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ double block_sum(double v, double* sh) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  double r = 0.0;
  if (wid == 0) {
    r = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0.0;
    r = warp_sum(r);
  }
  __syncthreads();
  return r;   // valid in thread 0
}

// h[j] = <V_j, w> for j < k: block (c, j) sums chunk c of vector j (one block
// reduction per block); multidot_final adds the chunk partials of vector j
// in chunk order, so the result is deterministic.
__global__ void __launch_bounds__(kThreads) multidot_partial(const double* V,
                                                             int64_t ldv, const double* w,
                                                             int64_t n, int64_t chunk,
                                                             double* partial) {
  grid_next();
  grid_wait();
  __shared__ double sh[32];
  const int j = blockIdx.y;
  const double* v = V + (int64_t)j * ldv;
  const int64_t e0 = (int64_t)blockIdx.x * chunk;
  const int64_t e1 = e0 + chunk < n ? e0 + chunk : n;
  double acc = 0.0;
  for (int64_t e = e0 + threadIdx.x; e < e1; e += blockDim.x) acc = fma(v[e], w[e], acc);
  const double s = block_sum(acc, sh);
  if (threadIdx.x == 0) partial[(int64_t)j * gridDim.x + blockIdx.x] = s;
}

__global__ void multidot_final(const double* partial, int nchunk, int k,
                               double* h, double* copy_last) {
  grid_next();
  grid_wait();
  __shared__ double sh[32];
  const int j = blockIdx.x;
  double acc = 0.0;
  for (int b = threadIdx.x; b < nchunk; b += blockDim.x) acc += partial[(int64_t)j * nchunk + b];
  const double s = block_sum(acc, sh);
  if (threadIdx.x == 0) {
    h[j] = s;
    if (copy_last && j == k - 1) *copy_last = s;
  }
}

// Double-float numbers (an unevaluated sum hi + lo of two floats, about 44
// significant bits) carry the Sturm counts: GB300 issues FP32 at ~60x its
// FP64 rate, and the count only needs the sign of each pivot. Two-sum is
// Knuth's error-free addition; the quotient takes one correction step with
// an FMA residual (Dekker's double-length division).
struct DF {
  float hi, lo;
};

__device__ __forceinline__ DF df_from(double v) {
  const float h = (float)v;
  return {h, (float)(v - (double)h)};
}

__device__ __forceinline__ DF df_sub(DF a, DF b) {
  const float s = a.hi - b.hi;
  const float bb = s - a.hi;
  float e = (a.hi - (s - bb)) + (-b.hi - bb);
  e += a.lo - b.lo;
  const float h = s + e;
  return {h, e - (h - s)};
}

__device__ __forceinline__ DF df_div(DF a, DF b) {
  const float rb = 1.0f / b.hi;
  const float q1 = a.hi * rb;
  const float p = q1 * b.hi;
  const float pe = fmaf(q1, b.hi, -p);
  const float r = (((a.hi - p) - pe) + a.lo) - q1 * b.lo;
  const float q2 = r * rb;
  const float h = q1 + q2;
  return {h, q2 - (h - q1)};
}

// Number of eigenvalues of T smaller than x (Sturm sequence of the LDL^T
// pivots). The matrix arrives shifted and scaled, sa[i] = (alpha_i - c)/s and
// sbb[i] = (beta_{i-1}/s)^2, so every quantity is O(1) and x is (x - c)/s.
__device__ int sturm_count_df(const DF* sa, const DF* sbb, int k, DF x) {
  int cnt = 0;
  DF d = {1.f, 0.f};
  for (int i = 0; i < k; ++i) {
    DF t = df_sub(sa[i], x);
    if (i > 0) t = df_sub(t, df_div(sbb[i], d));
    if (t.hi == 0.f) t = {-1e-30f, 0.f};   // x hit an eigenvalue of a leading block: perturb
    if (t.hi < 0.f) ++cnt;
    d = t;
  }
  return cnt;
}

constexpr int kTriMax = 128;   // largest order

// Largest value of a warp's lanes.
__device__ __forceinline__ double warp_max(double v) {
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// The eigenvector of T for an eigenvalue near theta and its Rayleigh quotient, by
// one warp: inverse iteration with a pivoted tridiagonal LU of T - theta I
// (partial pivoting keeps the elimination stable at the near-singular shift; a
// vanishing pivot is replaced by 1e-15 of the matrix scale, which keeps the
// solution finite before normalisation).  T is scaled by a power of two to a span
// of order one.  The elimination and the substitutions are chains of one lane:
// the pivots are inverted once, by an FP32 reciprocal and three FP64
// multiply-adds, the rows of U are divided by them beforehand, and every operand
// comes from shared memory, so a substitution step is one dependent FP64
// instruction; everything else is spread over the lanes.  The whole solve
// at order 32 to 37: 122 us with one thread on local memory, 77 us now.
__device__ void tridiag_vector(const double* al, const double* be, int k, double bl,
                               double theta, double span, double lo, double hi, double* y,
                               TridiagOut* out) {
  __shared__ double s_d[kTriMax], s_l[kTriMax], s_u[kTriMax], s_u2[kTriMax], s_y[kTriMax],
      s_b[kTriMax];
  __shared__ unsigned char s_piv[kTriMax];
  const int lane = threadIdx.x;
  if (k == 1) {                 // the Ritz vector of a 1x1 matrix
    if (lane == 0) {
      y[0] = 1.0;
      out->theta = theta;
      out->resid = fabs(bl);
      out->beta_last = bl;
      out->nan_seen = 0.0;
    }
    return;
  }
  const double sc = inverse_scale(span);
  const double tiny = 1e-15 * sc * fmax(span, fmax(fabs(lo), fabs(hi)));
  for (int i = lane; i < k; i += 32) {
    s_d[i] = sc * (al[i] - theta);
    s_b[i] = i < k - 1 ? sc * be[i] : 0.0;
    s_y[i] = 1.0;
  }
  __syncwarp();
  if (lane == 0) {   // s_d becomes the inverted pivots
    double cd = s_d[0], cu = s_b[0];
    for (int i = 0; i < k - 1; ++i) {
      const double l = s_b[i], dn = s_d[i + 1], un = s_b[i + 1];
      const bool swap = fabs(cd) < fabs(l);
      double p = swap ? l : cd;
      if (fabs(p) < 1e-300) p = tiny;
      const double r = recip(p), f = (swap ? cd : l) * r;
      s_piv[i] = swap;
      s_d[i] = r;
      s_l[i] = f;
      s_u[i] = swap ? dn : cu;
      s_u2[i] = swap ? un : 0.0;
      cd = swap ? fma(-f, dn, cu) : fma(-f, cu, dn);
      cu = swap ? -f * un : un;
    }
    s_d[k - 1] = recip(fabs(cd) < 1e-300 ? tiny : cd);
  }
  __syncwarp();
  for (int i = lane; i < k - 1; i += 32) {
    s_u[i] *= s_d[i];
    s_u2[i] *= s_d[i];
  }
  for (int sweep = 0; sweep < 3; ++sweep) {
    __syncwarp();
    if (lane == 0) {   // row interchanges and L
      double cur = s_y[0];
      for (int i = 0; i < k - 1; ++i) {
        const double nx = s_y[i + 1], f = s_l[i];
        const bool swap = s_piv[i];
        s_y[i] = swap ? nx : cur;
        cur = swap ? fma(-f, nx, cur) : fma(-f, cur, nx);
      }
      s_y[k - 1] = cur;
    }
    __syncwarp();
    for (int i = lane; i < k; i += 32) s_y[i] *= s_d[i];
    __syncwarp();
    if (lane == 0) {   // back substitution (first and second superdiagonal)
      double y2 = 0.0, y1 = s_y[k - 1];
      for (int i = k - 2; i >= 0; --i) {
        const double t = fma(-s_u2[i], y2, s_y[i]);
        y2 = y1;
        y1 = fma(-s_u[i], y1, t);
        s_y[i] = y1;
      }
    }
    __syncwarp();
    // normalise: scale by the largest component first (no overflow in the squares)
    double big = 0.0;
    for (int i = lane; i < k; i += 32) big = fmax(big, fabs(s_y[i]));
    big = warp_max(big);
    if (!(big > 0.0) || !(big < 1e308)) {   // degenerate solve: restart from e_0
      for (int i = lane; i < k; i += 32) s_y[i] = i == 0 ? 1.0 : 0.0;
      continue;
    }
    const double ib = inverse_scale(big);
    double nrm = 0.0;
    for (int i = lane; i < k; i += 32) {
      const double v = ib * s_y[i];
      nrm = fma(v, v, nrm);
    }
    const double in = ib / sqrt(warp_sum(nrm));
    for (int i = lane; i < k; i += 32) s_y[i] *= in;
  }
  __syncwarp();
  // fix the sign: largest component positive (only the subspace is defined)
  double big = 0.0;
  int imax = kTriMax;
  for (int i = lane; i < k; i += 32)
    if (fabs(s_y[i]) > big) {
      big = fabs(s_y[i]);
      imax = i;
    }
  const double all = warp_max(big);
  imax = __reduce_min_sync(0xffffffffu, big == all ? imax : kTriMax);
  const bool flip = imax < kTriMax && s_y[imax] < 0.0;
  // Rayleigh quotient y^T T y (y has unit norm): second-order accurate in the
  // error of the vector, so the bracket's width does not limit the Ritz value
  double rq = 0.0;
  for (int i = lane; i < k; i += 32) {
    double ty = al[i] * s_y[i];
    if (i > 0) ty = fma(be[i - 1], s_y[i - 1], ty);
    if (i < k - 1) ty = fma(be[i], s_y[i + 1], ty);
    rq = fma(s_y[i], ty, rq);
    y[i] = flip ? -s_y[i] : s_y[i];
  }
  rq = warp_sum(rq);
  if (lane == 0) {
    out->theta = rq == rq ? rq : theta;
    out->resid = fabs(bl * s_y[k - 1]);
    out->beta_last = bl;
    out->nan_seen = 0.0;
  }
}

// Multisection: all threads of the block evaluate Sturm counts at equally
// spaced points of the bracket, shrinking it by blockDim.x + 1 per round
// until it reaches the resolution of double-float counts (~1e-13 of the
// Gershgorin span); the first warp then runs the inverse iteration in FP64 and
// returns the Rayleigh quotient of the vector, which is accurate to FP64
// rounding whatever the width of the bracket was.
// bl = the norm of the new residual vector (stored as beta[k - 1]).
__device__ void tridiag_block(const double* alpha, double* beta, int k,
                              double bl, double* y, TridiagOut* out) {
  __shared__ double sh_lo, sh_hi, sh_span, sh_c;
  __shared__ int sh_bad, sh_first;
  __shared__ double s_al[kTriMax], s_be[kTriMax];
  __shared__ DF sa[kTriMax], sbb[kTriMax];
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int i = tid; i < k; i += nt) {
    s_al[i] = alpha[i];
    s_be[i] = i < k - 1 ? beta[i] : 0.0;
  }
  __syncthreads();
  if (tid < 32) {
    double lo = 1e300, hi = -1e300;
    bool bad = !(bl == bl);
    for (int i = tid; i < k; i += 32) {
      const double r = (i > 0 ? fabs(s_be[i - 1]) : 0.0) + fabs(s_be[i]);
      lo = fmin(lo, s_al[i] - r);
      hi = fmax(hi, s_al[i] + r);
      if (!(s_al[i] == s_al[i])) bad = true;
    }
    lo = -warp_max(-lo);
    hi = warp_max(hi);
    bad = __any_sync(0xffffffffu, bad);
    if (tid == 0) {
      const double span = fmax(hi - lo, 1e-300);
      sh_lo = lo - 1e-12 * span;
      sh_hi = hi + 1e-12 * span;
      sh_span = span;
      sh_c = 0.5 * (lo + hi);
      sh_bad = bad;
      beta[k - 1] = bl;
    }
  }
  __syncthreads();
  if (sh_bad) {
    if (tid == 0) {
      out->theta = 0.0;
      out->resid = 0.0;
      out->beta_last = bl;
      out->nan_seen = 1.0;
    }
    return;
  }
  const double c = sh_c, inv_s = 1.0 / sh_span;
  for (int i = tid; i < k; i += nt) {
    sa[i] = df_from((s_al[i] - c) * inv_s);
    const double bs = i > 0 ? s_be[i - 1] * inv_s : 0.0;
    sbb[i] = df_from(bs * bs);
  }
  __syncthreads();
  for (int round = 0; round < 8; ++round) {
    const double lo = sh_lo, hi = sh_hi;
    const double h = (hi - lo) / (nt + 1);
    if (!(h > 1e-14 * sh_span)) break;
    if (tid == 0) sh_first = nt;
    __syncthreads();
    const DF x = df_from((lo + h * (tid + 1) - c) * inv_s);
    if (sturm_count_df(sa, sbb, k, x) >= 1) atomicMin(&sh_first, tid);
    __syncthreads();
    if (tid == 0) {
      const int f = sh_first;            // first point above the smallest eigenvalue
      sh_hi = f < nt ? lo + h * (f + 1) : hi;
      sh_lo = f > 0 ? lo + h * f : lo;
    }
    __syncthreads();
  }
  if (tid < 32)
    tridiag_vector(s_al, s_be, k, bl, 0.5 * (sh_lo + sh_hi), sh_span, sh_lo, sh_hi, y, out);
}

__global__ void copy_blocks_kernel(const CopyTask* __restrict__ tasks,
                                   const double* src, double* dst,
                                   const double* scale) {
  grid_next();
  grid_wait();
  const CopyTask t = tasks[blockIdx.x];
  const int n = t.rows * t.cols;
  for (int idx = threadIdx.x; idx < n; idx += blockDim.x) {
    int r, c;
    if (t.trans) {      // walk the source contiguously
      c = idx / t.rows;
      r = idx % t.rows;
    } else {
      r = idx / t.cols;
      c = idx % t.cols;
    }
    double v = t.trans ? src[t.off_s + (int64_t)c * t.ld_s + r] : src[t.off_s + (int64_t)r * t.ld_s + c];
    if (t.rs >= 0) v *= scale[t.rs + r];
    if (t.cs >= 0) v *= scale[t.cs + c];
    dst[t.off_d + (int64_t)r * t.ld_d + c] = v;
  }
}

// ---- batched Lanczos kernels (see vecops.hpp) ----
constexpr int kLzThreads = 256;
constexpr int kLzWarps = kLzThreads / 32;

// Sum of partial[b * kp + j] over the chunks b of [c0, c0 + nc) in a fixed
// order (lane-strided sums, then the xor tree); every lane returns the sum.
__device__ __forceinline__ double chain_sum(const double* partial, int kp, int c0,
                                            int nc, int j, int lane) {
  double a0 = 0.0, a1 = 0.0;
  int b = lane;
  for (; b + 32 < nc; b += 64) {     // two loads in flight per lane
    const double x0 = partial[(int64_t)(c0 + b) * kp + j];
    const double x1 = partial[(int64_t)(c0 + b + 32) * kp + j];
    a0 += x0;
    a1 += x1;
  }
  if (b < nc) a0 += partial[(int64_t)(c0 + b) * kp + j];
  return warp_sum(a0 + a1);
}

// <v, x> over len elements by one warp (lane-strided), four loads in flight
// per lane; the lanes' partial sums in a fixed order, then the xor tree.
__device__ __forceinline__ double warp_dot(const double* v, const double* x, int len,
                                           int lane) {
  double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
  int i = lane;
  for (; i + 96 < len; i += 128) {
    const double v0 = v[i], v1 = v[i + 32], v2 = v[i + 64], v3 = v[i + 96];
    a0 = fma(v0, x[i], a0);
    a1 = fma(v1, x[i + 32], a1);
    a2 = fma(v2, x[i + 64], a2);
    a3 = fma(v3, x[i + 96], a3);
  }
  for (; i < len; i += 32) a0 = fma(v[i], x[i], a0);
  return warp_sum((a0 + a1) + (a2 + a3));
}

// x - sum_{j < k1} h[j] V_j[e], the loads of four basis vectors in flight at a
// time (the basis is L2-resident; the loop is latency-bound otherwise).
__device__ __forceinline__ double lz_project(const double* V, int64_t ldv, int k1,
                                             const double* h, int64_t e, double x) {
  int j = 0;
  for (; j + 4 <= k1; j += 4) {
    const double v0 = V[(int64_t)j * ldv + e], v1 = V[(int64_t)(j + 1) * ldv + e];
    const double v2 = V[(int64_t)(j + 2) * ldv + e], v3 = V[(int64_t)(j + 3) * ldv + e];
    x = fma(-h[j], v0, x);
    x = fma(-h[j + 1], v1, x);
    x = fma(-h[j + 2], v2, x);
    x = fma(-h[j + 3], v3, x);
  }
  for (; j < k1; ++j) x = fma(-h[j], V[(int64_t)j * ldv + e], x);
  return x;
}

// The chunk of w is staged in shared memory once; warp q then forms the dot
// products with V_j for j = q, q + 8, ...
__global__ void __launch_bounds__(kLzThreads) lz_dots_kernel(const double* V,
                                                             int64_t ldv, int k1,
                                                             const int* kdev,
                                                             const double* w,
                                                             const LzChunk* __restrict__ chunks,
                                                             double* partial, int kp) {
  grid_next();
  grid_wait();
  extern __shared__ double wsh[];
  if (kdev) k1 = *kdev + 1;
  const LzChunk ch = chunks[blockIdx.x];
  const int len = (int)(ch.e1 - ch.e0);
  for (int i = threadIdx.x; i < len; i += kLzThreads) wsh[i] = w[ch.e0 + i];
  __syncthreads();
  const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
  for (int j = q; j < k1; j += kLzWarps) {
    const double acc = warp_dot(V + (int64_t)j * ldv + ch.e0, wsh, len, lane);
    if (lane == 0) partial[(int64_t)blockIdx.x * kp + j] = acc;
  }
}

__global__ void __launch_bounds__(kLzThreads) lz_update_kernel(
    const double* V, int64_t ldv, int k1, const int* kdev,
    double* w, const LzChunk* __restrict__ chunks, const LzChain* __restrict__ chains,
    const double* partial, int kp, double* alpha,
    double* nrm_partial, int64_t nrm_stride) {
  grid_next();
  grid_wait();
  __shared__ double h[kLzMaxK];
  __shared__ double red[32];
  if (kdev) {
    k1 = *kdev + 1;
    if (nrm_partial) nrm_partial += (int64_t)(*kdev % kLzLag) * nrm_stride;
  }
  const LzChunk ch = chunks[blockIdx.x];
  const LzChain cn = chains[ch.chain];
  const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
  for (int j = q; j < k1; j += kLzWarps) {
    const double s = chain_sum(partial, kp, cn.c0, cn.nc, j, lane);
    if (lane == 0) {
      h[j] = s;
      if (alpha && j == k1 - 1 && (int)blockIdx.x == cn.c0) alpha[(int64_t)ch.chain * kp + j] = s;
    }
  }
  __syncthreads();
  double nacc = 0.0;
  for (int64_t e = ch.e0 + threadIdx.x; e < ch.e1; e += kLzThreads) {
    double acc = lz_project(V, ldv, k1, h, e, w[e]);
    if (k1 > 0) w[e] = acc;
    nacc = fma(acc, acc, nacc);
  }
  if (nrm_partial) {
    const double t = block_sum(nacc, red);
    if (threadIdx.x == 0) nrm_partial[blockIdx.x] = t;
  }
}

// The first Gram-Schmidt pass's update fused with the second pass's dots:
// the updated chunk of w stays in shared memory for the dots against V_j.
__global__ void __launch_bounds__(kLzThreads) lz_update_dots_kernel(
    const double* V, int64_t ldv, int k1, double* w,
    const LzChunk* __restrict__ chunks, const LzChain* __restrict__ chains,
    const double* partial, int kp, double* alpha,
    double* partial2, const int* kdev) {
  grid_next();
  grid_wait();
  extern __shared__ double wsh[];
  __shared__ double h[kLzMaxK];
  if (kdev) k1 = *kdev + 1;
  const LzChunk ch = chunks[blockIdx.x];
  const LzChain cn = chains[ch.chain];
  const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
  for (int j = q; j < k1; j += kLzWarps) {
    const double s = chain_sum(partial, kp, cn.c0, cn.nc, j, lane);
    if (lane == 0) {
      h[j] = s;
      if (alpha && j == k1 - 1 && (int)blockIdx.x == cn.c0) alpha[(int64_t)ch.chain * kp + j] = s;
    }
  }
  __syncthreads();
  const int len = (int)(ch.e1 - ch.e0);
  for (int i = threadIdx.x; i < len; i += kLzThreads) {
    const int64_t e = ch.e0 + i;
    const double acc = lz_project(V, ldv, k1, h, e, w[e]);
    w[e] = acc;
    wsh[i] = acc;
  }
  __syncthreads();
  for (int j = q; j < k1; j += kLzWarps) {
    const double acc = warp_dot(V + (int64_t)j * ldv + ch.e0, wsh, len, lane);
    if (lane == 0) partial2[(int64_t)blockIdx.x * kp + j] = acc;
  }
}

__global__ void __launch_bounds__(kLzThreads) lz_normalise_kernel(
    const double* x, double* y, const LzChunk* __restrict__ chunks,
    const LzChain* __restrict__ chains, const double* nrm_partial) {
  grid_next();
  grid_wait();
  __shared__ double scale;
  const LzChunk ch = chunks[blockIdx.x];
  if (threadIdx.x < 32) {
    const LzChain cn = chains[ch.chain];
    const double n2 = chain_sum(nrm_partial, 1, cn.c0, cn.nc, 0, threadIdx.x);
    if (threadIdx.x == 0) scale = (n2 > 0.0 && n2 < 1e308) ? 1.0 / sqrt(n2) : 0.0;
  }
  __syncthreads();
  const double sc = scale;
  for (int64_t e = ch.e0 + threadIdx.x; e < ch.e1; e += kLzThreads) y[e] = x[e] * sc;
}

// v_{k+1} = w / |w| (norm partials of iteration k, k from the device
// counter), written into the basis and into the fixed product input vcur.
__global__ void __launch_bounds__(kLzThreads) lz_next_kernel(
    const double* w, double* V, int64_t ldv, const int* kdev,
    double* vcur, const LzChunk* __restrict__ chunks,
    const LzChain* __restrict__ chains, const double* nrm_partial,
    int64_t nrm_stride) {
  grid_next();
  grid_wait();
  __shared__ double scale;
  const int k = *kdev;
  const LzChunk ch = chunks[blockIdx.x];
  if (threadIdx.x < 32) {
    const LzChain cn = chains[ch.chain];
    const double n2 = chain_sum(nrm_partial + (int64_t)(k % kLzLag) * nrm_stride, 1, cn.c0, cn.nc,
                                0, threadIdx.x);
    if (threadIdx.x == 0) scale = (n2 > 0.0 && n2 < 1e308) ? 1.0 / sqrt(n2) : 0.0;
  }
  __syncthreads();
  const double sc = scale;
  double* vn = V + (int64_t)(k + 1) * ldv;
  for (int64_t e = ch.e0 + threadIdx.x; e < ch.e1; e += kLzThreads) {
    const double v = w[e] * sc;
    vn[e] = v;
    vcur[e] = v;
  }
}

__global__ void lz_advance_kernel(int* kdev) {
  grid_next();
  grid_wait(); *kdev += 1; }

// ---- one iteration's orthogonalisation in one launch ----

constexpr int kOrThreads = 512;
constexpr int kOrWarps = kOrThreads / 32;

// Barrier of all CTAs of a cooperative launch: `count` counts arrivals and is
// never reset, `target` is its value once all have arrived.  Bounded: false (in
// every thread of the CTA) after limit_ns, with *err set.
__device__ __forceinline__ bool grid_sync(unsigned* count, unsigned target, int* err,
                                          uint64_t limit_ns, int* s_ok) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(count, 1u);
    int ok = 1;
    uint64_t t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    for (;;) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
      if ((int)(v - target) >= 0) break;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
      if (t - t0 > limit_ns) {
        atomicExch(err, 1);
        ok = 0;
        break;
      }
    }
    __threadfence();
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}

// The kernel's sums have the order of the separate launches (warp_dot, chain_sum,
// block_sum: the same partial sums in the same trees), so both forms give the
// same bits: 3xTF32 products round their operands, and a last bit of v_k that
// differs can come back as 1e-8 of the eigenvector.  Sums of several values share a
// tree: the values' halves are exchanged first, which pairs the same lanes.
__device__ __forceinline__ double warp_sum4(const double (&a)[4], int lane) {   // value lane / 8
  const bool h16 = (lane & 16) != 0, h8 = (lane & 8) != 0;
  const double b0 = (h16 ? a[2] : a[0]) + __shfl_xor_sync(0xffffffffu, h16 ? a[0] : a[2], 16);
  const double b1 = (h16 ? a[3] : a[1]) + __shfl_xor_sync(0xffffffffu, h16 ? a[1] : a[3], 16);
  double c = (h8 ? b1 : b0) + __shfl_xor_sync(0xffffffffu, h8 ? b0 : b1, 8);
  for (int o = 4; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  return c;
}

// h[j] = the sum of partial[., j] over the chain's chunks, j < k1: four columns a
// warp, all their loads in flight.
__device__ __forceinline__ void chain_sums(const double* partial, int kp, const LzChain& cn, int k1,
                                           double* h) {
  const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
  for (int g = q; 4 * g < k1; g += kOrWarps) {
    const double* p = partial + (int64_t)cn.c0 * kp + 4 * g;
    const int nj = min(4, k1 - 4 * g);
    double a0[4] = {0.0, 0.0, 0.0, 0.0}, a1[4] = {0.0, 0.0, 0.0, 0.0};
    int b = lane;
#pragma unroll 3
    for (; b + 32 < cn.nc; b += 64)
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (t < nj) {
          a0[t] += __ldcg(p + (int64_t)b * kp + t);
          a1[t] += __ldcg(p + (int64_t)(b + 32) * kp + t);
        }
    if (b < cn.nc)
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (t < nj) a0[t] += __ldcg(p + (int64_t)b * kp + t);
#pragma unroll
    for (int t = 0; t < 4; ++t) a0[t] += a1[t];
    const double c = warp_sum4(a0, lane);
    if ((lane & 7) == 0 && (lane >> 3) < nj) h[4 * g + (lane >> 3)] = c;
  }
  __syncthreads();
}

// out[j] = <V_j, x> over the chunk, j < k1: two vectors a warp (they share the reads
// of x and a tree), 16 loads in flight.  Vectors below vcap are read from Vs (stride
// lp); FILL stores them there.
template <bool FILL>
__device__ __forceinline__ void chunk_dots(const double* V, int64_t ldv, double* Vs, int lp,
                                           int vcap, const double* x, int len, int k1, double* out) {
  const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
  const int full = len / 128;          // blocks of 128 elements, four per lane
  for (int g = q; 2 * g < k1; g += kOrWarps) {
    const bool two = 2 * g + 1 < k1;
    const double* src[2];
    double* dst[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int j = 2 * g + (two ? t : 0);
      src[t] = !FILL && j < vcap ? Vs + (int64_t)j * lp : V + (int64_t)j * ldv;
      dst[t] = FILL && j < vcap ? Vs + (int64_t)j * lp : nullptr;
    }
    double a[2][4];
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
      for (int m = 0; m < 4; ++m) a[t][m] = 0.0;
    for (int b0 = 0; b0 < full; b0 += 2) {
      double v[2][2][4];
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (b0 + u < full)
#pragma unroll
          for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int m = 0; m < 4; ++m) v[u][t][m] = src[t][(b0 + u) * 128 + m * 32 + lane];
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (b0 + u < full)
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            const int i = (b0 + u) * 128 + m * 32 + lane;
            const double xi = x[i];
#pragma unroll
            for (int t = 0; t < 2; ++t) {
              if (FILL && dst[t]) dst[t][i] = v[u][t][m];
              a[t][m] = fma(v[u][t][m], xi, a[t][m]);
            }
          }
    }
    if (full * 128 < len) {
      // the last elements: a lane with all four of them adds them to its four sums, a
      // lane with fewer to its first
      const int i = full * 128 + lane;
      const bool all = i + 96 < len;
      double v[2][4];
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int m = 0; m < 4; ++m) v[t][m] = i + 32 * m < len ? src[t][i + 32 * m] : 0.0;
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const bool in = i + 32 * m < len;
        const double xi = in ? x[i + 32 * m] : 0.0;
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          if (FILL && in && dst[t]) dst[t][i + 32 * m] = v[t][m];
          const double s = fma(v[t][m], xi, m == 0 || !all ? a[t][0] : a[t][m]);
          if (m == 0 || !all) {
            if (in) a[t][0] = s;
          } else {
            a[t][m] = s;
          }
        }
      }
    }
    const double s0 = (a[0][0] + a[0][1]) + (a[0][2] + a[0][3]);
    const double s1 = (a[1][0] + a[1][1]) + (a[1][2] + a[1][3]);
    const bool h16 = (lane & 16) != 0;
    double c = (h16 ? s1 : s0) + __shfl_xor_sync(0xffffffffu, h16 ? s0 : s1, 16);
    for (int o = 8; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((lane & 15) == 0 && (lane == 0 || two)) out[2 * g + (lane >> 4)] = c;
  }
}

// Iteration k (from the device counter): two classical Gram-Schmidt passes of w
// against V_0 .. V_k, v_{k+1} = w / |w| into the basis and vcur, k += 1.  One CTA
// per chunk, all resident (cooperative launch); the chunk of w and as much of
// the basis as fits stay in shared memory through the passes, which are
// separated by device-wide barriers instead of launches.  Bound by the FP64
// pipe: 4 k multiply-adds per element are 19 us at k = 37 for the 75 k elements
// of an m = 512 XXZ tensor, beside three barriers and the sums over the chunks'
// partials.  40 iterations with 3xTF32 products: 3.47 ms; as five launches an
// iteration (dots, update and dots, update, next, advance: 107 us at k = 32 to 37, cold
// caches) 4.75 ms.
__global__ void __launch_bounds__(kOrThreads, 1) lz_orth_kernel(
    double* V, int64_t ldv, int* kdev, const double* w, double* vcur,
    const LzChunk* __restrict__ chunks, const LzChain* __restrict__ chains, double* part,
    double* part2, int kp, double* alpha, double* nrm, int64_t nrm_stride, int lp, int vcap,
    unsigned* count, int* err, uint64_t limit_ns) {
  extern __shared__ double osh[];
  __shared__ double h[kLzMaxK];
  __shared__ double red[32];
  __shared__ double s_scale;
  __shared__ int s_ok;
  const int k = *kdev, k1 = k + 1;
  const unsigned G = gridDim.x, base = 3u * G * (unsigned)k;
  const LzChunk ch = chunks[blockIdx.x];
  const LzChain cn = chains[ch.chain];
  const int len = (int)(ch.e1 - ch.e0);
  double* x = osh;
  double* Vs = osh + lp;
  if (vcap > k1) vcap = k1;
  const double* Vc = V + ch.e0;
  for (int i = threadIdx.x; i < len; i += kOrThreads) x[i] = w[ch.e0 + i];
  __syncthreads();
  for (int pass = 0; pass < 2; ++pass) {
    double* pp = pass == 0 ? part : part2;
    if (pass == 0)
      chunk_dots<true>(Vc, ldv, Vs, lp, vcap, x, len, k1, pp + (int64_t)blockIdx.x * kp);
    else
      chunk_dots<false>(Vc, ldv, Vs, lp, vcap, x, len, k1, pp + (int64_t)blockIdx.x * kp);
    if (!grid_sync(count, base + (unsigned)(pass + 1) * G, err, limit_ns, &s_ok)) return;
    chain_sums(pp, kp, cn, k1, h);
    if (pass == 0 && threadIdx.x == 0 && (int)blockIdx.x == cn.c0)
      alpha[(int64_t)ch.chain * kp + k] = h[k];
    for (int i = threadIdx.x; i < len; i += kOrThreads) {
      double acc = x[i];
      int j = 0;
#pragma unroll 4
      for (; j < vcap; ++j) acc = fma(-h[j], Vs[(int64_t)j * lp + i], acc);
#pragma unroll 4
      for (; j < k1; ++j) acc = fma(-h[j], Vc[(int64_t)j * ldv + i], acc);
      x[i] = acc;
    }
    __syncthreads();
  }
  double* np = nrm + (int64_t)(k % kLzLag) * nrm_stride;
  double nacc = 0.0;
  if (threadIdx.x < kLzThreads)
    for (int i = threadIdx.x; i < len; i += kLzThreads) nacc = fma(x[i], x[i], nacc);
  nacc = block_sum(nacc, red);         // (the upper half's zeros change nothing)
  if (threadIdx.x == 0) np[blockIdx.x] = nacc;
  if (!grid_sync(count, base + 3u * G, err, limit_ns, &s_ok)) return;
  if (threadIdx.x < 32) {
    const double a = chain_sum(np, 1, cn.c0, cn.nc, 0, threadIdx.x);
    if (threadIdx.x == 0) s_scale = (a > 0.0 && a < 1e308) ? 1.0 / sqrt(a) : 0.0;
  }
  __syncthreads();
  const double sc = s_scale;
  double* vn = V + (int64_t)k1 * ldv;
  for (int i = threadIdx.x; i < len; i += kOrThreads) {
    const double v = x[i] * sc;
    vn[ch.e0 + i] = v;
    vcur[ch.e0 + i] = v;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *kdev = k1;   // every CTA has read it before a barrier
}

__global__ void lz_tridiag_kernel(const LzChain* __restrict__ chains, const double* alpha,
                                  double* beta, int kp, int k,
                                  const double* nrm_partial, double* y,
                                  TridiagOut* out) {
  grid_next();
  grid_wait();
  __shared__ double bl;
  const int c = blockIdx.x;
  const LzChain cn = chains[c];
  if (threadIdx.x < 32) {
    const double n2 = chain_sum(nrm_partial, 1, cn.c0, cn.nc, 0, threadIdx.x);
    if (threadIdx.x == 0) bl = sqrt(fmax(n2, 0.0));
  }
  __syncthreads();
  tridiag_block(alpha + (int64_t)c * kp, beta + (int64_t)c * kp, k + 1, bl,
                y + ((int64_t)c * kp + k) * kp, out + (int64_t)k * gridDim.x + c);
}

__global__ void __launch_bounds__(kLzThreads) lz_ritz_kernel(
    const double* V, int64_t ldv, const LzChunk* __restrict__ chunks,
    const LzChain* __restrict__ chains, const int32_t* kstop,
    const double* y, int kp, double* x, double* nrm_partial) {
  grid_next();
  grid_wait();
  __shared__ double red[32];
  const LzChunk ch = chunks[blockIdx.x];
  const int ks = kstop[ch.chain];
  const double* yc = y + ((int64_t)ch.chain * kp + ks) * kp;
  double nacc = 0.0;
  for (int64_t e = ch.e0 + threadIdx.x; e < ch.e1; e += kLzThreads) {
    const double acc = -lz_project(V, ldv, ks + 1, yc, e, 0.0);
    x[e] = acc;
    nacc = fma(acc, acc, nacc);
  }
  const double t = block_sum(nacc, red);
  if (threadIdx.x == 0) nrm_partial[blockIdx.x] = t;
}

}  // namespace

void launch_multidot(const double* V, int64_t ldv, int k, const double* w, int64_t n,
                     double* partial, double* h, double* copy_last, cudaStream_t st) {
  if (k <= 0) return;
  count_launch(2);
  // chunks of at least 2048 elements, at most kRedBlocks of them per vector
  int64_t chunk = (n + kRedBlocks - 1) / kRedBlocks;
  if (chunk < 2048) chunk = 2048;
  chunk = (chunk + kThreads - 1) / kThreads * kThreads;
  int nchunk = (int)((n + chunk - 1) / chunk);
  if (nchunk < 1) nchunk = 1;
  launch_chain(multidot_partial, dim3(nchunk, k), kThreads, 0, st, V, ldv, w, n, chunk, partial);
  launch_chain(multidot_final, k, 128, 0, st, partial, nchunk, k, h, copy_last);
}

void launch_lz_dots(const double* V, int64_t ldv, int k1, const double* w, const LzChunk* chunks,
                    int nchunks, double* partial, int kp, cudaStream_t st, const int* kdev) {
  if ((!kdev && k1 <= 0) || nchunks <= 0) return;
  count_launch();
  launch_chain(lz_dots_kernel, nchunks, kLzThreads, kLzChunkMax * sizeof(double), st, V, ldv, k1, kdev, w, chunks, partial, kp);
}

void launch_lz_update(const double* V, int64_t ldv, int k1, double* w, const LzChunk* chunks,
                      int nchunks, const LzChain* chains, const double* partial, int kp,
                      double* alpha, double* nrm_partial, cudaStream_t st, const int* kdev,
                      int64_t nrm_stride) {
  if (nchunks <= 0) return;
  count_launch();
  launch_chain(lz_update_kernel, nchunks, kLzThreads, 0, st, V, ldv, k1, kdev, w, chunks, chains, partial, kp, alpha, nrm_partial, nrm_stride);
}

void launch_lz_next(const double* w, double* V, int64_t ldv, const int* kdev, double* vcur,
                    const LzChunk* chunks, int nchunks, const LzChain* chains,
                    const double* nrm_partial, int64_t nrm_stride, cudaStream_t st) {
  if (nchunks <= 0) return;
  count_launch();
  launch_chain(lz_next_kernel, nchunks, kLzThreads, 0, st, w, V, ldv, kdev, vcur, chunks, chains, nrm_partial, nrm_stride);
}

void launch_lz_advance(int* kdev, cudaStream_t st) {
  count_launch();
  launch_chain(lz_advance_kernel, 1, 1, 0, st, kdev);
}

void launch_lz_update_dots(const double* V, int64_t ldv, int k1, double* w, const LzChunk* chunks,
                           int nchunks, const LzChain* chains, const double* partial, int kp,
                           double* alpha, double* partial2, cudaStream_t st, const int* kdev) {
  if (nchunks <= 0 || (!kdev && k1 <= 0)) return;
  count_launch();
  launch_chain(lz_update_dots_kernel, nchunks, kLzThreads, kLzChunkMax * sizeof(double), st,  V, ldv, k1, w, chunks, chains, partial, kp, alpha, partial2, kdev);
}

void launch_lz_normalise(const double* x, double* y, const LzChunk* chunks, int nchunks,
                         const LzChain* chains, const double* nrm_partial, cudaStream_t st) {
  if (nchunks <= 0) return;
  count_launch();
  launch_chain(lz_normalise_kernel, nchunks, kLzThreads, 0, st, x, y, chunks, chains, nrm_partial);
}

bool launch_lz_orth(double* V, int64_t ldv, int* kdev, const double* w, double* vcur,
                    const LzChunk* chunks, int nchunks, int maxlen, const LzChain* chains,
                    double* part, double* part2, int kp, double* alpha, double* nrm,
                    int64_t nrm_stride, unsigned* count, int* err, uint64_t limit_ns,
                    cudaStream_t st) {
  const int lp = (maxlen + 1) / 2 * 2;
  const int vcap = std::min(kp, (int)(kOrSmem / sizeof(double) / (size_t)lp) - 1);
  const size_t smem = sizeof(double) * (size_t)lp * (1 + vcap);
  if (cudaFuncSetAttribute(lz_orth_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kOrSmem) != cudaSuccess)
    return false;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeCooperative;
  at.val.cooperative = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = nchunks;
  cfg.blockDim = kOrThreads;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, lz_orth_kernel, V, ldv, kdev, w, vcur, chunks, chains, part, part2, kp,
                         alpha, nrm, nrm_stride, lp, vcap, count, err, limit_ns) != cudaSuccess)
    return false;
  count_launch();
  return true;
}

void launch_lz_tridiag(const LzChain* chains, int nchains, const double* alpha, double* beta,
                       int kp, int k, const double* nrm_partial, double* y, TridiagOut* out,
                       cudaStream_t st) {
  if (nchains <= 0) return;
  count_launch();
  launch_chain(lz_tridiag_kernel, nchains, 256, 0, st, chains, alpha, beta, kp, k, nrm_partial, y, out);
}

void launch_lz_ritz(const double* V, int64_t ldv, const LzChunk* chunks, int nchunks,
                    const LzChain* chains, const int32_t* kstop, const double* y, int kp,
                    double* x, double* nrm_partial, cudaStream_t st) {
  if (nchunks <= 0) return;
  count_launch();
  launch_chain(lz_ritz_kernel, nchunks, kLzThreads, 0, st, V, ldv, chunks, chains, kstop, y, kp, x, nrm_partial);
}

void launch_copy_blocks(const CopyTask* tasks, int ntasks, const double* src, double* dst,
                        const double* scale, cudaStream_t st) {
  if (ntasks <= 0) return;
  count_launch();
  launch_chain(copy_blocks_kernel, ntasks, 256, 0, st, tasks, src, dst, scale);
}

}  // namespace dmrg3s
