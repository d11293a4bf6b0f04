// FP64 kernels of the block-sparse contraction (CUDA cores).
//
// The grouped GEMM computes every block product of one contraction step of
// the order (((L M) W) R) of Sec. V of arXiv:1501.05504 in one launch: one CTA
// per output tile, summing all K-segments of its task.  The
// combination kernel applies the MPO step (T2 = sum W T1), which costs
// O(m^2 d^2 w^2) and is bound by memory bandwidth.
#include <atomic>

#include "kernels.hpp"
#include "launch.hpp"

namespace dmrg3s {

namespace {

constexpr int NT = 256;
constexpr int kGemmSmem = 2 * 16 * 65;   // doubles: the chunks of A and B of a 64 x 64 tile

// One SIZE x SIZE output tile: every thread sums R x R elements over the k of its
// K-group (SIZE = 8: four groups of 64 threads, their sums added at the end).
// Bound by the FP64 pipe (a warp's multiply-add takes ~64 cycles of a
// sub-partition), so the work is what counts: rows and k beyond the block are
// left out of the loops, and the next chunk's loads are in flight during the
// current one's products.
template <int SIZE, Trans TA, Trans TB>
__device__ __forceinline__ void gemm_tile(const GemmTile& tile, const GemmTask& task,
                                          const GemmSeg* __restrict__ segs, const double* A,
                                          const double* B, double* C, double* sh) {
  constexpr int KS = SIZE == 8 ? 4 : 1;                  // K-groups
  constexpr int TX = SIZE == 8 ? 8 : 16, R = SIZE / TX;  // threads a side, elements a thread and side
  constexpr int BK = SIZE == 8 ? 64 : SIZE == 16 ? 32 : 16;
  constexpr int LD = SIZE + 1, E = SIZE * BK / NT;       // elements of a chunk a thread loads
  static_assert(2 * BK * LD <= kGemmSmem, "shared memory");
  double* As = sh;
  double* Bs = sh + BK * LD;
  const int tid = threadIdx.x;
  const int grp = KS == 1 ? 0 : tid / (TX * TX), t = KS == 1 ? tid : tid % (TX * TX);
  const int tx = t % TX, ty = t / TX;
  const int m0 = tile.tm * SIZE, n0 = tile.tn * SIZE;
  double acc[R][R];
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int j = 0; j < R; ++j) acc[i][j] = 0.0;
  double ra[E], rb[E];
  int sgi = 0, k0 = 0;
  GemmSeg sg{};
  if (task.nseg > 0) sg = segs[task.seg0];
  while (sgi < task.nseg && sg.K <= 0)
    if (++sgi < task.nseg) sg = segs[task.seg0 + sgi];
  // the loads of chunk k0 of segment sg
  auto load = [&]() {
    const double* Ap = A + sg.offA;
    const double* Bp = B + sg.offB;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int idx = tid + e * NT;
      const int m = TA == Trans::N ? idx / BK : idx % SIZE, ka = TA == Trans::N ? idx % BK : idx / SIZE;
      const int gm = m0 + m, gk = k0 + ka;
      ra[e] = gm < task.M && gk < sg.K
                  ? (TA == Trans::N ? Ap[(int64_t)gm * sg.lda + gk] : Ap[(int64_t)gk * sg.lda + gm])
                  : 0.0;
      const int n = TB == Trans::N ? idx % SIZE : idx / BK, kb = TB == Trans::N ? idx / SIZE : idx % BK;
      const int gn = n0 + n, gb = k0 + kb;
      rb[e] = gn < task.N && gb < sg.K
                  ? (TB == Trans::N ? Bp[(int64_t)gb * sg.ldb + gn] : Bp[(int64_t)gn * sg.ldb + gb])
                  : 0.0;
    }
  };
  if (sgi < task.nseg) load();
  while (sgi < task.nseg) {
    const int kc = min(BK, sg.K - k0);
    if (sg.scale != 1.0) {
#pragma unroll
      for (int e = 0; e < E; ++e) ra[e] *= sg.scale;
    }
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int idx = tid + e * NT;
      As[TA == Trans::N ? (idx % BK) * LD + idx / BK : (idx / SIZE) * LD + idx % SIZE] = ra[e];
      Bs[TB == Trans::N ? (idx / SIZE) * LD + idx % SIZE : (idx % BK) * LD + idx / BK] = rb[e];
    }
    __syncthreads();
    k0 += BK;
    while (sgi < task.nseg && k0 >= sg.K) {
      k0 = 0;
      if (++sgi < task.nseg) sg = segs[task.seg0 + sgi];
    }
    if (sgi < task.nseg) load();
    const int kq = KS == 1 ? kc : (kc + KS - 1) / KS;
    const int kend = min(kc, (grp + 1) * kq);
    if (m0 + ty < task.M) {
#pragma unroll 4
      for (int k = grp * kq; k < kend; ++k) {
        double a[R], b[R];
#pragma unroll
        for (int i = 0; i < R; ++i) a[i] = As[k * LD + ty + TX * i];
#pragma unroll
        for (int j = 0; j < R; ++j) b[j] = Bs[k * LD + tx + TX * j];
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
          for (int j = 0; j < R; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
      }
    }
    __syncthreads();
  }
  if (KS > 1) {
    sh[tid] = acc[0][0];
    __syncthreads();
    if (grp > 0) return;
    double s = sh[t];
#pragma unroll
    for (int g = 1; g < KS; ++g) s += sh[g * TX * TX + t];
    acc[0][0] = s;
  }
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int gm = m0 + ty + TX * i;
    if (gm >= task.M) continue;
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int gn = n0 + tx + TX * j;
      if (gn < task.N) C[task.offC + (int64_t)gm * task.ldc + gn] = acc[i][j];
    }
  }
}

template <Trans TA, Trans TB>
__global__ void __launch_bounds__(NT) gemm_f64_kernel(const GemmTile* __restrict__ tiles,
                                                      const GemmTask* __restrict__ tasks,
                                                      const GemmSeg* __restrict__ segs,
                                                      const double* A,
                                                      const double* B,
                                                      double* C) {
  grid_next();
  grid_wait();
  __shared__ double sh[kGemmSmem];
  const GemmTile tile = tiles[blockIdx.x];
  const GemmTask task = tasks[tile.task];
  if (tile.size == 8) gemm_tile<8, TA, TB>(tile, task, segs, A, B, C, sh);
  else if (tile.size == 16) gemm_tile<16, TA, TB>(tile, task, segs, A, B, C, sh);
  else if (tile.size == 32) gemm_tile<32, TA, TB>(tile, task, segs, A, B, C, sh);
  else gemm_tile<64, TA, TB>(tile, task, segs, A, B, C, sh);
}

__global__ void __launch_bounds__(256) combine_f64_kernel(const CombChunk* __restrict__ chunks,
                                                         const CombTask* __restrict__ tasks,
                                                         const CombTerm* __restrict__ terms,
                                                         const double* in,
                                                         double* out,
                                                         double scale) {
  grid_next();
  grid_wait();
  const CombChunk ch = chunks[blockIdx.x];
  const CombTask t = tasks[ch.task];
  const int n = ch.nrows * t.cols;
  for (int idx = threadIdx.x; idx < n; idx += blockDim.x) {
    const int r = ch.row0 + idx / t.cols, c = idx % t.cols;
    double acc = 0.0;
    for (int k = 0; k < t.nt; ++k) {
      const CombTerm tm = terms[t.t0 + k];
      acc = fma(tm.coef, in[tm.offIn + (int64_t)r * tm.ldi + c], acc);
    }
    out[t.offOut + (int64_t)r * t.ldo + c] = scale * acc;
  }
}

// ---- double-float combinations (inputs: tensor-core output pairs) ----
// Knuth's two-sum and an FMA-based product keep ~48 bits; all on the FP32
// pipe (the intrinsics also keep the compiler from contracting the sums).
__device__ __forceinline__ void df_acc(float ch, float cl, float2 x, float& ah, float& al) {
  const float p = __fmul_rn(ch, x.x);
  float pe = __fmaf_rn(ch, x.x, -p);
  pe = __fmaf_rn(ch, x.y, pe);
  pe = __fmaf_rn(cl, x.x, pe);
  const float s = __fadd_rn(ah, p);
  const float bb = __fsub_rn(s, ah);
  float e = __fadd_rn(__fsub_rn(ah, __fsub_rn(s, bb)), __fsub_rn(p, bb));
  e = __fadd_rn(e, __fadd_rn(al, pe));
  ah = __fadd_rn(s, e);
  al = __fsub_rn(e, __fsub_rn(ah, s));
}

// sum_k coef_k in_k for output element (r, c) of a chunk's task, as a pair
__device__ __forceinline__ void df_combine(const CombTask& t, const CombTerm* __restrict__ terms,
                                           const float2* in, int r, int c, float sh,
                                           float sl, float& ah, float& al) {
  ah = 0.f;
  al = 0.f;
  for (int k = 0; k < t.nt; ++k) {
    const CombTerm tm = terms[t.t0 + k];
    df_acc(tm.chi, tm.clo, in[tm.offIn + (int64_t)r * tm.ldi + c], ah, al);
  }
  if (sh != 1.f || sl != 0.f) {
    const float h = ah, l = al;
    ah = 0.f;
    al = 0.f;
    df_acc(sh, sl, make_float2(h, l), ah, al);
  }
}

__global__ void __launch_bounds__(256) combine_pairs_f64_kernel(
    const CombChunk* __restrict__ chunks, const CombTask* __restrict__ tasks,
    const CombTerm* __restrict__ terms, const float2* in, double* out,
    float sh, float sl) {
  grid_next();
  grid_wait();
  const CombChunk ch = chunks[blockIdx.x];
  const CombTask t = tasks[ch.task];
  const int n = ch.nrows * t.cols;
  for (int idx = threadIdx.x; idx < n; idx += blockDim.x) {
    const int r = ch.row0 + idx / t.cols, c = idx % t.cols;
    float ah, al;
    df_combine(t, terms, in, r, c, sh, sl, ah, al);
    out[t.offOut + (int64_t)r * t.ldo + c] = (double)ah + (double)al;
  }
}

std::atomic<int64_t> g_launches{0};

// One CTA per entry.  Each segment is cut into pieces of 1024 elements, dealt to
// the CTA's warps in turn: the blocks of a charge-conserving tensor are often
// only a few hundred elements, which a CTA-wide loop per segment visits one
// memory latency after the other.
constexpr int kDotPiece = 1024;
__global__ void __launch_bounds__(256) dots_kernel(const DotTask* __restrict__ tasks,
                                                   const DotSeg* __restrict__ segs,
                                                   const double* A,
                                                   const double* B,
                                                   double* out) {
  grid_next();
  grid_wait();
  const DotTask t = tasks[blockIdx.x];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double acc0 = 0.0, acc1 = 0.0, acc2 = 0.0, acc3 = 0.0;
  int turn = 0;                       // pieces dealt so far, modulo the warps
  for (int k = 0; k < t.nseg; ++k) {
    const DotSeg g = segs[t.seg0 + k];
    const int64_t np = (g.len + kDotPiece - 1) / kDotPiece;
    for (int64_t q = (warp - turn) & 7; q < np; q += 8) {
      const int64_t e1 = min(g.len, (q + 1) * kDotPiece);
      int64_t e = q * kDotPiece + lane;
      const double* a = A + g.offA;
      const double* b = B + g.offB;
      for (; e + 96 < e1; e += 128) {
        acc0 = fma(a[e], b[e], acc0);
        acc1 = fma(a[e + 32], b[e + 32], acc1);
        acc2 = fma(a[e + 64], b[e + 64], acc2);
        acc3 = fma(a[e + 96], b[e + 96], acc3);
      }
      for (; e < e1; e += 32) acc0 = fma(a[e], b[e], acc0);
    }
    turn = (int)((turn + np) & 7);
  }
  double acc = (acc0 + acc1) + (acc2 + acc3);
  __shared__ double red[8];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double sum = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) sum += red[w];
    out[t.out] = sum;
  }
}

}  // namespace

int64_t launch_count() { return g_launches.load(); }
void count_launch(int n) { g_launches += n; }

void launch_gemm_f64(Trans ta, Trans tb, const GemmTile* tiles, int ntiles, const GemmTask* tasks,
                     const GemmSeg* segs, const double* A, const double* B, double* C,
                     cudaStream_t st) {
  if (ntiles <= 0) return;
  count_launch();
  dim3 grid(ntiles), block(NT);
  if (ta == Trans::N && tb == Trans::N)
    launch_chain(gemm_f64_kernel<Trans::N, Trans::N>, grid, block, 0, st, tiles, tasks, segs, A, B, C);
  else if (ta == Trans::N && tb == Trans::T)
    launch_chain(gemm_f64_kernel<Trans::N, Trans::T>, grid, block, 0, st, tiles, tasks, segs, A, B, C);
  else if (ta == Trans::T && tb == Trans::N)
    launch_chain(gemm_f64_kernel<Trans::T, Trans::N>, grid, block, 0, st, tiles, tasks, segs, A, B, C);
  else
    launch_chain(gemm_f64_kernel<Trans::T, Trans::T>, grid, block, 0, st, tiles, tasks, segs, A, B, C);
}

void launch_combine_pairs_f64(const CombChunk* chunks, int nchunks, const CombTask* tasks,
                              const CombTerm* terms, const float2* in, double* out,
                              double scale, cudaStream_t st) {
  if (nchunks <= 0) return;
  count_launch();
  const float sh = (float)scale, sl = (float)(scale - (double)sh);
  launch_chain(combine_pairs_f64_kernel, nchunks, 256, 0, st, chunks, tasks, terms, in, out, sh, sl);
}

void launch_combine_f64(const CombChunk* chunks, int nchunks, const CombTask* tasks,
                        const CombTerm* terms, const double* in, double* out, double scale,
                        cudaStream_t st) {
  if (nchunks <= 0) return;
  count_launch();
  launch_chain(combine_f64_kernel, nchunks, 256, 0, st, chunks, tasks, terms, in, out, scale);
}

void launch_dots(const DotTask* tasks, int ntasks, const DotSeg* segs, const double* A,
                 const double* B, double* out, cudaStream_t st) {
  if (ntasks <= 0) return;
  count_launch();
  launch_chain(dots_kernel, ntasks, 256, 0, st, tasks, segs, A, B, out);
}

}  // namespace dmrg3s
