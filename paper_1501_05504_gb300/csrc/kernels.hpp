// Device task tables and launchers of the block-sparse contraction kernels.
//
// All operand addresses are element offsets relative to base pointers passed
// at launch, so one uploaded table serves every matrix-vector product of a
// Lanczos run (only the vector pointers change).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace dmrg3s {

// One K-segment of a grouped GEMM task: C += scale * op(A) op(B) over K.
struct GemmSeg {
  int64_t offA, offB;
  int32_t lda, ldb, K, pad;
  double scale;
};

// One output block C (M x N, row-major with leading dimension ldc) of a
// grouped GEMM.  Segments [seg0, seg0 + nseg) are summed; nseg == 0 writes 0.
struct GemmTask {
  int64_t offC;
  int32_t ldc, M, N, seg0, nseg, pad;
};

// One size x size output tile of a task (64, 32, 16 or 8).
struct GemmTile {
  int32_t task, tm, tn, size;
};

// Linear combination of blocks: out = sum_k coef_k in_k (rows x cols).
struct CombTask {
  int64_t offOut;
  int32_t ldo, rows, cols, t0, nt, pad;
};
struct CombTerm {
  int64_t offIn;
  int32_t ldi;
  float chi;        // coef = chi + clo (FP32 pair, filled by the planner)
  double coef;
  float clo;
  int32_t pad;
};
// Work unit of the combination kernel: up to kCombRows rows of one task.
struct CombChunk {
  int32_t task, row0, nrows, pad;
};
constexpr int kCombRows = 16;

enum class Trans { N, T };

// ---- tensor-core operands: packed tiles ----
// A packed matrix (R x K) is stored in tiles of 8 rows x 32 k, tile (g, c) at
// float offset (c * R8 + g) * 256 (R8 = ceil(R / 8) row groups, KC =
// ceil(K / 32) k-chunks).  A tile is one 1 KB atom of the K-major 128-byte
// swizzled layout of the tcgen05 shared-memory descriptors: row r % 8 is a
// 128-byte line (32 k), and its 16-byte chunk j = (k % 32) / 4 sits at chunk
// position j ^ (r % 8), i.e. element (r, k) at float offset (r % 8) * 32 +
// (((k % 32) / 4) ^ (r % 8)) * 4 + k % 4 (the swizzle spreads the eight rows
// the tensor core reads together over all shared-memory banks).  Entries
// beyond R or K are zero.  A 128-row slab of one k-chunk is therefore
// contiguous (16 KB) and moves into shared memory with one bulk copy.  Every
// operand has a hi and a lo part (the 3xTF32 split) at the same offsets of
// two arrays.
constexpr int kPackTile = 256;             // floats per 8 x 32 tile
struct PackBlock {
  // element (r, k) of the packed matrix is scale * src[off + r * ld + k]
  // (trans = 0) or scale * src[off + k * ld + r] (trans = 1)
  int64_t src, dst;                        // dst: float offset of tile (0, 0)
  double scale;
  int32_t ld, R, K, trans, R8, KC, tile0;  // tile0: first tile in the launch numbering
  float pow2;                              // scale when it is a power of two (applied to the
                                           // FP32 parts, exactly), else 0
};
// One K-segment of a tensor-core task: packed A (rows M) and B (rows N).
struct TcSeg {
  int64_t pa, pb;
  int32_t ra8, rb8, kc, pad;
};
// One 128 x 128 output tile: the task's K-segments in order, nchunks k-chunks in all.
struct TcUnit {
  int32_t task, tm, tn, nchunks;
};
// A combination task whose output is written packed (the stage-3 operand).
struct PackOut {
  int64_t dst;
  int32_t R8, KC, trans, tile0;
};

// ---- FP64 products by exact FP16 slices (kernels_sliced.cu) ----
// A sliced operand block (R rows x K) is stored in tiles of 8 rows x 64 k of
// FP16 digits, one tile per slice: tile (chunk c, slice i, row group g) at
// element offset dst + ((c * kSlices + i) * R8 + g) * kSlTile, with R8 the row
// groups rounded up to an even number (so that a tile column is a multiple of
// 16 columns of an MMA).  A tile is one 1 KB atom of the K-major 128-byte
// swizzled layout: row r % 8 is a 128-byte line (64 k), its 16-byte piece j =
// (k % 64) / 8 at position j ^ (r % 8).
constexpr int kSlices = 8;
constexpr int kSlTile = 512;               // FP16 elements of a tile
// A row scale: the exponent field F of the row's largest element (below 2^(F - 1022);
// possibly outside an FP64 number's range) + kSlBias; 0 for a zero row, kSlSpecial
// for one with Inf or NaN.
constexpr int32_t kSlSpecial = 0x40000000, kSlBias = 4096;
// One block of a scale group: element (r, k) is coef * src[src + r ld + k]
// (trans = 0) or coef * src[src + k ld + r] (trans = 1).
// t0: its first 64-wide chunk among the chunks of its group.  d0: its first entry of
// the operand's grading (SlOperand), or -1.
struct SlMember {
  int64_t src, dst;
  double coef;
  int32_t ld, K, KC, trans, t0, d0;
};
// Up to 32 consecutive k of blocks that share a grading: d[d0 + k] (k < nk) = the
// exponent of the largest element at that k of the views [v0, v0 + nv), so that
// |element| 2^-d < 1 (0 for none, or with Inf or NaN).
struct SlGrade {
  int32_t d0, nk, v0, nv;
};
struct SlView {
  int64_t src;             // of the first k
  int32_t ld, R, trans, pad;
};
// Blocks with the same rows whose rows share scales: scales[e0 + r]; a CTA of the
// slicing kernel per `per` row groups (1, 2, 4 or 8), from cta0 on.
// `shift` raises the scales by that power of two: headroom of the integer sums.
struct SlGroup {
  int32_t R, R8, m0, nm, nt, e0, cta0, shift, which, per;   // nt: chunks; which: its operand
  int32_t ctas() const { return (R8 + per - 1) / per; }
};
// Spans a unit may sum before the headroom has to grow (the levels of a span
// stay below 2^58.1 in the 64-bit sum).
constexpr int kSlSpans = 28;
// One K-segment of a task where its FP64 operands are (read for listed elements
// only), and the first entry of its grading or -1; GemmTask / GemmSeg order.
struct SlSeg {
  int64_t offA, offB;
  double scale;
  int32_t lda, ldb, K, d0;
};
// One output tile of up to 128 rows x tile_n columns (rows and cols: what lies
// inside the block), written at C + offC with leading dimension ldc; row scales
// of A from ea, column scales of B from eb; spans accumulation spans.
// m0, n0: its place in the task (for rows with Inf or NaN).  The largest
// exponent of every output row (column) is collected in the scales from em on.
struct SlUnit {
  int64_t offC;
  int32_t ldc, rows, cols, nw, spans, ea, eb, m0, n0, seg0, nseg;
  int32_t shift;    // of A's row scales (SlGroup.shift)
  int32_t em;       // first row scale of the output as a later operand, or -1
  int32_t sel;      // which pair of FP64 operands (SlSource) its segments read
  uint32_t least;   // least |sum| that is taken without a look at its terms, in 2^32 of H
  int32_t d0;       // first grading entry of its columns for the collected scales, or -1
};
// The units' 64-wide k-chunks in the order a CTA runs them.  The copies: slice
// i of A is `ga` tiles at a + i sa, slice j of B `gb` tiles at b + j sb (FP16
// elements); `word` is the MMA issuer's view: kSlSteps = its k16 steps (1-4),
// kSlFirst / kSlLast = first / last chunk of a span (at most 64 k),
// kSlLongFirst / kSlLongLast = of a long span (four spans, levels 4-7), kSlMove
// = the accumulators' columns move (another nw than the chunk before), and nw
// from bit kSlNw on.
struct SlChunk {
  int64_t a, b;
  int32_t sa, sb;
  int32_t ga, gb;
};
constexpr uint32_t kSlSteps = 7, kSlFirst = 8, kSlLast = 16, kSlLongFirst = 32, kSlLongLast = 64,
                   kSlMove = 128, kSlNw = 8;
constexpr int kSlLongSpan = 4;
// An operand: its FP64 array, its packed array, its row scales; `scale`
// multiplies every coefficient; element (r, k) also takes the factor 2^(sign d[d0 + k]).
struct SlOperand {
  const double* src;
  uint16_t* out;
  int32_t* scales;
  double scale;
  const int32_t* d;
  int32_t sign, pad;
};
// The launch also clears `nclear` scales (which a later launch collects) and the
// `nfix` counters of the SlFix lists.
struct SlOperands {
  SlOperand op[4];
  int32_t* clear;
  int32_t* fix;
  int32_t nclear, nfix;
};
// The elements of a product that its slices may hold with fewer digits than FP64
// would: `count` parts of units (a drain warp's 32 rows x 16 columns; part w of
// unit u is 16 u + w) listed in `list`, with a word of 32 rows for each column in
// mask[16 (16 u + w) ..].
struct SlFix {
  int32_t* count;
  int32_t* list;
  uint32_t* mask;
};
constexpr int kSlParts = 16;
constexpr int64_t kSlFixInts = 17;         // of list and mask, for a part
constexpr int32_t kSlForce = 1 << 30;      // on a list entry: form the elements whatever their terms' size
// A block of an operand whose row scales are known (collected by the launch
// that wrote it): tiles [tile0, tile0 + R8 KC), tile t = (chunk, row group) with
// t = chunk R8 + group.
struct SlPiece {
  int64_t src, dst;
  int32_t ld, K, KC, trans, R, R8, e0, shift, tile0, d0;   // d0: as in SlMember (sign -1)
};
// Row scales and slices of every block of every group (a group has ctas() CTAs from its
// cta0 on; cta_group[c] = the group of CTA c).
void launch_slice(const SlGroup* groups, const int32_t* cta_group, int nctas,
                  const SlMember* members, const SlOperands& ops, cudaStream_t st);
// The gradings of a site tensor (kernels_sliced.cu).
void launch_grade(const SlGrade* items, int nitems, const SlView* views, const double* src, int32_t* d,
                  cudaStream_t st);
// Slices of the pieces, a warp per tile; first[c] = the piece of tile 8 c.
void launch_slice_known(const SlPiece* pieces, int npieces, const int32_t* first, int ntiles,
                        const double* src, uint16_t* out, const int32_t* scales, const int32_t* d,
                        cudaStream_t st);

// C = sum over the task's segments of op(A) op(B), one rounding to FP64 (see
// kernels_sliced.cu).  CTA b runs units [cta_unit[b], cta_unit[b + 1]) and
// chunks [cta_chunk[b], cta_chunk[b + 1]).  src, segs: the FP64
// operands, read for rows with Inf or NaN only.  collect: the row scales of the
// output as an operand (of its rows, or of its columns), cleared before.
struct SlTables {
  const SlUnit* units;
  const SlChunk* chunks;
  const uint32_t* words;
  const int32_t *cta_unit, *cta_chunk;
  const SlSeg* segs;
  int ncta, nunits;
  bool chain;       // short enough for a chained launch (launch.hpp)
};
struct SlSource {
  const double *A, *B, *A1, *B1;     // A1, B1: of the units with sel = 1
  int32_t ta, tb;                    // stored transposed (as in launch_gemm_f64)
  double scale;
  int32_t sign, pad;                 // of A's grading (SlOperand.sign); B has the other one
};
// d: the gradings (SlUnit.d0; the scales of column c are collected as those of the
// elements times 2^-d).  fix (its count cleared before): receives the elements to form from the FP64
// operands, which a second launch does.
void launch_gemm_sliced(const SlTables& t, const uint16_t* pA, const uint16_t* pB,
                        const int32_t* eA, const int32_t* eB, const SlSource& src, double* C,
                        int32_t* collect, bool collect_cols, const int32_t* d, const SlFix& fix, int* err,
                        uint64_t wait_ns, cudaStream_t st);

// Blockwise inner products: out[task.out] = sum over the task's segments of
// <A[offA .. offA+len), B[offB .. offB+len)> (FP64, fixed summation order).
struct DotSeg {
  int64_t offA, offB, len;
};
struct DotTask {
  int64_t out;
  int32_t seg0, nseg;
};

// Process-wide count of kernels launched by this library.
int64_t launch_count();
void count_launch(int n = 1);

// FP64 grouped GEMM on the CUDA cores.  opA = A (M x K, lda) or A^T (A stored
// K x M); opB = B (K x N, ldb) or B^T (B stored N x K).
void launch_gemm_f64(Trans ta, Trans tb, const GemmTile* tiles, int ntiles, const GemmTask* tasks,
                     const GemmSeg* segs, const double* A, const double* B, double* C,
                     cudaStream_t st);

// out = scale * sum_k coef_k in_k for every task.
// Tensor-core grouped GEMM (tcgen05): passes = 1 (TF32) or 3 (3xTF32) over
// packed operands (hi, lo parts; lo unused when passes == 1), persistent CTAs
// over the units (a static schedule: one unit list per CTA).  Two output forms:
//  - packed = false: every output element as a double-float pair (hi, lo) at
//    (float2*)Chi + offC + m ldc + n (8 bytes per element, like the double it
//    stands for); Clo unused;
//  - packed = true: the output block packed as the A operand of a following
//    tensor-core stage (R = M rows, K = N, tile layout above, hi at Chi, lo at
//    Clo, lo only with passes == 3), with offC = its float offset and ldc =
//    its R8; entries beyond N in the last k-chunk and rows M .. 8 R8 - 1 are
//    written as zero.
// err is a device flag set to 1 when a wait gave up after wait_ns nanoseconds.
// One CTA per unit list: CTA b runs units [cta_start[b], cta_start[b + 1]).
void launch_gemm_tc(int passes, bool packed, const TcUnit* units, const int32_t* cta_start,
                    int ncta, const GemmTask* tasks, const TcSeg* segs, const float* Ahi,
                    const float* Alo, const float* Bhi, const float* Blo, float* Chi, float* Clo,
                    int* err, uint64_t wait_ns, bool chain, cudaStream_t st);

// Packs FP64 blocks into tensor-core operands: hi = tf32(x), lo = tf32(x - hi)
// (lo may be null), in the tile layout above.
void launch_pack(const PackBlock* blocks, int nblocks, int ntiles, const double* src, float* hi,
                 float* lo, cudaStream_t st);

// Combinations of double-float pair inputs (the tensor-core outputs), in
// double-float arithmetic on the FP32 pipe: out = scale * sum_k coef_k in_k.
// _pack writes the result as the packed 3xTF32 operand (hi, lo; lo may be
// null) of a following tensor-core stage (one PackOut per task), _f64 writes
// FP64.
void launch_combine_pairs_pack(const PackOut* outs, int ntasks, int ntiles, const CombTask* tasks,
                               const CombTerm* terms, const float2* in, float* out_hi,
                               float* out_lo, double scale, cudaStream_t st);
void launch_combine_pairs_f64(const CombChunk* chunks, int nchunks, const CombTask* tasks,
                              const CombTerm* terms, const float2* in, double* out,
                              double scale, cudaStream_t st);

void launch_combine_f64(const CombChunk* chunks, int nchunks, const CombTask* tasks,
                        const CombTerm* terms, const double* in, double* out, double scale,
                        cudaStream_t st);

// One CTA per task; deterministic (no atomics).
void launch_dots(const DotTask* tasks, int ntasks, const DotSeg* segs, const double* A,
                 const double* B, double* out, cudaStream_t st);

}  // namespace dmrg3s
