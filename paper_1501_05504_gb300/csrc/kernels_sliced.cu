// FP64 block products on the tensor cores: operands cut into exact FP16 slices
// (the splitting of Ozaki, Ogita, Oishi and Rump, 2012, with the integer slices
// that Mukunoki, Ozaki, Ogita and Imamura, 2020, run on tensor cores).
//
// Every row of a packed operand (an output row of A, an output column of B)
// carries one power-of-two scale over the whole contracted index; relative to
// it an element is a 71-bit fixed-point number v (|v| <= 2^71, rounded to
// nearest), written in eight balanced digits of 9 bits,
//   v = sum_i q_i 2^(63 - 9 i),   -256 <= q_i <= 256,
// each exact in FP16.  With both operands sliced,
//   C = 2^(scales) sum_l 2^(126 - 9 l) S_l,   S_l = sum_{i + j = l} A_i B_j,
// and the 36 digit products of the levels l = 0 .. 7 are formed (levels >= 8
// lie below 2^-72 of the row scales).  One S_l collects at most 64 k before
// it is drained for l <= 3, 256 k for l >= 4.  Levels 0-3 are exact integers in
// the FP32 accumulators (|S_l| <= (l + 1) 64 2^16 <= 2^24); levels 4-7 are while
// their sums stay below 2^24 (17 sigma of rounding digits), and rows with one near 2^24
// or above (digits that repeat along k) are listed (below).
// The drained levels are summed exactly in integers: H (64 bits, in units of level
// 4; the row scales leave it room for the task's spans) and L (27 bits below it),
// and the output is H 2^27 + L rounded once to FP64 with integer instructions.
//
// Precision: an FP64 product keeps 53 bits of every term, however small beside the
// others of its row; here a term is held to 2^-72 of the row scales.  Over K
// terms the rounding of the slices and the missing levels amount to about E =
// sqrt(K) 2^-72 of the scales (0.95 rms a term), so an output element with
// S = sum |a| |b| >= 3 2^54 E loses less by them than by the roundings of an FP64
// sum (2^-53 of S each), and is stored: |C| >= that bound shows it, or the sum of any
// one span (levels 0 and 1; the lower ones reach 25000 units of level 1).  Any
// other element (small terms of a graded row, cancelling terms) is listed, and a second
// launch (fix_kernel) looks at it: it computes S of the part, and what stays below the
// bound is formed from the FP64 operands, term by term (rows with large levels always,
// in compensated sums).  So no element is further from the exact sum than the plain
// form's bound, whatever the grading.
//
// Why: GB300 multiplies FP64 at 2 multiply-adds per SM and clock (1.1 TFLOP/s
// measured) and FP16 with FP32 accumulation at ~1700 times that, so 36 exact
// products cost less than a fortieth of one FP64 product.
//
// Kernel: persistent CTAs (one per SM, 576 threads) over output tiles of
// 128 x 64.  The eight levels are eight accumulators of nw <= 64 columns side
// by side in tensor memory (all 512 of its columns), and the B slices lie back to
// back in shared memory, so digit A_i meets the slices B_0 .. B_(7-i) in MMAs of up
// to 256 columns (one issue serves up to four digit products, and the A digit is read
// from shared memory once for all of them).
//   warp 0     one lane issues the bulk copies: the eight B slices of a 64-wide
//              k-chunk in one of two 64 KB buffers, the A slices through a ring
//              of 16 KB slabs
//   warp 1     one lane issues tcgen05.mma (kind::f16); level l is committed to
//              its own barrier right after digit A_l, while the later digits
//              still run
//   warps 2-17 drain: 32 rows x 16 columns each, H and L in registers
// Every wait is bounded as in the other tensor-core kernel.
//
// Inside a tile it is bound by the MMAs and by shared-memory bandwidth: the 36 products
// of 16 k take 1312 cycles for 64 columns.  Measured (the plain form / this): the m = 2048
// cylinder's environment update, 13 Gflop, 12.1 / 0.93 ms; the m = 512 XXZ operator, 0.18
// Gflop, 219 / 120 us, where eight launches, the slicing and short units (2 to 4 spans)
// count as much.  (With seven slices, no gradings and no fix launches, and so with
// small terms held to 2^-63 of the scales only: 0.75 ms and 71 us.)
#include <algorithm>
#include <atomic>
#include <cstdint>

#include "kernels.hpp"
#include "fp64.cuh"
#include "launch.hpp"
#include "tc_common.cuh"

namespace dmrg3s {

namespace {

constexpr int kFirstDrainWarp = 2, kDrainWarps = 16;
constexpr int kThreads = 32 * (kFirstDrainWarp + kDrainWarps);
constexpr int kSlabA = 16384;                          // 128 rows x 64 k of one slice
constexpr int kSlots = 4;                              // A ring
constexpr int kBufB = kSlices * 8192;                  // 64 columns x 64 k of all slices
constexpr int kOffA = 2 * kBufB;
constexpr int kOffStage = kOffA + kSlots * kSlabA;
constexpr int kStageRow = 5;                           // doubles per staged row (4 + 1 pad)
constexpr int kStageWarp = 32 * kStageRow * 8;
constexpr int kSmemBytes = kOffStage + kDrainWarps * kStageWarp;
constexpr uint32_t kTmemCols = 512;
// A drained level is turned into an integer by an FP32 addition (the low bits
// of x + 1.5 2^23 are x + 2^22; a conversion instruction takes 8 cycles a warp
// and sub-partition, the addition one).  Two levels of at most 2^21 make one
// unsigned 32-bit word, (a + 2^21) 512 + b + (the bits of 1.5 2^23), so H grows
// by kBiasH per span besides the levels, and by kBiasOne and kBiasLow (27 bits below it)
// per long span; larger levels (possible, but far outside what rounding digits give)
// take the conversion.
constexpr uint32_t kBiasOne = 0x4B400000u;
constexpr unsigned long long kBiasPair = (2097152ull << 9) + kBiasOne;
constexpr uint32_t kLowMask = (1u << 27) - 1;
constexpr unsigned long long kBiasLow = (unsigned long long)kBiasOne * ((1u << 18) + (1u << 9) + 1u);
constexpr unsigned long long kBiasH = (kBiasPair << 27) + (kBiasPair << 9);

// Instruction descriptor of kind::f16: D = F32, A = B = F16, both K-major.
__device__ __forceinline__ uint32_t idesc_f16(uint32_t n) {
  return (1u << 4) | ((n >> 3) << 17) | ((128u >> 4) << 24);
}

// Lower word of the shared-memory descriptor (smem_desc) of an address; the
// upper word is the same for all.  A K step of 16 (32 bytes) adds 2.
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr) { return ((addr >> 4) & 0x3FFF) | (1u << 16); }
constexpr uint32_t kDescHi = 64u | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint64_t desc(uint32_t lo) { return ((uint64_t)kDescHi << 32) | lo; }

__device__ __forceinline__ void mma_f16(uint32_t dtmem, uint64_t ad, uint64_t bd, uint32_t idesc,
                                        uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
      "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
      : "memory");
}

// ks MMAs of 16 k each from one pair of slabs (acc: whether the first adds).
__device__ __forceinline__ void mma_steps(uint32_t d, uint32_t a, uint32_t b, uint32_t idesc, int ks,
                                          uint32_t acc) {
  if (ks == 4) {
    mma_f16(d, desc(a), desc(b), idesc, acc);
    mma_f16(d, desc(a + 2), desc(b + 2), idesc, 1u);
    mma_f16(d, desc(a + 4), desc(b + 4), idesc, 1u);
    mma_f16(d, desc(a + 6), desc(b + 6), idesc, 1u);
  } else {
    for (int kk = 0; kk < ks; ++kk) mma_f16(d, desc(a + 2 * kk), desc(b + 2 * kk), idesc, kk ? 1u : acc);
  }
}

// Loads of 8 columns (32 lanes); several in flight before one wait.
__device__ __forceinline__ void tmem_ld8_async(uint32_t taddr, uint32_t* v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]),
                 "=r"(v[6]), "=r"(v[7])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld8(uint32_t (&v)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]),
                 "+r"(v[6]), "+r"(v[7])::"memory");
}
// Waits for the loads; v passes through it, so that no use moves before it.
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&v)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]),
                 "+r"(v[6]), "+r"(v[7]), "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]),
                 "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15])::"memory");
}

// (H 2^27 + L) 2^ex (L < 2^27) rounded to the nearest FP64 value: 32-bit integer
// instructions on the 96-bit sum (an FP64 conversion or addition holds GB300's
// FP64 unit for 64 cycles a warp), without branches, so that several elements
// are in flight.  (A negative sum is complemented, one unit below its
// magnitude: 2^-79 of the scales.)  Sets `out` when the result needs the
// general form below: exponent outside the normal range, or no bit above the
// last 32 of the 96.
__device__ __forceinline__ double fixed_to_f64(long long H, uint32_t L, int ex, bool* out) {
  const uint32_t h0 = (uint32_t)H, h1 = (uint32_t)((unsigned long long)H >> 32);
  uint32_t x0 = (h0 << 27) | L, x1 = __funnelshift_l(h0, h1, 27), x2 = (uint32_t)((int32_t)h1 >> 5);
  const uint32_t s = (uint32_t)((int32_t)x2 >> 31);
  x0 ^= s;
  x1 ^= s;
  x2 ^= s;
  const bool z = x2 == 0;                           // the leading limb first
  const uint32_t y2 = z ? x1 : x2, y1 = z ? x0 : x1, y0 = z ? 0u : x0;
  uint32_t lz;
  asm("bfind.shiftamt.u32 %0, %1;" : "=r"(lz) : "r"(y2));
  const uint32_t w1 = __funnelshift_l(y1, y2, lz), w0 = __funnelshift_l(y0, y1, lz);
  uint32_t r0, r1, c;
  asm("add.cc.u32 %0, %3, 0x400;\n\taddc.cc.u32 %1, %4, 0;\n\taddc.u32 %2, 0, 0;"
      : "=r"(r0), "=r"(r1), "=r"(c)
      : "r"(w0), "r"(w1));
  // exponent field less one: the leading bit of r1 >> 11 adds it (it is gone
  // when the rounding carried out)
  const int f = ex + (95 + 1022) - (z ? 32 : 0) - (int)lz + 2 * (int)c;
  const bool zero = (y2 | y1) == 0;
  *out = *out || (!zero && ((uint32_t)f >= 2045u || y2 == 0));
  const uint32_t hi = ((r1 >> 11) + ((uint32_t)f << 20)) | (s & 0x80000000u);
  return __hiloint2double((int)(zero ? 0u : hi), (int)(zero ? 0u : __funnelshift_r(r0, r1, 11)));
}

// The same for any range, in FP64 arithmetic.
__device__ __noinline__ double fixed_to_f64_any(long long H, uint32_t L, int ex) {
  const double top = (double)(H >> 32) * 4294967296.0, low = (double)(H & 0xFFFFFFFFll);
  return ldexp(fma(top + low, 134217728.0, (double)L), ex);
}

// The row scale that x 2^-d asks for (a subnormal counts as the smallest exponent).
__device__ __forceinline__ int scale_of(double x, int d) {
  const uint32_t hi = (uint32_t)__double2hiint(x) & 0x7FFFFFFFu;
  const int f = (int)(hi >> 20);
  if (f == 0x7FF) return kSlSpecial;
  return (hi | (uint32_t)__double2loint(x)) == 0u ? 0 : max(f, 1) - d + kSlBias;
}

__global__ void __launch_bounds__(kThreads, 1)
    gemm_sliced_kernel(const SlTables tab, const uint16_t* pA,
                       const uint16_t* pB, const int32_t* eA,
                       const int32_t* eB,
                       double* C, int32_t* collect, int collect_cols, const int32_t* d,
                       const SlFix fix, int* err, uint64_t wait_ns) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t afull[kSlots], aempty[kSlots], bfull[2], bempty[2];
  __shared__ __align__(8) uint64_t lfull[kSlices], lempty[kSlices], done;
  __shared__ uint32_t tmem_base;
  __shared__ volatile int abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid == 0) {
    for (int s = 0; s < kSlots; ++s) {
      mbar_init(&afull[s], 1);
      mbar_init(&aempty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&bfull[s], 1);
      mbar_init(&bempty[s], 1);
    }
    for (int l = 0; l < kSlices; ++l) {
      mbar_init(&lfull[l], 1);
      mbar_init(&lempty[l], kDrainWarps);
    }
    mbar_init(&done, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_base)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  const WaitCtl wc{&abort_flag, err, wait_ns};
  grid_wait();

  if (warp == 0) {
    // ---------------- bulk-copy producer ----------------
    if (lane == 0) {
      const int c_end = tab.cta_chunk[blockIdx.x + 1];
      int ci = tab.cta_chunk[blockIdx.x];
      uint32_t qa = 0, bf = 0;               // A slabs and B buffers filled
      SlChunk next{};
      if (ci < c_end) next = tab.chunks[ci];
      for (bool ok = true; ci < c_end && ok; ++ci) {
        const SlChunk ch = next;
        if (ci + 1 < c_end) next = tab.chunks[ci + 1];
        const int bs = (int)(bf & 1);
        if (bf >= 2 && !mbar_wait(&bempty[bs], ((bf >> 1) - 1) & 1, wc)) break;
        unsigned char* bb = smem + bs * kBufB;
        mbar_expect_tx(&bfull[bs], (uint32_t)(kSlices * ch.gb) * 1024u);
        if (ch.gb * kSlTile == ch.sb) {      // all slices of the chunk are contiguous
          bulk_g2s(bb, pB + ch.b, (uint32_t)(kSlices * ch.gb) * 1024u, &bfull[bs]);
        } else {
          for (int j = 0; j < kSlices; ++j)
            bulk_g2s(bb + j * ch.gb * 1024, pB + ch.b + (int64_t)j * ch.sb, (uint32_t)ch.gb * 1024u,
                     &bfull[bs]);
        }
        ++bf;
        for (int i = 0; i < kSlices; ++i, ++qa) {
          const int st = (int)(qa % kSlots);
          if (qa >= (uint32_t)kSlots && !mbar_wait(&aempty[st], ((qa / kSlots) - 1) & 1, wc)) {
            ok = false;
            break;
          }
          mbar_expect_tx(&afull[st], (uint32_t)ch.ga * 1024u);
          bulk_g2s(smem + kOffA + st * kSlabA, pA + ch.a + (int64_t)i * ch.sa,
                   (uint32_t)ch.ga * 1024u, &afull[st]);
        }
      }
      // copies still in flight must land before the CTA's memory is released:
      // the last phase of every slot and buffer that was filled
      for (uint32_t s = 0; s < (uint32_t)kSlots; ++s) {
        const uint32_t n = qa > s ? (qa - s + kSlots - 1) / kSlots : 0;
        if (n) mbar_drain(&afull[s], (n - 1) & 1);
      }
      for (uint32_t s = 0; s < 2; ++s) {
        const uint32_t n = bf > s ? (bf - s + 1) / 2 : 0;
        if (n) mbar_drain(&bfull[s], (n - 1) & 1);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    // the whole warp walks the chunks and one elected lane issues: the operands
    // of tcgen05.mma sit in uniform registers, and inside a branch of a single
    // known lane moving them there costs ~150 cycles an MMA instead of ~44.  The
    // next slab's barrier is tested while this one's MMAs are issued, and the
    // chunk words are read one ahead.
    const bool one = elect_one();
    const int c_end = tab.cta_chunk[blockIdx.x + 1];
    int ci = tab.cta_chunk[blockIdx.x];
    uint32_t slot = 0, aph = 0, bs = 0, bph = 0;
    uint32_t ph = 0, pl = 0;             // spans (levels 0-3), long spans (levels 4-7)
    uint32_t next = ci < c_end ? tab.words[ci] : 0u;
    const uint32_t s0 = smem_u32(smem);
    const uint32_t tmem_u = __reduce_or_sync(0xffffffffu, tmem);
    bool ok = true;
    bool b_ready = false, a_ready = false;
    // levels [l0, l1) drained since their last commit
    auto drained = [&](int l0, int l1, uint32_t n) {
      bool w = true;
      for (int l = l0; l < l1 && w; ++l) w = mbar_wait(&lempty[l], (n - 1) & 1, wc);
      return __all_sync(0xffffffffu, w) != 0;
    };
    for (; ci < c_end && ok; ++ci) {
      const uint32_t w = __reduce_or_sync(0xffffffffu, next);   // in a uniform register
      if (ci + 1 < c_end) next = tab.words[ci + 1];
      const uint32_t nw = w >> kSlNw;
      const int ks = (int)(w & kSlSteps);
      if (!__all_sync(0xffffffffu, b_ready) &&
          !__all_sync(0xffffffffu, mbar_wait(&bfull[bs], bph, wc)))
        break;
      const uint32_t sb = desc_lo(s0 + bs * kBufB);
      if ((w & kSlFirst) && ph > 0) {
        // levels 0-3 (after a change of nw, which moves the levels' columns: all)
        ok = drained(0, 4, ph) && (!(w & kSlMove) || pl == 0 || drained(4, kSlices, pl));
        if (!ok) break;
      }
#pragma unroll
      for (int i = 0; i < kSlices; ++i) {
        if (!__all_sync(0xffffffffu, a_ready) &&
            !__all_sync(0xffffffffu, mbar_wait(&afull[slot], aph, wc))) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t sa = desc_lo(s0 + kOffA + slot * kSlabA);
        const uint32_t cur = slot;
        if (++slot == kSlots) {
          slot = 0;
          aph ^= 1;
        }
        a_ready = mbar_test(&afull[slot], aph);
        // B slices 0 .. 7 - i in one MMA, or in two when they are more than 256
        // columns (the first digit always: its levels 4-7 are drained later)
        const uint32_t all = (uint32_t)(kSlices - i);
        const uint32_t n1 = i == 0 ? 4u : (i < 4 && all * nw > 256u) ? 3u : all;
        const bool two = i < 4 && n1 < all;
        const bool wait2 = i == 0 && (w & kSlLongFirst) && pl > 0;
        if (wait2) {
          if (one)
            mma_steps(tmem_u, sa, sb, idesc_f16(n1 * nw), ks, (w & kSlFirst) ? 0u : 1u);
          __syncwarp();
          if (!drained(4, kSlices, pl)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        }
        if (one) {
          if (!wait2)
            mma_steps(tmem_u + (uint32_t)i * nw, sa, sb, idesc_f16(n1 * nw), ks,
                      (i == 0 && (w & kSlFirst)) ? 0u : 1u);
          if (two)
            mma_steps(tmem_u + ((uint32_t)i + n1) * nw, sa, sb + n1 * nw * 8u,
                      idesc_f16((all - n1) * nw), ks, (i == 0 && (w & kSlLongFirst)) ? 0u : 1u);
          mma_commit(&aempty[cur]);
          if (w & (i < 4 ? kSlLast : kSlLongLast)) mma_commit(&lfull[i]);   // level i is complete
          if (i == kSlices - 1) mma_commit(&bempty[bs]);
        }
        __syncwarp();
      }
      if (!ok) break;
      if (w & kSlLast) ++ph;
      if (w & kSlLongLast) ++pl;
      bs ^= 1;
      if (bs == 0) bph ^= 1;
      b_ready = ci + 1 < c_end && mbar_test(&bfull[bs], bph);
    }
    // every product issued must finish before the tensor memory is freed
    if (one) {
      mma_commit(&done);
      mbar_drain(&done, 0);
    }
    __syncwarp();
  } else {
    // ---------------- drain and epilogue ----------------
    // 16 warps (four per scheduler hide the tensor memory's latency), each the
    // 32 rows of its quarter and 16 columns
    const int quarter = warp & 3, part = (warp - kFirstDrainWarp) >> 2;
    const uint32_t tcol = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(part * 16);
    double* stage =
        reinterpret_cast<double*>(smem + kOffStage + (warp - kFirstDrainWarp) * kStageWarp);
    uint32_t ph = 0, pl = 0;
    bool ok = true;
    const int u_end = tab.cta_unit[blockIdx.x + 1];
    for (int u = tab.cta_unit[blockIdx.x]; u < u_end && ok; ++u) {
      const SlUnit& un = tab.units[u];
      if (u + 1 < u_end)
        asm volatile("prefetch.global.L1 [%0];" ::"l"(reinterpret_cast<const char*>(&tab.units[u + 1]) + lane * 2));
      const uint32_t nw = (uint32_t)un.nw;
      const int spans = un.spans;
      // (a warp beyond the tile only arrives)
      const bool mine = (uint32_t)(part * 16) < nw && quarter * 32 < un.rows;
      unsigned long long H[16];                          // units of level 4 (levels 0-3 biased)
      uint32_t L[16];                                    // below them, units of level 7
      bool large = false;                                // a level 4-7 near 2^24 or above
      uint32_t sized = 0;                                // columns with a span of enough size
      const uint32_t enough = min(32u * un.least + 25000u, 1u << 30);
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        H[j] = 0;
        L[j] = 0;
      }
      const int row0 = quarter * 32, row = row0 + lane, n0 = part * 16;
      // (rows and columns of the padding get a scale in the normal range)
      const int fa = row < un.rows && spans > 0 ? eA[un.ea + row] : kSlBias + 1057;
      const int fb_lane = lane < 16 && n0 + lane < un.cols && spans > 0 ? eB[un.eb + n0 + lane] : kSlBias + 1057;
      for (int sp = 0; sp < spans && ok; ++sp, ++ph) {
        const bool longer = sp % kSlLongSpan == kSlLongSpan - 1 || sp == spans - 1;
#pragma unroll
        for (int l = 0; l < 4; l += 2) {                 // levels (0, 1), (2, 3)
          // one decision per warp: tcgen05.ld is a warp-wide instruction
          if (!__all_sync(0xffffffffu, mbar_wait(&lfull[l + 1], ph & 1, wc))) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          if (mine) {
#pragma unroll
            for (int h = 0; h < 16; h += 8) {
              uint32_t v[16];
              tmem_ld8_async(tcol + (uint32_t)l * nw + h, v);
              tmem_ld8_async(tcol + (uint32_t)(l + 1) * nw + h, v + 8);
              tmem_wait_ld(v);
              float m = 0.f;
#pragma unroll
              for (int j = 0; j < 8; ++j)
                m = fmaxf(m, fmaxf(fabsf(__uint_as_float(v[j])), fabsf(__uint_as_float(v[8 + j]))));
              if (!__any_sync(0xffffffffu, !(m < 2097152.f))) {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                  const uint32_t w =
                      __float_as_uint(__fadd_rn(__uint_as_float(v[j]), 10485760.f)) * 512u +
                      __float_as_uint(__fadd_rn(__uint_as_float(v[8 + j]), 12582912.f));
                  H[h + j] += (unsigned long long)w * (l == 0 ? 134217728u : 512u);
                  if (l == 0 && w - (uint32_t)kBiasPair + enough > 2u * enough) sized |= 1u << (h + j);
                }
              } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                  const long long a = (long long)__float2int_rn(__uint_as_float(v[j])) * 512 +
                                      __float2int_rn(__uint_as_float(v[8 + j]));
                  H[h + j] += ((unsigned long long)a + kBiasPair) * (l == 0 ? 134217728u : 512u);
                  if (l == 0 && llabs(a) > (long long)enough) sized |= 1u << (h + j);
                }
              }
            }
          }
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) {
            mbar_arrive(&lempty[l]);
            mbar_arrive(&lempty[l + 1]);
          }
        }
        if (!ok || !longer) continue;
        // level 4 into H, then levels 5-7 together: t = S_5 2^18 + S_6 2^9 + S_7 + L is at most
        // 63 bits, its upper part belongs to H
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          const int l = g == 0 ? 4 : kSlices - 1;
          for (int w = g == 0 ? 4 : 5; w <= l && ok; ++w)
            if (!__all_sync(0xffffffffu, mbar_wait(&lfull[w], pl & 1, wc))) ok = false;
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          if (mine && g == 0) {
            uint32_t v[16];
            tmem_ld8_async(tcol + 4u * nw, v);
            tmem_ld8_async(tcol + 4u * nw + 8, v + 8);
            tmem_wait_ld(v);
            float m = 0.f;
#pragma unroll
            for (int j = 0; j < 16; ++j) m = fmaxf(m, fabsf(__uint_as_float(v[j])));
            if (!__any_sync(0xffffffffu, !(m < 4194304.f))) {
#pragma unroll
              for (int j = 0; j < 16; ++j) H[j] += __float_as_uint(__fadd_rn(__uint_as_float(v[j]), 12582912.f));
            } else {
              large = large || (row < un.rows && !(m < 16000000.f));   // (lanes beyond hold garbage)
#pragma unroll
              for (int j = 0; j < 16; ++j)
                H[j] += (unsigned long long)(long long)__float2int_rn(__uint_as_float(v[j])) + kBiasOne;
            }
          } else if (mine) {
#pragma unroll
            for (int h = 0; h < 16; h += 8) {
              uint32_t v[16], u[16];
              tmem_ld8_async(tcol + 5u * nw + h, v);
              tmem_ld8_async(tcol + 6u * nw + h, v + 8);
              tmem_ld8_async(tcol + 7u * nw + h, u);
              tmem_wait_ld(v);
              tmem_wait_ld8(u);
              float m = 0.f;
#pragma unroll
              for (int j = 0; j < 8; ++j)
                m = fmaxf(m, fmaxf(fmaxf(fabsf(__uint_as_float(v[j])), fabsf(__uint_as_float(v[8 + j]))),
                                   fabsf(__uint_as_float(u[j]))));
              if (!__any_sync(0xffffffffu, !(m < 4194304.f))) {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                  const uint32_t a = __float_as_uint(__fadd_rn(__uint_as_float(v[j]), 12582912.f));
                  const uint32_t b = __float_as_uint(__fadd_rn(__uint_as_float(v[8 + j]), 12582912.f));
                  const uint32_t c = __float_as_uint(__fadd_rn(__uint_as_float(u[j]), 12582912.f)) + L[h + j];
                  const unsigned long long t = (unsigned long long)a * 262144u + ((unsigned long long)b * 512u + c);
                  H[h + j] += t >> 27;
                  L[h + j] = (uint32_t)t & kLowMask;
                }
              } else {
                large = large || (row < un.rows && !(m < 16000000.f));
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                  const long long t = (long long)__float2int_rn(__uint_as_float(v[j])) * 262144 +
                                      (long long)__float2int_rn(__uint_as_float(v[8 + j])) * 512 +
                                      __float2int_rn(__uint_as_float(u[j])) + (long long)(kBiasLow + L[h + j]);
                  H[h + j] += (unsigned long long)(t >> 27);
                  L[h + j] = (uint32_t)t & kLowMask;
                }
              }
            }
          }
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0)
            for (int w = g == 0 ? 4 : 5; w <= l; ++w) mbar_arrive(&lempty[w]);
        }
        if (!ok) break;
        ++pl;
      }
      if (!ok) break;
      if (!mine) continue;
      // rows of 4 consecutive doubles through the warp's staging rows
      // the biases: X = H 2^27 + L less `longs` kBiasLow
      const unsigned long long longs = (unsigned long long)((spans + kSlLongSpan - 1) / kSlLongSpan);
      const unsigned long long low = longs * kBiasLow;
      const unsigned long long bh = (unsigned long long)spans * kBiasH + longs * kBiasOne + (low >> 27);
      const uint32_t bl = (uint32_t)low & kLowMask;
      const int rows = un.rows, cols = un.cols;
      double* Cu = C + un.offC + n0;
      const int64_t ldc = un.ldc;
      const int em = un.em, shift = un.shift;
      // largest scale of the row (of column `lane`), and this lane's column's grading
      int fmax = 0;
      const int d_lane = em >= 0 && un.d0 >= 0 && lane < 16 && n0 + lane < cols ? d[un.d0 + n0 + lane] : 0;
      // a zero row or column has no error; elements of rows and columns with Inf or
      // NaN (their slices are zero) are listed
      const uint32_t zero_col = __ballot_sync(0xffffffffu, lane < 16 && fb_lane == 0);
      const uint32_t bad_col = __ballot_sync(0xffffffffu, lane < 16 && fb_lane == kSlSpecial);
      const uint32_t least = fa == 0 ? 0u : un.least;
      uint32_t listed = fa == kSlSpecial || large ? 0xffffu : bad_col;   // this lane's columns
#pragma unroll
      for (int c4 = 0; c4 < 16; c4 += 4) {
        if (n0 + c4 >= cols) break;
        bool out = false;                    // of this lane's elements inside the tile
        int ex[4];
        double val[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint32_t lo = L[c4 + i] - bl;                  // (a borrow leaves the sign bit)
          const long long h = (long long)(H[c4 + i] - bh) - (long long)(lo >> 31);
          const int hs = (int)(h >> 32);
          if ((uint32_t)(hs ^ (hs >> 31)) < least) listed |= 1u << (c4 + i) & ~(zero_col | sized);
          bool o = false;
          ex[i] = fa + shift + __shfl_sync(0xffffffffu, fb_lane, c4 + i) - (2123 + 2 * kSlBias);
          val[i] = fixed_to_f64(h, lo & kLowMask, ex[i], &o);
          out = out || (o && row < rows && n0 + c4 + i < cols);
        }
        if (out)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint32_t lo = L[c4 + i] - bl;
            val[i] = fixed_to_f64_any((long long)(H[c4 + i] - bh) - (long long)(lo >> 31), lo & kLowMask, ex[i]);
          }
#pragma unroll
        for (int i = 0; i < 4; ++i) stage[lane * kStageRow + i] = val[i];
        if (em >= 0) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int dc = un.d0 >= 0 ? __shfl_sync(0xffffffffu, d_lane, c4 + i) : 0;
            int f = scale_of(val[i], dc);
            if (row >= rows || n0 + c4 + i >= cols || (listed >> (c4 + i) & 1u)) f = 0;
            if (collect_cols) {
              f = __reduce_max_sync(0xffffffffu, f);
              fmax = lane == c4 + i ? f : fmax;
            } else {
              fmax = max(fmax, f);
            }
          }
        }
        __syncwarp();
#pragma unroll
        for (int it = 0; it < 4; ++it) {
          const int r = it * 8 + (lane >> 2), cc = lane & 3;
          if (row0 + r < rows && n0 + c4 + cc < cols)
            Cu[(row0 + r) * ldc + c4 + cc] = stage[r * kStageRow + cc];
        }
        __syncwarp();
      }
      if (em >= 0) {
        const bool inside = collect_cols ? lane < 16 && n0 + lane < cols : row < rows;
        if (inside && fmax) atomicMax(collect + em + (collect_cols ? n0 + lane : row), fmax);
      }
      if (row >= rows) listed = 0;
      if (cols - n0 < 16) listed &= (1u << (cols - n0)) - 1u;
      if (__any_sync(0xffffffffu, listed != 0)) {
        const int p = u * kSlParts + warp - kFirstDrainWarp;
        uint32_t w = 0;
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          const uint32_t x = __ballot_sync(0xffffffffu, listed >> c & 1u);
          w = lane == c ? x : w;
        }
        if (lane < 16) fix.mask[p * 16 + lane] = w;
        const bool force = __any_sync(0xffffffffu, large);
        if (lane == 0) fix.list[atomicAdd(fix.count, 1)] = force ? p | kSlForce : p;
      }
      __syncwarp();
    }
  }
  grid_next();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(kTmemCols)
                 : "memory");
}

// ---- listed elements ---------------------------------------------------------------
// One CTA per listed part (32 rows x 16 columns) at a time.  More than a few elements:
// a first pass forms S = sum |a| |b| of the whole part relative to the scales, on the
// FP32 pipe (truncated operands: a lower bound to K 2^-24, what is below 2^-60 of a
// scale taken as that); those whose S reaches the bound are done, and those whose S
// is zero, since every product then has a factor zero.  The others are formed by a
// warp each, or by several, its lanes over k, or, where they are many, by the part's
// FP64 sums.  Empty lists cost the launch.  XXZ operator m = 512, plain form
// 220 us: a site tensor log-uniform over 40 decades, nearly all elements formed, 695 us
// with a warp an element alone and 461 so; one with 2 % of its elements not zero, 1187
// and 615; one with normal elements 113 both ways.
constexpr int kFixThreads = 256, kFixWarps = kFixThreads / 32;
constexpr int kFixFew = 16, kFixMany = 96;
constexpr int kFixK = 32;
constexpr int kFixCtas = 4 * 152;

// |x| / 2^(e - 1023) truncated, at least 2^-60 unless zero; Inf beyond the range
__device__ __forceinline__ float part_of(double x, int e) {
  const int f = exponent_of(x);
  if ((__double_as_longlong(x) << 1) == 0ll) return 0.f;
  return f == 0 || f - e < -60 ? 0x1p-60f : f - e > 127 ? INFINITY : fabsf(float_of(x, e));
}

// acc + a b, with what its roundings leave added to lo (Ogita, Rump and Oishi, 2005).
__device__ __forceinline__ double dot2(double a, double b, double acc, double& lo) {
  const double p = __dmul_rn(a, b), e = fma(a, b, -p);
  const double s = __dadd_rn(acc, p), z = __dadd_rn(s, -acc);
  lo += __dadd_rn(__dadd_rn(acc, -__dadd_rn(s, -z)), __dadd_rn(p, -z)) + e;
  return s;
}

// acc[h] = sum of the segments' products for row lane, column warp + 8 h of a part, or
// (SIZE) of their magnitudes relative to the scales.
template <bool SIZE, class T>
__device__ __forceinline__ void part_sums(const SlUnit& un, const SlSeg* __restrict__ segs, const double* A,
                                          const double* B, const SlSource& src, const int32_t* d, int row0,
                                          int n0, const int* s_fa, const int* s_fb, T (*sa)[33], T (*sb)[16],
                                          T (&acc)[2]) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  acc[0] = acc[1] = (T)0;
  for (int g = 0; g < un.nseg; ++g) {
    const SlSeg q = segs[un.seg0 + g];
    const double cf = SIZE ? q.scale * src.scale : q.scale;
    const int ce = exponent_of(cf);
    // (a subnormal coefficient: no S, the elements are formed)
    const T w = !SIZE ? (T)cf : cf == 0.0 ? (T)0 : ce == 0 ? (T)NAN : (T)part_of(cf, ce);
    T part[2] = {(T)0, (T)0}, low[2] = {(T)0, (T)0};
    for (int k0 = 0; k0 < q.K; k0 += kFixK) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int e = tid + i * kFixThreads;
        const int r = src.ta ? e & 31 : e >> 5, k = src.ta ? e >> 5 : e & 31;
        double x = 0.0;
        int dk = 0;
        if (row0 + r < un.rows && k0 + k < q.K) {
          const int64_t m = un.m0 + row0 + r, kk = k0 + k;
          x = src.ta ? A[q.offA + kk * q.lda + m] : A[q.offA + m * q.lda + kk];
          if (SIZE && q.d0 >= 0) dk = src.sign * d[q.d0 + kk];
        }
        sa[k][r] = SIZE ? (T)part_of(x, s_fa[r] - (ce - 1023) - dk) : (T)x;
      }
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int e = tid + i * kFixThreads;
        const int c = src.tb ? e >> 5 : e & 15, k = src.tb ? e & 31 : e >> 4;
        double x = 0.0;
        int dk = 0;
        if (n0 + c < un.cols && k0 + k < q.K) {
          const int64_t n = un.n0 + n0 + c, kk = k0 + k;
          x = src.tb ? B[q.offB + n * q.ldb + kk] : B[q.offB + kk * q.ldb + n];
          if (SIZE && q.d0 >= 0) dk = -src.sign * d[q.d0 + kk];
        }
        sb[k][c] = SIZE ? (T)part_of(x, s_fb[c] - dk) : (T)x;
      }
      __syncthreads();
      // (columns beyond the segment are zero.)  The 32 terms in four sums, and their sum
      // into the total with its rounding kept
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        T r[4] = {(T)0, (T)0, (T)0, (T)0};
#pragma unroll
        for (int k = 0; k < kFixK; ++k) r[k & 3] = fma(sa[k][lane], sb[k][warp + 8 * h], r[k & 3]);
        const T t = (r[0] + r[1]) + (r[2] + r[3]), sum = part[h] + t, z = sum - part[h];
        if (!SIZE) low[h] += (part[h] - (sum - z)) + (t - z);
        part[h] = sum;
      }
      __syncthreads();
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (!SIZE && fabs(low[h]) < (T)1e308) part[h] += low[h];      // (Inf and NaN: the plain sum)
      acc[h] = fma(w, part[h], acc[h]);
    }
  }
}

__global__ void __launch_bounds__(kFixThreads, 4)
    fix_kernel(const SlUnit* __restrict__ units, const SlSeg* __restrict__ segs, const SlFix fix,
               const int32_t* eA, const int32_t* eB, const __grid_constant__ SlSource src, double* C,
               int32_t* collect, int collect_cols, const int32_t* d) {
  grid_next();
  grid_wait();
  __shared__ union {
    struct { double a[kFixK][33], b[kFixK][16]; } d;
    struct { float a[kFixK][33], b[kFixK][16]; } f;
  } tile;
  __shared__ uint32_t mask[16];
  __shared__ int s_fa[32], s_fb[16];
  __shared__ double s_sum[kFixWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int count = *fix.count, mine = fix.list[blockIdx.x];   // (the list has an entry for every CTA)
  for (int it = blockIdx.x; it < count; it += gridDim.x) {
    const int entry = it == (int)blockIdx.x ? mine : fix.list[it], p = entry & ~kSlForce;
    const bool force = (entry & kSlForce) != 0;
    const SlUnit un = units[p / kSlParts];
    const int w = p % kSlParts, row0 = ((w + kFirstDrainWarp) & 3) * 32, n0 = (w >> 2) * 16;
    __syncthreads();                        // (the part before is done)
    if (tid < 16) mask[tid] = fix.mask[p * 16 + tid];
    __syncthreads();
    const double* A = un.sel ? src.A1 : src.A;
    const double* B = un.sel ? src.B1 : src.B;
    double* Cp = C + un.offC + (int64_t)row0 * un.ldc + n0;
    // the element's exponent among the scales of the output as a later operand
    auto keep = [&](int r, int c, double v) {
      if (un.em < 0) return;
      const int f = scale_of(v, un.d0 >= 0 ? d[un.d0 + n0 + c] : 0);
      if (f) atomicMax(collect + un.em + (collect_cols ? n0 + c : row0 + r), f);
    };
    // this lane's column of the mask, and how many elements it and those before it list
    uint32_t word = 0;
    int upto = 0;
    const auto listed = [&]() {
      word = lane < 16 ? mask[lane] : 0u;
      upto = __popc(word);
#pragma unroll
      for (int o = 1; o < 16; o *= 2) {
        const int v = __shfl_up_sync(0xffffffffu, upto, o);
        if (lane >= o) upto += v;
      }
      return __shfl_sync(0xffffffffu, upto, 15);
    };
    int total = listed();
    if (total > kFixFew && !force) {
      // S of row lane, columns warp and warp + 8
      if (tid < 16) s_fb[tid] = n0 + tid < un.cols ? eB[un.eb + n0 + tid] + 1 - kSlBias : 0;
      if (warp == 1) s_fa[lane] = row0 + lane < un.rows ? eA[un.ea + row0 + lane] + un.shift + 1 - kSlBias : 0;
      __syncthreads();
      float size[2];
      part_sums<true, float>(un, segs, A, B, src, d, row0, n0, s_fa, s_fb, tile.f.a, tile.f.b, size);
      const float least = (float)un.least * 0x1p-20f;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = warp + 8 * h;
        const bool in = (mask[c] >> lane & 1u) != 0;
        // (rows and columns with Inf or NaN have no scale)
        const bool special = s_fa[lane] > kSlSpecial / 2 || s_fb[c] > kSlSpecial / 2;
        const bool form = in && (special || !(size[h] == 0.f || (size[h] >= least && size[h] < 1e30f)));
        if (in && !form) keep(lane, c, Cp[(int64_t)lane * un.ldc + c]);
        const uint32_t left = __ballot_sync(0xffffffffu, form);
        __syncwarp();
        if (lane == 0) mask[c] = left;
      }
      __syncthreads();
      total = listed();
    }
    if (total > kFixMany && !force) {
      double sum[2];
      part_sums<false, double>(un, segs, A, B, src, d, row0, n0, s_fa, s_fb, tile.d.a, tile.d.b, sum);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = warp + 8 * h;
        if (mask[c] >> lane & 1u) {
          const double v = src.scale * sum[h];
          Cp[(int64_t)lane * un.ldc + c] = v;
          keep(lane, c, v);
        }
      }
      continue;
    }
    // `ways` warps an element, each some of its segments
    const int ways = total > 4 ? 1 : total > 2 ? 2 : total > 1 ? 4 : 8;
    const int way = warp % ways;
    for (int e0 = 0; e0 < total; e0 += kFixWarps / ways) {
      const int e = e0 + warp / ways;
      const int at = min(e, total - 1);
      const int c = __ffs(__ballot_sync(0xffffffffu, upto > at)) - 1;
      uint32_t bits = __shfl_sync(0xffffffffu, word, c);
      for (int left = at - (__shfl_sync(0xffffffffu, upto, c) - __popc(bits)); left > 0; --left) bits &= bits - 1u;
      const int r = __ffs(bits) - 1;
      const int64_t m = un.m0 + row0 + r, n = un.n0 + n0 + c;
      double acc = 0.0, rest = 0.0;
      for (int g = e < total ? way : un.nseg; g < un.nseg; g += ways) {
        const SlSeg q = segs[un.seg0 + g];
        const double* a = A + q.offA + (src.ta ? m : m * q.lda);
        const double* b = B + q.offB + (src.tb ? n * q.ldb : n);
        const int64_t da = src.ta ? q.lda : 1, db = src.tb ? 1 : q.ldb;
        double s0 = 0.0, l0 = 0.0;
        if (force) {
          for (int k = lane; k < q.K; k += 32) s0 = dot2(a[k * da], b[k * db], s0, l0);
          acc = dot2(q.scale, s0, acc, rest);
          rest = fma(q.scale, l0, rest);
        } else {
#pragma unroll 4
          for (int k = lane; k < q.K; k += 32) s0 = fma(a[k * da], b[k * db], s0);
          acc = fma(q.scale, s0, acc);
        }
      }
      if (fabs(rest) < 1e308) acc += rest;      // (Inf and NaN: the plain sum)
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (ways > 1) {
        __syncthreads();
        if (lane == 0) s_sum[warp] = acc;
        __syncthreads();
        for (int x = 1; x < ways; ++x) acc += s_sum[min(warp + x, kFixWarps - 1)];
      }
      if (lane == 0 && way == 0 && e < total) {
        const double v = src.scale * acc;
        Cp[(int64_t)r * un.ldc + c] = v;
        keep(r, c, v);
      }
    }
  }
}

// ---- slicing -----------------------------------------------------------------------
// One CTA per 8 rows of a scale group (the packed blocks that share row
// scales; of several row groups where there are few chunks: with idle warps the
// kernel was at 20 % of its issue rate, XXZ m = 512 operator 23 us): the largest exponent of every row over all blocks of the group,
// then the slices.  A warp handles 8 rows x 64 k of one block at a time, lane l
// k = 2 l and 2 l + 1 of every row, so that the reads of a row and the writes
// of a slice's row are whole 128-byte lines; blocks stored with k as the slow
// index go through shared memory.  The elements of a warp's first tile stay in
// registers between the two passes, any further tile is read again (from L2).  Integer arithmetic only: the significand is shifted to the row
// scale and cut into digits.  All operands of a stage that are at hand are
// sliced by one launch.

// A coefficient: |c| = m 2^(f - 1086) with its significand m normalised to 64 bits
// (a subnormal one too).
struct Coef {
  unsigned long long m;
  int f;                  // exponent field (below 1 for a subnormal)
  bool pow2, neg, bad;
};
__device__ __forceinline__ Coef make_coef(double c) {
  Coef r;
  const unsigned long long b = (unsigned long long)__double_as_longlong(c);
  int f = (int)((b >> 52) & 0x7FF);
  unsigned long long m = b << 12 >> 1;               // (bit 63: the leading one)
  r.neg = (b >> 63) != 0;
  r.bad = f == 0x7FF;
  if (f) {
    m |= 1ull << 63;
  } else {
    const int z = __clzll((long long)m);             // 64 for a zero
    f = 1 - z;
    m = z < 64 ? m << z : 0ull;
  }
  r.pow2 = m == (1ull << 63);
  r.m = m;
  r.f = f;
  return r;
}

// Effective exponent field of coef * x 2^d, which is below 2^(field - 1022); kMinField
// for a zero.
constexpr int kMinField = -1000000;
__device__ __forceinline__ int eff_field(double x, const Coef& c, int d) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int f = (int)((b >> 52) & 0x7FF);
  if (f == 0x7FF) return kSlSpecial;
  if ((b << 1) == 0ull || c.m == 0ull) return kMinField;
  return (f ? f : 1) + c.f + d - (c.pow2 ? 1023 : 1022);
}

// The eight digits of coef * x 2^d relative to the row field F, biased by 256 each:
// digit 0 (10 bits) returned, digits 1-7 in *low, digit i in bits 63 - 9 i ...  The
// significand (of the product: its upper 64 bits) is shifted to the 71 bits below
// 2^(F - 1022).
__device__ __forceinline__ uint32_t digits(double x, const Coef& c, int d, int F, unsigned long long* low) {
  constexpr unsigned long long kBias = (256ull << 54) | (256ull << 45) | (256ull << 36) |
                                       (256ull << 27) | (256ull << 18) | (256ull << 9) | 256ull;
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  int f = (int)((b >> 52) & 0x7FF);
  unsigned long long m = b & 0xFFFFFFFFFFFFFull;
  if (f) {
    m = (m | 1ull << 52) << 11;
  } else {
    const int z = __clzll((long long)m);
    m = z < 64 ? m << z : 0ull;
    f = 12 - z;
  }
  if (!c.pow2) m = __umul64hi(m, c.m);
  const int s = F - (f + c.f + d - (c.pow2 ? 1023 : 1022));      // v = m 2^7 >> s
  unsigned long long lo = 0;
  uint32_t hi = 0;
  if (s <= 7) {
    const int l = 7 - max(s, 0);
    lo = m << l;
    hi = (uint32_t)((m >> 32) >> (32 - l));                        // l <= 7
  } else if (s < 72) {
    const unsigned long long t = m >> (s - 8);                     // to nearest, half away from zero
    lo = (t >> 1) + (t & 1ull);
  }
  if (((b >> 63) != 0) != c.neg) {
    lo = 0ull - lo;
    hi = ~hi + (lo == 0ull ? 1u : 0u);
  }
  lo += kBias;
  hi += 128u + (lo < kBias ? 1u : 0u);
  *low = lo;
  return hi << 1 | (uint32_t)(lo >> 63);
}

constexpr int kTRow = 66;      // doubles per row of a transposed tile (64 + 2 pad)

// x[2 r + h] = element (r0 + r, 64 c + 2 lane + h) of a block (0 outside its nr
// rows and K columns); tile: the warp's shared memory.
__device__ __forceinline__ void load_tile(const double* src, int64_t ld, int K, int trans,
                                          int nr, int c, int lane, double* tile, double (&x)[16]) {
  const int k = c * 64 + 2 * lane;
  if (!trans) {
    const double* p = src + k;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      x[2 * r] = r < nr && k < K ? p[r * ld] : 0.0;
      x[2 * r + 1] = r < nr && k + 1 < K ? p[r * ld + 1] : 0.0;
    }
  } else {
    const double* p = src + (lane & 7);
    double v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int kk = c * 64 + 4 * i + (lane >> 3);
      v[i] = (lane & 7) < nr && kk < K ? p[kk * ld] : 0.0;
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 16; ++i) tile[(lane & 7) * kTRow + 4 * i + (lane >> 3)] = v[i];
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      x[2 * r] = tile[r * kTRow + 2 * lane];
      x[2 * r + 1] = tile[r * kTRow + 2 * lane + 1];
    }
  }
}

// The digits of row r of a tile (its scale f; zero: no digits): this lane's
// pair of k, 4 bytes of the swizzled 16-byte piece lane / 4 of every slice.
__device__ __forceinline__ void store_row(uint16_t* base, int64_t slice, int r, double x0, double x1,
                                          const Coef& cf, int2 d, bool zero, int f, int lane) {
  uint16_t* row = base + r * 64 + (((lane >> 2) ^ r) << 3) + 2 * (lane & 3);
  if (zero) {                            // (the same for the whole warp)
#pragma unroll
    for (int i = 0; i < kSlices; ++i) *reinterpret_cast<uint32_t*>(row + i * slice) = 0u;
    return;
  }
  unsigned long long d0, d1;
  const uint32_t t0 = digits(x0, cf, d.x, f, &d0);
  const uint32_t t1 = digits(x1, cf, d.y, f, &d1);
#pragma unroll
  for (int i = 0; i < kSlices; ++i) {
    // digit + 256 in 0 .. 512: as FP16, 1024 + (digit + 256) has these bits
    // exactly; one packed subtraction of 1280 leaves the digits
    const uint32_t f0 = i == 0 ? t0 : (uint32_t)(d0 >> (63 - 9 * i)) & 0x1FFu;
    const uint32_t f1 = i == 0 ? t1 : (uint32_t)(d1 >> (63 - 9 * i)) & 0x1FFu;
    const uint32_t hw = (f0 | (f1 << 16)) | 0x64006400u;
    uint32_t res;
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(res) : "r"(hw), "r"(0x65006500u));
    *reinterpret_cast<uint32_t*>(row + i * slice) = res;
  }
}

// The member of a group that holds its chunk t: lanes compare 32 members at a time
// (a walk would wait for one table entry after the other).
__device__ __forceinline__ int member_of(const SlMember* __restrict__ m, int nm, int t, int lane) {
  int n = 0;
  for (int b = 0; b < nm; b += 32) {
    const bool le = b + lane < nm && m[b + lane].t0 <= t;
    const int c = __popc(__ballot_sync(0xffffffffu, le));
    n += c;
    if (c < 32) break;
  }
  return n - 1;
}

constexpr int kSliceWarps = 8;
__global__ void __launch_bounds__(32 * kSliceWarps, 3)
    slice_kernel(const SlGroup* __restrict__ groups, const int32_t* __restrict__ cta_group,
                 const SlMember* __restrict__ members,
                 const __grid_constant__ SlOperands ops) {
  grid_next();
  grid_wait();
  __shared__ int smax[8 * 8];                        // of up to eight row groups
  __shared__ double tr[kSliceWarps * 8 * kTRow];
  const int cta = (int)blockIdx.x;
  const SlGroup gr = groups[cta_group[cta]];
  const SlOperand op = ops.op[gr.which];
  const SlMember* mem = members + gr.m0;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // the warp's row group, and its place among the `nw` warps of that group
  const int nw = kSliceWarps / gr.per, sub = warp / nw, wi = warp % nw;
  const int r0 = ((cta - gr.cta0) * gr.per + sub) * 8, nr = min(8, gr.R - r0);   // (<= 0: padding)
  int* gmax = smax + 8 * sub;
  for (int i = (int)(blockIdx.x * blockDim.x + threadIdx.x); i < ops.nclear; i += (int)(gridDim.x * blockDim.x))
    ops.clear[i] = 0;
  if (blockIdx.x == 0 && (int)threadIdx.x < ops.nfix) ops.fix[threadIdx.x] = 0;
  if (threadIdx.x < 64) smax[threadIdx.x] = kMinField;
  __syncthreads();
  auto load = [&](const SlMember& mb, int t, double (&x)[16]) {
    load_tile(op.src + mb.src + (mb.trans ? (int64_t)r0 : (int64_t)r0 * mb.ld), mb.ld, mb.K, mb.trans, nr,
              t - mb.t0, lane, tr + warp * 8 * kTRow, x);
  };
  // the grading of this lane's two k
  auto grading = [&](const SlMember& mb, int t) {
    const int k = (t - mb.t0) * 64 + 2 * lane;
    int2 d = make_int2(0, 0);
    if (mb.d0 >= 0 && op.d) {
      if (k < mb.K) d.x = op.sign * op.d[mb.d0 + k];
      if (k + 1 < mb.K) d.y = op.sign * op.d[mb.d0 + k + 1];
    }
    return d;
  };
  double x[16];
  if (nr > 0) {
    int mx[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) mx[r] = kMinField;
    // the warp's chunks, the last one first: the first stays in registers
    const int last = gr.nt > wi ? wi + (gr.nt - 1 - wi) / nw * nw : -1;
    for (int t = last; t >= 0; t -= nw) {
      const SlMember mb = mem[member_of(mem, gr.nm, t, lane)];
      const Coef cf = make_coef(mb.coef * op.scale);
      const int2 d = grading(mb, t);
      load(mb, t, x);
#pragma unroll
      for (int e = 0; e < 16; ++e)
        mx[e >> 1] = max(mx[e >> 1], cf.bad ? kSlSpecial : eff_field(x[e], cf, e & 1 ? d.y : d.x));
    }
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int w = __reduce_max_sync(0xffffffffu, mx[r]);
      if (lane == r && w != kMinField) atomicMax(&gmax[r], w);
    }
  }
  __syncthreads();
  if (wi == 0 && lane < nr) {
    const int v = gmax[lane];
    op.scales[gr.e0 + r0 + lane] = v == kMinField ? 0 : v == kSlSpecial ? v : v + kSlBias;
  }
  if (r0 >= 8 * gr.R8) return;
  for (int t = wi; t < gr.nt; t += nw) {
    const SlMember mb = mem[member_of(mem, gr.nm, t, lane)];
    const Coef cf = make_coef(mb.coef * op.scale);
    const int2 d = grading(mb, t);
    if (t != wi || nr <= 0) load(mb, t, x);
    uint16_t* base = op.out + mb.dst + ((int64_t)(t - mb.t0) * kSlices * gr.R8 + (r0 >> 3)) * kSlTile;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int f = gmax[r];             // zero rows and rows with Inf or NaN have no digits
      store_row(base, (int64_t)gr.R8 * kSlTile, r, x[2 * r], x[2 * r + 1], cf, d,
                f == kMinField || f == kSlSpecial, f + gr.shift, lane);
    }
  }
}

// Grading.  The rows of a site tensor carry the Schmidt weights of the bond that the
// product sums over; in the environment's identity channels only one term of a sum is
// not zero, and the terms of small weight would be held with few digits beside the
// others of their column.  So the site tensor's row k is taken as 2^-d_k and the
// environment's column as 2^d_k, exactly, with d_k the exponent of the largest element
// (of a sample) of the site tensor at k; and in the same way the stage-2 output of H_eff, whose
// columns carry the weights of the other bond, and the second environment.  (With any d the results are right; without one, the
// fix launch would form most of a graded tensor's copies.)  A sample of 32 elements a
// block makes it one load latency and a little: 3 us.
__global__ void __launch_bounds__(256)
    grade_kernel(const SlGrade* __restrict__ items, const SlView* __restrict__ views, const double* src,
                 int32_t* d) {
  grid_next();
  grid_wait();
  __shared__ int best[32];
  const SlGrade it = items[blockIdx.x];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x < 32) best[threadIdx.x] = 0;
  __syncthreads();
  // (32 elements of every view and k are enough to see the weights)
  for (int v = 0; v < it.nv; ++v) {
    const SlView w = views[it.v0 + v];
    double x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = w.trans ? warp + 8 * i : lane;
      const int64_t r = (int64_t)(w.trans ? lane : warp + 8 * i) * max(w.R, 32) / 32;
      x[i] = k < it.nk && r < w.R ? src[w.src + (w.trans ? k * (int64_t)w.ld + r : r * w.ld + k)] : 0.0;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int f = exponent_of(x[i]);
      if (w.trans) {
        const int m = __reduce_max_sync(0xffffffffu, f);
        if (lane == 0) atomicMax(&best[warp + 8 * i], m);
      } else if (f) {
        atomicMax(&best[lane], f);
      }
    }
  }
  __syncthreads();
  if ((int)threadIdx.x < it.nk) {
    const int f = best[threadIdx.x];
    d[it.d0 + threadIdx.x] = f == 0 || f == 0x7FF ? 0 : f - 1022;
  }
}

// Known row scales (the products that wrote the blocks collected them): one
// pass, a warp per tile.
__global__ void __launch_bounds__(256)
    slice_known_kernel(const SlPiece* __restrict__ pieces, int npieces,
                       const int32_t* __restrict__ first, int ntiles, const double* src,
                       uint16_t* out, const int32_t* scales, const int32_t* d) {
  grid_next();
  grid_wait();
  __shared__ double tr[8][8 * kTRow];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int t = (int)blockIdx.x * 8 + warp;
  if (t >= ntiles) return;
  int pi = first[blockIdx.x];
  while (pi + 1 < npieces && pieces[pi + 1].tile0 <= t) ++pi;
  const SlPiece p = pieces[pi];
  const int local = t - p.tile0, c = local / p.R8, g = local - c * p.R8;
  const int r0 = g * 8, nr = min(8, p.R - r0);
  const int fl = lane < nr ? scales[p.e0 + r0 + lane] : 0;
  const int k = c * 64 + 2 * lane;
  int2 dk = make_int2(0, 0);
  if (p.d0 >= 0) {
    if (k < p.K) dk.x = -d[p.d0 + k];
    if (k + 1 < p.K) dk.y = -d[p.d0 + k + 1];
  }
  double x[16];
  load_tile(src + p.src + (p.trans ? (int64_t)r0 : (int64_t)r0 * p.ld), p.ld, p.K, p.trans, nr, c, lane,
            tr[warp], x);
  const Coef cf{1ull << 63, 1023, true, false, false};     // no coefficient
  uint16_t* base = out + p.dst + ((int64_t)c * kSlices * p.R8 + g) * kSlTile;
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int f = __shfl_sync(0xffffffffu, fl, r);
    store_row(base, (int64_t)p.R8 * kSlTile, r, x[2 * r], x[2 * r + 1], cf, dk, f == 0 || f == kSlSpecial,
              f - kSlBias + p.shift, lane);
  }
}

}  // namespace

void launch_slice(const SlGroup* groups, const int32_t* cta_group, int nctas,
                  const SlMember* members, const SlOperands& ops, cudaStream_t st) {
  if (nctas <= 0) return;
  count_launch();
  launch_chain(slice_kernel, nctas, 32 * kSliceWarps, 0, st, groups, cta_group, members, ops);
}

void launch_grade(const SlGrade* items, int nitems, const SlView* views, const double* src, int32_t* d,
                  cudaStream_t st) {
  if (nitems <= 0) return;
  count_launch();
  launch_chain(grade_kernel, nitems, 256, 0, st, items, views, src, d);
}

void launch_slice_known(const SlPiece* pieces, int npieces, const int32_t* first, int ntiles,
                        const double* src, uint16_t* out, const int32_t* scales, const int32_t* d,
                        cudaStream_t st) {
  if (ntiles <= 0) return;
  count_launch();
  launch_chain(slice_known_kernel, (ntiles + 7) / 8, 256, 0, st, pieces, npieces, first, ntiles, src, out, scales, d);
}

void launch_gemm_sliced(const SlTables& t, const uint16_t* pA, const uint16_t* pB,
                        const int32_t* eA, const int32_t* eB, const SlSource& src, double* C,
                        int32_t* collect, bool collect_cols, const int32_t* d, const SlFix& fix, int* err,
                        uint64_t wait_ns, cudaStream_t st) {
  if (t.ncta <= 0) return;
  // the shared-memory limit is a per-device attribute of the kernel
  static std::atomic<uint64_t> done{0};
  int dev = 0;
  cudaGetDevice(&dev);
  const uint64_t bit = dev >= 0 && dev < 64 ? (1ull << dev) : 0ull;
  if (!bit || !(done.load() & bit)) {
    cudaFuncSetAttribute(gemm_sliced_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         kSmemBytes);
    if (bit) done.fetch_or(bit);
  }
  count_launch(2);
  {
    const PlainLaunches plain(!t.chain);
    launch_chain(gemm_sliced_kernel, t.ncta, kThreads, kSmemBytes, st, t, pA, pB, eA, eB, C, collect,
                 collect_cols ? 1 : 0, d, fix, err, wait_ns);
  }
  const int64_t parts = (int64_t)t.nunits * kSlParts;
  launch_chain(fix_kernel, (unsigned)std::min<int64_t>(parts, kFixCtas), kFixThreads, 0, st, t.units, t.segs, fix,
               eA, eB, src, C, collect, collect_cols ? 1 : 0, d);
}

}  // namespace dmrg3s
