// Tensor-core grouped GEMM for sm_103a (tcgen05, TMEM accumulators, bulk
// asynchronous copies), and the kernels that pack its operands.
//
// Operands are FP64 tensors split into x = hi + lo with hi = tf32(x),
// lo = tf32(x - hi) (Ootomo and Yokota's split, 2022) and packed in tiles of
// 8 rows x 32 k in the K-major core-matrix order of the shared-memory matrix
// descriptors (kernels.hpp).  A 128-row slab of one 32-wide k-chunk is then a
// contiguous 16 KB run, so each operand slab reaches shared memory with one
// bulk copy (cp.async.bulk, completion counted in bytes on an mbarrier); no
// thread touches operand data on its way to the tensor core.
//
// Products per k-chunk of one 128 x 128 output tile:
//   kPasses = 1: D_main += A_hi B_hi                                (TF32)
//   kPasses = 3: D_main += A_hi B_hi,  D_corr += A_hi B_lo + A_lo B_hi  (3xTF32)
// The small correction terms keep their own TMEM accumulator over the whole
// K range (their FP32 rounding is ~2^-11 below the result).  The main
// accumulator is drained every kSpan k-chunks (128 k for kSpan = 4: 16
// accumulations of hi * hi products) into double-float registers with
// Knuth's two-sum, so FP32 rounding only ever sees a short span of main
// products.  The 512 TMEM columns hold two main and two correction buffers
// (four main buffers for TF32), so the tensor core can start the next tile
// while the drain warps still finish and store the previous one.  The last N
// tile of a block issues the narrowest MMA width (a multiple of 16) that
// covers it.  No FP64 instruction runs in the kernel (GB300's FP64 rate is
// ~1/1000 of its TF32 rate).
//
// Warp roles of the persistent CTA (one per SM, 384 threads = 3 warpgroups):
//   warp 0     one lane issues the bulk copies into a 3-stage shared-memory ring
//   warp 1     owns the tensor memory; walks the chunks as a whole, an elected
//              lane issues tcgen05.mma and commits each stage and each
//              accumulator to mbarriers
//   warps 2-3  idle (their warpgroup hands its registers to the drain warps)
//   warps 4-11 drain: warp w reads TMEM lanes 32 (w % 4) .. +31 (its row
//              quarter) and columns 64 ((w - 4) / 4) .. +63 of every tile, keeps
//              their double-float sums (128 registers) and stores the tile
//              through a small shared-memory transpose (coalesced rows of
//              (hi, lo) pairs).
// The CTA starts with 168 registers per thread (384 x 168 = 64,512 of the
// SM's 65,536); warpgroup 0 gives up to 56 (setmaxnreg.dec) and the two drain
// warpgroups take 224 (setmaxnreg.inc): 128 x 56 + 256 x 224 = 64,512.
// Units (output tiles) come in one list per CTA, balanced by the planner; the
// copy and MMA warps read the tables one entry ahead.  With that and the elected
// issue the 3xTF32 operator takes 188 us on the m = 2048 cylinder (201 before) and
// 38 us on the m = 512 XXZ chain (41 before).
//
// Every wait on an mbarrier is bounded by the elapsed %globaltimer time given
// by the host.  A wait that runs out sets the device error word and a shared
// abort flag that every other wait also watches; all roles then leave their
// loops, the copy lane waits for its copies still in flight, the MMA lane for
// its products (a fixed one-second limit for these drains), and the CTA frees
// its tensor memory and returns.  Nothing traps.
#include <atomic>
#include <cstdint>

#include "kernels.hpp"
#include "launch.hpp"
#include "tc_common.cuh"

namespace dmrg3s {

namespace {

constexpr int TBM = 128, TBN = 128, TBK = 32;
constexpr int kStages = 3;
constexpr int kThreads = 384;                       // 12 warps
constexpr int kFirstDrainWarp = 4;
constexpr int kDrainWarps = 8;
constexpr int kSlab = TBM * TBK * 4;                // bytes of one 128 x 32 slab (16 KB)
constexpr int kStageBytes = 4 * kSlab;              // A hi, A lo, B hi, B lo
constexpr int kEpiRow = 9;                          // float2 per staged row (8 + 1 pad)
constexpr int kEpiWarp = 4096;                      // bytes of one drain warp's staging (4 atoms)
constexpr int kSmemBytes = kStages * kStageBytes + kDrainWarps * kEpiWarp;
constexpr int kSpanChunks = 4;                      // k-chunks per drain of the main accumulator

// Instruction descriptor of kind::tf32: D = F32, A = B = TF32, both K-major,
// N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t idesc_tf32(int M, int N) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ float to_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

__device__ __forceinline__ void mma_tf32(uint32_t dtmem, uint64_t ad, uint64_t bd, uint32_t idesc,
                                         uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
      "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
      : "memory");
}

// Knuth's two-sum: (s, e) with s + e = a + b exactly.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

template <int kPasses, int kSpan, bool kPackedOut>
__global__ void __launch_bounds__(kThreads, 1)
    gemm_tc_kernel(const TcUnit* __restrict__ units, const int32_t* __restrict__ cta_start,
                   const GemmTask* __restrict__ tasks,
                   const TcSeg* __restrict__ segs, const float* Ahi,
                   const float* Alo, const float* Bhi,
                   const float* Blo, float* Chi,
                   float* Clo, int* err, uint64_t wait_ns) {
  extern __shared__ __align__(1024) unsigned char smem[];
  constexpr bool kLo = kPasses == 3;
  constexpr uint32_t kTmemCols = 512;
  constexpr int kMain = kLo ? 2 : 4;                 // main buffers of 128 columns
  constexpr uint32_t kCorrCol = kMain * TBN;         // two correction buffers (3xTF32)
  __shared__ __align__(8) uint64_t full[kStages], empty[kStages];
  __shared__ __align__(8) uint64_t mfull[kMain], mempty[kMain], cfull[2], cempty[2], done;
  __shared__ uint32_t tmem_base;
  __shared__ volatile int abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < kMain; ++b) {
      mbar_init(&mfull[b], 1);
      mbar_init(&mempty[b], kDrainWarps);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&cfull[b], 1);
      mbar_init(&cempty[b], kDrainWarps);
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
  const int u_begin = cta_start[blockIdx.x], u_end = cta_start[blockIdx.x + 1];
  if (warp < kFirstDrainWarp) asm volatile("setmaxnreg.dec.sync.aligned.u32 56;" ::: "memory");

  if (warp == 0) {
    // ---------------- bulk-copy producer ----------------
    if (lane == 0) {
      int pend[kStages];
#pragma unroll
      for (int s = 0; s < kStages; ++s) pend[s] = -1;
      uint32_t q = 0;
      bool ok = true;
      // the tables are read one unit and one segment ahead
      int n_tm = 0, n_tn = 0, n_nseg = 0, n_seg0 = 0;
      auto load = [&](int u) {
        const TcUnit un = units[u];
        n_tm = un.tm * 16;
        n_tn = un.tn * 16;
        n_nseg = tasks[un.task].nseg;
        n_seg0 = tasks[un.task].seg0;
      };
      if (u_begin < u_end) load(u_begin);
      for (int u = u_begin; u < u_end && ok; ++u) {
        const int tm16 = n_tm, tn16 = n_tn, nseg = n_nseg, seg0 = n_seg0;
        TcSeg sg_next{};
        if (nseg > 0) sg_next = segs[seg0];
        if (u + 1 < u_end) load(u + 1);
        for (int k = 0; k < nseg && ok; ++k) {
          const TcSeg sg = sg_next;
          if (k + 1 < nseg) sg_next = segs[seg0 + k + 1];
          const int ga = min(16, sg.ra8 - tm16), gb = min(16, sg.rb8 - tn16);
          const uint32_t ba = (uint32_t)ga * 1024u, bb = (uint32_t)gb * 1024u;
          for (int c = 0; c < sg.kc; ++c, ++q) {
            const int st = (int)(q % kStages);
            if (q >= (uint32_t)kStages && !mbar_wait(&empty[st], ((q / kStages) - 1) & 1, wc)) {
              ok = false;
              break;
            }
            unsigned char* base = smem + st * kStageBytes;
            const int64_t oa = sg.pa + ((int64_t)c * sg.ra8 + tm16) * kPackTile;
            const int64_t ob = sg.pb + ((int64_t)c * sg.rb8 + tn16) * kPackTile;
            mbar_expect_tx(&full[st], (ba + bb) * (kLo ? 2u : 1u));
            bulk_g2s(base, Ahi + oa, ba, &full[st]);
            bulk_g2s(base + 2 * kSlab, Bhi + ob, bb, &full[st]);
            if (kLo) {
              bulk_g2s(base + kSlab, Alo + oa, ba, &full[st]);
              bulk_g2s(base + 3 * kSlab, Blo + ob, bb, &full[st]);
            }
            pend[st] = (int)((q / kStages) & 1);
          }
        }
      }
      // copies still in flight must land before the CTA's memory is released
      for (int s = 0; s < kStages; ++s)
        if (pend[s] >= 0) mbar_drain(&full[s], (uint32_t)pend[s]);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    // (the whole warp walks the chunks, an elected lane issues: elect_one)
    const bool one = elect_one();
    const uint32_t tmem_u = __reduce_or_sync(0xffffffffu, tmem);
    const uint32_t s0 = smem_u32(smem);
    uint32_t st = 0, sph = 0, p = 0, uc = 0;
    bool ok = true, ready = false;
    int T_next = 0, n_next = 0;
    auto load = [&](int u) {
      const TcUnit un = units[u];
      T_next = un.nchunks;
      n_next = min(TBN, tasks[un.task].N - un.tn * TBN);
    };
    if (u_begin < u_end) load(u_begin);
    for (int u = u_begin; u < u_end && ok; ++u) {
      const int T = (int)__reduce_or_sync(0xffffffffu, (unsigned)T_next);
      // MMA width: the columns of this tile, rounded up to a multiple of 16
      const uint32_t idesc =
          __reduce_or_sync(0xffffffffu, idesc_tf32(TBM, (n_next + 15) & ~15));
      if (u + 1 < u_end) load(u + 1);
      if (T == 0) continue;
      const uint32_t cb = uc & 1;
      const uint32_t dcorr = tmem_u + kCorrCol + cb * TBN;
      if (kLo && uc >= 2 &&
          !__all_sync(0xffffffffu, mbar_wait(&cempty[cb], ((uc >> 1) - 1) & 1, wc)))
        break;
      uint32_t dmain = 0;
      for (int t = 0; t < T; ++t) {
        const bool span0 = t % kSpan == 0;
        if (span0) {
          const uint32_t mb = p % kMain;
          if (p >= (uint32_t)kMain &&
              !__all_sync(0xffffffffu, mbar_wait(&mempty[mb], ((p / kMain) - 1) & 1, wc))) {
            ok = false;
            break;
          }
          dmain = tmem_u + mb * TBN;
        }
        if (!__all_sync(0xffffffffu, ready) &&
            !__all_sync(0xffffffffu, mbar_wait(&full[st], sph, wc))) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t sah = s0 + st * kStageBytes, sal = sah + kSlab;
        const uint32_t sbh = sah + 2 * kSlab, sbl = sah + 3 * kSlab;
        const uint32_t cur = st;
        if (++st == kStages) {
          st = 0;
          sph ^= 1;
        }
        ready = mbar_test(&full[st], sph);           // the next stage's, while this one is issued
        if (one) {
#pragma unroll
          for (int kk = 0; kk < TBK / 8; ++kk) {     // K = 8 per instruction (32 bytes)
            const uint32_t off = kk * 32;            // 8 k = 32 bytes of the 128-byte line
            mma_tf32(dmain, smem_desc(sah + off), smem_desc(sbh + off), idesc,
                     (span0 && kk == 0) ? 0u : 1u);
            if (kLo) {
              mma_tf32(dcorr, smem_desc(sah + off), smem_desc(sbl + off), idesc,
                       (t == 0 && kk == 0) ? 0u : 1u);
              mma_tf32(dcorr, smem_desc(sal + off), smem_desc(sbh + off), idesc, 1u);
            }
          }
          mma_commit(&empty[cur]);                   // the stage is free once these are done
          if (t % kSpan == kSpan - 1 || t == T - 1)
            mma_commit(&mfull[p % kMain]);           // a span of main products is ready
          if (kLo && t == T - 1) mma_commit(&cfull[cb]);
        }
        __syncwarp();
        if (t % kSpan == kSpan - 1 || t == T - 1) ++p;
      }
      if (!ok) break;
      ++uc;
    }
    // every product issued must finish before the tensor memory is freed
    if (one) {
      mma_commit(&done);
      mbar_drain(&done, 0);
    }
    __syncwarp();
  } else if (warp >= kFirstDrainWarp) {
    // ---------------- drain and epilogue ----------------
    asm volatile("setmaxnreg.inc.sync.aligned.u32 224;" ::: "memory");
    const int quarter = warp & 3, half = (warp - kFirstDrainWarp) >> 2;
    const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
    const uint32_t col0 = (uint32_t)(half * 64);
    float2* stage_out =
        reinterpret_cast<float2*>(smem + kStages * kStageBytes + (warp - kFirstDrainWarp) * kEpiWarp);
    uint32_t p = 0, uc = 0;
    bool ok = true;
    for (int u = u_begin; u < u_end && ok; ++u) {
      const TcUnit un = units[u];
      const GemmTask t = tasks[un.task];
      float ah[64], al[64];
#pragma unroll
      for (int j = 0; j < 64; ++j) {
        ah[j] = 0.f;
        al[j] = 0.f;
      }
      // columns the MMA writes (its width; the rest of the buffer is stale)
      const int nmma = (min(TBN, t.N - un.tn * TBN) + 15) & ~15;
      if (un.nchunks > 0) {
        const int nsp = (un.nchunks + kSpan - 1) / kSpan;
        for (int j = 0; j < nsp; ++j, ++p) {
          const uint32_t mb = p % kMain;
          // one decision per warp: tcgen05.ld is a warp-wide instruction
          if (!__all_sync(0xffffffffu, mbar_wait(&mfull[mb], (p / kMain) & 1, wc))) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            if ((int)col0 + h * 16 >= nmma) break;
            uint32_t v[16];
            tmem_ld16(tmem + lane_off + mb * TBN + col0 + h * 16, v);
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              float s, e;
              two_sum(ah[h * 16 + i], __uint_as_float(v[i]), s, e);
              ah[h * 16 + i] = s;
              al[h * 16 + i] = __fadd_rn(al[h * 16 + i], e);
            }
          }
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(&mempty[mb]);
        }
        if (!ok) break;
        if (kLo) {
          const uint32_t cb = uc & 1;
          if (!__all_sync(0xffffffffu, mbar_wait(&cfull[cb], (uc >> 1) & 1, wc))) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            if ((int)col0 + h * 16 >= nmma) break;
            uint32_t v[16];
            tmem_ld16(tmem + lane_off + kCorrCol + cb * TBN + col0 + h * 16, v);
#pragma unroll
            for (int i = 0; i < 16; ++i)
              al[h * 16 + i] = __fadd_rn(al[h * 16 + i], __uint_as_float(v[i]));
          }
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(&cempty[cb]);
        }
        ++uc;
      }
      const int row0 = un.tm * TBM + quarter * 32;
      const int n0 = un.tn * TBN + half * 64;
      if (kPackedOut) {
        // packed split operand of the next stage: the warp's 32 rows are 4
        // whole 8-row atoms of each 32-wide k-chunk, contiguous in global
        // memory; they are staged in shared memory in the swizzled order
        // (lane = row) and written with one bulk copy per chunk and part
        const int R8 = t.ldc, KC32 = (t.N + 31) / 32 * 32;
        const int g0 = row0 >> 3, ng = min(4, R8 - g0);
        const int r = row0 + lane, rr = lane & 7;
        unsigned char* stg = reinterpret_cast<unsigned char*>(stage_out);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int k0 = n0 + 32 * h;
          if (k0 >= KC32 || ng <= 0) break;
#pragma unroll
          for (int part = 0; part < (kLo ? 2 : 1); ++part) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              float v[4];
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const int kk = 32 * h + 4 * j + i;
                float x = 0.f;
                if (r < t.M && k0 + 4 * j + i < t.N) {
                  const float a = ah[kk], hv = to_tf32(a);
                  // a - hv is exact (hv is a rounded to the 10-bit TF32 mantissa)
                  x = part == 0 ? hv : to_tf32(__fadd_rn(__fsub_rn(a, hv), al[kk]));
                }
                v[i] = x;
              }
              *reinterpret_cast<float4*>(stg + (lane >> 3) * 1024 + rr * 128 + ((j ^ rr) << 4)) =
                  make_float4(v[0], v[1], v[2], v[3]);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) {
              float* dst = (part == 0 ? Chi : Clo) + t.offC + ((int64_t)(k0 >> 5) * R8 + g0) * kPackTile;
              bulk_s2g(dst, stg, (uint32_t)ng * 1024u);
              bulk_wait_read();            // the staging buffer is reused next
            }
            __syncwarp();
          }
        }
      } else {
        // renormalise (hi, lo) and store: 8 columns at a time through the
        // warp's staging rows, written back as rows of 8 consecutive pairs
        float2* C = reinterpret_cast<float2*>(Chi);
#pragma unroll
        for (int c8 = 0; c8 < 64; c8 += 8) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            float s, e;
            two_sum(ah[c8 + i], al[c8 + i], s, e);
            stage_out[lane * kEpiRow + i] = make_float2(s, e);
          }
          __syncwarp();
#pragma unroll
          for (int it = 0; it < 8; ++it) {
            const int r = it * 4 + (lane >> 3), cc = lane & 7;
            const int gm = row0 + r, gn = n0 + c8 + cc;
            if (gm < t.M && gn < t.N)
              C[t.offC + (int64_t)gm * t.ldc + gn] = stage_out[r * kEpiRow + cc];
          }
          __syncwarp();
        }
      }
    }
    if (kPackedOut && lane == 0) bulk_wait_all();   // the tile stores are complete
    __syncwarp();
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

// hi + lo split of a double without FP64 arithmetic (GB300's FP64 pipe would
// bound the packing): hi = x rounded to 11 significant bits (to nearest, ties
// away from zero, from the integer significand), lo = tf32(x - hi) with the
// exact remainder formed from the significand bits.  Returns false for
// values outside the FP32 normal range and for Inf/NaN, which the caller
// splits the plain way.
__device__ __forceinline__ bool split_bits(double x, float& hi, float& lo) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const uint32_t hw = (uint32_t)(b >> 32), lw = (uint32_t)b;
  const int e = (int)((hw >> 20) & 0x7FF);
  const uint32_t sign = hw & 0x80000000u;
  if (e == 0) {                       // zero or an FP64 subnormal (below the FP32 range)
    hi = __uint_as_float(sign);
    lo = 0.f;
    return true;
  }
  const int ef = e - 1023 + 127;
  if (e == 0x7FF || ef <= 0 || ef >= 254) return false;
  const int hm = (int)((hw & 0xFFFFFu) | 0x100000u);      // top 21 significand bits
  const int r = (hm >> 10) + ((hm >> 9) & 1);              // 11 bits, rounded half away
  hi = __uint_as_float(sign | (((uint32_t)ef << 23) + ((uint32_t)(r - 1024) << 13)));
  const int dh = hm - (r << 10);                           // |dh| <= 512
  // (x - hi) / 2^(e - 1075) = dh 2^32 + lw, rounded once to FP32 by the sum
  const float rem = __fadd_rn(__fmul_rn((float)dh, 4294967296.f), __uint2float_rn(lw));
  const float v = ldexpf(rem, e - 1075);
  lo = to_tf32(sign ? -v : v);
  return true;
}

// The block of tile `tile` (blocks in increasing tile0 order), by a whole warp:
// 32 probes a step instead of one (a binary search waits for a dependent load
// per halving).
template <class T>
__device__ __forceinline__ int block_of_tile(const T* b, int n, int tile) {
  const int lane = threadIdx.x & 31;
  int lo = 0, len = n;                 // the block lies in [lo, lo + len)
  while (len > 1) {
    const int step = (len + 31) >> 5;
    const int i = lo + lane * step;
    const bool le = lane * step < len && b[i].tile0 <= tile;
    const int k = __popc(__ballot_sync(0xffffffffu, le)) - 1;
    len = min(step, len - k * step);
    lo += k * step;
  }
  return lo;
}

// One warp per 8 x 32 tile: lane l handles row l / 4 and k = 4 j + l % 4 of
// 16-byte chunk j (j = 0..7), stored at its swizzled position.
__global__ void __launch_bounds__(256)
    pack_kernel(const PackBlock* __restrict__ blocks, int nblocks, int ntiles,
                const double* src, float* hi, float* lo) {
  grid_next();
  grid_wait();
  const int tile = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (tile >= ntiles) return;
  const int lane = threadIdx.x & 31;
  const PackBlock b = blocks[block_of_tile(blocks, nblocks, tile)];
  const int local = tile - b.tile0;                  // tile = (c, g) with local = c R8 + g
  const int c = local / b.R8, g = local - c * b.R8;
  const int rr = lane >> 2, r = g * 8 + rr;
  const int64_t out = b.dst + (int64_t)local * kPackTile + rr * 32 + (lane & 3);
  // a power-of-two scale multiplies the FP32 parts exactly; any other one is
  // applied in FP64 before the split
  const bool f64scale = b.scale != 1.0 && b.pow2 == 0.f;
  const float fs = b.pow2 != 0.f ? b.pow2 : 1.f;
  double v[8];                   // every load before the first store
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int k = c * 32 + j * 4 + (lane & 3);
    v[j] = 0.0;
    if (r < b.R && k < b.K)
      v[j] = b.trans ? src[b.src + (int64_t)k * b.ld + r] : src[b.src + (int64_t)r * b.ld + k];
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    double x = v[j];
    float h, l;
    if (f64scale) x *= b.scale;
    if (!split_bits(x, h, l)) {
      h = to_tf32((float)x);
      l = to_tf32((float)(x - (double)h));
    }
    hi[out + ((j ^ rr) << 2)] = h * fs;
    if (lo) lo[out + ((j ^ rr) << 2)] = l * fs;
  }
}

// Double-float accumulation of a coefficient pair times an input pair.
__device__ __forceinline__ void df_acc(float ch, float cl, float2 x, float& ah, float& al) {
  const float p = __fmul_rn(ch, x.x);
  float pe = __fmaf_rn(ch, x.x, -p);
  pe = __fmaf_rn(ch, x.y, pe);
  pe = __fmaf_rn(cl, x.x, pe);
  float s, e;
  two_sum(ah, p, s, e);
  e = __fadd_rn(e, __fadd_rn(al, pe));
  ah = __fadd_rn(s, e);
  al = __fsub_rn(e, __fsub_rn(ah, s));
}

// Stage 2 into the packed operand of stage 3: one warp per 8 x 32 tile of a
// task's packed output; the value is scale * sum_k coef_k in_k in double-float
// arithmetic, then split hi = tf32(v), lo = tf32(v - hi).
__global__ void __launch_bounds__(256)
    combine_pairs_pack_kernel(const PackOut* __restrict__ outs, int ntasks, int ntiles,
                              const CombTask* __restrict__ tasks, const CombTerm* __restrict__ terms,
                              const float2* in, float* out_hi,
                              float* out_lo, float sh, float sl) {
  grid_next();
  grid_wait();
  const int tile = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (tile >= ntiles) return;
  const int lane = threadIdx.x & 31;
  const int ti = block_of_tile(outs, ntasks, tile);
  const PackOut o = outs[ti];
  const CombTask t = tasks[ti];
  const int local = tile - o.tile0;
  const int c = local / o.R8, g = local - c * o.R8;
  const int rr = lane >> 2, r = g * 8 + rr;
  const int R = o.trans ? t.cols : t.rows, K = o.trans ? t.rows : t.cols;
  const int64_t out = o.dst + (int64_t)local * kPackTile + rr * 32 + (lane & 3);
  const bool scaled = sh != 1.f || sl != 0.f;
#pragma unroll 2
  for (int j = 0; j < 8; ++j) {
    const int k = c * 32 + j * 4 + (lane & 3);
    float h = 0.f, l = 0.f;
    if (r < R && k < K) {
      const int row = o.trans ? k : r, col = o.trans ? r : k;
      float ah = 0.f, al = 0.f;
      for (int m = 0; m < t.nt; ++m) {
        const CombTerm tm = terms[t.t0 + m];
        df_acc(tm.chi, tm.clo, in[tm.offIn + (int64_t)row * tm.ldi + col], ah, al);
      }
      if (scaled) {
        const float xh = ah, xl = al;
        ah = 0.f;
        al = 0.f;
        df_acc(sh, sl, make_float2(xh, xl), ah, al);
      }
      h = to_tf32(ah);
      // ah - h is exact (h is ah rounded to the 10-bit TF32 mantissa)
      l = to_tf32(__fadd_rn(__fsub_rn(ah, h), al));
    }
    out_hi[out + ((j ^ rr) << 2)] = h;
    if (out_lo) out_lo[out + ((j ^ rr) << 2)] = l;
  }
}

template <int P, bool kPacked>
void launch_one(const TcUnit* units, const int32_t* cta_start, int ncta, const GemmTask* tasks,
                const TcSeg* segs, const float* Ah, const float* Al, const float* Bh,
                const float* Bl, float* Chi, float* Clo, int* err, uint64_t wait_ns,
                cudaStream_t st) {
  // the shared-memory limit is a per-device attribute of the kernel
  static std::atomic<uint64_t> done{0};
  int dev = 0;
  cudaGetDevice(&dev);
  const uint64_t bit = dev >= 0 && dev < 64 ? (1ull << dev) : 0ull;
  if (!bit || !(done.load() & bit)) {
    cudaFuncSetAttribute(gemm_tc_kernel<P, kSpanChunks, kPacked>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (bit) done.fetch_or(bit);
  }
  launch_chain(gemm_tc_kernel<P, kSpanChunks, kPacked>, ncta, kThreads, kSmemBytes, st, units, cta_start, tasks, segs, Ah, Al, Bh, Bl, Chi, Clo, err, wait_ns);
}

}  // namespace

void launch_pack(const PackBlock* blocks, int nblocks, int ntiles, const double* src, float* hi,
                 float* lo, cudaStream_t st) {
  if (ntiles <= 0 || nblocks <= 0) return;
  count_launch();
  launch_chain(pack_kernel, (ntiles + 7) / 8, 256, 0, st, blocks, nblocks, ntiles, src, hi, lo);
}

void launch_combine_pairs_pack(const PackOut* outs, int ntasks, int ntiles, const CombTask* tasks,
                               const CombTerm* terms, const float2* in, float* out_hi,
                               float* out_lo, double scale, cudaStream_t st) {
  if (ntiles <= 0 || ntasks <= 0) return;
  count_launch();
  const float sh = (float)scale, sl = (float)(scale - (double)sh);
  launch_chain(combine_pairs_pack_kernel, (ntiles + 7) / 8, 256, 0, st, outs, ntasks, ntiles, tasks, terms, in, out_hi, out_lo, sh, sl);
}

void launch_gemm_tc(int passes, bool packed, const TcUnit* units, const int32_t* cta_start,
                    int ncta, const GemmTask* tasks, const TcSeg* segs, const float* Ahi,
                    const float* Alo, const float* Bhi, const float* Blo, float* Chi, float* Clo,
                    int* err, uint64_t wait_ns, bool chain, cudaStream_t st) {
  if (ncta <= 0) return;
  const PlainLaunches plain(!chain);
  count_launch();
  if (passes == 3) {
    if (packed)
      launch_one<3, true>(units, cta_start, ncta, tasks, segs, Ahi, Alo, Bhi, Blo, Chi, Clo, err,
                          wait_ns, st);
    else
      launch_one<3, false>(units, cta_start, ncta, tasks, segs, Ahi, Alo, Bhi, Blo, Chi, nullptr,
                           err, wait_ns, st);
  } else {
    if (packed)
      launch_one<1, true>(units, cta_start, ncta, tasks, segs, Ahi, Alo, Bhi, Blo, Chi, Clo, err,
                          wait_ns, st);
    else
      launch_one<1, false>(units, cta_start, ncta, tasks, segs, Ahi, Alo, Bhi, Blo, Chi, nullptr,
                           err, wait_ns, st);
  }
}

}  // namespace dmrg3s
