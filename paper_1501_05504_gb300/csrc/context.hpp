// Library context: device, workspace arena, cached device-resident plans.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <memory>
#include <string>
#include <unordered_map>
#include <vector>

#include "dmrg3s.h"
#include "plan.hpp"

namespace dmrg3s {

// Tables of a sliced FP64 stage (SlStage).
struct DeviceSliced {
  SlSeg* segs = nullptr;
  SlUnit* units = nullptr;
  SlChunk* chunks = nullptr;
  uint32_t* words = nullptr;
  int32_t *cta_unit = nullptr, *cta_chunk = nullptr;
};
SlTables sliced_tables(const DeviceSliced& d, const SlStage& s);

// Device copy of the MPO-entry gradient's tables.
struct DeviceGradPlan {
  GradPlan host;
  void* mem = nullptr;
  struct Gemm {
    GemmTile* tiles = nullptr;
    GemmTask* tasks = nullptr;
    GemmSeg* segs = nullptr;
  } g1, gy;
  DotTask* tasks = nullptr;
  DotSeg* segs = nullptr;
  DeviceSliced s;
  SlGroup* sl_groups = nullptr;
  SlMember* sl_members = nullptr;
  int32_t* sl_cta_group = nullptr;
  ~DeviceGradPlan();
};
constexpr size_t kMaxGradPlans = 256;     // cached per context

// Device copy of a plan's task tables.
struct DevicePlan {
  Plan host;
  // the tables of the plain form, and those of the tensor-core and the sliced form once
  // a call has needed them (need_form), each in one allocation
  void *mem = nullptr, *mem_tc = nullptr, *mem_sl = nullptr;
  GemmTile* g1_tiles = nullptr;
  GemmTask* g1_tasks = nullptr;
  GemmSeg* g1_segs = nullptr;
  CombChunk* c2_chunks = nullptr;
  CombTask* c2_tasks = nullptr;
  CombTerm* c2_terms = nullptr;
  GemmTile* g3_tiles = nullptr;
  GemmTask* g3s_tasks = nullptr;     // split-K stage 3 (tensor-core form)
  // tensor-core tables: units, segments and operand packs of stages 1 and 3,
  // and the packed outputs of stage 2
  TcUnit* g1_units = nullptr;
  int32_t* g1_cta = nullptr;
  TcSeg* g1_tsegs = nullptr;
  PackBlock* g1_packA = nullptr;
  PackBlock* g1_packB = nullptr;
  TcUnit* g3s_units = nullptr;
  int32_t* g3s_cta = nullptr;
  TcSeg* g3s_tsegs = nullptr;
  PackBlock* g3s_packA = nullptr;
  PackBlock* g3s_packB = nullptr;
  PackOut* c2_pack = nullptr;
  GemmTask* g12_tasks = nullptr;     // fused stages 1 + 2 of the tensor-core H_eff
  TcUnit* g12_units = nullptr;
  int32_t* g12_cta = nullptr;
  TcSeg* g12_tsegs = nullptr;
  PackBlock* g12_packA = nullptr;
  PackBlock* g12_packB = nullptr;
  CombChunk* c3r_chunks = nullptr;
  CombTask* c3r_tasks = nullptr;
  CombTerm* c3r_terms = nullptr;
  GemmTask* g3_tasks = nullptr;
  GemmSeg* g3_segs = nullptr;
  // sliced FP64 form: stages 1 + 2, stage 3, the sum of its partials
  DeviceSliced s12, s3;
  SlGroup* sl_groups = nullptr;
  SlMember* sl_members = nullptr;
  int32_t* sl_cta_group = nullptr;
  SlGrade* grades = nullptr;
  SlView* views = nullptr;
  SlPiece* t2 = nullptr;
  int32_t* t2_first = nullptr;
  CombChunk* s3r_chunks = nullptr;
  CombTask* s3r_tasks = nullptr;
  CombTerm* s3r_terms = nullptr;
  ~DevicePlan();
};

// Per-kernel timing with CUDA events recorded on the launching stream around
// every grouped-GEMM and combination launch while profiling is on.
enum ProfKind {
  kProfGemm = 0,        // grouped-GEMM launches
  kProfCombine = 1,     // MPO combination launches
  kProfEig = 2,         // phases of a local update: eigensolver
  kProfExpand = 3,      //   expansion term
  kProfSvd = 4,         //   gather of M~, per-sector SVD, selection, new tensors
  kProfRemainder = 5,   //   S V^dagger (or U S) into the neighbour
  kProfEnv = 6,         //   environment update
  kProfEnergy = 7,      //   energy after truncation
  kProfAuxGemm = 8,     // FP64 grouped GEMMs outside H_eff/expansion/environment:
                        //   the remainder of the truncation, the MPO-entry gradient
  kProfJacobi = 9,      // one Jacobi sweep of the truncation's SVD (all its round launches)
  kProfKinds = 10
};
struct ProfRec {
  int kind;
  cudaEvent_t e0, e1;
  double flops, bytes;
  int64_t launches = 1;   // kernel launches between e0 and e1
};
struct Profiler {
  bool on = false;
  std::vector<ProfRec> recs;
  std::vector<cudaEvent_t> pool;
  cudaEvent_t take() {
    cudaEvent_t e;
    if (!pool.empty()) {
      e = pool.back();
      pool.pop_back();
    } else {
      cudaEventCreate(&e);
    }
    return e;
  }
  int begin(int kind, double flops, double bytes, cudaStream_t st) {
    ProfRec r{kind, take(), take(), flops, bytes};
    cudaEventRecord(r.e0, st);
    recs.push_back(r);
    return (int)recs.size() - 1;
  }
  void end(int id, cudaStream_t st) { cudaEventRecord(recs[id].e1, st); }
  void reset() {
    for (auto& r : recs) {
      pool.push_back(r.e0);
      pool.push_back(r.e1);
    }
    recs.clear();
  }
  ~Profiler() {
    reset();
    for (auto e : pool) cudaEventDestroy(e);
  }
};

// FNV-1a fingerprint builder used as the plan-cache key.
struct Hasher {
  uint64_t h = 1469598103934665603ull;
  void bytes(const void* p, size_t n) {
    const unsigned char* c = (const unsigned char*)p;
    for (size_t i = 0; i < n; ++i) {
      h ^= c[i];
      h *= 1099511628211ull;
    }
  }
  template <class T>
  void pod(const T& v) { bytes(&v, sizeof(T)); }
  template <class T>
  void vec(const std::vector<T>& v) {
    pod(v.size());
    if (!v.empty()) bytes(v.data(), v.size() * sizeof(T));
  }
  void bond(const Bond& b);
  void site(const SiteLayout& s);
  void env(const EnvLayout& e);
  void mpo(const MpoLayout& w);
};

// 128-bit fingerprint of a call's raw arguments (charges, dimensions, channel
// charges, MPO entries; not the data pointers).  A call whose arguments have
// been checked and planned before finds its plan by it, without building the
// layouts again: two multiplicative hashes over 8-byte words, ~1 us for the 7 KB
// of a Hubbard site, where layouts, checks and the plan key take ~30 us.
struct RawKey {
  uint64_t a = 0x243F6A8885A308D3ull, b = 0x13198A2E03707344ull;
  bool ok = true;          // false: malformed arguments (the checked path reports them)
  void word(uint64_t x) {
    a = (a ^ x) * 0x9E3779B97F4A7C15ull;
    a ^= a >> 32;
    b = (b + x) * 0xC2B2AE3D27D4EB4Full;
    b ^= b >> 29;
  }
  void bytes(const void* p, size_t n) {
    if (n && !p) {
      ok = false;
      return;
    }
    word(n);
    const char* c = static_cast<const char*>(p);
    for (; n >= 8; n -= 8, c += 8) {
      uint64_t x;
      std::memcpy(&x, c, 8);
      word(x);
    }
    if (n) {
      uint64_t x = 0;
      std::memcpy(&x, c, n);
      word(x);
    }
  }
  bool range(int64_t v, int64_t lo, int64_t hi) {
    ok = ok && v >= lo && v <= hi;
    return ok;
  }
  void bond(int nsym, const dmrg3s_bond& q) {
    if (!range(nsym, 0, DMRG3S_MAX_NSYM) || !range(q.nsec, 1, 1 << 20)) return;
    word((uint64_t)nsym << 32 | (uint32_t)q.nsec);
    if (nsym) bytes(q.q, sizeof(int32_t) * (size_t)nsym * q.nsec);
    bytes(q.dim, sizeof(int64_t) * (size_t)q.nsec);
  }
  void site(const dmrg3s_site& s) {
    if (!range(s.nsym, 0, DMRG3S_MAX_NSYM) || !range(s.d, 1, 1 << 12)) return;
    word((uint64_t)s.d);
    if (s.nsym) bytes(s.qp, sizeof(int32_t) * (size_t)s.nsym * s.d);
    bond(s.nsym, s.left);
    if (ok) bond(s.nsym, s.right);
  }
  void env(const dmrg3s_env& e) {
    if (!range(e.nsym, 0, DMRG3S_MAX_NSYM) || !range(e.w, 1, 1 << 16)) return;
    word((uint64_t)e.w);
    if (e.nsym) bytes(e.t, sizeof(int32_t) * (size_t)e.nsym * e.w);
    bond(e.nsym, e.bond);
  }
  void mpo(const dmrg3s_mpo_site& m, bool values) {
    if (!range(m.nsym, 0, DMRG3S_MAX_NSYM) || !range(m.d, 1, 1 << 12) || !range(m.wl, 1, 1 << 16) ||
        !range(m.wr, 1, 1 << 16))
      return;
    word((uint64_t)m.d << 32 | (uint32_t)m.nsym);
    word((uint64_t)m.wl << 32 | (uint32_t)m.wr);
    if (m.nsym) {
      bytes(m.qp, sizeof(int32_t) * (size_t)m.nsym * m.d);
      bytes(m.tl, sizeof(int32_t) * (size_t)m.nsym * m.wl);
      bytes(m.tr, sizeof(int32_t) * (size_t)m.nsym * m.wr);
    }
    const size_t n = (size_t)m.d * m.d * m.wl * m.wr;
    if (!m.W) ok = false;
    if (ok && values) bytes(m.W, sizeof(double) * n);
  }
  bool operator==(const RawKey& o) const { return a == o.a && b == o.b; }
};
struct RawKeyHash {
  size_t operator()(const RawKey& k) const { return (size_t)(k.a ^ (k.b << 1)); }
};

constexpr size_t kMaxArgs = 4096;
template <class Map, class Plan>
void remember(Map* m, const RawKey& key, const Plan* p) {
  if (!key.ok) return;
  if (m->size() >= kMaxArgs) m->clear();
  (*m)[key] = p;
}

struct Context {
  Profiler prof;
  int device = 0;
  char* ws = nullptr;           // workspace arena
  size_t ws_bytes = 0;
  double* pinned = nullptr;     // small pinned host buffer for scalar read-backs (64 doubles)
  int* d_err = nullptr;         // device error word latched by bounded waits (tensor-core kernel)
  uint64_t wait_ns = 1000000000ull;   // limit of every bounded device wait (dmrg3s_set_wait_limit)
  cudaStream_t aux = nullptr;   // side stream: the Lanczos tridiagonal solve beside the next product
  cudaEvent_t ev_ready = nullptr, ev_done = nullptr;
  cudaEvent_t ev_lz[3] = {nullptr, nullptr, nullptr};   // Lanczos results of iterations k mod 3
  double* pinned_big = nullptr;   // pinned read-back area of the batched Lanczos (grown on demand)
  size_t pinned_big_n = 0;        // its size in doubles
  std::unordered_map<uint64_t, std::unique_ptr<DevicePlan>> plans;
  std::unordered_map<uint64_t, std::unique_ptr<DeviceGradPlan>> grad_plans;
  // plans by the raw arguments of the calls that use them (entries of `plans`,
  // which live as long as the context; of `grad_plans`, dropped with them).  At most
  // kMaxArgs of each: the MPO's values are among the arguments, and a program that
  // varies them makes a new entry with every call.
  std::unordered_map<RawKey, const DevicePlan*, RawKeyHash> by_args;
  std::unordered_map<RawKey, const DeviceGradPlan*, RawKeyHash> grad_by_args;
  std::string last_error;
};

inline dmrg3s_status fail(Context* c, dmrg3s_status st, const std::string& msg) {
  if (c) c->last_error = msg;
  return st;
}

inline dmrg3s_status use_device(Context* c) {
  int cur = -1;
  if (cudaGetDevice(&cur) != cudaSuccess) return fail(c, DMRG3S_ERR_CUDA, "cudaGetDevice failed");
  if (cur != c->device && cudaSetDevice(c->device) != cudaSuccess)
    return fail(c, DMRG3S_ERR_CUDA, "cudaSetDevice failed");
  return DMRG3S_OK;
}

// Cached plans.  Each returns the device plan for the given structures,
// building and uploading it on first use.
dmrg3s_status heff_plan(Context* c, const EnvLayout& le, const MpoLayout& w, const EnvLayout& re,
                        const SiteLayout& a, const DevicePlan** out);
dmrg3s_status expand_plan(Context* c, int dir, const EnvLayout& e, const MpoLayout& w,
                          const SiteLayout& m, const SiteLayout& P, const FusedBond& f,
                          const DevicePlan** out);
dmrg3s_status env_plan(Context* c, int dir, const EnvLayout& e, const MpoLayout& w,
                       const SiteLayout& a, const EnvLayout& o, const DevicePlan** out);

// Bump allocator over the context workspace: returns an aligned pointer at
// byte offset *cursor and advances it; DMRG3S_ERR_OOM when it does not fit.
inline dmrg3s_status carve(Context* c, size_t* cursor, size_t bytes, void** out) {
  size_t off = (*cursor + 255) / 256 * 256;
  if (off + bytes > c->ws_bytes)
    return fail(c, DMRG3S_ERR_OOM, "context workspace too small (need " +
                                       std::to_string(off + bytes) + " bytes)");
  *out = c->ws + off;
  *cursor = off + bytes;
  return DMRG3S_OK;
}

// Lanczos with CGS2 for the smallest eigenpair of H_eff (step 1 of Sec. V).
// x: start vector on input, normalised Ritz vector on output (n doubles).
// The workspace from byte offset `cursor` on is used for the Krylov basis.
dmrg3s_status lanczos_run(Context* c, const DevicePlan& heff, const double* Ldata,
                          const double* Rdata, double* x, int64_t n, int kmax, double tol,
                          size_t cursor, cudaStream_t st, double* theta, int* iters,
                          dmrg3s_precision prec = DMRG3S_FP64);

// The same for several independent problems at once: `heff` is a plan whose
// vector operand holds every problem back to back (problem c at elements
// [off, off + n) of X, off a multiple of 32, ldx >= every off + n), so that one
// launch per stage applies all their H_eff.  Each problem keeps its own
// stopping rule (kmax, tol); theta and iters get one entry per problem.
struct LzSpec {
  int64_t off, n;
  int kmax;
  double tol;
};
dmrg3s_status lanczos_batch(Context* c, const DevicePlan& heff, const double* Ldata,
                            const double* Rdata, double* X, int64_t ldx,
                            const std::vector<LzSpec>& probs, size_t cursor, cudaStream_t st,
                            dmrg3s_precision prec, std::vector<double>* theta,
                            std::vector<int>* iters);
// Pinned host area of at least n doubles (c->pinned_big).
dmrg3s_status pinned_reserve(Context* c, size_t n);

// Upload a host plan (allocates the device tables).  Returns CUDA errors.
dmrg3s_status upload_plan(Plan&& host, std::unique_ptr<DevicePlan>* out);
// Builds and uploads what a call in this precision needs beside the plain tables, once
// (a 3xTF32 operator never reads the sliced tables, and an FP64 one never the TF32
// tables).  Before plan_ws_doubles, sliced_fits and run_plan.
dmrg3s_status need_form(Context* c, const DevicePlan& p, dmrg3s_precision prec);

// Enqueue the stages of a plan.  Bases as documented for each plan Kind.
// Tensor-core mode: the stage-1 and stage-3 operands are packed (hi, lo
// parts, tile layout of kernels.hpp) into the workspace:
//   [T1 pairs: ws1][packed T2 (stage-2 output)][g1 A packed][g1 B packed]
//   [g3 A or B packed (the operand that is not T2)][stage-3 partial pairs: ws3]
// (the fused H_eff has no T1 slot, and its stage-1 operands are g12's: the
// coefficient-scaled L blocks and the site tensor)
// (offsets in doubles, each slot 1 KB aligned; a packed operand of n floats
// per part takes n doubles: hi then lo).  A caller that has already packed an
// operand into its slot passes a hint and run_plan skips that pack (the
// Lanczos loop packs L and R once per run).
struct SplitHints {
  bool g1A = false, g1B = false, g3A = false, g3B = false;
  // H_eff only: packed L (stage-1 A) and R (stage-3 B) held outside the
  // workspace (a prepared operator); when set they replace those slots
  const float *g1A_hi = nullptr, *g1A_lo = nullptr, *g3B_hi = nullptr, *g3B_lo = nullptr;
  // FP64: which form runs (kF64Auto: sliced when the plan has it and its
  // intermediates fit the workspace)
  int f64 = 0;
};
constexpr int kF64Auto = 0, kF64Plain = 1, kF64Sliced = 2;
struct TcSlots {
  int64_t t2p, a1, b1, x3, p3, end;   // offsets in doubles from the workspace start
};
inline int64_t slot_round(int64_t d) { return (d + 127) / 128 * 128; }   // 1 KB
inline TcSlots tc_slots(const Plan& p) {
  // the fused H_eff never forms T1; its stage-1 operands are g12's
  const TcStage& s1 = p.fused ? p.g12.tc : p.g1.tc;
  TcSlots s;
  s.t2p = p.fused ? 0 : slot_round(p.ws1);
  s.a1 = s.t2p + slot_round(p.nT2p);
  s.b1 = s.a1 + slot_round(s1.nA);
  s.x3 = s.b1 + slot_round(s1.nB);
  const int64_t n3 = p.kind == Kind::Heff ? p.g3s.tc.nB : p.g3s.tc.nA;
  s.p3 = s.x3 + slot_round(p.has_g3 ? n3 : 0);
  s.end = s.p3 + slot_round(p.ws3);
  return s;
}
// Sliced FP64 mode:
//   [T2][s12 A][s12 B][s3 A][s3 B][row scales: s12 A, s12 B, s3 A, s3 B; grading;
//   counters, list and masks of listed elements][stage-3 partials]
// (offsets in doubles, 1 KB aligned; without stage 3 the output is not here).
struct SlSlots {
  int64_t t2, a1, b1, a3, b3, e, p3, end;
};
// The list of listed elements from `at` on (counter i of the launch's `n`).
inline SlFix sl_fix(int32_t* at, int i, int n, size_t units) {
  int32_t* list = at + n;
  return SlFix{at + i, list, reinterpret_cast<uint32_t*>(list + kSlParts * units)};
}
inline SlSlots sl_slots(const Plan& p) {
  SlSlots s;
  s.t2 = 0;
  s.a1 = slot_round(p.has_g3 ? p.ws2 : 0);
  s.b1 = s.a1 + slot_round((p.s12.nA + 3) / 4);
  s.a3 = s.b1 + slot_round((p.s12.nB + 3) / 4);
  s.b3 = s.a3 + slot_round((p.s3.nA + 3) / 4);
  s.e = s.b3 + slot_round((p.s3.nB + 3) / 4);
  const int64_t parts = kSlParts * (int64_t)std::max(p.s12.units.size(), p.s3.units.size());
  s.p3 = s.e + slot_round(((int64_t)p.s12.neA + p.s12.neB + p.s3.neA + p.s3.neB + p.ngrade + 2 +
                           kSlFixInts * parts + 1) / 2);
  s.end = s.p3 + slot_round(p.ws3s);
  return s;
}
inline bool sliced_fits(const Plan& p, size_t ws_bytes) {
  return p.sliced && (size_t)sl_slots(p).end * sizeof(double) <= ws_bytes;
}
// Workspace (in doubles) a plan needs at least in the given precision (FP64:
// the plain form; the sliced one runs where it fits).
inline int64_t plan_ws_doubles(const Plan& p, dmrg3s_precision prec) {
  return prec == DMRG3S_FP64 ? p.ws1 + p.ws2 : tc_slots(p).end;
}

// `prec` selects the form: plain or sliced FP64 (the sliced one forms stage 2 within
// stage 1's products), or the tensor-core one.
dmrg3s_status run_plan(Context* c, const DevicePlan& p, const double* g1A, const double* g1B,
                       double* ws1, double* c2out, double c2scale, const double* g3A,
                       const double* g3B, double* g3C, cudaStream_t st,
                       dmrg3s_precision prec = DMRG3S_FP64, const SplitHints* hints = nullptr);

// MPO-entry gradient G (d*d*wl*wr doubles, device, layout of W) of
// <M|H_eff|M> for the given environments; intermediates in the workspace.
dmrg3s_status grad_plan(Context* c, const EnvLayout& le, const MpoLayout& w, const EnvLayout& re,
                        const SiteLayout& a, const DeviceGradPlan** out);
dmrg3s_status run_mpo_grad(Context* c, const DeviceGradPlan& p, const double* L, const double* M,
                           const double* R, double* G, cudaStream_t st);

}  // namespace dmrg3s
