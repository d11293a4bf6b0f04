// Host-side planning of the block-sparse contractions.  See plan.hpp.
#include "plan.hpp"

#include "launch.hpp"
#include "validate.hpp"

#include <algorithm>
#include <array>
#include <atomic>
#include <cmath>
#include <functional>
#include <map>
#include <queue>
#include <unordered_map>

namespace dmrg3s {

void GemmStage::add(int64_t offC, int ldc, int M, int N, const std::vector<GemmSeg>& s) {
  if (M <= 0 || N <= 0) return;
  GemmTask t{};
  t.offC = offC;
  t.ldc = ldc;
  t.M = M;
  t.N = N;
  t.seg0 = (int32_t)segs.size();
  t.nseg = (int32_t)s.size();
  const int id = (int)tasks.size();
  tasks.push_back(t);
  for (const auto& g : s) {
    segs.push_back(g);
    flops += 2.0 * M * (double)N * g.K;
  }
  const int ntm = (M + 63) / 64, ntn = (N + 63) / 64;
  for (int a = 0; a < ntm; ++a)
    for (int b = 0; b < ntn; ++b) tiles.push_back(GemmTile{id, a, b, 64});
}

// GB300's FP64 pipe (2 multiply-adds a cycle and SM) makes a k-step of a size x
// size tile cost size^2 / 2 cycles of its SM whatever the operands' traffic, so
// the largest tile is not the fastest one: a stage takes about its padded work
// over the SMs plus its longest tile.  In 64 x 64 tiles the small calls ran a few
// CTAs for a long time, mostly on padding: the prepared operator took 233 us on
// the XXZ chain at m = 100, 165 on the Hubbard chain at m = 200 and 89 on one
// 8 x 8 block; 15, 12 and 11 now.  A large stage is as good in any size (m = 512
// XXZ 220 us, 80 % of the FP64 rate; 883 in 64 x 64 tiles, whose last wave and
// ragged edges left the chip idle).
std::vector<GemmTile> choose_tiles(const GemmStage& g) {
  constexpr int64_t kMost = 32768;                    // tiles of a stage in a smaller size
  constexpr double kTile = 300.0, kChunk = 600.0;     // cycles: a CTA's start, a chunk's latency
  int best = 64;
  double least = 0.0;
  for (const int size : {64, 32, 16, 8}) {
    const int bk = size == 8 ? 64 : size == 16 ? 32 : 16;
    double sum = 0.0, most = 0.0;
    int64_t n = 0;
    for (const GemmTask& t : g.tasks) {
      double cycles = 0.0, chunks = 0.0;
      for (int k = 0; k < t.nseg; ++k) {
        const int K = g.segs[t.seg0 + k].K;
        cycles += 0.5 * size * size * K;
        chunks += (K + bk - 1) / bk;
      }
      const int64_t tiles = (int64_t)((t.M + size - 1) / size) * ((t.N + size - 1) / size);
      n += tiles;
      sum += (double)tiles * (cycles + kTile);
      most = std::max(most, cycles + kChunk * chunks);
    }
    const double time = sum / plan_ctas() + most;
    if (size == 64 || (n <= kMost && time < least)) {
      best = size;
      least = time;
    }
  }
  std::vector<GemmTile> tiles;
  for (size_t id = 0; id < g.tasks.size(); ++id)
    for (int a = 0; a < (g.tasks[id].M + best - 1) / best; ++a)
      for (int b = 0; b < (g.tasks[id].N + best - 1) / best; ++b)
        tiles.push_back(GemmTile{(int32_t)id, a, b, best});
  return tiles;
}

void GemmStage::finalize_bytes(Trans, Trans) {
  std::vector<std::pair<int64_t, int64_t>> a, b;
  a.reserve(segs.size());
  b.reserve(segs.size());
  double elems = 0.0;
  for (const GemmTask& t : tasks) {
    elems += (double)t.M * t.N;
    for (int k = 0; k < t.nseg; ++k) {
      const GemmSeg& g = segs[t.seg0 + k];
      a.push_back({g.offA, (int64_t)t.M * g.K});
      b.push_back({g.offB, (int64_t)t.N * g.K});
    }
  }
  for (auto* v : {&a, &b}) {
    std::sort(v->begin(), v->end());
    v->erase(std::unique(v->begin(), v->end()), v->end());
    for (auto& x : *v) elems += (double)x.second;
  }
  bytes = 8.0 * elems;
}

void SliceTable::add(const std::vector<SlGroup>& g, const std::vector<SlMember>& m) {
  const int32_t which = (int32_t)cta.size() - 1, m0 = (int32_t)members.size();
  int32_t at = cta.back();
  for (SlGroup q : g) {
    q.which = which;
    q.m0 += m0;
    q.cta0 = at;
    // eight warps for one row group's chunks, or for two, four or eight groups with few
    q.per = q.nt > 4 ? 1 : q.nt > 2 ? 2 : q.nt > 1 ? 4 : 8;
    at += q.ctas();
    cta_group.insert(cta_group.end(), q.ctas(), (int32_t)groups.size());
    groups.push_back(q);
  }
  members.insert(members.end(), m.begin(), m.end());
  cta.push_back(at);
}

void CombStage::add(int64_t offOut, int ldo, int rows, int cols, const std::vector<CombTerm>& t) {
  if (rows <= 0 || cols <= 0) return;
  CombTask task{};
  task.offOut = offOut;
  task.ldo = ldo;
  task.rows = rows;
  task.cols = cols;
  task.t0 = (int32_t)terms.size();
  task.nt = (int32_t)t.size();
  const int id = (int)tasks.size();
  tasks.push_back(task);
  for (CombTerm tm : t) {
    tm.chi = (float)tm.coef;
    tm.clo = (float)(tm.coef - (double)tm.chi);
    terms.push_back(tm);
  }
  flops += 2.0 * rows * (double)cols * t.size();
  bytes += 8.0 * rows * (double)cols * (1 + t.size());
  for (int r = 0; r < rows; r += kCombRows)
    chunks.push_back(CombChunk{id, r, rows - r < kCombRows ? rows - r : kCombRows, 0});
}

namespace {
std::atomic<int> g_plan_ctas{152};
}  // namespace

void set_plan_ctas(int n) {
  if (n > 0 && n <= 4096) g_plan_ctas.store(n);
}
int plan_ctas() { return g_plan_ctas.load(); }

namespace {

// Static schedule of a stage's units over the persistent CTAs: longest
// processing time first onto the least loaded CTA.
void schedule(std::vector<TcUnit>& units, std::vector<int32_t>& cta_start,
              const std::vector<double>& cost) {
  const int n = (int)units.size();
  const int nc = std::max(1, std::min(plan_ctas(), n));
  std::vector<int> order(n);
  for (int i = 0; i < n; ++i) order[i] = i;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return cost[a] > cost[b]; });
  std::vector<std::vector<int>> lists(nc);
  using Load = std::pair<double, int>;               // (the lowest of equal ones first)
  std::priority_queue<Load, std::vector<Load>, std::greater<Load>> load;
  for (int c = 0; c < nc; ++c) load.push({0.0, c});
  for (int i : order) {
    const Load l = load.top();
    load.pop();
    lists[l.second].push_back(i);
    load.push({l.first + cost[i], l.second});
  }
  std::vector<TcUnit> out;
  out.reserve(n);
  cta_start.assign(nc + 1, 0);
  for (int c = 0; c < nc; ++c) {
    cta_start[c] = (int32_t)out.size();
    for (int i : lists[c]) out.push_back(units[i]);
  }
  cta_start[nc] = (int32_t)out.size();
  units.swap(out);
}

// A 128 x 128 unit's cost is its k-chunks, each weighted 0.7 as a fixed share
// (the A slab's copy and the issue latency, the same for every width) and 0.3
// by its MMA width, plus a fixed share for its drain and store.
void schedule_units(TcStage& tc, const std::vector<GemmTask>& tasks) {
  const int n = (int)tc.units.size();
  std::vector<double> cost(n);
  for (int i = 0; i < n; ++i) {
    const TcUnit& u = tc.units[i];
    const int nrem = std::min(128, tasks[u.task].N - u.tn * 128);
    cost[i] = u.nchunks * (0.7 + 0.3 * (double)((nrem + 15) / 16 * 16) / 128.0) + 4.0;
  }
  schedule(tc.units, tc.cta_start, cost);
  int64_t chunks = 0;
  for (const TcUnit& u : tc.units) chunks += u.nchunks;
  tc.chain = chunks <= (int64_t)kChainChunks * ((int64_t)tc.cta_start.size() - 1);
}

using Key = std::array<int, 4>;
struct Interm {
  int64_t off;
  int rows, cols;
};
struct Combo {
  int rows = 0, cols = 0;
  std::vector<CombTerm> terms;
};

inline GemmSeg seg(int64_t offA, int64_t lda, int64_t offB, int64_t ldb, int64_t K) {
  GemmSeg g{};
  g.offA = offA;
  g.offB = offB;
  g.lda = (int32_t)lda;
  g.ldb = (int32_t)ldb;
  g.K = (int32_t)K;
  g.scale = 1.0;
  return g;
}

// Stage 1 + 2 of the left side: T1[bl, s] = L[bl] M[s]; T2 terms.
void left_stages(const EnvLayout& le, const MpoLayout& W, const SiteLayout& M, Plan* p,
                 std::map<Key, Interm>* t1, std::map<Key, Combo>* t2) {
  p->g1.ta = Trans::N;
  p->g1.tb = Trans::N;
  int64_t off = 0;
  for (const Block& lb : le.blocks) {
    const int bl = lb.a, ip = lb.b, i = lb.c;
    for (int s = 0; s < M.d; ++s) {
      const int mb = M.block_of(s, i);
      if (mb < 0) continue;
      const Block& blk = M.blocks[mb];
      const int j = blk.c;
      const int64_t rows = le.bond.dim[ip], cols = M.right.dim[j], K = M.left.dim[i];
      if (t1) (*t1)[Key{bl, s, i, 0}] = Interm{off, (int)rows, (int)cols};
      p->g1.add(off, (int)cols, (int)rows, (int)cols, {seg(lb.off, K, blk.off, cols, K)});
      // stage 2 terms
      for (int so = 0; so < W.d; ++so)
        for (int br = 0; br < W.wr; ++br) {
          const double c = W.at(so, s, bl, br);
          if (c == 0.0) continue;
          Combo& cb = (*t2)[Key{br, so, ip, j}];
          cb.rows = (int)rows;
          cb.cols = (int)cols;
          CombTerm tm{};
          tm.offIn = off;
          tm.ldi = (int32_t)cols;
          tm.coef = c;
          cb.terms.push_back(tm);
        }
      off += rows * cols;
    }
  }
  p->ws1 = off;
}

// Stage 1 + 2 of the right side: U1[br, s] = M[s] R[br]^T; U2 terms.
void right_stages(const EnvLayout& re, const MpoLayout& W, const SiteLayout& M, Plan* p,
                  std::map<Key, Combo>* u2) {
  p->g1.ta = Trans::N;
  p->g1.tb = Trans::T;
  int64_t off = 0;
  for (const Block& mb : M.blocks) {
    const int s = mb.a, i = mb.b, j = mb.c;
    for (int br = 0; br < re.w; ++br) {
      const int rb = re.block_of(br, j);
      if (rb < 0) continue;
      const Block& rblk = re.blocks[rb];
      const int jp = rblk.b;
      const int64_t rows = M.left.dim[i], cols = re.bond.dim[jp], K = M.right.dim[j];
      p->g1.add(off, (int)cols, (int)rows, (int)cols, {seg(mb.off, K, rblk.off, K, K)});
      for (int so = 0; so < W.d; ++so)
        for (int bl = 0; bl < W.wl; ++bl) {
          const double c = W.at(so, s, bl, br);
          if (c == 0.0) continue;
          Combo& cb = (*u2)[Key{bl, so, i, jp}];
          cb.rows = (int)rows;
          cb.cols = (int)cols;
          CombTerm tm{};
          tm.offIn = off;
          tm.ldi = (int32_t)cols;
          tm.coef = c;
          cb.terms.push_back(tm);
        }
      off += rows * cols;
    }
  }
  p->ws1 = off;
}

// Materialise stage-2 blocks contiguously in ws2 (offsets in map order).
std::map<Key, Interm> materialise(const std::map<Key, Combo>& combos, Plan* p) {
  std::map<Key, Interm> out;
  int64_t off = 0;
  for (const auto& kv : combos) {
    const Combo& cb = kv.second;
    out[kv.first] = Interm{off, cb.rows, cb.cols};
    p->c2.add(off, cb.cols, cb.rows, cb.cols, cb.terms);
    off += (int64_t)cb.rows * cb.cols;
  }
  p->ws2 = off;
  return out;
}

// ---- tensor-core form of the stages ----

inline int32_t groups8(int64_t R) { return (int32_t)((R + 7) / 8); }
inline int32_t chunks32(int64_t K) { return (int32_t)((K + 31) / 32); }

// Packed placements of one operand array; identical views share one block.
struct Packer {
  std::map<std::pair<std::array<int64_t, 5>, double>, int64_t> seen;   // (view, scale) -> dst
  std::vector<PackBlock>* out;
  int64_t* n;
  int32_t* tiles;
  int64_t add(int64_t src, int64_t ld, int64_t R, int64_t K, int trans, double scale = 1.0) {
    const auto key = std::make_pair(std::array<int64_t, 5>{src, ld, R, K, trans}, scale);
    auto it = seen.find(key);
    if (it != seen.end()) return it->second;
    PackBlock b{};
    b.src = src;
    b.scale = scale;
    int ex = 0;
    b.pow2 = (std::frexp(scale, &ex) == 0.5 || std::frexp(scale, &ex) == -0.5) && ex > -100 && ex < 100
                 ? (float)scale
                 : 0.f;
    b.dst = *n;
    b.ld = (int32_t)ld;
    b.R = (int32_t)R;
    b.K = (int32_t)K;
    b.trans = trans;
    b.R8 = groups8(R);
    b.KC = chunks32(K);
    b.tile0 = *tiles;
    out->push_back(b);
    *n += (int64_t)b.R8 * b.KC * kPackTile;
    *tiles += b.R8 * b.KC;
    seen[key] = b.dst;
    return b.dst;
  }
};

// Placement of a block packed by stage 2: ws2 element offset -> (dst, R8, R, K).
struct CombPacked {
  int64_t dst;
  int32_t R8, R, K;
};

// Builds g.tc.  An operand with a map (c2A for A, c2B for B) is the stage-2
// output, already packed; its segments look their block up by the ws2 offset.
bool build_tc(GemmStage& g, const std::map<int64_t, CombPacked>* c2A,
              const std::map<int64_t, CombPacked>* c2B, std::string* err) {
  TcStage& tc = g.tc;
  tc = TcStage();
  Packer pa{{}, &tc.packA, &tc.nA, &tc.tilesA};
  Packer pb{{}, &tc.packB, &tc.nB, &tc.tilesB};
  auto lookup = [&](const std::map<int64_t, CombPacked>* m, int64_t off, int64_t R, int64_t K,
                    int64_t* dst, int32_t* r8) {
    auto it = m->find(off);
    if (it == m->end() || it->second.R != R || it->second.K != K) {
      *err = "tensor-core operand of stage 3 is not a stage-2 block";
      return false;
    }
    *dst = it->second.dst;
    *r8 = it->second.R8;
    return true;
  };
  for (const GemmTask& t : g.tasks) {
    int32_t nch = 0;
    for (int k = 0; k < t.nseg; ++k) {
      const GemmSeg& sg = g.segs[t.seg0 + k];
      TcSeg ts{};
      ts.kc = chunks32(sg.K);
      // A (rows M): ta = N stores M x K, ta = T stores K x M
      if (c2A) {
        if (!lookup(c2A, sg.offA, t.M, sg.K, &ts.pa, &ts.ra8)) return false;
      } else {
        ts.pa = pa.add(sg.offA, sg.lda, t.M, sg.K, g.ta == Trans::T ? 1 : 0);
        ts.ra8 = groups8(t.M);
      }
      // B (rows N): tb = N stores K x N, tb = T stores N x K
      if (c2B) {
        if (!lookup(c2B, sg.offB, t.N, sg.K, &ts.pb, &ts.rb8)) return false;
      } else {
        ts.pb = pb.add(sg.offB, sg.ldb, t.N, sg.K, g.tb == Trans::N ? 1 : 0);
        ts.rb8 = groups8(t.N);
      }
      tc.segs.push_back(ts);
      nch += ts.kc;
    }
    const int id = (int)(&t - g.tasks.data());
    for (int a = 0; a < (t.M + 127) / 128; ++a)
      for (int b = 0; b < (t.N + 127) / 128; ++b) tc.units.push_back(TcUnit{id, a, b, nch});
  }
  schedule_units(tc, g.tasks);
  return true;
}

// Packs every stage-2 output block (orientation `trans`) and returns the map
// from its ws2 offset to the packed placement.
std::map<int64_t, CombPacked> pack_c2(Plan* p, int trans) {
  std::map<int64_t, CombPacked> m;
  p->c2pack.clear();
  p->nT2p = 0;
  p->tilesT2 = 0;
  for (const CombTask& t : p->c2.tasks) {
    PackOut o{};
    const int64_t R = trans ? t.cols : t.rows, K = trans ? t.rows : t.cols;
    o.dst = p->nT2p;
    o.R8 = groups8(R);
    o.KC = chunks32(K);
    o.trans = trans;
    o.tile0 = p->tilesT2;
    p->c2pack.push_back(o);
    m[t.offOut] = CombPacked{o.dst, o.R8, (int32_t)R, (int32_t)K};
    p->nT2p += (int64_t)o.R8 * o.KC * kPackTile;
    p->tilesT2 += o.R8 * o.KC;
  }
  return m;
}

// Units per GPU the split-K grouping of stage 3 aims at (two per SM of a GB300).
constexpr int64_t kTargetUnits = 2 * 152;

// The fused stages 1 + 2 of H_eff: one task per stage-2 block T2 (packed
// output at its c2pack placement), one K-segment per MPO term of that block:
// A = coef * L[bl] (the stage-1 A operand of the term's T1 block), B = M[s].
bool build_fused(Plan* p, const std::map<int64_t, CombPacked>& c2p, std::string* err) {
  std::map<int64_t, int> t1_task;      // T1 element offset -> stage-1 task
  for (size_t i = 0; i < p->g1.tasks.size(); ++i) t1_task[p->g1.tasks[i].offC] = (int)i;
  GemmStage& g = p->g12;
  g = GemmStage();
  g.ta = p->g1.ta;
  g.tb = p->g1.tb;
  TcStage& tc = g.tc;
  Packer pa{{}, &tc.packA, &tc.nA, &tc.tilesA};
  Packer pb{{}, &tc.packB, &tc.nB, &tc.tilesB};
  for (const CombTask& ct : p->c2.tasks) {
    auto it = c2p.find(ct.offOut);
    if (it == c2p.end()) {
      *err = "fused stage: stage-2 block without a packed placement";
      return false;
    }
    GemmTask t{};
    t.offC = it->second.dst;
    t.ldc = it->second.R8;
    t.M = ct.rows;
    t.N = ct.cols;
    t.seg0 = (int32_t)g.segs.size();
    t.nseg = ct.nt;
    int32_t nch = 0;
    for (int k = 0; k < ct.nt; ++k) {
      const CombTerm& tm = p->c2.terms[ct.t0 + k];
      auto jt = t1_task.find(tm.offIn);
      if (jt == t1_task.end()) {
        *err = "fused stage: MPO term without a stage-1 block";
        return false;
      }
      const GemmTask& t1 = p->g1.tasks[jt->second];
      if (t1.nseg != 1 || t1.M != ct.rows || t1.N != ct.cols) {
        *err = "fused stage: stage-1 block shape";
        return false;
      }
      const GemmSeg& s1 = p->g1.segs[t1.seg0];
      g.segs.push_back(s1);
      TcSeg ts{};
      ts.kc = chunks32(s1.K);
      ts.pa = pa.add(s1.offA, s1.lda, t.M, s1.K, g.ta == Trans::T ? 1 : 0, tm.coef);
      ts.ra8 = groups8(t.M);
      ts.pb = pb.add(s1.offB, s1.ldb, t.N, s1.K, g.tb == Trans::N ? 1 : 0);
      ts.rb8 = groups8(t.N);
      tc.segs.push_back(ts);
      nch += ts.kc;
    }
    const int id = (int)g.tasks.size();
    g.tasks.push_back(t);
    for (int a = 0; a < (t.M + 127) / 128; ++a)
      for (int b = 0; b < (t.N + 127) / 128; ++b) tc.units.push_back(TcUnit{id, a, b, nch});
  }
  schedule_units(tc, g.tasks);
  // algorithmic work: that of stages 1 and 2, which this stage replaces
  g.flops = p->g1.flops + p->c2.flops;
  g.bytes = p->g1.bytes + p->c2.bytes;
  p->fused = true;
  return true;
}

// ---- sliced FP64 form ----

// Blocks of one operand of a stage, grouped by the tasks that use them: blocks
// that meet in one task share their row scales.
struct Slicer {
  struct Blk {
    SlMember m;
    int32_t R, spans;      // spans: of the longest task that uses the block
    int32_t shift;         // of its group (at the group's first block)
  };
  std::vector<Blk> blks;
  std::vector<int> parent;
  std::unordered_multimap<int64_t, int> seen;                 // source offset -> blocks
  int find(int i) {
    while (parent[i] != i) i = parent[i] = parent[parent[i]];
    return i;
  }
  int add(int64_t src, int64_t ld, int64_t R, int64_t K, int trans, double coef) {
    const auto range = seen.equal_range(src);
    for (auto it = range.first; it != range.second; ++it) {
      const Blk& q = blks[it->second];
      if (q.m.coef == coef && q.m.ld == ld && q.R == R && q.m.K == K && q.m.trans == trans) return it->second;
    }
    Blk b{};
    b.m.src = src;
    b.m.coef = coef;
    b.m.ld = (int32_t)ld;
    b.m.K = (int32_t)K;
    b.m.KC = (int32_t)((K + 63) / 64);
    b.m.trans = trans;
    b.m.d0 = -1;
    b.R = (int32_t)R;
    const int id = (int)blks.size();
    blks.push_back(b);
    parent.push_back(id);
    seen.emplace(src, id);
    return id;
  }
  void join(int a, int b) {
    a = find(a);
    b = find(b);
    if (a != b) parent[std::max(a, b)] = std::min(a, b);
  }
  static int32_t groups(int64_t R) { return (int32_t)((R + 15) / 16 * 2); }
  // Places every block and group; e0[block] = first scale of its group.
  void layout(bool headroom, std::vector<SlGroup>* g, std::vector<SlMember>* m, int64_t* n,
              int32_t* ne, std::vector<int32_t>* e0) {
    // blocks by their group (a group's first block is its lowest)
    std::vector<int32_t> first(blks.size() + 1, 0), by(blks.size());
    for (int i = 0; i < (int)blks.size(); ++i) ++first[find(i) + 1];
    for (size_t i = 1; i < first.size(); ++i) first[i] += first[i - 1];
    std::vector<int32_t> at(first.begin(), first.end() - 1);
    for (int i = 0; i < (int)blks.size(); ++i) by[at[find(i)]++] = i;
    e0->assign(blks.size(), 0);
    m->reserve(blks.size());
    for (int root = 0; root < (int)blks.size(); ++root) {
      const int nm = first[root + 1] - first[root];
      if (!nm) continue;
      SlGroup gr{};
      gr.R = blks[root].R;
      gr.R8 = groups(gr.R);
      gr.m0 = (int32_t)m->size();
      gr.nm = nm;
      gr.e0 = *ne;
      int spans = 0;
      for (int k = 0; k < nm; ++k) spans = std::max(spans, blks[by[first[root] + k]].spans);
      while (headroom && spans > kSlSpans << gr.shift) ++gr.shift;
      blks[root].shift = gr.shift;
      for (int k = 0; k < nm; ++k) {
        const int i = by[first[root] + k];
        blks[i].m.t0 = gr.nt;
        gr.nt += blks[i].m.KC;
        blks[i].m.dst = *n;
        *n += (int64_t)gr.R8 * blks[i].m.KC * kSlices * kSlTile;
        (*e0)[i] = gr.e0;
        m->push_back(blks[i].m);
      }
      *ne += gr.R;
      g->push_back(gr);
    }
  }
};

// The bound below which a sum of K terms is listed (kernels_sliced.cu): 3 2^54
// sqrt(K) 0.95 2^-72 of the scales, in units of 2^32 H (2^-20 of the scales).
constexpr double kSlLeast = 3.0 * 0.95 * 4.0;

// Views of the site tensor along the k of a block (by its source offset): what the
// grading of those k is taken from.
using GradeViews = std::unordered_map<int64_t, std::vector<SlView>>;

// The grading of the blocks that meet along k (grade_kernel): blocks of A and B in one
// segment share it, so the classes are the sectors of the contracted bond.  The
// views are those of A's blocks (of_a) or of B's.
bool grade_blocks(const GemmStage& g, const std::vector<int>& ia, const std::vector<int>& ib, bool of_a,
                  const GradeViews& from, Slicer* a, Slicer* b, std::vector<SlGrade>* items,
                  std::vector<SlView>* views, int32_t* n, std::string* err) {
  const int na = (int)a->blks.size();
  std::vector<int> parent(na + b->blks.size());
  for (size_t i = 0; i < parent.size(); ++i) parent[i] = (int)i;
  auto find = [&](int i) {
    while (parent[i] != i) i = parent[i] = parent[parent[i]];
    return i;
  };
  for (size_t k = 0; k < g.segs.size(); ++k) {
    const int x = find(ia[k]), y = find(na + ib[k]);
    parent[std::max(x, y)] = std::min(x, y);
  }
  auto member = [&](int i) -> SlMember& { return i < na ? a->blks[i].m : b->blks[i - na].m; };
  std::vector<int32_t> d0(parent.size(), -1);
  std::vector<std::vector<SlView>> site(parent.size());
  for (int i = 0; i < (int)parent.size(); ++i) {
    const int r = find(i);
    if (d0[r] < 0) {
      d0[r] = *n;
      *n += member(i).K;
    }
    if (member(i).K != member(r).K) {
      *err = "sliced stage: blocks of unequal length share a grading";
      return false;
    }
    member(i).d0 = d0[r];
    if ((i < na) == of_a) {
      const auto it = from.find(member(i).src);
      if (it != from.end()) site[r].insert(site[r].end(), it->second.begin(), it->second.end());
    }
  }
  for (size_t r = 0; r < site.size(); ++r) {
    if (d0[r] < 0) continue;
    // (a block of the site tensor may be seen through several blocks)
    std::vector<SlView>& v = site[r];
    std::sort(v.begin(), v.end(), [](const SlView& x, const SlView& y) { return x.src < y.src; });
    v.erase(std::unique(v.begin(), v.end(), [](const SlView& x, const SlView& y) { return x.src == y.src; }),
            v.end());
    const int K = member((int)r).K;
    for (int k = 0; k < K; k += 32) {
      items->push_back(SlGrade{d0[r] + k, std::min(32, K - k), (int32_t)views->size(), (int32_t)v.size()});
      for (SlView w : v) {
        w.src += w.trans ? (int64_t)k * w.ld : k;
        views->push_back(w);
      }
    }
  }
  return true;
}

// Sliced form of a stage: GemmSeg.scale is the coefficient of A (coefA) or B.  With
// `grade`, the blocks take a grading from these views of A's (of_a) or B's blocks.
bool build_sliced(const GemmStage& g, bool coefA, Plan* grade, bool of_a, const GradeViews& from, SlStage* out,
                  std::string* err) {
  SlStage& s = *out;
  s = SlStage();
  Slicer a, b;
  std::vector<int> ia(g.segs.size()), ib(g.segs.size());
  for (const GemmTask& t : g.tasks) {
    // at most this many spans (a span takes consecutive chunks up to 4 k16 steps)
    int chunks = 0;
    for (int k = 0; k < t.nseg; ++k) chunks += (g.segs[t.seg0 + k].K + 63) / 64;
    for (int k = 0; k < t.nseg; ++k) {
      const GemmSeg& q = g.segs[t.seg0 + k];
      // A (rows M): ta = N stores M x K; B (rows N): tb = T stores N x K
      ia[t.seg0 + k] = a.add(q.offA, q.lda, t.M, q.K, g.ta == Trans::T ? 1 : 0, coefA ? q.scale : 1.0);
      ib[t.seg0 + k] = b.add(q.offB, q.ldb, t.N, q.K, g.tb == Trans::N ? 1 : 0, coefA ? 1.0 : q.scale);
      a.blks[ia[t.seg0 + k]].spans = std::max(a.blks[ia[t.seg0 + k]].spans, chunks);
      if (k) {
        a.join(ia[t.seg0], ia[t.seg0 + k]);
        b.join(ib[t.seg0], ib[t.seg0 + k]);
      }
    }
  }
  for (size_t i = 0; i < a.blks.size(); ++i)
    if (a.blks[i].R != a.blks[a.find((int)i)].R) {
      *err = "sliced stage: blocks of unequal rows share scales";
      return false;
    }
  for (size_t i = 0; i < b.blks.size(); ++i)
    if (b.blks[i].R != b.blks[b.find((int)i)].R) {
      *err = "sliced stage: blocks of unequal rows share scales";
      return false;
    }
  if (grade && !grade_blocks(g, ia, ib, of_a, from, &a, &b, &grade->grades, &grade->views, &grade->ngrade, err))
    return false;
  std::vector<int32_t> ea, eb;
  a.layout(true, &s.gA, &s.mA, &s.nA, &s.neA, &ea);
  b.layout(false, &s.gB, &s.mB, &s.nB, &s.neB, &eb);
  for (size_t k = 0; k < g.segs.size(); ++k) {
    const GemmSeg& q = g.segs[k];
    s.segs.push_back(SlSeg{q.offA, q.offB, q.scale, q.lda, q.ldb, q.K, a.blks[ia[k]].m.d0});
  }
  // narrower units when the 64-wide ones leave SMs without work
  auto count = [&](int tn) {
    int64_t n = 0;
    for (const GemmTask& t : g.tasks) n += (int64_t)((t.M + 127) / 128) * ((t.N + tn - 1) / tn);
    return n;
  };
  int tile_n = 64;
  while (tile_n > 16 && count(tile_n - 16) <= plan_ctas()) tile_n -= 16;
  // cycles of a unit of nw columns: the MMAs of the 36 digit products (max(100, N / 2)
  // each, up to 256 columns in one), against the slabs' copies at ~48 B per cycle;
  // then the drains and the store
  const auto unit_cost = [&](const GemmTask& t, int tm, int nw) {
    double mma = 0.0;
    for (int i = 0; i < kSlices; ++i) {
      const int all = kSlices - i, n1 = i == 0 ? 4 : all * nw > 256 ? 3 : all;
      mma += std::max(100.0, 0.5 * n1 * nw) + (n1 < all ? std::max(100.0, 0.5 * (all - n1) * nw) : 0.0);
    }
    int steps = 0, chunks = 0;
    for (int k = 0; k < t.nseg; ++k) {
      steps += (g.segs[t.seg0 + k].K + 15) / 16;
      chunks += (g.segs[t.seg0 + k].K + 63) / 64;
    }
    const int ga = std::min(16, Slicer::groups(t.M) - tm * 16);
    const double copy = chunks * (double)kSlices * 1024.0 * (ga + nw / 8) / 48.0;
    return std::max(std::max(mma * steps, copy), 2200.0 * chunks) + 3000.0;
  };
  // a task that would keep its SMs busy for longer than the others take in all gets
  // narrower units, down to 32 columns (H_eff: the block that sums every channel has
  // eight times the terms of the others)
  double total = 0.0;
  for (const GemmTask& t : g.tasks)
    total += unit_cost(t, 0, tile_n) * ((t.M + 127) / 128) * ((t.N + tile_n - 1) / tile_n);
  std::vector<int> tile(g.tasks.size(), tile_n);
  for (size_t i = 0; i < g.tasks.size(); ++i)
    while (tile[i] > 32 && unit_cost(g.tasks[i], 0, std::min(tile[i], (g.tasks[i].N + 15) / 16 * 16)) >
                               1.2 * total / plan_ctas())
      tile[i] -= 16;
  std::vector<TcUnit> units;
  std::vector<double> cost;
  for (const GemmTask& t : g.tasks) {
    const int id = (int)(&t - g.tasks.data()), tn = tile[id];
    for (int i = 0; i < (t.M + 127) / 128; ++i)
      for (int j = 0; j < (t.N + tn - 1) / tn; ++j) {
        units.push_back(TcUnit{id, i, j, 0});
        cost.push_back(unit_cost(t, i, std::min(tn, (t.N + 15) / 16 * 16 - j * tn)));
      }
  }
  std::vector<int32_t> cta;
  schedule(units, cta, cost);
  // what each CTA runs: its units, and their chunks one after the other
  s.cta_unit = cta;
  s.cta_chunk.assign(cta.size(), 0);
  for (size_t c = 0; c + 1 < cta.size(); ++c) {
    s.cta_chunk[c] = (int32_t)s.chunks.size();
    int prev_nw = 0;
    for (int32_t ui = cta[c]; ui < cta[c + 1]; ++ui) {
      const GemmTask& t = g.tasks[units[ui].task];
      SlUnit un{};
      un.em = -1;
      un.d0 = -1;
      un.m0 = units[ui].tm * 128;
      const int tn = tile[units[ui].task];
      un.n0 = units[ui].tn * tn;
      un.offC = t.offC + (int64_t)un.m0 * t.ldc + un.n0;
      un.ldc = t.ldc;
      un.rows = std::min(128, t.M - un.m0);
      un.cols = std::min(tn, t.N - un.n0);
      un.nw = (un.cols + 15) / 16 * 16;
      un.seg0 = t.seg0;
      un.nseg = t.nseg;
      if (t.nseg > 0) {
        un.ea = ea[ia[t.seg0]] + un.m0;
        un.eb = eb[ib[t.seg0]] + un.n0;
        un.shift = a.blks[a.find(ia[t.seg0])].shift;
      }
      int64_t terms = 0;
      for (int k = 0; k < t.nseg; ++k) terms += g.segs[t.seg0 + k].K;
      un.least = (uint32_t)std::ceil(kSlLeast * std::sqrt((double)terms));
      const int ra8 = Slicer::groups(t.M), rb8 = Slicer::groups(t.N);
      const size_t first = s.words.size();
      int used = 0;
      for (int k = 0; k < t.nseg; ++k) {
        const int k16 = (g.segs[t.seg0 + k].K + 15) / 16;
        for (int q = 0; 4 * q < k16; ++q) {
          const int ks = std::min(4, k16 - 4 * q);
          uint32_t w = (uint32_t)ks | (uint32_t)un.nw << kSlNw;
          // spans: consecutive chunks while their k16 steps sum to at most 4
          if (s.words.size() == first || used + ks > 4) {
            if (s.words.size() > first) s.words.back() |= kSlLast;
            w |= kSlFirst;
            if (un.spans % kSlLongSpan == 0) {
              if (un.spans) s.words.back() |= kSlLongLast;
              w |= kSlLongFirst;
            }
            ++un.spans;
            used = 0;
          }
          if (s.words.size() == first && un.nw != prev_nw) w |= kSlMove;
          used += ks;
          s.words.push_back(w);
          SlChunk ch{};
          ch.sa = ra8 * kSlTile;
          ch.sb = rb8 * kSlTile;
          ch.a = a.blks[ia[t.seg0 + k]].m.dst + (int64_t)q * kSlices * ch.sa + (int64_t)(un.m0 / 8) * kSlTile;
          ch.b = b.blks[ib[t.seg0 + k]].m.dst + (int64_t)q * kSlices * ch.sb + (int64_t)(un.n0 / 8) * kSlTile;
          ch.ga = std::min(16, ra8 - un.m0 / 8);
          ch.gb = un.nw / 8;
          s.chunks.push_back(ch);
        }
      }
      if (s.words.size() > first) {
        s.words.back() |= kSlLast | kSlLongLast;
        prev_nw = un.nw;
      }
      s.units.push_back(un);
    }
  }
  if (!cta.empty()) s.cta_chunk.back() = (int32_t)s.chunks.size();
  return true;
}

// Stages 1 + 2 as one grouped GEMM in FP64: one task per stage-2 block, one
// K-segment per MPO term, scaled by its coefficient.
bool fuse_f64(const Plan& p, GemmStage* out, std::string* err) {
  std::unordered_map<int64_t, int> t1_task;      // T1 element offset -> stage-1 task
  t1_task.reserve(p.g1.tasks.size());
  for (size_t i = 0; i < p.g1.tasks.size(); ++i) t1_task[p.g1.tasks[i].offC] = (int)i;
  GemmStage& g = *out;
  g = GemmStage();
  g.ta = p.g1.ta;
  g.tb = p.g1.tb;
  for (const CombTask& ct : p.c2.tasks) {
    GemmTask t{};
    t.offC = ct.offOut;
    t.ldc = ct.ldo;
    t.M = ct.rows;
    t.N = ct.cols;
    t.seg0 = (int32_t)g.segs.size();
    t.nseg = ct.nt;
    for (int k = 0; k < ct.nt; ++k) {
      const CombTerm& tm = p.c2.terms[ct.t0 + k];
      auto jt = t1_task.find(tm.offIn);
      if (jt == t1_task.end()) {
        *err = "fused stage: MPO term without a stage-1 block";
        return false;
      }
      const GemmTask& t1 = p.g1.tasks[jt->second];
      if (t1.nseg != 1 || t1.M != ct.rows || t1.N != ct.cols) {
        *err = "fused stage: stage-1 block shape";
        return false;
      }
      GemmSeg q = p.g1.segs[t1.seg0];
      q.scale = tm.coef;
      g.segs.push_back(q);
    }
    g.tasks.push_back(t);
  }
  g.flops = p.g1.flops + p.c2.flops;   // algorithmic: the stages it replaces
  g.bytes = p.g1.bytes + p.c2.bytes;
  return true;
}

// Stage 3 in `groups` consecutive groups of K-segments per output block, each
// into its own partial block (offsets from 0), and the sum of the partials.
void split_k(const GemmStage& g3, int groups, GemmStage* parts, CombStage* sum, int64_t* n) {
  parts->ta = g3.ta;
  parts->tb = g3.tb;
  int64_t poff = 0;
  for (const GemmTask& t : g3.tasks) {
    std::vector<CombTerm> terms;
    const int ng = std::min<int>(groups, std::max(1, (int)t.nseg));
    for (int gi = 0; gi < ng; ++gi) {
      const int k0 = (int)((int64_t)t.nseg * gi / ng), k1 = (int)((int64_t)t.nseg * (gi + 1) / ng);
      std::vector<GemmSeg> sg(g3.segs.begin() + t.seg0 + k0, g3.segs.begin() + t.seg0 + k1);
      if (sg.empty() && t.nseg > 0) continue;
      parts->add(poff, t.N, t.M, t.N, sg);
      CombTerm tm{};
      tm.offIn = poff;
      tm.ldi = t.N;
      tm.coef = 1.0;
      terms.push_back(tm);
      poff += (int64_t)t.M * t.N;
    }
    sum->add(t.offC, t.ldc, t.M, t.N, terms);
  }
  *n = poff;
  parts->flops = g3.flops;        // same algorithmic work as stage 3
  parts->bytes = g3.bytes;
  sum->flops = 0.0;               // the partial sums are bookkeeping, not algorithm
  sum->bytes = 0.0;
}

// Smaller combination chunks when a stage would have too few of them: up to
// kCombCtas CTAs per SM (all the threads an SM holds) while each still has
// kCombElems elements, two per thread; two CTAs per SM when there are fewer
// elements.  The sum of the cylinder's 0.9 M stage-3 partials, with two CTAs an
// SM bound by the loads in flight, took 23 us of a 215 us 3xTF32 operator; the
// operator takes 202 us (with the packing's tile search in one step).
constexpr int kCombCtas = 8;
constexpr int kCombElems = 512;
void rechunk(CombStage& c) {
  int64_t elems = 0;
  for (const CombTask& t : c.tasks) elems += (int64_t)t.rows * t.cols;
  const int64_t target = std::max<int64_t>(
      2 * plan_ctas(), std::min<int64_t>(elems / kCombElems, kCombCtas * plan_ctas()));
  int rpc = kCombRows;
  auto count = [&](int r) {
    int64_t n = 0;
    for (const CombTask& t : c.tasks) n += (t.rows + r - 1) / r;
    return n;
  };
  while (rpc > 1 && count(rpc) < target) rpc /= 2;
  if (rpc == kCombRows) return;
  c.chunks.clear();
  for (size_t id = 0; id < c.tasks.size(); ++id) {
    const int rows = c.tasks[id].rows;
    for (int r = 0; r < rows; r += rpc)
      c.chunks.push_back(CombChunk{(int32_t)id, r, rows - r < rpc ? rows - r : rpc, 0});
  }
}

// The stage-2 output as stage 3's operand: its blocks as pieces, and where
// every unit of stage 2 collects its row scales (EnvLR: its columns' scales).
bool plan_t2(Plan* p, const std::vector<SlGroup>& groups, const std::vector<SlMember>& members,
             std::string* err) {
  // block offset -> its first row scale, grading entry
  std::unordered_map<int64_t, std::pair<int32_t, int32_t>> e0;
  e0.reserve(members.size());
  for (const SlGroup& g : groups)
    for (int k = 0; k < g.nm; ++k) {
      const SlMember& m = members[g.m0 + k];
      SlPiece q{};
      q.src = m.src;
      q.dst = m.dst;
      q.ld = m.ld;
      q.K = m.K;
      q.KC = m.KC;
      q.trans = m.trans;
      q.R = g.R;
      q.R8 = g.R8;
      q.e0 = g.e0;
      q.shift = g.shift;
      q.d0 = m.d0;
      q.tile0 = p->t2_tiles;
      p->t2_tiles += g.R8 * m.KC;
      p->t2.push_back(q);
      if (!e0.emplace(m.src, std::make_pair(g.e0, m.d0)).second) {
        *err = "sliced stage: a stage-2 block with two sets of scales";
        return false;
      }
    }
  int32_t at = 0;
  for (int32_t t = 0; t < p->t2_tiles; t += 8) {
    while (at + 1 < (int32_t)p->t2.size() && p->t2[at + 1].tile0 <= t) ++at;
    p->t2_first.push_back(at);
  }
  const bool cols = p->kind == Kind::EnvLR;
  for (SlUnit& u : p->s12.units) {
    // the unit's block: its offset less the unit's place in it
    const auto it = e0.find(u.offC - (int64_t)u.m0 * u.ldc - u.n0);
    u.em = it == e0.end() ? -1 : it->second.first + (cols ? u.n0 : u.m0);
    // (a graded operand: A of H_eff, whose k are the block's columns)
    u.d0 = it == e0.end() || it->second.second < 0 ? -1 : it->second.second + u.n0;
    const int32_t ne = p->kind == Kind::Heff ? p->s3.neA : p->s3.neB;
    if (u.em >= 0 && (u.em + (cols ? u.cols : u.rows) > ne || (u.d0 >= 0 && u.d0 + u.cols > p->ngrade))) {
      *err = "sliced stage: collected scales out of bounds";
      return false;
    }
  }
  return true;
}

// Least work of a contraction that takes the sliced form, whose time hardly falls
// below 60 us: flops that fill the products' tiles (128 rows, 16 columns, 16 k; a
// sector of 40 states wastes two thirds of them).  Plain against sliced calls (us; Mflop,
// the share that fills): operators, XXZ m = 256 (22, 0.26) 47 and 83, m = 320 (43, 0.34)
// 78 and 94, m = 400 (84, 0.50) 119 and 99, m = 512 (177, 0.53) 219 and 118; Hubbard m = 700
// (38, 0.34) 65 and 98, m = 1024 (127, 0.48) 163 and 117; one block, m = 96 (32, 0.75) 52 and
// 80, m = 128 (76, 1) 93 and 83.  Expansions, Hubbard m = 700 (19, 0.35) 36 and 55, m = 1024 (64,
// 0.5) 86 and 68; gradients, Hubbard m = 700 (37) 99 and 103, m = 1024 (126) 225 and 168.
constexpr double kSlicedMinFlops = 11e6;
double tile_fill(const GemmStage& g, const GemmStage* h) {
  double work = 0.0, tiles = 0.0;
  for (const GemmStage* s : {&g, h})
    if (s)
      for (const GemmTask& t : s->tasks)
        for (int k = 0; k < t.nseg; ++k) {
          const double K = s->segs[t.seg0 + k].K;
          work += (double)t.M * t.N * K;
          tiles += std::ceil(t.M / 128.0) * 128.0 * std::ceil(t.N / 16.0) * 16.0 * std::ceil(K / 16.0) * 16.0;
        }
  return tiles > 0.0 ? work / tiles : 0.0;
}
// Largest ratio of the fused stage's work to stage 1's: the sliced products
// run 2 (0.2 Gflop) to 13 (13 Gflop) times as fast as the plain ones; a model
// MPO has a ratio near 1.2.  Below it, the least work grows with the ratio.
constexpr double kSlicedMaxTerms = 6.0;

// The sliced FP64 form, where there is enough work for it.
}  // namespace

void plan_sliced(Plan* p) {
  const int64_t nA1 = p->nA1, nB1 = p->nB1, nOut2 = p->nOut2, nA3 = p->nA3, nB3 = p->nB3, nC3 = p->nC3;
  std::string why, *err = &why;
  p->sliced = false;
  p->sliced_tried = true;
  const double flops = p->flops() * tile_fill(p->g1, p->has_g3 ? &p->g3 : nullptr);
  if (flops < kSlicedMinFlops) return;
  // a dense MPO tensor: too many terms per stage-1 block to form each anew
  double terms = 0.0, blocks = 0.0;
  for (const CombTask& t : p->c2.tasks) terms += (double)t.nt * t.rows * t.cols;
  for (const GemmTask& t : p->g1.tasks) blocks += (double)t.M * t.N;
  if (terms > kSlicedMaxTerms * blocks || flops * blocks < kSlicedMinFlops * terms)
    return;
  const bool left = p->kind == Kind::Heff || p->kind == Kind::ExpandLR || p->kind == Kind::EnvLR;
  bool ok = fuse_f64(*p, &p->f12, err);
  // the site tensor (B of the left kinds, A of the right ones): along k, and along
  // the other index of the blocks that H_eff's stage 3 contracts
  GradeViews along, across;
  for (const GemmTask& t : p->f12.tasks)
    for (int k = 0; ok && k < t.nseg; ++k) {
      const GemmSeg& q = p->f12.segs[t.seg0 + k];
      auto& v = along[left ? q.offB : q.offA];
      if (v.empty()) v.push_back(left ? SlView{q.offB, q.ldb, t.N, 1, 0} : SlView{q.offA, q.lda, t.M, 0, 0});
      if (p->kind == Kind::Heff) {
        auto& w = across[t.offC];
        if (w.empty() || w.back().src != q.offB) w.push_back(SlView{q.offB, q.ldb, q.K, 0, 0});
      }
    }
  ok = ok && build_sliced(p->f12, left, p, !left, along, &p->s12, err) &&
       sliced_ok(p->f12, p->s12, nA1, nB1, nOut2, p->ngrade, err);
  if (ok && p->has_g3) {
    int64_t units1 = 0;
    int maxseg = 1;
    for (const GemmTask& t : p->g3.tasks) {
      units1 += (int64_t)((t.M + 127) / 128) * ((t.N + 63) / 64);
      maxseg = std::max(maxseg, (int)t.nseg);
    }
    int G = units1 > 0 ? (int)((kTargetUnits + units1 - 1) / units1) : 1;
    G = std::max(1, std::min(G, maxseg));
    if (G > 1) {
      split_k(p->g3, G, &p->f3, &p->s3r, &p->ws3s);
      rechunk(p->s3r);
      ok = comb_ok(p->s3r.tasks, p->s3r.terms, std::max<int64_t>(p->ws3s, 1), nC3, err);
    } else {
      p->f3 = p->g3;
      p->f3.tiles.clear();
    }
    ok = ok && build_sliced(p->f3, true, p->kind == Kind::Heff ? p : nullptr, true, across, &p->s3, err) &&
         sliced_ok(p->f3, p->s3, nA3, nB3, G > 1 ? std::max<int64_t>(p->ws3s, 1) : nC3, p->ngrade, err);
  }
  if (ok) {
    const bool t2_is_a = p->kind == Kind::Heff;
    p->slices.add(t2_is_a ? p->s3.gB : p->s3.gA, t2_is_a ? p->s3.mB : p->s3.mA);
    p->slices.add(left ? p->s12.gA : p->s12.gB, left ? p->s12.mA : p->s12.mB);
    p->slices.add(left ? p->s12.gB : p->s12.gA, left ? p->s12.mB : p->s12.mA);
    ok = slice_table_ok(p->slices, err) && grades_ok(p->grades, p->views, left ? nB1 : nA1, p->ngrade, err);
    if (ok && p->has_g3) ok = plan_t2(p, t2_is_a ? p->s3.gA : p->s3.gB, t2_is_a ? p->s3.mA : p->s3.mB, err);
  }
  p->sliced = ok;                    // (tables that fail a check: the plain form)
}

namespace {

// Bounds of every table against the buffers the stages address.
dmrg3s_status finish(Plan* p, int64_t nA1, int64_t nB1, int64_t nOut2, int64_t nA3, int64_t nB3,
                     int64_t nC3, std::string* err) {
  p->nA1 = nA1;
  p->nB1 = nB1;
  p->nOut2 = nOut2;
  p->nA3 = p->has_g3 ? nA3 : 0;
  p->nB3 = p->has_g3 ? nB3 : 0;
  p->nC3 = p->has_g3 ? nC3 : 0;
  p->g1.finalize_bytes(p->g1.ta, p->g1.tb);
  if (p->has_g3) p->g3.finalize_bytes(p->g3.ta, p->g3.tb);
  const int64_t w1 = p->ws1 > 0 ? p->ws1 : 1;
  if (!gemm_ok(p->g1.ta, p->g1.tb, p->g1.tasks, p->g1.segs, nA1, nB1, w1, err) ||
      !comb_ok(p->c2.tasks, p->c2.terms, w1, nOut2, err) ||
      (p->has_g3 && !gemm_ok(p->g3.ta, p->g3.tb, p->g3.tasks, p->g3.segs, nA3, nB3, nC3, err))) {
    *err = "internal planning error: " + *err;
    return DMRG3S_ERR_SHAPE;
  }
  p->g1.tiles = choose_tiles(p->g1);
  p->g3.tiles = choose_tiles(p->g3);
  rechunk(p->c2);
  return DMRG3S_OK;
}

}  // namespace

dmrg3s_status plan_tensor_core(Plan* p, std::string* err) {
  const int64_t nA1 = p->nA1, nB1 = p->nB1, nA3 = p->nA3, nB3 = p->nB3, nC3 = p->nC3;
  if (p->has_g3) {
    // split-K form of stage 3: the K-segments of every output block in G
    // consecutive groups, G chosen so that the units fill the GPU about twice
    // (kTargetUnits); each group writes a partial block, then a fixed-order sum
    int64_t units1 = 0;
    int maxseg = 1;
    for (const GemmTask& t : p->g3.tasks) {
      units1 += (int64_t)((t.M + 127) / 128) * ((t.N + 127) / 128);
      maxseg = std::max(maxseg, (int)t.nseg);
    }
    int G = units1 > 0 ? (int)((kTargetUnits + units1 - 1) / units1) : 1;
    G = std::max(1, std::min(G, maxseg));
    split_k(p->g3, G, &p->g3s, &p->c3r, &p->ws3);
    const int64_t w3 = p->ws3 > 0 ? p->ws3 : 1;
    if (!gemm_ok(p->g3s.ta, p->g3s.tb, p->g3s.tasks, p->g3s.segs, nA3, nB3, w3, err) ||
        !comb_ok(p->c3r.tasks, p->c3r.terms, w3, nC3, err)) {
      *err = "internal planning error: " + *err;
      return DMRG3S_ERR_SHAPE;
    }
  }
  // tensor-core form.  H_eff: stages 1 and 2 fused (g12) writing T2 packed
  // for stage 3.  The others: stage 1 packs both operands, and stage 3 takes
  // the stage-2 output packed by the combination (B of the environments).
  bool ok = true;
  if (p->kind == Kind::Heff) {
    const std::map<int64_t, CombPacked> m = pack_c2(p, 0);
    ok = build_fused(p, m, err) && build_tc(p->g3s, &m, nullptr, err) &&
         tc_ok(p->g12.tasks, p->g12.tc, nA1, nB1, p->g12.tc.nA, p->g12.tc.nB, err) &&
         packed_tasks_ok(p->g12.tasks, p->nT2p, err);
  } else {
    ok = build_tc(p->g1, nullptr, nullptr, err);
    if (ok && p->has_g3) {
      const int trans = p->kind == Kind::EnvLR ? 1 : 0;
      const std::map<int64_t, CombPacked> m = pack_c2(p, trans);
      ok = build_tc(p->g3s, nullptr, &m, err);
    }
    if (ok) ok = tc_ok(p->g1.tasks, p->g1.tc, nA1, nB1, p->g1.tc.nA, p->g1.tc.nB, err);
  }
  if (ok && p->has_g3) {
    const bool c2_is_a = p->kind == Kind::Heff;
    ok = tc_ok(p->g3s.tasks, p->g3s.tc, nA3, nB3, c2_is_a ? p->nT2p : p->g3s.tc.nA,
               c2_is_a ? p->g3s.tc.nB : p->nT2p, err) &&
         packout_ok(p->c2.tasks, p->c2pack, p->nT2p, err);
  }
  if (!ok) {
    *err = "internal planning error: " + *err;
    return DMRG3S_ERR_SHAPE;
  }
  rechunk(p->c3r);
  p->tc_built = true;
  return DMRG3S_OK;
}

namespace {
// Appends stage `src` to `dst` with its operand offsets moved by oA / oB and
// its output offsets by oC.
void append_gemm(GemmStage& dst, const GemmStage& src, int64_t oA, int64_t oB, int64_t oC) {
  const int32_t t0 = (int32_t)dst.tasks.size(), s0 = (int32_t)dst.segs.size();
  for (GemmTask t : src.tasks) {
    t.offC += oC;
    t.seg0 += s0;
    dst.tasks.push_back(t);
  }
  for (GemmSeg g : src.segs) {
    g.offA += oA;
    g.offB += oB;
    dst.segs.push_back(g);
  }
  for (GemmTile t : src.tiles) {
    t.task += t0;
    dst.tiles.push_back(t);
  }
  dst.flops += src.flops;
}
void append_comb(CombStage& dst, const CombStage& src, int64_t oIn, int64_t oOut, double scale) {
  const int32_t t0 = (int32_t)dst.tasks.size(), m0 = (int32_t)dst.terms.size();
  for (CombTask t : src.tasks) {
    t.offOut += oOut;
    t.t0 += m0;
    dst.tasks.push_back(t);
  }
  for (CombTerm m : src.terms) {
    m.offIn += oIn;
    if (scale != 1.0) {
      m.coef *= scale;
      m.chi = (float)m.coef;
      m.clo = (float)(m.coef - (double)m.chi);
    }
    dst.terms.push_back(m);
  }
  for (CombChunk ch : src.chunks) {
    ch.task += t0;
    dst.chunks.push_back(ch);
  }
  dst.flops += src.flops;
  dst.bytes += src.bytes;
}
}  // namespace

dmrg3s_status merge_plans(Kind kind, const std::vector<PlanPart>& parts, int64_t nA1, int64_t nB1,
                          int64_t nOut2, int64_t nA3, int64_t nB3, int64_t nC3, Plan* out,
                          std::string* err) {
  *out = Plan();
  Plan& m = *out;
  m.kind = kind;
  m.has_g3 = kind == Kind::Heff || kind == Kind::EnvLR || kind == Kind::EnvRL;
  if (parts.empty()) {
    *err = "merge of no plans";
    return DMRG3S_ERR_ARG;
  }
  m.g1.ta = parts[0].p->g1.ta;
  m.g1.tb = parts[0].p->g1.tb;
  m.g3.ta = parts[0].p->g3.ta;
  m.g3.tb = parts[0].p->g3.tb;
  int64_t o1 = 0, o2 = 0;
  for (const PlanPart& q : parts) {
    const Plan& p = *q.p;
    if (p.kind != kind || p.g1.ta != m.g1.ta || p.g1.tb != m.g1.tb ||
        (m.has_g3 && (p.g3.ta != m.g3.ta || p.g3.tb != m.g3.tb))) {
      *err = "merged plans differ in kind";
      return DMRG3S_ERR_ARG;
    }
    append_gemm(m.g1, p.g1, q.oA1, q.oB1, o1);
    append_comb(m.c2, p.c2, o1, m.has_g3 ? o2 : q.oOut2, q.c2scale);
    if (m.has_g3) {
      const bool t2_is_a = kind == Kind::Heff;
      append_gemm(m.g3, p.g3, t2_is_a ? o2 : q.oA3, t2_is_a ? q.oB3 : o2, q.oC3);
    }
    o1 += p.ws1;
    o2 += m.has_g3 ? p.ws2 : 0;
  }
  m.ws1 = o1;
  m.ws2 = o2;
  if (m.has_g3) {
    if (kind == Kind::Heff) nA3 = o2;
    else nB3 = o2;
    nOut2 = o2;
  }
  return finish(&m, nA1, nB1, nOut2, nA3, nB3, nC3, err);
}

dmrg3s_status check_site_mpo(const SiteLayout& s, const MpoLayout& W, std::string* err) {
  if (s.nsym != W.nsym) {
    *err = "site tensor and MPO have different nsym";
    return DMRG3S_ERR_SHAPE;
  }
  if (s.d != W.d) {
    *err = "site tensor and MPO have different physical dimension";
    return DMRG3S_ERR_SHAPE;
  }
  if (!same_charges(s.qp, W.qp)) {
    *err = "site tensor and MPO have different physical charges";
    return DMRG3S_ERR_QN;
  }
  return DMRG3S_OK;
}

dmrg3s_status check_env(const EnvLayout& e, const Bond& bond, int w, const std::vector<Charge>& t,
                        const char* what, std::string* err) {
  if (e.nsym != bond.nsym) {
    *err = std::string(what) + ": nsym differs from the site tensor";
    return DMRG3S_ERR_SHAPE;
  }
  if (!same_bond(e.bond, bond)) {
    *err = std::string(what) + ": bond differs from the site tensor's bond";
    return DMRG3S_ERR_SHAPE;
  }
  if (e.w != w) {
    *err = std::string(what) + ": MPO bond dimension differs from W";
    return DMRG3S_ERR_SHAPE;
  }
  if (!same_charges(e.t, t)) {
    *err = std::string(what) + ": channel charges differ from W";
    return DMRG3S_ERR_QN;
  }
  return DMRG3S_OK;
}

dmrg3s_status plan_heff(const EnvLayout& le, const MpoLayout& W, const EnvLayout& re,
                        const SiteLayout& M, Plan* p, std::string* err) {
  p->kind = Kind::Heff;
  std::map<Key, Combo> t2c;
  left_stages(le, W, M, p, nullptr, &t2c);
  std::map<Key, Interm> t2 = materialise(t2c, p);
  p->has_g3 = true;
  p->g3.ta = Trans::N;
  p->g3.tb = Trans::T;
  for (const Block& hb : M.blocks) {
    const int so = hb.a, ip = hb.b, jp = hb.c;
    std::vector<GemmSeg> segs;
    for (int br = 0; br < W.wr; ++br) {
      const int j = M.nsym ? M.right.find(sub(M.right.q[jp], re.t[br])) : 0;
      if (j < 0) continue;
      const int rb = re.block_of(br, j);
      if (rb < 0 || re.blocks[rb].b != jp) continue;
      auto it = t2.find(Key{br, so, ip, j});
      if (it == t2.end()) continue;
      const int64_t K = M.right.dim[j];
      segs.push_back(seg(it->second.off, K, re.blocks[rb].off, K, K));
    }
    p->g3.add(hb.off, (int)hb.cols, (int)hb.rows, (int)hb.cols, segs);
  }
  return finish(p, le.size, M.size, p->ws2, p->ws2, re.size, M.size, err);
}

dmrg3s_status plan_expand_lr(const EnvLayout& le, const MpoLayout& W, const SiteLayout& M,
                             const SiteLayout& P, const FusedBond& fused, Plan* p,
                             std::string* err) {
  p->kind = Kind::ExpandLR;
  std::map<Key, Combo> t2c;
  left_stages(le, W, M, p, nullptr, &t2c);
  const int nsrc = M.right.nsec();
  for (const Block& pb : P.blocks) {
    const int so = pb.a, ip = pb.b, k = pb.c;
    for (int br = 0; br < W.wr; ++br) {
      const int j = M.nsym ? M.right.find(sub(P.right.q[k], W.tr[br])) : 0;
      if (j < 0 || fused.target[(size_t)br * nsrc + j] != k) continue;
      const int64_t coff = fused.offset[(size_t)br * nsrc + j];
      auto it = t2c.find(Key{br, so, ip, j});
      static const std::vector<CombTerm> none;
      p->c2.add(pb.off + coff, (int)pb.cols, (int)pb.rows, (int)M.right.dim[j],
                it == t2c.end() ? none : it->second.terms);
    }
  }
  p->ws2 = 0;
  return finish(p, le.size, M.size, P.size, 0, 0, 0, err);
}

dmrg3s_status plan_env_lr(const EnvLayout& le, const MpoLayout& W, const SiteLayout& M,
                          const EnvLayout& out, Plan* p, std::string* err) {
  p->kind = Kind::EnvLR;
  std::map<Key, Combo> t2c;
  left_stages(le, W, M, p, nullptr, &t2c);
  std::map<Key, Interm> t2 = materialise(t2c, p);
  p->has_g3 = true;
  p->g3.ta = Trans::T;
  p->g3.tb = Trans::N;
  for (const Block& ob : out.blocks) {
    const int br = ob.a, ib = ob.b, ik = ob.c;
    std::vector<GemmSeg> segs;
    for (int so = 0; so < M.d; ++so) {
      const int ip = M.nsym ? M.left.find(sub(M.right.q[ib], M.qp[so])) : 0;
      if (ip < 0) continue;
      const int ab = M.block_of(so, ip);
      if (ab < 0 || M.blocks[ab].c != ib) continue;
      auto it = t2.find(Key{br, so, ip, ik});
      if (it == t2.end()) continue;
      const int64_t K = M.left.dim[ip];
      segs.push_back(seg(M.blocks[ab].off, M.right.dim[ib], it->second.off, M.right.dim[ik], K));
    }
    p->g3.add(ob.off, (int)ob.cols, (int)ob.rows, (int)ob.cols, segs);
  }
  return finish(p, le.size, M.size, p->ws2, M.size, p->ws2, out.size, err);
}

dmrg3s_status plan_expand_rl(const EnvLayout& re, const MpoLayout& W, const SiteLayout& M,
                             const SiteLayout& P, const FusedBond& fused, Plan* p,
                             std::string* err) {
  p->kind = Kind::ExpandRL;
  std::map<Key, Combo> u2c;
  right_stages(re, W, M, p, &u2c);
  const int nsrc = M.left.nsec();
  for (const Block& pb : P.blocks) {
    const int so = pb.a, k = pb.b, jp = pb.c;
    for (int bl = 0; bl < W.wl; ++bl) {
      const int i = M.nsym ? M.left.find(sub(P.left.q[k], W.tl[bl])) : 0;
      if (i < 0 || fused.target[(size_t)bl * nsrc + i] != k) continue;
      const int64_t roff = fused.offset[(size_t)bl * nsrc + i];
      auto it = u2c.find(Key{bl, so, i, jp});
      static const std::vector<CombTerm> none;
      p->c2.add(pb.off + roff * pb.cols, (int)pb.cols, (int)M.left.dim[i], (int)pb.cols,
                it == u2c.end() ? none : it->second.terms);
    }
  }
  p->ws2 = 0;
  return finish(p, M.size, re.size, P.size, 0, 0, 0, err);
}

dmrg3s_status plan_env_rl(const EnvLayout& re, const MpoLayout& W, const SiteLayout& M,
                          const EnvLayout& out, Plan* p, std::string* err) {
  p->kind = Kind::EnvRL;
  std::map<Key, Combo> u2c;
  right_stages(re, W, M, p, &u2c);
  std::map<Key, Interm> u2 = materialise(u2c, p);
  p->has_g3 = true;
  p->g3.ta = Trans::N;
  p->g3.tb = Trans::T;
  for (const Block& ob : out.blocks) {
    const int bl = ob.a, ib = ob.b, ik = ob.c;
    std::vector<GemmSeg> segs;
    for (int so = 0; so < M.d; ++so) {
      const int bb = M.block_of(so, ib);
      if (bb < 0) continue;
      const int jp = M.blocks[bb].c;
      auto it = u2.find(Key{bl, so, ik, jp});
      if (it == u2.end()) continue;
      const int64_t K = M.right.dim[jp];
      segs.push_back(seg(M.blocks[bb].off, K, it->second.off, K, K));
    }
    p->g3.add(ob.off, (int)ob.cols, (int)ob.rows, (int)ob.cols, segs);
  }
  return finish(p, M.size, re.size, p->ws2, M.size, p->ws2, out.size, err);
}

dmrg3s_status plan_mpo_grad(const EnvLayout& le, const MpoLayout& W, const EnvLayout& re,
                            const SiteLayout& M, GradPlan* p, std::string* err) {
  // stage 1 exactly as for H_eff; the T1 blocks are then indexed by (bl, s)
  Plan tmp;
  std::map<Key, Interm> t1;
  std::map<Key, Combo> unused;
  left_stages(le, W, M, &tmp, &t1, &unused);
  p->g1 = tmp.g1;
  p->ws1 = tmp.ws1;
  struct T1Blk {
    int ip, j;
    int64_t off, len;
  };
  std::map<std::pair<int, int>, std::vector<T1Blk>> by_bl_s;
  for (const auto& kv : t1) {
    const int bl = kv.first[0], s = kv.first[1], i = kv.first[2];
    const int lb = le.block_of(bl, i), mb = M.block_of(s, i);
    if (lb < 0 || mb < 0) continue;
    by_bl_s[{bl, s}].push_back(T1Blk{le.blocks[lb].b, M.blocks[mb].c, kv.second.off,
                                     (int64_t)kv.second.rows * kv.second.cols});
  }
  // Y[br, s'](al', ar) = M[s'](al', ar') R[br](ar', ar)
  p->gy.ta = Trans::N;
  p->gy.tb = Trans::N;
  std::map<Key, Interm> y;
  int64_t off = 0;
  for (const Block& mb : M.blocks) {
    const int so = mb.a, ip = mb.b, jp = mb.c;
    for (int br = 0; br < W.wr; ++br) {
      const int j = M.nsym ? M.right.find(sub(M.right.q[jp], re.t[br])) : 0;
      if (j < 0) continue;
      const int rb = re.block_of(br, j);
      if (rb < 0 || re.blocks[rb].b != jp) continue;
      const int64_t rows = M.left.dim[ip], cols = M.right.dim[j], K = M.right.dim[jp];
      y[Key{br, so, ip, j}] = Interm{off, (int)rows, (int)cols};
      p->gy.add(off, (int)cols, (int)rows, (int)cols, {seg(mb.off, K, re.blocks[rb].off, cols, K)});
      off += rows * cols;
    }
  }
  p->wsy = off;
  p->nG = (int64_t)W.d * W.d * W.wl * W.wr;
  for (int so = 0; so < W.d; ++so)
    for (int s = 0; s < W.d; ++s)
      for (int bl = 0; bl < W.wl; ++bl)
        for (int br = 0; br < W.wr; ++br) {
          DotTask t{};
          t.out = (((int64_t)so * W.d + s) * W.wl + bl) * W.wr + br;
          t.seg0 = (int32_t)p->segs.size();
          auto it = by_bl_s.find({bl, s});
          if (it != by_bl_s.end())
            for (const T1Blk& b : it->second) {
              auto yt = y.find(Key{br, so, b.ip, b.j});
              if (yt == y.end()) continue;
              p->segs.push_back(DotSeg{b.off, yt->second.off, b.len});
              p->dot_flops += 2.0 * b.len;
            }
          t.nseg = (int32_t)p->segs.size() - t.seg0;
          p->tasks.push_back(t);
        }
  p->g1.finalize_bytes(p->g1.ta, p->g1.tb);
  p->gy.finalize_bytes(p->gy.ta, p->gy.tb);
  p->g1.tiles = choose_tiles(p->g1);
  p->gy.tiles = choose_tiles(p->gy);
  const int64_t w1 = p->ws1 > 0 ? p->ws1 : 1, wy = p->wsy > 0 ? p->wsy : 1;
  if (!gemm_ok(p->g1.ta, p->g1.tb, p->g1.tasks, p->g1.segs, le.size, M.size, w1, err) ||
      !gemm_ok(p->gy.ta, p->gy.tb, p->gy.tasks, p->gy.segs, M.size, re.size, wy, err)) {
    *err = "internal planning error: " + *err;
    return DMRG3S_ERR_SHAPE;
  }
  // sliced form over the virtual operand arrays A = [L | M], B = [M | R] and
  // the output [T1 | Y]; then each operand's blocks back to its own array
  p->sliced = false;
  if (p->flops() * tile_fill(p->g1, &p->gy) >= kSlicedMinFlops) {
    const int64_t nL = le.size, nM = M.size, nR = re.size;
    GemmStage g;
    g.ta = p->g1.ta;
    g.tb = p->g1.tb;
    append_gemm(g, p->g1, 0, 0, 0);
    append_gemm(g, p->gy, nL, nM, w1);
    bool ok = p->g1.ta == p->gy.ta && p->g1.tb == p->gy.tb && build_sliced(g, true, nullptr, false, {}, &p->s, err) &&
              sliced_ok(g, p->s, nL + nM, nM + nR, w1 + wy, 0, err);
    auto split = [&](std::vector<SlGroup>& gs, std::vector<SlMember>& ms, int64_t n0) {
      std::vector<SlGroup> ga, gb;
      for (SlGroup q : gs) {
        const bool second = ms[q.m0].src >= n0;
        for (int k = 0; k < q.nm; ++k) {
          ok = ok && (ms[q.m0 + k].src >= n0) == second;
          if (second) ms[q.m0 + k].src -= n0;
        }
        (second ? gb : ga).push_back(q);
      }
      p->slices.add(ga, ms);
      p->slices.add(gb, ms);
    };
    if (ok) {
      split(p->s.gA, p->s.mA, nL);
      split(p->s.gB, p->s.mB, nM);
      for (size_t k = p->g1.segs.size(); k < p->s.segs.size(); ++k) {
        p->s.segs[k].offA -= nL;
        p->s.segs[k].offB -= nM;
      }
      for (SlUnit& u : p->s.units) u.sel = u.seg0 >= (int32_t)p->g1.segs.size() ? 1 : 0;
      ok = slice_table_ok(p->slices, err);
    }
    if (!ok) {
      *err = "internal planning error: " + *err;
      return DMRG3S_ERR_SHAPE;
    }
    p->sliced = true;
  }
  for (const DotSeg& g : p->segs)
    if (g.offA < 0 || g.offB < 0 || g.len < 0 || g.offA + g.len > p->ws1 ||
        g.offB + g.len > p->wsy) {
      *err = "internal planning error: gradient segment out of bounds";
      return DMRG3S_ERR_SHAPE;
    }
  return DMRG3S_OK;
}

}  // namespace dmrg3s
