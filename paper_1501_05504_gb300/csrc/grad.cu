// MPO-entry gradient of the DMRG3S energy functional.
//
// <Psi|H|Psi> is linear in every MPO tensor W_i (the network of Sec. II), so
// its derivative with respect to the entries of W_i is the same network with
// W_i taken out:
//   G_i[s', s, bl, br] = sum L_{i-1}[bl](al', al) M_i[s'](al', ar') M_i[s](al, ar)
//                            R_{i+1}[br](ar', ar)
// and, divided by <Psi|Psi>, dE/dtheta = sum_i <G_i, dW_i/dtheta> at fixed
// Psi (Hellmann-Feynman at a stationary state).  The contraction reuses the
// first stage of the H_eff order of Sec. V (T1 = L M), contracts the bra copy
// of M with R on the other side (Y = M R), and finishes with one blockwise
// inner product per entry of G.  FP64 throughout.
#include <cstring>

#include "context.hpp"
#include "dmrg3s.h"
#include "validate.hpp"

namespace dmrg3s {

// Sliced form (kernels_sliced.cu): L and R and both views of M sliced by one
// launch, T1 and Y by one grouped GEMM, then the inner products.  It runs
// where its intermediates fit the workspace, else the plain form.
dmrg3s_status run_mpo_grad(Context* c, const DeviceGradPlan& dp, const double* L, const double* M,
                           const double* R, double* G, cudaStream_t st) {
  const GradPlan& p = dp.host;
  if ((size_t)(p.ws1 + p.wsy) * sizeof(double) > c->ws_bytes)
    return fail(c, DMRG3S_ERR_OOM, "context workspace too small for the gradient intermediates");
  double* ws1 = reinterpret_cast<double*>(c->ws);
  const int64_t w1 = p.ws1 > 0 ? p.ws1 : 1, wy = p.wsy > 0 ? p.wsy : 1;
  double* wsy = ws1 + (p.sliced ? w1 : p.ws1);
  Profiler& pr = c->prof;
  const int64_t a = slot_round(w1 + wy), b = a + slot_round((p.s.nA + 3) / 4),
                e = b + slot_round((p.s.nB + 3) / 4),
                parts = kSlParts * (int64_t)p.s.units.size(),
                end = e + slot_round(((int64_t)p.s.neA + p.s.neB + 1 + kSlFixInts * parts + 1) / 2);
  if (p.sliced && (size_t)end * sizeof(double) <= c->ws_bytes) {
    uint16_t* pA = reinterpret_cast<uint16_t*>(ws1 + a);
    uint16_t* pB = reinterpret_cast<uint16_t*>(ws1 + b);
    int32_t* eA = reinterpret_cast<int32_t*>(ws1 + e);
    int32_t* eB = eA + p.s.neA;
    SlOperands ops{};
    ops.op[0] = SlOperand{L, pA, eA, 1.0, nullptr, 0};
    ops.op[1] = SlOperand{M, pA, eA, 1.0, nullptr, 0};
    ops.op[2] = SlOperand{M, pB, eB, 1.0, nullptr, 0};
    ops.op[3] = SlOperand{R, pB, eB, 1.0, nullptr, 0};
    ops.fix = eB + p.s.neB;
    ops.nfix = 1;
    launch_slice(dp.sl_groups, dp.sl_cta_group, p.slices.cta.back(), dp.sl_members, ops, st);
    const int id = pr.on ? pr.begin(kProfAuxGemm, p.g1.flops + p.gy.flops, p.g1.bytes + p.gy.bytes, st) : -1;
    launch_gemm_sliced(sliced_tables(dp.s, p.s), pA, pB, eA, eB, SlSource{L, M, M, R, 0, 0, 1.0, 0, 0}, ws1,
                       nullptr, false, nullptr, sl_fix(ops.fix, 0, 1, p.s.units.size()), c->d_err, c->wait_ns, st);
    if (id >= 0) pr.end(id, st);
  } else {
    wsy = ws1 + p.ws1;
    const DeviceGradPlan::Gemm* d[2] = {&dp.g1, &dp.gy};
    const GemmStage* g[2] = {&p.g1, &p.gy};
    const double *A[2] = {L, M}, *B[2] = {M, R};
    double* C[2] = {ws1, wsy};
    for (int i = 0; i < 2; ++i) {
      if (g[i]->tiles.empty()) continue;
      const int id = pr.on ? pr.begin(kProfAuxGemm, g[i]->flops, g[i]->bytes, st) : -1;
      launch_gemm_f64(g[i]->ta, g[i]->tb, d[i]->tiles, (int)g[i]->tiles.size(), d[i]->tasks, d[i]->segs,
                      A[i], B[i], C[i], st);
      if (id >= 0) pr.end(id, st);
    }
  }
  launch_dots(dp.tasks, (int)p.tasks.size(), dp.segs, ws1, wsy, G, st);
  if (cudaGetLastError() != cudaSuccess) return fail(c, DMRG3S_ERR_CUDA, "gradient launch");
  return DMRG3S_OK;
}

}  // namespace dmrg3s

using namespace dmrg3s;

extern "C" dmrg3s_status dmrg3s_mpo_grad_site(dmrg3s_ctx ctx, const dmrg3s_env* L,
                                              const dmrg3s_mpo_site* W, const dmrg3s_env* R,
                                              const dmrg3s_site* M, double* G,
                                              dmrg3s_stream stream) {
  Context* c = reinterpret_cast<Context*>(ctx);
  if (!c || !L || !W || !R || !M || !G) return fail(c, DMRG3S_ERR_ARG, "NULL argument");
  dmrg3s_status st;
  RawKey key;
  key.env(*L);
  key.mpo(*W, true);       // (its values are checked against the charges)
  key.env(*R);
  key.site(*M);
  const DeviceGradPlan* p = nullptr;
  if (key.ok) {
    auto it = c->grad_by_args.find(key);
    if (it != c->grad_by_args.end()) p = it->second;
  }
  if (!p) {
    std::string err;
    EnvLayout le, re;
    MpoLayout w;
    SiteLayout m;
    if ((st = make_env(L, &le, &err)) || (st = make_env(R, &re, &err)) ||
        (st = make_mpo(W, &w, &err)) || (st = make_site(M, &m, &err)))
      return fail(c, st, err);
    if ((st = check_site_mpo(m, w, &err)) ||
        (st = check_env(le, m.left, w.wl, w.tl, "L", &err)) ||
        (st = check_env(re, m.right, w.wr, w.tr, "R", &err)))
      return fail(c, st, err);
    if (!L->data || !R->data || !M->data) return fail(c, DMRG3S_ERR_ARG, "NULL device data pointer");
    if ((st = use_device(c))) return st;
    if ((st = grad_plan(c, le, w, re, m, &p))) return st;
    remember(&c->grad_by_args, key, p);
  }
  if (!L->data || !R->data || !M->data) return fail(c, DMRG3S_ERR_ARG, "NULL device data pointer");
  if ((st = use_device(c))) return st;
  return run_mpo_grad(c, *p, L->data, M->data, R->data, G, reinterpret_cast<cudaStream_t>(stream));
}
