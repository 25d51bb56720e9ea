// Curvilinear (moving-mesh) solve and the adjoint solves.
//
// Geometry (Sec. 4.2, Appendix B): psi is restricted to every level by full
// weighting and the triad, volume element and B = sqrt(g) g^-1 are rebuilt there;
// the coarsest level's operator is inverted exactly (pseudo-inverse).
// Solve (Sec. 4.3): L phi = f with L = M / J, f = delta - sum(delta J)/sum(J)
// (Eq. solvability), weighted-Jacobi V-cycles in FP32 inside a double-float
// defect correction, gauge: mean of phi removed.
// Adjoint (Sec. 4.8, Eq. adj_rhs / adj_op, written with the exact transpose):
// M^T lam = phi_bar - mean(phi_bar) by the same V-cycle on M^T / J,
// delta_bar = J (lam - sum(J lam)/sum(J)), psi_bar through the geometry.
// With the symmetric variant (opts.curv_sym) both solves use S, its own transpose.
#include <cstring>
#include <vector>

#include "kernels.h"
#include "loop.h"
#include "solver.h"

using namespace gbmg;

namespace {

enum CurvScal { S_SUMJ = 6, S_MW = 9, S_SLAM = 10, S_PINV = 20 };  // (S_PINV holds an int)

// operator form of the forward (tr false) or transposed (tr true) problem: 0 = M, 1 = M^T, 2 = S
int curv_form(const gbmg_ctx* c, bool tr) { return c->o.curv_sym ? 2 : (tr ? 1 : 0); }

// nu weighted-Jacobi sweeps of e (ping-pong with eo)
gbmg_status curv_smooth(gbmg_ctx* c, int l, float*& e, float*& eo, const float* r, int nu, bool tr) {
  const Level& L = c->lv[l];
  for (int k = 0; k < nu; ++k) {
    ProfScope ps(c, l == 0 ? GBMG_PROF_CURV0 : GBMG_PROF_OFF);
    TRY(launch_curv_jacobi(c->stream, L.d, L.cc, r, e, eo, curv_form(c, tr), (float)c->o.omega));
    std::swap(e, eo);
  }
  return GBMG_OK;
}

// Curvilinear V-cycle for L_l e = r (or the transposed-solve operator), one kernel
// per operation (Sec. 4.3, Eq. curv_error; Appendix B), from e = 0.  On entry e holds the
// first pre-smoothing sweep, which is pointwise and written by the kernel that makes r
// (nu1 = 0: zeros).
gbmg_status vcycle_curv(gbmg_ctx* c, int l, float*& e, float*& eo, const float* r, bool tr) {
  const Level& L = c->lv[l];
  if (l == c->L - 1) {
    TRY(launch_coarse_matvec<float>(c->stream, c->nc, tr ? c->G32T : c->G32, r, e));
    return GBMG_OK;
  }
  TRYS(curv_smooth(c, l, e, eo, r, c->o.nu1 - 1, tr));
  const Level& C = c->lv[l + 1];
  float* ce = (float*)C.e;
  float* ceo = (float*)C.e2;
  const bool smoothed = l + 1 < c->L - 1;
  float* const first = smoothed && c->o.nu1 > 0 ? ce : nullptr;
  if (curv_residual_restrict_ok(L.d)) {
    TRY(launch_curv_residual_restrict(c->stream, L.d, L.cc, r, e, curv_form(c, tr), (float*)C.r, C.cc, first,
                                      (float)c->o.omega));
  } else {
    TRY(launch_curv_residual(c->stream, L.d, L.cc, r, e, (float*)L.t, curv_form(c, tr)));
    TRY(launch_curv_restrict(c->stream, L.d, (const float*)L.t, (float*)C.r, C.cc, first, (float)c->o.omega));
  }
  if (smoothed && c->o.nu1 == 0) TRY(cudaMemsetAsync(ce, 0, (size_t)ncell(C.d) * sizeof(float), c->stream));
  TRYS(vcycle_curv(c, l + 1, ce, ceo, (const float*)C.r, tr));
  TRY(launch_prolong_add<float>(c->stream, C.d, ce, e));
  TRYS(curv_smooth(c, l, e, eo, r, c->o.nu2, tr));
  return GBMG_OK;
}

// Buffers of one cycle: the potential before and after, and the finest level's error
// buffer that holds the cycle's first sweep and the other one of the pair.
struct CurvBufs {
  float2 *phi, *phi_next;
  float *e, *eo;
};

// The buffers after a cycle: the potential's pair swaps; the V-cycle ends in e or eo after
// its nu1 - 1 + nu2 swaps, and the next first sweep goes to the other one.
CurvBufs curv_next(const gbmg_ctx* c, const CurvBufs& b) {
  const int swaps = c->L > 1 ? (c->o.nu1 > 0 ? c->o.nu1 - 1 : 0) + c->o.nu2 : 0;
  return swaps % 2 ? CurvBufs{b.phi_next, b.phi, b.e, b.eo} : CurvBufs{b.phi_next, b.phi, b.eo, b.e};
}

// One cycle of the curvilinear solve on c->stream: FP32 V-cycle on r0, then phi_next = phi +
// e, r0 = the double-float residual with the partial sums of its norm, and the next cycle's
// first sweep in one kernel.  b becomes the next cycle's buffers.  curv_cycle adds the norm
// and copies the scalars to pinned host memory.  Without timed families the whole loop is
// one graph (loop.h); otherwise: the launches depend only on the context, the orientation and the buffers, which alternate
// with the potential's parity, so after a cycle has run eagerly each (orientation, parity)
// is captured once as a CUDA graph and replayed (the coefficients change in place; timed
// families are timed by event nodes).
gbmg_status curv_cycle_step(gbmg_ctx* c, bool tr, float* r0, CurvBufs& b) {
  const Level& L0 = c->lv[0];
  double* sc = c->scal;
  float* e = b.e;
  float* eo = b.eo;
  TRYS(vcycle_curv(c, 0, e, eo, r0, tr));
  // (a single-level hierarchy's cycle is the coarsest solve: its next cycle needs no sweep)
  const bool first = c->L > 1 && c->o.nu1 > 0;
  {
    ProfScope ps(c, GBMG_PROF_DF0);
    TRY(launch_curv_df_step(c->stream, L0.d, L0.cc, c->F_df, sc + S_MEAN_F, tr ? 0 : 1, b.phi, e, b.phi_next,
                            curv_form(c, tr), r0, first ? eo : nullptr, (float)c->o.omega, c->partials, nullptr));
  }
  if (c->L > 1 && !first) TRY(cudaMemsetAsync(eo, 0, (size_t)ncell(L0.d) * sizeof(float), c->stream));
  b = curv_next(c, b);
  return GBMG_OK;
}
gbmg_status curv_cycle(gbmg_ctx* c, bool tr, float* r0, CurvBufs& b) {
  const Level& L0 = c->lv[0];
  double* sc = c->scal;
  TRYS(curv_cycle_step(c, tr, r0, b));
  TRY(launch_norm_sum(c->stream, c->partials, curv_df_partials(L0.d, curv_form(c, tr)), sc + S_R2));
  TRY(launch_scalars_to_host(c->stream, c->scal, c->host_scal_dev, 8));
  return GBMG_OK;
}

// Mixed-precision solve of L u = f (forward, f = src - weighted mean) or of the
// transposed problem M^T u = src - mean(src) (tr).  u_in NULL starts from zero;
// u_out NULL leaves the result in c->curv_phi only.
gbmg_status curv_solve_impl(gbmg_ctx* c, const double* src, const double* u_in, double* u_out, double tol, int maxv,
                            gbmg_stats& st, bool tr) {
  const Level& L0 = c->lv[0];
  const long long n = ncell(L0.d);
  double* part = c->partials;
  double* part1 = c->partials + c->npart;
  double* part2 = c->partials + 2 * c->npart;
  double* sc = c->scal;
  const long long pr = df_partial_count(n), pc = curv_df_partials(L0.d, curv_form(c, tr));
  TRY(launch_f64_to_df(c->stream, n, src, c->F_df, part));
  if (!tr) {
    TRY(launch_wsum(c->stream, n, src, L0.cc.J, part, part1));
    TRY(launch_finalize(c->stream, part, pr, sc + S_SUM_F, 1.0));
    TRY(launch_finalize(c->stream, part1, pr, sc + S_SUMJ, 1.0));
    TRY(launch_ratio(c->stream, sc + S_SUM_F, sc + S_SUMJ, sc + S_MEAN_F));
  } else {
    TRY(launch_finalize(c->stream, part, pr, sc + S_MEAN_F, 1.0 / (double)n));
  }
  if (u_in) {
    TRY(launch_f64_to_df(c->stream, n, u_in, c->phi_df, nullptr));
  } else {
    TRY(cudaMemsetAsync(c->phi_df, 0, (size_t)n * sizeof(float2), c->stream));
  }
  float* r0 = (float*)L0.r;
  CurvBufs b{c->phi_df, c->phi_df2, (float*)L0.e, (float*)L0.e2};
  const bool first = c->L > 1 && c->o.nu1 > 0;
  TRY(launch_curv_df_step(c->stream, L0.d, L0.cc, c->F_df, sc + S_MEAN_F, tr ? 0 : 1, b.phi, nullptr, nullptr,
                          curv_form(c, tr), r0, first ? b.e : nullptr, (float)c->o.omega, part, part1));
  if (c->L > 1 && !first) TRY(cudaMemsetAsync(b.e, 0, (size_t)n * sizeof(float), c->stream));
  const int k = tr ? 1 : 0;
  if (loop_usable(c) && !c->loop_exec[k]) {
    CurvBufs q = b;
    build_loop(c, [&]() { return curv_cycle_step(c, tr, r0, q); }, pc, c->loop_exec[k], c->loop_kernels[k]);
  }
  if (loop_usable(c) && c->loop_exec[k]) {
    TRY(launch_loop_begin(c->stream, part, part1, pc, tol, maxv, sc + S_R2, sc + S_F2, c->loop_dev, c->loop_host_dev));
    TRYS(loop_launch(c, c->loop_exec[k]));
    if (u_out) {
      const int* cycles = &c->loop_dev->cycles;
      TRY(launch_df_update(c->stream, n, c->phi_df, nullptr, part2, c->phi_df2, cycles));
      TRY(launch_finalize(c->stream, part2, pr, sc + S_MEAN_PHI, 1.0 / (double)n));
      TRY(launch_df_to_f64(c->stream, n, c->phi_df, sc + S_MEAN_PHI, u_out, c->phi_df2, cycles));
    }
    TRYS(loop_result(c, c->loop_kernels[k], st));
    c->curv_phi = st.cycles % 2 ? c->phi_df2 : c->phi_df;
    return GBMG_OK;
  }
  TRY(launch_norm_sum(c->stream, part, pc, sc + S_R2));
  TRY(launch_norm_sum(c->stream, part1, pc, sc + S_F2));
  double rel = 0.0;
  TRYS(read_rel(c, rel));
  Monitor mon(st, tol, maxv);
  mon.start(rel);
  while (!mon.done()) {
    sync_graph_mask(c);
    const bool graphs = c->curv_warm[k] && !c->cyc_off;
    const int g = 2 * k + (b.phi == c->phi_df ? 0 : 1);
    CurvBufs next = b;
    if (graphs && !c->curv_exec[g])
      TRYS(capture_graph(c, 2 + g,
                         [&]() {
                           CurvBufs q = b;
                           return curv_cycle(c, tr, r0, q);
                         },
                         c->curv_exec[g], c->curv_kernels[g]));
    const bool replay = graphs && c->curv_exec[g];
    if (replay) {
      TRY(cudaGraphLaunch(c->curv_exec[g], c->stream));
      note_launches(c->curv_kernels[g]);
      next = curv_next(c, b);
    } else {
      TRYS(curv_cycle(c, tr, r0, next));
      c->curv_warm[k] = true;
    }
    b = next;
    TRYS(rel_from_host(c, rel));
    if (replay) gprof_collect(c, 2 + g);
    if (mon.record(rel)) break;
  }
  c->curv_phi = b.phi;
  if (u_out) {
    TRY(launch_df_update(c->stream, n, b.phi, nullptr, part2));
    TRY(launch_finalize(c->stream, part2, pr, sc + S_MEAN_PHI, 1.0 / (double)n));
    TRY(launch_df_to_f64(c->stream, n, b.phi, sc + S_MEAN_PHI, u_out));
  }
  return GBMG_OK;
}

gbmg_status ensure_adjoint_scratch(gbmg_ctx* c) {
  const long long n = ncell(c->lv[0].d);
  if (!c->adj_lam) {
    TRY(cudaMalloc((void**)&c->adj_lam, (size_t)n * sizeof(double)));
    c->owned.push_back(c->adj_lam);
  }
  if (!c->adj_S) {
    TRY(cudaMalloc((void**)&c->adj_S, (size_t)n * 6 * sizeof(double)));
    c->owned.push_back(c->adj_S);
  }
  return GBMG_OK;
}

}  // namespace

gbmg_status gbmg::curv_solve(gbmg_ctx* c, const double* F, double* phi, double tol, int maxv, gbmg_stats& st) {
  return curv_solve_impl(c, F, phi, phi, tol, maxv, st, false);
}

namespace {

// The operator's diagonal on every level (the V-cycle does not smooth the coarsest, but
// mg_curv_smooth takes it too).
gbmg_status build_diag(gbmg_ctx* c) {
  for (const Level& L : c->lv) {
    TRY(launch_curv_diag(c->stream, L.d, L.cc, curv_form(c, false), (float*)L.cc.D));
  }
  return GBMG_OK;
}

// The coarsest inverses on the host, where the GPU has no room for the kernel's resident grid
// (up to 130 CTAs: a partition of a few SMs).  The same bits.
gbmg_status coarsest_on_host(gbmg_ctx* c, const char* who) {
  const size_t nc = c->nc, n2 = nc * nc;
  std::vector<float> Jc(nc);
  std::vector<double> Lm(n2), G;
  TRY(cudaMemcpyAsync(Jc.data(), c->lv[c->L - 1].cc.J, nc * sizeof(float), cudaMemcpyDeviceToHost, c->stream));
  for (int tr = 0; tr < 2; ++tr) {
    TRY(cudaMemcpyAsync(Lm.data(), c->dense + tr * n2, n2 * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    TRY(cudaStreamSynchronize(c->stream));
    for (float v : Jc)
      if (!(v > 0.f)) return fail(GBMG_ERR_INVALID_ARG, std::string(who) + ": non-positive volume element on the coarsest level");
    const std::vector<double> w(Jc.begin(), Jc.end());
    if (!dense_pinv((int)nc, Lm, w, G)) return fail(GBMG_ERR_INVALID_ARG, std::string(who) + ": coarsest operator is singular");
    const std::vector<float> G32(G.begin(), G.end());
    TRY(cudaMemcpy(tr ? c->G64T : c->G64, G.data(), n2 * sizeof(double), cudaMemcpyHostToDevice));
    TRY(cudaMemcpy(tr ? c->G32T : c->G32, G32.data(), n2 * sizeof(float), cudaMemcpyHostToDevice));
  }
  return GBMG_OK;
}

// Exact inverses of the coarsest operator and of its transposed-solve twin (minimum-norm,
// left null vector J), built from the coarsest level's coefficients.  Waits for the stream.
gbmg_status build_coarsest(gbmg_ctx* c, const char* who) {
  const Level& C = c->lv[c->L - 1];
  const int nc = c->nc;
  const size_t n2 = (size_t)nc * nc;
  int* const status = reinterpret_cast<int*>(c->scal + S_PINV);
  for (int tr = 0; tr < 2; ++tr)
    TRY(launch_curv_dense(c->stream, C.d, C.cc, curv_form(c, tr != 0), c->dense + tr * n2));
  const cudaError_t e = c->refuse ? cudaErrorCooperativeLaunchTooLarge
                                  : launch_coarse_inverse(c->stream, nc, c->dense, c->dense + 2 * n2, C.cc.J, c->G64,
                                                          c->G64T, c->G32, c->G32T, status);
  if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
    (void)cudaGetLastError();
    return coarsest_on_host(c, who);
  }
  if (e != cudaSuccess) return cuda_fail(e, "launch_coarse_inverse");
  TRY(launch_scalars_to_host(c->stream, c->scal + S_PINV, c->host_scal_dev + S_PINV, 1));
  TRY(cudaStreamSynchronize(c->stream));
  int flags;
  std::memcpy(&flags, c->host_scal + S_PINV, sizeof(flags));
  if (flags & 4) return fail(GBMG_ERR_CUDA, std::string(who) + ": the coarsest inversion timed out");
  if (flags & 2) return fail(GBMG_ERR_INVALID_ARG, std::string(who) + ": non-positive volume element on the coarsest level");
  if (flags & 1) return fail(GBMG_ERR_INVALID_ARG, std::string(who) + ": coarsest operator is singular");
  return GBMG_OK;
}

}  // namespace

extern "C" gbmg_status mg_set_geometry(gbmg_ctx* c, const double* psi_dev) {
  if (!c || !psi_dev) return fail(GBMG_ERR_INVALID_ARG, "mg_set_geometry: NULL argument");
  if (c->o.op != GBMG_OP_CURV19) return fail(GBMG_ERR_STATE, "mg_set_geometry: context is not curvilinear");
  DeviceGuard g(c->device);
  c->geom_ready = false;
  for (int l = 0; l < c->L; ++l) {
    Level& L = c->lv[l];
    if (l == 0) {
      TRY(cudaMemcpyAsync(L.psi, psi_dev, (size_t)ncell(L.d) * sizeof(double), cudaMemcpyDeviceToDevice, c->stream));
    } else {
      TRY(launch_restrict<double>(c->stream, c->lv[l - 1].d, c->lv[l - 1].psi, L.psi, true));
    }
    CurvCoefOut o;
    o.J = (float*)L.cc.J;
    for (int k = 0; k < 6; ++k) o.B[k] = (float*)L.cc.B[k];
    TRY(launch_geom(c->stream, L.d, L.psi, L.h, o));
  }
  TRYS(build_diag(c));
  TRYS(build_coarsest(c, "mg_set_geometry"));
  c->geom_ready = true;
  c->geom_from_psi = true;
  return GBMG_OK;
}

extern "C" gbmg_status mg_set_coefficients(gbmg_ctx* c, const float* J_dev, const float* B_dev) {
  if (!c || !J_dev || !B_dev) return fail(GBMG_ERR_INVALID_ARG, "mg_set_coefficients: NULL argument");
  if (c->o.op != GBMG_OP_CURV19) return fail(GBMG_ERR_STATE, "mg_set_coefficients: context is not curvilinear");
  DeviceGuard g(c->device);
  c->geom_ready = false;
  c->geom_from_psi = false;
  const size_t b0 = (size_t)ncell(c->lv[0].d) * sizeof(float);
  for (int l = 0; l < c->L; ++l) {
    Level& L = c->lv[l];
    if (l == 0) {
      TRY(cudaMemcpyAsync((float*)L.cc.J, J_dev, b0, cudaMemcpyDeviceToDevice, c->stream));
      for (int k = 0; k < 6; ++k)
        TRY(cudaMemcpyAsync((float*)L.cc.B[k], (const char*)B_dev + k * b0, b0, cudaMemcpyDeviceToDevice, c->stream));
    } else {
      // coarse coefficients: full-weighting restriction of the finer level's coefficients
      const Level& F = c->lv[l - 1];
      TRY(launch_restrict<float>(c->stream, F.d, F.cc.J, (float*)L.cc.J, true));
      for (int k = 0; k < 6; ++k) TRY(launch_restrict<float>(c->stream, F.d, F.cc.B[k], (float*)L.cc.B[k], true));
    }
  }
  TRYS(build_diag(c));
  TRYS(build_coarsest(c, "mg_set_coefficients"));
  c->geom_ready = true;
  return GBMG_OK;
}

extern "C" gbmg_status mg_solve_adjoint(gbmg_ctx* c, const double* phi_bar_dev, double* source_bar_dev,
                                        double* psi_bar_dev, const double* phi_dev, const double* source_dev,
                                        double tol, int max_vcycles, gbmg_stats* stats) {
  g_last_error.clear();
  if (!c || !phi_bar_dev || !source_bar_dev) return fail(GBMG_ERR_INVALID_ARG, "mg_solve_adjoint: NULL argument");
  if (!(tol >= 0.0)) return fail(GBMG_ERR_INVALID_ARG, "mg_solve_adjoint: tol must be >= 0");
  DeviceGuard g(c->device);
  const Level& L0 = c->lv[0];
  const long long n = ncell(L0.d);
  if (c->o.op == GBMG_OP_FLAT7) {
    // A is symmetric: source_bar = P A^+ P phi_bar is the same solve on the cotangent
    if (psi_bar_dev) return fail(GBMG_ERR_INVALID_ARG, "mg_solve_adjoint: psi_bar is only defined for the curvilinear operator");
    TRY(cudaMemsetAsync(source_bar_dev, 0, (size_t)n * sizeof(double), c->stream));
    return mg_solve(c, phi_bar_dev, nullptr, source_bar_dev, tol, max_vcycles, stats);
  }
  if (!c->geom_ready) return fail(GBMG_ERR_STATE, "mg_solve_adjoint: no geometry set");
  if (psi_bar_dev && (!phi_dev || !source_dev))
    return fail(GBMG_ERR_INVALID_ARG, "mg_solve_adjoint: psi_bar needs the forward solution and source");
  if (psi_bar_dev && !c->geom_from_psi)
    return fail(GBMG_ERR_STATE, "mg_solve_adjoint: psi_bar needs a geometry set from psi, not raw coefficients");
  TRYS(ensure_adjoint_scratch(c));
  gbmg_stats st;
  std::memset(&st, 0, sizeof(st));
  TRYS(curv_solve_impl(c, phi_bar_dev, nullptr, nullptr, tol, max_vcycles, st, true));
  double* part = c->partials;
  double* part1 = c->partials + c->npart;
  double* sc = c->scal;
  const long long pr = df_partial_count(n);
  // lam in FP64, s_lam = sum(J lam) / sum(J), delta_bar = J (lam - s_lam)
  TRY(launch_jscale(c->stream, n, c->curv_phi, L0.cc.J, nullptr, nullptr, c->adj_lam));
  TRY(launch_wsum(c->stream, n, c->adj_lam, L0.cc.J, part, part1));
  TRY(launch_finalize(c->stream, part, pr, sc + S_SUM_F, 1.0));
  TRY(launch_finalize(c->stream, part1, pr, sc + S_SUMJ, 1.0));
  TRY(launch_ratio(c->stream, sc + S_SUM_F, sc + S_SUMJ, sc + S_SLAM));
  TRY(launch_jscale(c->stream, n, c->curv_phi, L0.cc.J, sc + S_SLAM, source_bar_dev, nullptr));
  if (psi_bar_dev) {
    TRY(launch_wsum(c->stream, n, source_dev, L0.cc.J, part, part1));
    TRY(launch_finalize(c->stream, part, pr, sc + S_SUM_F, 1.0));
    TRY(launch_finalize(c->stream, part1, pr, sc + S_SUMJ, 1.0));
    TRY(launch_ratio(c->stream, sc + S_SUM_F, sc + S_SUMJ, sc + S_MW));
    TRY(launch_psibar(c->stream, L0.d, L0.psi, phi_dev, c->curv_phi, source_dev, sc + S_MW, sc + S_SLAM, L0.h,
                      c->o.curv_sym, (float2*)c->adj_S, psi_bar_dev));
  }
  TRY(cudaStreamSynchronize(c->stream));
  c->last = st;
  if (stats) *stats = st;
  return (gbmg_status)st.status;
}

// ------------------------------------------------------------------ components

extern "C" gbmg_status mg_curv_apply(gbmg_ctx* c, int level, int dtype, int transpose, int divide_by_J,
                                     const void* u, void* out) {
  if (!c || !u || !out || level < 0 || level >= c->L || (dtype != GBMG_F32 && dtype != GBMG_F64))
    return fail(GBMG_ERR_INVALID_ARG, "mg_curv_apply: bad argument");
  if (c->o.op != GBMG_OP_CURV19 || !c->geom_ready) return fail(GBMG_ERR_STATE, "mg_curv_apply: no geometry set");
  DeviceGuard g(c->device);
  const Level& L = c->lv[level];
  if (dtype == GBMG_F64)
    TRY(launch_curv_apply<double>(c->stream, L.d, L.cc, (const double*)u, (double*)out, curv_form(c, transpose != 0), divide_by_J ? 1 : 0));
  else
    TRY(launch_curv_apply<float>(c->stream, L.d, L.cc, (const float*)u, (float*)out, curv_form(c, transpose != 0), divide_by_J ? 1 : 0));
  return GBMG_OK;
}

// FP32 tiled kernels of the V-cycle's levels, one launch each (for tests and composition).
static gbmg_status curv_component_check(gbmg_ctx* c, int level, const void* a, const void* b, const void* o,
                                        const char* who) {
  if (!c || !a || !b || !o || level < 0 || level >= c->L) return fail(GBMG_ERR_INVALID_ARG, std::string(who) + ": bad argument");
  if (c->o.op != GBMG_OP_CURV19 || !c->geom_ready) return fail(GBMG_ERR_STATE, std::string(who) + ": no geometry set");
  return GBMG_OK;
}

extern "C" gbmg_status mg_curv_residual(gbmg_ctx* c, int level, int transpose, const float* r, const float* u,
                                        float* out) {
  TRYS(curv_component_check(c, level, r, u, out, "mg_curv_residual"));
  DeviceGuard g(c->device);
  const Level& L = c->lv[level];
  TRY(launch_curv_residual(c->stream, L.d, L.cc, r, u, out, curv_form(c, transpose != 0)));
  return GBMG_OK;
}

extern "C" gbmg_status mg_curv_smooth(gbmg_ctx* c, int level, int transpose, const float* e_in, const float* r,
                                      float* e_out) {
  TRYS(curv_component_check(c, level, r, r, e_out, "mg_curv_smooth"));
  if (e_in == e_out) return fail(GBMG_ERR_INVALID_ARG, "mg_curv_smooth: e_in and e_out must differ");
  DeviceGuard g(c->device);
  const Level& L = c->lv[level];
  const int form = curv_form(c, transpose != 0);
  if (e_in) TRY(launch_curv_jacobi(c->stream, L.d, L.cc, r, e_in, e_out, form, (float)c->o.omega));
  else TRY(launch_curv_jacobi_zero(c->stream, L.d, L.cc, r, e_out, (float)c->o.omega));
  return GBMG_OK;
}

extern "C" gbmg_status mg_curv_geometry(gbmg_ctx* c, int level, float* J_out, float* B_out) {
  if (!c || level < 0 || level >= c->L) return fail(GBMG_ERR_INVALID_ARG, "mg_curv_geometry: bad argument");
  if (c->o.op != GBMG_OP_CURV19 || !c->geom_ready) return fail(GBMG_ERR_STATE, "mg_curv_geometry: no geometry set");
  DeviceGuard g(c->device);
  const Level& L = c->lv[level];
  const size_t b = (size_t)ncell(L.d) * sizeof(float);
  if (J_out) TRY(cudaMemcpyAsync(J_out, L.cc.J, b, cudaMemcpyDeviceToDevice, c->stream));
  if (B_out)
    for (int k = 0; k < 6; ++k)
      TRY(cudaMemcpyAsync((char*)B_out + k * b, L.cc.B[k], b, cudaMemcpyDeviceToDevice, c->stream));
  return GBMG_OK;
}

extern "C" gbmg_status mg_curv_vcycle(gbmg_ctx* c, int transpose, const float* r, float* e_out) {
  if (!c || !r || !e_out) return fail(GBMG_ERR_INVALID_ARG, "mg_curv_vcycle: NULL argument");
  if (c->o.op != GBMG_OP_CURV19 || !c->geom_ready) return fail(GBMG_ERR_STATE, "mg_curv_vcycle: no geometry set");
  DeviceGuard g(c->device);
  const Level& L0 = c->lv[0];
  const long long n = ncell(L0.d);
  float* e = (float*)L0.e;
  float* eo = (float*)L0.e2;
  if (c->L > 1 && c->o.nu1 > 0) TRY(launch_curv_jacobi_zero(c->stream, L0.d, L0.cc, r, e, (float)c->o.omega));
  else TRY(cudaMemsetAsync(e, 0, (size_t)n * 4, c->stream));
  TRYS(vcycle_curv(c, 0, e, eo, r, transpose != 0));
  TRY(cudaMemcpyAsync(e_out, e, (size_t)n * 4, cudaMemcpyDeviceToDevice, c->stream));
  return GBMG_OK;
}
