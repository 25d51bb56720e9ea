// The device-side cycle loop of the solves (loop.cu) and its construction.
#pragma once
#include "solver.h"

namespace gbmg {

// pr2, pf2: n partials each of ||r||^2 and ||F||^2 of the initial residual.  Sums them,
// starts the books in L (device) and H (the device address of mapped host memory).
cudaError_t launch_loop_begin(cudaStream_t st, const double* pr2, const double* pf2, long long n, double tol, int maxv,
                              double* r2_out, double* f2_out, LoopState* L, LoopState* H);
cudaError_t launch_loop_gate(cudaStream_t st, const LoopState* L, cudaGraphConditionalHandle w);
cudaError_t launch_loop_check(cudaStream_t st, const double* part, long long n, double* r2_out, LoopState* L,
                              LoopState* H, cudaGraphConditionalHandle w, cudaGraphConditionalHandle f, int second);

// A loop runs unless cycle graphs are off, families are being timed (the event nodes of a
// timed cycle cannot stand in a conditional body) or an earlier construction failed.
inline bool loop_usable(const gbmg_ctx* c) { return !c->cyc_off && !c->loop_off && c->prof_mask == 0 && c->loop_dev; }

// Builds the loop graph into `exec`: gate, WHILE (cycle 0, check, IF (cycle 1, check)).
// cycle() queues one cycle on c->stream and leaves its `npart` residual partials in
// c->partials; it is called twice, for the two parities in turn.  On any failure the context
// goes back to a graph launch per cycle (loop_off) and nothing is left behind.
template <class Cycle>
void build_loop(gbmg_ctx* c, Cycle cycle, long long npart, cudaGraphExec_t& exec, long long& kernels) {
  cudaStream_t user = c->stream;
  const long long k0 = launch_count();
  cudaGraph_t g = nullptr, ended = nullptr;
  cudaGraphExec_t x = nullptr;
  long long per_cycle = 0;
  auto attempt = [&]() -> bool {
    if (!c->cap_stream && cudaStreamCreateWithFlags(&c->cap_stream, cudaStreamNonBlocking) != cudaSuccess) return false;
    c->stream = c->cap_stream;
    if (cudaGraphCreate(&g, 0) != cudaSuccess) return false;
    cudaGraphConditionalHandle w, f;
    if (cudaGraphConditionalHandleCreate(&w, g, 0, cudaGraphCondAssignDefault) != cudaSuccess) return false;
    // captures body() into `into`; the last node it leaves is the one later work depends on
    auto record = [&](cudaGraph_t into, auto body, cudaGraphNode_t* last) -> bool {
      if (cudaStreamBeginCaptureToGraph(c->stream, into, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal) !=
          cudaSuccess)
        return false;
      bool ok = body();
      cudaStreamCaptureStatus cs;
      const cudaGraphNode_t* deps = nullptr;
      const cudaGraphEdgeData* edges = nullptr;
      size_t nd = 0;
      ok = ok && cudaStreamGetCaptureInfo(c->stream, &cs, nullptr, nullptr, &deps, &edges, &nd) == cudaSuccess && nd == 1;
      if (ok) *last = deps[0];
      return cudaStreamEndCapture(c->stream, &ended) == cudaSuccess && ok;
    };
    auto conditional = [&](cudaGraph_t in, cudaGraphNode_t after, cudaGraphConditionalHandle h,
                           cudaGraphConditionalNodeType type, cudaGraph_t* body) -> bool {
      cudaGraphNodeParams p = {};
      p.type = cudaGraphNodeTypeConditional;
      p.conditional.handle = h;
      p.conditional.type = type;
      p.conditional.size = 1;
      cudaGraphNode_t n;
      if (cudaGraphAddNode(&n, in, &after, nullptr, 1, &p) != cudaSuccess) return false;
      *body = p.conditional.phGraph_out[0];
      return true;
    };
    cudaGraphNode_t last;
    cudaGraph_t b0, b1;
    if (!record(g, [&]() { return launch_loop_gate(c->stream, c->loop_dev, w) == cudaSuccess; }, &last)) return false;
    if (!conditional(g, last, w, cudaGraphCondTypeWhile, &b0)) return false;
    if (cudaGraphConditionalHandleCreate(&f, b0, 0, cudaGraphCondAssignDefault) != cudaSuccess) return false;
    auto body = [&](int second) {
      return cycle() == GBMG_OK && launch_loop_check(c->stream, c->partials, npart, c->scal + S_R2, c->loop_dev,
                                                     c->loop_host_dev, w, f, second) == cudaSuccess;
    };
    const long long k1 = launch_count();
    if (!record(b0, [&]() { return body(0); }, &last)) return false;
    per_cycle = launch_count() - k1;
    if (!conditional(b0, last, f, cudaGraphCondTypeIf, &b1)) return false;
    if (!record(b1, [&]() { return body(1); }, &last)) return false;
    return cudaGraphInstantiate(&x, g, 0) == cudaSuccess;
  };
  const bool ok = attempt();
  c->stream = user;
  note_launches(-(launch_count() - k0));
  if (g) cudaGraphDestroy(g);
  if (!ok) {
    (void)cudaGetLastError();
    if (x) cudaGraphExecDestroy(x);
    c->loop_off = true;
    return;
  }
  exec = x;
  kernels = per_cycle;
}

// Launches the loop after launch_loop_begin; ev marks its end on the stream.
inline gbmg_status loop_launch(gbmg_ctx* c, cudaGraphExec_t exec) {
  if (!c->loop_ev) TRY(cudaEventCreateWithFlags(&c->loop_ev, cudaEventDisableTiming));
  TRY(cudaGraphLaunch(exec, c->stream));
  note_launch();
  TRY(cudaEventRecord(c->loop_ev, c->stream));
  return GBMG_OK;
}

// Waits for the loop (not for work queued after it) and reads its books.
inline gbmg_status loop_result(gbmg_ctx* c, long long kernels, gbmg_stats& st) {
  TRY(cudaEventSynchronize(c->loop_ev));
  const LoopState& H = *c->loop_host;
  st.cycles = H.cycles;
  st.status = H.status;
  st.rel_res0 = H.rel0;
  st.rel_res = H.rel;
  for (int k = 0; k < H.cycles && k < 64; ++k) st.res_hist[k] = H.hist[k];
  note_launches(kernels * H.cycles);
  return GBMG_OK;
}

}  // namespace gbmg
