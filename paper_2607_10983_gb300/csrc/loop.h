// The device-side cycle loop of the solves (loop.cu) and its construction.
#pragma once
#include "solver.h"

namespace gbmg {

// pr2, pf2: n partials each of ||r||^2 and ||F||^2 of the initial residual.  Sums them,
// starts the books in L (device) and H (the device address of mapped host memory).
cudaError_t launch_loop_begin(cudaStream_t st, const double* pr2, const double* pf2, long long n, double tol, int maxv,
                              double* r2_out, double* f2_out, LoopState* L, LoopState* H);
// The sum of n partials in the order of the loop's checks, for the solves that the host drives:
// their histories have the same bits.
cudaError_t launch_norm_sum(cudaStream_t st, const double* part, long long n, double* out);
cudaError_t launch_loop_gate(cudaStream_t st, const LoopState* L, cudaGraphConditionalHandle w);
cudaError_t launch_loop_check(cudaStream_t st, const double* part, long long n, double* r2_out, LoopState* L,
                              LoopState* H, cudaGraphConditionalHandle w, cudaGraphConditionalHandle f, int second);

// A loop runs unless cycle graphs are off, families are being timed (the event nodes of a
// timed cycle cannot stand in a conditional body) or an earlier construction failed.
inline bool loop_usable(const gbmg_ctx* c) { return !c->cyc_off && !c->loop_off && c->prof_mask == 0 && c->loop_dev; }

// Captures what body() queues on `s` as a graph of its own and adds it to `into` as one node,
// after `dep` (nullable).  Not captured straight into a conditional node's body: a launch that
// is refused during the capture invalidates it, the driver then destroys the graph that was
// written to, and destroying its parent crashes the process.  (The child node costs nothing: 20
// kernels per turn of a loop 18.15 us either way.)
template <class Body>
gbmg_status add_captured(cudaStream_t s, cudaGraph_t into, const cudaGraphNode_t* dep, Body body,
                         cudaGraphNode_t* node) {
  cudaGraph_t part = nullptr;
  TRY(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
  const gbmg_status st = body();
  cudaError_t e = cudaStreamEndCapture(s, &part);
  if (st == GBMG_OK && e == cudaSuccess) e = cudaGraphAddChildGraphNode(node, into, dep, dep ? 1 : 0, part);
  if (part) cudaGraphDestroy(part);
  TRYS(st);
  TRY(e);
  return GBMG_OK;
}

// A node of `in` that runs *body while (type) the condition h holds, after `after`.
inline gbmg_status add_conditional(cudaGraph_t in, cudaGraphNode_t after, cudaGraphConditionalHandle h,
                                   cudaGraphConditionalNodeType type, cudaGraph_t* body, cudaGraphNode_t* node) {
  cudaGraphNodeParams p = {};
  p.type = cudaGraphNodeTypeConditional;
  p.conditional.handle = h;
  p.conditional.type = type;
  p.conditional.size = 1;
  TRY(cudaGraphAddNode(node, in, &after, nullptr, 1, &p));
  *body = p.conditional.phGraph_out[0];
  return GBMG_OK;
}

// Builds the loop graph into `exec`: gate, WHILE (cycle 0, check, IF (cycle 1, check)).
// cycle() queues one cycle on c->stream and leaves its `npart` residual partials in
// c->partials; it is called twice, for the two parities in turn.  On any failure the context
// goes back to a graph launch per cycle (loop_off) and nothing is left behind.
template <class Cycle>
void build_loop(gbmg_ctx* c, Cycle cycle, long long npart, cudaGraphExec_t& exec, long long& kernels) {
  cudaStream_t user = c->stream;
  const long long k0 = launch_count();
  cudaGraph_t g = nullptr;
  cudaGraphExec_t x = nullptr;
  long long per_cycle = 0;
  auto attempt = [&]() -> gbmg_status {
    if (!c->cap_stream) TRY(cudaStreamCreateWithFlags(&c->cap_stream, cudaStreamNonBlocking));
    c->stream = c->cap_stream;
    TRY(cudaGraphCreate(&g, 0));
    cudaGraphConditionalHandle w, f;
    TRY(cudaGraphConditionalHandleCreate(&w, g, 0, cudaGraphCondAssignDefault));
    cudaGraphNode_t last, node;
    cudaGraph_t b0, b1;
    TRYS(add_captured(c->stream, g, nullptr, [&]() -> gbmg_status {
      TRY(launch_loop_gate(c->stream, c->loop_dev, w));
      return GBMG_OK;
    }, &last));
    TRYS(add_conditional(g, last, w, cudaGraphCondTypeWhile, &b0, &node));
    TRY(cudaGraphConditionalHandleCreate(&f, b0, 0, cudaGraphCondAssignDefault));
    auto body = [&](int second) -> gbmg_status {
      TRYS(cycle());
      if (second && c->refuse) TRY(cudaStreamSynchronize(c->stream));  // (refused: the stream is captured)
      TRY(launch_loop_check(c->stream, c->partials, npart, c->scal + S_R2, c->loop_dev, c->loop_host_dev, w, f, second));
      return GBMG_OK;
    };
    const long long k1 = launch_count();
    TRYS(add_captured(c->stream, b0, nullptr, [&]() { return body(0); }, &last));
    per_cycle = launch_count() - k1;
    TRYS(add_conditional(b0, last, f, cudaGraphCondTypeIf, &b1, &node));
    TRYS(add_captured(c->stream, b1, nullptr, [&]() { return body(1); }, &last));
    TRY(cudaGraphInstantiate(&x, g, 0));
    return GBMG_OK;
  };
  const bool ok = attempt() == GBMG_OK;
  c->stream = user;
  note_launches(-(launch_count() - k0));
  if (g) cudaGraphDestroy(g);
  if (!ok) {
    (void)cudaGetLastError();
    g_last_error.clear();
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
