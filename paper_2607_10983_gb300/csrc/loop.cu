// The defect-correction loop on the device (Sec. 3.2): a solve's cycles as one CUDA graph
// with a conditional WHILE node, so that the host launches one graph and waits once per
// solve.  What it replaces, a graph launch and a stream synchronisation per cycle, left the
// GPU idle for about 16 us per cycle: 130 of the 604 us of a cold 64^3 solve.
//
// The loop's body is two cycles, one per parity of the ping-pong buffers, the second inside
// an IF node; after each a check kernel sums the residual's partials, keeps the books of
// Monitor (host_math.h) and sets the conditions.
#include "loop.h"

namespace gbmg {

namespace {

// FP64 runs at under 2 operations per clock on an SM, so the sums take four warps and a
// tree of theirs, not a block of 1024 threads of which most add zeros (5.9 -> 3.1 us for the
// 128 partials of 64^3 alone, with the host copy left to the last check; 4.2 in that solve, up to
// 6.4 with the thousands of larger meshes).
constexpr int LT = 128;

// valid in every thread
__device__ double sum_partials(const double* __restrict__ p, long long n, double* sh) {
  double s = 0.0;
  for (long long i = threadIdx.x; i < n; i += LT) s += p[i];
  s = warp_sum(s);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  return (sh[0] + sh[1]) + (sh[2] + sh[3]);
}

// Monitor::done
__device__ void loop_done(LoopState& L) {
  L.go = 0;
  if (!isfinite(L.rel)) L.status = GBMG_ERR_NONFINITE;
  else if (L.rel <= L.tol) return;
  else if (L.cycles >= L.maxv) L.status = GBMG_ERR_NOT_CONVERGED;
  else L.go = 1;
}

// The books to the host's copy, by the whole block after thread 0 has closed them.
__device__ void report(const LoopState* L, LoopState* H) {
  __syncthreads();
  if (L->go) return;
  const int n = L->cycles < 64 ? L->cycles : 64;
  for (int i = threadIdx.x; i < n; i += LT) H->hist[i] = L->hist[i];
  if (threadIdx.x == 0) {
    H->cycles = L->cycles;
    H->status = L->status;
    H->rel0 = L->rel0;
    H->rel = L->rel;
  }
  __threadfence_system();
}

__global__ void __launch_bounds__(LT) k_loop_begin(const double* __restrict__ pr2, const double* __restrict__ pf2,
                                                   long long n, double tol, int maxv, double* __restrict__ r2_out,
                                                   double* __restrict__ f2_out, LoopState* L, LoopState* H) {
  __shared__ double sh[4];
  const double r2 = sum_partials(pr2, n, sh);
  const double f2 = sum_partials(pf2, n, sh);
  if (threadIdx.x == 0) {
    *r2_out = r2;
    *f2_out = f2;
    L->tol = tol;
    L->maxv = maxv;
    L->cycles = 0;
    L->status = GBMG_OK;
    L->f2 = f2;
    L->rel0 = L->rel = L->prev1 = f2 > 0.0 ? sqrt(r2 / f2) : sqrt(r2);
    L->prev2 = -1.0;
    loop_done(*L);
  }
  report(L, H);
}

__global__ void k_loop_gate(const LoopState* L, cudaGraphConditionalHandle w) {
  if (threadIdx.x == 0) cudaGraphSetConditional(w, (unsigned)L->go);
}

__global__ void __launch_bounds__(LT) k_loop_check(const double* __restrict__ part, long long n,
                                                   double* __restrict__ r2_out, LoopState* L, LoopState* H,
                                                   cudaGraphConditionalHandle w, cudaGraphConditionalHandle f,
                                                   int second) {
  __shared__ double sh[4];
  LoopState S;  // read while the partials are on their way
  S.cycles = L->cycles;
  S.maxv = L->maxv;
  S.status = L->status;
  S.tol = L->tol;
  S.f2 = L->f2;
  S.prev1 = L->prev1;
  S.prev2 = L->prev2;
  const double r2 = sum_partials(part, n, sh);
  if (threadIdx.x == 0) {
    *r2_out = r2;
    // Monitor::record: prev1, prev2 are the residuals one and two cycles back
    const double rel = S.f2 > 0.0 ? sqrt(r2 / S.f2) : sqrt(r2);
    const bool diverged = S.cycles >= 1 && isfinite(rel) && rel > 10.0 * S.prev2;
    S.rel = rel;
    if (S.cycles < 64) L->hist[S.cycles] = rel;
    S.cycles += 1;
    S.go = 0;
    if (diverged) S.status = GBMG_ERR_DIVERGED;
    else loop_done(S);
    cudaGraphSetConditional(w, (unsigned)S.go);
    if (!second) cudaGraphSetConditional(f, (unsigned)S.go);
    L->cycles = S.cycles;
    L->status = S.status;
    L->go = S.go;
    L->rel = rel;
    L->prev2 = S.prev1;
    L->prev1 = rel;
  }
  report(L, H);
}

__global__ void __launch_bounds__(LT) k_norm_sum(const double* __restrict__ p, long long n, double* __restrict__ out) {
  __shared__ double sh[4];
  const double s = sum_partials(p, n, sh);
  if (threadIdx.x == 0) *out = s;
}

}  // namespace

cudaError_t launch_norm_sum(cudaStream_t st, const double* part, long long n, double* out) {
  k_norm_sum<<<1, LT, 0, st>>>(part, n, out);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_loop_begin(cudaStream_t st, const double* pr2, const double* pf2, long long n, double tol, int maxv,
                              double* r2_out, double* f2_out, LoopState* L, LoopState* H) {
  k_loop_begin<<<1, LT, 0, st>>>(pr2, pf2, n, tol, maxv, r2_out, f2_out, L, H);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_loop_gate(cudaStream_t st, const LoopState* L, cudaGraphConditionalHandle w) {
  k_loop_gate<<<1, 32, 0, st>>>(L, w);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_loop_check(cudaStream_t st, const double* part, long long n, double* r2_out, LoopState* L,
                              LoopState* H, cudaGraphConditionalHandle w, cudaGraphConditionalHandle f, int second) {
  k_loop_check<<<1, LT, 0, st>>>(part, n, r2_out, L, H, w, f, second);
  note_launch();
  return cudaGetLastError();
}

}  // namespace gbmg
