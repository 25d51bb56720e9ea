// What the persistent kernel of the batched solves (batch.cu) and the kernels of their phase
// graph (batch_graph.cu) share: descriptors and a few device helpers.
#pragma once
#include <cuda_runtime.h>

#include <functional>
#include <vector>

#include "dfk.cuh"
#include "kernels.h"
#include "legs.cuh"
#include "solver.h"
#include "stencil.cuh"

namespace gbmg {
namespace batchk {

constexpr int BMAXL = 16;
constexpr int CHUNK = 4096;      // default tile (chunk) size in cells
constexpr int MINCHUNK = 1024;   // smallest tile the tables are sized for
constexpr int MAXCHUNK = 65536;

// per-problem scalars
enum { P_MEAN = 0, P_F2 = 1, P_R2 = 2, P_REL = 3, P_PREV1 = 4, P_PREV2 = 5, P_MPHI = 6, P_N = 8 };
// status codes inside the kernel: 0 = still iterating, -1 = converged, else a gbmg_status
enum { ST_ACTIVE = 0, ST_CONVERGED = -1 };

struct BProb {
  int L, nc;
  Dims d[BMAXL];
  float* r[BMAXL];
  float* ea[BMAXL];
  float* eb[BMAXL];
  float* dv[BMAXL];
  float* t[BMAXL];
  const float* G;
  float2* F;
  float2* phi;   // double-float phi, and the second buffer of the fused update (phi2)
  float2* phi2;
  const double* src;
  double* out;
  int c0, nch;      // first level-0 chunk and count
  unsigned fmask;   // bit l: level l runs the fused legs
  int dffused;      // the finest level runs the fused double-float update (even nx)
  int ls;           // first level of the single-CTA bottom cycle (levels ls .. L-1), 0: none
};

struct BDesc {
  int count, maxL, degree, maxv;
  int chunk[BMAXL];  // tile (chunk) size in cells per level
  double tol;
  float c1[16];
  float ca[BMAXL][8];  // folded Chebyshev constants a = c2 D^-1 and b = a / h^2 per level and step
  float cb[BMAXL][8];
  float ih2[BMAXL];    // 1 / h_l^2
  const legs::Coef* coef;       // folded Chebyshev constants per level (device)
  const long long* doff[BMAXL];  // per level: prefix over problems of fused down-leg planes
  const long long* uoff[BMAXL];  // per level: the same for the up leg
  long long dtot[BMAXL], utot[BMAXL];
  const int* dfoff;              // prefix over problems of fused double-float items
  int dftot;
  double* dfpart;                // per double-float item: partial sum of r^2
  double* dfpart2;               // per double-float item: partial sum of (F - m)^2 (first residual)
  unsigned perop;                // bit l: some problem runs level l per operation (not the coarsest)
  unsigned coarse;               // bit l: some problem's coarsest level is l (outside a bottom cycle)
  const SmallCycle* small;       // per problem: parameters of its bottom cycle (ls > 0)
  int anysmall;                  // some problem runs a bottom cycle
  int* phicur;                   // per problem: 0 = phi, 1 = phi2 holds the current iterate
  BProb* p;
  // chunk tables per level: problem index and first cell
  int* cprob[BMAXL];
  long long* cstart[BMAXL];
  int nchunk[BMAXL];
  double* part0;  // per level-0 chunk partials
  double* part1;
  double* sc;     // count * P_N scalars
  int* status;    // count: ST_ACTIVE, then a gbmg_status
  int* cycles;    // count
  double* hist;   // count * 64
  double* rel0;   // count
  unsigned long long* tdone;  // count, %globaltimer at completion
  unsigned long long* tstart;
  int* any_active;
};

__device__ __forceinline__ unsigned long long globaltimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// level l of problem P runs the fused legs
__device__ __forceinline__ bool lv_fused(const BProb& P, int l) { return (P.fmask >> l) & 1u; }
// buffer holding the final correction of level l after its up leg
__device__ __forceinline__ float* final_e(const BProb& P, int l) {
  return (l < P.L - 1 && lv_fused(P, l)) ? P.eb[l] : P.ea[l];
}

// ---- the phase graph (batch_graph.cu)

// Work lists of its kernels (prefixes over the problems): planes of the legs per level, items
// of fz planes of the double-float step, with their partial sums.
struct Phases {
  const long long* doff[BMAXL];
  const long long* uoff[BMAXL];
  long long dtot[BMAXL], utot[BMAXL];
  const int* foff;
  int ftot, fz;
  double* fpart;   // r^2
  double* fpart2;  // (F - m)^2, first residual
};

struct PhaseGraph {
  bool usable = false;
  Phases t{};
  legs::Coef coef[BMAXL];
  size_t bottom_sm = 0;
  char* mem = nullptr;
  // bottom: shared memory of the largest bottom cycle
  gbmg_status init(const std::vector<gbmg_ctx*>& ctx, const BProb* prob, const BDesc& D, size_t bottom);
  // *graph: one solve, captured on gs, with head() before it and tail() after it (also set on
  // an error, for the caller to destroy); refuse (testing): fails in the loop's capture
  gbmg_status build(cudaStream_t gs, const BDesc& D, cudaGraph_t* graph, const std::function<gbmg_status()>& head,
                    const std::function<gbmg_status()>& tail, bool refuse) const;
  ~PhaseGraph();
};

}  // namespace batchk
}  // namespace gbmg
