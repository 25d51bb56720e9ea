// Batched solves as a graph of phase kernels: what the persistent kernel of batch.cu does
// between two grid barriers is a kernel here, and its cycle loop a conditional WHILE node.
//
// The persistent kernel holds every phase under one register limit at 12 warps per SM, so
// its phases ran 1.5 to 2 times as long as the kernels of single solves: 14.3 ms for 48
// problems of 64^3, 96^3 and 128^3, seven cycles (finest level per cycle: down 372, up 532,
// update 595 us; here 7.9 ms, the update 324 us, all down legs together 269 and all up legs 340).
// As kernels of their own the legs have the single solves' tiles and register limits (beside the
// batch's descriptors the down legs spill 16 bytes at degree 3 and 12 at degree 4, the up leg 4 at
// degree 4; those of single solves none), the double-float step has two CTAs per SM, and the bottom
// cycle 1024 threads; a launch boundary costs about what the grid barrier did.  Each value
// sees the same operations as in the persistent kernel (the chunks of the means and their
// summation order too), so both give the same iterates bit for bit; the residual norms are
// summed over other tiles.
//
// For batches whose every level runs the fused legs or a bottom cycle (degrees 1 to 4, even
// nx, levels of at least 16^3 above the bottom); others keep the persistent kernel.
#include <algorithm>

#include "batch.cuh"
#include "loop.h"
#include "small_cta.cuh"

namespace gbmg {
namespace batchk {

namespace {

constexpr int SMS = 152;
constexpr int ET = 384;  // threads of the chunk kernels: the persistent kernel's, for the same partial sums
using GDf = dfk::DTile<32, 32, 2, 320>;

// the problem p with off[p] <= v < off[p + 1]
template <typename I>
__device__ __forceinline__ int problem_of(const I* __restrict__ off, int count, I v) {
  int lo = 0, hi = count;
  while (hi - lo > 1) {
    const int mid = (lo + hi) / 2;
    (off[mid] <= v ? lo : hi) = mid;
  }
  return lo;
}

template <int V>
__global__ void __maxnreg__(legs::max_regs<typename legs::DownTile<V>::T>())
k_batch_down(BDesc B, Phases T, int l, legs::Coef cf) {
  using TL = typename legs::DownTile<V>::T;
  extern __shared__ __align__(16) float smf[];
  long long a = (long long)blockIdx.x * T.dtot[l] / gridDim.x;
  const long long b = (long long)(blockIdx.x + 1) * T.dtot[l] / gridDim.x;
  int p = problem_of(T.doff[l], B.count, a);
  while (a < b) {
    while (T.doff[l][p + 1] <= a) ++p;
    const BProb& P = B.p[p];
    const Dims d = P.d[l];
    const long long loc = a - T.doff[l][p];
    const int tile = (int)(loc / d.nz), z0 = (int)(loc - (long long)tile * d.nz);
    const int zend = (int)(z0 + (b - a) < d.nz ? z0 + (b - a) : d.nz);
    const int tiles_x = (d.nx + TL::TX - 1) / TL::TX;
    if (B.status[p] == ST_ACTIVE)
      legs::down_segment<V, TL>(d, P.r[l], P.ea[l], P.r[l + 1], tile % tiles_x * TL::TX, tile / tiles_x * TL::TY, z0,
                                zend, B.ih2[l], cf, smf);
    a += zend - z0;
    __syncthreads();
  }
}

template <int V>
__global__ void __maxnreg__(legs::max_regs<typename legs::UpTile<V>::T>())
k_batch_up(BDesc B, Phases T, int l, legs::Coef cf) {
  using TL = typename legs::UpTile<V>::T;
  extern __shared__ __align__(16) float smf[];
  long long a = (long long)blockIdx.x * T.utot[l] / gridDim.x;
  const long long b = (long long)(blockIdx.x + 1) * T.utot[l] / gridDim.x;
  int p = problem_of(T.uoff[l], B.count, a);
  while (a < b) {
    while (T.uoff[l][p + 1] <= a) ++p;
    const BProb& P = B.p[p];
    const Dims d = P.d[l];
    const long long loc = a - T.uoff[l][p];
    const int tile = (int)(loc / d.nz), z0 = (int)(loc - (long long)tile * d.nz);
    const int zend = (int)(z0 + (b - a) < d.nz ? z0 + (b - a) : d.nz);
    const int tiles_x = (d.nx + TL::TX - 1) / TL::TX;
    if (B.status[p] == ST_ACTIVE)
      legs::up_segment<V, TL>(d, P.ea[l], final_e(P, l + 1), P.r[l], P.eb[l], tile % tiles_x * TL::TX,
                              tile / tiles_x * TL::TY, z0, zend, B.ih2[l], cf, smf);
    a += zend - z0;
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kSmallThreads, 1) k_batch_bottom(BDesc B) {
  extern __shared__ __align__(16) float smf[];
  __shared__ SmallCycle sc;  // its parameters are read in every phase
  static_assert(sizeof(SmallCycle) % 4 == 0 && sizeof(SmallCycle) / 4 <= kSmallThreads, "");
  const BProb& P = B.p[blockIdx.x];
  if (B.status[blockIdx.x] != ST_ACTIVE) return;
  if (threadIdx.x < sizeof(SmallCycle) / 4) ((int*)&sc)[threadIdx.x] = ((const int*)&B.small[blockIdx.x])[threadIdx.x];
  __syncthreads();
  smallcta::vcycle(sc, P.r[P.ls], P.ea[P.ls], smf);
}

// One item (tile, z chunk) of the update and residual, with its own partial sums; FIRST: the
// residual of the guess.
template <bool FIRST>
__global__ void __launch_bounds__(GDf::NT, 2) k_batch_df(BDesc B, Phases T) {
  extern __shared__ __align__(16) float smf[];
  __shared__ double sh[32];
  const int it = blockIdx.x;
  const int p = problem_of(T.foff, B.count, it);
  if (B.status[p] != ST_ACTIVE) return;
  const BProb& P = B.p[p];
  const Dims d = P.d[0];
  const int loc = it - T.foff[p];
  const int tiles_x = (d.nx + GDf::TX - 1) / GDf::TX, nzc = (d.nz + T.fz - 1) / T.fz;
  const int tile = loc / nzc, z0 = (loc - tile * nzc) * T.fz;
  const int cur = B.phicur[p];
  const float2 m1 = f64_to_df(B.sc[p * P_N + P_MEAN]);
  float r2 = 0.f, f2 = 0.f;
  PAcc ps{bcast(0.f), bcast(0.f)};
  dfk::df_segment<GDf>(d, cur ? P.phi2 : P.phi, FIRST ? nullptr : final_e(P, 0), P.F,
                       DF2{bcast(m1.x), bcast(m1.y)}, FIRST ? nullptr : (cur ? P.phi : P.phi2), P.r[0],
                       tile % tiles_x * GDf::TX, tile / tiles_x * GDf::TY, z0, min(z0 + T.fz, d.nz), smf, r2, ps, f2);
  const double s = block_sum_f(r2, sh);
  if (threadIdx.x == 0) T.fpart[it] = s;
  if (FIRST) {
    const double sf = block_sum_f(f2, sh);
    if (threadIdx.x == 0) T.fpart2[it] = sf;
  }
}

// Relative residuals, histories and statuses, a warp per problem; the loop goes on while a
// problem is active.
template <bool FIRST>
__global__ void __launch_bounds__(1024) k_batch_books(BDesc B, Phases T, cudaGraphConditionalHandle w) {
  const int lane = threadIdx.x & 31;
  int active = 0;
  for (int pi = threadIdx.x >> 5; pi < B.count; pi += 32) {
    if (!FIRST && B.status[pi] != ST_ACTIVE) continue;
    double* const s = B.sc + pi * P_N;
    double r2 = 0.0, f2 = 0.0;
    for (int k = T.foff[pi] + lane; k < T.foff[pi + 1]; k += 32) {
      r2 += T.fpart[k];
      if (FIRST) f2 += T.fpart2[k];
    }
    r2 = warp_sum(r2);
    f2 = FIRST ? warp_sum(f2) : s[P_F2];
    if (lane) continue;
    const double rel = f2 > 0.0 ? sqrt(r2 / f2) : sqrt(r2);
    int cyc = FIRST ? 0 : B.cycles[pi];
    const double prev1 = FIRST ? -1.0 : s[P_PREV1], prev2 = FIRST ? -1.0 : s[P_PREV2];
    if (FIRST) {
      s[P_F2] = f2;
      B.rel0[pi] = rel;
    } else {
      if (cyc < 64) B.hist[pi * 64 + cyc] = rel;
      B.cycles[pi] = ++cyc;
      B.phicur[pi] ^= 1;  // the update wrote the other buffer
    }
    s[P_REL] = rel;
    int st = ST_ACTIVE;
    if (!isfinite(rel)) st = GBMG_ERR_NONFINITE;
    else if (rel <= B.tol) st = ST_CONVERGED;
    else if (!FIRST && prev2 > 0.0 && rel > 10.0 * prev2) st = GBMG_ERR_DIVERGED;
    else if (cyc >= B.maxv) st = GBMG_ERR_NOT_CONVERGED;
    s[P_PREV2] = prev1;
    s[P_PREV1] = rel;
    if (st != ST_ACTIVE) {
      B.status[pi] = st;
      B.tdone[pi] = globaltimer();
    } else {
      active = 1;
    }
  }
  active = __syncthreads_or(active);
  if (threadIdx.x == 0) cudaGraphSetConditional(w, active ? 1u : 0u);
}

// Level-0 chunks with the persistent kernel's partial sums: load(P, i, k) of four cells, then
// use(P, i, k, acc) in order (loads one at a time: 392 + 168 us instead of 249 + 120 for
// 51.9 M cells).
template <typename Load, typename Use>
__device__ __forceinline__ void chunks(const BDesc& B, double* part, double* sh, Load load, Use use) {
  for (int c = blockIdx.x; c < B.nchunk[0]; c += gridDim.x) {
    const int pi = B.cprob[0][c];
    const BProb& P = B.p[pi];
    const long long s0 = B.cstart[0][c];
    const long long n = ncell(P.d[0]);
    const long long s1 = s0 + B.chunk[0] < n ? s0 + B.chunk[0] : n;
    DfAcc acc{0.f, 0.f};
    for (long long i = s0 + threadIdx.x; i < s1; i += 4 * ET) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (i + k * ET < s1) load(pi, P, i + k * ET, k);
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (i + k * ET < s1) use(pi, P, i + k * ET, k, acc);
    }
    const double b = block_sum_acc(acc, sh);
    if (threadIdx.x == 0) part[c] = b;
  }
}

// Double-float copies of sources and guesses, and the chunk sums of the sources.
__global__ void __launch_bounds__(ET) k_batch_prologue(BDesc B) {
  __shared__ double sh[32];
  if (blockIdx.x == 0 && threadIdx.x == 0) *B.tstart = globaltimer();
  double f[4], g[4];
  chunks(B, B.part0, sh,
         [&](int, const BProb& P, long long i, int k) {
           f[k] = P.src[i];
           g[k] = P.out[i];
         },
         [&](int, const BProb& P, long long i, int k, DfAcc& acc) {
           const float2 v = f64_to_df(f[k]);
           P.F[i] = v;
           P.phi[i] = f64_to_df(g[k]);
           acc.add(v.x);
           acc.c += v.y;
         });
}

__global__ void __launch_bounds__(ET) k_batch_phi_sum(BDesc B) {
  __shared__ double sh[32];
  float2 v[4];
  chunks(B, B.part0, sh,
         [&](int pi, const BProb& P, long long i, int k) { v[k] = (B.phicur[pi] ? P.phi2 : P.phi)[i]; },
         [&](int, const BProb&, long long, int k, DfAcc& acc) {
           acc.add(v[k].x);
           acc.c += v[k].y;
         });
}

// The mean of a field from its chunk sums, added in order by one thread.
__global__ void __launch_bounds__(256) k_batch_mean(BDesc B, int slot) {
  __shared__ double sh[256];
  const int pi = blockIdx.x;
  const BProb& P = B.p[pi];
  double s = 0.0;
  for (int k0 = 0; k0 < P.nch; k0 += 256) {
    const int m = min(256, P.nch - k0);
    if (threadIdx.x < m) sh[threadIdx.x] = B.part0[P.c0 + k0 + threadIdx.x];
    __syncthreads();
    if (threadIdx.x == 0)
      for (int k = 0; k < m; ++k) s += sh[k];
    __syncthreads();
  }
  if (threadIdx.x) return;
  if (slot == P_MEAN) B.phicur[pi] = 0;
  B.sc[pi * P_N + slot] = s / (double)ncell(P.d[0]);
}

__global__ void __launch_bounds__(ET) k_batch_output(BDesc B) {
  for (int c = blockIdx.x; c < B.nchunk[0]; c += gridDim.x) {
    const int pi = B.cprob[0][c];
    const BProb& P = B.p[pi];
    const float2* ph = B.phicur[pi] ? P.phi2 : P.phi;
    float2 ms = f64_to_df(B.sc[pi * P_N + P_MPHI]);
    ms.x = -ms.x;
    ms.y = -ms.y;
    const long long s0 = B.cstart[0][c];
    const long long n = ncell(P.d[0]);
    const long long s1 = s0 + B.chunk[0] < n ? s0 + B.chunk[0] : n;
    for (long long i = s0 + threadIdx.x; i < s1; i += blockDim.x) P.out[i] = df_to_f64(df_add(ph[i], ms));
  }
}

struct Kernels {
  void (*down)(BDesc, Phases, int, legs::Coef);
  void (*up)(BDesc, Phases, int, legs::Coef);
  int down_t, up_t, down_ty, up_ty;
  size_t down_sm, up_sm;
};
template <int V>
Kernels kernels() {
  return Kernels{k_batch_down<V>, k_batch_up<V>, legs::DownTile<V>::T::NT, legs::UpTile<V>::T::NT,
                 legs::DownTile<V>::T::TY, legs::UpTile<V>::T::TY, legs::down_smem<V>(), legs::up_smem<V>()};
}
Kernels kernels_of(int degree) {
  switch (degree) {
    case 1: return kernels<1>();
    case 2: return kernels<2>();
    case 3: return kernels<3>();
    default: return kernels<4>();
  }
}

constexpr size_t kDfSmem = 3 * (size_t)GDf::PLANE * sizeof(float);

}  // namespace

PhaseGraph::~PhaseGraph() {
  if (mem) cudaFree(mem);
}

gbmg_status PhaseGraph::init(const std::vector<gbmg_ctx*>& ctx, const BProb* prob, const BDesc& D, size_t bottom) {
  usable = D.degree >= 1 && D.degree <= 4 && D.perop == 0 && D.coarse == 0;
  for (int i = 0; i < D.count; ++i) usable = usable && prob[i].dffused && prob[i].ls > 0;
  if (!usable) return GBMG_OK;
  const Kernels K = kernels_of(D.degree);
  const int count = D.count;
  auto cdiv = [](long long a, long long b) { return (a + b - 1) / b; };
  // prefixes over the problems: down planes per level, up planes per level; update items
  std::vector<long long> off((size_t)2 * D.maxL * (count + 1), 0);
  std::vector<int> fo(count + 1, 0);
  for (int l = 0; l < D.maxL; ++l)
    for (int i = 0; i < count; ++i) {
      long long nd = 0, nu = 0;
      if (prob[i].fmask >> l & 1u) {
        const Dims d = ctx[i]->lv[l].d;
        nd = cdiv(d.nx, 64) * cdiv(d.ny, K.down_ty) * d.nz;
        nu = cdiv(d.nx, 64) * cdiv(d.ny, K.up_ty) * d.nz;
      }
      long long* const o = off.data() + (size_t)l * (count + 1);
      o[i + 1] = o[i] + nd;
      long long* const u = o + (size_t)D.maxL * (count + 1);
      u[i + 1] = u[i] + nu;
    }
  // planes of an update item: 32 (for 48 problems 324 us per cycle; 16 and 48 329, 8 and 128
  // 363), fewer where that leaves less than two items for a CTA's place (two on an SM)
  for (t.fz = 32;; t.fz /= 2) {
    for (int i = 0; i < count; ++i) {
      const Dims d = ctx[i]->lv[0].d;
      fo[i + 1] = fo[i] + (int)(cdiv(d.nx, GDf::TX) * cdiv(d.ny, GDf::TY) * cdiv(d.nz, t.fz));
    }
    t.ftot = fo[count];
    if (t.ftot >= 4 * SMS || t.fz == 8) break;
  }
  const size_t b0 = (off.size() * sizeof(long long) + 255) / 256 * 256;
  const size_t b1 = (fo.size() * sizeof(int) + 255) / 256 * 256;
  TRY(cudaMalloc((void**)&mem, b0 + b1 + 2 * (size_t)t.ftot * sizeof(double)));
  TRY(cudaMemcpy(mem, off.data(), off.size() * sizeof(long long), cudaMemcpyHostToDevice));
  TRY(cudaMemcpy(mem + b0, fo.data(), fo.size() * sizeof(int), cudaMemcpyHostToDevice));
  for (int l = 0; l < D.maxL; ++l) {
    t.doff[l] = (const long long*)mem + (size_t)l * (count + 1);
    t.uoff[l] = t.doff[l] + (size_t)D.maxL * (count + 1);
    t.dtot[l] = off[(size_t)l * (count + 1) + count];
    t.utot[l] = off[(size_t)(D.maxL + l) * (count + 1) + count];
    coef[l] = legs::make_coef(ctx[0]->cc1.data(), ctx[0]->cc2.data(), D.degree, (double)(1 << l));
  }
  t.foff = (const int*)(mem + b0);
  t.fpart = (double*)(mem + b0 + b1);
  t.fpart2 = t.fpart + t.ftot;
  bottom_sm = bottom;
  auto smem = [](const void* k, size_t s) {
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)s);
  };
  TRY(smem((const void*)K.down, K.down_sm));
  TRY(smem((const void*)K.up, K.up_sm));
  // (the limit belongs to the kernel, not to this batch: a smaller bottom cycle's size would
  // refuse the launches of a batch made before)
  TRY(smem((const void*)k_batch_bottom, kSmallSmem));
  TRY(smem((const void*)k_batch_df<true>, kDfSmem));
  TRY(smem((const void*)k_batch_df<false>, kDfSmem));
  return GBMG_OK;
}

gbmg_status PhaseGraph::build(cudaStream_t gs, const BDesc& D, cudaGraph_t* graph,
                              const std::function<gbmg_status()>& head, const std::function<gbmg_status()>& tail,
                              bool refuse) const {
  const Kernels K = kernels_of(D.degree);
  const int chunks = std::min(D.nchunk[0], 8 * SMS);
  cudaGraph_t g = nullptr, turn = nullptr;
  TRY(cudaGraphCreate(&g, 0));
  *graph = g;
  cudaGraphConditionalHandle w;
  TRY(cudaGraphConditionalHandleCreate(&w, g, 0, cudaGraphCondAssignDefault));
  cudaGraphNode_t last, loop;
  TRYS(add_captured(gs, g, nullptr, [&]() -> gbmg_status {
    TRYS(head());
    k_batch_prologue<<<chunks, ET, 0, gs>>>(D);
    k_batch_mean<<<D.count, 256, 0, gs>>>(D, P_MEAN);
    k_batch_df<true><<<t.ftot, GDf::NT, kDfSmem, gs>>>(D, t);
    k_batch_books<true><<<1, 1024, 0, gs>>>(D, t, w);
    TRY(cudaGetLastError());
    return GBMG_OK;
  }, &last));
  TRYS(add_conditional(g, last, w, cudaGraphCondTypeWhile, &turn, &loop));
  TRYS(add_captured(gs, turn, nullptr, [&]() -> gbmg_status {
    for (int l = 0; l + 1 < D.maxL; ++l)
      if (t.dtot[l])
        K.down<<<(int)std::min<long long>(t.dtot[l], SMS), K.down_t, K.down_sm, gs>>>(D, t, l, coef[l]);
    k_batch_bottom<<<D.count, kSmallThreads, bottom_sm, gs>>>(D);
    for (int l = D.maxL - 2; l >= 0; --l)
      if (t.utot[l]) K.up<<<(int)std::min<long long>(t.utot[l], SMS), K.up_t, K.up_sm, gs>>>(D, t, l, coef[l]);
    k_batch_df<false><<<t.ftot, GDf::NT, kDfSmem, gs>>>(D, t);
    k_batch_books<false><<<1, 1024, 0, gs>>>(D, t, w);
    TRY(cudaGetLastError());
    if (refuse) TRY(cudaStreamSynchronize(gs));  // (refused: the stream is captured)
    return GBMG_OK;
  }, &last));
  TRYS(add_captured(gs, g, &loop, [&]() -> gbmg_status {
    k_batch_phi_sum<<<chunks, ET, 0, gs>>>(D);
    k_batch_mean<<<D.count, 256, 0, gs>>>(D, P_MPHI);
    k_batch_output<<<chunks, ET, 0, gs>>>(D);
    TRY(cudaGetLastError());
    return tail();
  }, &last));
  return GBMG_OK;
}

}  // namespace batchk
}  // namespace gbmg
