// Fused double-float kernel of the finest level: phi' = phi + e in double-float and
// the next defect-correction residual r' = F - m - A phi' (Sec. 3.2) in one pass.
//
// A CTA owns an output tile of TX x TY cells in (x, y) and a chunk of z planes; it
// updates phi on the tile plus a one-cell halo and forms the residual one plane
// behind.  Work unit: the pair of x-neighbouring cells, with the error-free
// double-float sums done by packed FP32x2 instructions lane by lane (bit-identical to
// the scalar double-float kernels).  A thread owns a column of R pairs; shared memory
// holds the updated planes split by x parity and hi/lo part, in a ring of three; the
// z window stays in registers.  One barrier per plane.
#include <cstdio>

#include "dfk.cuh"

namespace gbmg {

namespace {

using namespace dfk;

// ------------------------------------------------------------------ finest level, double-float

// phi' = phi + e (double-float) on the tile plus a one-cell halo, then
// r' = F - m - A phi' on the tile, one plane behind; block partial sums of r'^2,
// of phi' and (pf2 non-null) of (F - m)^2.  e NULL: phi' = phi (first residual of a
// solve); phi_out NULL: phi' is not stored.
// SPLIT: the chains of squares are cut every eight planes (32 squares) and added up with
// compensation.
template <class TL, bool SPLIT>
__global__ void __launch_bounds__(TL::NT, 2)
k_df_update_residual(Dims d, const float2* __restrict__ phi_in, const float* __restrict__ e,
                     const float2* __restrict__ F, const double* __restrict__ m_dev, float2* __restrict__ phi_out,
                     float* __restrict__ r_out, double* __restrict__ pr2, double* __restrict__ psum,
                     double* __restrict__ pf2, int zc) {
  extern __shared__ float smf[];
  __shared__ double shr[32];
  const int x0 = blockIdx.x * TL::TX, y0 = blockIdx.y * TL::TY, z0 = blockIdx.z * zc;
  const int zend = min(z0 + zc, d.nz);
  const float2 m1 = f64_to_df(m_dev[0]);
  const DF2 m{bcast(m1.x), bcast(m1.y)};
  float r2 = 0.f, f2 = 0.f;
  PAcc ps{bcast(0.f), bcast(0.f)};
  DfAcc r2s{0.f, 0.f}, f2s{0.f, 0.f};
  auto flush = [&](float& r, float& f) {
    if (!SPLIT) return;
    r2s.add(r);
    if (pf2) f2s.add(f);
    r = f = 0.f;
  };
  df_segment<TL>(d, phi_in, e, F, m, phi_out, r_out, x0, y0, z0, zend, smf, r2, ps, f2, flush);
  flush(r2, f2);
  DfAcc acc{ps.s.x, ps.c.x};
  acc.add(ps.s.y);
  acc.c += ps.c.y;
  const double b2 = SPLIT ? block_sum_pair(r2s, shr) : block_sum_f(r2, shr);
  const double bs = block_sum_acc(acc, shr);
  const double bf = !pf2 ? 0.0 : (SPLIT ? block_sum_pair(f2s, shr) : block_sum_f(f2, shr));
  if (threadIdx.x == 0) {
    const int bid = block_linear_id();
    pr2[bid] = b2;
    psum[bid] = bs;
    if (pf2) pf2[bid] = bf;
  }
}

using DFT = DTile<64, 16, 2, 320>;


}  // namespace

// ---- double-float update

// z chunk of the double-float update.  Large meshes: at least four waves of two CTAs per
// SM, so that enough loads are in flight.  Meshes that have no four waves of 16-plane
// chunks: the chunk with the shortest critical path, whole waves of 304 CTAs times the
// chunk and its two extra planes (16-plane chunks left most SMs idle there: 64^3 20.2 -> 6.6
// us, 160 x 128 x 224 42 -> 36 us, 256^3 108 -> 104 us).
long long df_tiles(Dims d) {
  return (long long)((d.nx + DFT::TX - 1) / DFT::TX) * ((d.ny + DFT::TY - 1) / DFT::TY);
}
bool df_four_waves(Dims d) { return df_tiles(d) * ((d.nz + 15) / 16) >= 4 * 2 * 152; }
int df_zchunk(Dims d) {
  const long long tiles = df_tiles(d);
  if (df_four_waves(d)) {
    int zc = d.nz;
    while (tiles * ((d.nz + zc - 1) / zc) < 4 * 2 * 152) zc = (zc + 1) / 2;
    return zc;
  }
  int best = d.nz;
  long long best_cost = -1;
  for (int zc = 2; zc <= d.nz; ++zc) {
    const long long waves = (tiles * ((d.nz + zc - 1) / zc) + 2 * 152 - 1) / (2 * 152);
    if (best_cost < 0 || waves * (zc + 2) < best_cost) best_cost = waves * (zc + 2), best = zc;
  }
  return best;
}

long long df_update_residual_partials(Dims d) {
  const int zc = df_zchunk(d);
  return (long long)((d.nx + DFT::TX - 1) / DFT::TX) * ((d.ny + DFT::TY - 1) / DFT::TY) * ((d.nz + zc - 1) / zc);
}

cudaError_t launch_df_update_residual(cudaStream_t st, Dims d, const float2* phi_in, const float* e, const float2* F,
                                      const double* m_dev, float2* phi_out, float* r_out, double* pr2, double* psum,
                                      double* pf2) {
  if (d.nx % 2) return cudaErrorInvalidValue;  // x-pairs
  const size_t sm = 3 * (size_t)DFT::PLANE * sizeof(float);
  const int zc = df_zchunk(d);
  const dim3 grid((d.nx + DFT::TX - 1) / DFT::TX, (d.ny + DFT::TY - 1) / DFT::TY, (d.nz + zc - 1) / zc);
  // chunks that the rule for small meshes makes longer than 16 planes (up to 64) would sum up to
  // 256 squares in one FP32 chain, where 16 planes sum 64
  const bool split = zc > 16 && !df_four_waves(d);
  static DeviceSet done[2] = {{0}, {0}};
  const auto kernel = split ? k_df_update_residual<DFT, true> : k_df_update_residual<DFT, false>;
  const cudaError_t err = allow_smem(done[split], kernel, sm);
  if (err != cudaSuccess) return err;
  kernel<<<grid, DFT::NT, sm, st>>>(d, phi_in, e, F, m_dev, phi_out, r_out, pr2, psum, pf2, zc);
  note_launch();
  return cudaGetLastError();
}

}  // namespace gbmg
