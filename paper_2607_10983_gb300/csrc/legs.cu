// Temporally blocked FP32 level kernels (the single-GPU form of the paper's
// communication-avoiding whole-level fusion, Sec. 3.4 implementation list): one
// HBM pass per level visit and leg instead of one per operation.
//
//   k_down_fused : Chebyshev pre-smoothing from e = 0 (degree V), residual and
//                  full-weighting restriction.  Reads r, writes e and R(r - A e).
//   k_up_fused   : trilinear prolongation + correction and Chebyshev
//                  post-smoothing.  Reads e, e_c, r; writes the new e.
//
// Blocking scheme.  A CTA owns an output tile of TX x TY cells in (x, y) and a range
// of z planes; it computes on the tile plus a halo (H cells in y, H rounded up to
// whole pairs in x), so that every stage, which needs its input on one more ring of
// cells, still produces valid values on the tile.  The CTA streams through z: each
// iteration loads one input plane and every stage advances one plane, stage s one
// plane behind stage s-1.  One barrier per iteration.
//
// Work unit: the pair of x-neighbouring cells (even x, odd x), computed with packed
// FP32x2 instructions; a thread owns a column of R pairs stacked in y.  Shared
// memory holds each stage's current plane split by x parity (even cells, odd cells),
// so the x neighbours of a pair are two conflict-free scalar loads; y neighbours
// inside the column and the two older z planes stay in registers.  Every lane of a
// packed instruction rounds like the scalar intrinsic of the one-kernel-per-operation
// path, in the same order, so the results are bit-identical to it.
//
// Schedule: persistent grid of one CTA per SM; the (tile, plane) pairs form one
// tile-major list and CTA b runs the contiguous range [b T / G, (b+1) T / G), as one
// z segment per tile it touches (each segment with its own warm-up planes).  Each
// tile's z stream starts at its own phase (tile_phase), so that neighbouring tiles
// stream the same planes at about the same time and their shared halo rows are read
// from DRAM about once.
#include "legs.cuh"

namespace gbmg {

namespace {

using namespace legs;

template <int V, class TL>
__global__ void __maxnreg__(max_regs<TL>())
k_down_fused(Dims d, const float* __restrict__ r, float* __restrict__ e_out, float* __restrict__ rc, Sched sc,
             float inv_h2, Coef cf) {
  extern __shared__ float sm[];
  long long a = (long long)blockIdx.x * sc.total / gridDim.x;
  const long long b = (long long)(blockIdx.x + 1) * sc.total / gridDim.x;
  while (a < b) {
    const long long tile = a / d.nz;
    const int p0 = (int)(a - tile * d.nz);
    const int z0 = (tile_phase(tile * d.nz, d.nz, sc.total, gridDim.x) + p0) % d.nz;
    int len = (int)(b - a < d.nz - p0 ? b - a : d.nz - p0);
    if (len > d.nz - z0) len = d.nz - z0;  // not taken (tile_phase): a run never crosses plane nz
    down_segment<V, TL>(d, r, e_out, rc, (int)(tile % sc.tiles_x) * TL::TX, (int)(tile / sc.tiles_x) * TL::TY, z0,
                        z0 + len, inv_h2, cf, sm);
    a += len;
    __syncthreads();
  }
}

template <int V, class TL>
__global__ void __maxnreg__(max_regs<TL>())
k_up_fused(Dims d, const float* __restrict__ e_in, const float* __restrict__ ec, const float* __restrict__ r,
           float* __restrict__ e_out, Sched sc, float inv_h2, Coef cf) {
  extern __shared__ float sm[];
  long long a = (long long)blockIdx.x * sc.total / gridDim.x;
  const long long b = (long long)(blockIdx.x + 1) * sc.total / gridDim.x;
  while (a < b) {
    const long long tile = a / d.nz;
    const int p0 = (int)(a - tile * d.nz);
    const int z0 = (tile_phase(tile * d.nz, d.nz, sc.total, gridDim.x) + p0) % d.nz;
    int len = (int)(b - a < d.nz - p0 ? b - a : d.nz - p0);
    if (len > d.nz - z0) len = d.nz - z0;  // not taken (tile_phase): a run never crosses plane nz
    up_segment<V, TL>(d, e_in, ec, r, e_out, (int)(tile % sc.tiles_x) * TL::TX, (int)(tile / sc.tiles_x) * TL::TY,
                      z0, z0 + len, inv_h2, cf, sm);
    a += len;
    __syncthreads();
  }
}

// ------------------------------------------------------------------ launch

int sm_count() {
  static const int n = []() {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 1)
      v = 152;
    return v;
  }();
  return n;
}

// A CTA whose range crosses a tile's end runs two segments, each with its warm-up planes.
// Where that costs more than leaving some SMs idle, every tile gets the same number of CTAs
// (six tiles of 80^3 or 96^3 on 150 CTAs: 21 -> 13 us; 512^3 keeps all SMs).
template <class TL>
Sched make_sched(Dims d, int warm, int& ctas) {
  Sched sc;
  sc.tiles_x = (d.nx + TL::TX - 1) / TL::TX;
  const long long tiles = (long long)sc.tiles_x * ((d.ny + TL::TY - 1) / TL::TY);
  sc.total = tiles * d.nz;
  const long long sms = sm_count();
  const long long g = sc.total < sms ? sc.total : sms;
  const long long k = sms / tiles < d.nz ? sms / tiles : d.nz;  // CTAs per tile
  ctas = (int)g;
  if (k > 0 && g % tiles != 0 && (d.nz + k - 1) / k + warm < (sc.total + g - 1) / g + 2 * warm) ctas = (int)(k * tiles);
  return sc;
}

template <int V>
cudaError_t down_v(cudaStream_t st, Dims d, const float* r, float* e, float* rc, float ih2, const Coef& cf) {
  using TL = typename DownTile<V>::T;
  const size_t sm = down_smem<V>();
  static DeviceSet done{0};
  const cudaError_t err = allow_smem(done, k_down_fused<V, TL>, sm);
  if (err != cudaSuccess) return err;
  int ctas = 0;
  const Sched sc = make_sched<TL>(d, 2 * V + 3, ctas);
  k_down_fused<V, TL><<<ctas, TL::NT, sm, st>>>(d, r, e, rc, sc, ih2, cf);
  note_launch();
  return cudaGetLastError();
}

template <int V>
cudaError_t up_v(cudaStream_t st, Dims d, const float* e_in, const float* ec, const float* r, float* e_out,
                 float ih2, const Coef& cf) {
  using TL = typename UpTile<V>::T;
  const size_t sm = up_smem<V>();
  static DeviceSet done{0};
  const cudaError_t err = allow_smem(done, k_up_fused<V, TL>, sm);
  if (err != cudaSuccess) return err;
  int ctas = 0;
  const Sched sc = make_sched<TL>(d, 2 * V, ctas);
  k_up_fused<V, TL><<<ctas, TL::NT, sm, st>>>(d, e_in, ec, r, e_out, sc, ih2, cf);
  note_launch();
  return cudaGetLastError();
}

}  // namespace

bool fused_degree_supported(int degree) { return degree >= 1 && degree <= 4; }

cudaError_t launch_down_fused(cudaStream_t st, int degree, Dims d, const float* r, float* e, float* rc, double h,
                              const double* c1, const double* c2) {
  if (d.nx % 2 || d.ny % 2 || d.nz % 2) return cudaErrorInvalidValue;  // levels that are coarsened are even
  const Coef cf = make_coef(c1, c2, degree, h);
  const float ih2 = (float)(1.0 / (h * h));
  switch (degree) {
    case 1: return down_v<1>(st, d, r, e, rc, ih2, cf);
    case 2: return down_v<2>(st, d, r, e, rc, ih2, cf);
    case 3: return down_v<3>(st, d, r, e, rc, ih2, cf);
    case 4: return down_v<4>(st, d, r, e, rc, ih2, cf);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_up_fused(cudaStream_t st, int degree, Dims d, const float* e_in, const float* ec, const float* r,
                            float* e_out, double h, const double* c1, const double* c2) {
  if (d.nx % 2 || d.ny % 2 || d.nz % 2) return cudaErrorInvalidValue;
  const Coef cf = make_coef(c1, c2, degree, h);
  const float ih2 = (float)(1.0 / (h * h));
  switch (degree) {
    case 1: return up_v<1>(st, d, e_in, ec, r, e_out, ih2, cf);
    case 2: return up_v<2>(st, d, e_in, ec, r, e_out, ih2, cf);
    case 3: return up_v<3>(st, d, e_in, ec, r, e_out, ih2, cf);
    case 4: return up_v<4>(st, d, e_in, ec, r, e_out, ih2, cf);
  }
  return cudaErrorInvalidValue;
}

}  // namespace gbmg
