// Single-CTA kernel of the bottom of the FP32 V-cycle (device code in small_cta.cuh).
#include "small_cta.cuh"

namespace gbmg {

namespace {

__global__ void __launch_bounds__(kSmallThreads, 1) k_small_vcycle(const __grid_constant__ SmallCycle P,
                                                                   const float* __restrict__ r_in,
                                                                   float* __restrict__ e_out) {
  extern __shared__ __align__(16) float sm[];
  smallcta::vcycle(P, r_in, e_out, sm);
}

}  // namespace

size_t small_cycle_smem(const SmallCycle& P) {
  size_t f = 0;
  for (int l = 0; l < P.nl; ++l) f += (size_t)ncell(P.d[l]) * (l < P.nl - 1 ? 5 : 2);
  return f * sizeof(float);
}

cudaError_t launch_small_vcycle(cudaStream_t st, const SmallCycle& P, const float* r_in, float* e_out) {
  if (P.nl < 2 || P.nl > kSmallMaxL || ncell(P.d[0]) > kSmallCells || P.degree < 1 || P.degree > 16 ||
      P.nc != ncell(P.d[P.nl - 1]))
    return cudaErrorInvalidValue;
  const size_t sm = small_cycle_smem(P);
  if (sm > kSmallSmem) return cudaErrorInvalidValue;
  static DeviceSet done{0};
  const cudaError_t err = allow_smem(done, k_small_vcycle, kSmallSmem);
  if (err != cudaSuccess) return err;
  k_small_vcycle<<<1, kSmallThreads, sm, st>>>(P, r_in, e_out);
  note_launch();
  return cudaGetLastError();
}

}  // namespace gbmg
