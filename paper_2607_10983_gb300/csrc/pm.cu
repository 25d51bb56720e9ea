// Particle-mesh steps around the Poisson solve (Sec. 2.1 "The PM gravity solve";
// Sec. 3.4, force evaluation = paint, solve, gradient, read): cloud-in-cell paint
// and read on the finest level of a context.  Positions in cell units, node
// (i, j, k) at position (i, j, k), periodic; per axis node floor(x) gets weight
// 1 - f and node floor(x) + 1 weight f, f = x - floor(x), formed in FP64 from the
// FP32 position (exact).  Read is the transpose of paint.
#include "kernels.h"
#include "solver.h"

namespace gbmg {

namespace {

struct Corners {
  long long off[8];
  double w[8];
};

// the 8 corners in the order dz, dy, dx (dx fastest) with their weights (wx wy) wz
__device__ __forceinline__ Corners cic_corners(Dims d, const float* __restrict__ pos, long long p) {
  Corners c;
  double f[3];
  int i0[3], i1[3];  // node floor(x) and floor(x) + 1, wrapped onto the mesh
  const int n[3] = {d.nx, d.ny, d.nz};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const double x = (double)pos[3 * p + a];
    const double fl = floor(x);
    f[a] = __dsub_rn(x, fl);
    int i = (int)fl % n[a];
    i = i < 0 ? i + n[a] : i;
    i0[a] = i;
    i1[a] = i + 1 == n[a] ? 0 : i + 1;
  }
  int k = 0;
#pragma unroll
  for (int dz = 0; dz < 2; ++dz) {
    const double wz = dz ? f[2] : __dsub_rn(1.0, f[2]);
    const long long iz = dz ? i1[2] : i0[2];
#pragma unroll
    for (int dy = 0; dy < 2; ++dy) {
      const double wy = dy ? f[1] : __dsub_rn(1.0, f[1]);
      const long long iy = dy ? i1[1] : i0[1];
#pragma unroll
      for (int dx = 0; dx < 2; ++dx) {
        const double wx = dx ? f[0] : __dsub_rn(1.0, f[0]);
        const long long ix = dx ? i1[0] : i0[0];
        c.off[k] = (iz * d.ny + iy) * d.nx + ix;
        c.w[k] = __dmul_rn(__dmul_rn(wx, wy), wz);
        ++k;
      }
    }
  }
  return c;
}

// ---- paint
//
// What bounds it: the eight FP64 atomics per particle (0.25 ms for 256^3 particles on a 256^3
// mesh).  With the weights formed in FP64 the kernel took 1.11 ms: some thirty FP64
// operations per particle at under 2 per clock and SM.  They are integers here.  A position
// of at least 2^-8 cells in magnitude (or zero) is a multiple of 2^-31, so f and 1 - f are
// 31-bit fixed-point numbers, wx wy is exact in 62 bits, and each product with wz and the
// mass keeps 64 leading bits before the one rounding to FP64 (the FP64 form rounds after
// each product).  Other positions and masses take the FP64 form.

// A finite mass as sign, 64-bit mantissa with its leading bit set, and exponent of that bit.
struct Mass {
  unsigned long long mant, sign;
  int e;
  bool one, ok;  // exactly 1; usable here (normal, with room for the weights' exponents)
};
__device__ __forceinline__ Mass split_mass(double m) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(m);
  const int e = (int)(b >> 52 & 0x7ffu);
  return Mass{(b << 11) | (1ull << 63), b & (1ull << 63), e - 1023, b == 0x3ff0000000000000ull, e > 150 && e < 2040};
}
__device__ __forceinline__ Mass split_mass(float m) {
  const unsigned b = __float_as_uint(m);
  const int e = (int)(b >> 23 & 0xffu);
  return Mass{((unsigned long long)b << 40) | (1ull << 63), (unsigned long long)(b & 0x80000000u) << 32, e - 127,
              b == 0x3f800000u, e > 0 && e < 255};
}

// Position x as node floor(x) and fraction in units of 2^-31; false when it is not such a
// multiple (or not finite, or beyond 2^22).
__device__ __forceinline__ bool split_position(float x, int& node, unsigned& f) {
  const unsigned b = __float_as_uint(x);
  const int e = (int)(b >> 23 & 0xffu);
  const bool zero = (b << 1) == 0;
  long long v = (long long)((b & 0x7fffffu) | 0x800000u) << min(max(e - 119, 0), 30);
  if (b & 0x80000000u) v = -v;
  if (zero) v = 0;
  node = (int)(v >> 31);
  f = (unsigned)v & 0x7fffffffu;
  return zero || (e >= 119 && e < 149);
}

__global__ void k_cic_paint(Dims d, const float* __restrict__ pos, const float* __restrict__ mass, double m0,
                            long long np, double* __restrict__ rho) {
  const int n[3] = {d.nx, d.ny, d.nz};
  const Mass ms = split_mass(m0);
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < np; p += (long long)gridDim.x * blockDim.x) {
    const Mass m = mass ? split_mass(mass[p]) : ms;
    int i0[3], i1[3];
    unsigned f[3];
    bool fast = m.ok;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      fast = split_position(pos[3 * p + a], i0[a], f[a]) && fast;
      if ((unsigned)i0[a] >= (unsigned)n[a]) {
        const int r = i0[a] % n[a];
        i0[a] = r < 0 ? r + n[a] : r;
      }
      i1[a] = i0[a] + 1 == n[a] ? 0 : i0[a] + 1;
    }
    if (!fast) {
      const Corners c = cic_corners(d, pos, p);
      const double md = mass ? (double)mass[p] : m0;
#pragma unroll
      for (int k = 0; k < 8; ++k) atomicAdd(rho + c.off[k], __dmul_rn(md, c.w[k]));
      continue;
    }
#pragma unroll
    for (int dy = 0; dy < 2; ++dy)
#pragma unroll
      for (int dx = 0; dx < 2; ++dx) {
        const unsigned long long wx = dx ? f[0] : 0x80000000u - f[0], wy = dy ? f[1] : 0x80000000u - f[1];
        const unsigned long long wxy = wx * wy;
        if (wxy == 0) continue;
        const int s = __clzll((long long)wxy);
        const unsigned long long A = wxy << s;
        double* const at = rho + (long long)(dy ? i1[1] : i0[1]) * d.nx + (dx ? i1[0] : i0[0]);
#pragma unroll
        for (int dz = 0; dz < 2; ++dz) {
          const unsigned wz = dz ? f[2] : 0x80000000u - f[2];
          if (wz == 0) continue;
          const int sz = __clz((int)wz);
          unsigned long long P = __umul64hi(A, (unsigned long long)(wz << sz) << 32);
          int lz = (int)(P >> 63) ^ 1;
          P <<= lz;
          int e = 2 - lz - s - sz;  // exponent of the leading bit
          if (!m.one) {
            P = __umul64hi(P, m.mant);
            lz = (int)(P >> 63) ^ 1;
            P <<= lz;
            e += m.e + 1 - lz;
          }
          // to 53 bits, ties to even; the sum carries the implicit bit into the exponent
          const unsigned rest = (unsigned)P & 0x7ffu;
          P >>= 11;
          P += (rest > 0x400u || (rest == 0x400u && (P & 1ull))) ? 1ull : 0ull;
          const unsigned long long bits = m.sign | (((unsigned long long)(e + 1022) << 52) + P);
          atomicAdd(at + (long long)(dz ? i1[2] : i0[2]) * d.ny * d.nx, __longlong_as_double((long long)bits));
        }
      }
  }
}

__global__ void k_cic_read(Dims d, const double* __restrict__ field, int ncomp, const float* __restrict__ pos,
                           long long np, double* __restrict__ out) {
  const long long n = ncell(d);
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < np; p += (long long)gridDim.x * blockDim.x) {
    const Corners c = cic_corners(d, pos, p);
    for (int q = 0; q < ncomp; ++q) {
      const double* f = field + q * n;
      double v = 0.0;
#pragma unroll
      for (int k = 0; k < 8; ++k) v = __dadd_rn(v, __dmul_rn(c.w[k], f[c.off[k]]));
      out[p * ncomp + q] = v;
    }
  }
}

// ---- single-precision force path: phi -> FP32, fourth-order gradient in FP32, CIC read in FP32

__global__ void k_phi_to_f32(long long n, const double* __restrict__ phi, float* __restrict__ out) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    out[i] = (float)phi[i];
}

__device__ __forceinline__ int wrap_any(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

// g = -(-u_{i+2} + 8 u_{i+1} - 8 u_{i-1} + u_{i-2}) / 12 along x, y, z (the force, h = 1), the
// components of a cell together: the read then takes eight 16-byte loads per particle
// instead of twenty-four of 4 bytes.  z-marching, the z neighbours in registers.
__global__ void k_force_grid(Dims d, const float* __restrict__ u, float4* __restrict__ g, int zc) {
  const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 8 + threadIdx.y;
  if (x >= d.nx || y >= d.ny) return;
  const int z0 = blockIdx.z * zc, z1 = min(z0 + zc, d.nz);
  const long long sz = (long long)d.nx * d.ny;
  const int row = y * d.nx, i = row + x;
  const int xm = row + wrap_any(x - 1, d.nx), xp = row + wrap_any(x + 1, d.nx), xmm = row + wrap_any(x - 2, d.nx),
            xpp = row + wrap_any(x + 2, d.nx);
  const int ym = wrap_any(y - 1, d.ny) * d.nx + x, yp = wrap_any(y + 1, d.ny) * d.nx + x,
            ymm = wrap_any(y - 2, d.ny) * d.nx + x, ypp = wrap_any(y + 2, d.ny) * d.nx + x;
  const float c8 = 8.f / 12.f, c1 = 1.f / 12.f;
  float w[5];
#pragma unroll
  for (int k = 0; k < 4; ++k) w[k + 1] = u[wrap_any(z0 - 2 + k, d.nz) * sz + i];
  for (int z = z0; z < z1; ++z) {
    const float* const q = u + z * sz;
#pragma unroll
    for (int k = 0; k < 4; ++k) w[k] = w[k + 1];
    w[4] = u[wrap_any(z + 2, d.nz) * sz + i];
    float4 v;
    v.x = c8 * (q[xm] - q[xp]) + c1 * (q[xpp] - q[xmm]);
    v.y = c8 * (q[ym] - q[yp]) + c1 * (q[ypp] - q[ymm]);
    v.z = c8 * (w[1] - w[3]) + c1 * (w[4] - w[0]);
    v.w = 0.f;
    g[z * sz + i] = v;
  }
}

__global__ void k_force_read(Dims d, const float4* __restrict__ g, const float* __restrict__ pos, long long np,
                             float* __restrict__ out) {
  const int nn[3] = {d.nx, d.ny, d.nz};
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < np; p += (long long)gridDim.x * blockDim.x) {
    int i0[3], i1[3];
    float f[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float x = pos[3 * p + a];
      const float fl = floorf(x);
      f[a] = x - fl;
      int i = (int)fl;
      if ((unsigned)i >= (unsigned)nn[a]) {
        i %= nn[a];
        i = i < 0 ? i + nn[a] : i;
      }
      i0[a] = i;
      i1[a] = i + 1 == nn[a] ? 0 : i + 1;
    }
    float4 v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k)
      v[k] = __ldg(g + ((long long)(k & 4 ? i1[2] : i0[2]) * d.ny + (k & 2 ? i1[1] : i0[1])) * d.nx + (k & 1 ? i1[0] : i0[0]));
    float acc[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int dz = 0; dz < 2; ++dz) {
      const float wz = dz ? f[2] : 1.f - f[2];
#pragma unroll
      for (int dy = 0; dy < 2; ++dy) {
        const float wzy = wz * (dy ? f[1] : 1.f - f[1]);
#pragma unroll
        for (int dx = 0; dx < 2; ++dx) {
          const float w = wzy * (dx ? f[0] : 1.f - f[0]);
          const float4 c = v[4 * dz + 2 * dy + dx];
          acc[0] = fmaf(w, c.x, acc[0]);
          acc[1] = fmaf(w, c.y, acc[1]);
          acc[2] = fmaf(w, c.z, acc[2]);
        }
      }
    }
    out[3 * p] = acc[0];
    out[3 * p + 1] = acc[1];
    out[3 * p + 2] = acc[2];
  }
}

int particle_blocks(long long np) {
  long long b = (np + 255) / 256;
  if (b > 152 * 16) b = 152 * 16;
  return (int)(b < 1 ? 1 : b);
}

}  // namespace

}  // namespace gbmg

using namespace gbmg;

extern "C" gbmg_status mg_cic_paint(gbmg_ctx* c, const float* pos_dev, const float* mass_dev, double mass,
                                    long long n_particles, double* rho_dev) {
  if (!c || !rho_dev || n_particles < 0 || (n_particles > 0 && !pos_dev))
    return fail(GBMG_ERR_INVALID_ARG, "mg_cic_paint: bad argument");
  DeviceGuard g(c->device);
  const Dims d = c->lv[0].d;
  TRY(cudaMemsetAsync(rho_dev, 0, (size_t)ncell(d) * sizeof(double), c->stream));
  if (n_particles == 0) return GBMG_OK;
  k_cic_paint<<<particle_blocks(n_particles), 256, 0, c->stream>>>(d, pos_dev, mass_dev, mass, n_particles, rho_dev);
  note_launch();
  TRY(cudaGetLastError());
  return GBMG_OK;
}

extern "C" gbmg_status mg_cic_read(gbmg_ctx* c, const double* field_dev, int ncomp, const float* pos_dev,
                                   long long n_particles, double* out_dev) {
  if (!c || !field_dev || ncomp < 1 || ncomp > 3 || n_particles < 0 || (n_particles > 0 && (!pos_dev || !out_dev)))
    return fail(GBMG_ERR_INVALID_ARG, "mg_cic_read: bad argument");
  DeviceGuard g(c->device);
  if (n_particles == 0) return GBMG_OK;
  k_cic_read<<<particle_blocks(n_particles), 256, 0, c->stream>>>(c->lv[0].d, field_dev, ncomp, pos_dev, n_particles,
                                                                 out_dev);
  note_launch();
  TRY(cudaGetLastError());
  return GBMG_OK;
}

extern "C" gbmg_status mg_force(gbmg_ctx* c, const double* phi_dev, const float* pos_dev, long long n_particles,
                                float* force_out_dev) {
  if (!c || !phi_dev || n_particles < 0 || (n_particles > 0 && (!pos_dev || !force_out_dev)))
    return fail(GBMG_ERR_INVALID_ARG, "mg_force: bad argument");
  DeviceGuard g(c->device);
  const Dims d = c->lv[0].d;
  const long long n = ncell(d);
  if (!c->force_scratch) {
    TRY(cudaMalloc((void**)&c->force_scratch, (size_t)n * 5 * sizeof(float)));
    c->owned.push_back(c->force_scratch);
  }
  float4* gr = (float4*)c->force_scratch;  // the force grid, then phi in FP32
  float* u = c->force_scratch + 4 * n;
  k_phi_to_f32<<<(int)df_partial_count(n), 256, 0, c->stream>>>(n, phi_dev, u);
  note_launch();
  TRY(cudaGetLastError());
  // z planes per thread: 16, fewer while the mesh does not give every SM four blocks
  const long long cols = (long long)((d.nx + 31) / 32) * ((d.ny + 7) / 8);
  int zc = 16;
  while (zc > 1 && cols * ((d.nz + zc - 1) / zc) < 4 * 152) zc /= 2;
  k_force_grid<<<dim3((d.nx + 31) / 32, (d.ny + 7) / 8, (d.nz + zc - 1) / zc), dim3(32, 8), 0, c->stream>>>(d, u, gr, zc);
  note_launch();
  TRY(cudaGetLastError());
  if (n_particles == 0) return GBMG_OK;
  k_force_read<<<particle_blocks(n_particles), 256, 0, c->stream>>>(d, gr, pos_dev, n_particles, force_out_dev);
  note_launch();
  TRY(cudaGetLastError());
  return GBMG_OK;
}
