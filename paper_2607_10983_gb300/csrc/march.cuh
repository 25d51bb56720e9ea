// Tile machinery of the z-marching curvilinear kernels (curv_march.cu): a CTA owns a
// 32 x 16 tile of cells and a run of z planes; the haloed planes of u and of the six
// components of B pass through a three-slot shared-memory ring filled by 16-byte
// asynchronous copies.
//
// A thread owns R rows of one x column in the low lane of packed FP32x2 registers and the
// rows 8 further on in the high lane.  Every neighbour of a packed row is the same offset
// for both lanes, so no operand is ever re-paired, and a warp reads 32 consecutive floats
// per shared load (no bank conflict).
//
// Each field keeps the rows and columns its neighbours need: u and xy on all sides, xx and
// xz in x, yy and yz in y, zz none.  A field with x neighbours holds the aligned 40 cells
// x0 - 4 .. x0 + 35 of a row: two 4-byte copies per row for the two cells x0 - 1 and
// x0 + 32 moved fewer bytes but took one sector and one request each, and the sweep of
// 256^3 ran in 245 us with them against 122 us without any x halo.
#pragma once
#include "kernels.h"
#include "packed.cuh"

namespace gbmg {
namespace march {

constexpr int MX = 32, MY = 16;            // tile
constexpr int PA = MX + 8, PB = MX;        // row pitch with and without x neighbours
constexpr int NF = 7;                      // fields: u and B
enum { FU = 0, FXX = 1, FYY = 2, FZZ = 3, FXY = 4, FXZ = 5, FYZ = 6 };
constexpr bool has_x(int f) { return f == FU || f == FXX || f == FXY || f == FXZ; }
constexpr bool has_y(int f) { return f == FU || f == FYY || f == FXY || f == FYZ; }
constexpr int f_chunks(int f) { return (has_y(f) ? MY + 2 : MY) * (has_x(f) ? PA : PB) / 4; }
constexpr int f_off(int f) {  // floats before field f in a slot
  int o = 0;
  for (int k = 0; k < f; ++k) o += f_chunks(k) * 4;
  return o;
}
constexpr int SLOT = f_off(NF);            // floats of one ring slot

__device__ __forceinline__ void cp_async16(unsigned dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async8(unsigned dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ int wrap_mod(int i, int n) {
  const int r = i % n;
  return r < 0 ? r + n : r;
}

struct Fields {
  const float* p[NF];
};

// Fields sharing a halo shape share their chunk offsets: 0 = u, xy; 1 = xx, xz; 2 = yy,
// yz; 3 = zz.
constexpr int f_group(int f) { return has_x(f) ? (has_y(f) ? 0 : 1) : (has_y(f) ? 2 : 3); }

// The copies of one plane of the fields F0 .. NF - 1 by NT threads (128 or 256): thread t
// copies chunk t of every field (its place in the slot is t 16-byte units into the field);
// with 128 threads the chunks from 128 on, of all fields one after the other, are dealt
// out as extras.
template <int NT, int F0 = 0>
struct Copier {
  static constexpr int extra_count() {
    int n = 0;
    for (int f = F0; f < NF; ++f) n += f_chunks(f) > NT ? f_chunks(f) - NT : 0;
    return n;
  }
  static constexpr int NE = (extra_count() + NT - 1) / NT;
  int off[4];                          // in-plane offset of the thread's chunk per group
  const float* x_src[NE ? NE : 1];     // extras: chunk of plane 0 (NULL: none), place in a slot
  unsigned x_dst[NE ? NE : 1];

  static __device__ __forceinline__ int chunk_off(Dims d, int x0, int y0, bool hx, bool hy, int c) {
    const int per = hx ? PA / 4 : PB / 4;
    const int row = c / per, q = c % per;
    return wrap_mod(y0 + row - (hy ? 1 : 0), d.ny) * d.nx + wrap_mod(x0 + 4 * q - (hx ? 4 : 0), d.nx);
  }
  __device__ __forceinline__ void init(Dims d, const Fields& P, int x0, int y0) {
    const int tid = threadIdx.x;
    off[0] = chunk_off(d, x0, y0, true, true, tid);
    off[1] = chunk_off(d, x0, y0, true, false, tid);
    off[2] = chunk_off(d, x0, y0, false, true, tid);
    off[3] = chunk_off(d, x0, y0, false, false, tid);
#pragma unroll
    for (int k = 0; k < NE; ++k) {
      int q = tid + k * NT;
      x_src[k] = nullptr;
      x_dst[k] = 0;
#pragma unroll
      for (int f = F0; f < NF; ++f) {
        const int n = f_chunks(f) > NT ? f_chunks(f) - NT : 0;
        if (q >= 0 && q < n) {
          x_src[k] = P.p[f] + chunk_off(d, x0, y0, has_x(f), has_y(f), NT + q);
          x_dst[k] = (unsigned)((f_off(f) - f_off(F0)) * 4 + (NT + q) * 16);
        }
        q -= n;
      }
    }
  }
  // the plane at offset zo into the slot at shared address sa
  __device__ __forceinline__ void issue(const Fields& P, long long zo, unsigned sa) const {
    const unsigned t = sa + threadIdx.x * 16u;
#pragma unroll
    for (int f = F0; f < NF; ++f)
      if (f_chunks(f) >= NT || threadIdx.x < f_chunks(f))
        cp_async16(t + (unsigned)(f_off(f) - f_off(F0)) * 4u, P.p[f] + (zo + off[f_group(f)]));
#pragma unroll
    for (int k = 0; k < NE; ++k)
      if (x_src[k]) cp_async16(sa + x_dst[k], x_src[k] + zo);
  }
};

// Shared-memory view of a thread whose first low-lane row is tile row `row`: one packed
// value of field F, dr rows and dx cells away, in the slot at offset s (floats).
struct View {
  const float* a;  // pitch PA, tile row -1 at haloed row 0
  const float* b;  // pitch PB
  __device__ __forceinline__ View(const float* sm, int row, int lane)
      : a(sm + (row + 1) * PA + 4 + lane), b(sm + (row + 1) * PB + lane) {}
  template <int F>
  __device__ __forceinline__ float2 at(int s, int dr, int dx) const {
    constexpr int p = has_x(F) ? PA : PB;
    const float* q = (has_x(F) ? a : b) + s + f_off(F) + (has_y(F) ? 0 : -p) + dr * p + dx;
    return make_float2(q[0], q[8 * p]);
  }
};

// z planes per CTA: among runs of 2 .. nz planes the one with the least work on the
// critical path, whole waves of `resident` CTAs times the run plus its two extra planes (from 4
// planes on: a sweep of 80 x 64 x 96 9.5 instead of 9.2 us, of 64^3 7.4 instead of 6.7).
inline int march_zchunk(Dims d, int resident) {
  const long long tiles = (long long)((d.nx + MX - 1) / MX) * ((d.ny + MY - 1) / MY);
  int best = d.nz;
  long long best_cost = -1;
  for (int n = 1; n <= d.nz; ++n) {
    const int zc = (d.nz + n - 1) / n;
    if (zc < 2 && n > 1) break;
    const long long waves = (tiles * ((d.nz + zc - 1) / zc) + resident - 1) / resident;
    const long long cost = waves * (zc + 2);
    if (best_cost < 0 || cost < best_cost) best_cost = cost, best = zc;
  }
  return best;
}
inline dim3 march_grid(Dims d, int zc) {
  return dim3((d.nx + MX - 1) / MX, (d.ny + MY - 1) / MY, (d.nz + zc - 1) / zc);
}

}  // namespace march
}  // namespace gbmg
