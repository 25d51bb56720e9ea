// The bottom of the FP32 V-cycle (the levels that fit in shared memory) by one CTA of
// kSmallThreads threads, for the kernel of single solves and for the batches' phase graph: a
// level visit of the one-kernel-per-operation chain costs a launch per
// operation while each operation is a few thousand cells; here the same operations run
// as phases of one CTA separated by __syncthreads, each cell with the chain's arithmetic
// (the same bits).  The batched persistent kernel, whose registers the legs fill, runs the one-cell
// form of small_cycle.cuh instead: this one inlined there spilled the legs (48 problems in
// 16.6 instead of 14.9 ms).
//
// What bounds it: about twenty dependent phases, each a round of shared loads and a
// barrier, and fetching the code, which runs once per launch.  So
//   - a thread's item is a column of four z cells: all its loads are issued before the
//     first value is used, its z neighbours come from registers, and its indices are formed
//     once per level visit instead of once per cell and phase;
//   - r and the Chebyshev direction stay in registers over a smoothing pass when every item
//     has its own thread;
//   - the first pre-smoothing step, of a zero iterate, is pointwise;
//   - each phase's code exists once, in a loop over levels and steps (unrolled over the
//     levels the kernel took 22 us with warm caches and 36 us between the passes of a large
//     mesh).
// 16^3, 8^3, 4^3: 25 -> 15.6 us inside the cycles of 64^3, 36 -> 15.9 us inside those of 512^3.
#pragma once
#include "kernels.h"
#include "stencil.cuh"

namespace gbmg {
namespace smallcta {

// A column of up to four z cells: offset of its first cell, relative offsets of the x and y
// neighbours, offsets of the cells below and above, and of its cells (beyond the column's
// end: the last cell again, loaded and not stored).
struct Item {
  int cnt, xm, xp, ym, yp, below, above;
  int x, y, z;
  int i[4];
  __device__ __forceinline__ void set(Dims d, int it) {
    const int ncol = d.nx * d.ny;
    const int zb = it / ncol, col = it - zb * ncol;
    y = col / d.nx;
    x = col - y * d.nx;
    z = 4 * zb;
    cnt = min(d.nz - z, 4);
    xm = x == 0 ? d.nx - 1 : -1;
    xp = x == d.nx - 1 ? 1 - d.nx : 1;
    ym = (y == 0 ? d.ny - 1 : -1) * d.nx;
    yp = (y == d.ny - 1 ? 1 - d.ny : 1) * d.nx;
#pragma unroll
    for (int q = 0; q < 4; ++q) i[q] = (z + min(q, cnt - 1)) * ncol + col;
    below = (z == 0 ? d.nz - 1 : z - 1) * ncol + col;
    above = (z + cnt == d.nz ? 0 : z + cnt) * ncol + col;
  }
};
__device__ __forceinline__ int item_count(Dims d) { return d.nx * d.ny * ((d.nz + 3) / 4); }

// values and neighbour sums of an item's cells
__device__ __forceinline__ void load_item(const Item& I, const float* u, float (&c)[4], float (&s)[4]) {
  float xm[4], xp[4], ym[4], yp[4];
  const float lo = u[I.below], hi = u[I.above];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float* const p = u + I.i[q];
    c[q] = p[0];
    xm[q] = p[I.xm];
    xp[q] = p[I.xp];
    ym[q] = p[I.ym];
    yp[q] = p[I.yp];
  }
#pragma unroll
  for (int q = 0; q < 4; ++q)
    s[q] = lap_sum(xm[q], xp[q], ym[q], yp[q], q ? c[q - 1] : lo, q + 1 < I.cnt && q < 3 ? c[q + 1] : hi, c[q]);
}

// e_out = V-cycle(r_in) on level 0 of P; sm: small_cycle_smem(P) bytes.
__device__ __forceinline__ void vcycle(const SmallCycle& P, const float* __restrict__ r_in, float* __restrict__ e_out,
                                       float* sm) {
  const int tid = threadIdx.x, lane = tid & 31;
  constexpr int nt = kSmallThreads;
  // the coarsest inverse on its way while the levels above it run
  for (int i = tid * 32; i < P.nc * P.nc; i += nt * 32)
    asm volatile("prefetch.global.L2 [%0];" ::"l"(P.G + i));
  // level l's fields from base: r, e, e2, d (the coarsest: r, e); bit l of cur: e is in e2
  unsigned cur = 0;
  int l = 0, base = 0, n = (int)ncell(P.d[0]);
  bool down = true;
  Item I;
  I.set(P.d[0], tid);
  for (;;) {
    const Dims d = P.d[l];
    const int items = item_count(d);
    const bool one = items <= nt;  // every item has its own thread
    float* const R = sm + base;
    float* const DV = R + 3 * n;
    float* E = R + n + ((cur >> l & 1u) ? n : 0);
    float* E2 = R + n + ((cur >> l & 1u) ? 0 : n);
    // ---- a smoothing pass
    float r[4], dv[4] = {0.f, 0.f, 0.f, 0.f};
    int k = 0;
    if (down) {
      // from zero: e = 0, s = 0, the direction starts at zero
      const float a = P.a[l][0], b = P.b[l][0], c1 = P.c1[0];
      const bool load = l == 0;
#pragma unroll 1
      for (int it = tid; it < items; it += nt) {
        if (!one) I.set(d, it);
#pragma unroll
        for (int q = 0; q < 4; ++q) r[q] = load ? __ldg(r_in + I.i[q]) : R[I.i[q]];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float t = 0.f;
          const float e = cheb_step(0.f, r[q], 0.f, t, a, b, c1);
          dv[q] = t;
          if (q >= I.cnt) continue;
          if (load) R[I.i[q]] = r[q];
          E2[I.i[q]] = e;
          if (!one) DV[I.i[q]] = t;
        }
      }
      k = 1;
      float* const t = E;
      E = E2;
      E2 = t;
      __syncthreads();
    } else if (one && tid < items) {
#pragma unroll
      for (int q = 0; q < 4; ++q) r[q] = R[I.i[q]];
    }
#pragma unroll 1
    for (; k < P.degree; ++k) {
      const float a = P.a[l][k], b = P.b[l][k], c1 = P.c1[k];
      const bool store = l == 0 && !down && k == P.degree - 1;
#pragma unroll 1
      for (int it = tid; it < items; it += nt) {
        if (!one) {
          I.set(d, it);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            r[q] = R[I.i[q]];
            dv[q] = k > 0 ? DV[I.i[q]] : 0.f;
          }
        }
        float c[4], s[4], e[4];
        load_item(I, E, c, s);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (c1 == 0.f) dv[q] = 0.f;
          e[q] = cheb_step(c[q], r[q], s[q], dv[q], a, b, c1);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (q >= I.cnt) continue;
          if (store) e_out[I.i[q]] = e[q];
          else E2[I.i[q]] = e[q];
          if (!one) DV[I.i[q]] = dv[q];
        }
      }
      float* const t = E;
      E = E2;
      E2 = t;
      __syncthreads();
    }
    cur ^= (unsigned)(P.degree & 1) << l;
    if (down) {
      // ---- residual (into the free error buffer), restriction
      const float ih2 = P.inv_h2[l];
#pragma unroll 1
      for (int it = tid; it < items; it += nt) {
        if (!one) {
          I.set(d, it);
#pragma unroll
          for (int q = 0; q < 4; ++q) r[q] = R[I.i[q]];
        }
        float c[4], s[4];
        load_item(I, E, c, s);
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q < I.cnt) E2[I.i[q]] = resid_from_sum(r[q], s[q], ih2);
      }
      __syncthreads();
      const float* const T = E2;
      base += 4 * n;
      ++l;
      const Dims dc = P.d[l];
      const int pl = d.nx * d.ny, pc = dc.nx * dc.ny;
      float* const Rc = sm + base;
      n = (int)ncell(dc);
#pragma unroll 1
      for (int i = tid; i < n; i += nt) {
        const int Z = i / pc, q = i - Z * pc, Y = q / dc.nx, X = q - Y * dc.nx;
        const int x0 = 2 * X, xm = x0 == 0 ? d.nx - 1 : x0 - 1;
        const int zo[3] = {(Z == 0 ? d.nz - 1 : 2 * Z - 1) * pl, 2 * Z * pl, (2 * Z + 1) * pl};
        const int yo[3] = {(Y == 0 ? d.ny - 1 : 2 * Y - 1) * d.nx, 2 * Y * d.nx, (2 * Y + 1) * d.nx};
        float v[3][3][3];
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            const float* const p = T + zo[a] + yo[b];
            v[0][b][a] = p[xm];
            v[1][b][a] = p[x0];
            v[2][b][a] = p[x0 + 1];
          }
        float yv[3];
#pragma unroll
        for (int a = 0; a < 3; ++a)
          yv[a] = fw3(fw3z(v[a][0][0], v[a][0][1], v[a][0][2]), fw3z(v[a][1][0], v[a][1][1], v[a][1][2]),
                      fw3z(v[a][2][0], v[a][2][1], v[a][2][2]));
        Rc[i] = fw3(yv[0], yv[1], yv[2]);
      }
      I.set(dc, tid);
      __syncthreads();
      if (l < P.nl - 1) continue;
      // ---- coarsest: e = G r, one warp per row, lanes stride the columns; four rows at a
      // time, their loads together
      float* const Ec = Rc + n;
      constexpr int nw = nt >> 5;
#pragma unroll 1
      for (int row = tid >> 5; row < P.nc; row += 4 * nw) {
        const float* g[4];
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int q = 0; q < 4; ++q) g[q] = P.G + (long long)min(row + q * nw, P.nc - 1) * P.nc;
#pragma unroll 2
        for (int j = lane; j < P.nc; j += 32) {
          const float rv = Rc[j];
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[q] = t_fma(__ldg(g[q] + j), rv, acc[q]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[q] = t_add(acc[q], __shfl_xor_sync(0xffffffffu, acc[q], o));
        if (lane == 0)
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (row + q * nw < P.nc) Ec[row + q * nw] = acc[q];
      }
      __syncthreads();
      down = false;
    } else if (l == 0) {
      break;
    }
    // ---- up one level: prolongation + correction
    const Dims dc = P.d[l];
    const int pc = dc.nx * dc.ny;
    const float* const Ec = sm + base + n + ((cur >> l & 1u) ? n : 0);
    --l;
    const Dims df = P.d[l];
    n = (int)ncell(df);
    base -= 4 * n;
    const int itf = item_count(df);
    float* const Ef = sm + base + n + ((cur >> l & 1u) ? n : 0);
    I.set(df, tid);
#pragma unroll 1
    for (int it = tid; it < itf; it += nt) {
      if (it != tid) I.set(df, it);
      // coarse values under the column: planes K, K + 1, K + 2 (z is a multiple of four)
      const int X = I.x >> 1, Y = (I.y >> 1) * dc.nx, K = I.z >> 1;
      const bool dx = I.x & 1, dy = I.y & 1;
      const int X1 = X + 1 == dc.nx ? 0 : X + 1, Y1 = (I.y >> 1) + 1 == dc.ny ? 0 : Y + dc.nx;
      float w[3][4], cy[3], e[4];
#pragma unroll
      for (int k2 = 0; k2 < 3; ++k2) {
        const int Kk = min(K + k2, K + (I.cnt >> 1));  // beyond a short column: not used
        const float* const p = Ec + (Kk >= dc.nz ? Kk - dc.nz : Kk) * pc;
        w[k2][0] = p[Y + X];
        w[k2][1] = p[Y + X1];
        w[k2][2] = p[Y1 + X];
        w[k2][3] = p[Y1 + X1];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) e[q] = Ef[I.i[q]];
#pragma unroll
      for (int k2 = 0; k2 < 3; ++k2) {
        const float c0 = dx ? half_sum(w[k2][0], w[k2][1]) : w[k2][0], c1 = dx ? half_sum(w[k2][2], w[k2][3]) : w[k2][2];
        cy[k2] = dy ? half_sum(c0, c1) : c0;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q < I.cnt) Ef[I.i[q]] = t_add(e[q], q & 1 ? half_sum(cy[q >> 1], cy[(q >> 1) + 1]) : cy[q >> 1]);
    }
    __syncthreads();
  }
}

}  // namespace smallcta
}  // namespace gbmg
