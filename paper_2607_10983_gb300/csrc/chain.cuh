// The bottom of a V-cycle whose operations run one after the other on levels of a few thousand
// cells, in one launch: a cluster of CTAs with a hardware barrier between operations instead of
// a kernel each.  The FP64 flat chain uses it.
//
// What bounds such a chain is launches: 17 of 2 to 4 us with their gaps for two levels (16^3,
// 8^3) and the coarsest solve, of which the arithmetic is a small part.  16 CTAs are the
// largest cluster: FP64 (two operations per clock and SM) wants as many SMs as there are, and
// one cell per thread.  A CTA keeps its cells of every field in shared memory and reads its
// neighbours' there (distributed shared memory): through L2 a barrier waits for the stores and
// the next loads for L2, 2.1 us per operation and nothing gained (36.8 us for 17).  The
// operations are those of the kernels they replace, in their order (the same bits); each exists
// once in the code, which a kernel that runs once pays for on every launch.
// 16^3, 8^3 and 4^3 in FP64, degree 3: 31 -> 25 us a cycle.  The curvilinear chain in this form
// took 35 us against 31 in launches: each cell's coefficient loads (about 60) go to L2 again
// after every barrier.
#pragma once
#include <cooperative_groups.h>

#include "kernels.h"
#include "stencil.cuh"

namespace gbmg {
namespace chain {

constexpr int kMaxL = 8;
constexpr int kCtas = 16;

// Level 0's e (and d) hold the first pre-smoothing step; levels 1 .. nl - 2 get theirs from the
// restriction; level nl - 1 is solved with the dense pseudo-inverse.  Cell i of a level lives in
// CTA i >> sh, whose fields of the level start at byte off: e, e2, t, r, d (1 << sh cells each).
struct Level {
  Dims d;
  int sh, off;
};
template <typename T>
struct Fields {
  int nl, pre, post;   // levels; smoothing steps still to do before, and after the correction
  int nc;
  const T* G;
  T *e, *r, *d;        // level 0 (d: NULL without one); e receives the result
  Level lv[kMaxL];
};
enum { E = 0, E2 = 1, TMP = 2, R = 3, DV = 4, NFIELD = 5 };

// A field of a level, wherever its cells live: base = shared address in any CTA.
template <typename T>
struct View {
  unsigned base;
  int sh;
  __device__ __forceinline__ View(const Level& L, int field)
      : base(L.off + ((unsigned)(field * sizeof(T)) << L.sh)), sh(L.sh) {}
  __device__ __forceinline__ T operator[](int i) const {
    unsigned a = base + (unsigned)(i & ((1 << sh) - 1)) * (unsigned)sizeof(T);
    asm("mapa.shared::cluster.u32 %0, %0, %1;" : "+r"(a) : "r"(i >> sh));
    T v;
    if constexpr (sizeof(T) == 8) asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    else asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
  }
  // the CTA's own cells
  __device__ __forceinline__ T& own(char* sm, unsigned s0, int j) const {
    return reinterpret_cast<T*>(sm + (base - s0))[j];
  }
};

// a cell's coordinates
struct Cell {
  int x, y, z;
  __device__ __forceinline__ Cell(Dims d, int i) {
    const int q = i / d.nx;
    x = i - q * d.nx;
    z = q / d.ny;
    y = q - z * d.ny;
  }
};

// k_restrict's value at a coarse cell: z weights, then y, then x
template <typename T>
__device__ __forceinline__ T restrict_value(Dims df, const View<T>& f, const Cell& c) {
  int xs[3], ys[3], zs[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    xs[k] = wrapi(2 * c.x + k - 1, df.nx);
    ys[k] = wrapi(2 * c.y + k - 1, df.ny) * df.nx;
    zs[k] = wrapi(2 * c.z + k - 1, df.nz) * df.nx * df.ny;
  }
  T v[3][3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
      for (int k = 0; k < 3; ++k) v[a][b][k] = f[zs[k] + ys[b] + xs[a]];
  T yv[3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
    yv[a] = fw3(fw3(v[a][0][0], v[a][0][1], v[a][0][2]), fw3(v[a][1][0], v[a][1][1], v[a][1][2]),
                fw3(v[a][2][0], v[a][2][1], v[a][2][2]));
  return fw3(yv[0], yv[1], yv[2]);
}

// prolong_value of stencil.cuh
template <typename T>
__device__ __forceinline__ T prolong_cell(const View<T>& c, Dims dc, const Cell& f) {
  const int I = f.x >> 1, J = f.y >> 1, K = f.z >> 1;
  const bool dx = f.x & 1, dy = f.y & 1, dz = f.z & 1;
  const int I1 = wrap_hi(I + 1, dc.nx), J1 = wrap_hi(J + 1, dc.ny), K1 = wrap_hi(K + 1, dc.nz);
  auto cx = [&](int jj, int kk) -> T {
    const int row = (kk * dc.ny + jj) * dc.nx;
    const T a = c[row + I], b = c[row + I1];
    return dx ? half_sum(a, b) : a;
  };
  const T a = cx(J, K), b = cx(J1, K), p = cx(J, K1), q = cx(J1, K1);
  const T v0 = dy ? half_sum(a, b) : a, v1 = dy ? half_sum(p, q) : p;
  return dz ? half_sum(v0, v1) : v0;
}

// OP: const Fields<T>& f(); T step(l, k, in, e, r, d, i, cell): step k of level l's smoothing (k <
// 0: the residual) at cell i, d its direction; T first(l, r, d, i): the first step from zero.
template <class OP>
__device__ __forceinline__ void run(const OP& op) {
  using T = typename OP::T;
  extern __shared__ __align__(16) char sm[];
  const Fields<T>& F = op.f();
  cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  const int rank = cl.block_rank(), tid = threadIdx.x, nt = blockDim.x;
  const unsigned s0 = (unsigned)__cvta_generic_to_shared(sm);
  auto field = [&](int l, int f) {
    View<T> v(F.lv[l], f);
    v.base += s0;
    return v;
  };
  // body(i, j) for the CTA's cells i of level l, j their places
  auto cells = [&](int l, auto body) {
    const Level& L = F.lv[l];
    const int n = (int)ncell(L.d);
#pragma unroll 1
    for (int j = tid; j < 1 << L.sh; j += nt) {
      const int i = (rank << L.sh) + j;
      if (i < n) body(i, j);
    }
  };
  unsigned flip = 0;   // bit l: e2 holds level l's iterate
  cells(0, [&](int i, int j) {
    field(0, E).own(sm, s0, j) = F.e[i];
    field(0, R).own(sm, s0, j) = F.r[i];
    if (F.d) field(0, DV).own(sm, s0, j) = F.d[i];
  });
  cl.sync();
#pragma unroll 1
  for (int v = 0; v < 2 * (F.nl - 1); ++v) {
    const bool down = v < F.nl - 1;
    const int l = down ? v : 2 * (F.nl - 1) - 1 - v;
    const Dims dl = F.lv[l].d, dc = F.lv[l + 1].d;
    if (!down) {
      const View<T> e = field(l, flip >> l & 1u), ec = field(l + 1, flip >> (l + 1) & 1u);
      cells(l, [&](int i, int j) { e.own(sm, s0, j) = t_add(e.own(sm, s0, j), prolong_cell(ec, dc, Cell(dl, i))); });
      cl.sync();
    }
    const int steps = down ? F.pre + 1 : F.post;
#pragma unroll 1
    for (int k = 0; k < steps; ++k) {
      const bool res = down && k == F.pre;
      const View<T> in = field(l, flip >> l & 1u), r = field(l, R), d = field(l, DV);
      const View<T> out = field(l, res ? TMP : 1 - (flip >> l & 1u));
      const int ks = res ? -1 : (down ? k + OP::kDone : k);
      cells(l, [&](int i, int j) {
        out.own(sm, s0, j) = op.step(l, ks, in, in.own(sm, s0, j), r.own(sm, s0, j), d.own(sm, s0, j), i, Cell(dl, i));
      });
      if (!res) flip ^= 1u << l;
      cl.sync();
    }
    if (!down) continue;
    {
      const View<T> t = field(l, TMP);
      cells(l + 1, [&](int i, int j) {
        const T rv = restrict_value(dl, t, Cell(dc, i));
        field(l + 1, R).own(sm, s0, j) = rv;
        if (l + 1 < F.nl - 1) field(l + 1, E).own(sm, s0, j) = op.first(l + 1, rv, field(l + 1, DV).own(sm, s0, j), i);
      });
      cl.sync();
    }
    if (l + 1 < F.nl - 1) continue;
    // coarsest solve: k_coarse_matvec, the CTA's rows
    const View<T> r = field(l + 1, R);
    const int lane = tid & 31, sh = F.lv[l + 1].sh;
#pragma unroll 1
    for (int j = tid >> 5; j < 1 << sh; j += nt >> 5) {
      const int row = (rank << sh) + j;
      if (row >= F.nc) break;
      T acc = T(0);
      for (int q = lane; q < F.nc; q += 32) acc = t_fma(F.G[(long long)row * F.nc + q], r[q], acc);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc = t_add(acc, __shfl_xor_sync(0xffffffffu, acc, o));
      if (lane == 0) field(l + 1, E).own(sm, s0, j) = acc;
    }
    cl.sync();
  }
  const View<T> e = field(0, flip & 1u);
  cells(0, [&](int i, int j) { F.e[i] = e.own(sm, s0, j); });
}

// The levels' places; returns the shared memory of a CTA.
template <typename T>
size_t layout(Fields<T>& F) {
  size_t off = 0;
  for (int l = 0; l < F.nl; ++l) {
    int sh = 0;
    while ((long long)kCtas << sh < ncell(F.lv[l].d)) ++sh;
    F.lv[l].sh = sh;
    F.lv[l].off = (int)off;
    off += ((NFIELD * sizeof(T) << sh) + 15) / 16 * 16;
  }
  return off;
}

// Configuration of a kernel whose CTAs form one cluster of kCtas; its limits are set.
struct Config {
  cudaLaunchConfig_t c = {};
  cudaLaunchAttribute at = {};
};
template <typename K>
cudaError_t configure(Config& q, cudaStream_t st, K kernel, int threads, size_t smem) {
  cudaError_t e = cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  q.c.gridDim = dim3(kCtas);
  q.c.blockDim = dim3(threads);
  q.c.dynamicSmemBytes = smem;
  q.c.stream = st;
  q.at.id = cudaLaunchAttributeClusterDimension;
  q.at.val.clusterDim.x = kCtas;
  q.at.val.clusterDim.y = q.at.val.clusterDim.z = 1;
  q.c.attrs = &q.at;
  q.c.numAttrs = 1;
  return e;
}
// 16 CTAs are more than the portable cluster size: a device or a partition may have no room
// for them.
template <typename K>
bool fits(K kernel, int threads, size_t smem) {
  Config q;
  int n = 0;
  const bool ok = configure(q, nullptr, kernel, threads, smem) == cudaSuccess &&
                  cudaOccupancyMaxActiveClusters(&n, kernel, &q.c) == cudaSuccess && n > 0;
  if (!ok) (void)cudaGetLastError();
  return ok;
}
template <typename K, typename A>
cudaError_t launch(cudaStream_t st, K kernel, int threads, size_t smem, const A& args) {
  Config q;
  cudaError_t e = configure(q, st, kernel, threads, smem);
  if (e == cudaSuccess) e = cudaLaunchKernelEx(&q.c, kernel, args);
  if (e == cudaSuccess) note_launch();
  return e;
}

}  // namespace chain
}  // namespace gbmg
