// The legs of a small level's visit (between the bottom cycle and the levels that the
// z-streaming legs are made for), a block of 8^3 cells per CTA:
//
//   k_block_down : V Chebyshev steps from e = 0, residual, full-weighting restriction
//   k_block_up   : prolongation + correction, V Chebyshev steps
//
// What bounds such a visit is latency: as a chain of one kernel per operation the two legs of
// a 32^3 level take 18 us of launches, each a few thousand cells long; the streaming legs take
// 10 us each at any size up to 64^3, a plane per iteration.  Here a CTA holds its block and a
// halo wide enough for all steps in shared memory, computes every step on the whole region
// (the ring that a step cannot know is wrong and shrinks the valid region, the outputs lie
// inside), and one barrier separates the steps.  That is up to eight times the arithmetic,
// which idle SMs do for free on a small mesh.
//
// A thread owns half a z column, eight cells: r, d and e in registers, its z neighbours among
// them, and the x and y neighbours are two 16-byte loads per neighbouring column (columns of 16
// cells stored z-fastest with a stride of 20 words: eight lanes read all 32 banks).  The steps and
// the residual are one loop, not unrolled: a kernel that runs once is bound by fetching its code.
// Each cell gets the operations of the per-operation kernels in their order (the same bits).
// Degree 3, both legs: 32^3 18 -> 8.3 us (64 CTAs), 48^3 20.2 (streaming) and 12.1; from 64^3
// on the arithmetic of the halos counts (21.2 against 19.7 us) and the streaming legs run.
#include "legs.cuh"

namespace gbmg {

namespace {

constexpr int BO = 8;        // outputs per side
constexpr int BZ = 16;       // cells of a column: outputs and 4 cells on either side
constexpr int CS = 20;       // words of a stored column
constexpr int BC = 9;        // coarse nodes per side under the up leg's region

// steps of the loop: constants of the Chebyshev steps, then (down leg) of the residual
struct BlockCoef {
  float c1[4], a[4], mb[4];
};

template <int H>
struct BlockTile {
  static constexpr int E = BO + 2 * H, NCOL = E * E, NT = (2 * NCOL + 31) / 32 * 32;
  static constexpr int PLANE = NCOL * CS;
};

template <int H>
struct BlockPos {
  using T = BlockTile<H>;
  int cx, cy, ch;               // column, half
  int own, xm, xp, ym, yp;      // offsets of the half column and its neighbours (clamped)
  bool act;
  int gxy, gz;                  // offset in a plane, first z
  bool out;                     // holds outputs
  __device__ __forceinline__ void init(Dims d, int x0, int y0, int z0) {
    const int tid = threadIdx.x;
    act = tid < 2 * T::NCOL;
    ch = tid >= T::NCOL ? 1 : 0;
    const int col = act ? tid - ch * T::NCOL : 0;
    cy = col / T::E;
    cx = col - cy * T::E;
    own = col * CS + 8 * ch;
    xm = own - (cx > 0 ? CS : 0);
    xp = own + (cx < T::E - 1 ? CS : 0);
    ym = own - (cy > 0 ? T::E * CS : 0);
    yp = own + (cy < T::E - 1 ? T::E * CS : 0);
    const int x = x0 - H + cx, y = y0 - H + cy;
    gxy = legs::wrapmod(x, d.nx) + legs::wrapmod(y, d.ny) * d.nx;
    gz = legs::wrapmod(z0 - 4 + 8 * ch, d.nz);
    out = act && cx >= H && cx < H + BO && cy >= H && cy < H + BO && x < d.nx && y < d.ny;
  }
  __device__ __forceinline__ void load(Dims d, const float* __restrict__ f, float2 (&v)[4]) const {
    const int pst = d.nx * d.ny;
    float t[8];
    int z = gz;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      t[k] = __ldg(f + (size_t)z * pst + gxy);
      z = z + 1 == d.nz ? 0 : z + 1;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = make_float2(t[2 * k], t[2 * k + 1]);
  }
  // the half column's outputs: its upper half for ch = 0, its lower half for ch = 1
  __device__ __forceinline__ void store(Dims d, float* __restrict__ f, int z0, const float2 (&v)[4]) const {
    if (!out) return;
    const int pst = d.nx * d.ny;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int z = z0 + 4 * ch + k;
      const float2 p = ch ? v[k / 2] : v[2 + k / 2];
      if (z < d.nz) f[(size_t)z * pst + gxy] = k & 1 ? p.y : p.x;
    }
  }
  __device__ __forceinline__ void put(float* S, const float2 (&v)[4]) const {
    if (!act) return;
    float4* const p = reinterpret_cast<float4*>(S + own);
    p[0] = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
    p[1] = make_float4(v[2].x, v[2].y, v[3].x, v[3].y);
  }
  // lap_sum of the half column's cells; c: their values
  __device__ __forceinline__ void lap(const float* S, const float2 (&c)[4], float2 (&s)[4]) const {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float4 a = *reinterpret_cast<const float4*>(S + xm + 4 * h);
      const float4 b = *reinterpret_cast<const float4*>(S + xp + 4 * h);
      const float4 e = *reinterpret_cast<const float4*>(S + ym + 4 * h);
      const float4 g = *reinterpret_cast<const float4*>(S + yp + 4 * h);
      s[2 * h] = p_add(p_add(make_float2(a.x, a.y), make_float2(b.x, b.y)),
                       p_add(make_float2(e.x, e.y), make_float2(g.x, g.y)));
      s[2 * h + 1] = p_add(p_add(make_float2(a.z, a.w), make_float2(b.z, b.w)),
                           p_add(make_float2(e.z, e.w), make_float2(g.z, g.w)));
    }
    const float lo = ch ? S[own - 1] : c[0].x, hi = ch ? c[3].y : S[own + 8];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float zm = k ? c[k - 1].y : lo, zp = k < 3 ? c[k + 1].x : hi;
      s[k] = p_add(s[k], make_float2(t_fma(-6.f, c[k].x, zm), t_fma(-6.f, c[k].y, c[k].x)));
      s[k] = make_float2(t_add(s[k].x, c[k].y), t_add(s[k].y, zp));
    }
  }
};

template <int V>
__global__ void __launch_bounds__(BlockTile<V + 1>::NT)
k_block_down(Dims d, const float* __restrict__ r, float* __restrict__ e_out, float* __restrict__ rc, BlockCoef cf) {
  constexpr int H = V + 1;
  using T = BlockTile<H>;
  __shared__ __align__(16) float sm[2 * T::PLANE];
  const int x0 = blockIdx.x * BO, y0 = blockIdx.y * BO, z0 = blockIdx.z * BO;
  BlockPos<H> P;
  P.init(d, x0, y0, z0);
  float2 rv[4], e[4], dd[4];
  P.load(d, r, rv);
#pragma unroll
  for (int k = 0; k < 4; ++k) dd[k] = e[k] = p_mul(bcast(cf.a[0]), rv[k]);
  P.put(sm, e);
  __syncthreads();
#pragma unroll 1
  for (int s = 1; s <= V; ++s) {
    const float2 a = bcast(cf.a[s]), mb = bcast(cf.mb[s]), c1 = bcast(cf.c1[s]);
    float2 sn[4], w[4];
    P.lap(sm + (s & 1 ? 0 : T::PLANE), e, sn);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      w[k] = p_fma(mb, sn[k], p_mul(a, rv[k]));   // s = V: r - A e (a = 1)
      if (s < V) {
        dd[k] = p_fma(c1, dd[k], w[k]);
        w[k] = e[k] = p_add(e[k], dd[k]);
      }
    }
    P.put(sm + (s & 1 ? T::PLANE : 0), w);
    __syncthreads();
  }
  P.store(d, e_out, z0, e);
  // coarse outputs: z weights, then y, then x
  const int q = threadIdx.x;
  const int I = q & 3, J = q >> 2 & 3, K = q >> 4;
  const int X = (x0 >> 1) + I, Y = (y0 >> 1) + J, Z = (z0 >> 1) + K;
  if (q >= 64 || X >= d.nx / 2 || Y >= d.ny / 2 || Z >= d.nz / 2) return;
  const float* const S = sm + (V & 1 ? T::PLANE : 0) + ((H + 2 * J - 1) * T::E + H + 2 * I - 1) * CS + 2 * K + 3;
  float yv[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    float zv[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const float* const c = S + (b * T::E + a) * CS;
      zv[b] = fw3z(c[0], c[1], c[2]);
    }
    yv[a] = fw3(zv[0], zv[1], zv[2]);
  }
  rc[((size_t)Z * (d.ny / 2) + Y) * (d.nx / 2) + X] = fw3(yv[0], yv[1], yv[2]);
}

template <int V>
__global__ void __launch_bounds__(BlockTile<V>::NT)
k_block_up(Dims d, const float* __restrict__ e_in, const float* __restrict__ ec, const float* __restrict__ r,
           float* __restrict__ e_out, BlockCoef cf) {
  constexpr int H = V;
  using T = BlockTile<H>;
  __shared__ __align__(16) float sm[2 * T::PLANE];
  __shared__ float cs[BC * BC * BC];   // (y, x, z), z fastest
  const int x0 = blockIdx.x * BO, y0 = blockIdx.y * BO, z0 = blockIdx.z * BO;
  const int cnx = d.nx >> 1, cny = d.ny >> 1, cnz = d.nz >> 1;
  BlockPos<H> P;
  P.init(d, x0, y0, z0);
  float2 rv[4], e[4], dd[4];
  P.load(d, e_in, e);
  P.load(d, r, rv);
  for (int q = threadIdx.x; q < BC * BC * BC; q += T::NT) {
    const int i = q % BC, j = q / BC % BC, k = q / (BC * BC);
    const int X = legs::wrapmod((x0 >> 1) - 2 + i, cnx), Y = legs::wrapmod((y0 >> 1) - 2 + j, cny),
              Z = legs::wrapmod((z0 >> 1) - 2 + k, cnz);
    cs[(j * BC + i) * BC + k] = __ldg(ec + ((size_t)Z * cny + Y) * cnx + X);
  }
  __syncthreads();
  {
    // the column's coarse values (x, then y midpoints), then z midpoints
    const int xr = P.cx - H + 4, yr = P.cy - H + 4;
    const bool dx = xr & 1, dy = yr & 1;
    const float* const c = cs + ((yr >> 1) * BC + (xr >> 1)) * BC + 4 * P.ch;
    float v[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const float a = c[k], b = c[BC * BC + k];
      const float ax = dx ? half_sum(a, c[BC + k]) : a, bx = dx ? half_sum(b, c[BC * BC + BC + k]) : b;
      v[k] = dy ? half_sum(ax, bx) : ax;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      e[k] = p_add(e[k], make_float2(v[k], half_sum(v[k], v[k + 1])));
      dd[k] = bcast(0.f);
    }
  }
  P.put(sm, e);
  __syncthreads();
#pragma unroll 1
  for (int s = 0; s < V; ++s) {
    const float2 a = bcast(cf.a[s]), mb = bcast(cf.mb[s]), c1 = bcast(cf.c1[s]);
    float2 sn[4];
    P.lap(sm + (s & 1 ? T::PLANE : 0), e, sn);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      dd[k] = p_fma(c1, dd[k], p_fma(mb, sn[k], p_mul(a, rv[k])));
      e[k] = p_add(e[k], dd[k]);
    }
    if (s + 1 < V) {
      P.put(sm + (s & 1 ? 0 : T::PLANE), e);
      __syncthreads();
    }
  }
  P.store(d, e_out, z0, e);
}

BlockCoef block_coef(int degree, double h, const double* c1, const double* c2) {
  const legs::Coef L = legs::make_coef(c1, c2, degree, h);
  BlockCoef cf{};
  for (int i = 0; i < degree; ++i) cf.c1[i] = L.c1[i], cf.a[i] = L.a[i], cf.mb[i] = L.mb[i];
  cf.a[degree] = 1.f;
  cf.mb[degree] = -(float)(1.0 / (h * h));
  return cf;
}
dim3 block_grid(Dims d) { return dim3((d.nx + BO - 1) / BO, (d.ny + BO - 1) / BO, (d.nz + BO - 1) / BO); }

}  // namespace

cudaError_t launch_block_down(cudaStream_t st, int degree, Dims d, const float* r, float* e, float* rc, double h,
                              const double* c1, const double* c2) {
  const BlockCoef cf = block_coef(degree, h, c1, c2);
  const dim3 g = block_grid(d);
  switch (degree) {
    case 1: k_block_down<1><<<g, BlockTile<2>::NT, 0, st>>>(d, r, e, rc, cf); break;
    case 2: k_block_down<2><<<g, BlockTile<3>::NT, 0, st>>>(d, r, e, rc, cf); break;
    case 3: k_block_down<3><<<g, BlockTile<4>::NT, 0, st>>>(d, r, e, rc, cf); break;
    default: return cudaErrorInvalidValue;
  }
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_block_up(cudaStream_t st, int degree, Dims d, const float* e_in, const float* ec, const float* r,
                            float* e_out, double h, const double* c1, const double* c2) {
  const BlockCoef cf = block_coef(degree, h, c1, c2);
  const dim3 g = block_grid(d);
  switch (degree) {
    case 1: k_block_up<1><<<g, BlockTile<1>::NT, 0, st>>>(d, e_in, ec, r, e_out, cf); break;
    case 2: k_block_up<2><<<g, BlockTile<2>::NT, 0, st>>>(d, e_in, ec, r, e_out, cf); break;
    case 3: k_block_up<3><<<g, BlockTile<3>::NT, 0, st>>>(d, e_in, ec, r, e_out, cf); break;
    default: return cudaErrorInvalidValue;
  }
  note_launch();
  return cudaGetLastError();
}

}  // namespace gbmg
