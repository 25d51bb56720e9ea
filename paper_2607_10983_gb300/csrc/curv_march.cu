// Weighted-Jacobi sweep and residual of the curvilinear operator (Sec. 4.3) on levels
// above 32^3, FP32: z-marching tiles of packed row pairs (march.cuh), one operator form
// per kernel: M, M^T, or the symmetric variant S.
//
// What bounds it: a sweep moves 44 bytes per cell (e, B, r, J, D in; e out).  The form it
// replaces, one cell per thread with every neighbour read from shared memory through the
// operator templates, issued about 310 instructions and 66 shared wavefronts per 32 cells
// and sat at 0.46 of the copy bandwidth.  Here the differences D_b = u(+b) - u(-b) are
// formed once per cell instead of once per face and tangent, the y and z neighbours come
// from registers, and the diagonal D is read instead of formed.
//
// Rounding: every cell's operations are those of the operator templates of
// curv_kernels.cu in the same order (products fused the way the compiler fuses them
// there, made explicit), so both give the same bits.  Halves and quarters are exact, so B
// is summed instead of averaged over a face and the whole sum is 8 times the operator.
#include <cstdint>
#include <type_traits>

#include "march.cuh"

namespace gbmg {

namespace {

using namespace march;

__device__ __forceinline__ float2 p_neg(float2 a) { return make_float2(-a.x, -a.y); }
// S1 d1 - S2 d2, the second product rounded first
__device__ __forceinline__ float2 p_dif(float2 s1, float2 d1, float2 s2, float2 d2) {
  return p_fma(s1, d1, p_neg(p_mul(s2, d2)));
}

// The running state of a form for R packed rows (rows 0 .. R - 1, -1 and R its halo) and
// its step from plane t to t + 1: out[j] = 8 h^2 op(u) at plane t, row j, from the slots of
// planes t (c) and t + 1 (n).  WARM: only the state advances (planes before the run).

// ---- M.  8 F_a = (B_aa + B_aa') 4 (u' - u) + sum_{b != a} (B_ab + B_ab') (D_b + D_b'),
// the first product fused into the second, rounded one.
template <int R>
struct OpM {
  float2 um[R + 2], u0[R + 2];            // u at t - 1 and t
  float2 lm[R], l0[R], rm[R], r0[R];      // the same at x - 1 and x + 1
  float2 zz[R], xz[R], yz[R + 2];         // B at t
  float2 fz[R];                           // flux of the face below

  __device__ __forceinline__ void start(const View& V, int c, int n, float2 (&out)[R]) {
#pragma unroll
    for (int k = 0; k < R + 2; ++k) u0[k] = um[k] = V.at<FU>(c, k - 1, 0);
#pragma unroll
    for (int j = 0; j < R; ++j) {
      l0[j] = lm[j] = V.at<FU>(c, j, -1);
      r0[j] = rm[j] = V.at<FU>(c, j, 1);
      zz[j] = V.at<FZZ>(c, j, 0);
      xz[j] = V.at<FXZ>(c, j, 0);
      yz[j + 1] = V.at<FYZ>(c, j, 0);
      fz[j] = bcast(0.f);
    }
    yz[0] = yz[R + 1] = bcast(0.f);
    step<true>(V, c, n, out);
  }

  template <bool WARM>
  __device__ __forceinline__ void step(const View& V, int c, int n, float2 (&out)[R]) {
    const float2 four = bcast(4.f);
    float2 u1[R + 2], l1[R], r1[R], zz1[R], xz1[R], yz1[R];
#pragma unroll
    for (int k = 0; k < R + 2; ++k) u1[k] = V.at<FU>(n, k - 1, 0);
#pragma unroll
    for (int j = 0; j < R; ++j) {
      l1[j] = V.at<FU>(n, j, -1);
      r1[j] = V.at<FU>(n, j, 1);
      zz1[j] = V.at<FZZ>(n, j, 0);
      xz1[j] = V.at<FXZ>(n, j, 0);
      yz1[j] = V.at<FYZ>(n, j, 0);
    }
    // z faces t | t + 1
    float2 fzp[R], dx0[R + 2], dy0[R];
#pragma unroll
    for (int j = 0; j < R; ++j) {
      dx0[j + 1] = p_sub(r0[j], l0[j]);
      dy0[j] = p_sub(u0[j + 2], u0[j]);
      const float2 dx1 = p_sub(r1[j], l1[j]), dy1 = p_sub(u1[j + 2], u1[j]);
      const float2 f = p_fma(p_mul(four, p_add(zz[j], zz1[j])), p_sub(u1[j + 1], u0[j + 1]),
                             p_mul(p_add(xz[j], xz1[j]), p_add(dx0[j + 1], dx1)));
      fzp[j] = p_fma(p_add(yz[j + 1], yz1[j]), p_add(dy0[j], dy1), f);
    }
    if (!WARM) {
      const float2 ll = V.at<FU>(c, -1, -1), lh = V.at<FU>(c, R, -1);
      const float2 rl = V.at<FU>(c, -1, 1), rh = V.at<FU>(c, R, 1);
      dx0[0] = p_sub(rl, ll);
      dx0[R + 1] = p_sub(rh, lh);
      float2 dz[R + 2], xy[R + 2], yy[R + 2];
#pragma unroll
      for (int k = 0; k < R + 2; ++k) {
        dz[k] = p_sub(u1[k], um[k]);
        xy[k] = V.at<FXY>(c, k - 1, 0);
        yy[k] = V.at<FYY>(c, k - 1, 0);
      }
      // x faces: right minus left
#pragma unroll
      for (int j = 0; j < R; ++j) {
        const float2 xx = V.at<FXX>(c, j, 0);
        const float2 dyl = p_sub(j == R - 1 ? lh : l0[j + 1], j ? l0[j - 1] : ll);
        const float2 dyr = p_sub(j == R - 1 ? rh : r0[j + 1], j ? r0[j - 1] : rl);
        const float2 dzl = p_sub(l1[j], lm[j]), dzr = p_sub(r1[j], rm[j]);
        float2 f = p_fma(p_mul(four, p_add(xx, V.at<FXX>(c, j, 1))), p_sub(r0[j], u0[j + 1]),
                         p_mul(p_add(xy[j + 1], V.at<FXY>(c, j, 1)), p_add(dy0[j], dyr)));
        f = p_fma(p_add(xz[j], V.at<FXZ>(c, j, 1)), p_add(dz[j + 1], dzr), f);
        float2 g = p_fma(p_mul(four, p_add(xx, V.at<FXX>(c, j, -1))), p_sub(u0[j + 1], l0[j]),
                         p_mul(p_add(xy[j + 1], V.at<FXY>(c, j, -1)), p_add(dy0[j], dyl)));
        g = p_fma(p_add(xz[j], V.at<FXZ>(c, j, -1)), p_add(dz[j + 1], dzl), g);
        out[j] = p_sub(f, g);
      }
      // y faces between rows k - 1 and k
      float2 fy[R + 1];
#pragma unroll
      for (int k = 0; k < R + 1; ++k) {
        const float2 f = p_fma(p_mul(four, p_add(yy[k], yy[k + 1])), p_sub(u0[k + 1], u0[k]),
                               p_mul(p_add(xy[k], xy[k + 1]), p_add(dx0[k], dx0[k + 1])));
        fy[k] = p_fma(p_add(yz[k], yz[k + 1]), p_add(dz[k], dz[k + 1]), f);
      }
#pragma unroll
      for (int j = 0; j < R; ++j) out[j] = p_add(p_add(out[j], p_sub(fy[j + 1], fy[j])), p_sub(fzp[j], fz[j]));
    }
#pragma unroll
    for (int k = 0; k < R + 2; ++k) {
      um[k] = u0[k];
      u0[k] = u1[k];
    }
#pragma unroll
    for (int j = 0; j < R; ++j) {
      lm[j] = l0[j];
      l0[j] = l1[j];
      rm[j] = r0[j];
      r0[j] = r1[j];
      zz[j] = zz1[j];
      xz[j] = xz1[j];
      yz[j + 1] = yz1[j];
      fz[j] = fzp[j];
    }
    yz[0] = V.at<FYZ>(n, -1, 0);
    yz[R + 1] = V.at<FYZ>(n, R, 0);
  }
  __device__ __forceinline__ float2 centre(int j) const { return u0[j + 1]; }
};

// ---- M^T.  With q_ab(c) = (B_ab(c) + B_ab(c + a)) (u(c) - u(c + a)),
//   8 M^T u = sum_a 4 [q_aa(j - a) - q_aa(j)]
//           + sum_{b != a} [q_ab(j - b) - q_ab(j + b)] + [q_ab(j - a - b) - q_ab(j - a + b)],
// the first product of each bracket fused into the difference.
template <int R>
struct OpT {
  float2 u0[R + 2], l0[R + 2], r0[R + 2];  // u at t with its x neighbours
  float2 zz[R], xzl[R], xzr[R], yz[R + 2];  // B at t
  float2 zs[R], zd[R];                     // factors of q_zz on the face below
  float2 zxm[R], zym[R];                   // the zx and zy brackets of the face below
  // factors (S, d) of the xz faces right and left and of the yz faces, planes t - 1 and t
  float2 xrs[2][R], xrd[2][R], xls[2][R], xld[2][R], yzs[2][R + 1], yzd[2][R + 1];

  __device__ __forceinline__ void start(const View& V, int c, int n, float2 (&out)[R]) {
    const float2 Z = bcast(0.f);
#pragma unroll
    for (int k = 0; k < R + 2; ++k) u0[k] = l0[k] = r0[k] = yz[k] = Z;
#pragma unroll
    for (int j = 0; j < R; ++j) {
      zz[j] = xzl[j] = xzr[j] = zs[j] = zd[j] = zxm[j] = zym[j] = Z;
      xrs[0][j] = xrd[0][j] = xls[0][j] = xld[0][j] = xrs[1][j] = xrd[1][j] = xls[1][j] = xld[1][j] = Z;
    }
#pragma unroll
    for (int k = 0; k < R + 1; ++k) yzs[0][k] = yzd[0][k] = yzs[1][k] = yzd[1][k] = Z;
    step<true>(V, c, c, out);
    step<true>(V, c, n, out);
  }

  template <bool WARM>
  __device__ __forceinline__ void step(const View& V, int c, int n, float2 (&out)[R]) {
    const float2 four = bcast(4.f);
    float2 u1[R + 2], l1[R + 2], r1[R + 2], yz1[R + 2], xzl1[R], xzr1[R], zz1[R];
#pragma unroll
    for (int k = 0; k < R + 2; ++k) {
      u1[k] = V.at<FU>(n, k - 1, 0);
      l1[k] = V.at<FU>(n, k - 1, -1);
      r1[k] = V.at<FU>(n, k - 1, 1);
      yz1[k] = V.at<FYZ>(n, k - 1, 0);
    }
    float2 xrs1[R], xrd1[R], xls1[R], xld1[R], yzs1[R + 1], yzd1[R + 1];
#pragma unroll
    for (int j = 0; j < R; ++j) {
      zz1[j] = V.at<FZZ>(n, j, 0);
      xzl1[j] = V.at<FXZ>(n, j, -1);
      xzr1[j] = V.at<FXZ>(n, j, 1);
      const float2 xz1 = V.at<FXZ>(n, j, 0);
      xrs1[j] = p_add(xz1, xzr1[j]);
      xrd1[j] = p_sub(u1[j + 1], r1[j + 1]);
      xls1[j] = p_add(xzl1[j], xz1);
      xld1[j] = p_sub(l1[j + 1], u1[j + 1]);
    }
#pragma unroll
    for (int k = 0; k < R + 1; ++k) {
      yzs1[k] = p_add(yz1[k], yz1[k + 1]);
      yzd1[k] = p_sub(u1[k], u1[k + 1]);
    }
    // z faces t | t + 1
    float2 zsn[R], zdn[R], zxn[R], zyn[R], qs[R + 2], qd[R + 2];
#pragma unroll
    for (int k = 0; k < R + 2; ++k) {
      qs[k] = p_add(yz[k], yz1[k]);
      qd[k] = p_sub(u0[k], u1[k]);
    }
#pragma unroll
    for (int j = 0; j < R; ++j) {
      zsn[j] = p_add(zz[j], zz1[j]);
      zdn[j] = qd[j + 1];
      zxn[j] = p_dif(p_add(xzl[j], xzl1[j]), p_sub(l0[j + 1], l1[j + 1]), p_add(xzr[j], xzr1[j]),
                     p_sub(r0[j + 1], r1[j + 1]));
      zyn[j] = p_dif(qs[j], qd[j], qs[j + 2], qd[j + 2]);
    }
    if (!WARM) {
      // faces of the xy plane: x faces right and left of rows -1 .. R, y faces of columns
      // x - 1 and x + 1
      float2 xy[R + 2], xyl[R + 2], xyr[R + 2], yy[R + 2];
#pragma unroll
      for (int k = 0; k < R + 2; ++k) {
        xy[k] = V.at<FXY>(c, k - 1, 0);
        xyl[k] = V.at<FXY>(c, k - 1, -1);
        xyr[k] = V.at<FXY>(c, k - 1, 1);
        yy[k] = V.at<FYY>(c, k - 1, 0);
      }
      float2 yx[R + 1], ys[R + 1], yd[R + 1];
#pragma unroll
      for (int k = 0; k < R + 1; ++k) {
        yx[k] = p_dif(p_add(xyl[k], xyl[k + 1]), p_sub(l0[k], l0[k + 1]), p_add(xyr[k], xyr[k + 1]),
                      p_sub(r0[k], r0[k + 1]));
        ys[k] = p_add(yy[k], yy[k + 1]);
        yd[k] = p_sub(u0[k], u0[k + 1]);
      }
#pragma unroll
      for (int j = 0; j < R; ++j) {
        // a = x
        const float2 xx = V.at<FXX>(c, j, 0);
        float2 o = p_mul(four, p_dif(p_add(V.at<FXX>(c, j, -1), xx), p_sub(l0[j + 1], u0[j + 1]),
                                     p_add(xx, V.at<FXX>(c, j, 1)), p_sub(u0[j + 1], r0[j + 1])));
        const float2 xy1 = p_dif(p_add(xy[j], xyr[j]), p_sub(u0[j], r0[j]), p_add(xy[j + 2], xyr[j + 2]),
                                 p_sub(u0[j + 2], r0[j + 2]));
        const float2 xy2 = p_dif(p_add(xyl[j], xy[j]), p_sub(l0[j], u0[j]), p_add(xyl[j + 2], xy[j + 2]),
                                 p_sub(l0[j + 2], u0[j + 2]));
        o = p_add(o, p_add(xy1, xy2));
        o = p_add(o, p_add(p_dif(xrs[0][j], xrd[0][j], xrs1[j], xrd1[j]),
                           p_dif(xls[0][j], xld[0][j], xls1[j], xld1[j])));
        // a = y
        o = p_fma(four, p_dif(ys[j], yd[j], ys[j + 1], yd[j + 1]), o);
        o = p_add(o, p_add(yx[j + 1], yx[j]));
        o = p_add(o, p_add(p_dif(yzs[0][j + 1], yzd[0][j + 1], yzs1[j + 1], yzd1[j + 1]),
                           p_dif(yzs[0][j], yzd[0][j], yzs1[j], yzd1[j])));
        // a = z
        o = p_fma(four, p_dif(zs[j], zd[j], zsn[j], zdn[j]), o);
        o = p_add(o, p_add(zxn[j], zxm[j]));
        out[j] = p_add(o, p_add(zyn[j], zym[j]));
      }
    }
#pragma unroll
    for (int k = 0; k < R + 2; ++k) {
      u0[k] = u1[k];
      l0[k] = l1[k];
      r0[k] = r1[k];
      yz[k] = yz1[k];
    }
#pragma unroll
    for (int j = 0; j < R; ++j) {
      zz[j] = zz1[j];
      xzl[j] = xzl1[j];
      xzr[j] = xzr1[j];
      zs[j] = zsn[j];
      zd[j] = zdn[j];
      zxm[j] = zxn[j];
      zym[j] = zyn[j];
      xrs[0][j] = xrs[1][j];
      xrd[0][j] = xrd[1][j];
      xls[0][j] = xls[1][j];
      xld[0][j] = xld[1][j];
      xrs[1][j] = xrs1[j];
      xrd[1][j] = xrd1[j];
      xls[1][j] = xls1[j];
      xld[1][j] = xld1[j];
    }
#pragma unroll
    for (int k = 0; k < R + 1; ++k) {
      yzs[0][k] = yzs[1][k];
      yzd[0][k] = yzd[1][k];
      yzs[1][k] = yzs1[k];
      yzd[1][k] = yzd1[k];
    }
  }
  __device__ __forceinline__ float2 centre(int j) const { return u0[j + 1]; }
};

// ---- S.  Faces (B_aa + B_aa') and edges: the coefficient of the ab-edge is the sum over
// its four cells, first along a, then along b; per pair a < b the four edges k = 0 .. 3
// (base -a for k & 1, -b for k & 2) couple to the neighbour across them, signs + - - +.
template <int R>
struct OpS {
  float2 um[R + 2], u0[R + 2];                    // u at t - 1, t
  float2 lm[R], rm[R], l0[R + 2], r0[R + 2];
  float2 zz[R], zs[R];                            // B_zz at t, face sum below
  float2 axl[R], axr[R], ay[R + 1];               // x and y sums of xz, yz at t
  float2 cxl[R], cxr[R], cy[R + 1];               // edge sums t - 1 | t

  __device__ __forceinline__ void start(const View& V, int c, int n, float2 (&out)[R]) {
    const float2 Z = bcast(0.f);
#pragma unroll
    for (int k = 0; k < R + 2; ++k) um[k] = u0[k] = l0[k] = r0[k] = Z;
#pragma unroll
    for (int j = 0; j < R; ++j) lm[j] = rm[j] = zz[j] = zs[j] = axl[j] = axr[j] = cxl[j] = cxr[j] = Z;
#pragma unroll
    for (int k = 0; k < R + 1; ++k) ay[k] = cy[k] = Z;
    step<true>(V, c, c, out);
    step<true>(V, c, n, out);
  }

  template <bool WARM>
  __device__ __forceinline__ void step(const View& V, int c, int n, float2 (&out)[R]) {
    const float2 four = bcast(4.f);
    float2 u1[R + 2], l1[R + 2], r1[R + 2], yz1[R + 2];
#pragma unroll
    for (int k = 0; k < R + 2; ++k) {
      u1[k] = V.at<FU>(n, k - 1, 0);
      l1[k] = V.at<FU>(n, k - 1, -1);
      r1[k] = V.at<FU>(n, k - 1, 1);
      yz1[k] = V.at<FYZ>(n, k - 1, 0);
    }
    float2 zz1[R], axl1[R], axr1[R], ay1[R + 1], zsn[R], cxln[R], cxrn[R], cyn[R + 1];
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const float2 xz1 = V.at<FXZ>(n, j, 0);
      zz1[j] = V.at<FZZ>(n, j, 0);
      axl1[j] = p_add(V.at<FXZ>(n, j, -1), xz1);
      axr1[j] = p_add(xz1, V.at<FXZ>(n, j, 1));
      zsn[j] = p_add(zz[j], zz1[j]);
      cxln[j] = p_add(axl[j], axl1[j]);
      cxrn[j] = p_add(axr[j], axr1[j]);
    }
#pragma unroll
    for (int k = 0; k < R + 1; ++k) {
      ay1[k] = p_add(yz1[k], yz1[k + 1]);
      cyn[k] = p_add(ay[k], ay1[k]);
    }
    if (!WARM) {
      float2 xl[R + 2], xr[R + 2], yy[R + 2];
#pragma unroll
      for (int k = 0; k < R + 2; ++k) {
        const float2 xy = V.at<FXY>(c, k - 1, 0);
        xl[k] = p_add(V.at<FXY>(c, k - 1, -1), xy);
        xr[k] = p_add(xy, V.at<FXY>(c, k - 1, 1));
        yy[k] = V.at<FYY>(c, k - 1, 0);
      }
#pragma unroll
      for (int j = 0; j < R; ++j) {
        const float2 u = u0[j + 1];
        const float2 xx = V.at<FXX>(c, j, 0);
        // in units of 1/2 for the faces and 1/8 for the edges
        float2 o = p_dif(p_add(xx, V.at<FXX>(c, j, 1)), p_sub(r0[j + 1], u), p_add(V.at<FXX>(c, j, -1), xx),
                         p_sub(u, l0[j + 1]));
        o = p_add(o, p_dif(p_add(yy[j + 1], yy[j + 2]), p_sub(u0[j + 2], u), p_add(yy[j], yy[j + 1]),
                           p_sub(u, u0[j])));
        o = p_add(o, p_dif(zsn[j], p_sub(u1[j + 1], u), zs[j], p_sub(u, um[j + 1])));
        // xy edges: bases (0, 0), (-x, 0), (0, -y), (-x, -y)
        float2 e = p_mul(p_add(xr[j + 1], xr[j + 2]), p_sub(r0[j + 2], u));
        e = p_fma(p_neg(p_add(xl[j + 1], xl[j + 2])), p_sub(l0[j + 2], u), e);
        e = p_fma(p_neg(p_add(xr[j], xr[j + 1])), p_sub(r0[j], u), e);
        e = p_fma(p_add(xl[j], xl[j + 1]), p_sub(l0[j], u), e);
        o = p_fma(four, o, e);
        // xz edges
        e = p_mul(cxrn[j], p_sub(r1[j + 1], u));
        e = p_fma(p_neg(cxln[j]), p_sub(l1[j + 1], u), e);
        e = p_fma(p_neg(cxr[j]), p_sub(rm[j], u), e);
        e = p_fma(cxl[j], p_sub(lm[j], u), e);
        o = p_add(o, e);
        // yz edges
        e = p_mul(cyn[j + 1], p_sub(u1[j + 2], u));
        e = p_fma(p_neg(cyn[j]), p_sub(u1[j], u), e);
        e = p_fma(p_neg(cy[j + 1]), p_sub(um[j + 2], u), e);
        e = p_fma(cy[j], p_sub(um[j], u), e);
        out[j] = p_add(o, e);
      }
    }
#pragma unroll
    for (int k = 0; k < R + 2; ++k) {
      um[k] = u0[k];
      u0[k] = u1[k];
    }
#pragma unroll
    for (int j = 0; j < R; ++j) {
      lm[j] = l0[j + 1];
      rm[j] = r0[j + 1];
      zz[j] = zz1[j];
      zs[j] = zsn[j];
      axl[j] = axl1[j];
      axr[j] = axr1[j];
      cxl[j] = cxln[j];
      cxr[j] = cxrn[j];
    }
#pragma unroll
    for (int k = 0; k < R + 2; ++k) {
      l0[k] = l1[k];
      r0[k] = r1[k];
    }
#pragma unroll
    for (int k = 0; k < R + 1; ++k) {
      ay[k] = ay1[k];
      cy[k] = cyn[k];
    }
  }
  __device__ __forceinline__ float2 centre(int j) const { return u0[j + 1]; }
};

enum { SWEEP = 0, RESID = 1 };

// SWEEP: out = e + omega (J r h^2 - h^2 op(e)) / D; RESID: out = r - op(e) / (h^2 J).
template <int MODE, class OP, int R, int MINB, int UN>
__global__ void __launch_bounds__(256 / R, MINB)
k_curv_march(Dims d, Fields P, const float* __restrict__ r, const float* __restrict__ J, const float* __restrict__ D,
             float* __restrict__ out, float omega, float h2, float inv_h2, int zc) {
  constexpr int NT = 256 / R;
  extern __shared__ __align__(16) float smf[];
  const int lane = threadIdx.x & 31, row = (threadIdx.x >> 5) * R;
  const int x0 = blockIdx.x * MX, y0 = blockIdx.y * MY, z0 = blockIdx.z * zc;
  const int zend = min(z0 + zc, d.nz);
  const long long pst = (long long)d.nx * d.ny;
  Copier<NT> C;
  C.init(d, P, x0, y0);
  const unsigned sbase = (unsigned)__cvta_generic_to_shared(smf);
  auto issue = [&](int z, int slot) {
    const int zw = z < 0 ? z + d.nz : (z >= d.nz ? z - d.nz : z);
    C.issue(P, zw * pst, sbase + (unsigned)(slot * SLOT) * 4u);
    cp_commit();
  };
  // the thread's cells k: row k % R of the low (k < R) or high lane
  const int x = x0 + lane;
  bool own[2 * R];
  int off[2 * R];
#pragma unroll
  for (int k = 0; k < 2 * R; ++k) {
    const int y = y0 + row + k % R + (k / R) * 8;
    own[k] = x < d.nx && y < d.ny;
    off[k] = own[k] ? y * d.nx + x : 0;
  }
  float rn[2 * R], Jn[2 * R], Dn[2 * R];
#pragma unroll
  for (int k = 0; k < 2 * R; ++k) rn[k] = 0.f, Jn[k] = Dn[k] = 1.f;
  auto fetch = [&](int z) {
    const long long zo = z * pst;
#pragma unroll
    for (int k = 0; k < 2 * R; ++k) {
      if (!own[k]) continue;
      rn[k] = __ldg(r + zo + off[k]);
      Jn[k] = __ldg(J + zo + off[k]);
      if (MODE == SWEEP) Dn[k] = __ldg(D + zo + off[k]);
    }
  };
  const View V(smf, row, lane);
  issue(z0 - 1, 0);
  issue(z0, 1);
  fetch(z0);
  cp_wait_all();
  __syncthreads();
  issue(z0 + 1, 2);
  OP S;
  float2 o2[R];
  S.start(V, 0, SLOT, o2);
  // the slots of planes t and t + 1 and the one to fill rotate; UN = 3: three steps per turn,
  // so that the slot offsets are constants and the state's planes are renamed, not moved
  int t = z0, sc = 1, sn = 2, sf = 0;
  while (t < zend) {
#pragma unroll
    for (int s = 0; s < UN; ++s, ++t) {
      if (s > 0 && t >= zend) break;
      if (UN == 3) sc = (s + 1) % 3, sn = (s + 2) % 3, sf = s;
      cp_wait_all();
      __syncthreads();
      if (t + 1 < zend) issue(t + 2, sf);
      float rc[2 * R], Jc[2 * R], Dc[2 * R];
#pragma unroll
      for (int k = 0; k < 2 * R; ++k) {
        rc[k] = rn[k];
        Jc[k] = Jn[k];
        Dc[k] = Dn[k];
      }
      if (t + 1 < zend) fetch(t + 1);
      float2 uc[R];
#pragma unroll
      for (int j = 0; j < R; ++j) uc[j] = S.centre(j);
      S.template step<false>(V, sc * SLOT, sn * SLOT, o2);
      float* const oz = out + t * pst;
#pragma unroll
      for (int k = 0; k < 2 * R; ++k) {
        const float m = 0.125f * (k / R ? o2[k % R].y : o2[k % R].x);
        const float u = k / R ? uc[k % R].y : uc[k % R].x;
        float v;
        if (MODE == SWEEP) v = __fmaf_rn(omega, __fdiv_rn(__fmaf_rn(__fmul_rn(Jc[k], rc[k]), h2, -m), Dc[k]), u);
        else v = __fsub_rn(rc[k], __fdiv_rn(__fmul_rn(m, inv_h2), Jc[k]));
        if (own[k]) oz[off[k]] = v;
      }
      if (UN != 3) {
        const int q = sc;
        sc = sn;
        sn = sf;
        sf = q;
      }
    }
  }
}

template <int MODE, class OP, int R, int MINB, int UN>
cudaError_t launch(cudaStream_t st, Dims d, const CurvCoef& cf, const float* r, const float* e, float* out,
                   float omega) {
  constexpr size_t sm = 3 * (size_t)SLOT * sizeof(float);
  static DeviceSet done{0};
  const cudaError_t err = allow_smem(done, k_curv_march<MODE, OP, R, MINB, UN>, sm);
  if (err != cudaSuccess) return err;
  Fields P;
  P.p[FU] = e;
  for (int k = 0; k < 6; ++k) P.p[FXX + k] = cf.B[k];
  const int zc = march_zchunk(d, MINB * 152);
  k_curv_march<MODE, OP, R, MINB, UN><<<march_grid(d, zc), 256 / R, sm, st>>>(d, P, r, cf.J, cf.D, out, omega, cf.h2,
                                                                         1.0f / cf.h2, zc);
  note_launch();
  return cudaGetLastError();
}

// Rows per thread, CTAs per SM and unrolling of the plane loop, measured at 256^3 (sweep /
// residual, us; one row in 256 threads, 2 or 3 CTAs | two rows in 128 threads, 4, 3, 2 CTAs):
//   M    162 / 158 | 219 / 129 (spills), 138 / 130 (unrolled by three; 142 / 136 rolled), -
//   M^T  186 / 176 | -, 382 / 274 (spills), 179 / 169 (238 / 176 unrolled)
//   S    175 / 166 | -, 146 / 138, 169 / 161
// against 211 / 195, 220 / 218 and 234 / 220 for the one-cell tiles of curv_kernels.cu.
template <int MODE>
cudaError_t launch_form(cudaStream_t st, Dims d, const CurvCoef& cf, const float* r, const float* e, float* out,
                        int form, float omega) {
  switch (form) {
    case 0: return launch<MODE, OpM<2>, 2, 3, 3>(st, d, cf, r, e, out, omega);
    case 1: return launch<MODE, OpT<2>, 2, 2, 1>(st, d, cf, r, e, out, omega);
    default: return launch<MODE, OpS<2>, 2, 3, 1>(st, d, cf, r, e, out, omega);
  }
}
}  // namespace

bool curv_march_ok(Dims d, const CurvCoef& cf, const float* u) {
  uintptr_t p = (uintptr_t)u;
  for (int k = 0; k < 6; ++k) p |= (uintptr_t)cf.B[k];
  return d.nx % 4 == 0 && (p & 15) == 0 && (long long)d.nx * d.ny < (1ll << 31);
}
cudaError_t launch_march_jacobi(cudaStream_t st, Dims d, const CurvCoef& cf, const float* r, const float* e_in,
                                float* e_out, int form, float omega) {
  return launch_form<SWEEP>(st, d, cf, r, e_in, e_out, form, omega);
}
cudaError_t launch_march_residual(cudaStream_t st, Dims d, const CurvCoef& cf, const float* r, const float* u,
                                  float* out, int form) {
  return launch_form<RESID>(st, d, cf, r, u, out, form, 0.f);
}

}  // namespace gbmg
