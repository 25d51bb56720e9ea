// One double-float defect-correction step of the curvilinear solve on the finest level
// (Sec. 3.2, 4.3), as a z-marching tile kernel of packed row pairs (march.cuh):
//   u' = u + e,  r = (b - op(u') / h^2) / J,  e1 = the first sweep of the next cycle,
// with the block sums of r^2 and, for a solve's first residual, of (b / J)^2.
//
// What bounds it: instruction issue.  A step moves 64 bytes per cell; the one-cell tile of
// curv_kernels.cu spent about 600 (M) to 900 (M^T) instructions per cell on it, and the
// update and the first sweep were passes of their own.  Here a difference of two
// double-float values is formed once per cell and face instead of once per product that
// uses it, and every operation is a packed FP32x2 one on two rows.
//
// Rounding: each cell's operations are those of df_face_flux / df_apply_MT / df_apply_S
// (curv_kernels.cu) in the same order, so the residual has the same bits.  B is summed,
// not averaged, and the whole sum is 8 times as large (exact).
#include <cstdint>

#include "march.cuh"

namespace gbmg {

namespace {

using namespace march;

constexpr int NT = 256;
constexpr int PU = 36, URO = (MY + 2) * PU;       // pitch and floats of the hi or lo plane of u
constexpr int SB = SLOT - f_off(1);               // floats of the B planes of a slot
constexpr int DSLOT = SB + 2 * URO;               // floats of a slot
constexpr int NPAIR = 18 * (MY + 2);              // x-pairs of the haloed plane (x0 - 2 .. x0 + 33)
constexpr int RAW = 3 * DSLOT;                    // staging: float4 phi pairs, then float2 e pairs
constexpr size_t kSmem = (size_t)(RAW + NPAIR * 6) * sizeof(float);

__device__ __forceinline__ float2 p_neg(float2 a) { return make_float2(-a.x, -a.y); }

// a - b of double-float values as an unnormalised pair (df_sub of curv_kernels.cu)
__device__ __forceinline__ DF2 p_df_sub(DF2 a, DF2 b) {
  DF2 d;
  d.hi = p_sub(a.hi, b.hi);
  const float2 bb = p_sub(d.hi, a.hi);
  d.lo = p_sub(p_sub(a.hi, p_sub(d.hi, bb)), p_add(b.hi, bb));
  d.lo = p_add(d.lo, p_sub(a.lo, b.lo));
  return d;
}
// acc += w v, acc -= w v (df_acc_prod)
__device__ __forceinline__ void acc_prod(PAcc& a, float2 w, const DF2& v) {
  const float2 p = p_mul(w, v.hi);
  const float2 pe = p_fma(w, v.hi, p_neg(p));
  a.add(p);
  a.c = p_add(a.c, p_fma(w, v.lo, pe));
}
__device__ __forceinline__ void acc_prod_neg(PAcc& a, float2 w, const DF2& v) {
  const float2 p = p_mul(w, v.hi);
  const float2 pe = p_fma(w, v.hi, p_neg(p));
  a.add_neg(p);
  a.c = p_sub(a.c, p_fma(w, v.lo, pe));
}

// The thread's view of a slot (offset s): B as in View, u as hi and lo planes.
struct DfView {
  View V;
  const float* u;
  __device__ __forceinline__ DfView(const float* sm, int row, int lane)
      : V(sm - f_off(1), row, lane), u(sm + SB + (row + 1) * PU + 2 + lane) {}
  template <int F>
  __device__ __forceinline__ float2 at(int s, int dr, int dx) const {
    return V.at<F>(s, dr, dx);
  }
  __device__ __forceinline__ DF2 U(int s, int dr, int dx) const {
    const float* q = u + s + dr * PU + dx;
    return DF2{make_float2(q[0], q[8 * PU]), make_float2(q[URO], q[URO + 8 * PU])};
  }
};

// ---- M
struct DfM {
  DF2 um[3], lm, rm;   // u at t - 1: rows -1 .. 1, x - 1, x + 1
  DF2 dx, dy;          // D_x, D_y of the cell at t
  PAcc fz;             // flux of the face below

  // 8 times the flux of a face: d = u' - u, (S1, p, p'), (S2, q, q') the two tangents
  static __device__ __forceinline__ PAcc flux(float2 Sa, const DF2& d, float2 S1, const DF2& p, const DF2& p2,
                                              float2 S2, const DF2& q, const DF2& q2) {
    const float2 wa = p_mul(bcast(4.f), Sa);
    PAcc f;
    f.s = p_mul(wa, d.hi);
    f.c = p_fma(wa, d.lo, p_fma(wa, d.hi, p_neg(f.s)));
    acc_prod(f, S1, p);
    acc_prod(f, S1, p2);
    acc_prod(f, S2, q);
    acc_prod(f, S2, q2);
    return f;
  }
  __device__ __forceinline__ PAcc z_face(const DfView& V, int c, int n, const DF2& u, const DF2& u1, const DF2& dx1,
                                         const DF2& dy1) const {
    return flux(p_add(V.at<FZZ>(c, 0, 0), V.at<FZZ>(n, 0, 0)), p_df_sub(u1, u),
                p_add(V.at<FXZ>(c, 0, 0), V.at<FXZ>(n, 0, 0)), dx, dx1,
                p_add(V.at<FYZ>(c, 0, 0), V.at<FYZ>(n, 0, 0)), dy, dy1);
  }
  __device__ __forceinline__ void start(const DfView& V, int c, int n) {
    lm = V.U(c, 0, -1);
    rm = V.U(c, 0, 1);
#pragma unroll
    for (int k = 0; k < 3; ++k) um[k] = V.U(c, k - 1, 0);
    dx = p_df_sub(rm, lm);
    dy = p_df_sub(um[2], um[0]);
    const DF2 dx1 = p_df_sub(V.U(n, 0, 1), V.U(n, 0, -1)), dy1 = p_df_sub(V.U(n, 1, 0), V.U(n, -1, 0));
    fz = z_face(V, c, n, um[1], V.U(n, 0, 0), dx1, dy1);
    dx = dx1;
    dy = dy1;
  }
  static __device__ __forceinline__ void face(PAcc& a, const PAcc& f, bool plus) {
    if (plus) {
      a.add(f.s);
      a.c = p_add(a.c, f.c);
    } else {
      a.add_neg(f.s);
      a.c = p_sub(a.c, f.c);
    }
  }
  // acc -= 8 h^2 M u at plane t
  __device__ __forceinline__ void step(const DfView& V, int c, int n, PAcc& acc) {
    const DF2 u = V.U(c, 0, 0);
    DF2 dz;
    {
      // x faces, right then left
      const float2 xx = V.at<FXX>(c, 0, 0), xy = V.at<FXY>(c, 0, 0), xz = V.at<FXZ>(c, 0, 0);
      const DF2 u1 = V.U(n, 0, 0);
      dz = p_df_sub(u1, um[1]);
      const DF2 r = V.U(c, 0, 1), r1 = V.U(n, 0, 1);
      DF2 dyn = p_df_sub(V.U(c, 1, 1), V.U(c, -1, 1)), dzn = p_df_sub(r1, rm);
      face(acc, flux(p_add(xx, V.at<FXX>(c, 0, 1)), p_df_sub(r, u), p_add(xy, V.at<FXY>(c, 0, 1)), dy, dyn,
                     p_add(xz, V.at<FXZ>(c, 0, 1)), dz, dzn), false);
      rm = r;
      const DF2 l = V.U(c, 0, -1), l1 = V.U(n, 0, -1);
      dyn = p_df_sub(V.U(c, 1, -1), V.U(c, -1, -1));
      dzn = p_df_sub(l1, lm);
      face(acc, flux(p_add(V.at<FXX>(c, 0, -1), xx), p_df_sub(u, l), p_add(V.at<FXY>(c, 0, -1), xy), dyn, dy,
                     p_add(V.at<FXZ>(c, 0, -1), xz), dzn, dz), true);
      lm = l;
    }
    {
      // y faces, upper then lower
      const float2 yy = V.at<FYY>(c, 0, 0), xy = V.at<FXY>(c, 0, 0), yz = V.at<FYZ>(c, 0, 0);
      const DF2 p = V.U(c, 1, 0);
      DF2 dxn = p_df_sub(V.U(c, 1, 1), V.U(c, 1, -1)), dzn = p_df_sub(V.U(n, 1, 0), um[2]);
      face(acc, flux(p_add(yy, V.at<FYY>(c, 1, 0)), p_df_sub(p, u), p_add(xy, V.at<FXY>(c, 1, 0)), dx, dxn,
                     p_add(yz, V.at<FYZ>(c, 1, 0)), dz, dzn), false);
      um[2] = p;
      const DF2 m = V.U(c, -1, 0);
      dxn = p_df_sub(V.U(c, -1, 1), V.U(c, -1, -1));
      dzn = p_df_sub(V.U(n, -1, 0), um[0]);
      face(acc, flux(p_add(V.at<FYY>(c, -1, 0), yy), p_df_sub(u, m), p_add(V.at<FXY>(c, -1, 0), xy), dxn, dx,
                     p_add(V.at<FYZ>(c, -1, 0), yz), dzn, dz), true);
      um[0] = m;
    }
    {
      const DF2 dx1 = p_df_sub(V.U(n, 0, 1), V.U(n, 0, -1)), dy1 = p_df_sub(V.U(n, 1, 0), V.U(n, -1, 0));
      const PAcc f = z_face(V, c, n, u, V.U(n, 0, 0), dx1, dy1);
      face(acc, f, false);
      face(acc, fz, true);
      fz = f;
      dx = dx1;
      dy = dy1;
      um[1] = u;
    }
  }
};

// ---- M^T
struct DfT {
  // z faces t - 1 | t: B sums and u differences (zz; xz at x - 1, x + 1; yz on rows -1, 1)
  float2 szz, sxl, sxr, sym, syp;
  DF2 dzz, dxl, dxr, dym, dyp;
  // plane t - 1: xz faces right and left, yz faces above and below the row
  float2 srm, slm, sum_, sdm;
  DF2 drm, dlm, dum, ddm;

  __device__ __forceinline__ void z_faces(const DfView& V, int c, int n) {
    szz = p_add(V.at<FZZ>(c, 0, 0), V.at<FZZ>(n, 0, 0));
    sxl = p_add(V.at<FXZ>(c, 0, -1), V.at<FXZ>(n, 0, -1));
    sxr = p_add(V.at<FXZ>(c, 0, 1), V.at<FXZ>(n, 0, 1));
    sym = p_add(V.at<FYZ>(c, -1, 0), V.at<FYZ>(n, -1, 0));
    syp = p_add(V.at<FYZ>(c, 1, 0), V.at<FYZ>(n, 1, 0));
    dzz = p_df_sub(V.U(c, 0, 0), V.U(n, 0, 0));
    dxl = p_df_sub(V.U(c, 0, -1), V.U(n, 0, -1));
    dxr = p_df_sub(V.U(c, 0, 1), V.U(n, 0, 1));
    dym = p_df_sub(V.U(c, -1, 0), V.U(n, -1, 0));
    dyp = p_df_sub(V.U(c, 1, 0), V.U(n, 1, 0));
  }
  __device__ __forceinline__ void plane_faces(const DfView& V, int c) {
    const float2 xz = V.at<FXZ>(c, 0, 0), yz = V.at<FYZ>(c, 0, 0);
    const DF2 u = V.U(c, 0, 0);
    srm = p_add(xz, V.at<FXZ>(c, 0, 1));
    slm = p_add(V.at<FXZ>(c, 0, -1), xz);
    sum_ = p_add(yz, V.at<FYZ>(c, 1, 0));
    sdm = p_add(V.at<FYZ>(c, -1, 0), yz);
    drm = p_df_sub(u, V.U(c, 0, 1));
    dlm = p_df_sub(V.U(c, 0, -1), u);
    dum = p_df_sub(u, V.U(c, 1, 0));
    ddm = p_df_sub(V.U(c, -1, 0), u);
  }
  __device__ __forceinline__ void start(const DfView& V, int c, int n) {
    z_faces(V, c, n);
    plane_faces(V, c);
  }
  __device__ __forceinline__ void step(const DfView& V, int c, int n, PAcc& acc) {
    const float2 four = bcast(4.f);
    const DF2 u = V.U(c, 0, 0);
    const float2 xz1 = V.at<FXZ>(n, 0, 0), yz1 = V.at<FYZ>(n, 0, 0);
    const DF2 u1 = V.U(n, 0, 0);
    DF2 dr, dl, du, dd;  // differences of plane t across the cell's faces
    {
      // a = x
      const float2 xx = V.at<FXX>(c, 0, 0);
      const DF2 l = V.U(c, 0, -1), r = V.U(c, 0, 1);
      dl = p_df_sub(l, u);
      dr = p_df_sub(u, r);
      acc_prod_neg(acc, p_mul(four, p_add(V.at<FXX>(c, 0, -1), xx)), dl);
      acc_prod(acc, p_mul(four, p_add(xx, V.at<FXX>(c, 0, 1))), dr);
      const float2 xym = V.at<FXY>(c, -1, 0), xyp = V.at<FXY>(c, 1, 0);
      const DF2 m = V.U(c, -1, 0), p = V.U(c, 1, 0);
      acc_prod_neg(acc, p_add(xym, V.at<FXY>(c, -1, 1)), p_df_sub(m, V.U(c, -1, 1)));
      acc_prod(acc, p_add(xyp, V.at<FXY>(c, 1, 1)), p_df_sub(p, V.U(c, 1, 1)));
      acc_prod_neg(acc, p_add(V.at<FXY>(c, -1, -1), xym), p_df_sub(V.U(c, -1, -1), m));
      acc_prod(acc, p_add(V.at<FXY>(c, 1, -1), xyp), p_df_sub(V.U(c, 1, -1), p));
      acc_prod_neg(acc, srm, drm);
      acc_prod(acc, p_add(xz1, V.at<FXZ>(n, 0, 1)), p_df_sub(u1, V.U(n, 0, 1)));
      acc_prod_neg(acc, slm, dlm);
      acc_prod(acc, p_add(V.at<FXZ>(n, 0, -1), xz1), p_df_sub(V.U(n, 0, -1), u1));
    }
    {
      // a = y
      const float2 yy = V.at<FYY>(c, 0, 0);
      const DF2 m = V.U(c, -1, 0), p = V.U(c, 1, 0);
      dd = p_df_sub(m, u);
      du = p_df_sub(u, p);
      acc_prod_neg(acc, p_mul(four, p_add(V.at<FYY>(c, -1, 0), yy)), dd);
      acc_prod(acc, p_mul(four, p_add(yy, V.at<FYY>(c, 1, 0))), du);
      const float2 xyl = V.at<FXY>(c, 0, -1), xyr = V.at<FXY>(c, 0, 1);
      const DF2 l = V.U(c, 0, -1), r = V.U(c, 0, 1);
      acc_prod_neg(acc, p_add(xyl, V.at<FXY>(c, 1, -1)), p_df_sub(l, V.U(c, 1, -1)));
      acc_prod(acc, p_add(xyr, V.at<FXY>(c, 1, 1)), p_df_sub(r, V.U(c, 1, 1)));
      acc_prod_neg(acc, p_add(V.at<FXY>(c, -1, -1), xyl), p_df_sub(V.U(c, -1, -1), l));
      acc_prod(acc, p_add(V.at<FXY>(c, -1, 1), xyr), p_df_sub(V.U(c, -1, 1), r));
      acc_prod_neg(acc, sum_, dum);
      acc_prod(acc, p_add(yz1, V.at<FYZ>(n, 1, 0)), p_df_sub(u1, V.U(n, 1, 0)));
      acc_prod_neg(acc, sdm, ddm);
      acc_prod(acc, p_add(V.at<FYZ>(n, -1, 0), yz1), p_df_sub(V.U(n, -1, 0), u1));
    }
    // a = z: the faces below are carried
    acc_prod_neg(acc, p_mul(four, szz), dzz);
    const DfT o = *this;
    z_faces(V, c, n);
    acc_prod(acc, p_mul(four, szz), dzz);
    acc_prod_neg(acc, sxl, dxl);
    acc_prod(acc, sxr, dxr);
    acc_prod_neg(acc, o.sxl, o.dxl);
    acc_prod(acc, o.sxr, o.dxr);
    acc_prod_neg(acc, sym, dym);
    acc_prod(acc, syp, dyp);
    acc_prod_neg(acc, o.sym, o.dym);
    acc_prod(acc, o.syp, o.dyp);
    const float2 xz = V.at<FXZ>(c, 0, 0), yz = V.at<FYZ>(c, 0, 0);
    srm = p_add(xz, V.at<FXZ>(c, 0, 1));
    slm = p_add(V.at<FXZ>(c, 0, -1), xz);
    sum_ = p_add(yz, V.at<FYZ>(c, 1, 0));
    sdm = p_add(V.at<FYZ>(c, -1, 0), yz);
    drm = dr;
    dlm = dl;
    dum = du;
    ddm = dd;
  }
};

// ---- S
struct DfS {
  DF2 um[3], lm, rm;           // u at t - 1: rows -1 .. 1, x - 1, x + 1
  float2 szz;                  // B_zz sum t - 1 | t
  float2 cl, cr, cd, cu;       // edge sums t - 1 | t: xz left and right, yz below and above

  __device__ __forceinline__ void edges(const DfView& V, int c, int n) {
    szz = p_add(V.at<FZZ>(c, 0, 0), V.at<FZZ>(n, 0, 0));
    const float2 x0 = V.at<FXZ>(c, 0, 0), x1 = V.at<FXZ>(n, 0, 0), y0 = V.at<FYZ>(c, 0, 0), y1 = V.at<FYZ>(n, 0, 0);
    cl = p_add(p_add(V.at<FXZ>(c, 0, -1), x0), p_add(V.at<FXZ>(n, 0, -1), x1));
    cr = p_add(p_add(x0, V.at<FXZ>(c, 0, 1)), p_add(x1, V.at<FXZ>(n, 0, 1)));
    cd = p_add(p_add(V.at<FYZ>(c, -1, 0), y0), p_add(V.at<FYZ>(n, -1, 0), y1));
    cu = p_add(p_add(y0, V.at<FYZ>(c, 1, 0)), p_add(y1, V.at<FYZ>(n, 1, 0)));
  }
  __device__ __forceinline__ void start(const DfView& V, int c, int n) {
    lm = V.U(c, 0, -1);
    rm = V.U(c, 0, 1);
#pragma unroll
    for (int k = 0; k < 3; ++k) um[k] = V.U(c, k - 1, 0);
    edges(V, c, n);
  }
  __device__ __forceinline__ void step(const DfView& V, int c, int n, PAcc& acc) {
    const float2 four = bcast(4.f);
    const DF2 u = V.U(c, 0, 0);
    const float2 xx = V.at<FXX>(c, 0, 0), yy = V.at<FYY>(c, 0, 0);
    acc_prod_neg(acc, p_mul(four, p_add(xx, V.at<FXX>(c, 0, 1))), p_df_sub(V.U(c, 0, 1), u));
    acc_prod(acc, p_mul(four, p_add(V.at<FXX>(c, 0, -1), xx)), p_df_sub(u, V.U(c, 0, -1)));
    acc_prod_neg(acc, p_mul(four, p_add(yy, V.at<FYY>(c, 1, 0))), p_df_sub(V.U(c, 1, 0), u));
    acc_prod(acc, p_mul(four, p_add(V.at<FYY>(c, -1, 0), yy)), p_df_sub(u, V.U(c, -1, 0)));
    const float2 oz = szz, ol = cl, orr = cr, od = cd, ou = cu;
    edges(V, c, n);
    acc_prod_neg(acc, p_mul(four, szz), p_df_sub(V.U(n, 0, 0), u));
    acc_prod(acc, p_mul(four, oz), p_df_sub(u, um[1]));
    // xy edges
    const float2 xl = p_add(V.at<FXY>(c, 0, -1), V.at<FXY>(c, 0, 0)), xr = p_add(V.at<FXY>(c, 0, 0), V.at<FXY>(c, 0, 1));
    const float2 xlp = p_add(V.at<FXY>(c, 1, -1), V.at<FXY>(c, 1, 0)), xrp = p_add(V.at<FXY>(c, 1, 0), V.at<FXY>(c, 1, 1));
    const float2 xlm = p_add(V.at<FXY>(c, -1, -1), V.at<FXY>(c, -1, 0)),
                 xrm = p_add(V.at<FXY>(c, -1, 0), V.at<FXY>(c, -1, 1));
    acc_prod_neg(acc, p_add(xr, xrp), p_df_sub(V.U(c, 1, 1), u));
    acc_prod(acc, p_add(xl, xlp), p_df_sub(V.U(c, 1, -1), u));
    acc_prod(acc, p_add(xrm, xr), p_df_sub(V.U(c, -1, 1), u));
    acc_prod_neg(acc, p_add(xlm, xl), p_df_sub(V.U(c, -1, -1), u));
    // xz edges
    acc_prod_neg(acc, cr, p_df_sub(V.U(n, 0, 1), u));
    acc_prod(acc, cl, p_df_sub(V.U(n, 0, -1), u));
    acc_prod(acc, orr, p_df_sub(rm, u));
    acc_prod_neg(acc, ol, p_df_sub(lm, u));
    // yz edges
    acc_prod_neg(acc, cu, p_df_sub(V.U(n, 1, 0), u));
    acc_prod(acc, cd, p_df_sub(V.U(n, -1, 0), u));
    acc_prod(acc, ou, p_df_sub(um[2], u));
    acc_prod_neg(acc, od, p_df_sub(um[0], u));
    um[1] = u;
    um[0] = V.U(c, -1, 0);
    um[2] = V.U(c, 1, 0);
    lm = V.U(c, 0, -1);
    rm = V.U(c, 0, 1);
  }
};

struct DfArgs {
  const float2* u;
  const float* e;
  float2* u_out;
  const float2* src;
  const double* m;
  const float* J;
  const float* D;
  float* r;
  float* e1;
  double *pr2, *pf2;
  float omega, h2;
  int scale_J, zc;
};

template <class OP, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_curv_df_march(Dims d, Fields P, DfArgs A) {
  extern __shared__ __align__(16) float smf[];
  __shared__ double shr[32];
  const int tid = threadIdx.x, lane = tid & 31, row = tid >> 5;
  const int x0 = blockIdx.x * MX, y0 = blockIdx.y * MY, z0 = blockIdx.z * A.zc;
  const int zend = min(z0 + A.zc, d.nz);
  const long long pst = (long long)d.nx * d.ny;
  Copier<NT, 1> C;
  C.init(d, P, x0, y0);
  const unsigned sbase = (unsigned)__cvta_generic_to_shared(smf);
  // the thread's x-pairs of u: in-plane offset, place in the hi plane, inside the tile?
  int q_off[2], q_dst[2];
  bool q_in[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int q = tid + k * NT, qr = q / 18, qc = q % 18;
    q_off[k] = q < NPAIR ? wrap_mod(y0 - 1 + qr, d.ny) * d.nx + wrap_mod(x0 - 2 + 2 * qc, d.nx) : -1;
    q_dst[k] = qr * PU + 2 * qc;
    q_in[k] = qc >= 1 && qc <= 16 && qr >= 1 && qr <= 16 && x0 - 2 + 2 * qc < d.nx && y0 - 1 + qr < d.ny;
  }
  const unsigned rawp = sbase + RAW * 4u, rawe = rawp + NPAIR * 16u;
  auto issue = [&](int z, int slot) {
    const int zw = z < 0 ? z + d.nz : (z >= d.nz ? z - d.nz : z);
    const long long zo = zw * pst;
    C.issue(P, zo, sbase + (unsigned)(slot * DSLOT) * 4u);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (q_off[k] < 0) continue;
      cp_async16(rawp + (tid + k * NT) * 16u, A.u + (zo + q_off[k]));
      if (A.e) cp_async8(rawe + (tid + k * NT) * 8u, A.e + (zo + q_off[k]));
    }
    cp_commit();
  };
  // the thread's own staged pairs of plane z: update, split into the slot, write back
  auto convert = [&](int z, int slot) {
    float* const uh = smf + slot * DSLOT + SB;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (q_off[k] < 0) continue;
      const float4 v = reinterpret_cast<const float4*>(smf + RAW)[tid + k * NT];
      DF2 w{make_float2(v.x, v.z), make_float2(v.y, v.w)};
      if (A.e) w = p_df_add_f(w, reinterpret_cast<const float2*>(smf + RAW + NPAIR * 4)[tid + k * NT]);
      *reinterpret_cast<float2*>(uh + q_dst[k]) = w.hi;
      *reinterpret_cast<float2*>(uh + URO + q_dst[k]) = w.lo;
      if (A.e && q_in[k] && z >= z0 && z < zend)
        *reinterpret_cast<float4*>(A.u_out + (z * pst + q_off[k])) = make_float4(w.hi.x, w.lo.x, w.hi.y, w.lo.y);
    }
  };
  const int x = x0 + lane;
  bool own[2];
  int off[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int y = y0 + row + 8 * k;
    own[k] = x < d.nx && y < d.ny;
    off[k] = own[k] ? y * d.nx + x : 0;
  }
  float Jn[2] = {1.f, 1.f}, Dn[2] = {1.f, 1.f};
  float2 bn[2] = {bcast(0.f), bcast(0.f)};
  auto fetch = [&](int z) {
    const long long zo = z * pst;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (!own[k]) continue;
      Jn[k] = __ldg(A.J + zo + off[k]);
      bn[k] = __ldg(A.src + zo + off[k]);
      if (A.e1) Dn[k] = __ldg(A.D + zo + off[k]);
    }
  };
  float2 m = bcast(0.f);
  if (A.m) m = f64_to_df(A.m[0]);
  const DfView V(smf, row, lane);
  // with compensation every four planes (8 squares): a run may be the whole mesh high, and one
  // FP32 chain of 2 x 256 squares was 5e-6 off (the tiles that this kernel replaced summed 16 per
  // thread).  In shared memory: four more registers across the loop cost 2%.
  __shared__ DfAcc sums[2][NT];
  sums[0][tid] = sums[1][tid] = DfAcc{0.f, 0.f};
  float r2 = 0.f, f2 = 0.f;
  auto flush = [&]() {
    sums[0][tid].add(r2);
    if (A.pf2) sums[1][tid].add(f2);
    r2 = f2 = 0.f;
  };
  issue(z0 - 1, 0);
  fetch(z0);
  cp_wait_all();
  convert(z0 - 1, 0);
  issue(z0, 1);
  cp_wait_all();
  convert(z0, 1);
  __syncthreads();
  issue(z0 + 1, 2);
  OP S;
  S.start(V, 0, DSLOT);
  int sc = 1, sn = 2, sf = 0;
  for (int t = z0; t < zend; ++t) {
    cp_wait_all();
    convert(t + 1, sn);
    __syncthreads();
    if (t + 1 < zend) issue(t + 2, sf);
    float Jc[2], Dc[2];
    float2 bc[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      Jc[k] = Jn[k];
      Dc[k] = Dn[k];
      bc[k] = bn[k];
      if (A.m) bc[k] = df_add(bc[k], make_float2(-m.x, -m.y));
    }
    if (t + 1 < zend) fetch(t + 1);
    PAcc acc{bcast(0.f), bcast(0.f)};
    {
      const float w0 = 8.f * (A.scale_J ? Jc[0] * A.h2 : A.h2), w1 = 8.f * (A.scale_J ? Jc[1] * A.h2 : A.h2);
      acc_prod(acc, make_float2(w0, w1), DF2{make_float2(bc[0].x, bc[1].x), make_float2(bc[0].y, bc[1].y)});
    }
    S.step(V, sc * DSLOT, sn * DSLOT, acc);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float a = 0.125f * (k ? __fadd_rn(acc.s.y, acc.c.y) : __fadd_rn(acc.s.x, acc.c.x));
      const float rv = __fdiv_rn(a, __fmul_rn(Jc[k], A.h2));
      if (!own[k]) continue;
      const long long i = t * pst + off[k];
      A.r[i] = rv;
      if (A.e1) A.e1[i] = __fmaf_rn(A.omega, __fdiv_rn(__fmul_rn(__fmul_rn(Jc[k], rv), A.h2), Dc[k]), 0.f);
      r2 = __fmaf_rn(rv, rv, r2);
      if (A.pf2) {
        const float fv = A.scale_J ? (bc[k].x + bc[k].y) : (bc[k].x + bc[k].y) / Jc[k];
        f2 = __fmaf_rn(fv, fv, f2);
      }
    }
    if ((t & 3) == 3 || t + 1 == zend) flush();
    const int q = sc;
    sc = sn;
    sn = sf;
    sf = q;
  }
  if (A.pr2) {
    const double s = block_sum_pair(sums[0][tid], shr);
    if (tid == 0) A.pr2[block_linear_id()] = s;
  }
  if (A.pf2) {
    const double s = block_sum_pair(sums[1][tid], shr);
    if (tid == 0) A.pf2[block_linear_id()] = s;
  }
}

// CTAs (of 256 threads) per SM, measured at 256^3 with the update and one FP32 chain for the norm
// (us; 1, 2, 3 CTAs):
//   M 474, 399, 607 (spills)   M^T 498, 657 (spills), -   S 438, 373, 553 (spills)
// (with the norm's compensated sums M 389, M^T 509, S 364) against 354 / 478 / 400 for the residual alone in the one-cell tiles, the update's 50 and
// the first sweep's 82 of their own.
constexpr int kCtas[3] = {2, 1, 2};
template <class OP, int MINB>
cudaError_t launch(cudaStream_t st, Dims d, const Fields& P, DfArgs A) {
  static DeviceSet done{0};
  const cudaError_t err = allow_smem(done, k_curv_df_march<OP, MINB>, kSmem);
  if (err != cudaSuccess) return err;
  A.zc = march_zchunk(d, MINB * 152);
  k_curv_df_march<OP, MINB><<<march_grid(d, A.zc), NT, kSmem, st>>>(d, P, A);
  note_launch();
  return cudaGetLastError();
}

long long blocks(Dims d, int minb) {
  const dim3 g = march_grid(d, march_zchunk(d, minb * 152));
  return (long long)g.x * g.y * g.z;
}

}  // namespace

long long march_df_partials(Dims d, int form) { return blocks(d, kCtas[form]); }


cudaError_t launch_march_df_step(cudaStream_t st, Dims d, const CurvCoef& cf, const float2* src, const double* m_dev,
                                 int scale_J, const float2* u, const float* e, float2* u_out, int form, float* r,
                                 float* e1, float omega, double* pr2, double* pf2) {
  Fields P;
  P.p[FU] = nullptr;
  for (int k = 0; k < 6; ++k) P.p[FXX + k] = cf.B[k];
  const DfArgs A{u, e, u_out, src, m_dev, cf.J, cf.D, r, e1, pr2, pf2, omega, cf.h2, scale_J, 0};
  switch (form) {
    case 0: return launch<DfM, kCtas[0]>(st, d, P, A);
    case 1: return launch<DfT, kCtas[1]>(st, d, P, A);
    default: return launch<DfS, kCtas[2]>(st, d, P, A);
  }
}

}  // namespace gbmg
