// Finite-difference gradients on the periodic finest level (spacing 1) and their
// transposes, for losses of the form sum(w . grad phi):
//   order 4: (-u_{i+2} + 8 u_{i+1} - 8 u_{i-1} + u_{i-2}) / 12, the one-exchange
//            fourth-order gradient of the force evaluation (Sec. 3.4);
//   order 2: (u_{i+1} - u_{i-1}) / 2, the central difference of Sec. 4.1.
// Both stencils are antisymmetric on the periodic mesh, so the transpose is the
// negated divergence with the same stencil.  FP64 in and out (w in FP32), once per
// loss evaluation, outside the V-cycle.
#include <cstdint>

#include "kernels.h"
#include "packed.cuh"
#include "solver.h"

namespace gbmg {

namespace {

constexpr int BX = 32, BY = 8;
dim3 cell_grid(Dims d) { return dim3((d.nx + BX - 1) / BX, (d.ny + BY - 1) / BY, d.nz); }

// |s| <= 2 <= n: one conditional wrap instead of a modulo
__device__ __forceinline__ int wrap2(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }
__device__ __forceinline__ long long shifted(Dims d, int x, int y, int z, int axis, int s) {
  if (axis == 0) x = wrap2(x + s, d.nx);
  else if (axis == 1) y = wrap2(y + s, d.ny);
  else z = wrap2(z + s, d.nz);
  return lin(d, x, y, z);
}

template <typename V>
__device__ __forceinline__ double dstencil(const V* u, Dims d, int x, int y, int z, int axis, int order, int sign) {
  auto U = [&](int s) { return (double)u[shifted(d, x, y, z, axis, sign * s)]; };
  if (order == 4) return (-U(2) + 8.0 * U(1) - 8.0 * U(-1) + U(-2)) / 12.0;
  return (U(1) - U(-1)) * 0.5;
}

__global__ void k_grad(Dims d, int order, const double* __restrict__ u, double* __restrict__ out) {
  const int x = blockIdx.x * BX + threadIdx.x, y = blockIdx.y * BY + threadIdx.y, z = blockIdx.z;
  if (x >= d.nx || y >= d.ny) return;
  const long long n = ncell(d), i = lin(d, x, y, z);
  for (int a = 0; a < 3; ++a) out[a * n + i] = dstencil(u, d, x, y, z, a, order, 1);
}

// grad^T w = -div w with the same antisymmetric stencil, one cell in FP64
__device__ double gradT_f64(const float* w, Dims d, int x, int y, int z, int order) {
  const long long n = ncell(d);
  double v = 0.0;
  for (int a = 0; a < 3; ++a) v += dstencil(w + a * n, d, x, y, z, a, order, -1);
  return v;
}

// ---- grad^T w without FP64 arithmetic per term
//
// The FP64 pipe issues under 2 operations per clock and SM, and the straightforward cell
// (12 conversions, 12 sums, 3 divisions, and in the dot product a block reduction per
// cell) spends its time there: 1.47 ms (transpose) and 1.36 ms (dot product) at 256^3
// against 0.05 ms of memory traffic.  So the numerator N = 12 grad^T w (order 2: 2
// grad^T w), a sum of FP32 values with power-of-two weights, is accumulated as an
// expansion of three FP32 parts on packed x-pairs (exact to 2^-72, beyond FP64), and
// turned into the FP64 quotient by integer operations.  At 256^3: 0.156 ms, bound by
// instruction issue (about 190 FP32 additions and 60 integer operations per pair of cells).

// Sum of three FP32 parts s + c + c2, |c2| << |c| << |s|, lane by lane.
struct PAcc3 {
  float2 s, c, c2;
  __device__ __forceinline__ void add(float2 t) {
    float2 ns, e, nc, e2;
    p_two_sum(s, t, ns, e);
    p_two_sum(c, e, nc, e2);
    s = ns;
    c = nc;
    c2 = p_add(c2, e2);
  }
};

// (s + c + c2) / div, div = 12 or 2, rounded to FP64, by integer operations.  ok is
// cleared when the leading part is tiny, huge or not finite (the caller then
// evaluates the cell in FP64).
template <int DIV>
__device__ __forceinline__ double expansion_quotient(float s, float c, float c2, bool& ok) {
  // renormalise (the sum may have cancelled, so no order of the parts is assumed):
  // |mid| <= ulp(hi), |lo| <= ulp(mid) / 2
  float hi, t, mid, lo, u;
  two_sum(c, c2, t, u);
  two_sum(s, t, hi, mid);
  two_sum(mid, u, t, lo);
  mid = t;
  if (hi == 0.f && mid == 0.f) {  // an exact zero (not NaN)
    ok = true;
    return 0.0;
  }
  const unsigned hb = __float_as_uint(hi);
  const int eh = (int)((hb >> 23) & 0xffu);
  ok = eh > 60 && eh < 245;
  // 62-bit fixed point with hi's leading bit at 2^61
  auto fixed = [&](float v) -> long long {
    const unsigned b = __float_as_uint(v);
    const int e = (int)((b >> 23) & 0xffu);
    const unsigned m = e ? ((b & 0x7fffffu) | 0x800000u) : 0u;  // subnormal parts are below 2^-62 of hi
    const int sh = eh - e;                                      // >= 23 for mid, more for lo
    const unsigned long long q = (unsigned long long)m << 38;
    const long long f = sh < 62 ? (long long)(q >> sh) : 0ll;
    return (b ^ hb) & 0x80000000u ? -f : f;
  };
  unsigned long long S = ((unsigned long long)((hb & 0x7fffffu) | 0x800000u)) << 38;
  S += (unsigned long long)(fixed(mid) + fixed(lo));
  int e2 = eh - 127 - 1;                        // S = value * 2^(61 - (eh - 127)); halved
  if (DIV == 12) {
    S = __umul64hi(S, 0xaaaaaaaaaaaaaaabull) >> 1;  // floor(S / 3)
    e2 -= 1;                                    // and a quarter
  }
  const int lz = __clzll((long long)S);         // 1 .. 4
  S <<= lz;                                     // leading bit at 2^63
  e2 += 2 - lz;
  // round to 53 bits, ties to even
  const unsigned long long rest = S & 0x7ffull;
  S >>= 11;
  S += (rest > 0x400ull || (rest == 0x400ull && (S & 1ull))) ? 1ull : 0ull;
  const unsigned long long bits =
      ((unsigned long long)(hb >> 31) << 63) + ((unsigned long long)(e2 + 1022) << 52) + S;  // S carries the implicit bit
  return __longlong_as_double((long long)bits);
}

// grad^T w on the cells x .. x + W - 1 (W = 2: an x-pair, nx even, 8-byte aligned w) of
// row y for the planes [z0, zend): emit(z, value of cell x, value of cell x + 1).
template <int ORDER, int W, typename Emit>
__device__ __forceinline__ void gradT_column(Dims d, const float* __restrict__ w, int x, int y, int z0, int zend,
                                             Emit emit) {
  const long long n = ncell(d), pst = (long long)d.nx * d.ny;
  constexpr int DIV = ORDER == 4 ? 12 : 2;
  const float2 zero = bcast(0.f);
  auto ldc = [&](const float* p) -> float2 {
    if constexpr (W == 2) return __ldg(reinterpret_cast<const float2*>(p));
    else return make_float2(__ldg(p), 0.f);
  };
  // in-plane offsets of the x neighbours (of the pair: its two neighbouring pairs) and rows
  const int row = y * d.nx;
  const int xm = wrap2(x - (W == 2 ? 2 : 1), d.nx), xp = wrap2(x + (W == 2 ? 2 : 1), d.nx);
  const int xmm = wrap2(x - 2, d.nx), xpp = wrap2(x + 2, d.nx);  // W = 1
  const int ym = wrap2(y - 1, d.ny) * d.nx + x, yp = wrap2(y + 1, d.ny) * d.nx + x;
  const int ymm = wrap2(y - 2, d.ny) * d.nx + x, ypp = wrap2(y + 2, d.ny) * d.nx + x;
  const float* wz = w + 2 * n + row + x;
  auto plane = [&](int z) { return (long long)wrap2(z, d.nz) * pst; };
  float2 zw[5];  // wz at planes z - 2 .. z + 2
#pragma unroll
  for (int k = 0; k < 4; ++k) zw[k + 1] = ldc(wz + plane(z0 - 2 + k));
  for (int z = z0; z < zend; ++z) {
#pragma unroll
    for (int k = 0; k < 4; ++k) zw[k] = zw[k + 1];
    zw[4] = ldc(wz + plane(z + 2));
    const float* wx = w + z * pst;
    const float* wy = wx + n;
    float2 m1, p1, m2 = zero, p2 = zero;
    if constexpr (W == 2) {
      const float2 a = ldc(wx + row + xm), b = ldc(wx + row + x), c = ldc(wx + row + xp);
      m1 = make_float2(a.y, b.x);
      p1 = make_float2(b.y, c.x);
      m2 = a;
      p2 = c;
    } else {
      m1 = ldc(wx + row + xm);
      p1 = ldc(wx + row + xp);
      if (ORDER == 4) {
        m2 = ldc(wx + row + xmm);
        p2 = ldc(wx + row + xpp);
      }
    }
    const float2 k1 = bcast(ORDER == 4 ? 8.f : 1.f);
    auto neg = [](float2 v) { return make_float2(-v.x, -v.y); };
    PAcc3 acc;
    acc.s = p_mul(k1, m1);
    acc.c = acc.c2 = zero;
    // the transposed stencil: +8 w_{i-1} - 8 w_{i+1} - w_{i-2} + w_{i+2}
    acc.add(neg(p_mul(k1, p1)));
    if (ORDER == 4) {
      acc.add(neg(m2));
      acc.add(p2);
    }
    acc.add(p_mul(k1, ldc(wy + ym)));
    acc.add(neg(p_mul(k1, ldc(wy + yp))));
    if (ORDER == 4) {
      acc.add(neg(ldc(wy + ymm)));
      acc.add(ldc(wy + ypp));
    }
    acc.add(p_mul(k1, zw[1]));
    acc.add(neg(p_mul(k1, zw[3])));
    if (ORDER == 4) {
      acc.add(neg(zw[0]));
      acc.add(zw[4]);
    }
    bool ok0, ok1 = true;
    double v0 = expansion_quotient<DIV>(acc.s.x, acc.c.x, acc.c2.x, ok0), v1 = 0.0;
    if (W == 2) v1 = expansion_quotient<DIV>(acc.s.y, acc.c.y, acc.c2.y, ok1);
    if (!ok0) v0 = gradT_f64(w, d, x, y, z, ORDER);
    if (!ok1) v1 = gradT_f64(w, d, x + 1, y, z, ORDER);
    emit(z, v0, v1);
  }
}

template <int ORDER, int W>
__global__ void k_grad_T(Dims d, const float* __restrict__ w, double* __restrict__ out, int gz) {
  const int x = (blockIdx.x * BX + threadIdx.x) * W, y = blockIdx.y * BY + threadIdx.y;
  if (x >= d.nx || y >= d.ny) return;
  const int z0 = blockIdx.z * gz, zend = min(z0 + gz, d.nz);
  double* const o = out + (long long)y * d.nx + x;
  const long long pst = (long long)d.nx * d.ny;
  gradT_column<ORDER, W>(d, w, x, y, z0, zend, [&](int z, double v0, double v1) {
    if constexpr (W == 2) *reinterpret_cast<double2*>(o + z * pst) = make_double2(v0, v1);
    else o[z * pst] = v0;
  });
}

// (double)f by integer operations (conversions run at the FP64 pipe's rate), f zero or normal.
__device__ __forceinline__ bool widens(float f) {
  const unsigned m = __float_as_uint(f) & 0x7fffffffu;
  return m == 0u || (m >= 0x00800000u && m < 0x7f800000u);
}
__device__ __forceinline__ double widen(float f) {
  const unsigned b = __float_as_uint(f), m = b & 0x7fffffffu;
  return __hiloint2double((int)((m ? (m >> 3) + 0x38000000u : 0u) | (b & 0x80000000u)), (int)(b << 29));
}

// Block partials of sum(w . grad u), from differences of u.  The sum of u grad^T w over the cells
// is the same number, but its terms have u's size instead of its gradient's: 15 times the
// error on a potential of 160^3 (spectrum k^-6), 10 times with a constant in u.  Here a constant
// drops out of the differences before anything else.  12 FP64 operations per cell (order 4; the
// divisions wait for the block's sum) bound it at the FP64 pipe's 1.6 per clock and SM: 0.407 ms
// at 256^3, order 2 0.208 (0.51 and 0.31 with the conversions of w in that pipe; one cell per
// thread with its divisions and a block reduction 1.36; the sum of u grad^T w 0.27 and 0.16).
template <int ORDER, int W>
__global__ void k_grad_dot(Dims d, const double* __restrict__ u, const float* __restrict__ w,
                           double* __restrict__ partials, int gz) {
  __shared__ double sh[32];
  const int x = (blockIdx.x * BX + threadIdx.x) * W, y = blockIdx.y * BY + threadIdx.y;
  double v = 0.0;
  if (x < d.nx && y < d.ny) {
    const int z0 = blockIdx.z * gz, zend = min(z0 + gz, d.nz);
    const long long n = ncell(d), pst = (long long)d.nx * d.ny;
    auto ldu = [&](const double* p) -> double2 {
      if constexpr (W == 2) return __ldg(reinterpret_cast<const double2*>(p));
      else return make_double2(__ldg(p), 0.0);
    };
    auto ldw = [&](const float* p) -> float2 {
      if constexpr (W == 2) return __ldg(reinterpret_cast<const float2*>(p));
      else return make_float2(__ldg(p), 0.f);
    };
    // w times the stencil's numerator; both differences first: a constant in u drops out
    auto term = [](double& s, double wv, double m2, double m1, double p1, double p2) {
      const double q = ORDER == 4 ? fma(8.0, p1 - m1, -(p2 - m2)) : p1 - m1;
      s = fma(wv, q, s);
    };
    double vx = 0.0, vy = 0.0, vz = 0.0;
    const long long row = (long long)y * d.nx, i = row + x;
    // the x neighbours: of the pair, its two neighbouring pairs
    const long long xm = row + wrap2(x - (W == 2 ? 2 : 1), d.nx), xp = row + wrap2(x + (W == 2 ? 2 : 1), d.nx);
    const long long xmm = row + wrap2(x - 2, d.nx), xpp = row + wrap2(x + 2, d.nx);  // W = 1
    const long long ym = (long long)wrap2(y - 1, d.ny) * d.nx + x, yp = (long long)wrap2(y + 1, d.ny) * d.nx + x;
    const long long ymm = (long long)wrap2(y - 2, d.ny) * d.nx + x, ypp = (long long)wrap2(y + 2, d.ny) * d.nx + x;
    double2 c[5];  // u at planes z - 2 .. z + 2
#pragma unroll
    for (int k = 0; k < 4; ++k) c[k + 1] = ldu(u + wrap2(z0 - 2 + k, d.nz) * pst + i);
    for (int z = z0; z < zend; ++z) {
#pragma unroll
      for (int k = 0; k < 4; ++k) c[k] = c[k + 1];
      c[4] = ldu(u + wrap2(z + 2, d.nz) * pst + i);
      const double* const up = u + z * pst;
      const float2 wx = ldw(w + z * pst + i), wy = ldw(w + n + z * pst + i), wz = ldw(w + 2 * n + z * pst + i);
      const double2 y1 = ldu(up + ym), y2 = ldu(up + yp);
      double2 y0 = y1, y3 = y2;
      if (ORDER == 4) {
        y0 = ldu(up + ymm);
        y3 = ldu(up + ypp);
      }
      const double2 a = ldu(up + xm), b = ldu(up + xp);
      double xl = 0.0, xr = 0.0;
      if (W == 1 && ORDER == 4) {
        xl = __ldg(up + xmm);
        xr = __ldg(up + xpp);
      }
      auto cells = [&](auto f64) {
        if constexpr (W == 2) {
          term(vx, f64(wx.x), a.x, a.y, c[2].y, b.x);
          term(vx, f64(wx.y), a.y, c[2].x, b.x, b.y);
          term(vy, f64(wy.y), y0.y, y1.y, y2.y, y3.y);
          term(vz, f64(wz.y), c[0].y, c[1].y, c[3].y, c[4].y);
        } else {
          term(vx, f64(wx.x), xl, a.x, b.x, xr);
        }
        term(vy, f64(wy.x), y0.x, y1.x, y2.x, y3.x);
        term(vz, f64(wz.x), c[0].x, c[1].x, c[3].x, c[4].x);
      };
      // (one branch for the pair: conversions under a predicate would run for every cell)
      if (widens(wx.x) && widens(wx.y) && widens(wy.x) && widens(wy.y) && widens(wz.x) && widens(wz.y))
        cells([](float f) { return widen(f); });
      else
        cells([](float f) { return (double)f; });
    }
    v = (vx + vy) + vz;
  }
  v = block_sum(v, sh);
  if (is_thread0()) partials[block_linear_id()] = v / (ORDER == 4 ? 12.0 : 2.0);
}

// z planes of one thread: 16 (four planes of the z window are loaded beside them), fewer
// on meshes that would not give every SM two blocks
int grad_planes(Dims d, int w) {
  const long long cols = (long long)((d.nx / w + BX - 1) / BX) * ((d.ny + BY - 1) / BY);
  int gz = 16;
  while (gz > 2 && cols * ((d.nz + gz - 1) / gz) < 2 * 152) gz /= 2;
  return gz;
}
dim3 grad_grid(Dims d, int w, int gz) {
  return dim3((d.nx / w + BX - 1) / BX, (d.ny + BY - 1) / BY, (d.nz + gz - 1) / gz);
}
// x-pairs: even rows, the FP32 field on 8 and the FP64 field on 16 bytes
bool grad_pairs(Dims d, const float* w, const double* f) {
  return d.nx % 2 == 0 && ((uintptr_t)w & 7) == 0 && ((uintptr_t)f & 15) == 0;
}

}  // namespace

}  // namespace gbmg

using namespace gbmg;

extern "C" gbmg_status mg_grad(gbmg_ctx* c, int order, int transpose, const void* in_dev, double* out_dev) {
  if (!c || !in_dev || !out_dev || (order != 2 && order != 4)) return fail(GBMG_ERR_INVALID_ARG, "mg_grad: bad argument");
  DeviceGuard g(c->device);
  const Dims d = c->lv[0].d;
  if (transpose) {
    const float* w = (const float*)in_dev;
    const bool pairs = grad_pairs(d, w, out_dev);
    const int gz = grad_planes(d, pairs ? 2 : 1);
    const dim3 g = grad_grid(d, pairs ? 2 : 1, gz), t(BX, BY);
    if (order == 4 && pairs) k_grad_T<4, 2><<<g, t, 0, c->stream>>>(d, w, out_dev, gz);
    else if (order == 4) k_grad_T<4, 1><<<g, t, 0, c->stream>>>(d, w, out_dev, gz);
    else if (pairs) k_grad_T<2, 2><<<g, t, 0, c->stream>>>(d, w, out_dev, gz);
    else k_grad_T<2, 1><<<g, t, 0, c->stream>>>(d, w, out_dev, gz);
  } else k_grad<<<cell_grid(d), dim3(BX, BY), 0, c->stream>>>(d, order, (const double*)in_dev, out_dev);
  note_launch();
  TRY(cudaGetLastError());
  return GBMG_OK;
}

extern "C" gbmg_status mg_grad_dot(gbmg_ctx* c, int order, const double* u_dev, const float* w_dev, double* out_dev) {
  if (!c || !u_dev || !w_dev || !out_dev || (order != 2 && order != 4))
    return fail(GBMG_ERR_INVALID_ARG, "mg_grad_dot: bad argument");
  DeviceGuard g(c->device);
  const Dims d = c->lv[0].d;
  const bool pairs = grad_pairs(d, w_dev, u_dev);
  const int gz = grad_planes(d, pairs ? 2 : 1);
  const dim3 gr = grad_grid(d, pairs ? 2 : 1, gz), t(BX, BY);
  if (order == 4 && pairs) k_grad_dot<4, 2><<<gr, t, 0, c->stream>>>(d, u_dev, w_dev, c->partials, gz);
  else if (order == 4) k_grad_dot<4, 1><<<gr, t, 0, c->stream>>>(d, u_dev, w_dev, c->partials, gz);
  else if (pairs) k_grad_dot<2, 2><<<gr, t, 0, c->stream>>>(d, u_dev, w_dev, c->partials, gz);
  else k_grad_dot<2, 1><<<gr, t, 0, c->stream>>>(d, u_dev, w_dev, c->partials, gz);
  note_launch();
  TRY(cudaGetLastError());
  TRY(launch_finalize(c->stream, c->partials, (long long)gr.x * gr.y * gr.z, out_dev, 1.0));
  return GBMG_OK;
}
