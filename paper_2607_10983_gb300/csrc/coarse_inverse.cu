// Minimum-norm inverses of the coarsest curvilinear operator and of its transposed-solve
// twin on the GPU (dense_pinv of host_math.cpp): Gauss-Jordan elimination with partial
// pivoting of the bordered (n + 1) x (n + 1) system, then the projection onto the range.
//
// Each orientation's matrix is inverted in place: a column of the right-hand identity
// becomes active when its row is the pivot, which is when the matrix column it replaces is
// finished.  A CTA owns a panel of NB columns in shared memory, a warp per column.  It
// applies the panels before its own as they appear in global memory, eliminates its own (one
// block barrier per pivot), writes the panel's multipliers and pivots to global memory,
// raises the panel's flag, and applies the panels after it.  All CTAs of a cooperative launch
// are resident, so the waits end; they are bounded all the same.  Every element sees the
// host code's operations in its order (products fused into the differences), so the inverse
// has its bits.
//
// What bounds it: the chain of n pivots (search, reciprocal, update of the next column); the
// n^3 FP64 multiply-adds, which run at under 2 per clock and SM, are spread over n / 8 SMs.
// The host took 0.75 ms per orientation for 125 unknowns and 4 ms for 216, with a copy and a
// synchronisation each way, twice per geometry.  A cluster of 16 CTAs exchanging columns
// through distributed shared memory took 147 / 476 / 1140 us for 64 / 125 / 216 unknowns:
// its remote stores, one per row and CTA, sat in front of every other shared access.  This
// one: 154 / 347 / 890 us (343 unknowns 2.0 ms, 480 3.9 ms).
#include "kernels.h"

namespace gbmg {

namespace {

constexpr int NB = 8;        // columns of a panel
constexpr int PT = 32 * NB;  // threads of a CTA
constexpr int kMaxPolls = 1 << 20;
constexpr int kMaxN = 512;   // unknowns of a coarsest level at most (mg_setup)

// Zero and NaN by the bits: FP64 comparisons run in the slow FP64 pipe, whose occupancy is
// what the elimination waits for.
__device__ __forceinline__ bool is_zero(double x) { return (__double_as_longlong(x) << 1) == 0; }

// A pivot: its reciprocal and row; ok: it did not vanish.
struct Step {
  double inv;
  int piv, ok;
};

int panel_count(int n) { return (n + 1 + NB - 1) / NB; }
size_t smem_bytes(int n) { return 2 * (size_t)NB * (n + 1) * sizeof(double) + 2 * (size_t)(n + 1) * sizeof(int); }

// Lm: two dense n x n operators (row-major); X: two (n + 1) x (n + 1) results; Fg, Sg: the
// multipliers and pivots of every column, two sets; flag: one per panel, two sets, zero;
// status: bit 0 a pivot vanished, bit 2 a wait ran out.
__global__ void __launch_bounds__(PT, 1) k_invert(int n, const double* __restrict__ Lm, double* __restrict__ X,
                                                  double* Fg, Step* Sg, int* flag, int* __restrict__ status) {
  extern __shared__ double sm[];
  __shared__ Step step[NB];
  __shared__ int give_up;
  const int m = n + 1, tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int panels = gridDim.x >> 1, o = blockIdx.x / panels, own = blockIdx.x - o * panels;
  const int j = own * NB + w;                          // the warp's column
  double* const col = sm + (size_t)w * m;
  double* const F = sm + (size_t)NB * m;               // multipliers of the panel at hand
  int* const row = reinterpret_cast<int*>(F + (size_t)NB * m);  // original index of each row
  int* const pivot = row + m;
  const double* const L = Lm + (size_t)o * n * n;
  double* const out = X + (size_t)o * m * m;
  double* const fo = Fg + (size_t)o * panels * NB * m;
  Step* const so = Sg + (size_t)o * panels * NB;
  int* const fl = flag + o * panels;
  if (j < m)
    for (int r = lane; r < m; r += 32) col[r] = j < n ? (r < n ? L[(size_t)r * n + j] : 1.0) : (r < n ? 1.0 : 0.0);
  for (int r = tid; r < m; r += PT) row[r] = r;
  if (tid == 0) give_up = 0;
  __syncthreads();

  // pivot step c (number p of its panel) on the warp's column
  auto update = [&](int c, int p) {
    const int piv = step[p].piv;
    const double* const f = F + (size_t)p * m;
    const double old = col[c];
    double v0 = 0.0;
    if (lane == 0) v0 = __dmul_rn(col[piv], step[p].inv);
    v0 = __shfl_sync(0xffffffffu, v0, 0);
    // (the trip count is the warp's, not the lane's: __syncwarp inside)
    for (int r0 = 0; r0 < m; r0 += 128) {
      double v[4], fr[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = min(r0 + lane + 32 * q, m - 1);
        v[q] = col[r];
        fr[q] = f[r];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (r0 + 32 * q >= m) break;
        const int r = r0 + lane + 32 * q;
        const double b = r == piv ? old : v[q];
        v[q] = r == c ? v0 : (is_zero(fr[q]) ? b : __fma_rn(-fr[q], v0, b));
      }
      __syncwarp();
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (r0 + lane + 32 * q < m) col[r0 + lane + 32 * q] = v[q];
    }
    __syncwarp();
  };

  for (int k = 0; k < panels; ++k) {
    const int cols = min(NB, m - k * NB);
    if (k != own) {
      // the panel's multipliers, once its flag is up
      if (tid == 0) {
        int up = 0;
        for (int t = 0; t < kMaxPolls && !up; ++t)
          asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(up) : "l"(fl + k) : "memory");
        if (!up) {
          give_up = 1;
          atomicOr(status, 4);
        }
      }
      __syncthreads();
      if (give_up) return;
      const double* const src = fo + (size_t)k * NB * m;
      for (int i = tid; i < cols * m; i += PT) F[i] = src[i];
      if (tid < cols) step[tid] = so[k * NB + tid];
      __syncthreads();
      if (j < m)
        for (int p = 0; p < cols; ++p) update(k * NB + p, p);
    } else {
      for (int p = 0; p < cols; ++p) {
        const int c = k * NB + p;
        double* const f = F + (size_t)p * m;
        if (w == p) {
          // largest magnitude on rows c .., the first of equals
          unsigned hi = 0, lo = 0;
          int at = m;
          for (int r = c + lane; r < m; r += 32) {
            unsigned long long b = (unsigned long long)__double_as_longlong(col[r]) & 0x7fffffffffffffffull;
            if (b > 0x7ff0000000000000ull) b = 0;  // a NaN is no pivot
            const unsigned h = (unsigned)(b >> 32), l = (unsigned)b;
            if (at == m || h > hi || (h == hi && l > lo)) hi = h, lo = l, at = r;
          }
          const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
          const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
          const int piv = (int)__reduce_min_sync(0xffffffffu, hi == mh && lo == ml ? (unsigned)at : (unsigned)m);
          const double fc = col[c], fp = col[piv];
          double inv = 0.0;
          if (lane == 0) inv = 1.0 / fp;
          inv = __shfl_sync(0xffffffffu, inv, 0);
          // the multipliers (the column after the row swap), and the identity column that
          // becomes active in its place
          for (int r0 = 0; r0 < m; r0 += 128) {
            double fr[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int r = r0 + lane + 32 * q;
              fr[q] = r == piv ? fc : (r == c ? fp : col[min(r, m - 1)]);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              if (r0 + 32 * q >= m) break;
              const int r = r0 + lane + 32 * q;
              const double v = r == c ? inv : (is_zero(fr[q]) ? 0.0 : -__dmul_rn(fr[q], inv));
              if (r < m) {
                f[r] = fr[q];
                col[r] = v;
              }
            }
          }
          if (lane == 0) {
            const double best = __longlong_as_double(((long long)mh << 32) | ml);
            step[p] = Step{inv, piv, best > 1e-300};
          }
        }
        __syncthreads();
        if (w != p && j < m) update(c, p);
      }
      __syncthreads();
      double* const dst = fo + (size_t)k * NB * m;
      for (int i = tid; i < cols * m; i += PT) dst[i] = F[i];
      if (tid < cols) {
        so[k * NB + tid] = step[tid];
        if (!step[tid].ok) atomicOr(status, 1);
      }
      __syncthreads();
      if (tid == 0) __threadfence();
      if (tid == 0) asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(fl + k), "r"(1) : "memory");
    }
    __syncthreads();
  }
  // the row swaps in order: column j holds the identity's column row[j]
  for (int c = tid; c < m; c += PT) pivot[c] = so[c].piv;
  __syncthreads();
  if (tid == 0)
    for (int c = 0; c < m; ++c) {
      const int piv = pivot[c], t = row[c];
      row[c] = row[piv];
      row[piv] = t;
    }
  __syncthreads();
  // column j holds the identity's column row[j]
  if (j < m)
    for (int r = lane; r < m; r += 32) out[(size_t)r * m + row[j]] = col[r];
}

// G = X (I - w w^T / w^T w) per row (w = J), in FP64 and FP32; status bit 1: a J not positive.
__global__ void __launch_bounds__(128) k_project(int n, const double* __restrict__ X, const float* __restrict__ J,
                                                 double* __restrict__ g64, double* __restrict__ g64t,
                                                 float* __restrict__ g32, float* __restrict__ g32t,
                                                 int* __restrict__ status) {
  extern __shared__ double sm[];
  __shared__ double xw, ww;
  const int i = blockIdx.x, m = n + 1, tid = threadIdx.x;
  const double* const x = X + (size_t)blockIdx.y * m * m + (size_t)i * m;
  double* const row = sm;
  double* const wv = sm + n;
  for (int j = tid; j < n; j += 128) {
    row[j] = x[j];
    wv[j] = (double)J[j];
    if (!(J[j] > 0.f)) atomicOr(status, 2);
  }
  __syncthreads();
  // the host's order: one chain of fused products each
  if (tid == 0) {
    double s = 0.0;
#pragma unroll 8
    for (int j = 0; j < n; ++j) s = __fma_rn(row[j], wv[j], s);
    xw = s;
  } else if (tid == 32) {
    double s = 0.0;
#pragma unroll 8
    for (int j = 0; j < n; ++j) s = __fma_rn(wv[j], wv[j], s);
    ww = s;
  }
  __syncthreads();
  double* const o64 = (blockIdx.y ? g64t : g64) + (size_t)i * n;
  float* const o32 = (blockIdx.y ? g32t : g32) + (size_t)i * n;
  for (int j = tid; j < n; j += 128) {
    const double g = __dsub_rn(row[j], __ddiv_rn(__dmul_rn(xw, wv[j]), ww));
    o64[j] = g;
    o32[j] = (float)g;
  }
}

}  // namespace

size_t coarse_inverse_work(int n) {
  const size_t m = n + 1, cols = (size_t)panel_count(n) * NB;
  return (2 * m * m + 2 * cols * m) * sizeof(double) + 2 * cols * sizeof(Step) + 2 * cols * sizeof(int);
}

cudaError_t launch_coarse_inverse(cudaStream_t st, int n, const double* dense, void* work, const float* J,
                                  double* g64, double* g64t, float* g32, float* g32t, int* status) {
  const int m = n + 1, panels = panel_count(n);
  const size_t cols = (size_t)panels * NB, sm = smem_bytes(n);
  double* X = (double*)work;
  double* F = X + 2 * (size_t)m * m;
  Step* S = (Step*)(F + 2 * cols * m);
  int* flag = (int*)(S + 2 * cols);
  // (the limit belongs to the kernel: the largest size, whatever other threads invert)
  cudaError_t e = cudaFuncSetAttribute(k_invert, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes(kMaxN));
  if (e == cudaSuccess) e = cudaMemsetAsync(status, 0, sizeof(int), st);
  if (e == cudaSuccess) e = cudaMemsetAsync(flag, 0, 2 * panels * sizeof(int), st);
  if (e != cudaSuccess) return e;
  void* args[] = {&n, &dense, &X, &F, &S, &flag, &status};
  e = cudaLaunchCooperativeKernel((const void*)k_invert, dim3(2 * panels), dim3(PT), args, sm, st);
  if (e != cudaSuccess) return e;
  note_launch();
  k_project<<<dim3(n, 2), 128, 2 * n * sizeof(double), st>>>(n, X, J, g64, g64t, g32, g32t, status);
  note_launch();
  return cudaGetLastError();
}

}  // namespace gbmg
