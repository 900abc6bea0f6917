// Spectral inner solves on the uniform channel: the projection's pressure
// problem, and the velocity problem inside the exact Stokes solve.
//
// The projection P~ = I - G (DG)^+ D of Section 4 needs the Neumann pressure
// problem (D^ D^T) phi = D^ w.  On the uniform channel that operator is the
// Kronecker sum of the periodic second difference along x and y and the
// cell-centred Neumann second difference along z, so Fourier modes along x
// and y diagonalise it and leave, for every mode (mx, my), the tridiagonal
// system
//     (lambda(mx) + lambda(my)) phi^ + T_z phi^ = r^,
//     lambda(m) = 2 - 2 cos(2 pi m / n),  T_z = tridiag(-1, 2, -1), ends 1
// along z.  The solve used inside FP64 iterative refinement (the projection's
// FAC iteration of Algorithm 1 with this solve in place of the V-cycle) is:
//   1. forward 2-D FFT of every z plane of the FP32 residual (one CTA per
//      plane, the plane in shared memory, radix-2 decimation in frequency:
//      modes come out in bit-reversed order, which nothing needs to undo);
//   2. per mode, the z system solved by the Thomas algorithm in FP32 (the
//      all-constant mode (0, 0) is singular: its z = 0 value is pinned to 0,
//      which fixes the pressure's free constant, and its column -- the
//      worst-conditioned one -- is solved exactly in FP64 by two scans);
//   3. inverse 2-D FFT of every plane (decimation in time, bit-reversed in,
//      natural out); the real part / n^2 is the correction.
// Grids: 3-D, nx == ny == n a power of two, 4 <= n <= 128; nz >= 2.
// The no-slip velocity operator has the same form with other ends of T_z (3 on
// cell centres, 2 on wall-normal faces) and no singular mode; its components'
// planes share the three launches.

#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

#include "../../include/selm_mg.h"
#include "selm_internal.h"
#include "selm_launch.h"
#include "selm_prof.h"

namespace selm {
namespace {

constexpr int kSpecThreads = 512;
constexpr int kThomasThreads = 128;

__device__ __forceinline__ int bitrev(int x, int logn) { return (int)(__brev((unsigned)x) >> (32 - logn)); }

// twiddles W[j] = exp(-2 pi i j / n), j < n / 2
__device__ void make_twiddles(float2* W, int n) {
  for (int j = threadIdx.x; j < (n >> 1); j += blockDim.x) {
    float s, c;
    sincospif(-2.0f * (float)j / (float)n, &s, &c);
    W[j] = make_float2(c, s);
  }
}

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// Butterfly q of a stage over all rows (columns == false: along x) or all
// columns (along y) of an n x n plane: line and pair index, with consecutive
// threads on consecutive addresses in both cases.  n = 2^logn and
// half = 2^lh, so the index arithmetic is shifts and masks.
__device__ __forceinline__ void stage_index(int q, int logn, int lh, bool columns, int* a0, int* a1, int* j) {
  const int n = 1 << logn;
  const int line = columns ? (q & (n - 1)) : (q >> (logn - 1));
  const int p = columns ? (q >> logn) : (q & ((n >> 1) - 1));
  const int grp = p >> lh;
  *j = p & ((1 << lh) - 1);
  const int i0 = (grp << (lh + 1)) + *j, i1 = i0 + (1 << lh);
  *a0 = columns ? (i0 << logn) + line : (line << logn) + i0;
  *a1 = columns ? (i1 << logn) + line : (line << logn) + i1;
}

// Forward transform along one axis, decimation in frequency: natural order in,
// bit-reversed order out.
__device__ void fft_dif(float2* A, const float2* W, int n, int logn, bool columns) {
  for (int s = logn; s >= 1; --s) {
    const int lh = s - 1, tw_shift = logn - s;
    for (int q = threadIdx.x; q < n * (n >> 1); q += blockDim.x) {
      int a0, a1, j;
      stage_index(q, logn, lh, columns, &a0, &a1, &j);
      const float2 x0 = A[a0], x1 = A[a1];
      A[a0] = make_float2(x0.x + x1.x, x0.y + x1.y);
      A[a1] = cmul(make_float2(x0.x - x1.x, x0.y - x1.y), W[j << tw_shift]);
    }
    __syncthreads();
  }
}

// Inverse transform (unscaled) along one axis, decimation in time:
// bit-reversed order in, natural order out.
__device__ void fft_dit_inv(float2* A, const float2* W, int n, int logn, bool columns) {
  for (int s = 1; s <= logn; ++s) {
    const int lh = s - 1, tw_shift = logn - s;
    for (int q = threadIdx.x; q < n * (n >> 1); q += blockDim.x) {
      int a0, a1, j;
      stage_index(q, logn, lh, columns, &a0, &a1, &j);
      float2 w = W[j << tw_shift];
      w.y = -w.y;   // exp(+2 pi i j / (2 half))
      const float2 x0 = A[a0], t = cmul(A[a1], w);
      A[a0] = make_float2(x0.x + t.x, x0.y + t.y);
      A[a1] = make_float2(x0.x - t.x, x0.y - t.y);
    }
    __syncthreads();
  }
}

// Forward: plane k of r (FP32, [nz][n][n]) -> spectrum S[k][.][.] with both
// mode indices in bit-reversed order (the solve along z does not care; the
// inverse transform takes that order as it comes).
__global__ void __launch_bounds__(kSpecThreads) k_spec_forward(const float* __restrict__ r, float2* __restrict__ S,
                                                               int n, int logn) {
  extern __shared__ float2 sm[];
  float2* A = sm;
  float2* W = sm + n * n;
  const int k = blockIdx.x;
  const float* rp = r + (long long)k * n * n;
  make_twiddles(W, n);
  // eight loads in flight per thread before their stores (n * n is a
  // multiple of 8 * blockDim for the supported sizes, else the tail loop)
  int q = threadIdx.x;
  for (; q + 7 * (int)blockDim.x < n * n; q += 8 * blockDim.x) {
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = rp[q + e * blockDim.x];
#pragma unroll
    for (int e = 0; e < 8; ++e) A[q + e * blockDim.x] = make_float2(v[e], 0.0f);
  }
  for (; q < n * n; q += blockDim.x) A[q] = make_float2(rp[q], 0.0f);
  __syncthreads();
  fft_dif(A, W, n, logn, false);
  fft_dif(A, W, n, logn, true);
  float2* Sp = S + (long long)k * n * n;
  for (int q = threadIdx.x; q < n * n; q += blockDim.x) Sp[q] = A[q];
}

// Inverse: spectrum plane k -> delta (FP32 real part / n^2).
__global__ void __launch_bounds__(kSpecThreads) k_spec_inverse(const float2* __restrict__ S, float* __restrict__ d,
                                                               int n, int logn) {
  extern __shared__ float2 sm[];
  float2* A = sm;
  float2* W = sm + n * n;
  const int k = blockIdx.x;
  const float2* Sp = S + (long long)k * n * n;
  make_twiddles(W, n);
  int q = threadIdx.x;
  for (; q + 7 * (int)blockDim.x < n * n; q += 8 * blockDim.x) {
    float2 v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = Sp[q + e * blockDim.x];
#pragma unroll
    for (int e = 0; e < 8; ++e) A[q + e * blockDim.x] = v[e];
  }
  for (; q < n * n; q += blockDim.x) A[q] = Sp[q];
  __syncthreads();
  fft_dit_inv(A, W, n, logn, false);
  fft_dit_inv(A, W, n, logn, true);
  const float inv = 1.0f / (float)(n * n);
  float* dp = d + (long long)k * n * n;
  for (int q = threadIdx.x; q < n * n; q += blockDim.x) dp[q] = A[q].x * inv;
}

// The wall axes of a system's components: rows, first plane of the component
// in the spectrum, and the diagonal of T_z in its first and last row (cell
// centres 3 with the no-slip ghost, 1 with the Neumann ghost; wall-normal
// faces 2).
struct WallAxes {
  int nz[kMaxComps];
  int first[kMaxComps];
  float end[kMaxComps];
};

// a[c] of a kernel parameter by selects: indexed with a run-time c, the whole
// struct is copied to local memory and every use of the value leaves the uniform
// registers (k_spec_thomas at 128^3: 23.1 instead of 16.6 us).
template <typename V>
__device__ __forceinline__ V param_at(const V (&a)[kMaxComps], unsigned c) {
  V v = a[0];
#pragma unroll
  for (unsigned q = 1; q < kMaxComps; ++q)
    if (c == q) v = a[q];
  return v;
}

// Thomas algorithm along z for the modes stored at (row py, column px)
// (mode indices bit-reversed), one thread per column, in place in S, in FP32;
// component blockIdx.y.
// Shared memory: per thread, the forward sweep's c' and the column
// ([nz][threads] each).  The all-constant mode (0, 0) is singular; the extra
// last block solves it alone (one warp, FP64): its z = 0 value is pinned to 0,
// which fixes the pressure's free constant, and the remaining rows of the
// Neumann T_z are a flux balance, g_k = x_k - x_{k-1} = sum_{j >= k} d_j and
// x_k = sum_{i <= k} g_i -- two scans.  (A no-slip operator has no singular
// mode: SINGULAR == false and no extra block.)  The Neumann form, with one
// component and its ends as constants, is the shorter chain per row: 16.6 us at
// 128^3, 19.2 with the ends as values.
template <bool SINGULAR>
__global__ void __launch_bounds__(kThomasThreads) k_spec_thomas(float2* __restrict__ S, int n, int logn, WallAxes wa,
                                                                float inv_scale) {
  extern __shared__ float tsm[];
  const int t = threadIdx.x;
  const int nz = SINGULAR ? wa.nz[0] : param_at(wa.nz, blockIdx.y);
  const float end = SINGULAR ? 1.0f : param_at(wa.end, blockIdx.y);
  if (!SINGULAR) S += (long long)param_at(wa.first, blockIdx.y) * n * n;
  const int per_row = n / (int)blockDim.x > 0 ? n / (int)blockDim.x : 1;
  const long long plane = (long long)n * n;
  if (SINGULAR && blockIdx.x == (unsigned)(n * per_row)) {   // the (0, 0) mode, stored at column 0 of row 0
    if (t >= 32) return;
    const int rows = nz - 1;                      // unknowns x_1 .. x_{nz-1}
    const int per = (rows + 31) / 32;             // consecutive rows per lane
    double gx[8], gy[8];                          // nz <= 257
    const int k0 = 1 + t * per;
    double sx = 0.0, sy = 0.0;
    // suffix sums of d within the lane's rows, then across lanes
    for (int e = per - 1; e >= 0; --e) {
      const int k = k0 + e;
      if (k < nz) {
        const float2 f = S[k * plane];
        sx += (double)f.x * inv_scale;
        sy += (double)f.y * inv_scale;
      }
      gx[e] = sx;
      gy[e] = sy;
    }
    // exclusive suffix scan of the lane totals over higher lanes
    double tx = sx, ty = sy;
    for (int o = 1; o < 32; o <<= 1) {
      const double ux = __shfl_down_sync(0xffffffffu, tx, o), uy = __shfl_down_sync(0xffffffffu, ty, o);
      if (t + o < 32) {
        tx += ux;
        ty += uy;
      }
    }
    const double hx = tx - sx, hy = ty - sy;   // sum over higher lanes
    double px_ = 0.0, py_ = 0.0;
    for (int e = 0; e < per; ++e) {
      gx[e] += hx;
      gy[e] += hy;
      if (k0 + e < nz) {
        px_ += gx[e];
        py_ += gy[e];
      }
      gx[e] = px_;   // now the lane-local prefix of g
      gy[e] = py_;
    }
    // exclusive prefix scan of the lane totals over lower lanes
    double qx = px_, qy = py_;
    for (int o = 1; o < 32; o <<= 1) {
      const double ux = __shfl_up_sync(0xffffffffu, qx, o), uy = __shfl_up_sync(0xffffffffu, qy, o);
      if (t >= o) {
        qx += ux;
        qy += uy;
      }
    }
    const double lx = qx - px_, ly = qy - py_;
    for (int e = 0; e < per; ++e) {
      const int k = k0 + e;
      if (k < nz) S[k * plane] = make_float2((float)(gx[e] + lx), (float)(gy[e] + ly));
    }
    if (t == 0) S[0] = make_float2(0.0f, 0.0f);
    return;
  }
  const int py = blockIdx.x / per_row;
  const int px = (blockIdx.x - py * per_row) * blockDim.x + t;
  const long long col = (long long)py * n + px;
  if (px >= n) return;
  const int mx = bitrev(px, logn), my = bitrev(py, logn);
  if (SINGULAR && mx == 0 && my == 0) return;   // solved by the last block
  float* cp = tsm;                                               // [nz][threads]
  float2* dd = reinterpret_cast<float2*>(tsm + nz * blockDim.x);  // [nz][threads]: the column
  // the whole column first (independent, coalesced loads), then the sweeps
  {
    int k = 0;
    for (; k + 8 <= nz; k += 8) {   // eight loads in flight before their stores
      float2 v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = S[(k + e) * plane + col];
#pragma unroll
      for (int e = 0; e < 8; ++e) dd[(k + e) * blockDim.x + t] = v[e];
    }
    for (; k < nz; ++k) dd[k * blockDim.x + t] = S[k * plane + col];
  }
  // lambda(m) = 2 - 2 cos(2 pi m / n) per axis
  const float lam = (2.0f - 2.0f * cospif(2.0f * (float)mx / (float)n)) +
                    (2.0f - 2.0f * cospif(2.0f * (float)my / (float)n));
  float cprev = 0.0f;
  float2 dprev = make_float2(0.0f, 0.0f);
  for (int k = 0; k < nz; ++k) {
    const float2 f = dd[k * blockDim.x + t];
    const float b = lam + ((k == 0 || k == nz - 1) ? end : 2.0f);
    const float m = b - (k == 0 ? 0.0f : -cprev);                   // a = -1
    const float r = 1.0f / m;
    const float cn = k == nz - 1 ? 0.0f : -r;
    dprev = make_float2((f.x * inv_scale + (k == 0 ? 0.0f : dprev.x)) * r,
                        (f.y * inv_scale + (k == 0 ? 0.0f : dprev.y)) * r);
    cp[k * blockDim.x + t] = cn;
    dd[k * blockDim.x + t] = dprev;
    cprev = cn;
  }
  float2 x = dprev;
  S[(nz - 1) * plane + col] = x;
  for (int k = nz - 2; k >= 0; --k) {
    const float cn = cp[k * blockDim.x + t];
    const float2 dn = dd[k * blockDim.x + t];
    x = make_float2(dn.x - cn * x.x, dn.y - cn * x.y);
    S[k * plane + col] = x;
  }
}

// ---- the staggered composite grid's pressure operator ---------------------------
// diag(vol) D G on the composite cells: fine layers of 2n x 2n cells below
// z = K H, base rows of n x n cells above, and across the interface one
// difference per base cell, (base value - mean of its four children) with
// weight W = 4 H / 3.  Fourier modes along x and y leave, per base mode
// kappa = (kx, ky), the base column of that mode and the fine columns of its
// four aliases (kx + {0, n}, ky + {0, n}), tied together by the interface only:
// with c_a = (1 + e^{-i pi k_a / n}) / 2 per axis, multiplied over x and y,
//     T_f x_a = b_a + c_a Q e_top,   T_c y = b_c - Q e_0,
//     Q = W (y_0 - 1/4 sum_a conj(c_a) x_a,top).
// Each column is eliminated from its wall to the interface, Q follows from the
// five ends, and the columns are substituted back.  The pivots are kept as
// d = w (1 + e), e_0 = lambda, e_m = lambda + e_{m-1} / (1 + e_{m-1}), which has
// no cancellation for small lambda.  In bit-reversed order the base mode at
// (py, px) has its aliases at (2 py + {0, 1}, 2 px + {0, 1}).  The constant
// mode's columns are solved by two FP64 scans (flux balance).
struct MacSpec {
  int n, logn, nf, nb;       // base edge, fine layers (2 K), base rows (n - K)
  float2* fine;              // [nf][2n][2n]
  float2* base;              // [nb][n][n]
};

// Planes of the residual (FP64, divided by its norm sqrt(*rr)) to spectra:
// fine layers, then base rows.
__global__ void __launch_bounds__(kSpecThreads) k_mac_forward(MacSpec M, const double* __restrict__ r,
                                                              const double* __restrict__ rr) {
  extern __shared__ float2 sm[];
  const bool f = (int)blockIdx.x < M.nf;
  const int logn = M.logn + (f ? 1 : 0), n = 1 << logn, N = n * n;
  const int k = f ? blockIdx.x : blockIdx.x - M.nf;
  const double* rp = f ? r + (long long)k * N : r + (long long)M.nf * 4 * M.n * M.n + (long long)k * N;
  float2* Sp = (f ? M.fine : M.base) + (long long)k * N;
  float2* A = sm;
  float2* W = sm + N;
  make_twiddles(W, n);
  const double scale = *rr > 0.0 ? rsqrt(*rr) : 0.0;
  int q = threadIdx.x;
  for (; q + 7 * (int)blockDim.x < N; q += 8 * blockDim.x) {
    double v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = rp[q + e * blockDim.x];
#pragma unroll
    for (int e = 0; e < 8; ++e) A[q + e * blockDim.x] = make_float2((float)(v[e] * scale), 0.0f);
  }
  for (; q < N; q += blockDim.x) A[q] = make_float2((float)(rp[q] * scale), 0.0f);
  __syncthreads();
  fft_dif(A, W, n, logn, false);
  fft_dif(A, W, n, logn, true);
  for (int q2 = threadIdx.x; q2 < N; q2 += blockDim.x) Sp[q2] = A[q2];
}

// Spectra to planes of z = S^-1 r (S is negative: the columns solve -S), times
// the residual's norm.
__global__ void __launch_bounds__(kSpecThreads) k_mac_inverse(MacSpec M, double* __restrict__ z,
                                                              const double* __restrict__ rr) {
  extern __shared__ float2 sm[];
  const bool f = (int)blockIdx.x < M.nf;
  const int logn = M.logn + (f ? 1 : 0), n = 1 << logn, N = n * n;
  const int k = f ? blockIdx.x : blockIdx.x - M.nf;
  double* zp = f ? z + (long long)k * N : z + (long long)M.nf * 4 * M.n * M.n + (long long)k * N;
  const float2* Sp = (f ? M.fine : M.base) + (long long)k * N;
  float2* A = sm;
  float2* W = sm + N;
  make_twiddles(W, n);
  int q = threadIdx.x;
  for (; q + 7 * (int)blockDim.x < N; q += 8 * blockDim.x) {
    float2 v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = Sp[q + e * blockDim.x];
#pragma unroll
    for (int e = 0; e < 8; ++e) A[q + e * blockDim.x] = v[e];
  }
  for (; q < N; q += blockDim.x) A[q] = Sp[q];
  __syncthreads();
  fft_dit_inv(A, W, n, logn, false);
  fft_dit_inv(A, W, n, logn, true);
  const double scale = -sqrt(*rr) / (double)N;
  for (int q2 = threadIdx.x; q2 < N; q2 += blockDim.x) zp[q2] = (double)A[q2].x * scale;
}

__device__ __forceinline__ float lambda_of(int m, int n) { return 2.0f - 2.0f * cospif(2.0f * (float)m / (float)n); }

// The columns of 32 base modes of one row py: warp c < 4 the fine columns of
// alias (c >> 1, c & 1), warp 4 the base columns.  Shared memory: per warp its
// columns and their multipliers (rows x 32), then the exchange of the ends.
// The block after the last one solves the constant mode.
__global__ void __launch_bounds__(160) k_mac_columns(MacSpec M) {
  extern __shared__ float csm[];
  const int n = M.n, nf = M.nf, nb = M.nb, n2 = 2 * n;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float H = 1.0f / (float)n, h = 0.5f * H, Wi = 4.0f / 3.0f * H;
  const long long fplane = (long long)n2 * n2, bplane = (long long)n * n;
  const int per_row = (n + 31) / 32;
  if ((int)blockIdx.x == n * per_row) {
    // constant mode: B_i the sum of b over rows 0..i (fine, then base); in units
    // of the cell means u = x / 4 (fine), y (base): u_{m+1} = u_m - B_m / (4 h),
    // across the interface - B / W, then - B / H; u_0 = 0
    if (warp != 0) return;
    const int rows = nf + nb, per = (rows + 31) / 32;   // at most 4 (rows <= 128)
    double b[4], s = 0.0;
    for (int e = 0; e < per; ++e) {
      const int i = lane * per + e;
      s += i < rows ? (double)(i < nf ? M.fine[i * fplane].x : M.base[(i - nf) * bplane].x) : 0.0;
      b[e] = s;
    }
    auto exclusive = [&](double total) {
      double t = total;
      for (int o = 1; o < 32; o <<= 1) {
        const double u = __shfl_up_sync(0xffffffffu, t, o);
        if (lane >= o) t += u;
      }
      return t - total;
    };
    const double hb = exclusive(s);
    double g = 0.0;
    for (int e = 0; e < per; ++e) {   // the step from row i to row i + 1
      const int i = lane * per + e;
      const double w = i + 1 < nf ? 4.0 * (0.5 / n) : i + 1 == nf ? 4.0 / 3.0 / n : 1.0 / n;
      const double before = g;
      g -= (b[e] + hb) / w;
      b[e] = before;                  // the prefix of the steps up to row i, within the lane
    }
    const double hg = exclusive(g);
    for (int e = 0; e < per; ++e) {
      const int i = lane * per + e;
      if (i >= rows) continue;
      const float u = (float)(b[e] + hg);
      if (i < nf)
        M.fine[i * fplane] = make_float2(4.0f * u, 0.0f);
      else
        M.base[(i - nf) * bplane] = make_float2(u, 0.0f);
    }
    return;
  }
  const int py = blockIdx.x / per_row, px = (blockIdx.x - py * per_row) * 32 + lane;
  const bool on = px < n;
  const int kx = on ? bitrev(px, M.logn) : 0, ky = bitrev(py, M.logn);
  const bool fine = warp < 4;
  const int ay = warp >> 1, ax = warp & 1;
  const int rows = fine ? nf : nb;
  // row m of the column counted from its wall: fine layer m, base row nb - 1 - m
  float2* col;
  long long step;
  float lam, w, cre = 1.0f, cim = 0.0f;   // c_a
  if (fine) {
    const int mx = kx + ax * n, my = ky + ay * n;
    col = M.fine + (long long)(2 * py + ay) * n2 + 2 * px + ax;
    step = fplane;
    lam = lambda_of(mx, n2) + lambda_of(my, n2);
    w = h;
    float sx, cx, sy, cy;
    sincospif(-(float)mx / (float)n, &sx, &cx);
    sincospif(-(float)my / (float)n, &sy, &cy);
    const float2 c = cmul(make_float2(0.5f * (1.0f + cx), 0.5f * sx), make_float2(0.5f * (1.0f + cy), 0.5f * sy));
    cre = c.x;
    cim = c.y;
  } else {
    col = M.base + (nb - 1) * bplane + (long long)py * n + px;
    step = -bplane;
    lam = lambda_of(kx, n) + lambda_of(ky, n);
    w = H;
  }
  const bool solve = on && rows > 0 && !(kx == 0 && ky == 0 && (!fine || warp == 0));
  // columns (float2) and multipliers 1 / (1 + e) of the warps one after another
  float2* x = reinterpret_cast<float2*>(csm) + (fine ? (long long)warp * nf * 32 : (long long)4 * nf * 32) + lane;
  float* mult = csm + 2 * (long long)(4 * nf + nb) * 32 + (fine ? (long long)warp * nf * 32 : (long long)4 * nf * 32) + lane;
  float4* ends = reinterpret_cast<float4*>(csm + 3 * (long long)(4 * nf + nb) * 32);   // [5][32]
  float2 b = make_float2(0.0f, 0.0f);
  float e = 0.0f;
  if (solve) {
    int m = 0;
    for (; m + 8 <= rows; m += 8) {   // eight loads in flight before their stores
      float2 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = col[(m + u) * step];
#pragma unroll
      for (int u = 0; u < 8; ++u) x[(m + u) * 32] = v[u];
    }
    for (; m < rows; ++m) x[m * 32] = col[m * step];
    // b'_m = b_m + b'_{m-1} / (1 + e_{m-1})
    float inv = 0.0f;
    for (m = 0; m < rows; ++m) {
      const float2 f = x[m * 32];
      b = make_float2(fmaf(b.x, inv, f.x), fmaf(b.y, inv, f.y));
      e = m == 0 ? lam : fmaf(e, inv, lam);
      inv = 1.0f / (1.0f + e);
      x[m * 32] = b;
      mult[m * 32] = inv;
    }
  }
  // the ends: x_end = (b' + q) / (w e), q the interface's contribution
  const float dinv = solve ? 1.0f / (w * e) : 0.0f;
  ends[warp * 32 + lane] = make_float4(b.x * dinv, b.y * dinv, dinv, 0.0f);
  __syncthreads();
  if (!solve) return;
  float2 Q = make_float2(0.0f, 0.0f);
  if (nf > 0 && nb > 0 && !(kx == 0 && ky == 0)) {
    float2 num = make_float2(0.0f, 0.0f);
    float den = 1.0f;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int mx = kx + (a & 1) * n, my = ky + (a >> 1) * n;
      float sx, cx, sy, cy;
      sincospif(-(float)mx / (float)n, &sx, &cx);
      sincospif(-(float)my / (float)n, &sy, &cy);
      const float2 c = cmul(make_float2(0.5f * (1.0f + cx), 0.5f * sx), make_float2(0.5f * (1.0f + cy), 0.5f * sy));
      const float4 t = ends[a * 32 + lane];
      const float2 ct = cmul(make_float2(c.x, -c.y), make_float2(t.x, t.y));
      num.x -= 0.25f * ct.x;
      num.y -= 0.25f * ct.y;
      den += Wi * 0.25f * (c.x * c.x + c.y * c.y) * t.z;
    }
    const float4 t = ends[4 * 32 + lane];
    num.x += t.x;
    num.y += t.y;
    den += Wi * t.z;
    Q = make_float2(Wi * num.x / den, Wi * num.y / den);
  }
  const float2 q = fine ? cmul(make_float2(cre, cim), Q) : make_float2(-Q.x, -Q.y);
  float2 v = make_float2((b.x + q.x) * dinv, (b.y + q.y) * dinv);
  col[(rows - 1) * step] = v;
  for (int m = rows - 2; m >= 0; --m) {   // x_m = (b'_m / w + x_{m+1}) / (1 + e_m)
    const float2 f = x[m * 32];
    const float g = mult[m * 32];
    v = make_float2(fmaf(f.x, 1.0f / w, v.x) * g, fmaf(f.y, 1.0f / w, v.y) * g);
    col[m * step] = v;
  }
}

template <typename K>
bool set_smem(K kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
}

}  // namespace

// Square power-of-two planes, columns that the shared memory of the z solve
// holds, and wall axes of known ends: the pressure's single Neumann component
// or no-slip velocity components.
bool spectral_supported(const LevelDev& L0) {
  for (int ci = 0; ci < L0.ncomp; ++ci) {
    const CompDev& c = L0.c[ci];
    if (c.nx != c.ny || c.nx != L0.c[0].nx || c.nx < 4 || c.nx > 128 || (c.nx & (c.nx - 1)) != 0 || c.nz < 2)
      return false;
    if (c.zkind == kAxisCellNeu ? L0.ncomp != 1 : c.zkind != kAxisCellDir && c.zkind != kAxisVertex) return false;
    if ((size_t)c.nz * kThomasThreads * 3 * sizeof(float) > 200 * 1024 || c.nz > 257) return false;
  }
  return true;
}

size_t spectral_bytes(const LevelDev& L0) { return (size_t)L0.size * sizeof(float2); }

cudaError_t spectral_inner_solve(const LevelDev& L0, const float* r, float* delta, void* spectrum, cudaStream_t st) {
  const CompDev& c = L0.c[0];
  const int n = c.nx;
  int logn = 0;
  while ((1 << logn) < n) ++logn;
  float2* S = (float2*)spectrum;
  WallAxes wa{};
  int planes = 0, nz = 0;
  for (int ci = 0; ci < L0.ncomp; ++ci) {   // the components' planes follow one another in the field
    wa.nz[ci] = L0.c[ci].nz;
    wa.first[ci] = planes;
    wa.end[ci] = L0.c[ci].zkind == kAxisCellDir ? 3.0f : L0.c[ci].zkind == kAxisCellNeu ? 1.0f : 2.0f;
    planes += L0.c[ci].nz;
    nz = nz > L0.c[ci].nz ? nz : L0.c[ci].nz;
  }
  const bool singular = c.zkind == kAxisCellNeu;
  const size_t fsm = (size_t)(n * n + n / 2) * sizeof(float2);
  // at least one warp per block (the (0, 0) block scans with a full warp)
  const int tthreads = n < 32 ? 32 : (n < kThomasThreads ? n : kThomasThreads);
  const int per_row = n / tthreads > 0 ? n / tthreads : 1;
  // per thread: FP32 c' and the column (float2)
  const size_t tsm = (size_t)nz * tthreads * 3 * sizeof(float);
  static std::atomic<int> ready[64];
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !ready[dev].load()) {
    if (!set_smem(k_spec_forward, 227 * 1024) || !set_smem(k_spec_inverse, 227 * 1024) ||
        !set_smem(k_spec_thomas<true>, 227 * 1024) || !set_smem(k_spec_thomas<false>, 227 * 1024))
      return cudaGetLastError();
    ready[dev].store(1);
  }
  prof::Scope ps(SELM_K_PROJECTION, st);
  k_spec_forward<<<planes, kSpecThreads, fsm, st>>>(r, S, n, logn);
  if (singular)
    k_spec_thomas<true><<<n * per_row + 1, tthreads, tsm, st>>>(S, n, logn, wa, (float)(1.0 / c.s));
  else
    k_spec_thomas<false><<<dim3(n * per_row, L0.ncomp), tthreads, tsm, st>>>(S, n, logn, wa, (float)(1.0 / c.s));
  k_spec_inverse<<<planes, kSpecThreads, fsm, st>>>(S, delta, n, logn);
  return cudaGetLastError();
}

bool mac_spectral_supported(int dim, int n, int K) {
  return dim == 3 && n >= 4 && n <= 64 && (n & (n - 1)) == 0 && K >= 0 && K <= n;
}

size_t mac_spectral_bytes(int n, int K) { return (size_t)n * n * (8 * K + n - K) * sizeof(float2); }

cudaError_t mac_spectral_solve(int n, int K, const double* r, double* z, const double* rr, void* spectrum,
                               cudaStream_t st) {
  MacSpec M{};
  M.n = n;
  while ((1 << M.logn) < n) ++M.logn;
  M.nf = 2 * K;
  M.nb = n - K;
  M.fine = (float2*)spectrum;
  M.base = M.fine + (size_t)M.nf * 4 * n * n;
  const int np = K > 0 ? 2 * n : n;
  const size_t fsm = (size_t)(np * np + np / 2) * sizeof(float2);
  const size_t csm = (size_t)(4 * M.nf + M.nb) * 32 * 3 * sizeof(float) + 5 * 32 * sizeof(float4);
  static std::atomic<int> ready[64];
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !ready[dev].load()) {
    if (!set_smem(k_mac_forward, 227 * 1024) || !set_smem(k_mac_inverse, 227 * 1024) ||
        !set_smem(k_mac_columns, 227 * 1024))
      return cudaGetLastError();
    if (dev >= 0 && dev < 64) ready[dev].store(1);
  }
  prof::Scope ps(SELM_K_PROJECTION, st);
  k_mac_forward<<<M.nf + M.nb, kSpecThreads, fsm, st>>>(M, r, rr);
  k_mac_columns<<<n * ((n + 31) / 32) + 1, 160, csm, st>>>(M);
  k_mac_inverse<<<M.nf + M.nb, kSpecThreads, fsm, st>>>(M, z, rr);
  return cudaGetLastError();
}

}  // namespace selm
