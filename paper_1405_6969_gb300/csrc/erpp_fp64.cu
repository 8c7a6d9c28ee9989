// erpp_fp64.cu -- the plain FP64 form of the gather and the scatter, and the
// gather of the velocity with its Laplacian for the general force.
//
// Particles in index order, no binning: a block evaluates the per-axis weights
// of Sec. 2.4's truncated Gaussian of its particles in double precision, a
// thread per particle and axis, then a warp walks each particle's window.  The
// gather reads the grid from global memory; the scatter adds fscale * D_p W_p(j) (fscale = -1/rho_f for
// the source) into the zeroed grid with FP64 global atomics.  This is the
// straightforward double-precision implementation the FP32 tile kernels are
// measured against.
//
// The Laplacian gather (ERPP_FULL_FORCE, Eq. force_particle) walks the same
// window with the weights' second derivatives as well; on FP32 grids its
// windows are computed once per particle and its particles visited in
// cell-block order.
#include <cuda_runtime.h>

#include "erpp_internal.cuh"

namespace {

constexpr int kWarps = 8;
constexpr int kMaxW = 32;
constexpr int kRowBuf = 64;  // row weights a warp keeps at a time

// Sum of a window's weights in four interleaved parts, pairwise at the end: for up to
// 8 nodes the order of a warp's butterfly.  One after the other, and with the
// quotients below as products with the rounded reciprocal alone, velocities gathered
// from 64^3 nodes were 2.7e-16 off (rms, against sums in more than 64 bits) instead
// of 2.0e-16 (1.9e-16 with a division per node); the FP64 step of 100k particles in
// 128^3 nodes takes 561 us for it, not 555.
struct WindowSum {
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  __device__ __forceinline__ void add(double v) {
    const double t = s[0] + v;
    s[0] = s[1];
    s[1] = s[2];
    s[2] = s[3];
    s[3] = t;
  }
  __device__ __forceinline__ double total() const { return (s[0] + s[2]) + (s[1] + s[3]); }
};

// What a window's weights are multiplied by, as a high and a low part: the quotient
// by dx times their sum rounded once or twice (a division per node takes the FP64
// pipe eight times as long).
struct WindowScale {
  double hi, lo;
};
__device__ __forceinline__ WindowScale window_scale(const erpp_kparams& kp, int a, double sum) {
  if (!kp.normalize) return {kp.raw_norm1, 0.0};
  const double den = kp.dx[a] * sum, r = 1.0 / den;
  return {r, fma(-r, den, 1.0) * r};
}
__device__ __forceinline__ double scaled(double e, const WindowScale& q) {
  return fma(e, q.hi, e * q.lo);
}

// Weights of one axis of a particle (raw or normalised), one thread: w[0..nw)
// stored with stride ws, the rest of the xs slots not written; returns nw (0 on
// an invalid position).
__device__ int axis_weights_f64(const erpp_kparams& kp, int a, double x, double* w, int ws,
                                int* jlo, uint32_t* err) {
  if (!(x >= 0.0 && x < kp.L[a])) {
    erpp_set_err(err, ERPP_ERRBIT_RANGE);
    return 0;
  }
  const erpp_axis_win aw =
      erpp_axis_window_lean(x, kp.inv_dx[a], kp.cp[a], kp.cp_int[a], kp.cp_frac[a]);
  const int nw = aw.hi - aw.lo + 1;
  if (nw > kp.xs || nw < 1) {
    erpp_set_err(err, ERPP_ERRBIT_BOUNDS);
    return 0;
  }
  const double s = __dmul_rn(x, kp.inv_dx[a]);
  WindowSum sum;
  for (int k = 0; k < nw; ++k) {
    const double d = ((double)(aw.lo + k) - s) * kp.dx[a];
    const double q = d * d;
    // -q / (2 sigma_R^2) by the reciprocal's high and low parts
    const double e = exp(fma(q, kp.gauss_hi, q * kp.gauss_lo));
    w[k * ws] = e;
    sum.add(e);
  }
  const WindowScale scale = window_scale(kp, a, sum.total());
  for (int k = 0; k < nw; ++k) w[k * ws] = scaled(w[k * ws], scale);
  *jlo = aw.lo;
  return nw;
}

// Particles of a block of the plain kernels: 32, or 8 where there are few (plain_few).
constexpr int kPlainMany = 32, kPlainFew = 8;

// Doubles that keep the weights and windows of a block of P particles between the
// gather and the source of one step.
__host__ __device__ constexpr size_t kept_doubles(int xs, int P) { return (size_t)3 * (xs + 1) * P; }

// A block's particles: window starts and lengths per axis (length 0: invalid); where
// they are few, the positions in units of the spacing and the weights' scales.  The
// weights are w[axis][k][particle], P + 1 apart in k.
template <int P>
struct Plain {
  int jlo[3][P], nw[3][P];
  double s[3][P];
  WindowScale scale[3][P];
};

// The weights of a block's particles, called by the whole block (it ends behind a
// barrier).  Many particles: a thread evaluates an axis of a particle.  Few: the
// exponentials by a thread each, between barriers, for a block would wait for xs of
// them one after the other; the same products and sums in the same order.
template <int P>
__device__ __forceinline__ void plain_weights(const erpp_kparams& kp, int64_t p0, int np,
                                              const double* __restrict__ x0,
                                              const double* __restrict__ x1,
                                              const double* __restrict__ x2, double* w,
                                              Plain<P>& sh, const double* __restrict__ kept,
                                              uint32_t* err) {
  constexpr int kS = P + 1;
  if (kept) {
    // evaluated by the step's gather at the same positions
    const double* src = kept + (size_t)blockIdx.x * kept_doubles(kp.xs, P);
    for (int i = threadIdx.x; i < 3 * kp.xs * P; i += blockDim.x)
      w[(i / P) * kS + (i & (P - 1))] = src[i];
    const int2* win = reinterpret_cast<const int2*>(src + 3 * kp.xs * P);
    for (int i = threadIdx.x; i < 3 * P; i += blockDim.x) {
      const int a = i / P, p = i & (P - 1);
      const int2 v = win[i];
      sh.jlo[a][p] = v.x;
      sh.nw[a][p] = v.y;
    }
    __syncthreads();
    return;
  }
  if (P == kPlainMany) {
    for (int i = threadIdx.x; i < 3 * P; i += blockDim.x) {
      const int a = i / P, p = i & (P - 1);
      if (p >= np) continue;
      const double x = a == 0 ? x0[p0 + p] : (a == 1 ? x1[p0 + p] : x2[p0 + p]);
      int lo = 0;
      sh.nw[a][p] = axis_weights_f64(kp, a, x, w + a * kp.xs * kS + p, kS, &lo, err);
      sh.jlo[a][p] = lo;
    }
    __syncthreads();
    return;
  }
  for (int i = threadIdx.x; i < 3 * P; i += blockDim.x) {
    const int a = i / P, p = i & (P - 1);
    int lo = 0, nw = 0;
    double s = 0.0;
    if (p < np) {
      const double x = a == 0 ? x0[p0 + p] : (a == 1 ? x1[p0 + p] : x2[p0 + p]);
      if (!(x >= 0.0 && x < kp.L[a])) {
        erpp_set_err(err, ERPP_ERRBIT_RANGE);
      } else {
        const erpp_axis_win aw =
            erpp_axis_window_lean(x, kp.inv_dx[a], kp.cp[a], kp.cp_int[a], kp.cp_frac[a]);
        lo = aw.lo;
        nw = aw.hi - aw.lo + 1;
        if (nw > kp.xs || nw < 1) {
          erpp_set_err(err, ERPP_ERRBIT_BOUNDS);
          nw = 0;
        }
        s = __dmul_rn(x, kp.inv_dx[a]);
      }
    }
    sh.jlo[a][p] = lo;
    sh.nw[a][p] = nw;
    sh.s[a][p] = s;
  }
  __syncthreads();
  const int all = 3 * kp.xs * P;
  for (int i = threadIdx.x; i < all; i += blockDim.x) {
    const int r = i / P, p = i & (P - 1);
    const int a = r >= 2 * kp.xs ? 2 : (r >= kp.xs ? 1 : 0), k = r - a * kp.xs;
    if (k >= sh.nw[a][p]) continue;
    const double d = ((double)(sh.jlo[a][p] + k) - sh.s[a][p]) * kp.dx[a];
    const double q = d * d;
    // -q / (2 sigma_R^2) by the reciprocal's high and low parts
    w[r * kS + p] = exp(fma(q, kp.gauss_hi, q * kp.gauss_lo));
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 3 * P; i += blockDim.x) {
    const int a = i / P, p = i & (P - 1);
    WindowSum sum;
    for (int k = 0; k < sh.nw[a][p]; ++k) sum.add(w[(a * kp.xs + k) * kS + p]);
    sh.scale[a][p] = window_scale(kp, a, sum.total());
  }
  __syncthreads();
  for (int i = threadIdx.x; i < all; i += blockDim.x) {
    const int r = i / P, p = i & (P - 1);
    const int a = r >= 2 * kp.xs ? 2 : (r >= kp.xs ? 1 : 0);
    if (r - a * kp.xs < sh.nw[a][p]) w[r * kS + p] = scaled(w[r * kS + p], sh.scale[a][p]);
  }
  __syncthreads();
}

__device__ __forceinline__ int wrap_idx(int j, int n) {
  return j < 0 ? j + n : (j >= n ? j - n : j);
}

// A warp's walk over the window of one particle: lanes (kx, row), nwx lanes a
// row and 32 / nwx rows at a time; wyz[] holds the products of the rows'
// weights (written here), f(lane's weight e_x, row weight, node) sees every node
// of the window once.
template <int P, typename F>
__device__ __forceinline__ void plain_walk(const erpp_kparams& kp, const double* w,
                                           const Plain<P>& sh, int p, double* wyz, F f) {
  constexpr int kPlainS = P + 1;
  const int (*jlo)[P] = sh.jlo;
  const int (*nw)[P] = sh.nw;
  const int lane = threadIdx.x & 31;
  const int nx = nw[0][p], ny = nw[1][p], nz = nw[2][p], rows = ny * nz;
  const double* wy = w + kp.xs * kPlainS + p;
  const double* wz = wy + kp.xs * kPlainS;
  const int R = nx <= 32 ? 32 / nx : 1;
  const int kx = lane % nx, r0 = lane / nx;
  const bool on = r0 < R;
  const double wx = w[kx * kPlainS + p];
  const int jx = wrap_idx(jlo[0][p] + kx, kp.n[0]);
  // row products in passes of as many rows as the buffer holds
  for (int c0 = 0; c0 < rows; c0 += kRowBuf) {
    const int nr = min(kRowBuf, rows - c0);
    __syncwarp();
    for (int r = lane; r < nr; r += 32) {
      const int z = (c0 + r) / ny, y = (c0 + r) - z * ny;
      wyz[r] = wy[y * kPlainS] * wz[z * kPlainS];
    }
    __syncwarp();
    int z = (c0 + r0) / ny, y = (c0 + r0) - z * ny;
    for (int r = r0; r < nr && on; r += R) {
      const size_t node = ((size_t)wrap_idx(jlo[2][p] + z, kp.n[2]) * kp.n[1] +
                           (size_t)wrap_idx(jlo[1][p] + y, kp.n[1])) * kp.n[0] + jx;
      f(wx, wyz[r], node);
      y += R;
      while (y >= ny) {
        y -= ny;
        ++z;
      }
    }
  }
}

// A block takes P particles: their weights first, then a warp per particle.  The FP64 pipe bounds both kernels (2
// lanes a clock on an SM, whatever the number of active lanes of an
// instruction): per particle the exponentials are evaluated once per node and
// axis instead of by all 32 lanes of a warp, the row weights once per row, and
// a node costs one operation per component.  100k particles, 216 nodes each, on
// 128^3: gather 1585 -> 302 us (100 us of it the weights), source 1480 -> 210 us
// with the weights that the step's gather leaves in w64, 290 us without.
template <int P>
__global__ void __launch_bounds__(kWarps * 32) k_gather_f64(erpp_kparams kp, int64_t n,
                                                            const double* __restrict__ x0,
                                                            const double* __restrict__ x1,
                                                            const double* __restrict__ x2,
                                                            const double* __restrict__ u,
                                                            double* up0, double* up1, double* up2,
                                                            double* __restrict__ keep,
                                                            uint32_t* err) {
  extern __shared__ double plain_smem[];
  __shared__ Plain<P> sh;
  constexpr int kPlainS = P + 1;
  double* const w = plain_smem;  // [3][xs][kPlainS]
  double* const rowbuf = w + 3 * kp.xs * kPlainS;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t p0 = (int64_t)blockIdx.x * P;
  const int np = (int)min((int64_t)P, n - p0);
  plain_weights<P>(kp, p0, np, x0, x1, x2, w, sh, nullptr, err);
  if (keep) {
    double* dst = keep + (size_t)blockIdx.x * kept_doubles(kp.xs, P);
    for (int i = threadIdx.x; i < 3 * kp.xs * P; i += blockDim.x)
      dst[i] = w[(i / P) * kPlainS + (i & (P - 1))];
    int2* win = reinterpret_cast<int2*>(dst + 3 * kp.xs * P);
    for (int i = threadIdx.x; i < 3 * P; i += blockDim.x)
      win[i] = make_int2(sh.jlo[i / P][i & (P - 1)], sh.nw[i / P][i & (P - 1)]);
  }
  const size_t nn = (size_t)kp.n[0] * kp.n[1] * kp.n[2];
  for (int p = warp; p < np; p += kWarps) {
    double a0 = 0.0, a1 = 0.0, a2 = 0.0;
    if (sh.nw[0][p] > 0 && sh.nw[1][p] > 0 && sh.nw[2][p] > 0) {
      double wx = 0.0;
      plain_walk<P>(kp, w, sh, p, rowbuf + warp * kRowBuf,
                 [&](double wl, double wr, size_t node) {
                   wx = wl;
                   a0 = fma(wr, __ldg(u + node), a0);
                   a1 = fma(wr, __ldg(u + nn + node), a1);
                   a2 = fma(wr, __ldg(u + 2 * nn + node), a2);
                 });
      wx *= kp.dV;
      a0 *= wx;
      a1 *= wx;
      a2 *= wx;
    }
    // sums over the lanes: two values change hands, then one
    const bool h16 = lane & 16, h8 = lane & 8;
    const double s0 = (h16 ? a2 : a0) + __shfl_xor_sync(0xffffffffu, h16 ? a0 : a2, 16);
    const double b1 = __shfl_xor_sync(0xffffffffu, a1, 16);
    const double s1 = a1 + b1;  // in both halves
    // lanes below 16: s0 = component 0; above: component 2; s1 everywhere
    double v = (h8 ? s1 : s0) + __shfl_xor_sync(0xffffffffu, h8 ? s0 : s1, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) up0[p0 + p] = v + kp.shear_rate * x1[p0 + p];
    if (lane == 8) up1[p0 + p] = v;
    if (lane == 16) up2[p0 + p] = v;
  }
}

template <int P>
__global__ void __launch_bounds__(kWarps * 32) k_scatter_f64(erpp_kparams kp, int64_t n,
                                                             const double* __restrict__ x0,
                                                             const double* __restrict__ x1,
                                                             const double* __restrict__ x2,
                                                             const double* __restrict__ D0,
                                                             const double* __restrict__ D1,
                                                             const double* __restrict__ D2,
                                                             double fscale, double* S,
                                                             const double* __restrict__ kept,
                                                             uint32_t* err) {
  extern __shared__ double plain_smem[];
  __shared__ Plain<P> sh;
  constexpr int kPlainS = P + 1;
  double* const w = plain_smem;  // [3][xs][kPlainS]
  double* const rowbuf = w + 3 * kp.xs * kPlainS;
  const int warp = threadIdx.x >> 5;
  const int64_t p0 = (int64_t)blockIdx.x * P;
  const int np = (int)min((int64_t)P, n - p0);
  plain_weights<P>(kp, p0, np, x0, x1, x2, w, sh, kept, err);
  const size_t nn = (size_t)kp.n[0] * kp.n[1] * kp.n[2];
  for (int p = warp; p < np; p += kWarps) {
    if (!(sh.nw[0][p] > 0 && sh.nw[1][p] > 0 && sh.nw[2][p] > 0)) continue;
    const double wl = w[((threadIdx.x & 31) % sh.nw[0][p]) * kPlainS + p];
    const double f0 = fscale * D0[p0 + p] * wl, f1 = fscale * D1[p0 + p] * wl,
                 f2 = fscale * D2[p0 + p] * wl;
    plain_walk<P>(kp, w, sh, p, rowbuf + warp * kRowBuf, [&](double, double wr, size_t node) {
      atomicAdd(S + node, f0 * wr);
      atomicAdd(S + nn + node, f1 * wr);
      atomicAdd(S + 2 * nn + node, f2 * wr);
    });
  }
}

size_t plain_smem_bytes(const erpp_kparams& kp, int P) {
  return sizeof(double) * ((size_t)3 * kp.xs * (P + 1) + (size_t)kWarps * kRowBuf);
}

// Few particles: a warp for each, so that no warp walks one window after another
// while SMs are idle.  Interpolation with blocks of 32 and of 8 in us, windows of 6
// nodes: 1000 particles 27 and 14.5, 10k 48 and 39, 30k 108 and 97, 100k 301 and 311;
// of 9: 54 and 19, 99 and 80, 232 and 212, 667 and 685; of 31: 1131 and 294, 2150 and
// 1635, 5104 and 4486, 15086 and 14801.
constexpr int64_t kFewMost = 50000;
bool plain_few(int64_t n) { return n <= kFewMost; }

// Weights of one axis and their second derivatives in the particle
// coordinate (raw or normalised like axis_weights_f64), evaluated in FP64 and
// stored as T.  With d = (j - s) dx: dw/dx_p = w d / sig2,
// d2w/dx_p2 = w (d^2 / sig2^2 - 1 / sig2); for the normalised w~ = w / Z the
// quotient rule gives w~'' = w~ (B - 2 A m1 - m2 + 2 m1^2), A = d / sig2,
// B = d^2 / sig2^2 - 1 / sig2, m1 and m2 the w~-means of A and B.
// The window is decided in FP64 (the oracle's exact membership); the weights
// are evaluated in T from the FP64 offset of each node (FP64 arithmetic runs
// at a small fraction of the FP32 rate: FP32 contexts keep it to the window).
template <typename T>
__device__ int axis_weights_d2(const erpp_kparams& kp, int a, double x, T* w, T* w2, int* jw,
                               uint32_t* err) {
  const int lane = threadIdx.x & 31;
  if (!(x >= 0.0 && x < kp.L[a])) {
    if (lane == 0) erpp_set_err(err, ERPP_ERRBIT_RANGE);
    return 0;
  }
  double s, lo, hi;
  erpp_axis_window(x, kp.inv_dx[a], kp.cp[a], &s, &lo, &hi);
  const int nw = (int)(hi - lo) + 1;
  if (nw > kMaxW || nw < 1) {
    if (lane == 0) erpp_set_err(err, ERPP_ERRBIT_BOUNDS);
    return 0;
  }
  const T sig2 = (T)kp.sig2;
  const T dxa = (T)kp.dx[a];
  T wv = T(0), A = T(0), B = T(0);
  if (lane < nw) {
    const T d = (T)((lo + (double)lane) - s) * dxa;
    wv = (T)kp.raw_norm1 * exp(-(d * d) / (T(2) * sig2));
    A = d / sig2;
    B = d * d / (sig2 * sig2) - T(1) / sig2;
  }
  T w2v;
  if (kp.normalize) {
    T sum = wv;
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    wv = wv / (dxa * sum);
    T m1 = dxa * wv * A, m2 = dxa * wv * B;
    for (int o = 16; o > 0; o >>= 1) {
      m1 += __shfl_xor_sync(0xffffffffu, m1, o);
      m2 += __shfl_xor_sync(0xffffffffu, m2, o);
    }
    w2v = wv * (B - T(2) * A * m1 - m2 + T(2) * m1 * m1);
  } else {
    w2v = wv * B;
  }
  w[lane] = wv;
  w2[lane] = w2v;
  if (lane < nw) {  // wrapped node index (the window starts at most 15 nodes below 0)
    int j = (int)lo + lane;
    j = j < 0 ? j + kp.n[a] : (j >= kp.n[a] ? j - kp.n[a] : j);
    jw[lane] = j;
  }
  return nw;
}

// Gather of u and of its Laplacian in the particle position, warp per
// particle; products and sums in the grid's type.
template <typename T>
__global__ void __launch_bounds__(kWarps * 32) k_gather_faxen(
    erpp_kparams kp, int64_t n, const double* __restrict__ x0, const double* __restrict__ x1,
    const double* __restrict__ x2, const T* __restrict__ u, double* up0, double* up1,
    double* up2, double* lap, int64_t lap_stride, uint32_t* err) {
  __shared__ T w[kWarps][3][kMaxW];
  __shared__ T w2[kWarps][3][kMaxW];
  __shared__ int jw[kWarps][3][kMaxW];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t p = (int64_t)blockIdx.x * kWarps + warp;
  if (p >= n) return;
  const double xv[3] = {x0[p], x1[p], x2[p]};
  int nw[3];
  bool ok = true;
  for (int a = 0; a < 3; ++a) {
    nw[a] = axis_weights_d2<T>(kp, a, xv[a], w[warp][a], w2[warp][a], jw[warp][a], err);
    ok = ok && nw[a] > 0;
  }
  __syncwarp();
  T acc[3] = {T(0), T(0), T(0)}, lac[3] = {T(0), T(0), T(0)};
  const size_t nn = (size_t)kp.n[0] * kp.n[1] * kp.n[2];
  if (ok) {
    const int total = nw[0] * nw[1] * nw[2];
    for (int f = lane; f < total; f += 32) {
      const int kx = f % nw[0];
      const int t = f / nw[0];
      const int ky = t % nw[1];
      const int kz = t / nw[1];
      const size_t node = ((size_t)jw[warp][2][kz] * kp.n[1] + (size_t)jw[warp][1][ky]) *
                              kp.n[0] + (size_t)jw[warp][0][kx];
      const T wx = w[warp][0][kx], wy = w[warp][1][ky], wz = w[warp][2][kz];
      const T W = wx * wy * wz;
      const T K = w2[warp][0][kx] * wy * wz + wx * w2[warp][1][ky] * wz +
                  wx * wy * w2[warp][2][kz];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const T uv = u[c * nn + node];
        acc[c] += W * uv;
        lac[c] += K * uv;
      }
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c)
    for (int o = 16; o > 0; o >>= 1) {
      acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
      lac[c] += __shfl_xor_sync(0xffffffffu, lac[c], o);
    }
  if (lane == 0) {
    up0[p] = kp.dV * (double)acc[0] + kp.shear_rate * xv[1];
    up1[p] = kp.dV * (double)acc[1];
    up2[p] = kp.dV * (double)acc[2];
    lap[p] = kp.dV * (double)lac[0];
    lap[lap_stride + p] = kp.dV * (double)lac[1];
    lap[2 * lap_stride + p] = kp.dV * (double)lac[2];
  }
}

// FP32 grids: the FP64 windows once per particle (one thread each), so that
// the gather's lanes work in FP32 only.  win[i] = (j_lo x, y, z, packed
// lengths nw_x | nw_y << 8 | nw_z << 16, 0 when invalid), frac[i] = s - j_lo
// per axis (s = x N / L).
__global__ void __launch_bounds__(256) k_faxen_windows(erpp_kparams kp, int64_t n,
                                                       const double* __restrict__ x0,
                                                       const double* __restrict__ x1,
                                                       const double* __restrict__ x2,
                                                       int4* __restrict__ win,
                                                       float4* __restrict__ frac, uint32_t* err) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double xv[3] = {x0[i], x1[i], x2[i]};
  int lo[3], nw[3];
  float fr[3];
  bool ok = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (!(xv[a] >= 0.0 && xv[a] < kp.L[a])) {
      ok = false;
      erpp_set_err(err, ERPP_ERRBIT_RANGE);
      lo[a] = 0;
      nw[a] = 0;
      fr[a] = 0.f;
      continue;
    }
    double s, l, h;
    erpp_axis_window(xv[a], kp.inv_dx[a], kp.cp[a], &s, &l, &h);
    lo[a] = (int)l;
    nw[a] = (int)(h - l) + 1;
    fr[a] = (float)(s - l);
    if (nw[a] > kMaxW || nw[a] < 1) {
      ok = false;
      erpp_set_err(err, ERPP_ERRBIT_BOUNDS);
    }
  }
  win[i] = make_int4(lo[0], lo[1], lo[2], ok ? (nw[0] | (nw[1] << 8) | (nw[2] << 16)) : 0);
  frac[i] = make_float4(fr[0], fr[1], fr[2], 0.f);
}

// Weights and second derivatives of one axis from a precomputed window (FP32),
// with the same formulas as axis_weights_d2.
__device__ void axis_weights_d2_f32(const erpp_kparams& kp, int a, int lo, int nw, float r,
                                    float* w, float* w2, int* jw) {
  const int lane = threadIdx.x & 31;
  const float sig2 = (float)kp.sig2;
  const float dxa = (float)kp.dx[a];
  float wv = 0.f, A = 0.f, B = 0.f;
  if (lane < nw) {
    const float d = ((float)lane - r) * dxa;
    wv = (float)kp.raw_norm1 * expf(-(d * d) / (2.f * sig2));
    A = d / sig2;
    B = d * d / (sig2 * sig2) - 1.f / sig2;
  }
  float w2v;
  if (kp.normalize) {
    float sum = wv;
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    wv = wv / (dxa * sum);
    float m1 = dxa * wv * A, m2 = dxa * wv * B;
    for (int o = 16; o > 0; o >>= 1) {
      m1 += __shfl_xor_sync(0xffffffffu, m1, o);
      m2 += __shfl_xor_sync(0xffffffffu, m2, o);
    }
    w2v = wv * (B - 2.f * A * m1 - m2 + 2.f * m1 * m1);
  } else {
    w2v = wv * B;
  }
  w[lane] = wv;
  w2[lane] = w2v;
  if (lane < nw) {
    int j = lo + lane;
    j = j < 0 ? j + kp.n[a] : (j >= kp.n[a] ? j - kp.n[a] : j);
    jw[lane] = j;
  }
}

// Particles in the order perm (by cell block), so that neighbouring warps
// read neighbouring grid rows and share them in L2.
__global__ void __launch_bounds__(kWarps * 32) k_gather_faxen_f32(
    erpp_kparams kp, int64_t n, const double* __restrict__ x1, const int4* __restrict__ win,
    const float4* __restrict__ frac, const int32_t* __restrict__ perm,
    const float* __restrict__ u, double* up0, double* up1, double* up2, double* lap,
    int64_t lap_stride) {
  __shared__ float w[kWarps][3][kMaxW];
  __shared__ float w2[kWarps][3][kMaxW];
  __shared__ int jw[kWarps][3][kMaxW];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t i = (int64_t)blockIdx.x * kWarps + warp;
  if (i >= n) return;
  const int64_t p = perm[i];
  const int4 wi = win[p];
  const float4 fr = frac[p];
  const int nw[3] = {wi.w & 255, (wi.w >> 8) & 255, (wi.w >> 16) & 255};
  const bool ok = wi.w != 0;
  if (ok) {
    axis_weights_d2_f32(kp, 0, wi.x, nw[0], fr.x, w[warp][0], w2[warp][0], jw[warp][0]);
    axis_weights_d2_f32(kp, 1, wi.y, nw[1], fr.y, w[warp][1], w2[warp][1], jw[warp][1]);
    axis_weights_d2_f32(kp, 2, wi.z, nw[2], fr.z, w[warp][2], w2[warp][2], jw[warp][2]);
  }
  __syncwarp();
  float acc[3] = {0.f, 0.f, 0.f}, lac[3] = {0.f, 0.f, 0.f};
  const size_t nn = (size_t)kp.n[0] * kp.n[1] * kp.n[2];
  // lanes as (kx, row): lane kx = lane % nw_x of rows lane / nw_x, + R, ...
  // (R = 32 / nw_x rows per pass); the row's (ky, kz) advance without divisions
  const int R = 32 / nw[0];
  const int kx = lane % nw[0];
  int r0 = lane / nw[0];
  if (ok && r0 < R) {
    const float wx = w[warp][0][kx], w2x = w2[warp][0][kx];
    const size_t jx = (size_t)jw[warp][0][kx];
    int ky = r0 % nw[1], kz = r0 / nw[1];
    for (; kz < nw[2];) {
      const float wy = w[warp][1][ky], wz = w[warp][2][kz];
      const float w2y = w2[warp][1][ky], w2z = w2[warp][2][kz];
      const float W = wx * (wy * wz);
      const float K = w2x * (wy * wz) + wx * (w2y * wz + wy * w2z);
      const size_t node =
          ((size_t)jw[warp][2][kz] * kp.n[1] + (size_t)jw[warp][1][ky]) * kp.n[0] + jx;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float uv = u[c * nn + node];
        acc[c] += W * uv;
        lac[c] += K * uv;
      }
      ky += R;
      while (ky >= nw[1]) {
        ky -= nw[1];
        ++kz;
      }
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c)
    for (int o = 16; o > 0; o >>= 1) {
      acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
      lac[c] += __shfl_xor_sync(0xffffffffu, lac[c], o);
    }
  if (lane == 0) {
    up0[p] = kp.dV * (double)acc[0] + kp.shear_rate * x1[p];
    up1[p] = kp.dV * (double)acc[1];
    up2[p] = kp.dV * (double)acc[2];
    lap[p] = kp.dV * (double)lac[0];
    lap[lap_stride + p] = kp.dV * (double)lac[1];
    lap[2 * lap_stride + p] = kp.dV * (double)lac[2];
  }
}

}  // namespace

namespace erpp {

cudaError_t launch_gather_faxen(erpp_ctx* ctx, const void* u, int64_t n,
                                const double* const x[3], double* const up[3], cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int blocks = (int)((n + kWarps - 1) / kWarps);
  if (ctx->fp64) {
    ++ctx->launches;
    k_gather_faxen<double><<<blocks, kWarps * 32, 0, st>>>(
        ctx->kp, n, x[0], x[1], x[2], (const double*)u, up[0], up[1], up[2], ctx->ff_lap,
        ctx->cap, ctx->err);
  } else {
    // FP32 grids: the particles ordered by cell block, the windows once per
    // particle into the tile path's geometry arrays (free between steps),
    // then the FP32 gather
    cudaError_t e = sort_by_cell_block(ctx, n, x, st);
    if (e != cudaSuccess) return e;
    ctx->launches += 2;
    k_faxen_windows<<<(int)((n + 255) / 256), 256, 0, st>>>(ctx->kp, n, x[0], x[1], x[2],
                                                             ctx->geo_c, ctx->geo_t, ctx->err);
    k_gather_faxen_f32<<<blocks, kWarps * 32, 0, st>>>(ctx->kp, n, x[1], ctx->geo_c, ctx->geo_t,
                                                       ctx->w_perm, (const float*)u, up[0],
                                                       up[1], up[2], ctx->ff_lap, ctx->cap);
  }
  return cudaGetLastError();
}

cudaError_t launch_gather_f64(erpp_ctx* ctx, const double* u, int64_t n,
                              const double* const x[3], double* const up[3], bool keep,
                              cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int P = plain_few(n) ? kPlainFew : kPlainMany;
  auto kern = plain_few(n) ? k_gather_f64<kPlainFew> : k_gather_f64<kPlainMany>;
  ++ctx->launches;
  kern<<<(unsigned)((n + P - 1) / P), kWarps * 32, plain_smem_bytes(ctx->kp, P), st>>>(
      ctx->kp, n, x[0], x[1], x[2], u, up[0], up[1], up[2], keep ? ctx->w64 : nullptr, ctx->err);
  return cudaGetLastError();
}

// The step's weights (24 (xs + 1) bytes a particle) are kept where there is memory
// for them, made by the first step outside a capture; the source evaluates its own
// otherwise, with the same values.
bool w64_reserve(erpp_ctx* ctx) {
  if (ctx->w64) return true;
  if (ctx->w64_refused || ctx->cap <= 0) return false;
  // whole blocks of either size
  const size_t blocks = (size_t)((ctx->cap + kPlainMany - 1) / kPlainMany);
  if (cudaMalloc(&ctx->w64, sizeof(double) * kept_doubles(ctx->kp.xs, kPlainMany) * blocks) !=
      cudaSuccess) {
    cudaGetLastError();
    ctx->w64 = nullptr;
    ctx->w64_refused = true;
  }
  return ctx->w64 != nullptr;
}

bool w64_ready(erpp_ctx* ctx, cudaStream_t st) {
  return ctx->w64 || (!stream_captures(st) && w64_reserve(ctx));
}

cudaError_t launch_scatter_f64(erpp_ctx* ctx, int64_t n, const double* const x[3],
                               const double* const D[3], double fscale, double* S, bool kept,
                               cudaStream_t st) {
  const erpp_kparams& kp = ctx->kp;
  size_t nn = (size_t)kp.n[0] * kp.n[1] * kp.n[2];
  cudaError_t e = cudaMemsetAsync(S, 0, sizeof(double) * 3 * nn, st);
  if (e != cudaSuccess) return e;
  if (n <= 0) return cudaSuccess;
  const int P = plain_few(n) ? kPlainFew : kPlainMany;
  auto kern = plain_few(n) ? k_scatter_f64<kPlainFew> : k_scatter_f64<kPlainMany>;
  ++ctx->launches;
  kern<<<(unsigned)((n + P - 1) / P), kWarps * 32, plain_smem_bytes(kp, P), st>>>(
      kp, n, x[0], x[1], x[2], D[0], D[1], D[2], fscale, S, kept ? ctx->w64 : nullptr, ctx->err);
  return cudaGetLastError();
}

}  // namespace erpp
