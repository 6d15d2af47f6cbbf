// Shared device definitions of the gbnfft CUDA library.
//
// Grid storage: the oversampled grid I_n is stored with cell l_t at array
// index l_t mod n_t, C order (dimension d-1 fastest).  With that layout the
// centred DFTs of Section 2 are plain cuFFT transforms.
//
// Points: after nfft_set_points every point j is described, in sorted order,
// by its original index perm[p], its in-bin cell offsets (packed) and its
// in-cell offsets delta_t = u_t - floor(u_t), u_t = n_t (x_t mod 1).  The
// subproblem list cuts every non-empty bin into runs of at most P points.
//
// Window taps: a point in cell c reaches cells c - m + s + i, i = 0..W-1,
// where (s, W) = (0, 2m+2) for the Gaussian and (1, 2m) for the Kaiser-Bessel
// window (whose weight is exactly zero at the two outer cells of the 2m + 2
// the method defines).  The distance u - l of tap i is delta + (m - s) - i.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace gbnfft {

constexpr int kMaxDim = 3;
constexpr int kMaxTaps = 32;

template <typename Real> struct Cplx;
template <> struct Cplx<float> { using type = float2; };
template <> struct Cplx<double> { using type = double2; };

template <typename C> __device__ __forceinline__ C cmake(double re, double im);
template <> __device__ __forceinline__ float2 cmake<float2>(double re, double im) { return make_float2((float)re, (float)im); }
template <> __device__ __forceinline__ double2 cmake<double2>(double re, double im) { return make_double2(re, im); }

// c + v w for a complex v and a real w: per component one round-to-nearest
// fma (as fmaf / fma); in FP32 both components in one paired instruction
// (FFMA2, sm_100 and later).
__device__ __forceinline__ float2 cmad(float2 v, float w, float2 c) { return __ffma2_rn(v, make_float2(w, w), c); }
__device__ __forceinline__ double2 cmad(double2 v, double w, double2 c) {
  return make_double2(fma(v.x, w, c.x), fma(v.y, w, c.y));
}
// v w, per component one round-to-nearest product (FP32: FMUL2).
__device__ __forceinline__ float2 cscale(float2 v, float w) { return __fmul2_rn(v, make_float2(w, w)); }
__device__ __forceinline__ double2 cscale(double2 v, double w) { return make_double2(v.x * w, v.y * w); }

// Window parameters, normalised so that psi(0) = 1 (the constant phi(0) is
// moved into the FP64 scaling factors on the host).  The shape parameter
// depends on sigma_t = n_t / N_t, so it is kept per dimension.
struct WindowDev {
  int kind;                 // 0 Gaussian, 1 Kaiser-Bessel, 2 B-spline, 3 sinc-power
  int m;                    // cut-off
  int shift;                // s: first tap is c - m + s
  int taps;                 // W
  double b[kMaxDim];        // shape parameter per dimension
  double kb_norm[kMaxDim];  // Kaiser-Bessel: 1 / (1 - exp(-2 b m)); B-spline: 1 / M_2m(0)
  float bf[kMaxDim];        // the same two, rounded to float once (FP32 kernels)
  float kb_normf[kMaxDim];
  float binvf[kMaxDim];     // 1 / b in float (FP32 Gaussian)
  // the window as polynomials (window_taps), per dimension [taps / 2][pairs];
  // null for the B-spline
  const float2* polyf[kMaxDim];
  const double2* polyd[kMaxDim];
};

// Coefficient pairs of the window's polynomials: degree 11 in FP32, 21 in
// FP64.  The Chebyshev coefficients of a window (psi(0) = 1) on a tap's unit
// interval that this leaves out add up to at most 4.1e-8 and 2.6e-16 (Gaussian,
// m = 1, sigma = 16; 1.5e-8 and 9e-18 at sigma = 2), and to 6e-9 and 6e-20 for
// the other windows and 1.4e-9 and 1.3e-19 from m = 2 on, over every sigma that
// a plan takes: less than an FP32 (FP64) tap near 1 is rounded by.
constexpr int kPolyF = 6;
constexpr int kPolyD = 11;

// psi(u) = phi(u / n) / phi(0) for the distance u (in cells).
//   Gaussian:       exp(-u^2 / b)
//   Kaiser-Bessel:  sinh(b z) / z * m / sinh(b m),  z = sqrt(m^2 - u^2), |u| < m
//   B-spline:       M_2m(u) / M_2m(0)           (window_psi_any only)
//   sinc-power:     sinc(pi b u)^(2m),  |u| < m
// The Kaiser-Bessel form is evaluated as
//   exp(-b u^2 / (z + m)) * m * ((1 - exp(-2 b z)) / z) * kb_norm
// so the large exponent b m cancels exactly instead of in floating point.
template <typename Real>
__device__ __forceinline__ Real window_psi(const WindowDev& w, int t, Real u);

// Centred cardinal B-spline M_order(u), |u| < order / 2, raised from the
// indicator of [0, 1) by the two-term recurrence of uniform B-splines
// (nonnegative terms only).  Only window_psi_any (the global kernels, which
// run every B-spline plan) calls it: the other kernels keep their registers.
template <typename Real>
__device__ __noinline__ Real cardinal_bspline_dev(int order, Real u) {
  const Real s = u + (Real)(order / 2);
  if (!(s > (Real)0 && s < (Real)order)) return (Real)0;
  Real v[kMaxTaps + 1];
  const int f = (int)floor(s);
  for (int i = 0; i <= order; ++i) v[i] = (Real)0;
  v[f] = (Real)1;
  for (int j = 2; j <= order; ++j) {
    const Real inv = (Real)1 / (Real)(j - 1);
    const int i0 = f - j + 1 > 0 ? f - j + 1 : 0, i1 = f < order - j ? f : order - j;
    for (int i = i0; i <= i1; ++i) {
      const Real si = s - (Real)i;
      v[i] = (si * v[i] + ((Real)j - si) * v[i + 1]) * inv;
    }
  }
  return v[0];
}

// FP32: the hardware reciprocal square root, reciprocal and exponential
// (a few ulp each) in place of correctly rounded division, sqrt and expm1.
// At the window's peak the result is exp(0) = 1 times 1/z, within 2 ulp;
// the exponentials' argument-proportional error and the cancellation in
// 1 - exp(-2 b z) for small z act only where the weight is far below one
// (at |u| = m it is about 2 b m exp(-b m)), so every weight stays within a
// few 1e-8 of psi(u) in absolute terms, the size of its FP32 rounding.
template <>
__device__ __forceinline__ float window_psi<float>(const WindowDev& w, int t, float u) {
  if (w.kind == 0) return expf(-(u * u) * w.binvf[t]);
  const float b = w.bf[t];
  const float m = (float)w.m;
  const float u2 = u * u;
  const float m2 = m * m;
  if (!(u2 < m2)) return 0.0f;
  if (w.kind == 3) {
    // sinc(pi c u) with c = b: sinpi needs no large-argument reduction
    const float zz = b * u;
    const float sc = zz != 0.0f ? __fdividef(sinpif(zz), 3.14159265358979f * zz) : 1.0f;
    const float r = sc * sc;
    float p = 1.0f;
    for (int i = 0; i < w.m; ++i) p *= r;
    return p;
  }
  const float z2 = m2 - u2;
  const float rz = rsqrtf(z2);   // 1 / z
  const float z = z2 * rz;
  const float e = __expf(__fdividef(-b * u2, z + m));
  const float s = (1.0f - __expf(-2.0f * b * z)) * rz;
  return e * m * s * w.kb_normf[t];
}

template <>
__device__ __forceinline__ double window_psi<double>(const WindowDev& w, int t, double u) {
  const double b = w.b[t];
  if (w.kind == 0) return exp(-(u * u) / b);
  const double m = (double)w.m;
  const double u2 = u * u;
  const double m2 = m * m;
  if (!(u2 < m2)) return 0.0;
  if (w.kind == 3) {
    const double zz = b * u;
    const double sc = zz != 0.0 ? sinpi(zz) / (3.141592653589793 * zz) : 1.0;
    const double r = sc * sc;
    double p = 1.0;
    for (int i = 0; i < w.m; ++i) p *= r;
    return p;
  }
  const double z = sqrt(m2 - u2);
  const double e = exp(-b * u2 / (z + m));
  const double s = -expm1(-2.0 * b * z) / z;
  return e * m * s * w.kb_norm[t];
}

// The W taps of a point at offset delta in [0, 1) of its cell, w[i] =
// psi(delta + m - s - i), for the windows that are smooth inside their
// support (all but the B-spline).  Tap i over its unit interval is a
// polynomial in x = 2 delta - 1, and the window's symmetry makes tap W - 1 - i
// the same one in -x: with E and O its even and odd parts in x^2, the two taps
// are E + x O and E - x O.  Two FP32 taps cost 5 paired FMAs and 2 FMAs; the
// formula (window_psi) costs 4 special-function instructions and about 16
// others per tap, in FP64 about 110 FP64 operations against 11.  x is exact
// to 2^-24 where u = delta + m - s would round at the size of m.

// A window cut at |u| = m is 0 from there on: its outer taps where u, rounded
// as window_psi rounds it, reaches the cut (delta = 0, or within rounding of a
// cell's ends).
template <int W, typename Real>
__device__ __forceinline__ void cut_taps(const WindowDev& win, Real delta, Real* w) {
  if (win.kind == 0) return;
  const Real base = delta + (Real)(win.m - win.shift), last = base - (Real)(W - 1), m2 = (Real)win.m * (Real)win.m;
  if (!(base * base < m2)) w[0] = (Real)0;
  if (!(last * last < m2)) w[W - 1] = (Real)0;
}

template <int W>
__device__ __forceinline__ void window_taps(const WindowDev& win, int t, float delta, float* w) {
  const float4* c = reinterpret_cast<const float4*>(win.polyf[t]);
  const float x = fmaf(2.0f, delta, -1.0f);
  const float s = x * x;
#pragma unroll
  for (int i = 0; i < W / 2; ++i) {
    float2 p;
#pragma unroll
    for (int k = kPolyF / 2 - 1; k >= 0; --k) {
      const float4 v = __ldg(c + i * (kPolyF / 2) + k);
      if (k == kPolyF / 2 - 1) p = make_float2(v.z, v.w);
      else p = cmad(p, s, make_float2(v.z, v.w));
      p = cmad(p, s, make_float2(v.x, v.y));
    }
    w[i] = fmaf(x, p.y, p.x);
    w[W - 1 - i] = fmaf(-x, p.y, p.x);
  }
  cut_taps<W>(win, delta, w);
}
template <int W>
__device__ __forceinline__ void window_taps(const WindowDev& win, int t, double delta, double* w) {
  const double2* c = win.polyd[t];
  const double x = fma(2.0, delta, -1.0);
  const double s = x * x;
#pragma unroll
  for (int i = 0; i < W / 2; ++i) {
    double2 p = __ldg(c + i * kPolyD + kPolyD - 1);
#pragma unroll
    for (int k = kPolyD - 2; k >= 0; --k) p = cmad(p, s, __ldg(c + i * kPolyD + k));
    w[i] = fma(x, p.y, p.x);
    w[W - 1 - i] = fma(-x, p.y, p.x);
  }
  cut_taps<W>(win, delta, w);
}

// One of them, tap k (kernels whose lanes take different taps).
__device__ __forceinline__ double window_tap(const WindowDev& win, int t, double delta, int k, int taps) {
  const bool mirror = k >= taps / 2;
  const double2* c = win.polyd[t] + (mirror ? taps - 1 - k : k) * kPolyD;
  const double x = fma(2.0, delta, -1.0);
  const double s = x * x;
  double2 p = __ldg(c + kPolyD - 1);
#pragma unroll
  for (int q = kPolyD - 2; q >= 0; --q) p = cmad(p, s, __ldg(c + q));
  if (win.kind != 0) {
    const double u = delta + (double)(win.m - win.shift) - (double)k, m = (double)win.m;
    if (!(u * u < m * m)) return 0.0;
  }
  return fma(mirror ? -x : x, p.y, p.x);
}

// Every window, the B-spline included (global kernels only).
template <typename Real>
__device__ __forceinline__ Real window_psi_any(const WindowDev& w, int t, Real u) {
  if (w.kind == 2) return cardinal_bspline_dev<Real>(2 * w.m, u) * (Real)w.kb_norm[t];
  return window_psi<Real>(w, t, u);
}

// One subproblem: a run of sorted points inside one bin of one item.
struct SubProblem {
  int bin;     // bin id within the item
  int start;   // first sorted position
  int count;
  int item;
  int form;    // how its points are interpolated (pencils)
};
constexpr int kFormGrid = 0;    // few points per plane: a warp per point straight from the grid
constexpr int kFormSlab = 1;    // a warp per point from a slab of planes
constexpr int kFormDense = 2;   // points share cells (kDenseRun of them per cell or more): a thread per point from a slab

struct GridGeom {
  int d;
  int n[kMaxDim];            // oversampled sizes (unused dims = 1)
  int bin[kMaxDim];          // bin edges (unused dims = 1)
  int nbins[kMaxDim];        // bins per dimension
  int tile[kMaxDim];         // bin + W - 1 (unused dims = 1)
  int64_t grid_cells;        // prod n
  int tile_cells;            // prod tile
  int fine;                  // sort keys per bin: 1, or its planes (a pencil's points in their order)
};

// One transform of a batch (a single plan is a batch of one), as the
// kernels see it.  Items of one kernel launch share d, the taps and the bin
// edges (so the tile shape); n, M, the window shape and the pointers may
// differ.
struct ItemDev {
  GridGeom geom;
  WindowDev win;
  int N[kMaxDim];
  int64_t NN;                  // |I_N|
  int64_t M;
  int nrhs;
  int bin_offset;              // first global bin id of the item
  int key_offset;              // first sort key of the item (geom.fine keys per bin)
  int64_t point_offset;        // first point of the item in the unsorted concatenation
  const double* x;             // M x d points (read by nfft_set_points only)
  void* grid;                  // nrhs grids of geom.grid_cells
  const double* inv_c[kMaxDim];
  const void* in;              // per call: f (adjoint) or fhat (forward), nrhs blocks
  void* out;                   // per call: fhat (adjoint) or f (forward)
};

// Point data after sorting (all arrays indexed by sorted position).
template <typename Real>
struct SortedPoints {
  const int* perm;           // sorted position -> point index within its item
  const uint32_t* local;     // packed in-bin cell offsets
  const Real* delta[kMaxDim];
  const SubProblem* subs;
  const int* sub_start;      // exclusive scan of subproblems per global bin
  const int* num_subs;       // device scalar: all subproblems
  const int* bin_count;      // points per global bin
  const int* grid_points;   // per item: points of its kFormGrid subproblems (pencils)
  const int* bin_start;      // first sorted position per global bin
};

// Pack / unpack of in-bin offsets: 32 bits split evenly over d dimensions.
__host__ __device__ __forceinline__ int local_bits(int d) { return d == 1 ? 32 : (d == 2 ? 16 : 10); }

__device__ __forceinline__ int unpack_local(uint32_t v, int d, int t) {
  if (d == 1) return (int)v;
  const int bits = local_bits(d);
  return (int)((v >> (bits * t)) & ((1u << bits) - 1u));
}

__device__ __forceinline__ int wrap_mod(int v, int n) {
  v %= n;
  return v < 0 ? v + n : v;
}

}  // namespace gbnfft
