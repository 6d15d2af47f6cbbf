// nfft_set_points kernels: argument reduction and counting sort of the points
// by spatial bin.  The bins are the on-device form of the paper's subcells
// (Section 3, Eqs. 7-8): a transform is the sum of the sub-transforms of any
// partition of the points, so every bin can be spread independently.
//
// All items of a batch are sorted in one pass: item i's points are global
// points [point_offsets[i], point_offsets[i+1]) and its bins are global bins
// [bin_offsets[i], bin_offsets[i+1]).
#include "kernels.h"

namespace gbnfft {

namespace {

// Largest i with offs[i] <= v (offs ascending, offs[0] = 0 <= v < offs[n]).
template <typename T>
__device__ __forceinline__ int find_item(const T* offs, int n, T v) {
  int lo = 0, hi = n;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (offs[mid] <= v) lo = mid;
    else hi = mid;
  }
  return lo;
}

// Reduce one coordinate to a cell c in [0, n) and the offset u - c of the
// cell coordinate u (Eq. 5 is 1-periodic in x, so any integer shift of x
// changes no exact sum), rounded once to Real.  An offset that rounds up to 1
// moves to the next cell with offset 0 (the same position).
//
// FP32 offsets: integer arithmetic throughout (FP64 is a slow pipe here).
// The fraction of |x| is taken from its mantissa bits as a 64-bit binary
// fraction F (exact for |x| >= 2^-12; below that the bits under 2^-64 are
// dropped), the fraction of x is F or 1 - F, and the 96-bit product n F
// splits into the cell (its bits 64 and up) and the offset (the 64 below),
// whose top 32 bits are rounded to float.
// FP64 offsets: the paper's reduction written out in FP64: x is brought into
// the torus [-1/2, 1/2) of Section 1 as x - floor(x + 1/2), u = n times
// that, c = floor(u) (then taken mod n) and the offset u - floor(u), so the
// offset carries only the rounding of that product, at most n/2 2^-53 cells
// (a reduction to [0, 1) would add the rounding of x + 1 for negative x, up
// to n 2^-53 cells).
__device__ __forceinline__ unsigned long long frac64(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff);
  const unsigned long long mant = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const int sh = 1075 - e;   // |x| = mant * 2^-sh
  unsigned long long f;
  if (e == 0 || sh <= 0) f = 0;           // zero, subnormal (taken as 0) or an integer
  else if (sh <= 64) f = mant << (64 - sh);
  else if (sh < 64 + 53) f = mant >> (sh - 64);
  else f = 0;
  if ((b >> 63) && f) f = 0ull - f;       // frac(-y) = 1 - frac(y)
  return f;
}

template <typename Real>
__device__ __forceinline__ void reduce_cell(double x, int n, int& c, Real& delta);
template <>
__device__ __forceinline__ void reduce_cell<float>(double x, int n, int& c, float& delta) {
  const unsigned long long f = frac64(x);
  const unsigned long long nn = (unsigned long long)n;
  c = (int)__umul64hi(f, nn);
  delta = __uint2float_rn((unsigned)((f * nn) >> 32)) * 2.3283064365386963e-10f;   // 2^-32
}
template <>
__device__ __forceinline__ void reduce_cell<double>(double x, int n, int& c, double& delta) {
  const double xw = x - floor(x + 0.5);
  const double u = (double)n * xw;
  const double cf = floor(u);
  c = (int)cf;
  if (c < 0) c += n;   // u >= -n/2 - 1 (x + 1/2 may round up to the next integer)
  delta = u - cf;
}

template <typename Real>
__device__ __forceinline__ void reduce_coord(double x, int n, int& c, Real& delta) {
  int ci;
  Real dr;
  reduce_cell<Real>(x, n, ci, dr);
  if (dr >= (Real)1) {
    dr = (Real)0;
    ci += 1;
  }
  if (ci >= n) ci -= n;
  c = ci;
  delta = dr;
}

__device__ __forceinline__ double load_coord(const double* x, int64_t j, int d, int t, bool& bad) {
  const double v = x[j * d + t];
  if (!isfinite(v)) {
    bad = true;
    return 0.0;
  }
  return v;
}

// Points per thread of the two point passes: a thread's points are kSortThreads
// apart (coalesced per slot) and every load and atomic of its points is
// issued before any result is used, so each thread keeps kSortPer memory
// requests in flight (the passes are bound by memory latency).
constexpr int kSortThreads = 256;
constexpr int kSortPer = 4;

template <typename Real>
__global__ void __launch_bounds__(kSortThreads) k_key_count(SortArgs s, int* __restrict__ key_count,
                                                            int2* __restrict__ key_rank) {
  const int64_t base = (int64_t)blockIdx.x * (kSortThreads * kSortPer) + threadIdx.x;
  const int lane = threadIdx.x & 31;
  int key[kSortPer];
  bool any_bad = false;
#pragma unroll
  for (int k = 0; k < kSortPer; ++k) {
    const int64_t gidx = base + (int64_t)k * kSortThreads;
    key[k] = -1;
    if (gidx < s.total_points) {
      const int item = find_item<int64_t>(s.point_offsets, s.n_items, gidx);
      const ItemDev& it = s.items[item];
      const int64_t j = gidx - it.point_offset;
      const double* x = s.x_override ? s.x_override : it.x;
      const GridGeom& g = it.geom;
      bool bad = false;
      int local = 0, plane = 0;
      for (int t = 0; t < g.d; ++t) {
        int c;
        Real dl;
        reduce_coord<Real>(load_coord(x, j, g.d, t, bad), g.n[t], c, dl);
        const int b = c / g.bin[t];
        if (t == 0) plane = c - b * g.bin[0];
        local = local * g.nbins[t] + b;
      }
      any_bad |= bad;
      key[k] = it.key_offset + local * g.fine + (g.fine > 1 ? plane : 0);
    }
  }
  if (any_bad) atomicOr(s.err, 1);
  // warp-aggregated ranks: lanes with the same bin share one atomic; the
  // atomics of all slots are in flight before their results are read
  unsigned peers[kSortPer];
  int got[kSortPer];
#pragma unroll
  for (int k = 0; k < kSortPer; ++k) {
    peers[k] = __match_any_sync(0xffffffffu, key[k]);
    got[k] = 0;
    if (key[k] >= 0 && lane == __ffs(peers[k]) - 1) got[k] = atomicAdd(&key_count[key[k]], __popc(peers[k]));
  }
#pragma unroll
  for (int k = 0; k < kSortPer; ++k) {
    const int first = __shfl_sync(peers[k], got[k], __ffs(peers[k]) - 1);
    const int64_t gidx = base + (int64_t)k * kSortThreads;
    if (key[k] >= 0) key_rank[gidx] = make_int2(key[k], first + __popc(peers[k] & ((1u << lane) - 1u)));
  }
}

template <typename Real>
__global__ void __launch_bounds__(kSortThreads) k_scatter(SortArgs s, const int* __restrict__ key_start,
                                                          const int2* __restrict__ key_rank, int* __restrict__ perm,
                                                          uint32_t* __restrict__ local, Real* d0, Real* d1, Real* d2) {
  const int64_t base = (int64_t)blockIdx.x * (kSortThreads * kSortPer) + threadIdx.x;
  Real* dst[3] = {d0, d1, d2};
  int2 br[kSortPer];
  int pos[kSortPer];
#pragma unroll
  for (int k = 0; k < kSortPer; ++k) {
    const int64_t gidx = base + (int64_t)k * kSortThreads;
    br[k] = gidx < s.total_points ? key_rank[gidx] : make_int2(-1, 0);
  }
#pragma unroll
  for (int k = 0; k < kSortPer; ++k) pos[k] = br[k].x >= 0 ? key_start[br[k].x] + br[k].y : -1;
#pragma unroll
  for (int k = 0; k < kSortPer; ++k) {
    const int64_t gidx = base + (int64_t)k * kSortThreads;
    if (pos[k] < 0) continue;
    const int item = find_item<int64_t>(s.point_offsets, s.n_items, gidx);
    const ItemDev& it = s.items[item];
    const int64_t j = gidx - it.point_offset;
    const double* x = s.x_override ? s.x_override : it.x;
    const GridGeom& g = it.geom;
    perm[pos[k]] = (int)j;
    if (g.fine > 1) continue;   // k_refine writes the rest
    bool bad = false;
    uint32_t packed = 0;
    const int bits = local_bits(g.d);
    for (int t = 0; t < g.d; ++t) {
      int c;
      Real dl;
      reduce_coord<Real>(load_coord(x, j, g.d, t, bad), g.n[t], c, dl);
      const uint32_t lc = (uint32_t)(c % g.bin[t]);
      packed |= (g.d == 1) ? lc : (lc << (bits * t));
      dst[t][pos[k]] = dl;
    }
    local[pos[k]] = packed;
  }
}

// The two point passes for one item of dimension D (single plans): the
// item's geometry is held in registers, and every coordinate of a thread's
// points is loaded before any is reduced (no item search, no reload of the
// item's fields per point).
template <int D>
struct OneItem {
  const double* x;
  int64_t poff;
  int koff, fine;
  int n[D], bw[D], nb[D];
  __device__ __forceinline__ explicit OneItem(const SortArgs& s) {
    const ItemDev& it = s.items[0];
    x = s.x_override ? s.x_override : it.x;
    poff = it.point_offset;
    koff = it.key_offset;
    fine = it.geom.fine;
#pragma unroll
    for (int t = 0; t < D; ++t) {
      n[t] = it.geom.n[t];
      bw[t] = it.geom.bin[t];
      nb[t] = it.geom.nbins[t];
    }
  }
};

template <typename Real, int D>
__global__ void __launch_bounds__(kSortThreads) k_key_count_one(SortArgs s, int* __restrict__ key_count,
                                                                int2* __restrict__ key_rank) {
  const int64_t base = (int64_t)blockIdx.x * (kSortThreads * kSortPer) + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const OneItem<D> one(s);
  double v[kSortPer][D];
#pragma unroll
  for (int k = 0; k < kSortPer; ++k) {
    const int64_t gidx = base + (int64_t)k * kSortThreads;
#pragma unroll
    for (int t = 0; t < D; ++t) v[k][t] = gidx < s.total_points ? one.x[(gidx - one.poff) * D + t] : 0.0;
  }
  int key[kSortPer];
  bool any_bad = false;
#pragma unroll
  for (int k = 0; k < kSortPer; ++k) {
    const int64_t gidx = base + (int64_t)k * kSortThreads;
    int local = 0, plane = 0;
#pragma unroll
    for (int t = 0; t < D; ++t) {
      double c0 = v[k][t];
      if (!isfinite(c0)) {
        any_bad = true;
        c0 = 0.0;
      }
      int c;
      Real dl;
      reduce_coord<Real>(c0, one.n[t], c, dl);
      const int b = c / one.bw[t];
      if (t == 0) plane = c - b * one.bw[0];
      local = local * one.nb[t] + b;
    }
    key[k] = gidx < s.total_points ? one.koff + local * one.fine + (one.fine > 1 ? plane : 0) : -1;
  }
  if (any_bad) atomicOr(s.err, 1);
  unsigned peers[kSortPer];
  int got[kSortPer];
#pragma unroll
  for (int k = 0; k < kSortPer; ++k) {
    peers[k] = __match_any_sync(0xffffffffu, key[k]);
    got[k] = 0;
    if (key[k] >= 0 && lane == __ffs(peers[k]) - 1) got[k] = atomicAdd(&key_count[key[k]], __popc(peers[k]));
  }
#pragma unroll
  for (int k = 0; k < kSortPer; ++k) {
    const int first = __shfl_sync(peers[k], got[k], __ffs(peers[k]) - 1);
    const int64_t gidx = base + (int64_t)k * kSortThreads;
    if (key[k] >= 0) key_rank[gidx] = make_int2(key[k], first + __popc(peers[k] & ((1u << lane) - 1u)));
  }
}

template <typename Real, int D>
__global__ void __launch_bounds__(kSortThreads) k_scatter_one(SortArgs s, const int* __restrict__ key_start,
                                                              const int2* __restrict__ key_rank, int* __restrict__ perm,
                                                              uint32_t* __restrict__ local, Real* d0, Real* d1, Real* d2) {
  const int64_t base = (int64_t)blockIdx.x * (kSortThreads * kSortPer) + threadIdx.x;
  Real* dst[3] = {d0, d1, d2};
  const OneItem<D> one(s);
  const bool whole = one.fine <= 1;   // else k_refine writes all but the index
  int2 br[kSortPer];
  double v[kSortPer][D];
#pragma unroll
  for (int k = 0; k < kSortPer; ++k) {
    const int64_t gidx = base + (int64_t)k * kSortThreads;
    const bool in = gidx < s.total_points;
    br[k] = in ? key_rank[gidx] : make_int2(-1, 0);
#pragma unroll
    for (int t = 0; t < D; ++t) v[k][t] = in && whole ? one.x[(gidx - one.poff) * D + t] : 0.0;
  }
  int pos[kSortPer];
#pragma unroll
  for (int k = 0; k < kSortPer; ++k) pos[k] = br[k].x >= 0 ? key_start[br[k].x] + br[k].y : -1;
  constexpr int bits = D == 1 ? 32 : (D == 2 ? 16 : 10);
#pragma unroll
  for (int k = 0; k < kSortPer; ++k) {
    if (pos[k] < 0) continue;
    const int64_t gidx = base + (int64_t)k * kSortThreads;
    perm[pos[k]] = (int)(gidx - one.poff);
    if (!whole) continue;
    uint32_t packed = 0;
#pragma unroll
    for (int t = 0; t < D; ++t) {
      const double c0 = isfinite(v[k][t]) ? v[k][t] : 0.0;
      int c;
      Real dl;
      reduce_coord<Real>(c0, one.n[t], c, dl);
      const uint32_t lc = (uint32_t)(c % one.bw[t]);
      packed |= (D == 1) ? lc : (lc << (bits * t));
      dst[t][pos[k]] = dl;
    }
    local[pos[k]] = packed;
  }
}

// Exclusive scan of n ints with one block of 1024 threads: each thread scans a
// contiguous chunk sequentially, the chunk totals are scanned in shared memory.
// Used for the per-tile partial sums of the multi-block scan below.
// clear: the input is left zero (the sort's counts, for the next call).
__global__ void __launch_bounds__(1024) k_scan(int* __restrict__ in, int* __restrict__ out, int n,
                                                int* __restrict__ total, bool clear) {
  __shared__ int part[1024];
  const int T = blockDim.x;
  const int chunk = (n + T - 1) / T;
  const int lo = min(n, threadIdx.x * chunk);
  const int hi = min(n, lo + chunk);
  int s = 0;
  for (int i = lo; i < hi; ++i) s += in[i];
  part[threadIdx.x] = s;
  __syncthreads();
  // Hillis-Steele inclusive scan of the chunk totals
  for (int off = 1; off < T; off <<= 1) {
    const int v = threadIdx.x >= off ? part[threadIdx.x - off] : 0;
    __syncthreads();
    part[threadIdx.x] += v;
    __syncthreads();
  }
  int run = part[threadIdx.x] - s;
  for (int i = lo; i < hi; ++i) {
    const int v = in[i];
    out[i] = run;
    if (clear) in[i] = 0;
    run += v;
  }
  if (total && threadIdx.x == T - 1) *total = part[T - 1];
}

// Multi-block exclusive scan: tiles of kScanTile ints.  k_scan_reduce sums
// each tile (coalesced), k_scan scans the tile sums, k_scan_apply scans each
// tile (16 consecutive ints per thread, then the block's thread totals) and
// adds its tile's offset.
constexpr int kScanThreads = 256;
constexpr int kScanPer = 16;
constexpr int kScanTile = kScanThreads * kScanPer;

// Exclusive prefix of v over the block's threads (in thread order).
__device__ __forceinline__ int block_exclusive(int v) {
  __shared__ int wsum[kScanThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) wsum[w] = inc;
  __syncthreads();
  int before = 0;
  for (int k = 0; k < w; ++k) before += wsum[k];
  return before + inc - v;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(const int* __restrict__ in, int n,
                                                               int* __restrict__ partials) {
  __shared__ int wsum[kScanThreads / 32];
  const int64_t base = (int64_t)blockIdx.x * kScanTile;
  int s = 0;
  for (int i = threadIdx.x; i < kScanTile; i += kScanThreads)
    if (base + i < n) s += in[base + i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int k = 0; k < kScanThreads / 32; ++k) t += wsum[k];
    partials[blockIdx.x] = t;
  }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_apply(int* __restrict__ in, int* __restrict__ out, int n,
                                                              const int* __restrict__ offsets, bool clear) {
  const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanPer;
  int v[kScanPer];
  int s = 0;
#pragma unroll
  for (int q = 0; q < kScanPer; ++q) {
    v[q] = base + q < n ? in[base + q] : 0;
    s += v[q];
  }
  int run = block_exclusive(s) + offsets[blockIdx.x];
#pragma unroll
  for (int q = 0; q < kScanPer; ++q) {
    if (base + q < n) {
      out[base + q] = run;
      if (clear) in[base + q] = 0;
    }
    run += v[q];
  }
}

__global__ void k_sub_count(SortArgs s, const int* __restrict__ key_start, int P, int* __restrict__ bin_count,
                            int* __restrict__ bin_start, int* __restrict__ sub_count) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= s.total_bins) return;
  const ItemDev& it = s.items[find_item<int>(s.bin_offsets, s.n_items, b)];
  const int key = it.key_offset + (b - it.bin_offset) * it.geom.fine;
  const int start = key_start[key], cnt = key_start[key + it.geom.fine] - start;
  bin_count[b] = cnt;
  bin_start[b] = start;
  sub_count[b] = (cnt + P - 1) / P;
}

// Points of a bin's pieces: at most P, and as even as can be (pencils: P, whole
// batches of their kernels).  In pieces of P and the rest, uniform points make
// tiles for a few points each: 2-D, N = 256^2, 100,000 points, bins of 390, P =
// 328, spreading + interpolation at 12 taps: FP32 149 + 74 us, even 118 + 45,
// three right-hand sides 347 + 227, even 280 + 149; FP64 447 + 430, even 320 + 266.
__device__ __forceinline__ int piece_size(int count, int P, int fine) {
  if (fine > 1) return P;
  const int pieces = max((count + P - 1) / P, 1);
  return (count + pieces - 1) / pieces;
}

__global__ void k_sub_fill(SortArgs s, const int* __restrict__ bin_count, const int* __restrict__ bin_start,
                           const int* __restrict__ sub_start, int P, SubProblem* __restrict__ subs,
                           int* __restrict__ grid_points) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < s.n_items) grid_points[b] = 0;   // (an item has a bin or more)
  if (b >= s.total_bins) return;
  const int cnt = bin_count[b];
  if (cnt == 0) return;
  const int item = find_item<int>(s.bin_offsets, s.n_items, b);
  const int local_bin = b - s.bin_offsets[item];
  const int s0 = sub_start[b];
  const int size = piece_size(cnt, P, s.items[item].geom.fine);
  for (int k = 0, off = 0; off < cnt; ++k, off += size) {
    SubProblem sp;
    sp.bin = local_bin;
    sp.start = bin_start[b] + off;
    sp.count = min(size, cnt - off);
    sp.item = item;
    sp.form = kFormGrid;
    subs[s0 + k] = sp;
  }
}

// k_sub_count, the scan of its counts and k_sub_fill in one block, for up to
// kSubSingle bins: one launch in place of three, and the records are written
// by all threads evenly instead of by each bin's thread.
constexpr int kSubSingle = 16384;

__global__ void __launch_bounds__(1024) k_subproblems(SortArgs s, const int* __restrict__ key_start, int P,
                                                       int* __restrict__ bin_count, int* __restrict__ bin_start,
                                                       int* __restrict__ sub_start, int* __restrict__ num_subs,
                                                       SubProblem* __restrict__ subs, int* __restrict__ grid_points) {
  for (int i = threadIdx.x; i < s.n_items; i += 1024) grid_points[i] = 0;
  __shared__ int wsum[32];
  const int nb = s.total_bins, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int chunk = (nb + 1023) / 1024;
  const int lo = min(nb, (int)threadIdx.x * chunk), hi = min(nb, lo + chunk);
  int mine = 0;
  for (int b = lo; b < hi; ++b) {
    const ItemDev& it = s.items[find_item<int>(s.bin_offsets, s.n_items, b)];
    const int key = it.key_offset + (b - it.bin_offset) * it.geom.fine;
    const int start = key_start[key], cnt = key_start[key + it.geom.fine] - start;
    bin_count[b] = cnt;
    bin_start[b] = start;
    mine += (cnt + P - 1) / P;
  }
  int inc = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) wsum[w] = inc;
  __syncthreads();
  int before = 0, total = 0;
  for (int k = 0; k < 32; ++k) {
    before += k < w ? wsum[k] : 0;
    total += wsum[k];
  }
  int run = before + inc - mine;
  for (int b = lo; b < hi; ++b) {
    sub_start[b] = run;
    run += (bin_count[b] + P - 1) / P;
  }
  if (threadIdx.x == 0) *num_subs = total;
  __syncthreads();
  for (int t = threadIdx.x; t < total; t += 1024) {
    const int b = find_item<int>(sub_start, nb, t);   // the last bin that starts at t or before: not an empty one
    const int item = find_item<int>(s.bin_offsets, s.n_items, b);
    const int size = piece_size(bin_count[b], P, s.items[item].geom.fine);
    const int off = (t - sub_start[b]) * size;
    SubProblem sp;
    sp.bin = b - s.bin_offsets[item];
    sp.start = bin_start[b] + off;
    sp.count = min(size, bin_count[b] - off);
    sp.item = item;
    sp.form = kFormGrid;
    subs[t] = sp;
  }
}

// The points of a pencil's subproblem (geom.fine > 1: in the order of their
// planes, by their indices only): their records written, in runs of kRefine
// points, ordered by cell, (l0, l1, l2), where there are as many points as
// cells.  Neighbouring points then share cells, which interpolation turns into
// shared-memory broadcasts (kFormDense).  The scatter writes 4 bytes per point to a random place
// instead of 20 in five arrays (32-byte sectors: 5 of them; M = 3 10^7: 1.23
// -> 0.21 ms); the coordinates are gathered here instead, and the records go
// out in order (0.81 ms with the sort, M = 10^6 uniform without it: 21 us).  Bitonic sort of
// 32-bit keys (cell, slot), four per thread in registers: a step's partner is
// in the thread, in another lane (a shuffle) or, from distance 128 on, in
// another warp (shared memory, 6 of the 55 steps; all steps in shared memory:
// 1.04 ms).
constexpr int kRefine = 1024;
constexpr int kRefineThreads = 256;
constexpr int kRefinePer = kRefine / kRefineThreads;

__global__ void __launch_bounds__(kRefineThreads) k_refine(SortArgs s, SubProblem* __restrict__ subs,
                                                           const int* __restrict__ num_subs, int* __restrict__ perm,
                                                           uint32_t* __restrict__ local, float* __restrict__ d0,
                                                           float* __restrict__ d1, float* __restrict__ d2,
                                                           int* __restrict__ grid_points) {
  static_assert(kRefinePer == 4, "four elements per thread");
  __shared__ __align__(16) uint32_t key[kRefine];
  __shared__ uint32_t loc[kRefine];
  __shared__ int idx[kRefine];
  __shared__ float del[3][kRefine];
  if ((int)blockIdx.x >= *num_subs) return;
  const SubProblem sub = subs[blockIdx.x];
  const ItemDev& it = s.items[sub.item];
  if (it.geom.fine <= 1) return;
  const double* x = s.x_override ? s.x_override : it.x;
  int n[3], bw[3];
#pragma unroll
  for (int t = 0; t < 3; ++t) {
    n[t] = it.geom.n[t];
    bw[t] = it.geom.bin[t];
  }
  int total_cells = 0, total_blocks = 0;   // of this thread's points, those that begin a cell, or planes of a slab
  int first_plane = 0, last_plane = 0;
  const int ahead = slab_ahead(it.win.taps);
  for (int r0 = 0; r0 < sub.count; r0 += kRefine) {
    const int cnt = min(kRefine, sub.count - r0), first = sub.start + r0;
    int size = 64;
    while (size < cnt) size *= 2;
    // every index, then every coordinate of a thread's points in flight together
    int j[kRefinePer];
    double v[kRefinePer][3];
#pragma unroll
    for (int q = 0; q < kRefinePer; ++q) {
      const int i = threadIdx.x + q * kRefineThreads;
      j[q] = i < cnt ? perm[first + i] : -1;
    }
#pragma unroll
    for (int q = 0; q < kRefinePer; ++q)
#pragma unroll
      for (int t = 0; t < 3; ++t) v[q][t] = j[q] >= 0 ? x[(int64_t)j[q] * 3 + t] : 0.0;
#pragma unroll
    for (int q = 0; q < kRefinePer; ++q) {
      const int i = threadIdx.x + q * kRefineThreads;
      if (j[q] >= 0) {
        uint32_t packed = 0, k = 0;
#pragma unroll
        for (int t = 0; t < 3; ++t) {
          int c;
          float dl;
          reduce_coord<float>(isfinite(v[q][t]) ? v[q][t] : 0.0, n[t], c, dl);
          const uint32_t lc = (uint32_t)(c % bw[t]);
          packed |= lc << (10 * t);
          k = t == 0 ? lc : (k << 5 | lc);   // edges of dimensions 1, 2 are below 32
          del[t][i] = dl;
        }
        idx[i] = j[q];
        loc[i] = packed;
        key[i] = k << 10 | (uint32_t)i;
      }
    }
    __syncthreads();
    // fewer points than cells: no run of the sort would be worth it
    const int l0 = (int)(loc[0] & 1023u);
    last_plane = (int)(loc[cnt - 1] & 1023u);
    if (r0 == 0) first_plane = l0;
    const int span = last_plane - l0 + 1;
    if (cnt < span * bw[1] * bw[2]) {
#pragma unroll
      for (int q = 0; q < kRefinePer; ++q) {
        const int i = threadIdx.x + q * kRefineThreads;
        if (i >= cnt) continue;
        local[first + i] = loc[i];
        d0[first + i] = del[0][i];
        d1[first + i] = del[1][i];
        d2[first + i] = del[2][i];
        ++total_cells;
        total_blocks += i == 0 || (int)(loc[i] & 1023u) / ahead != (int)(loc[i - 1] & 1023u) / ahead;
      }
      __syncthreads();
      continue;
    }
    // element 4 t + r of the sort in register r of thread t
    const int first_e = kRefinePer * threadIdx.x;
    uint32_t e[kRefinePer];
#pragma unroll
    for (int r = 0; r < kRefinePer; ++r) e[r] = first_e + r < cnt ? key[first_e + r] : 0xffffffffu;
    for (int k = 2; k <= size; k *= 2) {
      for (int d = k / 2; d >= 4 * 32; d /= 2) {   // partner in another warp
        __syncthreads();
        *reinterpret_cast<uint4*>(key + first_e) = make_uint4(e[0], e[1], e[2], e[3]);
        __syncthreads();
        const uint4 o = *reinterpret_cast<const uint4*>(key + (first_e ^ d));
        const bool low = ((first_e & d) == 0) == ((first_e & k) == 0);
        e[0] = low ? min(e[0], o.x) : max(e[0], o.x);
        e[1] = low ? min(e[1], o.y) : max(e[1], o.y);
        e[2] = low ? min(e[2], o.z) : max(e[2], o.z);
        e[3] = low ? min(e[3], o.w) : max(e[3], o.w);
      }
      for (int d = min(k / 2, 64); d >= 4; d /= 2) {   // in another lane
        const bool low = ((first_e & d) == 0) == ((first_e & k) == 0);
#pragma unroll
        for (int r = 0; r < kRefinePer; ++r) {
          const uint32_t o = __shfl_xor_sync(0xffffffffu, e[r], d / 4);
          e[r] = low ? min(e[r], o) : max(e[r], o);
        }
      }
      const bool up = (first_e & k) == 0;   // in this thread: (0, 2), (1, 3), then (0, 1), (2, 3)
      auto swap = [](uint32_t& x, uint32_t& y, bool ascending) {
        const uint32_t lo = min(x, y), hi = max(x, y);
        x = ascending ? lo : hi;
        y = ascending ? hi : lo;
      };
      if (k >= 4) {
        swap(e[0], e[2], up);
        swap(e[1], e[3], up);
      }
      swap(e[0], e[1], k == 2 ? true : up);
      swap(e[2], e[3], k == 2 ? false : up);
    }
    __syncthreads();
    *reinterpret_cast<uint4*>(key + first_e) = make_uint4(e[0], e[1], e[2], e[3]);
    __syncthreads();
    int cells = 0;   // of this thread's points, those that begin a cell
    for (int i = threadIdx.x; i < cnt; i += kRefineThreads) {
      cells += i == 0 || key[i] >> 10 != key[i - 1] >> 10;
      total_blocks += i == 0 || (int)(key[i] >> 20) / ahead != (int)(key[i - 1] >> 20) / ahead;
      const int p = (int)(key[i] & (kRefine - 1));
      perm[first + i] = idx[p];
      local[first + i] = loc[p];
      d0[first + i] = del[0][p];
      d1[first + i] = del[1][p];
      d2[first + i] = del[2][p];
    }
    total_cells += cells;
    __syncthreads();
  }
  // dense: kDenseRun points per occupied cell or more
  __shared__ int occupied, blocks;
  if (threadIdx.x == 0) occupied = blocks = 0;
  __syncthreads();
  atomicAdd(&occupied, total_cells);
  atomicAdd(&blocks, total_blocks);
  __syncthreads();
  if (threadIdx.x == 0) {
    const int planes = min(blocks * ahead, last_plane - first_plane + 1);   // of slabs
    const bool slab = 2 * sub.count >= slab_points(it.win.taps) * planes;
    const int form = sub.count >= kDenseRun * occupied ? kFormDense : (slab ? kFormSlab : kFormGrid);
    subs[blockIdx.x].form = form;
    if (form == kFormGrid) atomicAdd(&grid_points[sub.item], sub.count);
  }
}

inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

template <typename Real>
cudaError_t launch_key_count(const SortArgs& s, int* key_count, int2* key_rank, cudaStream_t st) {
  if (s.total_points == 0) return cudaSuccess;
  const unsigned blocks = blocks_for(s.total_points, kSortThreads * kSortPer);
  switch (s.single_d) {
    case 1: k_key_count_one<Real, 1><<<blocks, kSortThreads, 0, st>>>(s, key_count, key_rank); break;
    case 2: k_key_count_one<Real, 2><<<blocks, kSortThreads, 0, st>>>(s, key_count, key_rank); break;
    case 3: k_key_count_one<Real, 3><<<blocks, kSortThreads, 0, st>>>(s, key_count, key_rank); break;
    default: k_key_count<Real><<<blocks, kSortThreads, 0, st>>>(s, key_count, key_rank);
  }
  return cudaGetLastError();
}

int scan_partials_needed(int n) { return 2 * ((n + kScanTile - 1) / kScanTile) + 1; }

// Up to kScanSingle ints one block scans them in one launch (a few per
// thread); longer arrays take the three tiled launches.
constexpr int kScanSingle = 4 * kScanTile;

int scan_launches(int n) { return n <= kScanSingle ? 1 : 3; }

cudaError_t launch_scan(int* in, int* out, int n, int* total, int* partials, bool clear, cudaStream_t st) {
  if (n <= kScanSingle) {
    k_scan<<<1, 1024, 0, st>>>(in, out, n, total, clear);
    return cudaGetLastError();
  }
  const int tiles = (n + kScanTile - 1) / kScanTile;
  int* const offsets = partials + tiles;   // the scanned tile sums
  if (tiles > 0) k_scan_reduce<<<tiles, kScanThreads, 0, st>>>(in, n, partials);
  k_scan<<<1, 1024, 0, st>>>(partials, offsets, tiles, total, false);
  if (tiles > 0) k_scan_apply<<<tiles, kScanThreads, 0, st>>>(in, out, n, offsets, clear);
  return cudaGetLastError();
}

template <typename Real>
cudaError_t launch_scatter(const SortArgs& s, const int* key_start, const int2* key_rank, int* perm, uint32_t* local,
                           Real* const* delta, cudaStream_t st) {
  if (s.total_points == 0) return cudaSuccess;
  const unsigned blocks = blocks_for(s.total_points, kSortThreads * kSortPer);
  switch (s.single_d) {
    case 1:
      k_scatter_one<Real, 1><<<blocks, kSortThreads, 0, st>>>(s, key_start, key_rank, perm, local, delta[0], delta[1],
                                                              delta[2]);
      break;
    case 2:
      k_scatter_one<Real, 2><<<blocks, kSortThreads, 0, st>>>(s, key_start, key_rank, perm, local, delta[0], delta[1],
                                                              delta[2]);
      break;
    case 3:
      k_scatter_one<Real, 3><<<blocks, kSortThreads, 0, st>>>(s, key_start, key_rank, perm, local, delta[0], delta[1],
                                                              delta[2]);
      break;
    default:
      k_scatter<Real><<<blocks, kSortThreads, 0, st>>>(s, key_start, key_rank, perm, local, delta[0], delta[1],
                                                       delta[2]);
  }
  return cudaGetLastError();
}

int subproblem_launches(int nbins) { return nbins <= kSubSingle ? 1 : 2 + scan_launches(nbins); }

cudaError_t launch_subproblems(const SortArgs& s, const int* key_start, int P, int* bin_count, int* bin_start,
                               int* sub_count, int* sub_start, int* num_subs, int* partials, SubProblem* subs,
                               int* grid_points, cudaStream_t st) {
  if (s.total_bins <= kSubSingle) {
    k_subproblems<<<1, 1024, 0, st>>>(s, key_start, P, bin_count, bin_start, sub_start, num_subs, subs,
                                      grid_points);
    return cudaGetLastError();
  }
  k_sub_count<<<blocks_for(s.total_bins, 256), 256, 0, st>>>(s, key_start, P, bin_count, bin_start, sub_count);
  const cudaError_t e = launch_scan(sub_count, sub_start, s.total_bins, num_subs, partials, false, st);
  if (e != cudaSuccess) return e;
  k_sub_fill<<<blocks_for(s.total_bins, 256), 256, 0, st>>>(s, bin_count, bin_start, sub_start, P, subs, grid_points);
  return cudaGetLastError();
}

cudaError_t launch_refine(const SortArgs& s, int64_t max_subs, SubProblem* subs, const int* num_subs, int* perm,
                          uint32_t* local, float* const* delta, int* grid_points, cudaStream_t st) {
  if (max_subs <= 0) return cudaSuccess;
  k_refine<<<(unsigned)max_subs, kRefineThreads, 0, st>>>(s, subs, num_subs, perm, local, delta[0], delta[1], delta[2],
                                                                  grid_points);
  return cudaGetLastError();
}

template cudaError_t launch_key_count<float>(const SortArgs&, int*, int2*, cudaStream_t);
template cudaError_t launch_key_count<double>(const SortArgs&, int*, int2*, cudaStream_t);
template cudaError_t launch_scatter<float>(const SortArgs&, const int*, const int2*, int*, uint32_t*, float* const*,
                                           cudaStream_t);
template cudaError_t launch_scatter<double>(const SortArgs&, const int*, const int2*, int*, uint32_t*,
                                            double* const*, cudaStream_t);

}  // namespace gbnfft
