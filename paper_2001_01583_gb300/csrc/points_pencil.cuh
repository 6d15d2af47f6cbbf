// 3-D spreading and interpolation in FP32 along pencils.
//
// The sort keeps a bin's points in the order of their cell along dimension 0
// (GridGeom::fine), and a bin is a pencil: by x bx cells of dimensions 1, 2,
// long in dimension 0.  A block walks a run of a pencil's points along
// dimension 0 and never back, so a tile pays a halo in two dimensions only,
// (by + W - 1)(bx + W - 1) cells per plane of by bx: 3.2 of them at 8 taps
// where a bin of 8 x 8 x 16 cells flushes 5.1.
//
// Spreading holds the cells in registers, a window of W planes that moves
// with the points.  The tile of 8 NR x 8 NR columns (by = bx = 8 NR + 1 - W,
// so the halo fills it) is cut into NR x NR squares of 8 x 8 columns, a warp
// each; lane (ly, lx) holds columns (ly, lx) and (ly + 4, lx) of its warp's
// square.  A point adds wz(i) (wy(y) (wx(x) v)) to the W cells of every column
// it reaches; when the next point lies in a later plane, the planes left
// behind go to the grid (vector atomics: neighbouring pencils' halos overlap)
// and the window moves.  A warp takes only the points that reach its square
// (one ballot per 32 points); the weights of dimensions 1 and 2 are staged
// with zeros on both sides, so a lane outside a footprint adds zeros.
//   Why: with the tile in shared memory (points_planes.cuh) every cell update
//   is a shared load and store, 64 wavefronts of 128 bytes per point at 8
//   taps, and 32 more for the weights.  Here an update is one paired FMA on
//   registers; the price is lanes outside the footprint: a point of 8 taps
//   meets (16 / 9)^2 = 3.2 squares of 64 columns on average (NR = 2).  It is
//   bound by instruction issue (about 160 per point at 8 taps, 52 of them the
//   FMAs) at 20 warps per SM.  The window's halves lie in 64-bit registers,
//   pairs along dimension 0, so that a paired FMA takes two neighbouring
//   weights as they lie in shared memory.
//
// Interpolation loads slabs of the tile's planes into shared memory
// (k_interp_pencil).
//
// Measured on GB300 (Kaiser-Bessel, sigma = 2, spread / interpolation, against
// the kernels of points_planes.cuh and points_gm.cuh at their default bins):
//   N = 64^3, M = 10^6, m = 4, uniform: 222 / 206 us from 441 / 248
//     clustered (32 clusters, std 0.02): 209 / 180 us from 566 / 288
//   N = 90 x 128 x 74, M = 777777, m = 5: 311 / 532 us from 1069 / 989
//   N = 256^3, M = 3 10^7, m = 3, 64 clusters, std 0.01: 3.5 / 2.0 ms from
//     14.9 / 5.0
//   N = 128^3, 393216 ions, m = 6: 388 us from 2471 (spread only)
#pragma once

#include "points_planes.cuh"

namespace gbnfft {

// The pencil kernels' shape for W taps and NR x NR squares.
template <int W, int NR>
struct PencilShape {
  // columns per lane: a warp's part of the tile is 4 C rows by 8 columns
  // (C = 4 reads fewer weights per point and meets more idle lanes: 243 us
  // against 229 for N = 64^3, M = 10^6, 8 taps, and 3.9 against 3.6 ms for 6
  // taps on the largest configuration)
  static constexpr int C = 2;
  static constexpr int ROWS = 4 * C, WARPS = 8 * NR / ROWS * NR, THREADS = 32 * WARPS;
  // threads that stage one point, and points per batch (a multiple of 32)
  static constexpr int PARTS = NR == 2 ? 2 : 3, BP = NR == 2 ? THREADS / 2 : 96;
  // resident blocks asked of the compiler
  static constexpr int MIN_BLOCKS = NR == 2 ? (W <= 6 ? 7 : 5) : (W <= 12 ? 2 : 1);
  static constexpr int PADX = 8, PADY = ROWS;   // zeros on each side of wx and wy
  static constexpr int LENX = (W + 2 * PADX + 3) / 4 * 4, LENY = (W + 2 * PADY + 3) / 4 * 4;
  static_assert(PARTS * BP <= THREADS, "a thread stages at most one part");
};

// Floats of a staged point: wz | 0 wy 0 | 0 wx 0 (spreading: the complex v wx).  The stride is an odd number of 16-byte units, so that 8
// consecutive points' 16-byte stores fall in distinct banks.
template <int W, int NR>
struct PencilRow {
  using S = PencilShape<W, NR>;
  static constexpr int WY = (W + 3) / 4 * 4;
  static constexpr int WX = WY + S::LENY;
  static constexpr int S4 = (WX + 2 * S::LENX + 3) / 4;
  static constexpr int STRIDE = 4 * (S4 % 2 ? S4 : S4 + 1);
  static constexpr size_t BYTES = (size_t)(S::BP + 1) * STRIDE * sizeof(float);   // a row of zeros after the points'
};

// Shared memory: the staged points, the warps' lists, the points' packed cells.
template <int W, int NR>
constexpr size_t pencil_smem_bytes() {
  using S = PencilShape<W, NR>;
  return PencilRow<W, NR>::BYTES + (size_t)S::WARPS * S::BP * 16 + (size_t)S::BP * sizeof(uint32_t);
}

__device__ __forceinline__ void sts_f4(uint32_t a, float x, float y, float z, float w) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}

__device__ __forceinline__ void sts_u4(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}
__device__ __forceinline__ uint4 lds_u4(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}

// N consecutive floats (N even) to a 16-byte aligned shared address.
template <int N>
__device__ __forceinline__ void sts_row(uint32_t a, const float* v) {
#pragma unroll
  for (int i = 0; i + 3 < N; i += 4) sts_f4(a + 4u * i, v[i], v[i + 1], v[i + 2], v[i + 3]);
  if (N % 4 == 2) sts_f2(a + 4u * (N - 2), make_float2(v[N - 2], v[N - 1]));
}

// What a thread stages of its point of a batch, in registers: loaded while the
// batch before it is worked on.  PARTS threads per point, the parts in
// different warps (BP is a multiple of 32): dimension 0 (and, of two parts,
// 1), dimension 1, dimension 2 with the point's value or index.
template <int W, int NR>
struct PencilFetch {
  using S = PencilShape<W, NR>;
  using R = PencilRow<W, NR>;
  float da, db;     // offsets in the cell
  uint32_t loc;
  int jn;           // index of the next batch's point
  float2 v;

  static __device__ __forceinline__ int part() { return threadIdx.x / S::BP; }
  static __device__ __forceinline__ int slot() { return threadIdx.x % S::BP; }

  // the batch first .. first + nb - 1 of the subproblem's points up to end
  __device__ __forceinline__ void fetch(const PointKernelArgs<float>& a, const float2* f_in, int first, int end) {
    const int idx = first + slot();
    if (idx >= end) return;
    if (part() == 0) da = a.pts.delta[0][idx];
    if (part() == S::PARTS - 2) db = a.pts.delta[1][idx];
    if (part() == S::PARTS - 1) {
      da = a.pts.delta[2][idx];
      loc = a.pts.local[idx];
      v = f_in[jn];
      if (idx + S::BP < end) jn = a.pts.perm[idx + S::BP];
    }
  }

  __device__ __forceinline__ void start(const PointKernelArgs<float>& a, const float2* f_in, int first, int end) {
    da = db = 0.f;
    loc = 0;
    jn = 0;
    v = make_float2(0.f, 0.f);
    if (part() == S::PARTS - 1 && first + slot() < end) jn = a.pts.perm[first + slot()];
    fetch(a, f_in, first, end);
  }

  __device__ __forceinline__ void stage(const WindowDev& win, uint32_t wt_a, uint32_t* rec, int nb) const {
    const int t = slot();
    if (part() >= S::PARTS || t >= nb) return;
    const uint32_t row = wt_a + 4u * (uint32_t)(t * R::STRIDE);
    float w[W];
    if (part() == 0) {
      window_taps<W>(win, 0, da, w);
      sts_row<W>(row, w);
    }
    if (part() == S::PARTS - 2) {
      window_taps<W>(win, 1, db, w);
      sts_row<W>(row + 4u * (R::WY + S::PADY), w);
    }
    if (part() == S::PARTS - 1) {
      rec[t] = loc;
      window_taps<W>(win, 2, da, w);
#pragma unroll
      for (int i = 0; i < W; i += 2) {
        const float2 p = cscale(v, w[i]), q = cscale(v, w[i + 1]);
        sts_f4(row + 4u * (R::WX + 2 * (S::PADX + i)), p.x, p.y, q.x, q.y);
      }
    }
  }
};

// W floats (W even) from a 16-byte aligned shared address, as pairs.
template <int W>
__device__ __forceinline__ void lds_pairs(uint32_t a, Pair* w) {
#pragma unroll
  for (int i = 0; i + 1 < W / 2; i += 2)
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(w[i]), "=l"(w[i + 1]) : "r"(a + 8u * i));
  if ((W / 2) % 2) asm volatile("ld.shared.b64 %0, [%1];" : "=l"(w[W / 2 - 1]) : "r"(a + 8u * (W / 2 - 1)));
}

// A window of W values one value on: the first leaves, v comes last.
template <int W>
__device__ __forceinline__ void window_step(Pair* w, float v) {
#pragma unroll
  for (int i = 0; i < W / 2; ++i) w[i] = pair(halves(w[i]).y, i + 1 < W / 2 ? halves(w[i + 1]).x : v);
}

// The staged points that reach a warp's square, in their order (so planes
// ascend), into the warp's list: shared address of the point's row, of this
// square's first row and column in its padded weights, and its plane.  The
// list is filled up to a multiple of four with the row of zeros at the last
// point's plane.  Returns the filled length.
template <int W, int NR>
__device__ __forceinline__ int pencil_list(const uint32_t* rec, uint32_t wt_a, uint32_t list_a, int nb, int lane,
                                           int y0, int x0) {
  using S = PencilShape<W, NR>;
  using R = PencilRow<W, NR>;
  int n = 0, last = 0;
#pragma unroll
  for (int base = 0; base < S::BP; base += 32) {
    if (base >= nb) break;
    const int t = base + lane;
    const uint32_t loc = rec[t];   // t < BP; stale past nb
    const int dy = y0 - unpack_local(loc, 3, 1), dx = x0 - unpack_local(loc, 3, 2);
    const int l0 = unpack_local(loc, 3, 0);
    const bool reach = t < nb && dy > -S::PADY && dy < W && dx > -S::PADX && dx < W;
    const unsigned mask = __ballot_sync(0xffffffffu, reach);
    if (reach) {
      const uint32_t row = wt_a + 4u * (uint32_t)(t * R::STRIDE);
      sts_u4(list_a + 16u * (uint32_t)(n + __popc(mask & ((1u << lane) - 1u))), row,
             row + 4u * (uint32_t)(R::WY + S::PADY + dy), row + 4u * R::WX + 8u * (uint32_t)(S::PADX + dx), (uint32_t)l0);
    }
    if (mask) last = __shfl_sync(0xffffffffu, l0, 31 - __clz(mask));
    n += __popc(mask);
  }
  const int full = (n + 3) & ~3;
  if (n + lane < full) {
    const uint32_t zero = wt_a + 4u * (uint32_t)(S::BP * R::STRIDE);
    sts_u4(list_a + 16u * (uint32_t)(n + lane), zero, zero, zero, (uint32_t)last);
  }
  __syncwarp();
  return full;
}

// This block's subproblem; false when there is none.
__device__ __forceinline__ bool pencil_sub(const PointKernelArgs<float>& a, SubProblem& sub) {
  int lo, hi;
  launch_subs(a, lo, hi);
  const int sp = lo + (int)blockIdx.x;
  if (sp >= hi) return false;
  sub = a.pts.subs[sp];
  return true;
}

// The pencil's first plane in the grid, and this lane's columns (flat index
// inside a plane).
template <int C>
struct PencilCols {
  int z0, col[C];
  __device__ __forceinline__ PencilCols(const ItemDev& it, int bin, int y0, int x0, int lane) {
    const GridGeom& g = it.geom;
    int bc[kMaxDim];
    bin_coords(bin, g, bc);
    const int s = it.win.shift - it.win.m;
    z0 = bc[0] * g.bin[0] + s;
    const int x = wrap_mod(bc[2] * g.bin[2] + s + x0 + (lane & 7), g.n[2]);
#pragma unroll
    for (int c = 0; c < C; ++c)
      col[c] = wrap_mod(bc[1] * g.bin[1] + s + y0 + (lane >> 3) + 4 * c, g.n[1]) * g.n[2] + x;
  }
};

template <int W, int NR>
__global__ void __launch_bounds__(PencilShape<W, NR>::THREADS, PencilShape<W, NR>::MIN_BLOCKS)
    k_spread_pencil(PointKernelArgs<float> a) {
  using S = PencilShape<W, NR>;
  using R = PencilRow<W, NR>;
  constexpr int C = S::C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* wt = reinterpret_cast<float*>(smem_raw);
  uint4* list = reinterpret_cast<uint4*>(smem_raw + R::BYTES);   // [warps][BP]
  uint32_t* rec = reinterpret_cast<uint32_t*>(list + S::WARPS * S::BP);
  SubProblem sub;
  if (!pencil_sub(a, sub)) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int y0 = warp / NR * S::ROWS, x0 = warp % NR * 8;
  for (int e = threadIdx.x; e < (S::BP + 1) * R::STRIDE / 4; e += S::THREADS)
    reinterpret_cast<float4*>(wt)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
  const ItemDev& it = a.items[sub.item];
  const GridGeom& g = it.geom;
  const ItemCall call = item_call(a, it);
  const int r = blockIdx.y;
  const float2* f_in = static_cast<const float2*>(call.in) + (int64_t)r * it.M;
  float2* grid = static_cast<float2*>(it.grid) + (int64_t)r * g.grid_cells;
  const PencilCols<C> pc(it, sub.bin, y0, x0, lane);
  const int n0 = g.n[0], plane = g.n[1] * g.n[2];
  const uint32_t wt_a = (uint32_t)__cvta_generic_to_shared(wt);
  const uint32_t wy_l = 4u * (uint32_t)(lane >> 3), wx_l = 8u * (uint32_t)(lane & 7);
  const uint32_t list_a = (uint32_t)__cvta_generic_to_shared(list + warp * S::BP);
  // the window: real and imaginary parts of W cells per column, pairs along
  // dimension 0 (a paired FMA takes two neighbouring weights as they lie)
  Pair re[C][W / 2], im[C][W / 2];
#pragma unroll
  for (int c = 0; c < C; ++c)
#pragma unroll
    for (int i = 0; i < W / 2; ++i) re[c][i] = im[c][i] = 0;
  int cur = -1;        // plane of the window's first cell (in the pencil)
  bool live = false;   // the window holds something
  // the window's first plane to the grid, the window one plane on
  auto flush = [&]() {
    float2* const zp = grid + (int64_t)wrap_mod(pc.z0 + cur, n0) * plane;
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const float2 v = make_float2(halves(re[c][0]).x, halves(im[c][0]).x);
      if (v.x != 0.f || v.y != 0.f) grid_add(zp + pc.col[c], v);
    }
#pragma unroll
    for (int c = 0; c < C; ++c) {
      window_step<W>(re[c], 0.f);
      window_step<W>(im[c], 0.f);
    }
    ++cur;
  };
  auto move_to = [&](int l0) {
    if (live)
      for (int q = min(l0 - cur, W); q > 0; --q) flush();
    cur = l0;
    live = true;
  };
  auto add = [&](const uint4& e) {
    Pair wz[W / 2];
    float wy[C];
#pragma unroll
    for (int c = 0; c < C; ++c) wy[c] = lds_f1(e.y + wy_l + 16u * (uint32_t)c);
    const float2 v = lds_f2(e.z + wx_l);
    lds_pairs<W>(e.x, wz);
    Pair pr[C], pi[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
      pr[c] = pair(v.x * wy[c], v.x * wy[c]);
      pi[c] = pair(v.y * wy[c], v.y * wy[c]);
    }
#pragma unroll
    for (int i = 0; i < W / 2; ++i)
#pragma unroll
      for (int c = 0; c < C; ++c) {
        re[c][i] = pair_fma(wz[i], pr[c], re[c][i]);
        im[c][i] = pair_fma(wz[i], pi[c], im[c][i]);
      }
  };
  PencilFetch<W, NR> fetch;
  const int end = sub.start + sub.count;
  fetch.start(a, f_in, sub.start, end);
  for (int pb = 0; pb < sub.count; pb += S::BP) {
    const int nb = min(S::BP, sub.count - pb);
    __syncthreads();   // zeros written / previous batch no longer read
    fetch.stage(it.win, wt_a, rec, nb);
    __syncthreads();
    fetch.fetch(a, f_in, sub.start + pb + S::BP, end);
    const int n = pencil_list<W, NR>(rec, wt_a, list_a, nb, lane, y0, x0);
    for (int k = 0; k < n; k += 4) {
      const uint32_t la = list_a + 16u * (uint32_t)k;
      if (lds_i1(la + 12u) == cur && lds_i1(la + 60u) == cur) {   // planes ascend: all four are the window's
#pragma unroll
        for (int q = 0; q < 4; q += 2) {   // two entries on their way before the first is used
          const uint4 e0 = lds_u4(la + 16u * (uint32_t)q), e1 = lds_u4(la + 16u * (uint32_t)q + 16u);
          add(e0);
          add(e1);
        }
      } else {
#pragma unroll 1
        for (int q = 0; q < 4; ++q) {
          const uint4 e = lds_u4(la + 16u * (uint32_t)q);
          if ((int)e.w != cur) move_to((int)e.w);
          add(e);
        }
      }
    }
  }
  if (live)
    for (int k = 0; k < W; ++k) flush();
}

// Interpolation: a slab of the pencil's planes in shared memory, loaded by
// asynchronous copies, serves the points of AHEAD planes; up to THREADS points
// at a time.
//   dense subproblems (points ordered by cell): a thread per point.  The lanes
//     of a warp read the same or neighbouring cells, so a load is mostly a
//     broadcast, and a point needs W^3 / 32 of them and no reduction.
//   else: a warp per point, four of them reduced at once.  Lane (ix, q) reads
//     cell ix of PASSES rows of each plane; with the tile's pitch and the
//     choice of rows below the two halves of a warp read without bank
//     conflicts for 2, 4, 8 and 16 taps (128 bytes per wavefront) and nearly
//     so for the others.
template <int W, int NR>
struct SlabShape {
  static constexpr int THREADS = W <= 6 ? 192 : W <= 12 ? 128 : 256;
  static constexpr int SIDE = 8 * NR;   // tile columns per dimension
  // pitch of a tile row in cells, and whether a lane's rows are neighbours
  // (row q PASSES + k) or Q apart (q + Q k): the fewest wavefronts over all
  // positions of a footprint
  static constexpr int PITCH = W == 2 ? 18 : W == 4 ? 20 : W == 6 ? 22 : W == 8 ? 20 : W <= 12 ? 26 : W == 14 ? 30 : 24;
  static constexpr bool NEIGHBOURS = W == 8 || W == 12;
  static constexpr int PLANE = SIDE * PITCH;
  // (a slab is loaded whole, AHEAD + W - 1 planes, for every AHEAD planes of
  // points: more planes mean fewer reloads and fewer resident blocks.  8 taps,
  // uniform, M = 10^6: 254 us for 3 planes, 236 for 4, 213 for 7, 206 for 9, 210
  // for 12; 96000 points, three right-hand sides: 346, 259, 219, 195, 180.
  // N = 96^3, one right-hand side, 2 / 8 points per plane: 6 taps 102 / 151 us
  // for 7 planes, 96 / 137 for 9, 83 / 133 for 12, which takes dense subproblems
  // longer (the largest configuration 2.02 ms for 7, 2.09 for 12); 12 taps 459 / 634 for 2 planes and 256 threads,
  // 206 / 401 for 7 and 128, 217 / 428 for 12 and 256; 14 taps 1077 / 1627 for 1
  // and 128, 538 / 854 for 4 and 256, 321 / 623 for 12 and 256; 16 taps 1791 / 2628
  // for 1 and 128, 588 / 1126 for 8 and 256, 475 / 1006 for 14 and 256; 10 taps
  // 289 / 583 for 7, 264 / 564 for 12)
  static constexpr int AHEAD = slab_ahead(W);   // planes of points a slab serves
  static constexpr int PLANES = AHEAD + W - 1;
  static constexpr int Q = 32 / W, PASSES = (W + Q - 1) / Q;
  static constexpr bool FULL = 32 % W == 0 && Q * PASSES == W;
  // a staged point: wz | wy | wx, an odd number of 16-byte units apart
  static constexpr int S4 = (3 * W + 3) / 4, STRIDE = 4 * (S4 % 2 ? S4 : S4 + 1);
  static constexpr size_t smem_bytes() {
    return (size_t)PLANES * PLANE * sizeof(float2) + (size_t)THREADS * (STRIDE * sizeof(float) + 2 * sizeof(int)) +
           SIDE * SIDE * sizeof(int);
  }
};

template <int W, int NR>
__global__ void __launch_bounds__(SlabShape<W, NR>::THREADS) k_interp_pencil(PointKernelArgs<float> a) {
  using S = SlabShape<W, NR>;
  constexpr int T = S::THREADS;
  constexpr uint32_t PB = 8u * S::PLANE;   // bytes of a plane
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* slab = reinterpret_cast<float2*>(smem_raw);
  float* wt = reinterpret_cast<float*>(slab + S::PLANES * S::PLANE);   // [T][STRIDE]; dense: wz as [W][T]
  int* off = reinterpret_cast<int*>(wt + T * S::STRIDE);               // first cell of each point's footprint
  int* jt = off + T;
  int* col = jt + T;                                                   // grid index of a tile column in its plane
  SubProblem sub;
  if (!pencil_sub(a, sub) || (a.split_forms && !slab_takes(a, sub))) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const ItemDev& it = a.items[sub.item];
  const GridGeom& g = it.geom;
  const WindowDev& win = it.win;
  const ItemCall call = item_call(a, it);
  const int r = blockIdx.y;
  float2* f_out = static_cast<float2*>(call.out) + (int64_t)r * it.M;
  const float2* grid = static_cast<const float2*>(it.grid) + (int64_t)r * g.grid_cells;
  const int n0 = g.n[0], plane = g.n[1] * g.n[2];
  int bc[kMaxDim];
  bin_coords(sub.bin, g, bc);
  const int z0 = bc[0] * g.bin[0] + win.shift - win.m;
  for (int e = threadIdx.x; e < S::SIDE * S::SIDE; e += T)
    col[e] = wrap_mod(bc[1] * g.bin[1] + win.shift - win.m + e / S::SIDE, g.n[1]) * g.n[2] +
             wrap_mod(bc[2] * g.bin[2] + win.shift - win.m + e % S::SIDE, g.n[2]);
  const uint32_t slab_a = (uint32_t)__cvta_generic_to_shared(slab);
  const uint32_t wt_a = (uint32_t)__cvta_generic_to_shared(wt);
  const uint32_t off_a = (uint32_t)__cvta_generic_to_shared(off);
  // this lane's rows of a plane and its column, for a warp per point (a lane
  // without one reads the last and weighs it with 0)
  const int q = lane / W, ix = lane % W;
  uint32_t row_o[S::PASSES], wy_o[S::PASSES];
  bool has[S::PASSES];
#pragma unroll
  for (int k = 0; k < S::PASSES; ++k) {
    const int row = S::NEIGHBOURS ? q * S::PASSES + k : q + S::Q * k;
    has[k] = S::FULL || (q < S::Q && row < W);
    row_o[k] = 8u * (uint32_t)(min(row, W - 1) * S::PITCH + ix);
    wy_o[k] = wt_a + 4u * (uint32_t)(W + min(row, W - 1));
  }
  const uint32_t wx_o = wt_a + 4u * (uint32_t)(2 * W + ix);
  const int end = sub.start + sub.count;
  const int l_end = unpack_local(a.pts.local[end - 1], 3, 0);   // the last point's plane
  int base = -S::AHEAD;                                         // the slab's first plane
  for (int s = sub.start; s < end;) {
    const int idx = s + (int)threadIdx.x;
    const bool in = idx < end;
    const int l_first = unpack_local(a.pts.local[s], 3, 0);
    uint32_t loc = 0;
    float d0 = 0.f, d1 = 0.f, d2 = 0.f;
    int j = 0;
    if (in) {
      loc = a.pts.local[idx];
      d0 = a.pts.delta[0][idx];
      d1 = a.pts.delta[1][idx];
      d2 = a.pts.delta[2][idx];
      j = a.pts.perm[idx];
    }
    const int l0 = unpack_local(loc, 3, 0);
    const bool fresh = l_first >= base + S::AHEAD;   // block-uniform
    const int first = fresh ? l_first : base;
    const bool mine = in && l0 < first + S::AHEAD;
    // a prefix: planes ascend; past the barrier nobody reads the slab and the weights of the round before
    const int count = __syncthreads_count(mine);
    if (fresh) {
      base = first;
      const int planes = min(S::PLANES, l_end + W - base);
      int z = wrap_mod(z0 + base, n0);
      for (int p = 0; p < planes; ++p) {
        const float2* src = grid + (int64_t)z * plane;
        const uint32_t dst = slab_a + PB * (uint32_t)p;
#pragma unroll
        for (int e0 = 0; e0 < S::SIDE * S::SIDE; e0 += T) {
          const int e = e0 + threadIdx.x;
          if (e < S::SIDE * S::SIDE)
            cp_async_cell(dst + 8u * (uint32_t)(e / S::SIDE * S::PITCH + e % S::SIDE), src + col[e]);
        }
        z = z + 1 == n0 ? 0 : z + 1;
      }
    }
    const int cell = (l0 - base) * S::PLANE + unpack_local(loc, 3, 1) * S::PITCH + unpack_local(loc, 3, 2);
    if (sub.form == kFormDense) {
      float wy[W], wx[W];
      if (mine) {
        window_taps<W>(win, 0, d0, wx);
#pragma unroll
        for (int i = 0; i < W; ++i) wt[i * T + threadIdx.x] = wx[i];
        window_taps<W>(win, 1, d1, wy);
        window_taps<W>(win, 2, d2, wx);
      }
      if (fresh) {
        cp_async_wait_all();
        __syncthreads();
      }
      if (mine) {
        uint32_t at = slab_a + 8u * (uint32_t)cell;
        float2 sum = make_float2(0.f, 0.f);
#pragma unroll 1
        for (int iz = 0; iz < W; ++iz) {
          float2 ps = make_float2(0.f, 0.f);
#pragma unroll
          for (int iy = 0; iy < W; ++iy) {
            float2 row = make_float2(0.f, 0.f);
#pragma unroll
            for (int i = 0; i < W; ++i) row = cmad(lds_f2(at + 8u * (uint32_t)(iy * S::PITCH + i)), wx[i], row);
            ps = cmad(row, wy[iy], ps);
          }
          sum = cmad(ps, wt[iz * T + threadIdx.x], sum);
          at += PB;
        }
        f_out[j] = sum;
      }
    } else {
      if (mine) {
        const uint32_t row = wt_a + 4u * (uint32_t)(threadIdx.x * S::STRIDE);
        float w[3 * W];
        window_taps<W>(win, 0, d0, w);
        window_taps<W>(win, 1, d1, w + W);
        window_taps<W>(win, 2, d2, w + 2 * W);
        sts_row<3 * W>(row, w);
        off[threadIdx.x] = 8 * cell;
        jt[threadIdx.x] = j;
      }
      if (fresh) cp_async_wait_all();
      __syncthreads();
      for (int p0 = warp * 4; p0 < count; p0 += T / 32 * 4) {
        float v[8];
#pragma unroll
        for (int g4 = 0; g4 < 4; ++g4) {
          const uint32_t pp = (uint32_t)min(p0 + g4, count - 1);   // past the round: recomputed, not written
          const uint32_t po = 4u * S::STRIDE * pp;
          uint32_t at = slab_a + (uint32_t)lds_i1(off_a + 4u * pp);
          float wz[W];
#pragma unroll
          for (int i = 0; i + 3 < W; i += 4) {
            const float4 t = lds_f4(wt_a + po + 4u * i);
            wz[i] = t.x, wz[i + 1] = t.y, wz[i + 2] = t.z, wz[i + 3] = t.w;
          }
          if (W % 4) {
            const float2 t = lds_f2(wt_a + po + 4u * (W - 2));
            wz[W - 2] = t.x, wz[W - 1] = t.y;
          }
          float2 u[S::PASSES];
#pragma unroll
          for (int k = 0; k < S::PASSES; ++k) u[k] = make_float2(0.f, 0.f);
#pragma unroll
          for (int iz = 0; iz < W; ++iz) {
#pragma unroll
            for (int k = 0; k < S::PASSES; ++k) u[k] = cmad(lds_f2(at + row_o[k]), wz[iz], u[k]);
            at += PB;
          }
          float2 sum = make_float2(0.f, 0.f);
#pragma unroll
          for (int k = 0; k < S::PASSES; ++k) {
            const float wy = lds_f1(wy_o[k] + po);
            sum = cmad(u[k], has[k] ? wy : 0.f, sum);
          }
          const float2 sw = cscale(sum, lds_f1(wx_o + po));
          v[2 * g4] = sw.x;
          v[2 * g4 + 1] = sw.y;
        }
        const float re = butterfly8(v, lane);
        // value l >> 2 is point l >> 3, its real part when bit 2 is 0
        const float im = __shfl_down_sync(0xffffffffu, re, 4);
        const int g4 = lane >> 3;
        if ((lane & 7) == 0 && p0 + g4 < count) f_out[jt[p0 + g4]] = make_float2(re, im);
      }
    }
    s += count;
  }
}

// Taps and squares per side: tiles of 16 x 16 columns to 10 taps (10 taps on 24
// x 24: 412 / 645 us in place of 311 / 532 above), 24 x 24 beyond.
#define GBNFFT_PENCIL_CASES(X) X(2, 2) X(4, 2) X(6, 2) X(8, 2) X(10, 2) X(12, 3) X(14, 3) X(16, 3)

}  // namespace gbnfft
