// Real-space part of the Ewald energy, Eq. 11 (Section 5):
//   U^R = 1/2 sum'_n sum_{i,j} q_i q_j erfc(alpha |r_ij + n L|) / |r_ij + n L|
// over the pairs (and periodic images) closer than a cut-off r_c; the primed
// sum omits n = 0 for i = j.
//
// Three forms:
//   - columns (L / r_c >= 3): the box is cut into columns along z of edge
//     L / ncol >= r_c / 3, each cut into fine z bins, and the ions are
//     counting-sorted by (column, bin), so a column's ions are contiguous and
//     nearly ordered by z.  A warp takes two ions of one column; for each of
//     the 7 x 7 columns around it that comes within r_c it works out the z
//     range that does and runs its lanes over the ions of that range, both
//     partners of a lane's ion in the two halves of paired FP32 instructions.
//     47% of the candidates are partners; of the 125 cells of edge r_c / 2
//     around an ion, a thread per ion, 23% were, and every candidate ran the
//     whole pair term because one lane of 32 accepted it.  393216 ions,
//     r_c = 10, about 4000 partners each, with forces, a call: 13.2 -> 5.5 ms
//     (5.2 with FP32 sums per ion).  It is bound by issue and the FP32 pipe: 70
//     instructions per 64 candidates, 25 of them paired operations of two cycles,
//     and about 35 per range for its sums;
//     Lengths are in units of L.  An ion's x and y are FP32 offsets from its
//     column's axis, its z the sum of a multiple of 2^-10 and an FP32 remainder:
//     a separation along z is rounded to FP32 once, along x and y with its
//     columns' distance and its offsets, an error of at most 2e-8 L between
//     neighbours and 5e-8 L between third neighbours of 9 columns a side, 1.2e-9 and
//     2e-9 L of 128.  Pair terms and the sums over a range are FP32, an ion's sums
//     over its ranges FP64;
//   - the same with few partners and many ions (cell_partners): cells of edge
//     L / nc >= r_c / 2, a thread per ion over the 5^3 cells around its own.  A
//     range of the columns then holds fewer ions than a warp has lanes (13 of 32
//     at 250 partners), while this form's work falls with the partners.  FP32
//     offsets from the cells' centres, FP32 pair terms and sums over a cell, FP64
//     over the cells;
//     In both, with r_c <= L / 3 only the minimum image of a pair can be within
//     r_c, and it is found exactly once;
//   - all pairs (smaller boxes): the minimum image of every pair plus the 26
//     shifts by L, all in FP64, which is the definition itself (r_c < L).
// The energy 1/2 sum_i q_i phi_i is reduced in FP64, the blocks' partials in a
// fixed order; the order of ions inside a bin (atomics) and with it the last
// bits of an ion's FP32 sums change from run to run.
//
// Forces (the negative gradient of Eq. 11; the paper names MD as the use but
// prints no force formula): F_i = q_i sum_j q_j g(d) (r_i - r_j + n L) with
// g(d) = (erfc(alpha d) / d + 2 alpha / sqrt(pi) exp(-alpha^2 d^2)) / d^2,
// summed by the same forms (each ion sums its own force, no atomics).
#include <cmath>
#include <cstdint>

#include "gbnfft.h"
#include "kernels.h"
#include "warp.cuh"

namespace gbnfft {
namespace {

constexpr int kRsThreads = 256;
constexpr int kRsReach = 3;     // neighbour columns per side (column edge >= r_c / kRsReach)
constexpr int kRsCellReach = 2; // neighbour cells per side (cell edge >= r_c / kRsCellReach)
constexpr int kRsColumns = (2 * kRsReach + 1) * (2 * kRsReach + 1);
constexpr int kRsIons = 8;      // most ions a warp takes, two at a time
// Partners per ion (on average) below which the cells are taken: 500, and
// fewer where the ions do not fill the chip with threads (x ions per SM).  The
// cells' time is then the latency of one thread, about 345 + 0.92 us per
// partner, that of the columns about 300 + 1.27 x.  Forces, uniform ions, cells /
// columns: 36,000 ions and 120 partners 480 / 583 us, 300: 638 / 600; 165,888 ions
// and 60: 712 / 1264, 500: 1322 / 1244; 393,216 ions and 60: 1181 / 2485, 400: 2025
// / 2361, 1000: 3742 / 2630.
inline double cell_partners(double ions_per_sm) { return std::min(500.0, 1.4 * ions_per_sm - 50.0); }
constexpr double kRsGrid = 1024.0;

// (v, v), kept in its registers (the compiler rebuilt constant pairs in the loop).
__device__ __forceinline__ Pair pinned_pair(float v) {
  Pair p;
  asm volatile("mov.b64 %0, {%1, %1};" : "=l"(p) : "f"(v));
  return p;
}
// The hardware's 2^x, 1 / x and 1 / sqrt(x) (a few ulp) in both halves.
__device__ __forceinline__ Pair pair_exp2(Pair p) {
  const float2 v = halves(p);
  float a, b;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(a) : "f"(v.x));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(b) : "f"(v.y));
  return pair(a, b);
}
__device__ __forceinline__ Pair pair_rcp(Pair p) {
  const float2 v = halves(p);
  float a, b;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(a) : "f"(v.x));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(b) : "f"(v.y));
  return pair(a, b);
}
__device__ __forceinline__ Pair pair_rsqrt(Pair p) {
  const float2 v = halves(p);
  float a, b;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(a) : "f"(v.x));
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(b) : "f"(v.y));
  return pair(a, b);
}

__device__ __forceinline__ double warp_sum_f64(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block sum of v into partial[blockIdx.x] (fixed order).
__device__ __forceinline__ void block_partial(double v, double* partial) {
  __shared__ double ws[kRsThreads / 32];
  v = warp_sum_f64(v);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) ws[warp] = v;
  __syncthreads();
  if (warp == 0) {
    double s = lane < (int)(blockDim.x >> 5) ? ws[lane] : 0.0;
    s = warp_sum_f64(s);
    if (lane == 0) partial[blockIdx.x] = s;
  }
}

// Fraction of the box edge in [0, 1), and its cell of n.
__device__ __forceinline__ double rs_fraction(double r, double L) {
  const double u = r / L;
  const double s = u - floor(u);
  return s < 1.0 ? s : 0.0;
}
__device__ __forceinline__ int rs_cell(double s, int n) { return min((int)(s * n), n - 1); }

// (Column, z bin) of each ion and its rank there (cells: ncol = nz).
__global__ void k_rs_count(int64_t n, const double* __restrict__ r, double L, int ncol, int nz, int* __restrict__ count,
                           int2* __restrict__ cell_rank) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int cx = rs_cell(rs_fraction(r[i * 3], L), ncol), cy = rs_cell(rs_fraction(r[i * 3 + 1], L), ncol);
  const int cell = (cx * ncol + cy) * nz + rs_cell(rs_fraction(r[i * 3 + 2], L), nz);
  cell_rank[i] = make_int2(cell, atomicAdd(&count[cell], 1));
}

// Sorted records: (x, y offsets from the column's axis, z in two parts), the
// charge and the column.
__global__ void k_rs_scatter(int64_t n, const double* __restrict__ r, const double* __restrict__ q, double L, int ncol,
                             int nz, const int* __restrict__ start, const int2* __restrict__ cell_rank,
                             float4* __restrict__ rec, float* __restrict__ rec_q, int* __restrict__ rec_col,
                             int* __restrict__ rec_idx) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int2 cr = cell_rank[i];
  const int col = cr.x / nz;
  const double sx = rs_fraction(r[i * 3], L), sy = rs_fraction(r[i * 3 + 1], L), sz = rs_fraction(r[i * 3 + 2], L);
  const double zh = floor(sz * kRsGrid) / kRsGrid;
  const int p = start[cr.x] + cr.y;
  rec[p] = make_float4((float)(sx - (col / ncol + 0.5) / ncol), (float)(sy - (col % ncol + 0.5) / ncol), (float)zh,
                       (float)(sz - zh));
  // an ion without a position takes no part
  const bool placed = isfinite(r[i * 3]) && isfinite(r[i * 3 + 1]) && isfinite(r[i * 3 + 2]);
  rec_q[p] = placed ? (float)q[i] : 0.f;
  rec_col[p] = col;
  if (rec_idx) rec_idx[p] = (int)i;
}

// The same for cells: offsets from the cell's centre and the charge.
__global__ void k_rs_scatter_cells(int64_t n, const double* __restrict__ r, const double* __restrict__ q, double L,
                                   int nc, const int* __restrict__ start, const int2* __restrict__ cell_rank,
                                   float4* __restrict__ rec, int* __restrict__ rec_cell, int* __restrict__ rec_idx) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int2 cr = cell_rank[i];
  const int cc[3] = {cr.x / (nc * nc), cr.x / nc % nc, cr.x % nc};
  const double h = L / nc;
  float o[3];
  bool placed = true;
  for (int t = 0; t < 3; ++t) {
    const double x = r[i * 3 + t];
    placed = placed && isfinite(x);
    o[t] = (float)(rs_fraction(x, L) * L - (cc[t] + 0.5) * h);
  }
  const int p = start[cr.x] + cr.y;
  rec[p] = make_float4(o[0], o[1], o[2], placed ? (float)q[i] : 0.f);
  rec_cell[p] = cr.x;
  if (rec_idx) rec_idx[p] = (int)i;
}

constexpr float kTwoOverSqrtPiF = 1.1283791670955126f;
constexpr double kTwoOverSqrtPi = 1.1283791670955126;

// Few partners: a thread per sorted ion over the cells around its own; block
// partials of q_i phi_i.  FORCES: also the ion's force, written to its
// original index (F: n x 3 doubles).
template <bool FORCES>
__global__ void __launch_bounds__(kRsThreads) k_rs_cells(int n, int nc, float h, float rc2, float alpha,
                                                         const float4* __restrict__ rec,
                                                         const int* __restrict__ rec_cell,
                                                         const int* __restrict__ start, double* __restrict__ partial,
                                                         const int* __restrict__ rec_idx, double* __restrict__ F) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  double e = 0.0;
  if (i < n) {
    const float4 pi = rec[i];
    const int cell = rec_cell[i];
    const int cz = cell % nc, cy = cell / nc % nc, cx = cell / (nc * nc);
    double phi = 0.0, fx = 0.0, fy = 0.0, fz = 0.0;
    const float c2 = kTwoOverSqrtPiF * alpha, a2 = alpha * alpha;
    for (int dx = -kRsCellReach; dx <= kRsCellReach; ++dx) {
      const int x = cx + dx < 0 ? cx + dx + nc : (cx + dx >= nc ? cx + dx - nc : cx + dx);
      for (int dy = -kRsCellReach; dy <= kRsCellReach; ++dy) {
        const int y = cy + dy < 0 ? cy + dy + nc : (cy + dy >= nc ? cy + dy - nc : cy + dy);
        for (int dz = -kRsCellReach; dz <= kRsCellReach; ++dz) {
          const int z = cz + dz < 0 ? cz + dz + nc : (cz + dz >= nc ? cz + dz - nc : cz + dz);
          const int nb = (x * nc + y) * nc + z;
          const float sx = dx * h - pi.x, sy = dy * h - pi.y, sz = dz * h - pi.z;
          float acc = 0.0f, ax = 0.0f, ay = 0.0f, az = 0.0f;
          for (int j = start[nb]; j < start[nb + 1]; ++j) {
            const float4 pj = rec[j];
            const float rx = pj.x + sx, ry = pj.y + sy, rz = pj.z + sz;   // r_j - r_i
            const float d2 = rx * rx + ry * ry + rz * rz;
            if (d2 < rc2 && d2 > 0.0f) {
              const float rinv = rsqrtf(d2);
              const float ec = erfcf(alpha * d2 * rinv) * rinv;
              acc += pj.w * ec;
              if (FORCES) {
                const float g = pj.w * (ec + c2 * __expf(-a2 * d2)) * rinv * rinv;
                ax -= g * rx;
                ay -= g * ry;
                az -= g * rz;
              }
            }
          }
          phi += (double)acc;
          if (FORCES) {
            fx += (double)ax;
            fy += (double)ay;
            fz += (double)az;
          }
        }
      }
    }
    e = (double)pi.w * phi;
    if (FORCES) {
      const int64_t o = (int64_t)rec_idx[i] * 3;
      F[o] = (double)pi.w * fx;
      F[o + 1] = (double)pi.w * fy;
      F[o + 2] = (double)pi.w * fz;
    }
  }
  block_partial(e, partial);
}

// erfc(x) e^(x^2) for x >= 0 as t P(t), t = 1 / (1 + 0.42 x): P is the
// least relative error polynomial of degree 7 over x in [0, 6.5] (Chebyshev
// fit with iterated weights): 4e-8, 1e-7 with FP32 rounding.  Beyond, e^(-x^2)
// is below 1e-18.
constexpr float kErfcScale = 0.42f;

struct RsParams {
  int n, ncol, nz;
  int per_warp;     // ions a warp takes: even, at most kRsIons
  float rc2, near;  // (r_c / L)^2, r_c / (4 L)
  float alpha;      // alpha L
  float escale;     // -(alpha L)^2 log2(e)
  float c2;         // 2 alpha L / sqrt(pi)
  double phi_scale, f_scale;   // 1 / L, 1 / L^2
};

// A range of ions in a column: the offsets of its axis, the z shift of its image.
struct RsRange {
  int begin, end;
  float dx, dy, dz;
};

// Potential (and force) of each sorted ion; block partials of q_i phi_i.
// FORCES: also the ion's force, written to its original index (F: n x 3).
template <bool FORCES>
__global__ void __launch_bounds__(kRsThreads, 4) k_rs_columns(RsParams P, const float4* __restrict__ rec,
                                                           const float* __restrict__ rec_q,
                                                           const int* __restrict__ rec_col,
                                                           const int* __restrict__ start, double* __restrict__ partial,
                                                           const int* __restrict__ rec_idx, double* __restrict__ F) {
  __shared__ RsRange ranges[kRsThreads / 32][2 * kRsColumns];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  RsRange* mine = ranges[warp];
  const int first = (blockIdx.x * (kRsThreads / 32) + warp) * P.per_warp, last = min(P.n, first + P.per_warp);
  const float inv = 1.0f / (float)P.ncol, half = 0.5f * inv;
  constexpr float kErfc[8] = {0.236731262f, 0.240897215f,  0.187104512f,  0.292422239f,
                              -0.17306915f, 0.48496216f,   -0.345052719f, 0.0760044978f};
  // added to every squared distance, so that the pair term of an ion with
  // itself (masked) stays finite; far below what the records resolve
  constexpr float tiny = 1e-20f;
  Pair cf[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) cf[c] = pinned_pair(kErfc[c]);
  const Pair ps = pinned_pair(kErfcScale * P.alpha), one = pinned_pair(1.f), tn = pinned_pair(tiny);
  const Pair es = pinned_pair(P.escale), c2 = pinned_pair(P.c2);
  const float rc2 = P.rc2;
  double e = 0.0;
  for (int i = first; i < last;) {
    // two ions of one column, or one (then both halves hold it)
    const int col = rec_col[i];
    const float4 pa = rec[i];
    float4 pb = rec[min(i + 1, P.n - 1)];
    const float za = pa.z + pa.w;
    float zb = pb.z + pb.w;
    // close in z as well: their common range then wraps on one side at most
    const bool two = i + 1 < last && rec_col[i + 1] == col && fabsf(zb - za) <= P.near;
    if (!two) {
      pb = pa;
      zb = za;
    }
    const int cx = col / P.ncol, cy = col - cx * P.ncol;
    // the ranges of the columns around: up to two each (the z period)
    int count = 0;
    __syncwarp();
    for (int t0 = 0; t0 < kRsColumns; t0 += 32) {
      const int t = t0 + lane;
      const int ix = t / (2 * kRsReach + 1) - kRsReach, iy = t % (2 * kRsReach + 1) - kRsReach;
      RsRange rg;
      rg.dx = (float)ix * inv;
      rg.dy = (float)iy * inv;
      rg.dz = 0.f;
      const float mx = fmaxf(fminf(fabsf(rg.dx - pa.x), fabsf(rg.dx - pb.x)) - half, 0.f);
      const float my = fmaxf(fminf(fabsf(rg.dy - pa.y), fabsf(rg.dy - pb.y)) - half, 0.f);
      const float left = P.rc2 * 1.00001f - mx * mx - my * my;
      int b0 = 0, b1 = -1, w0 = 0, w1 = -1;   // bins in the box, and of the image above or below
      float wz = 0.f;
      int base = 0;
      if (t < kRsColumns && left > 0.f) {
        const int x = cx + ix < 0 ? cx + ix + P.ncol : (cx + ix >= P.ncol ? cx + ix - P.ncol : cx + ix);
        const int y = cy + iy < 0 ? cy + iy + P.ncol : (cy + iy >= P.ncol ? cy + iy - P.ncol : cy + iy);
        base = (x * P.ncol + y) * P.nz;
        const float reach = sqrtf(left);
        b0 = (int)floorf((fminf(za, zb) - reach) * (float)P.nz - 1e-3f);
        b1 = (int)floorf((fmaxf(za, zb) + reach) * (float)P.nz + 1e-3f);
        if (b0 < 0) {
          w0 = b0 + P.nz, w1 = P.nz - 1, wz = -1.f;
          b0 = 0;
        } else if (b1 >= P.nz) {
          w0 = 0, w1 = b1 - P.nz, wz = 1.f;
          b1 = P.nz - 1;
        }
      }
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int lo = k ? w0 : b0, hi = k ? w1 : b1;
        bool some = lo <= hi;
        if (some) {
          rg.begin = start[base + lo];
          rg.end = start[base + hi + 1];
          if (k) rg.dz = wz;
          some = rg.begin < rg.end;
        }
        const unsigned mask = __ballot_sync(0xffffffffu, some);
        if (some) mine[count + __popc(mask & ((1u << lane) - 1u))] = rg;
        count += __popc(mask);
      }
    }
    __syncwarp();
    double sum = 0.0;   // lane l: its share of value l >> 2 of (phi, f) of the first ion, then of the second
    for (int k = 0; k < count; ++k) {
      const RsRange rg = mine[k];
      const float sxa = rg.dx - pa.x, sxb = rg.dx - pb.x, sya = rg.dy - pa.y, syb = rg.dy - pb.y;
      Pair phi = 0, fx = 0, fy = 0, fz = 0;   // a range's sums: FP32, over its lanes too; FP64 over the ranges
      const float sha = rg.dz - pa.z, shb = rg.dz - pb.z, sla = -pa.w, slb = -pb.w;
#pragma unroll 2
      for (int j0 = rg.begin; j0 < rg.end; j0 += 32) {
        const int j = min(j0 + lane, rg.end - 1);
        const float4 rj = __ldg(rec + j);
        const float qj = j0 + lane < rg.end ? __ldg(rec_q + j) : 0.f;
        // single adds: a paired one would first copy rj into both halves
        const Pair X = pair(rj.x + sxa, rj.x + sxb), Y = pair(rj.y + sya, rj.y + syb);
        const Pair Z = pair_add(pair(rj.z + sha, rj.z + shb), pair(rj.w + sla, rj.w + slb));
        const Pair d2p = pair_fma(Z, Z, pair_fma(Y, Y, pair_fma(X, X, tn)));
        const float2 d2 = halves(d2p);
        const float qa = d2.x < rc2 && d2.x > tiny ? qj : 0.f, qb = d2.y < rc2 && d2.y > tiny ? qj : 0.f;
        const Pair rinv = pair_rsqrt(d2p);
        const Pair t = pair_rcp(pair_fma(pair_mul(d2p, rinv), ps, one)), ee = pair_exp2(pair_mul(d2p, es));
        Pair w = cf[7];
#pragma unroll
        for (int c = 6; c >= 0; --c) w = pair_fma(w, t, cf[c]);
        const Pair q2 = pair(qa, qb);
        const Pair ec = pair_mul(pair_mul(pair_mul(w, t), ee), rinv);   // erfc(alpha r) / r
        phi = pair_fma(q2, ec, phi);
        if (FORCES) {
          const Pair g = pair_mul(pair_mul(pair_fma(ee, c2, ec), pair_mul(rinv, rinv)), q2);
          fx = pair_fma(g, X, fx);
          fy = pair_fma(g, Y, fy);
          fz = pair_fma(g, Z, fz);
        }
      }
      const float2 p2 = halves(phi);
      if (FORCES) {
        const float2 x2 = halves(fx), y2 = halves(fy), z2 = halves(fz);
        const float v[8] = {p2.x, x2.x, y2.x, z2.x, p2.y, x2.y, y2.y, z2.y};
        sum += (double)butterfly8_shares(v, lane);
      } else {
        const bool second = lane >= 16;
        sum += (double)((second ? p2.y : p2.x) + __shfl_xor_sync(0xffffffffu, second ? p2.x : p2.y, 16));
      }
    }
#pragma unroll
    for (int o = FORCES ? 2 : 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    const int which = lane >> 4, comp = (lane >> 2) & 3;
    if ((lane & 3) == 0 && (which == 0 || two)) {
      const double qi = (double)rec_q[i + which];
      if (comp == 0) e += qi * sum * P.phi_scale;
      else if (FORCES) F[(int64_t)rec_idx[i + which] * 3 + comp - 1] = -qi * sum * P.f_scale;
    }
    i += two ? 2 : 1;
  }
  block_partial(e, partial);
}

// All pairs with the minimum image and the 26 shifts by L, FP64.  FORCES:
// also each ion's force (F: n x 3 doubles, input order).
template <bool FORCES>
__global__ void __launch_bounds__(kRsThreads) k_rs_pairs(int n, const double* __restrict__ r,
                                                         const double* __restrict__ q, double L, double rc,
                                                         double alpha, double* __restrict__ partial,
                                                         double* __restrict__ F) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  double e = 0.0;
  if (i < n) {
    const double xi = r[3 * i], yi = r[3 * i + 1], zi = r[3 * i + 2];
    double phi = 0.0, fx = 0.0, fy = 0.0, fz = 0.0;
    for (int j = 0; j < n; ++j) {
      double d[3] = {xi - r[3 * j], yi - r[3 * j + 1], zi - r[3 * j + 2]};
      for (int t = 0; t < 3; ++t) d[t] -= L * rint(d[t] / L);
      for (int s = 0; s < 27; ++s) {
        const double ax = d[0] + (s / 9 - 1) * L, ay = d[1] + ((s / 3) % 3 - 1) * L, az = d[2] + (s % 3 - 1) * L;
        const double dist = sqrt(ax * ax + ay * ay + az * az);
        if (dist > 0.0 && dist < rc) {
          const double ec = erfc(alpha * dist) / dist;
          phi += q[j] * ec;
          if (FORCES) {
            const double g = q[j] * (ec + kTwoOverSqrtPi * alpha * exp(-alpha * alpha * dist * dist)) / (dist * dist);
            fx += g * ax;   // (r_i - r_j + n L)
            fy += g * ay;
            fz += g * az;
          }
        }
      }
    }
    e = q[i] * phi;
    if (FORCES) {
      F[3 * i] = q[i] * fx;
      F[3 * i + 1] = q[i] * fy;
      F[3 * i + 2] = q[i] * fz;
    }
  }
  block_partial(e, partial);
}

// Fixed-order sum of the block partials; out = scale * sum.
__global__ void __launch_bounds__(kRsThreads) k_rs_total(const double* __restrict__ partial, int count, double scale,
                                                         double* __restrict__ out) {
  double s = 0.0;
  for (int k = threadIdx.x; k < count; k += blockDim.x) s += partial[k];
  block_partial(s, out);                    // thread 0 writes out[0]
  if (threadIdx.x == 0) out[0] *= scale;
}

}  // namespace
}  // namespace gbnfft

namespace gbnfft {
namespace {

// The energy (and with F the forces) of Eq. 11: shared by both entry points.
int real_space_impl(int64_t n, const double* r_dev, const double* q_dev, double L, double alpha, double rcut,
                    double* energy, double* F_dev, void* cuda_stream) {
  if (n < 0 || !energy || (n > 0 && (!r_dev || !q_dev))) return NFFT_ERR_INVALID_ARG;
  if (!(L > 0.0) || !(alpha > 0.0) || !(rcut > 0.0) || !(rcut < L) || !std::isfinite(L) || !std::isfinite(alpha))
    return NFFT_ERR_INVALID_ARG;
  if (n > ((int64_t)1 << 30)) return NFFT_ERR_UNSUPPORTED;
  *energy = 0.0;
  if (n == 0) return NFFT_OK;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  // L / rcut < 3: all pairs
  const bool sorted = std::floor(L / rcut) >= 3;
  if (!sorted && n > 65536) return NFFT_ERR_UNSUPPORTED;   // the all-pairs form is O(n^2)
  const int ni = (int)n;
  const int blocks = (ni + kRsThreads - 1) / kRsThreads;
  int device = 0, sms = 0;
  if (cudaGetDevice(&device) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) {
    cudaGetLastError();
    return NFFT_ERR_CUDA;
  }
  const double partners = 4.0 / 3.0 * M_PI * rcut * rcut * rcut / (L * L * L) * (double)n;
  const bool cells_form = sorted && partners < cell_partners((double)n / sms);
  // columns of edge L / side >= rcut / kRsReach (at least 9 per side, so the
  // 7 x 7 around one are distinct), z bins a quarter of that; or cells of edge
  // L / side >= rcut / kRsCellReach (at least 6 per side)
  const int side = !sorted ? 1
                   : cells_form ? (int)std::min(std::floor(kRsCellReach * L / rcut), 256.0)
                                : (int)std::min(std::floor(kRsReach * L / rcut), 128.0);
  const int nz = cells_form ? side : 4 * side;
  // As many ions per warp as still give the chip's resident warps (32 on each
  // SM) one each; a warp's ranges serve all its ions in turn.  With 8
  // each throughout, few ions left SMs idle: forces of 2592 ions 395 -> 325 us,
  // 6144: 402 -> 350, 12000: 512 -> 421, 20736: 611 -> 541; 49152: 1155 either way.
  const int per_warp = std::min(std::max(2 * (ni / (2 * 32 * sms)), 2), kRsIons);
  const int per_block = kRsThreads / 32 * per_warp;
  const int parts = sorted && !cells_form ? (ni + per_block - 1) / per_block : blocks;
  const int cells = side * side * nz;
  // scratch: partials and the total, and for the sorted forms records, charges,
  // (cell, rank), columns, counts, starts, scan scratch and record indices
  size_t bytes = sizeof(double) * (size_t)(parts + 1);
  if (sorted) {
    bytes += 16 + (sizeof(float4) + sizeof(int2) + sizeof(float) + sizeof(int)) * ((size_t)n + 1) +
             sizeof(int) * ((size_t)(2 * cells + 2) + (size_t)scan_partials_needed(cells + 1)) +
             (F_dev ? sizeof(int) * (size_t)n : 0);
  }
  char* buf = nullptr;
  if (cudaMalloc(&buf, bytes) != cudaSuccess) {
    cudaGetLastError();
    return NFFT_ERR_OOM;
  }
  int status = NFFT_OK;
  auto ck = [&](cudaError_t e) {
    if (e != cudaSuccess && status == NFFT_OK) status = NFFT_ERR_CUDA;
  };
  double* partial = reinterpret_cast<double*>(buf);
  double* total = partial + parts;
  if (sorted) {
    char* p = buf + sizeof(double) * (size_t)(parts + 1);
    float4* rec = reinterpret_cast<float4*>((reinterpret_cast<uintptr_t>(p) + 15) & ~(uintptr_t)15);
    int2* cell_rank = reinterpret_cast<int2*>(rec + n);
    float* rec_q = reinterpret_cast<float*>(cell_rank + n);
    int* rec_col = reinterpret_cast<int*>(rec_q + n);
    int* count = rec_col + n;
    int* start = count + cells + 1;
    int* scan_scratch = start + cells + 1;
    int* rec_idx = F_dev ? scan_scratch + scan_partials_needed(cells + 1) : nullptr;
    ck(cudaMemsetAsync(count, 0, sizeof(int) * (size_t)(cells + 1), st));
    k_rs_count<<<blocks, kRsThreads, 0, st>>>(n, r_dev, L, side, nz, count, cell_rank);
    ck(cudaGetLastError());
    ck(launch_scan(count, start, cells + 1, nullptr, scan_scratch, false, st));   // start[cells] = n
    if (cells_form) {
      k_rs_scatter_cells<<<blocks, kRsThreads, 0, st>>>(n, r_dev, q_dev, L, side, start, cell_rank, rec, rec_col,
                                                        rec_idx);
      ck(cudaGetLastError());
      const float h = (float)(L / side), rc2 = (float)(rcut * rcut);
      if (F_dev)
        k_rs_cells<true><<<blocks, kRsThreads, 0, st>>>(ni, side, h, rc2, (float)alpha, rec, rec_col, start, partial,
                                                        rec_idx, F_dev);
      else
        k_rs_cells<false><<<blocks, kRsThreads, 0, st>>>(ni, side, h, rc2, (float)alpha, rec, rec_col, start, partial,
                                                         nullptr, nullptr);
      ck(cudaGetLastError());
    } else {
      k_rs_scatter<<<blocks, kRsThreads, 0, st>>>(n, r_dev, q_dev, L, side, nz, start, cell_rank, rec, rec_q, rec_col,
                                                  rec_idx);
      ck(cudaGetLastError());
      RsParams P;
      P.n = ni;
      P.ncol = side;
      P.nz = nz;
      P.per_warp = per_warp;
      P.rc2 = (float)(rcut / L * (rcut / L));
      P.near = (float)(0.25 * rcut / L);
      P.alpha = (float)(alpha * L);
      P.escale = (float)(-alpha * L * alpha * L * 1.4426950408889634);
      P.c2 = (float)(kTwoOverSqrtPi * alpha * L);
      P.phi_scale = 1.0 / L;
      P.f_scale = 1.0 / (L * L);
      if (F_dev)
        k_rs_columns<true><<<parts, kRsThreads, 0, st>>>(P, rec, rec_q, rec_col, start, partial, rec_idx, F_dev);
      else
        k_rs_columns<false><<<parts, kRsThreads, 0, st>>>(P, rec, rec_q, rec_col, start, partial, nullptr, nullptr);
      ck(cudaGetLastError());
    }
  } else {
    if (F_dev)
      k_rs_pairs<true><<<blocks, kRsThreads, 0, st>>>(ni, r_dev, q_dev, L, rcut, alpha, partial, F_dev);
    else
      k_rs_pairs<false><<<blocks, kRsThreads, 0, st>>>(ni, r_dev, q_dev, L, rcut, alpha, partial, nullptr);
    ck(cudaGetLastError());
  }
  k_rs_total<<<1, kRsThreads, 0, st>>>(partial, parts, 0.5, total);
  ck(cudaGetLastError());
  double host = 0.0;
  ck(cudaMemcpyAsync(&host, total, sizeof(double), cudaMemcpyDeviceToHost, st));
  ck(cudaStreamSynchronize(st));
  cudaFree(buf);
  if (status == NFFT_OK) *energy = host;
  return status;
}

}  // namespace
}  // namespace gbnfft

extern "C" int nfft_ewald_real_space(int64_t n, const double* r_dev, const double* q_dev, double L, double alpha,
                                     double rcut, double* energy, void* cuda_stream) {
  return gbnfft::real_space_impl(n, r_dev, q_dev, L, alpha, rcut, energy, nullptr, cuda_stream);
}

extern "C" int nfft_ewald_real_space_forces(int64_t n, const double* r_dev, const double* q_dev, double L,
                                            double alpha, double rcut, double* F_dev, double* energy,
                                            void* cuda_stream) {
  if (n > 0 && !F_dev) return NFFT_ERR_INVALID_ARG;
  return gbnfft::real_space_impl(n, r_dev, q_dev, L, alpha, rcut, energy, n > 0 ? F_dev : nullptr, cuda_stream);
}
