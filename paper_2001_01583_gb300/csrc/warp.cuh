// Paired FP32 arithmetic in 64-bit registers and the eight-value warp sum.
#pragma once

#include <cuda_runtime.h>

namespace gbnfft {

// Two neighbouring floats in one 64-bit register pair (a window assembled from
// scalars as float2 was copied into aligned pairs for every point: 37 moves).
using Pair = unsigned long long;
__device__ __forceinline__ Pair pair(float lo, float hi) {
  Pair p;
  asm("mov.b64 %0, {%1, %2};" : "=l"(p) : "f"(lo), "f"(hi));
  return p;
}
__device__ __forceinline__ float2 halves(Pair p) {
  float2 v;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}
// a b + c in each half, one rounding each
__device__ __forceinline__ Pair pair_fma(Pair a, Pair b, Pair c) {
  Pair d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ Pair pair_mul(Pair a, Pair b) {
  Pair d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ Pair pair_add(Pair a, Pair b) {
  Pair d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// Eight values reduced over the warp at once by a transposed butterfly (7
// shuffles): after the exchanges over lane bits 4, 3 and 2 lane l keeps its
// share of value l >> 2; the four lanes of a value have its sum between them.
__device__ __forceinline__ float butterfly8_shares(const float* v, int lane) {
  const int b4 = (lane >> 4) & 1, b3 = (lane >> 3) & 1, b2 = (lane >> 2) & 1;
  float a4[4], a2[2];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float send = b4 ? v[j] : v[4 + j];
    const float keep = b4 ? v[4 + j] : v[j];
    a4[j] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const float send = b3 ? a4[j] : a4[2 + j];
    const float keep = b3 ? a4[2 + j] : a4[j];
    a2[j] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
  const float send = b2 ? a2[0] : a2[1];
  const float keep = b2 ? a2[1] : a2[0];
  return keep + __shfl_xor_sync(0xffffffffu, send, 4);
}
// The same with the shares added up (9 shuffles): lane l returns the sum of value l >> 2.
__device__ __forceinline__ float butterfly8(const float* v, int lane) {
  float a1 = butterfly8_shares(v, lane);
  a1 += __shfl_xor_sync(0xffffffffu, a1, 2);
  a1 += __shfl_xor_sync(0xffffffffu, a1, 1);
  return a1;
}

}  // namespace gbnfft
