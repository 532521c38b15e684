// Products of a block-packed FP32 (or bfloat16) star inverse (BlockLayout) with r, by 9x9 blocks
// held in registers.
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

#include "common.cuh"

namespace als {

// S_IJ r_J -> yI and S_IJ^T r_I -> yJ for block b of one block-packed patch at S
// (global or shared memory).  Diagonal blocks use the symmetric upper triangle.
// Storage of the block-packed FP32-cycle inverses: float, or bfloat16 (the opt-in
// ALS_STORE_BF16) widened to float on load; every product and sum runs in float.
template <bool GLOBAL>
__device__ __forceinline__ float4 ld4(const float* p) {
  if constexpr (GLOBAL) return __ldg(reinterpret_cast<const float4*>(p));
  else return *reinterpret_cast<const float4*>(p);
}
template <bool GLOBAL>
__device__ __forceinline__ float ld1(const float* p) {
  if constexpr (GLOBAL) return __ldg(p);
  else return *p;
}
template <bool GLOBAL>
__device__ __forceinline__ float4 ld4(const __nv_bfloat16* p) {   // four entries, one 8-byte load
  uint2 u;
  if constexpr (GLOBAL) u = __ldg(reinterpret_cast<const uint2*>(p));
  else u = *reinterpret_cast<const uint2*>(p);
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
  const float2 c = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
  return make_float4(a.x, a.y, c.x, c.y);
}
template <bool GLOBAL>
__device__ __forceinline__ float ld1(const __nv_bfloat16* p) {
  if constexpr (GLOBAL) return __bfloat162float(__ldg(p));
  else return __bfloat162float(*p);
}

// entries per patch of the block-packed layout in storage TS: the packed size rounded to
// 16 bytes (bulk copies and vector loads need 16-byte aligned rows)
template <typename TS>
__host__ __device__ constexpr int block_stride(int np) {
  return sizeof(TS) == 4 ? packed_stride(np) : (packed_size(np) + 7) & ~7;
}

template <bool GLOBAL, typename TS = float>
__device__ __forceinline__ void block_product(const BlockLayout& BL, const TS* __restrict__ S, int b, bool diag,
                                              const float (&rI)[9], const float (&rJ)[9], float (&yI)[9],
                                              float (&yJ)[9]) {
  float e[84];
#pragma unroll
  for (int q = 0; q < 11; ++q) {
    const float4 v = ld4<GLOBAL>(S + 4 * (q * BL.nbp + b));
    e[4 * q] = v.x; e[4 * q + 1] = v.y; e[4 * q + 2] = v.z; e[4 * q + 3] = v.w;
  }
  e[44] = ld1<GLOBAL>(S + 44 * BL.nbp + b);
  if (!diag) {
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      const float4 v = ld4<GLOBAL>(S + BL.q2 + 4 * (q * BL.noff + b));
      e[45 + 4 * q] = v.x; e[46 + 4 * q] = v.y; e[47 + 4 * q] = v.z; e[48 + 4 * q] = v.w;
    }
  }
#pragma unroll
  for (int k = 0; k < 9; ++k) { yI[k] = 0.f; yJ[k] = 0.f; }
  if (diag) {
#pragma unroll
    for (int rr = 0; rr < 9; ++rr)
#pragma unroll
      for (int cc = rr; cc < 9; ++cc) {
        const float sv = e[rr * 9 - (rr * (rr - 1)) / 2 + (cc - rr)];
        yI[rr] += sv * rI[cc];
        if (cc != rr) yI[cc] += sv * rI[rr];
      }
  } else {
    float yI2[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) yI2[k] = 0.f;
#pragma unroll
    for (int rr = 0; rr < 9; ++rr)
#pragma unroll
      for (int cc = 0; cc < 9; ++cc) {
        const float sv = e[rr * 9 + cc];
        if (cc & 1) yI2[rr] += sv * rJ[cc];   // two independent partial sums per row
        else yI[rr] += sv * rJ[cc];
        yJ[cc] += sv * rI[rr];
      }
#pragma unroll
    for (int k = 0; k < 9; ++k) yI[k] += yI2[k];
  }
}

__device__ __forceinline__ void block_of(const BlockLayout& BL, int b, int& I, int& J, bool& diag) {
  diag = b >= BL.noff;
  I = 0;
  J = 0;
  if (diag) {
    I = J = b - BL.noff;
  } else {
    int rem = b;
    while (rem >= BL.nbr - 1 - I) { rem -= BL.nbr - 1 - I; ++I; }
    J = I + 1 + rem;
  }
}

// the role's block products of one star: role 0: a = S_01 r_1, b = S_01^T r_0; role 1: a = S_00 r_0, b = S_11 r_1
template <bool GLOBAL, typename TS>
__device__ __forceinline__ void star2_products(const TS* __restrict__ S, int role, const float (&r0)[9],
                                               const float (&r1)[9], float (&a)[9], float (&b)[9]) {
  constexpr BlockLayout BL = BlockLayout(18);
  if (role == 0) {
    block_product<GLOBAL, TS>(BL, S, 0, false, r0, r1, a, b);
  } else {
    float unused[9];
    block_product<GLOBAL, TS>(BL, S, 1, true, r0, r0, a, unused);
    block_product<GLOBAL, TS>(BL, S, 2, true, r1, r1, b, unused);
  }
}

}  // namespace als
