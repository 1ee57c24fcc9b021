// Pieces shared by the kernels with an mma.sync contraction and a tcgen05
// inverse DFT (k_umma256.cu, k_umma512.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cstdint>

namespace mra {

template <bool FP16>
__device__ __forceinline__ void mma_frag(float (&d)[4], const uint4 &a, uint32_t b0, uint32_t b1) {
  if constexpr (FP16)
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
  else
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t pack_bf2u(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t *>(&h);
}

__device__ __forceinline__ uint4 load_frag(const unsigned char *p) {
  uint4 v;
  asm volatile("ld.global.nc.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

// Per k-step accumulators d of one (row, reference) pair and frequency ->
// {2 Re C, 2 Re C', 2 Im C, 2 Im C'} (see k_umma256.cu).
__device__ __forceinline__ void pair_sums(const float (&d)[4], float (&v)[4]) {
  v[0] = d[0] + d[3];
  v[1] = d[1] + d[2];
  v[2] = d[1] - d[2];
  v[3] = d[3] - d[0];
}

// Units of work are (row tile, range of reference tiles): `splits` ranges
// per row tile, chosen to minimise the time of the fullest SM,
// waves x (tiles per unit + the unit's load of its row fragments, about one
// tile).  One range when the row tiles fill many waves (each row tile's
// fragments are then loaded once); more when the stack is so small that
// whole row tiles would leave SMs idle.
inline int pick_splits(int64_t row_tiles, int ref_tiles, int sms) {
  int best = 1;
  int64_t best_cost = INT64_MAX;
  for (int s = 1; s <= ref_tiles; ++s) {
    const int per = (ref_tiles + s - 1) / s;
    if ((ref_tiles + per - 1) / per != s) continue;  // ranges must not be empty
    const int64_t cost = (row_tiles * s + sms - 1) / sms * (per + 1);
    if (cost < best_cost) {
      best_cost = cost;
      best = s;
    }
  }
  return best;
}

}  // namespace mra
