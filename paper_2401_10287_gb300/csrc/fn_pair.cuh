// Shared-memory layout and warp-level products of the BF16-mode pair kernels.
#pragma once
#include "fn_device.cuh"

namespace fn {

// Shared-memory position of column c of pair row `row` (32 words a row, the 8-word groups
// permuted by row mod 4): four consecutive rows' equal columns lie in different banks, and even
// column pairs stay together.
__device__ __forceinline__ int pair_at(int row, int c) { return row * 32 + (c ^ ((row & 3) << 3)); }

// c += rows (ra.., ra + 8..) of g times the weights [n][LDW] over 16 columns from k0, hi/lo splits of both.
template <int LDW>
__device__ __forceinline__ void pair_mma_k16(const float* gs, int ra, const __nv_bfloat16* whl,
                                             const __nv_bfloat16* wll, int k0, int grp, int tig, float (&c)[4][4]) {
  const int x = (k0 + 2 * tig) ^ ((ra & 3) << 3), y = (k0 + 2 * tig + 8) ^ ((ra & 3) << 3);   // ra + 8: the same permutation
  const float2 a0 = *(const float2*)(gs + ra * 32 + x), a1 = *(const float2*)(gs + (ra + 8) * 32 + x),
               a2 = *(const float2*)(gs + ra * 32 + y), a3 = *(const float2*)(gs + (ra + 8) * 32 + y);
  uint32_t ah[4], al[4];
  split_pack(a0.x, a0.y, ah[0], al[0]);
  split_pack(a1.x, a1.y, ah[1], al[1]);
  split_pack(a2.x, a2.y, ah[2], al[2]);
  split_pack(a3.x, a3.y, ah[3], al[3]);
#pragma unroll
  for (int nb = 0; nb < 4; ++nb) {
    const int off = (8 * nb + grp) * LDW + k0 + 2 * tig;
    const uint32_t bh0 = *(const uint32_t*)(whl + off), bh1 = *(const uint32_t*)(whl + off + 8);
    const uint32_t bl0 = *(const uint32_t*)(wll + off), bl1 = *(const uint32_t*)(wll + off + 8);
    mma_16816(c[nb], ah, bh0, bh1);
    mma_16816(c[nb], ah, bl0, bl1);
    mma_16816(c[nb], al, bh0, bh1);
  }
}

}  // namespace fn
