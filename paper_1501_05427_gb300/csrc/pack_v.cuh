// The operand images of the tensor-core contractions: columns vmap[0..R) of V (vmap null: 0, 1, ...)
// as K-major canonical BF16 images of N rows (right-hand sides) x 32 points per tile, the parts of
// a tile back to back (one bulk copy); rows r >= R and points >= n are zero.  The CTAs
// cta = 0..ctas-1 share the work.
#pragma once

#include <cuda_bf16.h>

#include "tc_common.cuh"

namespace ulisse {

// High and low part (mixed precision).
__device__ inline void pack_v2(const float* __restrict__ V, long long ldv,
                               const int* __restrict__ vmap, int R, int N, long long n,
                               long long ntiles, __nv_bfloat16* __restrict__ Vp, int cta, int ctas) {
  const int per = N * 32;
  for (long long idx = cta * (long long)blockDim.x + threadIdx.x; idx < ntiles * per;
       idx += (long long)ctas * blockDim.x) {
    const long long t = idx / per;
    const int rem = (int)(idx - t * per);
    const int r = rem / 32, jj = rem - r * 32;
    const long long j = t * 32 + jj;
    const float v = (r < R && j < n) ? V[(long long)(vmap ? vmap[r] : r) * ldv + j] : 0.f;
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    __nv_bfloat16* o = Vp + t * 2LL * per + tc::canon_offset(r, jj, 2, 4) / 2;
    o[0] = h;
    o[per] = __float2bfloat16_rn(v - __bfloat162float(h));
  }
}

// A tile of 32 points with N columns of V in three parts, and all tiles of a product: the tiles, then
// per tile and column a word with a bit for every point whose value is not finite.
constexpr size_t pack_v3_bytes(long long ntiles, int N) { return (size_t)ntiles * N * (3 * 32 * 2 + 4); }

// High, middle and low part: a float exactly (FP32 products).  The high part of the largest floats
// is rounded towards zero, as to nearest it is infinite; a value that is not finite stays whole in
// the high part.
__device__ inline void pack_v3(const float* __restrict__ V, long long ldv,
                               const int* __restrict__ vmap, int R, int N, long long n,
                               long long ntiles, __nv_bfloat16* __restrict__ Vp, int cta, int ctas) {
  const int per = N * 32;
  uint32_t* bad = reinterpret_cast<uint32_t*>(Vp + ntiles * 3LL * per);
  for (long long idx = cta * (long long)blockDim.x + threadIdx.x; idx < ntiles * per;
       idx += (long long)ctas * blockDim.x) {
    const long long t = idx / per;
    const int rem = (int)(idx - t * per);
    const int r = rem / 32, jj = rem - r * 32;
    const long long j = t * 32 + jj;
    const float v = (r < R && j < n) ? V[(long long)(vmap ? vmap[r] : r) * ldv + j] : 0.f;
    __nv_bfloat16 h = __float2bfloat16_rn(v);
    if (isinf(__bfloat162float(h))) h = __float2bfloat16_rz(v);
    const float v1 = isfinite(v) ? v - __bfloat162float(h) : 0.f;
    const __nv_bfloat16 m = __float2bfloat16_rn(v1);
    __nv_bfloat16* o = Vp + t * 3LL * per + tc::canon_offset(r, jj, 2, 4) / 2;
    o[0] = h;
    o[per] = m;
    o[2 * per] = __float2bfloat16_rn(v1 - __bfloat162float(m));
    // a warp holds the 32 points of one tile and column
    const uint32_t mask = __ballot_sync(0xffffffffu, !isfinite(v));
    if (jj == 0) bad[t * N + r] = mask;
  }
}

}  // namespace ulisse
