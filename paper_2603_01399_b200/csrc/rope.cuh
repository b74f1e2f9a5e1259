// QK-RMSNorm + RoPE of one head vector by a warp, and where the rows of a block go in the KV cache.
#pragma once

#include "common.cuh"

namespace quasar {

struct RopeArgs {
  __nv_bfloat16* qkv;            // [M][(Hq+2Hkv)*D]
  const __nv_bfloat16* q_norm;   // [D] or nullptr
  const __nv_bfloat16* k_norm;
  const float2* table;           // [position][D/2] cosine, sine
  const int32_t *seq_len, *block_len;
  BlockInfo bi;
  __nv_bfloat16 *k_cache, *v_cache;   // this layer's: [B][Hkv][s_max][D]
  int T_max, Hq, Hkv, D, s_max;
  float eps;
};

#ifdef __CUDACC__
// Lane l holds the rotation pairs (d, d + D/2), d = l + 32 p, in lo[p], hi[p]; they are normalised (gain not null), rotated to
// position `pos` and stored to dst.
template <int D>
__device__ __forceinline__ void rope_head(float (&lo)[D / 64], float (&hi)[D / 64], const __nv_bfloat16* gain, const float2* table,
                                          int pos, float eps, __nv_bfloat16* dst) {
  const int lane = threadIdx.x & 31;
  if (gain != nullptr) {
    float ss = 0.f;
#pragma unroll
    for (int p = 0; p < D / 64; ++p) ss += lo[p] * lo[p] + hi[p] * hi[p];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    const float r = 1.0f / sqrtf(ss / (float)D + eps);
#pragma unroll
    for (int p = 0; p < D / 64; ++p) {
      const int d = lane + 32 * p;
      lo[p] = lo[p] * r * __bfloat162float(gain[d]);
      hi[p] = hi[p] * r * __bfloat162float(gain[d + D / 2]);
    }
  }
#pragma unroll
  for (int p = 0; p < D / 64; ++p) {
    const int d = lane + 32 * p;
    const float2 cs = table[(size_t)pos * (D / 2) + d];
    dst[d] = __float2bfloat16_rn(lo[p] * cs.x - hi[p] * cs.y);
    dst[d + D / 2] = __float2bfloat16_rn(hi[p] * cs.x + lo[p] * cs.y);
  }
}
#endif

}  // namespace quasar
