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
// What a lane needs to rotate its pairs (d, d + D/2), d = lane + 32 p, of a head vector; loaded apart, so that the loads can be
// under way before the vector is there.
template <int D>
struct RopeLane {
  float2 cs[D / 64];
  float glo[D / 64], ghi[D / 64];
  bool normed;
};
template <int D>
__device__ __forceinline__ void rope_load(RopeLane<D>& r, const __nv_bfloat16* gain, const float2* table, int pos) {
  const int lane = threadIdx.x & 31;
  r.normed = gain != nullptr;
#pragma unroll
  for (int p = 0; p < D / 64; ++p) {
    const int d = lane + 32 * p;
    r.cs[p] = table[(size_t)pos * (D / 2) + d];
    r.glo[p] = r.normed ? __bfloat162float(gain[d]) : 1.f;
    r.ghi[p] = r.normed ? __bfloat162float(gain[d + D / 2]) : 1.f;
  }
}
// the pairs lo[p], hi[p] normalised (if the model does), rotated and stored to dst
template <int D>
__device__ __forceinline__ void rope_head(float (&lo)[D / 64], float (&hi)[D / 64], const RopeLane<D>& rl, float eps, __nv_bfloat16* dst) {
  const int lane = threadIdx.x & 31;
  if (rl.normed) {
    float ss = 0.f;
#pragma unroll
    for (int p = 0; p < D / 64; ++p) ss += lo[p] * lo[p] + hi[p] * hi[p];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    const float r = 1.0f / sqrtf(ss / (float)D + eps);
#pragma unroll
    for (int p = 0; p < D / 64; ++p) {
      lo[p] = lo[p] * r * rl.glo[p];
      hi[p] = hi[p] * r * rl.ghi[p];
    }
  }
#pragma unroll
  for (int p = 0; p < D / 64; ++p) {
    const int d = lane + 32 * p;
    dst[d] = __float2bfloat16_rn(lo[p] * rl.cs[p].x - hi[p] * rl.cs[p].y);
    dst[d + D / 2] = __float2bfloat16_rn(hi[p] * rl.cs[p].x + lo[p] * rl.cs[p].y);
  }
}
#endif

}  // namespace quasar
