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

// What a row of a 128-channel tile (one head of 128, or two of 64) needs besides its values, and whether it takes part.
struct RopeRow {
  RopeLane<128> r128;
  RopeLane<64> r64[2];
  int slot;   // the row's cache position, or -1
};
__device__ __forceinline__ void rope_row_load(RopeRow& p, const RopeArgs& r, int m, int n0) {
  const int b = m / r.T_max, i = m - b * r.T_max;
  const int valid = r.bi.valid[b], len = r.block_len[b], P = r.seq_len[b], depth = r.bi.depth[m];
  p.slot = valid != 0 && i < len ? P + i : -1;
  const int pos = p.slot < 0 ? 0 : P + depth;
  if (r.D == 128) {
    const int head = n0 / 128;
    rope_load<128>(p.r128, head < r.Hq ? r.q_norm : r.k_norm, r.table, pos);
  } else {
#pragma unroll
    for (int h = 0; h < 2; ++h) rope_load<64>(p.r64[h], n0 / 64 + h < r.Hq ? r.q_norm : r.k_norm, r.table, pos);
  }
}

// The row (of `width` channels in all), four channels a lane, f as the linear layer's bf16 output: q and k heads normalised, rotated
// and put in their places, v heads copied.
template <int D>
__device__ __forceinline__ void rope_row_store(const RopeArgs& r, const float (&f)[4], int m, int n0, int width, const RopeRow& p) {
  const int lane = threadIdx.x & 31;
  if (p.slot < 0) return;
  const int b = m / r.T_max;
#pragma unroll
  for (int h = 0; h < 128 / D; ++h) {
    const int head = n0 / D + h;
    // lane l takes the channels l + 32 k of the head, which lane (l + 32 k) / 4 holds
    float x[D / 32];
#pragma unroll
    for (int k = 0; k < D / 32; ++k) {
      const int from = (h * D + 32 * k + lane) >> 2;
      x[k] = 0.f;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float t = __shfl_sync(0xffffffffu, f[e], from);
        if ((lane & 3) == e) x[k] = t;
      }
    }
    if (head >= r.Hq + 2 * r.Hkv) continue;
    if (head >= r.Hq + r.Hkv) {
      __nv_bfloat16* dst = r.v_cache + (((size_t)b * r.Hkv + (head - r.Hq - r.Hkv)) * r.s_max + p.slot) * D;
#pragma unroll
      for (int k = 0; k < D / 32; ++k) dst[lane + 32 * k] = __float2bfloat16_rn(x[k]);
      continue;
    }
    float lo[D / 64], hi[D / 64];
#pragma unroll
    for (int q = 0; q < D / 64; ++q) { lo[q] = x[q]; hi[q] = x[q + D / 64]; }
    __nv_bfloat16* dst = head < r.Hq ? r.qkv + (size_t)m * width + (size_t)head * D
                                     : r.k_cache + (((size_t)b * r.Hkv + (head - r.Hq)) * r.s_max + p.slot) * D;
    if constexpr (D == 128) rope_head<128>(lo, hi, p.r128, r.eps, dst);
    else rope_head<64>(lo, hi, p.r64[h], r.eps, dst);
  }
}
#endif

}  // namespace quasar
