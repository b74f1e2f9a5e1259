// QK-RMSNorm + RoPE + KV append (Section 3.3: the "non-linear layers" stay in high precision), the RoPE table and the
// cache commit.  All are HBM/L2-bound on a few KB..MB; fp32 math, bf16 storage.
#include <math.h>

#include "common.cuh"
#include "tc_common.cuh"

namespace quasar {

namespace {

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---- RoPE table: cos/sin(pos * theta^(-2i/D)) evaluated in fp64, stored as fp32 -------------
__global__ void rope_table_kernel(float2* table, int max_pos, int D, double theta) {
  const int half = D / 2;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= max_pos * half) return;
  const int pos = idx / half, i = idx % half;
  const double inv_freq = pow(theta, -2.0 * (double)i / (double)D);
  double s, c;
  sincos((double)pos * inv_freq, &s, &c);
  table[idx] = make_float2((float)c, (float)s);
}

// ---- QK-RMSNorm + RoPE + KV append: one warp per (row, head) --------------------------------
template <int D>
__global__ void __launch_bounds__(128)
rope_append_kernel(__nv_bfloat16* __restrict__ qkv, const __nv_bfloat16* __restrict__ q_norm,
                   const __nv_bfloat16* __restrict__ k_norm, const float2* __restrict__ rope_table,
                   const int32_t* __restrict__ seq_len, const int32_t* __restrict__ block_len, BlockInfo bi, int T_max,
                   int Hq, int Hkv, float eps, __nv_bfloat16* __restrict__ k_cache, __nv_bfloat16* __restrict__ v_cache,
                   int s_max, int n_items) {
  tc::pdl_trigger();
  tc::pdl_wait();
  constexpr int kPairs = D / 64;  // rotation pairs (i, i + D/2) per lane
  const int item = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (item >= n_items) return;
  const int lane = threadIdx.x & 31;
  const int heads = Hq + 2 * Hkv;
  const int m = item / heads, head = item % heads;
  const int b = m / T_max, i = m % T_max;
  if (!bi.valid[b] || i >= block_len[b]) return;
  const int P = seq_len[b];
  __nv_bfloat16* src = qkv + (size_t)m * heads * D + (size_t)head * D;

  if (head >= Hq + Hkv) {  // v head: copy into the cache
    const int hk = head - Hq - Hkv;
    __nv_bfloat16* dst = v_cache + (((size_t)b * Hkv + hk) * s_max + (P + i)) * D;
    if (lane < D / 8) reinterpret_cast<uint4*>(dst)[lane] = reinterpret_cast<const uint4*>(src)[lane];
    return;
  }
  const bool is_q = head < Hq;
  const __nv_bfloat16* gain = is_q ? q_norm : k_norm;
  float lo[kPairs], hi[kPairs];
  float ss = 0.f;
#pragma unroll
  for (int p = 0; p < kPairs; ++p) {
    const int d = lane + 32 * p;
    lo[p] = __bfloat162float(src[d]);
    hi[p] = __bfloat162float(src[d + D / 2]);
    ss += lo[p] * lo[p] + hi[p] * hi[p];
  }
  if (gain != nullptr) {
    ss = warp_sum(ss);
    const float r = 1.0f / sqrtf(ss / (float)D + eps);
#pragma unroll
    for (int p = 0; p < kPairs; ++p) {
      const int d = lane + 32 * p;
      lo[p] = lo[p] * r * __bfloat162float(gain[d]);
      hi[p] = hi[p] * r * __bfloat162float(gain[d + D / 2]);
    }
  }
  const int pos = P + bi.depth[m];
  __nv_bfloat16* dst = is_q ? src : k_cache + (((size_t)b * Hkv + (head - Hq)) * s_max + (P + i)) * D;
#pragma unroll
  for (int p = 0; p < kPairs; ++p) {
    const int d = lane + 32 * p;
    const float2 cs = rope_table[(size_t)pos * (D / 2) + d];
    dst[d] = __float2bfloat16_rn(lo[p] * cs.x - hi[p] * cs.y);
    dst[d + D / 2] = __float2bfloat16_rn(hi[p] * cs.x + lo[p] * cs.y);
  }
}

// ---- commit: (tree) move accepted rows into place, then bump seq_len --------------------------
// One thread per 16-byte piece of a (layer, sequence, kv head) row; depths are walked in
// increasing order inside the thread, which keeps every source slot intact until it is read
// (the accepted row at depth d has block index >= d).
__global__ void kv_gather_kernel(__nv_bfloat16* __restrict__ k_cache, __nv_bfloat16* __restrict__ v_cache,
                                 const int32_t* __restrict__ seq_len, const int32_t* __restrict__ accept_len,
                                 const int32_t* __restrict__ accept_path, int L, int B_cache, int B, int T_max,
                                 int Hkv, int D, int s_max) {
  const int chunks = D / 8;
  const size_t total = (size_t)L * B * Hkv * chunks;
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= total) return;
  const int c = (int)(idx % chunks);
  size_t r = idx / chunks;
  const int hk = (int)(r % Hkv); r /= Hkv;
  const int b = (int)(r % B);
  const int l = (int)(r / B);
  const int n = accept_len[b];
  const int P = seq_len[b];
  if (n < 0 || n >= T_max || P < 0) return;
  const size_t base = (((size_t)l * B_cache + b) * Hkv + hk) * (size_t)s_max;
  for (int d = 1; d <= n; ++d) {
    const int j = accept_path[b * T_max + d];
    if (j == d || j < d || j >= T_max || P + j >= s_max) continue;
    uint4* kd = reinterpret_cast<uint4*>(k_cache + (base + P + d) * D) + c;
    uint4* vd = reinterpret_cast<uint4*>(v_cache + (base + P + d) * D) + c;
    *kd = *(reinterpret_cast<const uint4*>(k_cache + (base + P + j) * D) + c);
    *vd = *(reinterpret_cast<const uint4*>(v_cache + (base + P + j) * D) + c);
  }
}

__global__ void seq_bump_kernel(int32_t* seq_len, const int32_t* __restrict__ accept_len, int B, int T_max, int s_max) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  const int n = accept_len[b];
  if (n < 0 || n >= T_max) return;
  const int v = seq_len[b] + 1 + n;
  if (v <= s_max) seq_len[b] = v;
}

}  // namespace

int launch_rope_table(float2* table, int max_pos, int D, float theta, cudaStream_t stream) {
  const int total = max_pos * (D / 2);
  rope_table_kernel<<<(total + 255) / 256, 256, 0, stream>>>(table, max_pos, D, (double)theta);
  QUASAR_LAUNCH_CHECK();
  return QUASAR_OK;
}

int launch_rope_append(__nv_bfloat16* qkv, const __nv_bfloat16* q_norm, const __nv_bfloat16* k_norm,
                       const float2* rope_table, const int32_t* seq_len, const int32_t* block_len, BlockInfo bi, int B,
                       int T_max, int Hq, int Hkv, int D, float eps, __nv_bfloat16* k_cache_layer,
                       __nv_bfloat16* v_cache_layer, int s_max, cudaStream_t stream) {
  const int n_items = B * T_max * (Hq + 2 * Hkv);
  const int grid = (n_items + 3) / 4;
  if (D == 128) {
    return launch_dependent(rope_append_kernel<128>, dim3(grid), dim3(128), 0, true, stream, qkv, q_norm, k_norm, rope_table, seq_len, block_len, bi, T_max,
                                                       Hq, Hkv, eps, k_cache_layer, v_cache_layer, s_max, n_items);
  } else if (D == 64) {
    return launch_dependent(rope_append_kernel<64>, dim3(grid), dim3(128), 0, true, stream, qkv, q_norm, k_norm, rope_table, seq_len, block_len, bi, T_max,
                                                      Hq, Hkv, eps, k_cache_layer, v_cache_layer, s_max, n_items);
  } else {
    set_error("head_dim %d not supported (64 or 128)", D);
    return QUASAR_ERR_SHAPE;
  }
}

int launch_kv_commit(__nv_bfloat16* k_cache, __nv_bfloat16* v_cache, int32_t* seq_len, const int32_t* accept_len,
                     const int32_t* accept_path, int L, int B_cache, int B, int T_max, int Hkv, int D, int s_max,
                     cudaStream_t stream) {
  if (accept_path != nullptr) {
    const size_t total = (size_t)L * B * Hkv * (D / 8);
    kv_gather_kernel<<<(unsigned)((total + 255) / 256), 256, 0, stream>>>(k_cache, v_cache, seq_len, accept_len,
                                                                          accept_path, L, B_cache, B, T_max, Hkv, D,
                                                                          s_max);
    QUASAR_LAUNCH_CHECK();
  }
  seq_bump_kernel<<<(B + 63) / 64, 64, 0, stream>>>(seq_len, accept_len, B, T_max, s_max);
  QUASAR_LAUNCH_CHECK();
  return QUASAR_OK;
}

}  // namespace quasar
