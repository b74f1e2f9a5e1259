// QK-RMSNorm + RoPE + KV append (Section 3.3: the "non-linear layers" stay in high precision), the RoPE table and the
// cache commit.  All are HBM/L2-bound on a few KB..MB; fp32 math, bf16 storage.
#include <math.h>

#include "common.cuh"
#include "rope.cuh"
#include "tc_common.cuh"

namespace quasar {

namespace {

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

// ---- QK-RMSNorm + RoPE + KV append (where the qkv projection does not finish its rows itself: traces, wide int8 blocks that run
//      as one range, W8A8 and bf16 blocks of more than 128 rows): a warp per row and six neighbouring heads,
//      whose vectors are asked for at once, beside what says where the row goes.  One head a warp was a chain of round trips for
//      a kilobyte: 9.1 us at 512 rows of 48 heads. ----
constexpr int kRopeHeads = 6;

template <int D>
__global__ void __launch_bounds__(128) rope_append_kernel(const RopeArgs a, int n_items, int groups) {
  tc::pdl_wait();
  tc::pdl_trigger();   // (only now: the attention reads before its own wait what the kernels in front of this one's predecessor left)
  const int item = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (item >= n_items) return;
  const int lane = threadIdx.x & 31;
  const int heads = a.Hq + 2 * a.Hkv;
  const int m = item / groups, head0 = (item - m * groups) * kRopeHeads;
  const int b = m / a.T_max, i = m - b * a.T_max;
  __nv_bfloat16* row = a.qkv + (size_t)m * heads * D;
  float lo[kRopeHeads][D / 64], hi[kRopeHeads][D / 64];
#pragma unroll
  for (int h = 0; h < kRopeHeads; ++h) {
    const __nv_bfloat16* src = row + (size_t)min(head0 + h, heads - 1) * D;
#pragma unroll
    for (int p = 0; p < D / 64; ++p) {
      lo[h][p] = __bfloat162float(src[lane + 32 * p]);
      hi[h][p] = __bfloat162float(src[lane + 32 * p + D / 2]);
    }
  }
  const int valid = a.bi.valid[b], len = a.block_len[b], P = a.seq_len[b], depth = a.bi.depth[m];
  if (!valid || i >= len) return;
  RopeLane<D> rq, rk;
  rope_load<D>(rq, a.q_norm, a.table, P + depth);
  rope_load<D>(rk, a.k_norm, a.table, P + depth);
#pragma unroll
  for (int h = 0; h < kRopeHeads; ++h) {
    const int head = head0 + h;
    if (head >= heads) break;
    const bool is_q = head < a.Hq, is_v = head >= a.Hq + a.Hkv;
    if (is_v) {
      __nv_bfloat16* dst = a.v_cache + (((size_t)b * a.Hkv + (head - a.Hq - a.Hkv)) * a.s_max + (P + i)) * D;
#pragma unroll
      for (int p = 0; p < D / 64; ++p) {
        dst[lane + 32 * p] = __float2bfloat16_rn(lo[h][p]);
        dst[lane + 32 * p + D / 2] = __float2bfloat16_rn(hi[h][p]);
      }
      continue;
    }
    __nv_bfloat16* dst = is_q ? row + (size_t)head * D : a.k_cache + (((size_t)b * a.Hkv + (head - a.Hq)) * a.s_max + (P + i)) * D;
    if (is_q) rope_head<D>(lo[h], hi[h], rq, a.eps, dst);
    else rope_head<D>(lo[h], hi[h], rk, a.eps, dst);
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

int launch_rope_append(const RopeArgs& a, int B, cudaStream_t stream) {
  const int groups = (a.Hq + 2 * a.Hkv + kRopeHeads - 1) / kRopeHeads, n_items = B * a.T_max * groups;
  const dim3 grid((unsigned)((n_items + 3) / 4));
  if (a.D == 128) return launch_dependent(rope_append_kernel<128>, grid, dim3(128), 0, true, stream, 1, a, n_items, groups);
  if (a.D == 64) return launch_dependent(rope_append_kernel<64>, grid, dim3(128), 0, true, stream, 1, a, n_items, groups);
  set_error("head_dim %d not supported (64 or 128)", a.D);
  return QUASAR_ERR_SHAPE;
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
