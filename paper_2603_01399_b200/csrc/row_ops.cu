// The steps of the pass that work on whole activation rows and leave the operand of the linear layer that follows
// (Section 3.3: the "non-linear layers" stay in high precision, the online quantisation of Eq. 9 rides on them):
// embedding gather + first RMSNorm, RMSNorm, SwiGLU, and the attention output on its way into the o projection.
//
// The operand has one of three forms: the row as four digit rows (int8 weights, bf16 activations; see tc_linear.cuh),
// the row smoothed and quantised per token (W8A8, Eq. 9), or the bf16 row itself (bf16 weights).
//
// One CTA of 512 threads per row; a row of up to 24,576 elements stays in registers between its passes (statistic,
// maximum, codes), eight consecutive elements a thread and turn, longer rows are read again.  Latency-bound (a row is
// 8 to 48 KB out of L2): every input of a turn is one 128-bit load, the gains and smoothing factors - weights - are
// asked for before the kernel in front has finished, and all of these are dependent launches.
#include <math.h>

#include "common.cuh"
#include "tc_attention.cuh"
#include "tc_common.cuh"
#include "tc_linear.cuh"

namespace quasar {

namespace {

using tc::pdl_trigger;
using tc::pdl_wait;

constexpr int kRowThreads = 512;

__device__ __forceinline__ void unpack8(const uint4& v, float (&f)[8]) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    f[2 * e] = __uint_as_float(w[e] << 16);
    f[2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u);
  }
}
// rounds f to bf16 in place and returns the packed values
__device__ __forceinline__ uint4 round8(float (&f)[8]) {
  uint32_t w[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(f[2 * e], f[2 * e + 1]);
    w[e] = *reinterpret_cast<const uint32_t*>(&p);
    f[2 * e] = __uint_as_float(w[e] << 16);
    f[2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

__device__ __forceinline__ float block_sum(float v, float* s_buf) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) s_buf[threadIdx.x >> 5] = v;
  __syncthreads();
  v = s_buf[0];
#pragma unroll
  for (int i = 1; i < kRowThreads / 32; ++i) v += s_buf[i];   // warps in order
  return v;
}
// maximum of magnitudes (bit patterns, see magnitude())
__device__ __forceinline__ uint32_t block_max(uint32_t v, float* s_buf) {
  v = __reduce_max_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) s_buf[threadIdx.x >> 5] = __uint_as_float(v);
  __syncthreads();
  v = __float_as_uint(s_buf[0]);
#pragma unroll
  for (int i = 1; i < kRowThreads / 32; ++i) v = max(v, __float_as_uint(s_buf[i]));
  return v;
}

// sum and maximum of magnitudes of a block in one meeting; s_buf [64]
__device__ __forceinline__ void block_sum_max(float& sum, uint32_t& top, float* s_buf) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  top = __reduce_max_sync(0xffffffffu, top);
  if ((threadIdx.x & 31) == 0) {
    s_buf[threadIdx.x >> 5] = sum;
    s_buf[32 + (threadIdx.x >> 5)] = __uint_as_float(top);
  }
  __syncthreads();
  sum = s_buf[0];
  top = __float_as_uint(s_buf[32]);
#pragma unroll
  for (int i = 1; i < kRowThreads / 32; ++i) {   // warps in order
    sum += s_buf[i];
    top = max(top, __float_as_uint(s_buf[32 + i]));
  }
}

// The larger of a maximum so far and |f|, as bits.  Digits keep a NaN (the row becomes NaN); the step size of Eq. 9 is defined
// over the numbers and passes over it.
template <int OP>
__device__ __forceinline__ uint32_t take_max(uint32_t top, float f) {
  return OP == kOperandDigits ? max(top, magnitude(f)) : __float_as_uint(fmaxf(__uint_as_float(top), fabsf(f)));
}

// The smoothing factors of eight channels (one for all without smoothing)
__device__ __forceinline__ void load_smooth8(const float* smooth, int i, float (&s)[8]) {
  if (smooth == nullptr) {
#pragma unroll
    for (int e = 0; e < 8; ++e) s[e] = 1.f;
    return;
  }
  const float4 a = __ldg(reinterpret_cast<const float4*>(smooth) + 2 * i), b = __ldg(reinterpret_cast<const float4*>(smooth) + 2 * i + 1);
  s[0] = a.x; s[1] = a.y; s[2] = a.z; s[3] = a.w; s[4] = b.x; s[5] = b.y; s[6] = b.z; s[7] = b.w;
}

// Eq. 9 for eight elements: codes of the smoothed values
__device__ __forceinline__ uint2 smoothed_codes8(const float (&f)[8], const float (&s)[8], float scale) {
  uint32_t p[2] = {0u, 0u};
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const int q = max(-127, min(127, __float2int_rn(__fdiv_rn(__fmul_rn(f[e], s[e]), scale))));
    p[e >> 2] |= (uint32_t)(q & 0xff) << (8 * (e & 3));
  }
  return make_uint2(p[0], p[1]);
}

// The row's values (eight of vector i by value(i, j, f); j is the turn) as the operand.
template <int OP, int V, typename F>
__device__ __forceinline__ void write_operand(F&& value, int nvec, int m, const RowOperand& out, float* s_buf) {
  if (OP == kOperandBf16) {   // (the values have been stored as they were made)
    float f[8];
    if (V > 0) {
#pragma unroll
      for (int j = 0; j < (V > 0 ? V : 1); ++j)
        if ((int)threadIdx.x + j * kRowThreads < nvec) value((int)threadIdx.x + j * kRowThreads, j, f);
    } else {
      for (int i = threadIdx.x; i < nvec; i += kRowThreads) value(i, 0, f);
    }
    return;
  }
  const int64_t width = (int64_t)nvec * 8;
  float f[V > 0 ? V : 1][8];
  uint32_t top = 0;
  if (V > 0) {
#pragma unroll
    for (int j = 0; j < (V > 0 ? V : 1); ++j) {
      const int i = (int)threadIdx.x + j * kRowThreads;
      if (i < nvec) {
        value(i, j, f[j]);
#pragma unroll
        for (int e = 0; e < 8; ++e) top = take_max<OP>(top, f[j][e]);
      }
    }
  } else {
    for (int i = threadIdx.x; i < nvec; i += kRowThreads) {
      value(i, 0, f[0]);
#pragma unroll
      for (int e = 0; e < 8; ++e) top = take_max<OP>(top, f[0][e]);
    }
  }
  top = block_max(top, s_buf);
  const float amax = __uint_as_float(top);
  float up = 1.f, scale = 1.f;
  if (OP == kOperandDigits) digit_scale(top, up, scale);
  else scale = amax == 0.f ? 1.0f : __fdiv_rn(amax, 127.0f);
  if (threadIdx.x == 0) out.scale[m] = scale;
  auto put = [&](int i, const float (&v)[8]) {
    if (OP == kOperandDigits) {
      write_digits8(v, up, out.q + kDigitPlanes * (int64_t)m * width, width, (int64_t)i * 8);
    } else {
      uint32_t p[2] = {0u, 0u};
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int q = max(-127, min(127, __float2int_rn(__fdiv_rn(v[e], scale))));
        p[e >> 2] |= (uint32_t)(q & 0xff) << (8 * (e & 3));
      }
      *reinterpret_cast<uint2*>(out.q + (int64_t)m * width + (int64_t)i * 8) = make_uint2(p[0], p[1]);
    }
  };
  if (V > 0) {
#pragma unroll
    for (int j = 0; j < (V > 0 ? V : 1); ++j)
      if ((int)threadIdx.x + j * kRowThreads < nvec) put((int)threadIdx.x + j * kRowThreads, f[j]);
  } else {
    for (int i = threadIdx.x; i < nvec; i += kRowThreads) {
      value(i, 0, f[0]);
      put(i, f[0]);
    }
  }
}

// Sum of squares of a row in a FIXED order, whatever the spread of the row over the threads: pair p of the row (elements 2 p,
// 2 p + 1) belongs to adder p % adders, which takes its pairs in ascending order; 32 neighbouring adders join as a warp's
// butterfly does, and these sums are added in order (rows too long for registers: as the threads hold them).  A last-bit difference here turns into quantisation steps in the
// W8A8 form, so the order does not change with the kernel's shape.
__device__ __forceinline__ float sum_of_squares(const float* s_pair, int pairs, int adders, float* s_buf) {
  __syncthreads();   // the pairs' sums are there
  for (int t = threadIdx.x; t < adders; t += kRowThreads) {
    float ss = 0.f;
    for (int p = t; p < pairs; p += adders) ss += s_pair[p];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if ((t & 31) == 0) s_buf[t >> 5] = ss;
  }
  __syncthreads();
  float tot = 0.f;
  for (int i = 0; i < adders / 32; ++i) tot += s_buf[i];
  return tot;
}

// RMSNorm of the row whose vectors raw(i, j, f) gives, in operand form: y = bf16(x * rsqrt(mean(x^2) + eps) * g)
template <int OP, int V, typename F>
__device__ __forceinline__ void norm_row(F&& raw, const uint4 (&gain)[V > 0 ? V : 1], const __nv_bfloat16* g, int nvec, float eps, int adders,
                                         int m, const RowOperand& out, float* s_buf) {
  extern __shared__ float s_pair[];
  float x[V > 0 ? V : 1][8];
  float ss = 0.f;
  uint32_t top = 0;   // digits: the largest |x g|
  if (V > 0) {
#pragma unroll
    for (int j = 0; j < (V > 0 ? V : 1); ++j) {
      const int i = (int)threadIdx.x + j * kRowThreads;
      if (i < nvec) {
        raw(i, x[j]);
        float4 v;
        v.x = x[j][0] * x[j][0] + x[j][1] * x[j][1];
        v.y = x[j][2] * x[j][2] + x[j][3] * x[j][3];
        v.z = x[j][4] * x[j][4] + x[j][5] * x[j][5];
        v.w = x[j][6] * x[j][6] + x[j][7] * x[j][7];
        if (OP == kOperandCodes) reinterpret_cast<float4*>(s_pair)[i] = v;
        else ss += (v.x + v.y) + (v.z + v.w);
        if (OP == kOperandDigits) {
          float gg[8];
          unpack8(gain[V > 0 ? j : 0], gg);
#pragma unroll
          for (int e = 0; e < 8; ++e) top = take_max<OP>(top, x[j][e] * gg[e]);
        }
      }
    }
    // (The other forms need no particular order, only always the same one: without the pass through shared memory, and with the
    // maximum of a digit row in the same meeting, the chain pass took 2196 -> 2158 us, the batch of eight 3875 -> 3709.)
    if (OP == kOperandDigits) block_sum_max(ss, top, s_buf);
    else ss = OP == kOperandCodes ? sum_of_squares(s_pair, nvec * 4, adders, s_buf) : block_sum(ss, s_buf);
  } else {
    for (int i = threadIdx.x; i < nvec; i += kRowThreads) {
      raw(i, x[0]);
#pragma unroll
      for (int e = 0; e < 8; ++e) ss += x[0][e] * x[0][e];
    }
    ss = block_sum(ss, s_buf);
  }
  const float r = 1.0f / sqrtf(ss / (float)(nvec * 8) + eps);
  if constexpr (OP == kOperandDigits && V > 0) {
    // The row's maximum without another meeting of the block: top * r is it but for roundings, for which digit_scale leaves room.
    float up, scale;
    digit_scale(magnitude(__uint_as_float(top) * r), up, scale);
    if (threadIdx.x == 0) out.scale[m] = scale;
    const int64_t width = (int64_t)nvec * 8;
#pragma unroll
    for (int j = 0; j < V; ++j) {
      const int i = (int)threadIdx.x + j * kRowThreads;
      if (i >= nvec) break;
      float gg[8], f[8];
      unpack8(gain[j], gg);
#pragma unroll
      for (int e = 0; e < 8; ++e) f[e] = x[j][e] * r * gg[e];
      const uint4 y = round8(f);
      if (out.y != nullptr) reinterpret_cast<uint4*>(out.y + (size_t)m * nvec * 8)[i] = y;
      write_digits8(f, up, out.q + kDigitPlanes * (int64_t)m * width, width, (int64_t)i * 8);
    }
    return;
  }
  write_operand<OP, V>(
      [&](int i, int j, float (&f)[8]) {
        float gg[8];
        if (V > 0) {
          unpack8(gain[V > 0 ? j : 0], gg);
#pragma unroll
          for (int e = 0; e < 8; ++e) f[e] = x[V > 0 ? j : 0][e] * r * gg[e];
        } else {
          unpack8(__ldg(reinterpret_cast<const uint4*>(g) + i), gg);
          raw(i, f);
#pragma unroll
          for (int e = 0; e < 8; ++e) f[e] = f[e] * r * gg[e];
        }
        const uint4 y = round8(f);
        if (out.y != nullptr) reinterpret_cast<uint4*>(out.y + (size_t)m * nvec * 8)[i] = y;
        if (OP == kOperandCodes) {
          float s[8];
          load_smooth8(out.smooth, i, s);
#pragma unroll
          for (int e = 0; e < 8; ++e) f[e] = __fmul_rn(f[e], s[e]);
        }
      },
      nvec, m, out, s_buf + 32);
}

template <int V>
__device__ __forceinline__ void load_gain(uint4 (&gain)[V > 0 ? V : 1], const __nv_bfloat16* g, int nvec) {
  if (V > 0) {
#pragma unroll
    for (int j = 0; j < (V > 0 ? V : 1); ++j) {
      const int i = (int)threadIdx.x + j * kRowThreads;
      gain[j] = i < nvec ? __ldg(reinterpret_cast<const uint4*>(g) + i) : make_uint4(0, 0, 0, 0);
    }
  }
}

template <int OP, int V>
__global__ void __launch_bounds__(kRowThreads)
norm_kernel(const __nv_bfloat16* x, const __nv_bfloat16* __restrict__ g, int nvec, float eps, int adders, RowOperand out) {
  __shared__ float s_buf[64];
  pdl_trigger();
  uint4 gain[V > 0 ? V : 1];
  load_gain<V>(gain, g, nvec);
  pdl_wait();
  const int m = blockIdx.x;
  const uint4* row = reinterpret_cast<const uint4*>(x + (size_t)m * nvec * 8);
  norm_row<OP, V>([&](int i, float (&f)[8]) { unpack8(row[i], f); }, gain, g, nvec, eps, adders, m, out, s_buf);
}

template <int OP, int V>
__global__ void __launch_bounds__(kRowThreads)
swiglu_kernel(const __nv_bfloat16* gu, int nvec, RowOperand out) {
  __shared__ float s_buf[32];
  pdl_trigger();
  pdl_wait();
  const int m = blockIdx.x;
  const uint4* gr = reinterpret_cast<const uint4*>(gu + (size_t)m * nvec * 16);
  const uint4* ur = gr + nvec;
  write_operand<OP, V>(
      [&](int i, int j, float (&f)[8]) {
        float up[8];
        unpack8(gr[i], f);
        unpack8(ur[i], up);
#pragma unroll
        for (int e = 0; e < 8; ++e) f[e] = f[e] / (1.0f + expf(-f[e])) * up[e];
        const uint4 y = round8(f);
        if (out.y != nullptr) reinterpret_cast<uint4*>(out.y + (size_t)m * nvec * 8)[i] = y;
        if (OP == kOperandCodes) {
          float s[8];
          load_smooth8(out.smooth, i, s);
#pragma unroll
          for (int e = 0; e < 8; ++e) f[e] = __fmul_rn(f[e], s[e]);
        }
      },
      nvec, m, out, s_buf);
}

// The operand of rows whose largest magnitude is known (its bits in row_max, gathered by the kernel that wrote the rows): every
// element for itself.
constexpr int kElemThreads = 128;
template <int OP>
__global__ void __launch_bounds__(kElemThreads)
operand_kernel(const __nv_bfloat16* x, const unsigned* row_max, int nvec, RowOperand out) {
  pdl_trigger();
  const int m = blockIdx.y, i = blockIdx.x * kElemThreads + threadIdx.x;
  float s[8];
  if (OP == kOperandCodes && i < nvec) load_smooth8(out.smooth, i, s);
  pdl_wait();
  const uint32_t top = row_max[m];
  const float amax = __uint_as_float(top);
  float up = 1.f, scale = 1.f;
  if (OP == kOperandDigits) digit_scale(top, up, scale);
  else scale = amax == 0.f ? 1.0f : __fdiv_rn(amax, 127.0f);
  if (blockIdx.x == 0 && threadIdx.x == 0) out.scale[m] = scale;
  if (i >= nvec) return;
  float f[8];
  unpack8(reinterpret_cast<const uint4*>(x + (size_t)m * nvec * 8)[i], f);
  const int64_t width = (int64_t)nvec * 8;
  if (OP == kOperandDigits) {
    write_digits8(f, up, out.q + kDigitPlanes * (int64_t)m * width, width, (int64_t)i * 8);
  } else {
    *reinterpret_cast<uint2*>(out.q + (int64_t)m * width + (int64_t)i * 8) = smoothed_codes8(f, s, scale);
  }
}

// Puts an attention's partial results together and leaves the o projection's operand: a cluster of four CTAs per block row,
// each a quarter of the query heads, a warp per head.  A head's parts lie `stride` entries apart and are added in their order
// (tcgen05 form: the two groups of every CTA whose run of the list touched the head's segment, see tc_attention.cuh; the other
// form: the chunks of the keys); the copies of 8 or 16 parts are in flight together.  Latency-bound; 6 rows of 32 heads and 18 or 34
// parts took 10-17 us with one CTA per row or eight parts at a time and another kernel for the operand.
constexpr int kMergeCtas = 4, kMergeWarps = 16;

template <int OP, int D, bool LIST>
__global__ void __launch_bounds__(kMergeWarps * 32)
attention_merge_kernel(AttnList l, AttnParts parts, AttnChunks ch, int batch, RowOperand out) {
  __shared__ uint32_t s_buf[kMergeWarps];
  __shared__ float s_amax[kMergeCtas];   // of every CTA of the cluster
  extern __shared__ __align__(16) unsigned char s_row[];   // this CTA's heads, bf16; then each warp's parts of a batch
  pdl_trigger();
  if (OP != kOperandBf16) tc::cluster_arrive();   // (every CTA of the cluster has started before one writes into another's memory)
  if (!LIST) pdl_wait();   // (the list's description is older than the kernel in front, see tc_attention_kernel)
  const int rank = blockIdx.x % kMergeCtas, m = blockIdx.x / kMergeCtas, b = m / l.T_max, i = m % l.T_max;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  const int Hq = l.Hkv * l.G, h0 = rank * Hq / kMergeCtas, h1 = (rank + 1) * Hq / kMergeCtas;
  constexpr int kPer = D / 32;
  __shared__ float4 s_part[kMergeWarps][64];   // per warp: the non-empty parts' (index, weight, sum)
  bool live;
  int n0 = 0, stride, tiles = 0, row_tiles = 0, unit0 = 0, seg0 = 0, row0;
  unsigned total = 1, ctas = 1;
  if (LIST) {
    const AttnSeq q = l.seq[b];
    total = (unsigned)l.seq[l.B].unit0;
    tiles = q.tiles; row_tiles = q.row_tiles; unit0 = q.unit0; seg0 = q.seg0;
    live = tiles > 0 && i < l.block_len[b];
    ctas = attn_ctas(total);
    const int t = i / l.npt;
    unit0 += t * tiles;    // of head 0's row tile that holds this row
    seg0 += t;
    row0 = (i - t * l.npt) * l.G;
    stride = 128;
  } else {
    const int T = l.block_len[b];
    live = l.valid[b] != 0 && i < T;
    n0 = (l.seq_len[b] + T + ch.chunk - 1) / ch.chunk;
    stride = ch.Rpad;
    row0 = i * l.G;
  }
  if (LIST) pdl_wait();
  float* s_o = reinterpret_cast<float*>(s_row + (size_t)((Hq + kMergeCtas - 1) / kMergeCtas) * D * 2) + (size_t)warp * batch * D;
  uint32_t top = 0;   // of the operand's values, head by head as they are made
  for (int hq = h0 + warp; hq < h1; hq += warps) {
    uint32_t pk[kPer / 2];
#pragma unroll
    for (int e = 0; e < kPer / 2; ++e) pk[e] = 0u;
    if (live) {
      const int hk = hq / l.G, row = row0 + hq - hk * l.G;
      size_t at0;
      int n = n0;
      if (LIST) {   // CTA c takes the units [c * total / ctas, (c + 1) * total / ctas): the ones that share u0 .. u1 - 1
        const int u0 = unit0 + hk * row_tiles * tiles, u1 = u0 + tiles, s = seg0 + hk * row_tiles;
        int c0, c1;
        if (total < (1u << 24)) {
          c0 = (int)(((unsigned)(u0 + 1) * ctas - 1u) / total);
          c1 = (int)(((unsigned)u1 * ctas - 1u) / total);
        } else {
          c0 = (int)(((unsigned long long)(u0 + 1) * ctas - 1) / total);
          c1 = (int)(((unsigned long long)u1 * ctas - 1) / total);
        }
        n = 2 * (c1 - c0 + 1);
        at0 = (size_t)(c0 + s) * 256 + row;
      } else {
        at0 = ((size_t)b * l.Hkv + hk) * ch.nchunk * ch.Rpad + row;
      }
      auto part_ml = [&](int p) { return p < n ? __ldcg(&parts.ml[at0 + (size_t)p * stride]) : make_float2(-INFINITY, 0.f); };
      float2 ml[2] = {part_ml(lane), part_ml(lane + 32)};   // (64 parts in one round trip: more are rare)
      float mx = fmaxf(ml[0].x, ml[1].x);
      for (int p = lane + 64; p < n; p += 32) mx = fmaxf(mx, __ldcg(&parts.ml[at0 + (size_t)p * stride].x));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      float acc[kPer], den = 0.f;
#pragma unroll
      for (int e = 0; e < kPer; ++e) acc[e] = 0.f;
      for (int p0 = 0; p0 < n; p0 += 64) {
        if (p0 > 0) { ml[0] = part_ml(p0 + lane); ml[1] = part_ml(p0 + 32 + lane); }
        // the non-empty parts in a row (one without a visible key may never have been written)
        int cnt = 0;
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float w = ml[h].x == -INFINITY ? 0.f : exp2f(ml[h].x - mx);
          const unsigned some = __ballot_sync(0xffffffffu, w != 0.f);
          if (w != 0.f) s_part[warp][cnt + __popc(some & ((1u << lane) - 1u))] = make_float4(__int_as_float(p0 + 32 * h + lane), w, ml[h].y, 0.f);
          cnt += __popc(some);
        }
        __syncwarp();
        for (int j0 = 0; j0 < cnt; j0 += batch) {
          // the batch's copies in flight together (as loads into registers the compiler spreads them over their uses)
          const int nb = min(batch, cnt - j0);
#pragma unroll 4
          for (int q = 0; q < nb; ++q) {
            const float* src = parts.o + (at0 + (size_t)__float_as_int(s_part[warp][j0 + q].x) * stride) * D + lane * kPer;
            asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(tc::smem_u32(s_o + (q * 32 + lane) * kPer)), "l"(src),
                         "n"(kPer * 4)
                         : "memory");
          }
          asm volatile("cp.async.wait_all;\n" ::: "memory");   // (each lane reads only what it copied)
#pragma unroll 4
          for (int q = 0; q < nb; ++q) {
            const float4 part = s_part[warp][j0 + q];
            den += part.y * part.z;
#pragma unroll
            for (int e = 0; e < kPer; ++e) acc[e] += part.y * s_o[(q * 32 + lane) * kPer + e];
          }
        }
      }
      const float inv = 1.0f / den;
#pragma unroll
      for (int e = 0; e < kPer / 2; ++e) {
        const __nv_bfloat162 t = __floats2bfloat162_rn(acc[2 * e] * inv, acc[2 * e + 1] * inv);
        pk[e] = *reinterpret_cast<const uint32_t*>(&t);
      }
    }
    uint32_t* dst = reinterpret_cast<uint32_t*>(s_row) + (hq - h0) * (D / 2) + lane * (kPer / 2);
#pragma unroll
    for (int e = 0; e < kPer / 2; ++e) dst[e] = pk[e];
    if (OP != kOperandBf16) {
#pragma unroll
      for (int e = 0; e < kPer / 2; ++e) {
        float lo = __uint_as_float(pk[e] << 16), hi = __uint_as_float(pk[e] & 0xffff0000u);
        if (OP == kOperandCodes && out.smooth != nullptr) {
          const float2 f = __ldg(reinterpret_cast<const float2*>(out.smooth + hq * D + lane * kPer) + e);
          lo = __fmul_rn(lo, f.x);
          hi = __fmul_rn(hi, f.y);
        }
        top = take_max<OP>(take_max<OP>(top, lo), hi);
      }
    }
  }
  if (OP != kOperandBf16) {
    top = __reduce_max_sync(0xffffffffu, top);
    if (lane == 0) s_buf[warp] = top;
  }
  __syncthreads();
  const int nvec = (h1 - h0) * (D / 8), first = h0 * (D / 8);   // this CTA's 16-byte pieces of the row
  const int64_t width = (int64_t)Hq * D;
  float f[8], s[8];
  if (out.y != nullptr) {
    for (int v = threadIdx.x; v < nvec; v += blockDim.x)
      reinterpret_cast<uint4*>(out.y + (size_t)m * width)[first + v] = reinterpret_cast<const uint4*>(s_row)[v];
  }
  if (OP == kOperandBf16) return;
  tc::cluster_wait();
  if (warp == 0) {
    top = __reduce_max_sync(0xffffffffu, lane < warps ? s_buf[lane] : 0u);
    if (lane < kMergeCtas) tc::st_cluster_f32(tc::cluster_map(tc::smem_u32(s_amax + rank), (uint32_t)lane), __uint_as_float(top));
  }
  __syncwarp();
  tc::cluster_arrive();
  tc::cluster_wait();
  top = 0;
#pragma unroll
  for (int c = 0; c < kMergeCtas; ++c) top = max(top, __float_as_uint(s_amax[c]));
  const float amax = __uint_as_float(top);
  float up = 1.f, scale = 1.f;
  if (OP == kOperandDigits) digit_scale(top, up, scale);
  else scale = amax == 0.f ? 1.0f : __fdiv_rn(amax, 127.0f);
  if (rank == 0 && threadIdx.x == 0) out.scale[m] = scale;
  for (int v = threadIdx.x; v < nvec; v += blockDim.x) {
    unpack8(reinterpret_cast<const uint4*>(s_row)[v], f);
    if (OP == kOperandDigits) {
      write_digits8(f, up, out.q + kDigitPlanes * (int64_t)m * width, width, (int64_t)(first + v) * 8);
    } else {
      load_smooth8(out.smooth, first + v, s);
      *reinterpret_cast<uint2*>(out.q + (int64_t)m * width + (int64_t)(first + v) * 8) = smoothed_codes8(f, s, scale);
    }
  }
}

// One warp checks a sequence's tokens / parents / capacity and derives ancestor bit masks and depths.  A chain's are known
// in closed form; a tree's are walked in shared memory by one lane.
__device__ void prepare_sequence(const BlockArgs& a, int b, int* s_parent, unsigned long long* s_anc, int* s_depth) {
  const int lane = threadIdx.x & 31;
  const int T = a.block_len[b], P = a.seq_len[b];
  int err = 0;
  if (T < 1 || T > a.T_max || P < 0) err = QUASAR_ERR_INVALID_ARG;
  else if (P + T > a.s_max) err = QUASAR_ERR_CAPACITY;
  const int n = err ? 0 : T;
  int row_err[2] = {0, 0};
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int i = lane + 32 * h;
    if (i < n) {
      const int tok = a.tokens[b * a.T_max + i];
      const int par = a.parents ? a.parents[b * a.T_max + i] : i - 1;
      if (tok < 0 || tok >= a.vocab) row_err[h] = QUASAR_ERR_TOKEN;
      if ((i == 0 && par != -1) || (i > 0 && (par < 0 || par >= i))) row_err[h] = QUASAR_ERR_TREE;
      s_parent[i] = par;
    }
    const unsigned bad = __ballot_sync(0xffffffffu, row_err[h] != 0);
    if (bad && !err) err = __shfl_sync(0xffffffffu, row_err[h], __ffs(bad) - 1);   // the first faulty row's error
  }
  __syncwarp();
  if (!err && a.parents && lane == 0) {
    for (int i = 0; i < n; ++i) {
      const int p = s_parent[i];
      s_anc[i] = (1ull << i) | (i > 0 ? s_anc[p] : 0ull);
      s_depth[i] = i > 0 ? s_depth[p] + 1 : 0;
    }
  }
  __syncwarp();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int i = lane + 32 * h;
    if (i >= a.T_max) continue;
    const bool live = !err && i < n;
    a.bi.anc[b * a.T_max + i] = !live ? 0ull : a.parents ? s_anc[i] : (i == 63 ? ~0ull : (1ull << (i + 1)) - 1ull);
    a.bi.depth[b * a.T_max + i] = !live ? 0 : a.parents ? s_depth[i] : i;
    if (a.keys != nullptr) a.keys[b * a.T_max + i] = 0ull;   // the rows' arg-max starts
  }
  if (lane == 0) {
    a.bi.valid[b] = err ? 0 : 1;
    if (err && a.status) atomicMin(a.status, err);
  }
}

// Every sequence's place in the attention's list (AttnSeq): a warp, 32 sequences at a time, a running total behind the last.
__device__ void lay_out_list(const BlockArgs& a) {
  const int lane = threadIdx.x & 31;
  int units = 0, segs = 0;
  for (int b0 = 0; b0 < a.B; b0 += 32) {
    const int b = b0 + lane;
    AttnSeq q = {0, 0, 0, 0};
    if (b < a.B && a.bi.valid[b] != 0) {
      const int T = a.block_len[b];
      q.tiles = (a.seq_len[b] + T + 127) / 128;
      q.row_tiles = (T + a.npt - 1) / a.npt;
    }
    int u = q.tiles * q.row_tiles * a.Hkv, s = q.row_tiles * a.Hkv;
    const int own_u = u, own_s = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int pu = __shfl_up_sync(0xffffffffu, u, o), ps = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) { u += pu; s += ps; }
    }
    q.unit0 = units + u - own_u;
    q.seg0 = segs + s - own_s;
    if (b < a.B) a.seq[b] = q;
    units += __shfl_sync(0xffffffffu, u, 31);
    segs += __shfl_sync(0xffffffffu, s, 31);
  }
  if (lane == 0) a.seq[a.B] = AttnSeq{0, 0, units, segs};
}

// The pass's first kernel: CTA m < M gathers the embedding of row m into the residual stream and normalises it; CTA M does
// the bookkeeping, a warp per sequence in turn.
template <int OP, int V>
__global__ void __launch_bounds__(kRowThreads)
embed_norm_kernel(BlockArgs a, int M, const __nv_bfloat16* __restrict__ embed, __nv_bfloat16* x, const __nv_bfloat16* __restrict__ g,
                  int nvec, float eps, int adders, RowOperand out) {
  __shared__ float s_buf[64];
  pdl_trigger();
  const int m = blockIdx.x;
  if (m >= M) {
    __shared__ int s_parent[kRowThreads / 32][QUASAR_MAX_BLOCK], s_depth[kRowThreads / 32][QUASAR_MAX_BLOCK];
    __shared__ unsigned long long s_anc[kRowThreads / 32][QUASAR_MAX_BLOCK];
    const int warp = threadIdx.x >> 5;
    for (int k = threadIdx.x; k < a.n_clear; k += kRowThreads) a.clear[k] = 0u;
    for (int b = warp; b < a.B; b += kRowThreads / 32) {
      prepare_sequence(a, b, s_parent[warp], s_anc[warp], s_depth[warp]);
      __syncwarp();
    }
    __syncthreads();
    if (warp == 0) lay_out_list(a);
    return;
  }
  uint4 gain[V > 0 ? V : 1];
  load_gain<V>(gain, g, nvec);
  const int tok = a.tokens[m];
  const bool ok = tok >= 0 && tok < a.vocab;
  const uint4* src = reinterpret_cast<const uint4*>(embed) + (size_t)(ok ? tok : 0) * nvec;
  uint4* dst = reinterpret_cast<uint4*>(x) + (size_t)m * nvec;
  norm_row<OP, V>(
      [&](int i, float (&f)[8]) {
        const uint4 v = ok ? __ldg(src + i) : make_uint4(0, 0, 0, 0);
        dst[i] = v;
        unpack8(v, f);
      },
      gain, g, nvec, eps, adders, m, out, s_buf);
}

// One warp per sequence: the rows' top choices out of their arg-max keys, then greedy acceptance (Eq. 2 at temperature
// 0) in shared memory.
__global__ void __launch_bounds__(32)
accept_kernel(BlockArgs a, int32_t* __restrict__ accept_len, int32_t* __restrict__ bonus, int32_t* __restrict__ accept_path) {
  __shared__ int s_tok[QUASAR_MAX_BLOCK], s_par[QUASAR_MAX_BLOCK], s_top[QUASAR_MAX_BLOCK], s_path[QUASAR_MAX_BLOCK];
  pdl_trigger();
  pdl_wait();
  const int b = blockIdx.x, lane = threadIdx.x, base = b * a.T_max;
  const bool valid = a.bi.valid[b] != 0;
  const int T = valid ? a.block_len[b] : 0;
  for (int i = lane; i < a.T_max; i += 32) {
    s_path[i] = -1;
    if (i < T) {
      const unsigned long long k = a.keys[base + i];
      s_top[i] = k == 0ull ? 0 : (int)(0xffffffffu - (uint32_t)(k & 0xffffffffull));
      s_tok[i] = a.tokens[base + i];
      s_par[i] = a.parents ? a.parents[base + i] : i - 1;
    }
  }
  __syncwarp();
  int n = -1, bon = -1;   // a skipped sequence: -1 tells quasar_kv_commit to leave its cache and seq_len alone
  if (valid) {
    int cur = 0;
    n = 0;
    if (lane == 0) s_path[0] = 0;
    while (true) {   // the lowest row that follows `cur` and holds the verifier's choice
      const int want = s_top[cur];
      int nxt = -1;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = lane + 32 * h;
        const unsigned hit = __ballot_sync(0xffffffffu, c > cur && c < T && s_par[c] == cur && s_tok[c] == want);
        if (nxt < 0 && hit) nxt = 32 * h + __ffs(hit) - 1;
      }
      if (nxt < 0) break;
      cur = nxt;
      ++n;
      if (lane == 0) s_path[n] = cur;
    }
    bon = s_top[cur];
  }
  __syncwarp();
  if (lane == 0) {
    accept_len[b] = n;
    bonus[b] = bon;
  }
  if (accept_path != nullptr)
    for (int i = lane; i < a.T_max; i += 32) accept_path[base + i] = s_path[i];
}

// turns of 8 * 512 elements a row takes, rounded up to a form that exists; 0: too long for registers
int turns_of(int nvec) {
  const int v = (nvec + kRowThreads - 1) / kRowThreads;
  return v <= 1 ? 1 : v <= 2 ? 2 : v <= 3 ? 3 : v <= 6 ? 6 : 0;
}

template <typename... P, typename... A>
int launch_row(void (*kernel)(P...), int grid, size_t smem, bool pdl, cudaStream_t stream, A&&... args) {
  return launch_dependent(kernel, dim3((unsigned)grid), dim3(kRowThreads), smem, pdl, stream, 1, static_cast<A&&>(args)...);
}

// Dynamic shared memory of a norm that leaves codes: the pairs' sums of a row that stays in registers, at most 48 KB.  With what
// the kernels hold besides (16.3 KB of bookkeeping in the first one) that is more than a kernel gets unasked.
constexpr size_t kNormMaxSmem = (size_t)6 * kRowThreads * 16;
size_t norm_smem(int nvec) { return turns_of(nvec) > 0 ? (size_t)nvec * 16 : 0; }

#define ROW_DISPATCH(KERNEL, ...)                                                                                              \
  switch (turns_of(nvec)) {                                                                                                    \
    case 1: ROW_DISPATCH_OP(KERNEL, 1, __VA_ARGS__)                                                                            \
    case 2: ROW_DISPATCH_OP(KERNEL, 2, __VA_ARGS__)                                                                            \
    case 3: ROW_DISPATCH_OP(KERNEL, 3, __VA_ARGS__)                                                                            \
    case 6: ROW_DISPATCH_OP(KERNEL, 6, __VA_ARGS__)                                                                            \
    default: ROW_DISPATCH_OP(KERNEL, 0, __VA_ARGS__)                                                                           \
  }
#define ROW_DISPATCH_OP(KERNEL, V, ...)                                                                                        \
  switch (op) {                                                                                                                \
    case kOperandDigits: return launch_row(KERNEL<kOperandDigits, V>, __VA_ARGS__);                                            \
    case kOperandCodes: return launch_row(KERNEL<kOperandCodes, V>, __VA_ARGS__);                                              \
    default: return launch_row(KERNEL<kOperandBf16, V>, __VA_ARGS__);                                                          \
  }

}  // namespace

int launch_embed_norm(int op, const BlockArgs& a, const __nv_bfloat16* embed, __nv_bfloat16* x, const __nv_bfloat16* g, int H, float eps,
                      int adders, const RowOperand& out, cudaStream_t stream) {
  const int nvec = H / 8, M = a.B * a.T_max;
  if (op == kOperandCodes) {
    static DeviceOnce once;
    const int rc = allow_shared_memory(once, kNormMaxSmem, false,
                                       {(const void*)embed_norm_kernel<kOperandCodes, 1>, (const void*)embed_norm_kernel<kOperandCodes, 2>,
                                        (const void*)embed_norm_kernel<kOperandCodes, 3>, (const void*)embed_norm_kernel<kOperandCodes, 6>});
    if (rc != QUASAR_OK) return rc;
  }
  ROW_DISPATCH(embed_norm_kernel, M + 1, op == kOperandCodes ? norm_smem(nvec) : 0, false, stream, a, M, embed, x, g, nvec, eps, adders, out)
}

int launch_norm(int op, const __nv_bfloat16* x, const __nv_bfloat16* g, int M, int H, float eps, int adders, const RowOperand& out, cudaStream_t stream) {
  const int nvec = H / 8;
  if (op == kOperandCodes) {
    static DeviceOnce once;
    const int rc = allow_shared_memory(once, kNormMaxSmem, false,
                                       {(const void*)norm_kernel<kOperandCodes, 1>, (const void*)norm_kernel<kOperandCodes, 2>,
                                        (const void*)norm_kernel<kOperandCodes, 3>, (const void*)norm_kernel<kOperandCodes, 6>});
    if (rc != QUASAR_OK) return rc;
  }
  ROW_DISPATCH(norm_kernel, M, op == kOperandCodes ? norm_smem(nvec) : 0, true, stream, x, g, nvec, eps, adders, out)
}

int launch_swiglu(int op, const __nv_bfloat16* gu, int M, int F, const RowOperand& out, cudaStream_t stream) {
  const int nvec = F / 8;
  ROW_DISPATCH(swiglu_kernel, M, 0, true, stream, gu, nvec, out)
}

int launch_operand(int op, const __nv_bfloat16* x, const unsigned* row_max, int M, int K, const RowOperand& out, cudaStream_t stream) {
  if (op == kOperandBf16) return QUASAR_OK;   // the row itself is the operand
  const int nvec = K / 8;
  const dim3 grid((unsigned)((nvec + kElemThreads - 1) / kElemThreads), (unsigned)M);
  if (op == kOperandDigits) return launch_dependent(operand_kernel<kOperandDigits>, grid, dim3(kElemThreads), 0, true, stream, 1, x, row_max, nvec, out);
  return launch_dependent(operand_kernel<kOperandCodes>, grid, dim3(kElemThreads), 0, true, stream, 1, x, row_max, nvec, out);
}

namespace {
constexpr size_t kMergeMaxSmem = 208 * 1024;
template <int OP, int D, bool LIST>
int launch_merge(int warps, size_t smem, const AttnList& list, const AttnParts& parts, const AttnChunks& ch, int batch, int M,
                 const RowOperand& out, cudaStream_t stream) {
  static DeviceOnce once;
  const int rc = allow_shared_memory(once, kMergeMaxSmem, false, {(const void*)attention_merge_kernel<OP, D, LIST>});
  if (rc != QUASAR_OK) return rc;
  return launch_dependent(attention_merge_kernel<OP, D, LIST>, dim3((unsigned)(M * kMergeCtas)), dim3((unsigned)warps * 32), smem, true, stream,
                          kMergeCtas, list, parts, ch, batch, out);
}
}  // namespace

int launch_attention_merge(int op, const AttnList& list, const AttnParts& parts, const AttnChunks* chunks, int M, int D,
                           const RowOperand& out, cudaStream_t stream) {
  const int heads = (list.Hkv * list.G + kMergeCtas - 1) / kMergeCtas;   // of a CTA
  const int warps = heads < kMergeWarps ? heads : kMergeWarps;
  // few rows: round trips count (6 rows, 34 chunks of the W8A8 form: all at once), many: CTAs on an SM do
  int batch = M > 16 ? 8 : chunks == nullptr ? 16 : std::min(40, std::max(16, chunks->nchunk));
  auto bytes = [&] { return (size_t)heads * D * 2 + (size_t)warps * batch * D * 4; };
  while (bytes() > kMergeMaxSmem && batch > 1) batch /= 2;
  const size_t smem = bytes();
  if (smem > kMergeMaxSmem) { set_error("attention merge: %d query heads of %d", list.Hkv * list.G, D); return QUASAR_ERR_SHAPE; }
  const AttnChunks ch = chunks ? *chunks : AttnChunks{};
#define MERGE_AS(OP, DD, LIST) return launch_merge<OP, DD, LIST>(warps, smem, list, parts, ch, batch, M, out, stream)
#define MERGE(OP)                                     \
  if (D == 128) {                                     \
    if (chunks) MERGE_AS(OP, 128, false);             \
    MERGE_AS(OP, 128, true);                          \
  }                                                   \
  if (chunks) MERGE_AS(OP, 64, false);                \
  MERGE_AS(OP, 64, true);
  if (op == kOperandDigits) { MERGE(kOperandDigits) }
  if (op == kOperandCodes) { MERGE(kOperandCodes) }
  MERGE(kOperandBf16)
#undef MERGE_AS
#undef MERGE
}

int launch_accept(const BlockArgs& a, int32_t* accept_len, int32_t* bonus, int32_t* accept_path, cudaStream_t stream) {
  return launch_dependent(accept_kernel, dim3((unsigned)a.B), dim3(32), 0, true, stream, 1, a, accept_len, bonus, accept_path);
}

}  // namespace quasar
