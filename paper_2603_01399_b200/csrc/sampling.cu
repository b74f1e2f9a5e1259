// Stochastic acceptance of a drafted chain (Section 3.1 Eq. 2-3; Section 3.3 "Lossless Rejection
// Sampling"), on the logits the verification pass produced.  Per draft position: target probability
// p = softmax(logits / T) of the drafted token against the drafter's q, accepted while r < min(1, p / q)
// (Eq. 2); at the first rejection a corrective token is drawn from norm(max(0, p - q)) (Eq. 3); if every
// draft is accepted one more token is drawn from the target distribution of the last row.  Random numbers
// are inputs (r_accept per draft position, r_sample per sequence); a token is drawn from unnormalised
// weights by inversion: the smallest v with w_0 + ... + w_v > r_sample * sum(w).  A drafter that gives no
// distribution is the point mass on its token (a retrieval drafter proposes one token with certainty).
//
// Two kernels over at most 64 segments of kChunk tokens (or a multiple of it, above 262,140), all reductions in a fixed order (results repeat bit for bit).
//  1. softmax_segment_kernel: maximum and sum of exponentials of every segment of every block row.  Bound by
//     HBM: the logits are read once, 16 values per thread in flight.
//  2. draw_segment_kernel: every CTA puts the row statistics of its sequence together and walks the chain (a few
//     hundred values out of L2, cheaper than a launch of its own), sums the weights of its segment of the row to
//     draw from, and the last CTA of a sequence to finish picks the token: segment by a scan over the segment sums,
//     token by a scan over one segment.  Only one row per sequence is read again.
// One CTA per row and one per sequence, as this file had it before, left a 151,936-token row to 512 threads and the
// draw to one SM: 42 + 5 + 152 us at 8 x 9 rows; the segments spread both over the chip.
#include <math.h>

#include "common.cuh"

namespace quasar {

namespace {

constexpr int kSegThreads = 256;
constexpr int kPerThread = 16;
constexpr int kChunk = kSegThreads * kPerThread;   // 38 segments of a 152k vocabulary: even one short block fills the chip
constexpr int kMaxSegments = 64;

// segments of a row of V tokens and chunks per segment (up to 3 positions lie before the row, see row_lead)
struct SegPlan { int nseg, chunks; };
SegPlan seg_plan(int V) {
  const int64_t total = ((int64_t)V + 3 + kChunk - 1) / kChunk;
  SegPlan p;
  p.chunks = (int)((total + kMaxSegments - 1) / kMaxSegments);
  p.nseg = (int)((total + p.chunks - 1) / p.chunks);
  return p;
}

// A row starts anywhere (V may be odd), so segments are cut on 16-byte boundaries: `lead` values (0..3) of the first
// segment lie before the row.  Thread t holds positions 16 t .. 16 t + 15 of the segment.
__device__ __forceinline__ int row_lead(const float* row) { return (int)((reinterpret_cast<uintptr_t>(row) & 15u) >> 2); }

template <typename F>
__device__ __forceinline__ void load16(const float* row, int first, int V, float fill, F&& put) {
#pragma unroll
  for (int j = 0; j < kPerThread / 4; ++j) {
    const int v = first + 4 * j;
    if (v >= 0 && v + 4 <= V) {
      const float4 x = __ldg(reinterpret_cast<const float4*>(row + v));
      put(4 * j, x.x); put(4 * j + 1, x.y); put(4 * j + 2, x.z); put(4 * j + 3, x.w);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) put(4 * j + e, (v + e >= 0 && v + e < V) ? __ldg(row + v + e) : fill);
    }
  }
}

__device__ __forceinline__ float block_max(float v, float* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  float r = sh[0];
#pragma unroll
  for (int i = 1; i < kSegThreads / 32; ++i) r = fmaxf(r, sh[i]);
  __syncthreads();
  return r;
}
__device__ __forceinline__ float block_sum(float v, float* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  float r = 0.f;
#pragma unroll
  for (int i = 0; i < kSegThreads / 32; ++i) r += sh[i];   // warps in order
  __syncthreads();
  return r;
}

// part[(b * T_max + i) * nseg + s] = (maximum, sum of exp((x - maximum) / temperature)) of a segment; also clears the
// arrival counters of the kernel that follows.
__global__ void __launch_bounds__(kSegThreads)
softmax_segment_kernel(const float* __restrict__ logits, const int32_t* __restrict__ block_len, int T_max, int V, int nseg,
                       int chunks, float inv_t, float2* __restrict__ part, unsigned* __restrict__ arrivals) {
  __shared__ float sh[kSegThreads / 32];
  const int s = blockIdx.x, i = blockIdx.y, b = blockIdx.z;
  if (s == 0 && i == 0 && threadIdx.x == 0) arrivals[b] = 0;
  if (i >= block_len[b]) return;
  const float* row = logits + ((size_t)b * T_max + i) * V;
  float m = -INFINITY, sum = 0.f;
  for (int c = 0; c < chunks; ++c) {
    const int first = (s * chunks + c) * kChunk + threadIdx.x * kPerThread - row_lead(row);
    float x[kPerThread];
    load16(row, first, V, -INFINITY, [&](int j, float v) { x[j] = v; });
    float cm = x[0];
#pragma unroll
    for (int j = 1; j < kPerThread; ++j) cm = fmaxf(cm, x[j]);
    cm = fmaxf(block_max(cm, sh), m);
    if (cm > -INFINITY) {
      float cs = 0.f;
#pragma unroll
      for (int j = 0; j < kPerThread; ++j) cs += expf((x[j] - cm) * inv_t);
      cs = block_sum(cs, sh);
      sum = c == 0 ? cs : sum * expf((m - cm) * inv_t) + cs;
      m = cm;
    }
  }
  if (threadIdx.x == 0) part[((size_t)b * T_max + i) * nseg + s] = make_float2(m, sum);
}

struct DrawArgs {
  const float* logits;
  const int32_t* tokens;
  const int32_t* block_len;
  const float* q_probs;
  const float* r_accept;
  const float* r_sample;
  const float2* part;
  float* seg_sum;        // [B][nseg]
  unsigned* arrivals;    // [B]
  int32_t* accept_len;
  int32_t* next_token;
  int T_max, V, nseg, chunks;
  float inv_t;
};

struct Draw {   // what to draw from: a row, its softmax statistics, and what is taken off it
  const float* row;
  const float* qrow;   // residual of a drafter with a distribution, or nullptr
  int tok;             // residual of a point mass: the token, else -1
  float max, inv_sum;
};

// The weights of this thread's 16 positions of a chunk of the row.
__device__ __forceinline__ void draw_weights(const Draw& d, int chunk, int V, float inv_t, int& first, float (&w)[kPerThread]) {
  first = chunk * kChunk + threadIdx.x * kPerThread - row_lead(d.row);
  load16(d.row, first, V, -INFINITY, [&](int j, float v) { w[j] = expf((v - d.max) * inv_t) * d.inv_sum; });
  if (d.qrow != nullptr)
    load16(d.qrow, first, V, 0.f, [&](int j, float v) { w[j] = fmaxf(0.f, w[j] - v); });   // Eq. 3
#pragma unroll
  for (int j = 0; j < kPerThread; ++j)
    if (first + j == d.tok) w[j] = 0.f;                                                   // point-mass drafter
}

__global__ void __launch_bounds__(kSegThreads) draw_segment_kernel(DrawArgs a) {
  __shared__ float sh[kSegThreads / 32];
  __shared__ float4 s_row[QUASAR_MAX_BLOCK];      // per block row: max, sum, p of the next block token, q of it
  __shared__ int s_n, s_rejected, s_last, s_pick, s_seg;
  __shared__ float s_total, s_begin;
  const int s = blockIdx.x, b = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int T = min(a.block_len[b], a.T_max);

  // ---- row statistics: a warp per row, lanes over the segments ----
  for (int i = warp; i < T; i += kSegThreads / 32) {
    const float2* p = a.part + ((size_t)b * a.T_max + i) * a.nseg;
    float m = -INFINITY;
    for (int k = lane; k < a.nseg; k += 32) m = fmaxf(m, p[k].x);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    float sum = 0.f;
    for (int k = lane; k < a.nseg; k += 32) sum += p[k].y * expf((p[k].x - m) * a.inv_t);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) {
      float p_tok = 0.f, q_tok = 1.f;
      if (i + 1 < T) {
        const int tok = a.tokens[b * a.T_max + i + 1];
        const size_t at = ((size_t)b * a.T_max + i) * a.V + tok;
        if (tok >= 0 && tok < a.V) {
          p_tok = expf((a.logits[at] - m) * a.inv_t) / sum;
          if (a.q_probs != nullptr) q_tok = a.q_probs[at];
        } else {
          q_tok = 0.f;   // a token outside the vocabulary can only be rejected
        }
      }
      s_row[i] = make_float4(m, sum, p_tok, q_tok);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {   // Eq. 2 along the chain
    int n = 0, rejected = 0;
    for (int i = 0; i + 1 < T; ++i) {
      const float p_tok = s_row[i].z, q_tok = s_row[i].w;
      const float ratio = q_tok > 0.f ? fminf(1.f, p_tok / q_tok) : 0.f;
      if (!(q_tok > 0.f) || !(a.r_accept[b * a.T_max + i] < ratio)) { rejected = 1; break; }
      ++n;
    }
    s_n = n;
    s_rejected = rejected;
    if (s == 0) a.accept_len[b] = n;
  }
  __syncthreads();
  const int i = s_rejected ? s_n : T - 1;
  const size_t row_at = ((size_t)b * a.T_max + i) * a.V;
  Draw d;
  d.row = a.logits + row_at;
  d.qrow = (s_rejected && a.q_probs != nullptr) ? a.q_probs + row_at : nullptr;
  d.tok = (s_rejected && a.q_probs == nullptr) ? a.tokens[b * a.T_max + i + 1] : -1;
  if (d.tok < 0) d.tok = 0x7fffffff;       // no position: also not one of the (at most 3) before the row
  d.max = s_row[i].x;
  d.inv_sum = 1.0f / s_row[i].y;

  float w[kPerThread];
  int first;
  float seg = 0.f;
  for (int c = 0; c < a.chunks; ++c) {
    draw_weights(d, s * a.chunks + c, a.V, a.inv_t, first, w);
    float local = 0.f;
#pragma unroll
    for (int j = 0; j < kPerThread; ++j) local += w[j];
    seg += block_sum(local, sh);
  }
  if (threadIdx.x == 0) {
    __stcg(a.seg_sum + (size_t)b * a.nseg + s, seg);
    __threadfence();
    s_last = atomicAdd(a.arrivals + b, 1u) == (unsigned)a.nseg - 1u;
    s_pick = -1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();

  // ---- the last CTA of the sequence: segment, then token ----
  for (int attempt = 0; attempt < 2; ++attempt) {
    if (warp == 0) {
      // the segments' intervals [begin, end) tile [0, total): 32 at a time, an end is the next one's begin
      float carry = 0.f;
      for (int k0 = 0; k0 < a.nseg; k0 += 32) {
        float v = 0.f;
        if (k0 + lane < a.nseg) {
          if (attempt == 0) {
            v = __ldcg(a.seg_sum + (size_t)b * a.nseg + k0 + lane);
          } else {   // p itself: its segment sums are known from the statistics
            const float2 p = a.part[((size_t)b * a.T_max + i) * a.nseg + k0 + lane];
            v = p.y * expf((p.x - d.max) * a.inv_t) * d.inv_sum;
          }
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const float up = __shfl_up_sync(0xffffffffu, v, o);
          if (lane >= o) v += up;
        }
        carry += __shfl_sync(0xffffffffu, v, 31);
      }
      const float total = carry;
      const float target = a.r_sample[b] * total;
      int found = -1, last = -1;
      float begin_found = 0.f;
      carry = 0.f;
      for (int k0 = 0; k0 < a.nseg && found < 0; k0 += 32) {
        float v = 0.f;
        if (k0 + lane < a.nseg) {
          if (attempt == 0) {
            v = __ldcg(a.seg_sum + (size_t)b * a.nseg + k0 + lane);
          } else {
            const float2 p = a.part[((size_t)b * a.T_max + i) * a.nseg + k0 + lane];
            v = p.y * expf((p.x - d.max) * a.inv_t) * d.inv_sum;
          }
        }
        const float own = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const float up = __shfl_up_sync(0xffffffffu, v, o);
          if (lane >= o) v += up;
        }
        float excl = __shfl_up_sync(0xffffffffu, v, 1);
        if (lane == 0) excl = 0.f;
        const unsigned hit = __ballot_sync(0xffffffffu, own > 0.f && carry + excl <= target && target < carry + v);
        const unsigned pos = __ballot_sync(0xffffffffu, own > 0.f);
        if (pos) last = k0 + 31 - __clz(pos);
        if (hit) {
          const int l = __ffs(hit) - 1;
          found = k0 + l;
          begin_found = __shfl_sync(0xffffffffu, carry + excl, l);
        }
        carry += __shfl_sync(0xffffffffu, v, 31);
      }
      if (lane == 0) {
        s_total = total;
        s_seg = found >= 0 ? found : last;
        // r_sample * total rounded up to the total: no interval holds it, the last positive token is taken
        s_begin = found >= 0 ? begin_found : -INFINITY;
      }
    }
    __syncthreads();
    if (s_total > 0.f && s_seg >= 0) {
      const float target = s_begin > -INFINITY ? a.r_sample[b] * s_total : INFINITY;
      float base = s_begin > -INFINITY ? s_begin : 0.f;
      int last_pos = -1;
      for (int c = 0; c < a.chunks; ++c) {
        draw_weights(d, s_seg * a.chunks + c, a.V, a.inv_t, first, w);
        float local = 0.f;
#pragma unroll
        for (int j = 0; j < kPerThread; ++j) {
          local += w[j];
          if (w[j] > 0.f) last_pos = first + j;
        }
        float incl = local;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const float up = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += up;
        }
        float excl = __shfl_up_sync(0xffffffffu, incl, 1);
        if (lane == 0) excl = 0.f;
        if (lane == 31) sh[warp] = incl;
        __syncthreads();
        float before = base;
        for (int k = 0; k < warp; ++k) before += sh[k];
        if (local > 0.f && before + excl <= target && target < before + incl) {
          // walk the 16 positions that hold the target; if rounding leaves none, their last positive one
          float acc = before + excl;
          int pick = -1;
#pragma unroll
          for (int j = 0; j < kPerThread; ++j) {
            acc += w[j];
            if (pick < 0 && w[j] > 0.f && acc > target) pick = first + j;
          }
          s_pick = pick >= 0 ? pick : last_pos;
        }
        for (int k = 0; k < kSegThreads / 32; ++k) base += sh[k];
        __syncthreads();
        if (s_pick >= 0) break;
      }
      if (s_pick < 0) {   // the target lies in the last rounding of the segment's sum: its last positive position
        __syncthreads();
        if (last_pos >= 0) atomicMax(&s_pick, last_pos);
        __syncthreads();
      }
      break;
    }
    // max(0, p - q) is empty (p == q): the corrective token comes from p itself
    __syncthreads();
    d.qrow = nullptr;
    d.tok = 0x7fffffff;
  }
  if (threadIdx.x == 0) a.next_token[b] = s_pick < 0 ? 0 : s_pick;
}

size_t align256s(size_t v) { return (v + 255) / 256 * 256; }

}  // namespace

size_t accept_stochastic_workspace_bytes(int B, int T_max) {
  return align256s((size_t)B * T_max * kMaxSegments * sizeof(float2)) + align256s((size_t)B * kMaxSegments * sizeof(float)) +
         align256s((size_t)B * sizeof(unsigned));
}

int launch_accept_stochastic(const float* logits, const int32_t* tokens, const int32_t* block_len, const float* q_probs, int B,
                             int T_max, int V, float temperature, const float* r_accept, const float* r_sample,
                             int32_t* accept_len, int32_t* next_token, void* workspace, cudaStream_t stream) {
  unsigned char* ws = reinterpret_cast<unsigned char*>(workspace);
  const SegPlan p = seg_plan(V);
  DrawArgs a;
  float2* part = reinterpret_cast<float2*>(ws);
  ws += align256s((size_t)B * T_max * kMaxSegments * sizeof(float2));
  a.seg_sum = reinterpret_cast<float*>(ws);
  a.arrivals = reinterpret_cast<unsigned*>(ws + align256s((size_t)B * kMaxSegments * sizeof(float)));
  a.logits = logits; a.tokens = tokens; a.block_len = block_len; a.q_probs = q_probs;
  a.r_accept = r_accept; a.r_sample = r_sample; a.part = part;
  a.accept_len = accept_len; a.next_token = next_token;
  a.T_max = T_max; a.V = V; a.nseg = p.nseg; a.chunks = p.chunks;
  a.inv_t = 1.0f / temperature;
  softmax_segment_kernel<<<dim3(p.nseg, T_max, B), kSegThreads, 0, stream>>>(logits, block_len, T_max, V, p.nseg, p.chunks, a.inv_t,
                                                                             part, a.arrivals);
  QUASAR_LAUNCH_CHECK();
  draw_segment_kernel<<<dim3(p.nseg, B), kSegThreads, 0, stream>>>(a);
  QUASAR_LAUNCH_CHECK();
  return QUASAR_OK;
}

}  // namespace quasar
