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
#include "tc_common.cuh"

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
// segment lie before the row.
__device__ __forceinline__ int row_lead(const float* row) { return (int)((reinterpret_cast<uintptr_t>(row) & 15u) >> 2); }

// 16 values as four 128-bit loads `stride` positions apart
template <int stride, typename F>
__device__ __forceinline__ void load16(const float* row, int first, int V, float fill, F&& put) {
#pragma unroll
  for (int j = 0; j < kPerThread / 4; ++j) {
    const int v = first + stride * j;
    if (v >= 0 && v + 4 <= V) {
      const float4 x = __ldg(reinterpret_cast<const float4*>(row + v));
      put(4 * j, x.x); put(4 * j + 1, x.y); put(4 * j + 2, x.z); put(4 * j + 3, x.w);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) put(4 * j + e, (v + e >= 0 && v + e < V) ? __ldg(row + v + e) : fill);
    }
  }
}

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// (maximum, sum of exponentials against it) of two parts put together
__device__ __forceinline__ float2 join(float2 x, float2 y, float inv_t) {
  const float m = fmaxf(x.x, y.x);
  if (!(m > -INFINITY)) return make_float2(m, 0.f);
  return make_float2(m, x.y * expf((x.x - m) * inv_t) + y.y * expf((y.x - m) * inv_t));
}

// part[(b * T_max + i) * nseg + s] = (maximum, sum of exp((x - maximum) / temperature)) of a segment; also clears the
// arrival counters of the kernel that follows.
__global__ void __launch_bounds__(kSegThreads)
softmax_segment_kernel(const float* __restrict__ logits, const int32_t* __restrict__ block_len, int T_max, int V, int nseg,
                       int chunks, float inv_t, float2* __restrict__ part, unsigned* __restrict__ arrivals) {
  __shared__ float2 sh[kSegThreads / 32];
  tc::pdl_trigger();
  const int s = blockIdx.x, i = blockIdx.y, b = blockIdx.z;
  if (s == 0 && i == 0 && threadIdx.x == 0) arrivals[b] = 0;
  if (i >= block_len[b]) return;
  const float* row = logits + ((size_t)b * T_max + i) * V;
  float2 acc = make_float2(-INFINITY, 0.f);   // of this warp: one block-wide meeting per segment, not one per reduction
  for (int c = 0; c < chunks; ++c) {
    float x[kPerThread];
    load16<kChunk / 4>(row, (s * chunks + c) * kChunk + threadIdx.x * 4 - row_lead(row), V, -INFINITY, [&](int j, float v) { x[j] = v; });
    float m = x[0];
#pragma unroll
    for (int j = 1; j < kPerThread; ++j) m = fmaxf(m, x[j]);
    m = warp_max(m);
    float sum = 0.f;
    if (m > -INFINITY) {
#pragma unroll
      for (int j = 0; j < kPerThread; ++j) sum += expf((x[j] - m) * inv_t);
    }
    const float2 part_c = make_float2(m, warp_sum(sum));
    acc = c == 0 ? part_c : join(acc, part_c, inv_t);
  }
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    acc = sh[0];
#pragma unroll
    for (int w = 1; w < kSegThreads / 32; ++w) acc = join(acc, sh[w], inv_t);   // warps in order
    part[((size_t)b * T_max + i) * nseg + s] = acc;
  }
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
  load16<4>(d.row, first, V, -INFINITY, [&](int j, float v) { w[j] = expf((v - d.max) * inv_t) * d.inv_sum; });
  if (d.qrow != nullptr)
    load16<4>(d.qrow, first, V, 0.f, [&](int j, float v) { w[j] = fmaxf(0.f, w[j] - v); });   // Eq. 3
#pragma unroll
  for (int j = 0; j < kPerThread; ++j)
    if (first + j == d.tok) w[j] = 0.f;                                                   // point-mass drafter
}

__global__ void __launch_bounds__(kSegThreads) draw_segment_kernel(DrawArgs a) {
  __shared__ float sh[kSegThreads / 32];
  __shared__ float2 s_row[QUASAR_MAX_BLOCK];      // per block row: maximum and sum
  __shared__ float s_logit[QUASAR_MAX_BLOCK], s_q[QUASAR_MAX_BLOCK], s_r[QUASAR_MAX_BLOCK];   // of the next block token
  __shared__ int s_n, s_rejected, s_last, s_pick, s_seg;
  __shared__ float s_target, s_begin;
  const int s = blockIdx.x, b = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int T = min(a.block_len[b], a.T_max);
  const float r_sample = a.r_sample[b];

  // ---- row statistics: half a warp per row, its lanes over the segments; the last T threads fetch what the walk
  //      compares them with ----
  const int t_row = kSegThreads - 1 - (int)threadIdx.x;
  if (t_row < T) {
    float x = 0.f, q = 1.f, r = 0.f;
    if (t_row + 1 < T) {
      const int tok = a.tokens[b * a.T_max + t_row + 1];
      const size_t at = ((size_t)b * a.T_max + t_row) * a.V + tok;
      r = a.r_accept[b * a.T_max + t_row];
      if (tok >= 0 && tok < a.V) {
        x = a.logits[at];
        if (a.q_probs != nullptr) q = a.q_probs[at];
      } else {
        q = 0.f;   // a token outside the vocabulary can only be rejected
      }
    }
    s_logit[t_row] = x;
    s_q[t_row] = q;
    s_r[t_row] = r;
  }
  tc::pdl_wait();   // (what was fetched so far is older than the kernel in front)
  for (int i = threadIdx.x >> 4; i < (T + 1) / 2 * 2; i += kSegThreads / 16) {   // (both halves of a warp take every turn)
    const float2* p = a.part + ((size_t)b * a.T_max + i) * a.nseg;
    float2 v[kMaxSegments / 16];
#pragma unroll
    for (int k = 0; k < kMaxSegments / 16; ++k) {
      const int at = (threadIdx.x & 15) + 16 * k;
      v[k] = (i < T && at < a.nseg) ? p[at] : make_float2(-INFINITY, 0.f);
    }
    float m = -INFINITY;
#pragma unroll
    for (int k = 0; k < kMaxSegments / 16; ++k) m = fmaxf(m, v[k].x);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    float sum = 0.f;
#pragma unroll
    for (int k = 0; k < kMaxSegments / 16; ++k)
      if (v[k].y > 0.f) sum += v[k].y * expf((v[k].x - m) * a.inv_t);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (i < T && (threadIdx.x & 15) == 0) s_row[i] = make_float2(m, sum);
  }
  __syncthreads();
  if (threadIdx.x == 0) {   // Eq. 2 along the chain
    int n = 0, rejected = 0;
    for (int i = 0; i + 1 < T; ++i) {
      const float p_tok = expf((s_logit[i] - s_row[i].x) * a.inv_t) / s_row[i].y, q_tok = s_q[i];
      const float ratio = q_tok > 0.f ? fminf(1.f, p_tok / q_tok) : 0.f;
      if (!(q_tok > 0.f) || !(s_r[i] < ratio)) { rejected = 1; break; }
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
    local = warp_sum(local);
    if (lane == 0) sh[warp] = local;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kSegThreads / 32; ++k) seg += sh[k];   // warps in order
    if (c + 1 < a.chunks) __syncthreads();
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
      float own[kMaxSegments / 32], incl[kMaxSegments / 32];
#pragma unroll
      for (int k = 0; k < kMaxSegments / 32; ++k) {
        const int at = lane + 32 * k;
        own[k] = 0.f;
        if (at < a.nseg) {
          if (attempt == 0) {
            own[k] = __ldcg(a.seg_sum + (size_t)b * a.nseg + at);
          } else {   // p itself: its segment sums are known from the statistics
            const float2 p = a.part[((size_t)b * a.T_max + i) * a.nseg + at];
            own[k] = p.y > 0.f ? p.y * expf((p.x - d.max) * a.inv_t) * d.inv_sum : 0.f;
          }
        }
        incl[k] = own[k];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const float up = __shfl_up_sync(0xffffffffu, incl[k], o);
          if (lane >= o) incl[k] += up;
        }
      }
      float total = 0.f;
#pragma unroll
      for (int k = 0; k < kMaxSegments / 32; ++k) total += __shfl_sync(0xffffffffu, incl[k], 31);
      const float target = r_sample * total;
      int found = -1, last = -1;
      float begin_found = 0.f, carry = 0.f;
#pragma unroll
      for (int k = 0; k < kMaxSegments / 32; ++k) {
        float excl = __shfl_up_sync(0xffffffffu, incl[k], 1);
        if (lane == 0) excl = 0.f;
        const unsigned hit = __ballot_sync(0xffffffffu, own[k] > 0.f && carry + excl <= target && target < carry + incl[k]);
        const unsigned pos = __ballot_sync(0xffffffffu, own[k] > 0.f);
        if (pos) last = 32 * k + 31 - __clz(pos);
        if (hit && found < 0) {
          const int l = __ffs(hit) - 1;
          found = 32 * k + l;
          begin_found = __shfl_sync(0xffffffffu, carry + excl, l);
        }
        carry += __shfl_sync(0xffffffffu, incl[k], 31);
      }
      if (lane == 0) {
        s_seg = total > 0.f ? (found >= 0 ? found : last) : -1;
        // r_sample * total rounded up to the total: no interval holds it, the last positive token is taken
        s_begin = found >= 0 ? begin_found : 0.f;
        s_target = found >= 0 ? target : INFINITY;
      }
    }
    __syncthreads();
    if (s_seg >= 0) {
      const float target = s_target;
      float base = s_begin;
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
  return launch_dependent(draw_segment_kernel, dim3(p.nseg, B), dim3(kSegThreads), 0, true, stream, 1, a);
}

}  // namespace quasar
