// Drafting by prompt lookup (Section 4.1: the n-gram drafter of all of the paper's experiments; lookup
// range K = (K_min, K_max), Section 4.4 / Table 3).  For n = K_max down to K_min the last n tokens of a
// sequence are looked up in the tokens before them; the most recent earlier occurrence that is followed
// by at least one token wins and the up to gamma tokens that followed it become the draft; the longest n
// with such an occurrence is used.
//
// One CTA per sequence, one pass over the history whatever the range of n: an occurrence is told by where it ENDS (one
// position before the last token at most), and the length of the match backwards from there, capped at K_max, is the
// longest n that it serves.  The winner is the largest (length, end) - an integer maximum, so the result does not
// depend on the order of the threads.  Bound by latency (two dependent loads and a block reduction): 1024 threads take
// four positions each at once; one pass per n with 256 threads took 10.8 us at 4096 tokens, this 4-5 us.
#include "common.cuh"

namespace quasar {

namespace {

constexpr int kDraftThreads = 1024;
constexpr int kDraftUnroll = 4;

__global__ void __launch_bounds__(kDraftThreads)
ngram_draft_kernel(const int32_t* __restrict__ history, const int32_t* __restrict__ hist_len, int S, int gamma, int k_min,
                   int k_max, int32_t* __restrict__ draft, int32_t* __restrict__ draft_len) {
  __shared__ unsigned long long s_best;
  const int b = blockIdx.x;
  const int32_t* h = history + (size_t)b * S;
  const int L = min(max(hist_len[b], 0), S);
  if (threadIdx.x == 0) s_best = 0;
  __syncthreads();
  unsigned long long best = 0;   // (length of the match) << 32 | (end of the occurrence); 0: none
  if (L >= 2) {
    const int32_t last = h[L - 1];
    for (int e0 = threadIdx.x; e0 < L - 1; e0 += kDraftThreads * kDraftUnroll) {
      int32_t t[kDraftUnroll];
#pragma unroll
      for (int u = 0; u < kDraftUnroll; ++u) {
        const int e = e0 + u * kDraftThreads;
        t[u] = e < L - 1 ? h[e] : ~last;
      }
#pragma unroll
      for (int u = 0; u < kDraftUnroll; ++u) {
        if (t[u] != last) continue;
        const int e = e0 + u * kDraftThreads;
        int n = 1;
        while (n < k_max && n <= e && h[e - n] == h[L - 1 - n]) ++n;
        const unsigned long long key = (unsigned long long)(unsigned)n << 32 | (unsigned)e;
        if (n >= k_min && key > best) best = key;
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long other = __shfl_xor_sync(0xffffffffu, best, o);
    best = other > best ? other : best;
  }
  if ((threadIdx.x & 31) == 0 && best != 0) atomicMax(&s_best, best);
  __syncthreads();
  best = s_best;
  int len = 0, from = 0;
  if (best != 0) {
    from = (int)(best & 0xffffffffu) + 1;
    len = min(gamma, L - from);
  }
  for (int i = threadIdx.x; i < gamma; i += kDraftThreads) draft[(size_t)b * gamma + i] = i < len ? h[from + i] : -1;
  if (threadIdx.x == 0) draft_len[b] = len;
}

}  // namespace

int launch_ngram_draft(const int32_t* history, const int32_t* hist_len, int B, int S, int gamma, int k_min, int k_max,
                       int32_t* draft, int32_t* draft_len, cudaStream_t stream) {
  ngram_draft_kernel<<<B, kDraftThreads, 0, stream>>>(history, hist_len, S, gamma, k_min, k_max, draft, draft_len);
  QUASAR_LAUNCH_CHECK();
  return QUASAR_OK;
}

}  // namespace quasar
