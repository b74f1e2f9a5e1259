// The list of key tiles that the tcgen05 attention deals out to its CTAs (tc_attention.cu), and the places of its partial
// results, for the kernel that merges them (row_ops.cu).
#pragma once

#include "common.cuh"

namespace quasar {

constexpr int kAttnCtas = 148;    // one per SM
constexpr int kShapes = 128;       // sequences whose shapes a CTA keeps in shared memory (more are looked up as they come)

// block rows whose query heads of one kv head make up a row tile of the 128-row MMAs
constexpr int attn_nodes_per_tile(int G) { return 128 / G; }
constexpr int attn_row_tiles(int G, int T) { return (T + attn_nodes_per_tile(G) - 1) / attn_nodes_per_tile(G); }

// Segments in order of sequence, kv head, row tile (npt block rows x G query heads); a segment's units are its tiles
// of 128 keys.  CTA c takes the units [c * total / ctas, (c + 1) * total / ctas), and its partial results for segment s
// lie in slot c + s.
struct AttnList {
  const int32_t *seq_len, *block_len, *valid;
  const uint64_t* anc;    // [B*T_max]
  int B, T_max, Hkv, G, s_max, npt;
};

struct AttnParts {
  float* o;      // [slots][2 groups][128 rows][D] un-normalised outputs
  float2* ml;    // [slots][2][128] row maximum (power of two), sum
};

size_t tc_attention_workspace_bytes(int B, int T_max, int Hq, int Hkv, int D);
AttnParts tc_attention_parts(void* workspace, int B, int T_max, int Hq, int Hkv, int D);
int launch_tc_attention(const __nv_bfloat16* qkv, const __nv_bfloat16* k_cache_layer, const __nv_bfloat16* v_cache_layer,
                        const AttnList& list, int kv_batch, int D, const AttnParts& parts, int32_t* error, cudaStream_t stream);

// adds the partial results up into rows and leaves the o projection's operand (row_ops.cu)
int launch_attention_merge(int op, const AttnList& list, const AttnParts& parts, int M, int D, const RowOperand& out, cudaStream_t stream);

#ifdef __CUDACC__
// key tiles and row tiles of a sequence (none of a skipped one)
__device__ __forceinline__ void attn_shape(const AttnList& l, int b, int& tiles, int& row_tiles) {
  const int ok = l.valid[b], T = l.block_len[b], P = l.seq_len[b];   // (side by side: a skipped one's may be anything)
  tiles = ok ? (P + T + 127) / 128 : 0;
  row_tiles = ok ? (T + l.npt - 1) / l.npt : 0;
}

// units of all sequences (every lane of a converged warp gets the sum)
__device__ __forceinline__ long long attn_total(const AttnList& l) {
  long long sum = 0;
  for (int b = (int)(threadIdx.x & 31); b < l.B; b += 32) {
    int t, r;
    attn_shape(l, b, t, r);
    sum += (long long)t * r * l.Hkv;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  return sum;
}

// Walks the sequences in order: the first unit and segment of sequence b, and its shape.
struct AttnCursor {
  int b, seg0, tiles, row_tiles;
  long long unit0;
  __device__ __forceinline__ void shape(const AttnList& l, const int2* known) {   // known: the first kShapes sequences'
    if (b < kShapes) { tiles = known[b].x; row_tiles = known[b].y; }
    else attn_shape(l, b, tiles, row_tiles);
  }
  __device__ __forceinline__ void start(const AttnList& l, const int2* known) {
    b = 0;
    seg0 = 0;
    unit0 = 0;
    shape(l, known);
  }
  __device__ __forceinline__ void seek(const AttnList& l, const int2* known, long long u) {   // the sequence that holds unit u
    while (b < l.B && u >= unit0 + (long long)tiles * row_tiles * l.Hkv) {
      unit0 += (long long)tiles * row_tiles * l.Hkv;
      seg0 += row_tiles * l.Hkv;
      if (++b < l.B) shape(l, known);
    }
  }
};
#endif

}  // namespace quasar
