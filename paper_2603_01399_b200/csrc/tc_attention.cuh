// The list of key tiles that the tcgen05 attention deals out to its CTAs (tc_attention.cu), and the places of its partial
// results, for the kernel that merges them (row_ops.cu).
#pragma once

#include "common.cuh"

namespace quasar {

constexpr int kAttnCtas = 148;    // one per SM
constexpr int kShapes = 64;       // sequences whose places a CTA keeps in shared memory (more are looked up as they come)

// block rows whose query heads of one kv head make up a row tile of the 128-row MMAs
constexpr int attn_nodes_per_tile(int G) { return 128 / G; }
constexpr int attn_row_tiles(int G, int T) { return (T + attn_nodes_per_tile(G) - 1) / attn_nodes_per_tile(G); }

// Segments in order of sequence, kv head, row tile (npt block rows x G query heads); a segment's units are its tiles
// of 128 keys.  CTA c < ctas = min(148, total) takes the units [c * total / ctas, (c + 1) * total / ctas) - one at least -, and its partial results for segment s
// lie in slot c + s.
struct AttnList {
  const int32_t *seq_len, *block_len, *valid;
  const AttnSeq* seq;     // [B + 1]
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

// adds the partial results up into rows and leaves the o projection's operand (row_ops.cu); chunks: partial results of
// launch_attention instead of this list's
int launch_attention_merge(int op, const AttnList& list, const AttnParts& parts, const AttnChunks* chunks, int M, int D,
                           const RowOperand& out, cudaStream_t stream);

#ifdef __CUDACC__
__device__ __forceinline__ unsigned attn_ctas(unsigned total) { return total < (unsigned)kAttnCtas ? total : (unsigned)kAttnCtas; }

// Walks the sequences in order, to the one that holds a unit.
struct AttnCursor {
  int b;
  AttnSeq q;
  __device__ __forceinline__ void load(const AttnList& l, const AttnSeq* known) { q = b < kShapes ? known[b] : l.seq[b]; }   // known: the first kShapes
  __device__ __forceinline__ void start(const AttnList& l, const AttnSeq* known) {
    b = 0;
    load(l, known);
  }
  __device__ __forceinline__ void seek(const AttnList& l, const AttnSeq* known, int u) {
    while (b + 1 < l.B && u >= q.unit0 + q.tiles * q.row_tiles * l.Hkv) {
      ++b;
      load(l, known);
    }
  }
};
#endif

}  // namespace quasar
