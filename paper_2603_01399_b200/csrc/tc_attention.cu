// Grouped-query verify-attention on the 5th-generation tensor cores (the attention of the verification pass, Section 3.1:
// every block row attends to the cached context x_<t plus the block rows its mask allows - earlier rows for a chain,
// ancestors for a tree).
//
// The second HBM stream of the pass: K and V of the prefix are read once per layer, 4 D bytes per position and kv head.
// One kv head serves R = G * T query rows (G query heads x T block rows).  The rows are the 128-row operand of the MMAs:
//   S = Q K^T      operands in shared memory, 128 keys at a time, S in tensor memory (one lane per query row)
//   softmax        a thread owns a row: maximum, exponentials and their sum without any exchange between threads
//   O += P V       P goes back to tensor memory as a bf16 high and low part (two MMAs: about 16 bits of the
//                  probabilities) over S; V is read as it lies (keys x d, the MMA's transposed form)
// Two groups of four softmax warps take the key tiles in turn, each with an S and an O of its own (4 x 128 columns, all of
// the tensor memory), so that one group's softmax passes under the other's MMAs; nothing is exchanged between them.  The
// query rows come by TMA too, two pieces of work deep, and the MMAs run on from piece to piece.
// O is scaled only when a row's maximum grows by more than 2^8 over the one its sums stand against.
//
// Work split: the key tiles of all (sequence, kv head, row tile) segments form one list, and each of the 148 CTAs takes an
// equal run of it, whatever the lengths of the sequences; a run's part of a segment leaves two partial results (one per
// group: row maxima, sums, O), which attention_merge (row_ops.cu) adds in list order.
//
// What bounds it: HBM on long prefixes.  Per 128 keys (64 KB) an SM spends about 1540 cycles of MMAs, 1030 issue slots of
// softmax and 2900 cycles of its share of the memory's bandwidth.
#include <math.h>

#include "common.cuh"
#include "tc_attention.cuh"
#include "tc_common.cuh"

namespace quasar {

namespace {

using namespace tc;

constexpr int kKeys = 128;        // keys of a tile
constexpr int kThreadsA = 320;    // TMA warp, MMA warp, two groups of four softmax warps
constexpr int kSlots = 5;         // ring of K and V tiles in turn
constexpr float kLog2eA = 1.4426950408889634f;
constexpr float kGrow = 8.f;      // how far (in powers of two) a row's maximum may outgrow its reference

struct TcAttnArgs {
  AttnList list;
  float* o_part;              // [slots][2][128][D]
  float2* ml_part;            // [slots][2][128]
  int q_rows;                 // query rows a box of map_q brings: G * npt
  int32_t* error;
};

// 32 consecutive columns of this thread's lane
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* f) {
  uint32_t v[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,"
      "%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]),
        "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]),
        "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]),
        "=r"(v[30]), "=r"(v[31])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) f[i] = __uint_as_float(v[i]);
}

__device__ __forceinline__ float ex2(float x) {   // 2^x; results below the normal range are zero
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x));
  return y;
}

// Which of the 32 keys from key0 on a row may see: all before the block (key < P), in the block those of its ancestor mask
// (which has no bit beyond the block).
__device__ __forceinline__ uint32_t visible32(unsigned long long anc, int key0, int P) {
  const int off = key0 - P;
  if (off <= -32) return 0xffffffffu;
  if (off < 0) return (uint32_t)(anc << (-off)) | ((1u << (-off)) - 1u);
  return off < 64 ? (uint32_t)(anc >> off) : 0u;
}

// V as operand B: N = d (contiguous, 64 elements = 128 bytes per swizzled row), K = keys; groups of 8 keys 1024 bytes apart,
// the second 64 of d a sub-tile further
__device__ __forceinline__ uint64_t desc_v(const void* smem_tile) {
  uint64_t d = 0;
  d |= (uint64_t)((smem_u32(smem_tile) & 0x3ffff) >> 4);
  d |= (uint64_t)((kKeys * 128) >> 4) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// A CTA's run through the list: piece by piece (a piece = its tiles of one segment).
struct Walk {
  AttnCursor cur;
  const AttnSeq* known;
  int u, end;
  int b, hk, rt, t0, nt, seg;   // the piece: sequence, kv head, row tile, first key tile, key tiles, ordinal of the segment
  __device__ Walk(const AttnList& l, const AttnSeq* k, int total, int cta) : known(k) {
    const int ctas = (int)attn_ctas((unsigned)total);
    u = cta < ctas ? (int)((long long)cta * total / ctas) : 0;
    end = cta < ctas ? (int)((long long)(cta + 1) * total / ctas) : 0;
    cur.start(l, known);
  }
  __device__ bool next(const AttnList& l) {
    if (u >= end) return false;
    cur.seek(l, known, u);
    b = cur.b;
    const int in = u - cur.q.unit0, s = in / cur.q.tiles;
    t0 = in - s * cur.q.tiles;
    nt = min(cur.q.tiles - t0, end - u);
    hk = s / cur.q.row_tiles;
    rt = s - hk * cur.q.row_tiles;
    seg = cur.q.seg0 + s;
    u += nt;
    return true;
  }
};

template <int D>
__global__ void __launch_bounds__(kThreadsA, 1)
tc_attention_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                    const __grid_constant__ CUtensorMap map_v, const TcAttnArgs a) {
  constexpr int kSubs = D / 64;                     // 128-byte columns of a row
  constexpr int kSub = kKeys * 128;                 // bytes of one of them for a tile's keys (or the 128 query rows)
  constexpr int kTile = kSubs * kSub;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char* q_s = smem;                        // two pieces' query rows, then the ring
  unsigned char* ring = smem + 2 * kTile;
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + (size_t)kSlots * kTile);
  uint64_t* empty = full + kSlots;
  uint64_t* q_full = empty + kSlots;                // [2] a piece's query rows have landed
  uint64_t* q_empty = q_full + 2;                   // [2] its last S is complete
  uint64_t* s_full = q_empty + 2;                   // [2] S of a group's tile is complete
  uint64_t* p_ready = s_full + 2;                   // [2] P lies over it
  uint64_t* pv_done = p_ready + 2;                  // [2] O has the products of a group's part of a piece
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(pv_done + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    *abort_flag = 0;
    for (int s = 0; s < kSlots; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(q_full + i, 1);
      mbar_init(q_empty + i, 1);
      mbar_init(s_full + i, 1);
      mbar_init(p_ready + i, 4);
      mbar_init(pv_done + i, 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;   // columns: S (then P) of group 0, of group 1, O of group 0, of group 1
  // The sequences' places, fetched once and side by side (each role walks them on its own).  They come from the pass's first
  // kernel, which is complete: the kernel in front lets this one start only once it has waited for all before it.
  __shared__ AttnSeq s_seq[kShapes];
  __shared__ int s_total;
  for (int b = (int)threadIdx.x; b < min(a.list.B, kShapes); b += kThreadsA) s_seq[b] = a.list.seq[b];
  if (threadIdx.x == kThreadsA - 1) s_total = a.list.seq[a.list.B].unit0;
  __syncthreads();

  Walk w(a.list, s_seq, s_total, (int)blockIdx.x);
  if (warp != 0) pdl_wait();
  if (warp == 0) {
    // ---- TMA producer ----
    const uint64_t policy = l2_evict_first_policy();
    int s = 0, issued = 0, piece = 0;
    uint32_t ph = 0;
    bool ok = true;
    auto load_kv = [&](int i, int row, bool v) {
      unsigned char* at = ring + (size_t)i * kTile;
      mbar_expect_tx(full + i, kTile);
#pragma unroll
      for (int c = 0; c < kSubs; ++c) tma_load_2d_hint(at + c * kSub, v ? &map_v : &map_k, c * 128, row, full + i, policy);
    };
    // the first piece's tiles that lie in the cached context do not depend on the kernel in front
    bool more = w.next(a.list);
    int early = 0;
    if (more) {
      const int P = a.list.seq_len[w.b], row0 = (w.b * a.list.Hkv + w.hk) * a.list.s_max + w.t0 * kKeys;
      for (; early < min(2 * w.nt, kSlots) && (w.t0 + (early >> 1) + 1) * kKeys <= P; ++early) {
        if (elect_one()) load_kv(early, row0 + (early >> 1) * kKeys, (early & 1) != 0);
        __syncwarp();
      }
    }
    pdl_wait();
    if (lane == 0) pdl_trigger();
    for (; ok && more; more = w.next(a.list)) {
      const int row0 = (w.b * a.list.Hkv + w.hk) * a.list.s_max + w.t0 * kKeys;
      const int qb = piece & 1;
      if (!(ok = mbar_wait(q_empty + qb, ((uint32_t)(piece >> 1) & 1u) ^ 1u, abort_flag, a.error))) break;
      if (elect_one()) {
        mbar_expect_tx(q_full + qb, (uint32_t)(kSubs * a.q_rows * 128));
#pragma unroll
        for (int c = 0; c < kSubs; ++c)
          tma_load_3d(q_s + qb * kTile + c * kSub, &map_q, c * 128, w.hk * a.list.G, w.b * a.list.T_max + w.rt * a.list.npt, q_full + qb);
      }
      __syncwarp();
      ++piece;
      for (int t = 0; t < w.nt && ok; ++t) {
#pragma unroll 1
        for (int kv = 0; kv < 2; ++kv) {
          if (issued >= early) {
            if (!(ok = mbar_wait(empty + s, ph ^ 1u, abort_flag, a.error))) break;
            if (elect_one()) load_kv(s, row0 + t * kKeys, kv != 0);
            __syncwarp();
          }
          ++issued;
          if (++s == kSlots) { s = 0; ph ^= 1u; }
        }
      }
    }
    if (!ok) {   // given up: what is in flight lands (bounded) before the CTA leaves
      for (; issued < early; ++issued)
        if (++s == kSlots) { s = 0; ph ^= 1u; }
      for (int i = 0; i < min(kSlots, issued); ++i) {
        if (--s < 0) { s = kSlots - 1; ph ^= 1u; }
        const unsigned long long t0 = gtime_ns();
        while (!mbar_try(full + s, ph) && gtime_ns() - t0 < 100000ull) {}
      }
      for (int i = 0; i < min(2, piece); ++i) {
        const int p = piece - 1 - i;
        const unsigned long long t0 = gtime_ns();
        while (!mbar_try(q_full + (p & 1), (uint32_t)(p >> 1) & 1u) && gtime_ns() - t0 < 100000ull) {}
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer: S of tile i, then O of tile i - 1, on through the pieces.  (A commit covers every MMA before it, so the
    //      s_full of tile i + 2 also says that P of tile i, which it overwrites, has been used.) ----
    const uint32_t id_s = idesc(1, 1, 128, kKeys);
    const uint32_t id_o = idesc(1, 1, 128, D) | (1u << 16);   // B transposed
    uint32_t p_ph[2] = {0u, 0u};
    int slot = 0, piece = 0, i = 0;
    uint32_t ph = 0;
    bool ok = true;
    auto step_slot = [&]() { if (++slot == kSlots) { slot = 0; ph ^= 1u; } };
    // the product of the tile before: its V slot, and whether it is its group's first of the piece / the last of it
    bool pending = false, pend_first = false, pend_done = false;
    int pend_slot = 0;
    auto product = [&](int tile) {
      const int g = tile & 1;
      if (!(ok = mbar_wait(p_ready + g, p_ph[g], abort_flag, a.error))) return;
      p_ph[g] ^= 1u;
      fence_after();
      if (elect_one()) {
        const uint64_t dv = desc_v(ring + (size_t)pend_slot * kTile);
        const uint32_t tp = tmem + (uint32_t)(g * 128), to = tmem + (uint32_t)(256 + g * 128);
#pragma unroll
        for (int kk = 0; kk < kKeys / 16; ++kk) {   // 16 keys: the high part of P, then the low part
          const uint64_t dvk = dv + (uint64_t)((kk * 16 * 128) >> 4);
          const uint32_t tpk = tp + (uint32_t)((kk >> 1) * 32 + (kk & 1) * 8);
          mma_f16_ts(to, tpk, dvk, id_o, (!pend_first || kk > 0) ? 1u : 0u);
          mma_f16_ts(to, tpk + 16u, dvk, id_o, 1u);
        }
        commit(empty + pend_slot);
        if (pend_done) commit(pv_done + g);
      }
      __syncwarp();
    };
    while (ok && w.next(a.list)) {
      const int qb = piece & 1;
      if (!(ok = mbar_wait(q_full + qb, (uint32_t)(piece >> 1) & 1u, abort_flag, a.error))) break;
      ++piece;
      for (int t = 0; t < w.nt; ++t, ++i) {
        if (!(ok = mbar_wait(full + slot, ph, abort_flag, a.error))) break;
        fence_after();
        if (elect_one()) {
          const uint64_t dq = desc_sw128(q_s + qb * kTile), dk = desc_sw128(ring + (size_t)slot * kTile);
#pragma unroll
          for (int j = 0; j < D / 16; ++j) {
            const uint64_t off = (uint64_t)(((j >> 2) * kSub + (j & 3) * 32) >> 4);
            mma_f16_ss(tmem + (uint32_t)((i & 1) * 128), dq + off, dk + off, id_s, j > 0 ? 1u : 0u);
          }
          commit(s_full + (i & 1));
          commit(empty + slot);
          if (t == w.nt - 1) commit(q_empty + qb);
        }
        __syncwarp();
        step_slot();
        if (pending) product(i - 1);
        if (!ok) break;
        // (the softmax warps of this tile wait for its V themselves where they have to touch it)
        if (!(ok = mbar_wait(full + slot, ph, abort_flag, a.error))) break;
        pending = true;
        pend_slot = slot;
        pend_first = t < 2;
        pend_done = t + 2 >= w.nt;
        step_slot();
      }
    }
    if (ok && pending) product(i - 1);
  } else {
    // ---- softmax: warps 2..9.  Group 0 the warps 2..5, group 1 the warps 6..9; a warp's tensor-memory lanes are 32 (warp % 4)
    //      .. + 31, lane = query row of the tile ----
    const int g = (warp - 2) >> 2, q = warp & 3;
    const int row = q * 32 + lane;
    const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16);
    const uint32_t ts = lane_base + (uint32_t)(g * 128), to = lane_base + (uint32_t)(256 + g * 128);
    const float scale_log2 = kLog2eA / sqrtf((float)D);
    const int G = a.list.G;
    uint32_t s_ph = 0, pv_ph = 0;
    int done = 0;            // key tiles of the pieces before
    bool ok = true;
    while (ok && w.next(a.list)) {
      const int T = a.list.block_len[w.b], P = a.list.seq_len[w.b], Lk = P + T;
      const int node0 = w.rt * a.list.npt, rows = min(a.list.npt, T - node0) * G;
      const bool active = q * 32 < rows;   // (a warp without rows only keeps the hand-shakes going)
      const bool live = row < rows;
      const unsigned long long anc = live ? a.list.anc[w.b * a.list.T_max + node0 + row / G] : 0ull;
      float m_ref = -INFINITY, sum = 0.f;
      const size_t slot = ((size_t)(blockIdx.x + w.seg) * 2 + g) * 128 + row;
      const int t_first = (done & 1) ^ g;   // this group's first tile of the piece
      for (int t = t_first; t < w.nt; t += 2) {
        if (!(ok = __all_sync(0xffffffffu, mbar_wait(s_full + g, s_ph, abort_flag, a.error)))) break;
        s_ph ^= 1u;
        fence_after();
        const int k0 = (w.t0 + t) * kKeys;
        if (active) {
          const bool edge = k0 + kKeys > P;   // keys of the block in it, or beyond the end
          auto load = [&](int c, float (&s)[32]) {
            tmem_ld32(ts + (uint32_t)(c * 32), s);
            if (edge) {
              const uint32_t see = visible32(anc, k0 + c * 32, P);
#pragma unroll
              for (int j = 0; j < 32; ++j) s[j] = (see >> j) & 1u ? s[j] : -INFINITY;
            }
          };
          float mx = -INFINITY;
#pragma unroll 1
          for (int c = 0; c < kKeys / 32; ++c) {
            float s[32];
            load(c, s);
            float m4[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
            for (int j = 4; j < 32; ++j) m4[j & 3] = fmaxf(m4[j & 3], s[j]);
            mx = fmaxf(mx, fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])));
          }
          mx *= scale_log2;
          // a new reference for rows whose maximum has outgrown the old one: O and the sum are scaled down to it
          const bool grow = mx > m_ref + kGrow;   // (the first tile with a visible key always)
          if (__any_sync(0xffffffffu, grow)) {
            const float m_new = grow ? mx : m_ref;
            const float f = grow ? (m_ref == -INFINITY ? 0.f : exp2f(m_ref - m_new)) : 1.f;
            if (t > t_first) {   // (this S is complete, so the product of this group's tile before is)
#pragma unroll 1
              for (int c = 0; c < D / 32; ++c) {
                float o[32];
                tmem_ld32(to + (uint32_t)(c * 32), o);
                uint32_t ow[32];
#pragma unroll
                for (int j = 0; j < 32; ++j) ow[j] = __float_as_uint(o[j] * f);
                tmem_st32(to + (uint32_t)(c * 32), ow);
              }
            }
            sum *= f;
            m_ref = m_new;
          }
          const float m_use = m_ref == -INFINITY ? 0.f : m_ref;
          float sum0 = 0.f, sum1 = 0.f;
#pragma unroll 1
          for (int c = 0; c < kKeys / 32; ++c) {   // 32 keys at a time: 16 columns of high parts, then 16 of low parts
            float s[32];
            load(c, s);
            uint32_t p[32];
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const float p0 = ex2(fmaf(s[2 * j], scale_log2, -m_use)), p1 = ex2(fmaf(s[2 * j + 1], scale_log2, -m_use));
              sum0 += p0;
              sum1 += p1;
              const __nv_bfloat162 h2 = __floats2bfloat162_rn(p0, p1);
              p[j] = *reinterpret_cast<const uint32_t*>(&h2);
              const __nv_bfloat162 l2 = __floats2bfloat162_rn(p0 - __uint_as_float(p[j] << 16), p1 - __uint_as_float(p[j] & 0xffff0000u));
              p[16 + j] = *reinterpret_cast<const uint32_t*>(&l2);
            }
            tmem_st32(ts + (uint32_t)(c * 32), p);
          }
          sum += sum0 + sum1;
          tmem_st_wait();
        }
        if (k0 + kKeys > Lk) {
          // rows of V beyond the end of the sequence are whatever lies there: zero, since P = 0 does not silence a NaN
          const int c = 2 * (done + t) + 1;   // this tile's V in the ring's order
          if (!(ok = __all_sync(0xffffffffu, mbar_wait(full + c % kSlots, (uint32_t)(c / kSlots) & 1u, abort_flag, a.error)))) break;
          unsigned char* vt = ring + (size_t)(c % kSlots) * kTile;
          const int from = Lk - k0;
          for (int i = from * 8 * kSubs + (q * 32 + lane); i < kKeys * 8 * kSubs; i += 128) {
            const int r = i / (8 * kSubs), pc = i % (8 * kSubs);
            *reinterpret_cast<uint4*>(vt + (pc >> 3) * kSub + r * 128 + ((pc & 7) << 4)) = make_uint4(0, 0, 0, 0);
          }
          asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        }
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(p_ready + g);
      }
      if (!ok) break;
      if (w.nt > t_first) {   // the group's products are in O
        if (!(ok = __all_sync(0xffffffffu, mbar_wait(pv_done + g, pv_ph, abort_flag, a.error)))) break;
        pv_ph ^= 1u;
        fence_after();
      }
      if (active) {   // the piece's partial result
        if (live) a.ml_part[slot] = make_float2(m_ref, sum);
        if (w.nt > t_first) {
#pragma unroll
          for (int c = 0; c < D / 32; ++c) {
            float o[32];
            tmem_ld32(to + (uint32_t)(c * 32), o);
            if (live) {
              float4* dst = reinterpret_cast<float4*>(a.o_part + slot * D + c * 32);
#pragma unroll
              for (int j = 0; j < 8; ++j) dst[j] = make_float4(o[4 * j], o[4 * j + 1], o[4 * j + 2], o[4 * j + 3]);
            }
          }
        }
        fence_before();   // (the next piece's P, which follows in this warp's order, lets O be overwritten)
      }
      done += w.nt;
    }
  }
  __syncwarp();
  fence_before();
  __syncthreads();
  if (warp == 1) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512u) : "memory");
  }
}

template <int D>
int launch_d(const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv, const TcAttnArgs& a, int ctas, cudaStream_t stream) {
  constexpr size_t smem = (size_t)(2 + kSlots) * (D / 64) * kKeys * 128 + 1024 + 512;
  static DeviceOnce once;
  const int rc = allow_shared_memory(once, smem, false, {(const void*)tc_attention_kernel<D>});
  if (rc != QUASAR_OK) return rc;
  return launch_dependent(tc_attention_kernel<D>, dim3((unsigned)ctas), dim3(kThreadsA), smem, true, stream, 1, mq, mk, mv, a);
}

}  // namespace

size_t tc_attention_workspace_bytes(int B, int T_max, int Hq, int Hkv, int D) {
  const size_t slots = kAttnCtas + (size_t)B * Hkv * attn_row_tiles(Hq / Hkv, T_max);
  return slots * 2 * 128 * ((size_t)D * 4 + 8);
}

AttnParts tc_attention_parts(void* workspace, int B, int T_max, int Hq, int Hkv, int D) {
  const size_t slots = kAttnCtas + (size_t)B * Hkv * attn_row_tiles(Hq / Hkv, T_max);
  AttnParts p;
  p.o = reinterpret_cast<float*>(workspace);
  p.ml = reinterpret_cast<float2*>(p.o + slots * 2 * 128 * D);
  return p;
}

int launch_tc_attention(const __nv_bfloat16* qkv, const __nv_bfloat16* k_cache_layer, const __nv_bfloat16* v_cache_layer,
                        const AttnList& list, int kv_batch, int D, const AttnParts& parts, int32_t* error, cudaStream_t stream) {
  CUtensorMap mq, mk, mv;
  const uint64_t rows = (uint64_t)kv_batch * list.Hkv * list.s_max;
  int rc = make_map_sw128(&mk, k_cache_layer, rows, (uint64_t)D * 2, kKeys);
  if (rc != QUASAR_OK) return rc;
  rc = make_map_sw128(&mv, v_cache_layer, rows, (uint64_t)D * 2, kKeys);
  if (rc != QUASAR_OK) return rc;
  rc = make_map3_sw128(&mq, qkv, (uint64_t)D * 2, (uint64_t)list.Hkv * (list.G + 2), (uint64_t)list.B * list.T_max,
                       (uint32_t)list.G, (uint32_t)list.npt);
  if (rc != QUASAR_OK) return rc;
  TcAttnArgs a;
  a.q_rows = list.G * list.npt; a.list = list; a.o_part = parts.o; a.ml_part = parts.ml; a.error = error;
  return D == 128 ? launch_d<128>(mq, mk, mv, a, kAttnCtas, stream) : launch_d<64>(mq, mk, mv, a, kAttnCtas, stream);
}

}  // namespace quasar
