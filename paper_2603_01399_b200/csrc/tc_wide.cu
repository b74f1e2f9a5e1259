// Linear layers  Y = delta * (W X)  (Section 3.2 Eq. 8) with int8 weights and bf16 activations for WIDE blocks, on the
// 5th-generation tensor cores.
//
// The digit form (tc_linear.cu) pays four int8 MMA rows per activation row for never touching a weight byte with an
// instruction: right while the weights' way from memory is what takes the time, but beyond some 60 rows the MMAs do, and
// one bf16 MMA row costs what one int8 row does.  Here the weights become bf16 (exact: an int8 has 8 significant
// bits) on their way to operand A, once per weight and row tile:
//   TMA -> shared memory (int8) -> registers -> tensor memory (bf16, operand A)     X: TMA -> shared memory (operand B)
// Pairs of CTAs (cta_group::2) work on 256 channels x up to 256 rows: each brings and converts its own 128 channels and brings
// HALF of the rows, so an SM takes in 16 KB of weights and `brows` x 128 bytes of rows per 128 of K - for less the intake of an
// SM (about 105 KB per us) would not keep up with the MMAs - and shared memory serves reads and writes at 100 bytes a clock or
// less.  Operand A in tensor memory is what makes the rest fit: through shared memory it would add 32 KB of writes and reads a stage.
//
// Roles: TMA warp, MMA warp, sixteen converter warps (a group of four takes one half, 64 of K, of every other stage: 4 16-byte
// loads, 16 x (2 PRMT, 4 LOP3, 2 HADD2) and one tcgen05.st of 32 columns per thread), four epilogue warps.  What bounds it: a
// stage costs the integer pipes 780 cycles of conversion (0.41 us) and the MMAs 4 cycles a row, so up to some 190 rows a tile
// the conversion, beyond that the tensor cores: 24,576 x 4096 at 512 rows 118 us as digit rows, 82 here (1.25 PFLOP/s),
// LM head 675 -> 474 us (1.35); prompt chunks of 8 x 64 rows through the 8B model 12.5 -> 9.5 ms.  Tensor memory: accumulators of `brows` columns - two where that leaves room, so that a tile leaves
// for memory under the next one's MMAs - and a ring of 32-column pieces of operand A.
// Two forms: tiles in turn on one pair per SM pair; or, for matrices of few tiles, k-ranges of a tile in the pairs of one
// cluster, added through distributed shared memory in the order of the ranges.
//
// Every wait is bounded (2 s): on expiry the CTA raises an error word, stops waiting everywhere, releases its tensor
// memory and returns.
#include <math.h>

#include <algorithm>

#include "rope.cuh"
#include "tc_common.cuh"
#include "tc_linear.cuh"
#include "tc_wide.cuh"

namespace quasar {

namespace {

using namespace tc;

constexpr int kThreadsW = 704;           // TMA, MMA, 16 converter warps, 4 epilogue warps
constexpr int kWBytes = 128 * 128;       // a stage's weights of a CTA: 128 channels x 128 of K
constexpr int kPiece = 32;               // columns of a piece of operand A: 64 of K
constexpr int kTmem = 512;
constexpr size_t kSmemW = 227 * 1024;
constexpr size_t kFixedW = 1024 + 1024 + 8192;  // alignment of the ring; barriers and arg-max keys

struct WideArgs {
  const float* dw;             // [N]
  void* y;                     // [M][N] bf16 or fp32, or nullptr; SwiGLU: [M][N / 2] bf16
  const __nv_bfloat16* res;    // [M][N] or nullptr
  unsigned long long* keys;    // [M] or nullptr
  int32_t* error;
  int M, N, kblocks;
  int rows, brows, row_tiles, nsplit, stages;
  int accs, pieces;            // accumulators; pieces of operand A in the ring
  int acc_cols;                // columns from one accumulator to the next
  int units;
  int y_is_f32, early_weights;
  RopeArgs rope;               // kWideRope
};

// What is done with a unit's finished sums: stored; multiplied as gate and up units; or made q, k and v (QK-norm, RoPE, cache
// append: only behind ranges, whose exchange leaves whole rows of a head to a warp; a kernel and a pass over q, k and v less).
// A warp finishes its rows one after the other, so the gain shrinks with the rows, but the plan goes over to one range before it is
// gone.  us a layer against the separate kernel (passes of 4 layers on 256 positions; rows a warp in brackets):
//   rows                  65-72        96          128         176         208         224         240
//   6144 x 4096           -2.7 (1.6)   -2.4 (2.2)  -3.0 (2.9)  -2.0 (4.0)  -1.4 (4.7)  -1.0 (5.1)  one range
//   7168 x 5120           -3.1 (1.6)   -3.9 (2.2)  -2.7 (2.9)  -2.2 (4.0)  -1.2 (4.7)  -0.8 (5.1)  -0.8 (5.5)
//   3072 x 2048, heads of 64: -0.6 at 72 rows, -1.7 at 128, -2.3 at 176 in four ranges; -1.1 at 192 to 224 in two row tiles of two
// A pass of 8 x 9 rows through the 8B shape 4104 -> 3953 us, of a 17-node tree x 4 through the 14B shape 5523 -> 5364.  Tiles without
// ranges keep the separate kernel: eight rows a warp cost more than it does (8 x 64 rows 9592 -> 9765).
enum WideEpilogue { kWideStore = 0, kWideSwiglu = 1, kWideRope = 2 };

// four int8 -> four bf16, exactly: 0x43bb is 128 + bb for the low seven bits, and the sign bit asks for 256 instead of 128 to go
__device__ __forceinline__ void bf16x4(uint32_t w, uint32_t& lo, uint32_t& hi) {
  const uint32_t v[2] = {__byte_perm(w, 0x43434343u, 0x4140), __byte_perm(w, 0x43434343u, 0x4342)};
  uint32_t out[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const uint32_t t = v[i] & 0xff7fff7fu, c = v[i] & 0xff80ff80u;
    const __nv_bfloat162 d = __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&t), *reinterpret_cast<const __nv_bfloat162*>(&c));
    out[i] = *reinterpret_cast<const uint32_t*>(&d);
  }
  lo = out[0];
  hi = out[1];
}

// operand A from tensor memory, the pair form
__device__ __forceinline__ void mma_f16_ts_pair(uint32_t d, uint32_t ta, uint64_t db, uint32_t id, uint32_t accumulate) {
  asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d), "r"(ta),
               "l"(db), "r"(id), "r"(accumulate)
               : "memory");
}

__device__ __forceinline__ float round_bf16(float f) { return __bfloat162float(__float2bfloat16_rn(f)); }

// Channel of the matrix that lane `r` of a CTA's tile holds.  SwiGLU: of every 32 lanes 16 are gate units and 16 the same up units.
template <bool SWIGLU>
__device__ __forceinline__ int channel_of(int n0, int r, int N) {
  if (!SWIGLU) return n0 + r;
  const int u = n0 / 2 + (r >> 5) * 16 + (r & 15);
  return (r & 16) ? N / 2 + u : u;
}

template <bool SPLIT, int EPI>
__global__ void __launch_bounds__(kThreadsW, 1)
tc_wide_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_x, const WideArgs a) {
  constexpr bool SWIGLU = EPI == kWideSwiglu;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);   // the swizzle repeats every 1024 bytes
  const int b_half = a.brows / 2;                // rows of operand B of this CTA
  const int x_sub = b_half * 128;                // bytes of 64 of their K
  const int stage_bytes = kWBytes + 2 * x_sub;
  const int S = a.stages, NP = a.pieces;
  uint64_t* w_full = reinterpret_cast<uint64_t*>(smem + (size_t)S * stage_bytes);   // this CTA's weights have landed
  uint64_t* w_empty = w_full + S;          // and have been converted
  uint64_t* x_full = w_empty + S;          // both CTAs' rows have landed (the leader's)
  uint64_t* x_empty = x_full + S;          // and have been multiplied
  uint64_t* a_full = x_empty + S;          // [pieces] both CTAs have written the piece (the leader's)
  uint64_t* a_empty = a_full + NP;         // and it has been multiplied
  uint64_t* acc_full = a_empty + NP;       // [2]
  uint64_t* acc_empty = acc_full + 2;      // [2] (the leader's)
  unsigned long long* s_best = reinterpret_cast<unsigned long long*>(acc_empty + 2);   // [4][256] arg-max keys of the row tile's rows, by quarter
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(s_best + 1024);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // (warp: uniform)
  const int pair_x = (int)blockIdx.x & 1;
  const int split = SPLIT ? (int)blockIdx.y : 0;
  const uint32_t leader = (uint32_t)(2 * split);
  const uint16_t mask = (uint16_t)(3u << (2 * split));
  const int first = (int)blockIdx.x >> 1, step = (int)gridDim.x >> 1;
  const int kb0 = SPLIT ? (int)((long long)split * a.kblocks / a.nsplit) : 0;
  const int kb1 = SPLIT ? (int)((long long)(split + 1) * a.kblocks / a.nsplit) : a.kblocks;
  auto row_of = [&](int u) { return (u % a.row_tiles) * a.rows; };
  auto chan_of = [&](int u) { return (2 * (u / a.row_tiles) + pair_x) * 128; };

  if (threadIdx.x == 0) {
    *abort_flag = 0;
    for (int s = 0; s < S; ++s) {
      mbar_init(w_full + s, 1);
      mbar_init(w_empty + s, 8);
      mbar_init(x_full + s, 1);
      mbar_init(x_empty + s, 1);
    }
    for (int i = 0; i < NP; ++i) {
      mbar_init(a_full + i, 8);     // four warps of each CTA
      mbar_init(a_empty + i, 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(acc_full + i, 1);
      mbar_init(acc_empty + i, 8);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  for (int i = threadIdx.x; i < 1024; i += kThreadsW) s_best[i] = 0ull;
  __syncwarp();
  cluster_arrive();   // every CTA's barriers exist before another one's arrivals
  cluster_wait();
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)), "r"((uint32_t)kTmem) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;\n" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t tmem_a = tmem + (uint32_t)(a.accs * a.acc_cols);
  // (A tcgen05 kernel behind this one waits for it while it holds tensor memory.  Behind the qkv projection it is the attention, which
  // counts on everything in front of THIS kernel being complete: see below.)
  if (EPI != kWideRope && threadIdx.x == 0) pdl_trigger();

  if (warp == 0) {
    // ---- TMA producer ----
    const uint64_t policy = l2_evict_first_policy();
    auto load_w = [&](int s, int kb, int n0) {
      unsigned char* at = smem + (size_t)s * stage_bytes;
      mbar_expect_tx(w_full + s, kWBytes);
      if (SWIGLU) {
#pragma unroll
        for (int i = 0; i < 8; ++i)   // 16 gate rows, the same 16 up rows, ...
          tma_load_2d(at + i * 2048, &map_w, kb * 128, n0 / 2 + (i >> 1) * 16 + (i & 1) * (a.N / 2), w_full + s);
      } else if (a.row_tiles == 1) {
        tma_load_2d_hint(at, &map_w, kb * 128, n0, w_full + s, policy);
      } else {                        // (row tiles that share a weight tile read it at about the same time: it may stay in L2 for them)
        tma_load_2d(at, &map_w, kb * 128, n0, w_full + s);
      }
    };
    auto load_x = [&](int s, int kb, int m0) {
      unsigned char* at = smem + (size_t)s * stage_bytes + kWBytes;
      if (pair_x == 0) mbar_expect_tx(x_full + s, (uint32_t)(4 * x_sub));
      const uint32_t bar = cluster_map(smem_u32(x_full + s), leader);
#pragma unroll
      for (int h = 0; h < 2; ++h) tma_load_2d_pair<false>(at + h * x_sub, &map_x, kb * 256 + h * 128, m0 + pair_x * b_half, bar, policy);
    };
    const int ahead = first < a.units ? min(S, kb1 - kb0) : 0;
    if (a.early_weights) {   // the weights of the first stages do not depend on the kernel in front
      for (int i = 0; i < ahead; ++i) {
        if (elect_one()) load_w(i, kb0 + i, chan_of(first));
        __syncwarp();
      }
    }
    pdl_wait();
    int s = 0, issued = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int u = first; u < a.units && ok; u += step) {
      const int n0 = chan_of(u), m0 = row_of(u);
      for (int kb = kb0; kb < kb1; ++kb) {
        const bool early = a.early_weights && issued < ahead;
        if (!early && !(ok = mbar_wait(w_empty + s, ph ^ 1u, abort_flag, a.error))) break;
        if (!early && elect_one()) load_w(s, kb, n0);
        __syncwarp();
        if (!(ok = mbar_wait(x_empty + s, ph ^ 1u, abort_flag, a.error))) { ++issued; break; }
        if (elect_one()) load_x(s, kb, m0);
        __syncwarp();
        ++issued;
        if (++s == S) { s = 0; ph ^= 1u; }
      }
    }
    if (!ok) {   // given up: what is in flight lands (bounded) before the CTA leaves
      const unsigned long long t0 = gtime_ns();
      while (gtime_ns() - t0 < 200000ull) {}
    }
  } else if (warp == 1) {
    if (pair_x == 0) {   // ---- MMA issuer ----
      const uint32_t id = idesc(1, 1, 256, a.brows);
      int s = 0, buf = 0, piece = 0;
      uint32_t ph = 0, bph = 0, pph = 0;
      bool ok = true;
      for (int u = first; u < a.units && ok; u += step) {
        if (!(ok = mbar_wait(acc_empty + buf, bph ^ 1u, abort_flag, a.error))) break;
        fence_after();
        const uint32_t d = tmem + (uint32_t)(buf * a.acc_cols);
        for (int kb = kb0; kb < kb1 && ok; ++kb) {
          if (!(ok = mbar_wait(x_full + s, ph, abort_flag, a.error))) break;
          const uint64_t db = desc_sw128(smem + (size_t)s * stage_bytes + kWBytes);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (!(ok = mbar_wait(a_full + piece, pph, abort_flag, a.error))) break;
            fence_after();
            if (elect_one()) {
              const uint64_t dbh = db + (uint64_t)((uint32_t)(h * x_sub) >> 4);
              const uint32_t ta = tmem_a + (uint32_t)(piece * kPiece);
#pragma unroll
              for (int j = 0; j < 4; ++j)   // 16 of K: 8 columns of A, 32 bytes along the rows of B
                mma_f16_ts_pair(d, ta + (uint32_t)(8 * j), dbh + (uint64_t)(2 * j), id, (kb > kb0 || h > 0 || j > 0) ? 1u : 0u);
              commit_pair(a_empty + piece, mask);
              if (h == 1) commit_pair(x_empty + s, mask);
            }
            __syncwarp();
            if (++piece == NP) { piece = 0; pph ^= 1u; }
          }
          if (++s == S) { s = 0; ph ^= 1u; }
        }
        if (ok && elect_one()) commit_pair(acc_full + buf, mask);
        __syncwarp();
        if (++buf == a.accs) { buf = 0; bph ^= 1u; }
      }
    }
  } else if (warp < 18) {
    // ---- converters: a group of four warps takes half h of every other stage; a thread one channel ----
    const int g = (warp - 2) >> 2, h = g & 1, q = warp & 3, r = q * 32 + lane;
    const uint32_t lane_a = tmem_a + ((uint32_t)(q * 32) << 16);
    int s = 0, piece = g;
    uint32_t ph = 0, pph = 0;
    bool ok = true;
    int turn = g >> 1;   // 0: this stage is the group's
    for (int u = first; u < a.units && ok; u += step) {
      for (int kb = kb0; kb < kb1; ++kb, turn ^= 1) {
        if (turn != 0) {
          if (++s == S) { s = 0; ph ^= 1u; }
          continue;
        }
        if (!(ok = __all_sync(0xffffffffu, mbar_wait(w_full + s, ph, abort_flag, a.error)))) break;
        const unsigned char* row = smem + (size_t)s * stage_bytes + r * 128;
        uint32_t w[16];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const uint4 v = *reinterpret_cast<const uint4*>(row + (((h * 4 + c) ^ (r & 7)) << 4));
          w[4 * c] = v.x; w[4 * c + 1] = v.y; w[4 * c + 2] = v.z; w[4 * c + 3] = v.w;
        }
        uint32_t p[32];
#pragma unroll
        for (int i = 0; i < 16; ++i) bf16x4(w[i], p[2 * i], p[2 * i + 1]);
        __syncwarp();
        if (lane == 0) mbar_arrive(w_empty + s);
        if (!(ok = __all_sync(0xffffffffu, mbar_wait(a_empty + piece, pph ^ 1u, abort_flag, a.error)))) break;
        fence_after();
        tmem_st32(lane_a + (uint32_t)(piece * kPiece), p);
        tmem_st_wait();
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(cluster_map(smem_u32(a_full + piece), leader));
        if ((piece += 4) >= NP) { piece -= NP; pph ^= 1u; }
        if (++s == S) { s = 0; ph ^= 1u; }
      }
    }
  }
  if (!SPLIT && warp >= 18) {
    // ---- epilogue: a thread one channel, 16 rows at a time ----
    const int q = warp & 3, r = q * 32 + lane;
    pdl_wait();   // the residual comes from a kernel in front
    const bool one_row_tile = step % a.row_tiles == 0;
    int buf = 0;
    uint32_t bph = 0;
    for (int u = first; u < a.units; u += step) {
      const int m0 = row_of(u), rows = min(a.rows, a.M - m0), n0 = chan_of(u), n = channel_of<SWIGLU>(n0, r, a.N);
      const int F = a.N / 2, unit = n0 / 2 + (r >> 5) * 16 + (r & 15);
      const bool live = SWIGLU ? unit < F : n < a.N;
      const float dw = live ? __ldg(a.dw + (SWIGLU ? unit : n)) : 1.f, dw_up = SWIGLU && live ? __ldg(a.dw + F + unit) : 1.f;
      if (!__all_sync(0xffffffffu, mbar_wait(acc_full + buf, bph, abort_flag, a.error))) break;
      fence_after();
      const uint32_t t0 = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * a.acc_cols);
      for (int r0 = 0; r0 < rows; r0 += 16) {
        uint32_t v[16];
        tmem_ld16_async(t0 + (uint32_t)r0, v);
        const int count = rows - r0;
        uint16_t res[16];
        if (!SWIGLU && a.res != nullptr) load_res16(res, a.res, live, (size_t)(m0 + r0), n, a.N, count);
        tmem_ld_wait(v);
        if (SWIGLU) {
          const bool up_lane = (lane & 16) != 0;
          __nv_bfloat16* y = reinterpret_cast<__nv_bfloat16*>(a.y);
#pragma unroll
          for (int j = 0; j < 16; j += 2) {   // gate lanes finish row j, up lanes row j + 1
            const uint32_t other = __shfl_xor_sync(0xffffffffu, up_lane ? v[j] : v[j + 1], 16);
            const float gt = round_bf16(__uint_as_float(up_lane ? other : v[j]) * dw);
            const float uv = round_bf16(__uint_as_float(up_lane ? v[j + 1] : other) * dw_up);
            const int m = r0 + j + (up_lane ? 1 : 0);
            if (live && m < rows) y[(size_t)(m0 + m) * F + unit] = __float2bfloat16_rn(gt / (1.0f + expf(-gt)) * uv);
          }
        }
        if (!SWIGLU) {
          float f[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) f[j] = __uint_as_float(v[j]) * dw;
          if (a.keys != nullptr) best16(f, live, n, count, s_best + q * 256 + r0);
          if (a.y != nullptr) store16(f, live, (size_t)(m0 + r0), n, a.N, count, a.y, a.y_is_f32 != 0, a.res != nullptr, res);
        }
      }
      if (a.keys != nullptr && !one_row_tile) {   // the next tile is of other rows: the warp hands on what it has
        __syncwarp();
        for (int r0 = 0; r0 < rows; r0 += 16) {
          unsigned long long& k = s_best[q * 256 + r0 + lane % 16];
          if (lane < 16 && r0 + lane < rows && k != 0) {
            atomicMax(a.keys + m0 + r0 + lane, k);
            k = 0;
          }
        }
      }
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(cluster_map(smem_u32(acc_empty + buf), leader));
      if (++buf == a.accs) { buf = 0; bph ^= 1u; }
    }
    if (a.keys != nullptr && one_row_tile && first < a.units) {
      asm volatile("bar.sync 1, 128;\n" ::: "memory");   // (every epilogue warp comes here, one that has given up too)
      const int m0 = row_of(first);
      for (int t = (int)threadIdx.x - 576; t < min(a.rows, a.M - m0); t += 128) {
        unsigned long long k = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) k = s_best[i * 256 + t] > k ? s_best[i * 256 + t] : k;
        if (k != 0) atomicMax(a.keys + m0 + t, k);
      }
    }
  }
  if (EPI == kWideRope && warp == 18) {
    pdl_wait();
    if (lane == 0) pdl_trigger();
  }
  if (SPLIT && warp >= 2) {
    // ---- this range's sums to shared memory, [row][channel] (the ring is idle then: every load has landed and every MMA read it) ----
    const int q = warp & 3, r = q * 32 + lane;
    const uint32_t t0 = tmem + ((uint32_t)(q * 32) << 16);
    if (__all_sync(0xffffffffu, mbar_wait(acc_full, 0, abort_flag, a.error))) {
      fence_after();
      float* red = reinterpret_cast<float*>(smem);
      for (int r0 = ((warp - 2) >> 2) * 16; r0 < a.brows; r0 += 80) {
        uint32_t v[16];
        tmem_ld16(t0 + (uint32_t)r0, v);
#pragma unroll
        for (int j = 0; j < 16; ++j) red[(r0 + j) * 128 + r] = __uint_as_float(v[j]);
      }
    }
  }
  __syncwarp();
  fence_before();
  cluster_arrive();
  cluster_wait();
  if (warp == 1) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"((uint32_t)kTmem) : "memory");
  }
  if (SPLIT) {
    pdl_wait();
    if (*abort_flag == 0) {
      // this CTA's share of the tile's rows, four channels a lane
      const int m0 = row_of(first), n = chan_of(first) + lane * 4, rows = min(a.rows, a.M - m0);
      const int per = (rows + a.nsplit - 1) / a.nsplit, r_end = min(rows, (split + 1) * per);
      const uint32_t red_addr = smem_u32(smem);
      float dw[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) dw[e] = n + e < a.N ? __ldg(a.dw + n + e) : 1.f;
      for (int m = split * per + warp; m < r_end; m += kThreadsW / 32) {
        RopeRow rope;
        if constexpr (EPI == kWideRope) rope_row_load(rope, a.rope, m0 + m, chan_of(first));
        uint4 p[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (k < a.nsplit) p[k] = ld_cluster_v4(cluster_map(red_addr + (uint32_t)(m * 128 + lane * 4) * 4, (uint32_t)(2 * k + pair_x)));
        float f[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (k >= a.nsplit) break;
          const uint32_t v[4] = {p[k].x, p[k].y, p[k].z, p[k].w};
#pragma unroll
          for (int e = 0; e < 4; ++e) f[e] = k == 0 ? __uint_as_float(v[e]) : f[e] + __uint_as_float(v[e]);
        }
        if constexpr (EPI == kWideRope) {
#pragma unroll
          for (int e = 0; e < 4; ++e) f[e] = round_bf16(f[e] * dw[e]);
          if (a.rope.D == 128) rope_row_store<128>(a.rope, f, m0 + m, chan_of(first), a.N, rope);
          else rope_row_store<64>(a.rope, f, m0 + m, chan_of(first), a.N, rope);
          continue;
        }
        unsigned long long best = 0;
        const size_t idx = (size_t)(m0 + m) * a.N + n;
        if (a.keys == nullptr && (a.N & 3) == 0) {   // (then four channels are inside or outside together, and aligned)
          if (n >= a.N) continue;
#pragma unroll
          for (int e = 0; e < 4; ++e) f[e] *= dw[e];
          if (a.res != nullptr) {
            const uint2 rr = *reinterpret_cast<const uint2*>(a.res + idx);
            f[0] = round_bf16(f[0]) + __uint_as_float(rr.x << 16);
            f[1] = round_bf16(f[1]) + __uint_as_float(rr.x & 0xffff0000u);
            f[2] = round_bf16(f[2]) + __uint_as_float(rr.y << 16);
            f[3] = round_bf16(f[3]) + __uint_as_float(rr.y & 0xffff0000u);
          }
          if (a.y_is_f32) {
            *reinterpret_cast<float4*>(reinterpret_cast<float*>(a.y) + idx) = make_float4(f[0], f[1], f[2], f[3]);
          } else {
            const __nv_bfloat162 lo = __floats2bfloat162_rn(f[0], f[1]), hi = __floats2bfloat162_rn(f[2], f[3]);
            *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(a.y) + idx) =
                make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
          }
          continue;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (n + e >= a.N) break;
          float o = f[e] * dw[e];
          if (a.keys != nullptr && o == o) {
            const unsigned long long k = argmax_key(o, n + e);
            best = k > best ? k : best;
          }
          if (a.y == nullptr) continue;
          if (a.res != nullptr) o = round_bf16(o) + __bfloat162float(a.res[idx + e]);
          if (a.y_is_f32) reinterpret_cast<float*>(a.y)[idx + e] = o;
          else reinterpret_cast<__nv_bfloat16*>(a.y)[idx + e] = __float2bfloat16_rn(o);
        }
        if (a.keys != nullptr) {
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long other = __shfl_xor_sync(0xffffffffu, best, o);
            best = other > best ? other : best;
          }
          if (lane == 0 && best != 0) atomicMax(a.keys + m0 + m, best);
        }
      }
    }
    __syncwarp();
    cluster_arrive();   // nobody's shared memory goes away while another CTA may read it
    cluster_wait();
  }
}

struct WidePlan {
  int row_tiles, rows, brows, nsplit, stages, accs, pieces, acc_cols, ctas, tiles;
  double cost;
};

int allow_wide(int* device) {
  static DeviceOnce once;
  return allow_shared_memory(once, kSmemW, true, {(const void*)tc_wide_kernel<false, kWideStore>, (const void*)tc_wide_kernel<true, kWideStore>,
                                                  (const void*)tc_wide_kernel<false, kWideSwiglu>, (const void*)tc_wide_kernel<true, kWideRope>}, device);
}

// Clusters of s pairs that the device holds at once (they lie within a group of SMs, so long ones leave SMs unused).  Behind
// allow_wide, without which it holds none.  Where the question fails this plan goes by one, and the next one asks again.
int max_pair_clusters(int device, int s) {
  static DeviceAnswers<5> kept;
  return std::max(1, clusters_at_once(kept, device, s, (const void*)tc_wide_kernel<true, kWideStore>, kThreadsW, kSmemW, 2, (unsigned)s));
}

// Row tiles and k-ranges by an estimate of the time in us.  A stage (128 of K) takes its MMAs (7.0e6 multiply-adds per us on an
// SM), or its way into the SM, or 0.41 us of the hand-overs from load to conversion to MMA.  It ranks forms and is no forecast: gate+up
// at 72 rows takes 0.53 us a stage, the MMA rate is above what GEMMs reach, and launches of 512 rows take 1.3 to 1.7 times their
// estimate (qkv 18 / 27, o 18 / 31, gate+up 59 / 93, down 38 / 50).
WidePlan plan_wide(int device, int64_t M, int64_t N, int64_t K, bool swiglu, bool keys) {
  WidePlan best = {};
  const int kblocks = (int)((K + 127) / 128);
  const int tiles = (int)((N + 255) / 256);
  const int least = (int)((M + 255) / 256);
  for (int t = least; t <= least + 2 || t <= 2 * least; ++t) {
    WidePlan p = {};
    p.row_tiles = t;
    p.rows = (int)((M + t - 1) / t);
    p.brows = std::max(32, (p.rows + 15) / 16 * 16);
    p.tiles = tiles;
    p.accs = p.brows <= 192 ? 2 : 1;
    p.acc_cols = (p.brows + 31) / 32 * 32;
    p.pieces = (kTmem - p.accs * p.acc_cols) / kPiece;
    if (p.pieces > 8) p.pieces = 8;
    const int stage = kWBytes + p.brows * 128;
    p.stages = (int)((kSmemW - kFixedW) / stage);
    if (p.stages > 8) p.stages = 8;
    const double mma = p.brows * 128.0 * 128.0 / 7.0e6, intake = stage / 105e3;
    const double a = std::max(std::max(mma, intake), 0.41);
    const int units = tiles * t;
    for (int s = 1; s <= (swiglu ? 1 : 4) && s <= kblocks; ++s) {
      if (s == 1) {
        int n = 74;
        if (keys) n = 74 / t * t;   // (a CTA stays on its row tile then)
        if (n < 1) n = 74;
        n = std::min(n, units);
        const int turns = (units + n - 1) / n;
        const double drain = 0.006 * p.brows;   // of an accumulator
        p.cost = 4.0 + turns * (kblocks * a + (p.accs == 1 ? drain : 0.2)) + (p.accs == 2 ? drain : 0.0);
        p.ctas = 2 * n;
      } else {
        const int fit = max_pair_clusters(device, s);
        const int waves = (units + fit - 1) / fit;
        p.cost = waves * (6.0 + (kblocks + s - 1) / s * a + 0.012 * p.brows) + 0.3 * s;
        p.ctas = 2 * units;
      }
      p.cost = std::max(p.cost, (double)N * K / 6.3e6);
      p.nsplit = s;
      if (best.nsplit == 0 || p.cost < best.cost * 0.99) best = p;
    }
  }
  return best;
}

int launch_wide(int epi, const __nv_bfloat16* x, const int8_t* w, int64_t M, int64_t N, int64_t K, WideArgs a, bool pdl, cudaStream_t stream) {
  const bool swiglu = epi == kWideSwiglu;
  int device = 0, rc = allow_wide(&device);
  if (rc != QUASAR_OK) return rc;
  const WidePlan p = plan_wide(device, M, N, K, swiglu, a.keys != nullptr);
  CUtensorMap map_w, map_x;
  rc = make_map_sw128(&map_w, w, (uint64_t)N, (uint64_t)K, swiglu ? 16u : 128u);
  if (rc != QUASAR_OK) return rc;
  rc = make_map_sw128(&map_x, x, (uint64_t)M, (uint64_t)K * 2, (uint32_t)(p.brows / 2));
  if (rc != QUASAR_OK) return rc;
  a.M = (int)M; a.N = (int)N; a.kblocks = (int)((K + 127) / 128);
  a.rows = p.rows; a.brows = p.brows; a.row_tiles = p.row_tiles; a.nsplit = p.nsplit; a.stages = p.stages;
  a.accs = p.accs; a.pieces = p.pieces; a.acc_cols = p.acc_cols; a.units = p.tiles * p.row_tiles;
  a.early_weights = pdl ? 1 : 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)p.ctas, (unsigned)p.nsplit);
  cfg.blockDim = dim3(kThreadsW);
  cfg.dynamicSmemBytes = (size_t)p.stages * (kWBytes + p.brows * 128) + kFixedW;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = (unsigned)p.nsplit;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 2u : 1u;
  if (swiglu) QUASAR_CUDA_CHECK(cudaLaunchKernelEx(&cfg, tc_wide_kernel<false, kWideSwiglu>, map_w, map_x, a));
  else if (epi == kWideRope) QUASAR_CUDA_CHECK(cudaLaunchKernelEx(&cfg, tc_wide_kernel<true, kWideRope>, map_w, map_x, a));
  else if (p.nsplit > 1) QUASAR_CUDA_CHECK(cudaLaunchKernelEx(&cfg, tc_wide_kernel<true, kWideStore>, map_w, map_x, a));
  else QUASAR_CUDA_CHECK(cudaLaunchKernelEx(&cfg, tc_wide_kernel<false, kWideStore>, map_w, map_x, a));
  count_launch();
  return QUASAR_OK;
}

}  // namespace

// Digit rows put up to 64 rows into one tile, and up to there they are the better form: us as digits / here, at 48 rows 6144 x 4096
// 12.0 / 13.5, 4096 x 4096 10.3 / 11.4, 24,576 x 4096 26.1 / 30.9, 4096 x 12288 17.5 / 19.3, LM head of 151,936 channels 101 / 120; at
// 64 rows 15.3 / 13.7, 11.0 / 11.8, 29.3 / 31.5, 19.1 / 19.6, 116 / 127.  Beyond, in two tiles of digits, no shape but one is: at 72 rows
// 14.6 / 13.8, 12.8 / 12.2, 29.4 / 32.0, 22.9 / 20.0, 145 / 132, and with the steps that follow them in the epilogues the batch of
// eight (72 rows) takes 4540 us as digits, 4090 here.  One line for all shapes: a pass keeps its rows in one form.
// Whatever the rows, a contraction whose digit sums could pass the 32 bits of the integer MMAs comes here: digits and weights go
// down to -128, so up to 2^17 - 1 products fit.
bool tc_wide_better(int64_t M, int64_t K) { return M > kDigitRows || K > 131071; }

int launch_tc_wide(const __nv_bfloat16* x, const int8_t* w, const float* dw, int64_t M, int64_t N, int64_t K, void* y, bool y_is_f32,
                   const __nv_bfloat16* residual, unsigned long long* keys, int32_t* error, bool pdl, cudaStream_t stream) {
  WideArgs a = {};
  a.dw = dw; a.y = y; a.res = residual; a.keys = keys; a.error = error; a.y_is_f32 = y_is_f32 ? 1 : 0;
  return launch_wide(kWideStore, x, w, M, N, K, a, pdl, stream);
}

int launch_tc_wide_swiglu(const __nv_bfloat16* x, const int8_t* w, const float* dw, int64_t M, int64_t F, int64_t K, __nv_bfloat16* act,
                          int32_t* error, bool pdl, cudaStream_t stream) {
  WideArgs a = {};
  a.dw = dw; a.y = act; a.error = error;
  return launch_wide(kWideSwiglu, x, w, M, 2 * F, K, a, pdl, stream);
}

bool tc_wide_rope_fits(int64_t M, int64_t N, int64_t K) {
  int device = 0;
  return allow_wide(&device) == QUASAR_OK && plan_wide(device, M, N, K, false, false).nsplit > 1;   // (a failure is the launch's to report)
}

int launch_tc_wide_qkv_rope(const __nv_bfloat16* x, const int8_t* w, const float* dw, int64_t M, int64_t K, const RopeArgs& rope, int32_t* error,
                            cudaStream_t stream) {
  WideArgs a = {};
  a.dw = dw; a.error = error; a.rope = rope;
  return launch_wide(kWideRope, x, w, M, (int64_t)(rope.Hq + 2 * rope.Hkv) * rope.D, K, a, true, stream);
}

}  // namespace quasar
