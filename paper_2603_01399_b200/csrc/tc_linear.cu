// Linear layers  Y = delta * (W X)  (Section 3.2 Eq. 8 / Section 3.3 Eq. 10) on the 5th-generation tensor cores, for
// int8 weights with bf16 activations, int8 weights with int8 activations, and bf16 weights.
//
// Mapping.  The weights are the 128-row operand A (one tensor-memory lane per output channel), the activation rows -
// padded to a multiple of 16 - operand B.  A CTA owns up to 128 output channels x up to 128 activation rows x one range
// of the contraction; a stage of its ring is 128 bytes of every weight row (TMA, 128-byte swizzle) and the activations
// that meet them.
//   * int8 x int8 (kind::i8, s32 sums) and bf16 x bf16 (kind::f16): both tiles go from TMA straight into the MMA.
//   * int8 x bf16: operand A is read from TENSOR memory.  Eight converter warps turn a stage's rows into bf16 in
//     registers and store them with tcgen05.st.  int8 -> bf16 is exact and takes eight instructions for four weights:
//     with m = w & 127 and s = w & 128, the bytes m and s under the high byte 0x43 read 128 + m and 128 (or 256) as
//     bf16, and one packed subtraction leaves w.  The activations enter as they are: no fp16 copy of them, no row
//     scales, no kernel in front of this one.  (The form before this one converted to fp16 with four warps a CTA: each
//     stage waited for one warp's chain of load, convert, store, publish - 2.9 TB/s of weights at 72 rows.)
//
// Work split.  About two CTAs fit an SM, and a launch has to give every SM the same number of weight bytes: the tile
// height (a multiple of 8 channels) and the number of k-ranges are chosen together for that (plan_tc).  The k-ranges of
// a tile form a thread-block cluster; their sums meet through distributed shared memory, every CTA of the cluster
// finishing a share of the rows, in the order of the ranges (results repeat bit for bit): no partial sums in global
// memory, no second kernel, no counters.
//
// Every wait is bounded (2 s): on expiry the CTA raises an error word, stops waiting everywhere, releases its tensor
// memory and returns.
#include <math.h>

#include <algorithm>
#include <mutex>

#include "tc_common.cuh"
#include "tc_linear.cuh"

namespace quasar {

namespace tc {

static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

int make_map_sw128(CUtensorMap* map, const void* base, uint64_t rows, uint64_t row_bytes, uint32_t box_rows) {
  auto fn = encode_fn();
  if (fn == nullptr) {
    set_error("cuTensorMapEncodeTiled is not available from this driver");
    return QUASAR_ERR_CUDA;
  }
  const cuuint64_t dims[2] = {row_bytes, rows};
  const cuuint64_t strides[1] = {row_bytes};
  const cuuint32_t box[2] = {128u, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_error("cuTensorMapEncodeTiled failed (%d) for %llu x %llu bytes", (int)r, (unsigned long long)rows,
              (unsigned long long)row_bytes);
    return QUASAR_ERR_CUDA;
  }
  return QUASAR_OK;
}

}  // namespace tc

namespace {

using namespace tc;

// activations of the int8 forms: three digit rows (weight-only form) or one row of int8 codes (W8A8) per token
enum TcKind { kDigits = 0, kBf16 = 1, kCodes = 2 };

constexpr int kTileN = 128;              // channels of an MMA (operand A rows)
constexpr int kAStage = kTileN * 128;    // bytes of a stage's weights
constexpr int kThreadsTc = 320;          // TMA warp, MMA warp, eight converter / epilogue warps
constexpr int kTmemCols = 256;           // two CTAs share an SM's 512 columns: one accumulator column per row of operand B
constexpr size_t kMaxSmem = 227 * 1024;
constexpr size_t kSmemSlack = 1024 + 256;       // alignment of the ring, barriers

struct TcArgs {
  const float* dx;             // [M] step sizes of the int8 activations
  const float* dw;             // [N] step sizes of the int8 weights
  void* y;                     // [M][N] bf16 or fp32, or nullptr: only the arg-max is wanted
  const __nv_bfloat16* res;    // [M][N] or nullptr
  int32_t* acc_out;            // [M][N] raw int32 sums (int8 activations) or nullptr
  unsigned long long* keys;    // [M] running arg-max keys of the rows (see argmax_key), or nullptr
  int32_t* error;              // device status word or nullptr
  int M, N, kblocks;
  int chan;                    // channels of a tile
  int rows, brows;             // activation rows of a row tile; rows of operand B (three per activation row for digits), padded to 16
  int row_tiles, nsplit, stages;
  int y_is_f32;
  int early_weights;           // the weights may be asked for before the kernel in front has finished
};

template <int KIND>
__device__ __forceinline__ float finish(uint32_t bits, float dx, float dw) {
  if (KIND == kCodes) return __fmul_rn((float)(int)bits, __fmul_rn(dw, dx));   // Eq. 10
  if (KIND == kDigits) return (__uint_as_float(bits) * dx) * dw;               // dx: the power of two of the row
  return __uint_as_float(bits);
}

// one row, four channels from n on; `best`: the row's arg-max key so far
template <int KIND>
__device__ __forceinline__ void store4(const TcArgs& a, const uint32_t (&v)[4], int m, int n, float dx, unsigned long long& best) {
  const size_t idx = (size_t)m * a.N + n;
  const bool vec = (a.N & 3) == 0;   // then n + 3 < N, and every address below is aligned
  float f[4];
  if (vec) {
    float4 dw = make_float4(1.f, 1.f, 1.f, 1.f);
    if (KIND != kBf16) dw = __ldg(reinterpret_cast<const float4*>(a.dw + n));
    f[0] = finish<KIND>(v[0], dx, dw.x); f[1] = finish<KIND>(v[1], dx, dw.y);
    f[2] = finish<KIND>(v[2], dx, dw.z); f[3] = finish<KIND>(v[3], dx, dw.w);
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e) f[e] = finish<KIND>(v[e], dx, (KIND != kBf16 && n + e < a.N) ? a.dw[n + e] : 1.f);
  }
  if (a.keys != nullptr) {
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (n + e < a.N && f[e] == f[e]) {   // NaNs never enter
        const unsigned long long k = argmax_key(f[e], n + e);
        best = k > best ? k : best;
      }
  }
  if (a.y == nullptr) return;
  if (vec) {
    if (KIND == kCodes && a.acc_out != nullptr)
      *reinterpret_cast<int4*>(a.acc_out + idx) = make_int4((int)v[0], (int)v[1], (int)v[2], (int)v[3]);
    if (a.res != nullptr) {
      const uint2 r = *reinterpret_cast<const uint2*>(a.res + idx);
      const uint32_t rr[2] = {r.x, r.y};
#pragma unroll
      for (int e = 0; e < 4; ++e)
        f[e] = __bfloat162float(__float2bfloat16_rn(f[e])) +
               __uint_as_float((e & 1) ? (rr[e >> 1] & 0xffff0000u) : (rr[e >> 1] << 16));
    }
    if (a.y_is_f32) {
      *reinterpret_cast<float4*>(reinterpret_cast<float*>(a.y) + idx) = make_float4(f[0], f[1], f[2], f[3]);
    } else {
      const __nv_bfloat162 lo = __floats2bfloat162_rn(f[0], f[1]), hi = __floats2bfloat162_rn(f[2], f[3]);
      *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(a.y) + idx) =
          make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
    }
    return;
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    if (n + e >= a.N) break;
    if (KIND == kCodes && a.acc_out != nullptr) a.acc_out[idx + e] = (int)v[e];
    float o = f[e];
    if (a.res != nullptr) o = __bfloat162float(__float2bfloat16_rn(o)) + __bfloat162float(a.res[idx + e]);
    if (a.y_is_f32) reinterpret_cast<float*>(a.y)[idx + e] = o;
    else reinterpret_cast<__nv_bfloat16*>(a.y)[idx + e] = __float2bfloat16_rn(o);
  }
}

template <int KIND>
__global__ void __launch_bounds__(kThreadsTc, 2)
tc_linear_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_x, const TcArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);   // the swizzle repeats every 1024 bytes
  const int b_bytes = a.brows * 128;
  const int stage_bytes = kAStage + b_bytes;
  const int S = a.stages;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)S * stage_bytes);   // the stage's bytes have landed
  uint64_t* empty = full + S;             // its MMAs have read it
  uint64_t* accum_done = empty + S;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(accum_done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row_tile = (int)blockIdx.x % a.row_tiles, tile = (int)blockIdx.x / a.row_tiles;
  const int split = blockIdx.y;
  const int n0 = tile * a.chan, m0 = row_tile * a.rows;
  const int kb0 = (int)((long long)split * a.kblocks / a.nsplit), kb1 = (int)((long long)(split + 1) * a.kblocks / a.nsplit);
  const uint32_t tx = (uint32_t)(a.chan * 128 + b_bytes);

  if (threadIdx.x == 0) {
    *abort_flag = 0;
    for (int s = 0; s < S; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);
    }
    mbar_init(accum_done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)),
                 "r"((uint32_t)kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // Only now may the kernel behind this one start: a tcgen05 kernel further down the stream waits for this one while it
  // holds tensor memory, so every CTA here must have its own first.
  if (threadIdx.x == 0) pdl_trigger();

  if (warp == 0) {
    if (lane == 0) {   // ---- TMA producer ----
      const uint64_t policy = l2_evict_first_policy();
      const int ahead = min(S, kb1 - kb0);
      if (a.early_weights) {   // the weights of the first stages do not depend on the kernel in front
        for (int i = 0; i < ahead; ++i) {
          mbar_expect_tx(full + i, tx);
          tma_load_2d_hint(smem + (size_t)i * stage_bytes, &map_w, (kb0 + i) * 128, n0, full + i, policy);
        }
      }
      pdl_wait();
      int s = 0;
      uint32_t ph = 0;
      int kb = kb0;
      for (; kb < kb1; ++kb) {
        unsigned char* at = smem + (size_t)s * stage_bytes;
        if (!(a.early_weights && kb - kb0 < ahead)) {
          if (!mbar_wait(empty + s, ph ^ 1u, abort_flag, a.error)) break;
          mbar_expect_tx(full + s, tx);
          tma_load_2d_hint(at, &map_w, kb * 128, n0, full + s, policy);
        }
        tma_load_2d(at + kAStage, &map_x, kb * 128, KIND == kDigits ? 3 * m0 : m0, full + s);
        if (++s == S) { s = 0; ph ^= 1u; }
      }
      if (kb < kb1) {   // given up: what is in flight lands (bounded) before the CTA leaves
        for (int i = 0; i < min(S, kb - kb0); ++i) {
          if (--s < 0) { s = S - 1; ph ^= 1u; }
          const unsigned long long t0 = gtime_ns();
          while (!mbar_try(full + s, ph) && gtime_ns() - t0 < 100000ull) {}
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {   // ---- MMA issuer ----
      const uint32_t id = idesc(KIND == kBf16 ? 1 : 2, 1, kTileN, a.brows);
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!(ok = mbar_wait(full + s, ph, abort_flag, a.error))) break;
        fence_after();
        const unsigned char* at = smem + (size_t)s * stage_bytes;
        const uint64_t da = desc_sw128(at), db = desc_sw128(at + kAStage);
#pragma unroll
        for (int j = 0; j < 4; ++j) {   // 32 bytes along the rows of both
          const uint32_t acc = (kb > kb0 || j > 0) ? 1u : 0u;
          if (KIND == kBf16) mma_f16_ss(tmem_base, da + (uint64_t)(j * 2), db + (uint64_t)(j * 2), id, acc);
          else mma_i8_ss(tmem_base, da + (uint64_t)(j * 2), db + (uint64_t)(j * 2), id, acc);
        }
        commit(empty + s);
        if (++s == S) { s = 0; ph ^= 1u; }
      }
      if (ok) commit(accum_done);
    }
  } else {
    // ---- warps 2..9: the sums to shared memory, [row][channel] (the ring is idle then: every load has landed and every MMA
    //      has read its stage).  A warp may touch the tensor-memory lanes 32 (warp % 4) .. + 31; two warps share them. ----
    const int q = warp & 3, half = (warp - 2) >> 2;
    const int r = q * 32 + lane;
    const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
    if (__all_sync(0xffffffffu, mbar_wait(accum_done, 0, abort_flag, a.error))) {
      fence_after();
      uint32_t* red = reinterpret_cast<uint32_t*>(smem);
      for (int r0 = half * 16; r0 < a.rows; r0 += 32) {   // 16 activation rows at a time
        uint32_t v[16];
        if (KIND == kDigits) {
          uint32_t d[48];
#pragma unroll
          for (int c = 0; c < 3; ++c) tmem_ld16(lane_addr + (uint32_t)(3 * r0 + 16 * c), *reinterpret_cast<uint32_t(*)[16]>(d + 16 * c));
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const long long total = ((long long)(int)d[3 * j + 2] << 16) + ((long long)(int)d[3 * j + 1] << 8) + (long long)(int)d[3 * j];
            v[j] = __float_as_uint((float)total);
          }
        } else {
          tmem_ld16(lane_addr + (uint32_t)r0, v);
        }
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (r0 + j < a.rows) red[(r0 + j) * kTileN + r] = v[j];
      }
    }
  }
  __syncwarp();
  fence_before();
  if (a.nsplit > 1) {
    cluster_arrive();
    cluster_wait();
  } else {
    __syncthreads();
  }
  if (warp == 1) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"((uint32_t)kTmemCols) : "memory");
  }
  pdl_wait();   // every thread: the residual below may come from the kernel in front
  if (*abort_flag == 0) {
    // this CTA's share of the tile's rows, 32 threads a row, four channels a thread; the ranges in ascending order
    const int rows = min(a.rows, a.M - m0);
    const int per = (rows + a.nsplit - 1) / a.nsplit;
    const int r_begin = split * per, r_end = min(rows, r_begin + per);
    const int n = n0 + lane * 4;
    const bool live = lane * 4 < a.chan && n < a.N;
    const uint32_t red_addr = smem_u32(smem);
    for (int m = r_begin + warp; m < r_end; m += kThreadsTc / 32) {
      unsigned long long best = 0;
      if (live) {
      const uint32_t off = (uint32_t)(m * kTileN + lane * 4) * 4;
      uint32_t sum[4];
      if (a.nsplit == 1) {
        const uint4 p = *reinterpret_cast<const uint4*>(smem + off);
        sum[0] = p.x; sum[1] = p.y; sum[2] = p.z; sum[3] = p.w;
      } else {
        uint4 p[8];
#pragma unroll
        for (int k = 0; k < 8; ++k)
          if (k < a.nsplit) p[k] = ld_cluster_v4(cluster_map(red_addr + off, (uint32_t)k));
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          if (k >= a.nsplit) break;
          const uint32_t w[4] = {p[k].x, p[k].y, p[k].z, p[k].w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            if (k == 0) sum[e] = w[e];
            else if (KIND == kCodes) sum[e] += w[e];
            else sum[e] = __float_as_uint(__uint_as_float(sum[e]) + __uint_as_float(w[e]));
          }
        }
      }
      store4<KIND>(a, sum, m0 + m, n, KIND != kBf16 ? a.dx[m0 + m] : 1.f, best);
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
  if (a.nsplit > 1) {   // nobody's shared memory goes away while another CTA may read it
    cluster_arrive();
    cluster_wait();
  }
}

struct TcPlan {
  int chan, tiles, nsplit, row_tiles, rows, brows, kblocks, stages;
};

// Clusters of s CTAs that the device holds at once with one CTA on each SM (they lie within a group of SMs, so long ones
// leave SMs unused).
int max_clusters(const void* kernel, int s) {
  static std::mutex mu;
  static int seen[9] = {};
  std::lock_guard<std::mutex> lock(mu);
  if (seen[s] == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1, (unsigned)s);
    cfg.blockDim = dim3(kThreadsTc);
    cfg.dynamicSmemBytes = kMaxSmem;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 1;
    attr.val.clusterDim.y = (unsigned)s;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) cudaGetLastError();
    seen[s] = n < 1 ? 1 : n;
  }
  return seen[s];
}

// Tile height and k-ranges, by an estimate of the time in us: waves of CTAs, each a fixed cost and the largest of what its
// stages' latency, the SM's intake (about 95 KB per us) and the memory (6.2 MB of weights per us for all) ask for, with a
// cost for every range that joins the exchange of sums.  Measured at 6 rows: 4096 x 4096 in 4 ranges 9.1 us, in 8 9.3, in 2
// 10.6; 4096 x 12288 in 8 ranges 15.4 us, in 4 16.6, in 2 21.2; 6144 x 4096 in 4 ranges 10.5 us, in 6 (more clusters
// than fit at once) 14.2.
TcPlan plan_tc(int64_t M, int64_t N, int64_t K, int kind, const void* kernel) {
  TcPlan p;
  const int most = kind == kDigits ? 80 : 128;
  p.row_tiles = (int)((M + most - 1) / most);
  p.rows = (int)((M + p.row_tiles - 1) / p.row_tiles);
  p.brows = (p.rows * (kind == kDigits ? 3 : 1) + 15) / 16 * 16;
  p.kblocks = (int)(((kind == kBf16 ? 2 * K : K) + 127) / 128);
  const int stage = kAStage + p.brows * 128;
  // two CTAs on an SM as long as that leaves each three stages; wider blocks do better with one CTA and its deeper ring
  // (4096 x 4096 at 72 rows: 11.3 us with one, 12.9 with two)
  int per_sm = (int)((kMaxSmem / 2 - 1024 - kSmemSlack) / stage) >= 3 ? 2 : 1;
  const size_t room = per_sm == 2 ? kMaxSmem / 2 - 1024 : kMaxSmem;
  const int st = (int)((room - kSmemSlack) / stage);
  p.stages = st > 8 ? 8 : st;
  double best = 0;
  p.nsplit = 0;
  for (int s = 1; s <= 8 && s <= p.kblocks; ++s) {
    // (two CTAs of a cluster can share an SM)
    const long long fit = per_sm == 1 ? max_clusters(kernel, s) : std::max(2 * max_clusters(kernel, s), max_clusters(kernel, (s + 1) / 2));
    for (int c = 128; c >= 64; c -= 8) {
      const long long tiles = (N + c - 1) / c;
      const long long clusters = tiles * p.row_tiles;
      const long long waves = (clusters + fit - 1) / fit;
      const double ctas = (double)(clusters < fit ? clusters : fit) * s;
      const double kbs = (double)((p.kblocks + s - 1) / s);
      const double lat = 0.22 * kbs;
      const double sm = kbs * (ctas > 148 ? ctas / 148 : 1.0) * (c * 128.0 + p.brows * 128.0) / 95e3;
      const double mem = kbs * ctas * c * 128.0 / 6.2e6 / p.row_tiles;
      const double cost = (double)waves * (2.0 + sqrt(lat * lat + sm * sm + mem * mem)) + 0.15 * s;
      if (p.nsplit == 0 || cost < best * 0.99) {
        best = cost;
        p.nsplit = s;
        p.chan = c;
        p.tiles = (int)tiles;
      }
    }
  }
  return p;
}

template <int KIND>
int launch_kind(const CUtensorMap& map_w, const CUtensorMap& map_x, const TcArgs& a, const TcPlan& p, bool pdl, cudaStream_t stream) {
  const size_t smem = (size_t)p.stages * (kAStage + p.brows * 128) + kSmemSlack;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(p.tiles * p.row_tiles), (unsigned)p.nsplit);
  cfg.blockDim = dim3(kThreadsTc);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  int na = 0;
  if (p.nsplit > 1) {
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = 1;
    attr[na].val.clusterDim.y = (unsigned)p.nsplit;
    attr[na].val.clusterDim.z = 1;
    ++na;
  }
  if (pdl) {
    attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[na].val.programmaticStreamSerializationAllowed = 1;
    ++na;
  }
  cfg.attrs = attr;
  cfg.numAttrs = (unsigned)na;
  QUASAR_CUDA_CHECK(cudaLaunchKernelEx(&cfg, tc_linear_kernel<KIND>, map_w, map_x, a));
  count_launch();
  return QUASAR_OK;
}

int launch_any(int kind, const void* x, const float* dx, const void* w, const float* dw, int64_t M, int64_t N, int64_t K, void* y,
               bool y_is_f32, const __nv_bfloat16* residual, int32_t* acc_out, unsigned long long* keys, int32_t* error, bool pdl, cudaStream_t stream) {
  const void* kernel = kind == kDigits ? (const void*)tc_linear_kernel<kDigits>
                                       : (kind == kBf16 ? (const void*)tc_linear_kernel<kBf16> : (const void*)tc_linear_kernel<kCodes>);
  {
    static bool configured[3] = {false, false, false};
    if (!configured[kind]) {
      QUASAR_CUDA_CHECK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem));
      QUASAR_CUDA_CHECK(cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
      configured[kind] = true;
    }
  }
  const TcPlan p = plan_tc(M, N, K, kind, kernel);
  CUtensorMap map_w, map_x;
  int rc = make_map_sw128(&map_w, w, (uint64_t)N, (uint64_t)K * (kind == kBf16 ? 2 : 1), (uint32_t)p.chan);
  if (rc != QUASAR_OK) return rc;
  rc = make_map_sw128(&map_x, x, (uint64_t)M * (kind == kDigits ? 3 : 1), (uint64_t)K * (kind == kBf16 ? 2 : 1), (uint32_t)p.brows);
  if (rc != QUASAR_OK) return rc;
  TcArgs a;
  a.dx = dx; a.dw = dw; a.y = y; a.res = residual; a.acc_out = acc_out; a.keys = keys; a.error = error;
  a.M = (int)M; a.N = (int)N; a.kblocks = p.kblocks; a.chan = p.chan; a.rows = p.rows; a.brows = p.brows;
  a.row_tiles = p.row_tiles; a.nsplit = p.nsplit; a.stages = p.stages; a.y_is_f32 = y_is_f32 ? 1 : 0;
  a.early_weights = pdl ? 1 : 0;
  switch (kind) {
    case kDigits: return launch_kind<kDigits>(map_w, map_x, a, p, pdl, stream);
    case kBf16: return launch_kind<kBf16>(map_w, map_x, a, p, pdl, stream);
    default: return launch_kind<kCodes>(map_w, map_x, a, p, pdl, stream);
  }
}

}  // namespace

bool tc_linear_usable(int64_t M, int64_t N, int64_t K) {
  return M >= 1 && N >= 1 && K >= 16 && K % 16 == 0 && M <= (1 << 20) && N <= (1 << 30) && K <= (1 << 28);
}

// ---- activations as digit rows: row m of x becomes the rows 3 m .. 3 m + 2 of xd -------------------------------------
__global__ void __launch_bounds__(kDigitThreads)
digit_rows3_kernel(const __nv_bfloat16* __restrict__ x, int K, int8_t* __restrict__ xd, float* __restrict__ row_scale) {
  __shared__ float s_max[kDigitThreads / 32];
  pdl_trigger();
  const int64_t m = blockIdx.x;
  const uint4* row = reinterpret_cast<const uint4*>(x + m * K);
  float amax = 0.f;
  for (int i = threadIdx.x; i < K / 8; i += kDigitThreads) {
    const uint4 v = row[i];
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) amax = fmaxf(amax, fmaxf(fabsf(__uint_as_float(w[e] << 16)), fabsf(__uint_as_float(w[e] & 0xffff0000u))));
  }
  amax = digit_block_max(amax, s_max);
  float up, down;
  digit_scale(amax, up, down);
  if (threadIdx.x == 0) row_scale[m] = down;
  int8_t* d = xd + 3 * m * K;
  for (int i = threadIdx.x; i < K / 8; i += kDigitThreads) {
    const uint4 v = row[i];
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    float f[8];
#pragma unroll
    for (int e = 0; e < 4; ++e) { f[2 * e] = __uint_as_float(w[e] << 16); f[2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u); }
    write_digits8(f, up, d, K, i * 8);
  }
}

int launch_digit_rows3(const __nv_bfloat16* x, int64_t M, int64_t K, int8_t* xd, float* row_scale, cudaStream_t stream) {
  digit_rows3_kernel<<<(unsigned)M, kDigitThreads, 0, stream>>>(x, (int)K, xd, row_scale);
  QUASAR_LAUNCH_CHECK();
  return QUASAR_OK;
}

int launch_tc_linear_bf16(const __nv_bfloat16* x, const __nv_bfloat16* w, int64_t M, int64_t N, int64_t K, void* y, bool y_is_f32,
                          const __nv_bfloat16* residual, unsigned long long* keys, int32_t* error, bool pdl, cudaStream_t stream) {
  return launch_any(kBf16, x, nullptr, w, nullptr, M, N, K, y, y_is_f32, residual, nullptr, keys, error, pdl, stream);
}

int launch_tc_linear_digits(const int8_t* xd, const float* row_scale, const int8_t* w, const float* dw, int64_t M, int64_t N,
                            int64_t K, void* y, bool y_is_f32, const __nv_bfloat16* residual, unsigned long long* keys,
                            int32_t* error, bool pdl, cudaStream_t stream) {
  return launch_any(kDigits, xd, row_scale, w, dw, M, N, K, y, y_is_f32, residual, nullptr, keys, error, pdl, stream);
}

int launch_tc_linear_w8a8(const int8_t* xq, const float* dx, const int8_t* w, const float* dw, int64_t M, int64_t N, int64_t K,
                          void* y, bool y_is_f32, const __nv_bfloat16* residual, int32_t* acc_out, unsigned long long* keys,
                          int32_t* error, bool pdl, cudaStream_t stream) {
  return launch_any(kCodes, xq, dx, w, dw, M, N, K, y, y_is_f32, residual, acc_out, keys, error, pdl, stream);
}

}  // namespace quasar
