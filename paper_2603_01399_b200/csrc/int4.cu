// 4-bit group-wise weights (Section 6, "Ultra-low Bit Verification": weights of 4 bits or fewer, the first
// item of the paper's outlook).  The quantiser is Q of Section 3.2 Eq. 6 with the range [-7, 7] and one
// step size per output channel and group of 128 consecutive input channels; two codes per byte (the even
// input channel in the low nibble, two's complement).  The linear layer is Eq. 8 with one step per group:
//   Y[m][n] = sum_g delta[n][g] * sum_{k in g} X[m][k] * code[n][k]
// The weight stream is a quarter of the bf16 one (Section 3.4's M * bytes / BW term).
//
// Kernel: operand A is made in tensor memory from the codes (exact in bf16), operand B is the activation rows, one accumulator per
// group on the 5th-generation tensor cores:
//   TMA -> shared memory (packed codes) -> registers -> tensor memory (bf16)     X: global -> registers -> shared memory
// A code becomes a bf16 by placing (code + 8) under the exponent of 128 and subtracting 136 (exact), two codes per instruction.
// Shifting by 4 bits pairs code i with code i + 4, so the activations are staged in that order (0,4,1,5,2,6,3,7 within eight);
// the contraction index may be permuted freely as long as both operands agree.  A group's sums leave tensor memory under the
// next groups' MMAs and join the running fp32 sum with the group's step size.
// Tiles of 128 channels in turn on one CTA per SM, or, for matrices of few tiles, ranges of a tile's groups in the CTAs of a
// cluster, added through distributed shared memory in the order of the ranges.
// Every wait is bounded (2 s): on expiry the CTA stops waiting everywhere, releases its tensor memory and returns.
#include <algorithm>
#include <mutex>

#include "common.cuh"
#include "quant.cuh"
#include "tc_common.cuh"
#include "tc_linear.cuh"

namespace quasar {

namespace {

constexpr int kGroup = 128;
constexpr int kW4Threads = 576;    // TMA, MMA, 8 converter, 4 staging, 4 epilogue warps
constexpr int kW4Tile = 128;       // channels of a tile
constexpr int kW4Rows = 64;        // activation rows of a launch
constexpr int kW4Weights = kW4Tile * 128;   // bytes of a stage's weights: two groups
constexpr int kW4Pieces = 4;       // of operand A in tensor memory: a group each, 64 columns
constexpr int kW4Accs = 4;         // accumulators, 64 columns apart
constexpr size_t kW4Smem = 227 * 1024;
constexpr size_t kW4Fixed = 1024 + 512;     // alignment of the ring; barriers

// A thread takes eight consecutive values; the 16 lanes of a group share its maximum.  Four pieces per thread in flight.
constexpr int kQ4Pieces = 4;
__global__ void __launch_bounds__(256)
quantize_int4_kernel(const __nv_bfloat16* __restrict__ w, int64_t nvec, uint32_t* __restrict__ packed, float* __restrict__ delta) {
  const int64_t base = (int64_t)blockIdx.x * 256 * kQ4Pieces + threadIdx.x;
  uint4 raw[kQ4Pieces];
#pragma unroll
  for (int j = 0; j < kQ4Pieces; ++j) {
    const int64_t i = base + j * 256;
    raw[j] = i < nvec ? __ldg(reinterpret_cast<const uint4*>(w) + i) : make_uint4(0, 0, 0, 0);
  }
#pragma unroll
  for (int j = 0; j < kQ4Pieces; ++j) {
    const int64_t i = base + j * 256;
    float f[8], c[8];
    unpack_bf16x8(raw[j], f);
    AbsMax m;
#pragma unroll
    for (int e = 0; e < 8; ++e) m.take(f[e]);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
      m.num = fmaxf(m.num, __shfl_xor_sync(0xffffffffu, m.num, o));
      m.bits = max(m.bits, __shfl_xor_sync(0xffffffffu, m.bits, o));
    }
    const QuantStep st = quant_step(m.num == 0.f ? 1.0f : __fdiv_rn(m.num, 7.0f), m.has_nan());
    if (i >= nvec) continue;   // (whole groups: nvec is a multiple of 16)
    quantize8(f, st, 7, c);
    packed[i] = pack_nibbles8(c);
    if ((threadIdx.x & 15) == 0) delta[i >> 4] = st.delta;
  }
}

struct W4Args {
  const __nv_bfloat16* x;    // [M][K]
  const float* delta;        // [N][K/128]
  void* y;
  const __nv_bfloat16* res;
  int M, N, K, groups, stages_k;   // groups of the contraction, pairs of them
  int tiles, nsplit, ring, y_is_f32;
};

// eight packed codes -> four bf16 pairs (code i, code i + 4), i = 0..3
__device__ __forceinline__ void nib8_to_bf16(uint32_t w, uint32_t (&out)[4]) {
  const __nv_bfloat162 bias = __floats2bfloat162_rn(136.f, 136.f);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t v = ((w >> (4 * i)) & 0x000F000Fu) ^ 0x43084308u;     // bf16 128 + (code + 8): code + 8 is the nibble with its top bit turned
    const __nv_bfloat162 r = __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&v), bias);
    out[i] = *reinterpret_cast<const uint32_t*>(&r);
  }
}

using namespace tc;

// NB: 16s of activation rows
template <int NB>
__global__ void __launch_bounds__(kW4Threads, 1)
w4_kernel(const __grid_constant__ CUtensorMap map_w, const W4Args a) {
  constexpr int kRows = 16 * NB, kSub = kRows * 128;          // a slot of the rows: four sub-tiles of 64 of K
  constexpr int kStage = kW4Weights + 4 * kSub;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);   // the swizzle repeats every 1024 bytes
  const int S = a.ring;
  uint64_t* w_full = reinterpret_cast<uint64_t*>(smem + (size_t)S * kStage);   // a stage's codes have landed
  uint64_t* w_empty = w_full + S;            // and are in the converters' registers
  uint64_t* x_full = w_empty + S;            // its rows are staged
  uint64_t* x_empty = x_full + S;            // and have been multiplied
  uint64_t* a_full = x_empty + S;            // [pieces]
  uint64_t* a_empty = a_full + kW4Pieces;
  uint64_t* acc_full = a_empty + kW4Pieces;  // [accumulators]
  uint64_t* acc_empty = acc_full + kW4Accs;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + kW4Accs);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // (warp: uniform)
  const int split = (int)blockIdx.y, step = (int)gridDim.x;
  const int s0 = (int)((long long)split * a.stages_k / a.nsplit), s1 = (int)((long long)(split + 1) * a.stages_k / a.nsplit);

  if (threadIdx.x == 0) {
    *abort_flag = 0;
    for (int s = 0; s < S; ++s) {
      mbar_init(w_full + s, 1);
      mbar_init(w_empty + s, 8);
      mbar_init(x_full + s, 1);
      mbar_init(x_empty + s, 1);
    }
    for (int i = 0; i < kW4Pieces; ++i) {
      mbar_init(a_full + i, 4);
      mbar_init(a_empty + i, 1);
    }
    for (int i = 0; i < kW4Accs; ++i) {
      mbar_init(acc_full + i, 1);
      mbar_init(acc_empty + i, 4);
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
  const uint32_t tmem = *tmem_slot, tmem_a = tmem + (uint32_t)(kW4Accs * 64);

  if (warp == 0) {
    // ---- TMA producer ----
    const uint64_t policy = l2_evict_first_policy();
    int s = 0, issued = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < a.tiles && ok; t += step) {
      for (int k = s0; k < s1; ++k) {
        if (!(ok = mbar_wait(w_empty + s, ph ^ 1u, abort_flag, nullptr))) break;
        if (elect_one()) {
          mbar_expect_tx(w_full + s, kW4Weights);
          tma_load_2d_hint(smem + (size_t)s * kStage, &map_w, k * 128, t * kW4Tile, w_full + s, policy);
        }
        __syncwarp();
        ++issued;
        if (++s == S) { s = 0; ph ^= 1u; }
      }
    }
    if (!ok) {   // given up: what is in flight lands (bounded) before the CTA leaves
      for (int i = 0; i < min(S, issued); ++i) {
        if (--s < 0) { s = S - 1; ph ^= 1u; }
        const unsigned long long t0 = gtime_ns();
        while (!mbar_try(w_full + s, ph) && gtime_ns() - t0 < 100000ull) {}
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer ----
    const uint32_t id = idesc(1, 1, kW4Tile, kRows);
    int s = 0, piece = 0, acc = 0;
    uint32_t ph = 0, pph = 0, aph = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < a.tiles && ok; t += step) {
      for (int k = s0; k < s1 && ok; ++k) {
        if (!(ok = mbar_wait(x_full + s, ph, abort_flag, nullptr))) break;
        const uint64_t db = desc_sw128(smem + (size_t)s * kStage + kW4Weights);
#pragma unroll 1
        for (int j = 0; j < 2; ++j) {
          if (!(ok = mbar_wait(a_full + piece, pph, abort_flag, nullptr))) break;
          if (!(ok = mbar_wait(acc_empty + acc, aph ^ 1u, abort_flag, nullptr))) break;
          fence_after();
          if (elect_one()) {
            const uint32_t d = tmem + (uint32_t)(acc * 64), ta = tmem_a + (uint32_t)(piece * 64);
#pragma unroll
            for (int i = 0; i < 8; ++i)   // 16 of K: 8 columns of A, 32 bytes along the rows of B
              mma_f16_ts(d, ta + (uint32_t)(8 * i), db + (uint64_t)((uint32_t)((2 * j + (i >> 2)) * kSub) >> 4) + (uint64_t)(2 * (i & 3)), id, i > 0 ? 1u : 0u);
            commit(a_empty + piece);
            commit(acc_full + acc);
            if (j == 1) commit(x_empty + s);
          }
          __syncwarp();
          if (++piece == kW4Pieces) { piece = 0; pph ^= 1u; }
          if (++acc == kW4Accs) { acc = 0; aph ^= 1u; }
        }
        if (++s == S) { s = 0; ph ^= 1u; }
      }
    }
  } else if (warp < 10) {
    // ---- converters: four warps take group j of every stage; a thread one channel ----
    const int j = (warp - 2) >> 2, q = warp & 3, r = q * 32 + lane;
    const uint32_t lane_a = tmem_a + ((uint32_t)(q * 32) << 16);
    int s = 0, piece = j;
    uint32_t ph = 0, pph = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < a.tiles && ok; t += step) {
      for (int k = s0; k < s1; ++k) {
        if (!(ok = __all_sync(0xffffffffu, mbar_wait(w_full + s, ph, abort_flag, nullptr)))) break;
        const unsigned char* row = smem + (size_t)s * kStage + r * 128;
        uint32_t w[16];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const uint4 v = *reinterpret_cast<const uint4*>(row + (((j * 4 + c) ^ (r & 7)) << 4));
          w[4 * c] = v.x; w[4 * c + 1] = v.y; w[4 * c + 2] = v.z; w[4 * c + 3] = v.w;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(w_empty + s);
        if (!(ok = __all_sync(0xffffffffu, mbar_wait(a_empty + piece, pph ^ 1u, abort_flag, nullptr)))) break;
        fence_after();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t p[32];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            uint32_t o[4];
            nib8_to_bf16(w[8 * h + i], o);
            p[4 * i] = o[0]; p[4 * i + 1] = o[1]; p[4 * i + 2] = o[2]; p[4 * i + 3] = o[3];
          }
          tmem_st32(lane_a + (uint32_t)(piece * 64 + 32 * h), p);
        }
        tmem_st_wait();
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(a_full + piece);
        if ((piece += 2) >= kW4Pieces) { piece -= kW4Pieces; pph ^= 1u; }
        if (++s == S) { s = 0; ph ^= 1u; }
      }
    }
  } else if (warp < 14) {
    // ---- staging: a warp takes every fourth slot, 16 rows at a time, half a kilobyte a row ----
    int s = 0, turn = warp - 10;
    uint32_t ph = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < a.tiles && ok; t += step) {
      for (int k = s0; k < s1; ++k, turn = turn == 0 ? 3 : turn - 1) {
        if (turn != 0) {
          if (++s == S) { s = 0; ph ^= 1u; }
          continue;
        }
        unsigned char* slot = smem + (size_t)s * kStage + kW4Weights;
        // lane: eight elements, piece `lane` of the 32 of a row's slot
        const int kx = k * 256 + lane * 8, sub = lane >> 3, pc = lane & 7;
        bool waited = false;
#pragma unroll 1
        for (int r0 = 0; r0 < kRows; r0 += 16) {
          uint4 raw[16];
#pragma unroll
          for (int i = 0; i < 16; ++i)
            raw[i] = r0 + i < a.M && kx < a.K ? __ldg(reinterpret_cast<const uint4*>(a.x + (size_t)(r0 + i) * a.K + kx)) : make_uint4(0, 0, 0, 0);
          if (!waited) {
            if (!(ok = __all_sync(0xffffffffu, mbar_wait(x_empty + s, ph ^ 1u, abort_flag, nullptr)))) break;
            waited = true;
          }
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const int row = r0 + i;
            uint4 v;   // halves e0..e7 -> e0,e4,e1,e5,e2,e6,e3,e7
            v.x = __byte_perm(raw[i].x, raw[i].z, 0x5410);
            v.y = __byte_perm(raw[i].x, raw[i].z, 0x7632);
            v.z = __byte_perm(raw[i].y, raw[i].w, 0x5410);
            v.w = __byte_perm(raw[i].y, raw[i].w, 0x7632);
            *reinterpret_cast<uint4*>(slot + sub * kSub + row * 128 + ((pc ^ (row & 7)) << 4)) = v;
          }
        }
        if (!ok) break;
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(x_full + s);
        if (++s == S) { s = 0; ph ^= 1u; }
      }
    }
  } else {
    // ---- epilogue: a thread one channel ----
    const int q = warp & 3, r = q * 32 + lane;
    const uint32_t lane_d = tmem + ((uint32_t)(q * 32) << 16);
    const int g0 = 2 * s0, g1 = min(a.groups, 2 * s1), g_end = 2 * s1;
    float tot[kRows];
    int acc = 0;
    uint32_t aph = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < a.tiles && ok; t += step) {
      const int n = t * kW4Tile + r;
      const bool live = n < a.N;
      const float* dr = a.delta + (size_t)(live ? n : 0) * a.groups;
#pragma unroll
      for (int m = 0; m < kRows; ++m) tot[m] = 0.f;
      float d[4];   // step sizes, asked for four groups ahead
#pragma unroll
      for (int i = 0; i < 4; ++i) d[i] = g0 + i < g1 ? __ldg(dr + g0 + i) : 0.f;
      for (int g = g0; g < g_end && ok; g += 4) {
        float dn[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) dn[i] = g + 4 + i < g1 ? __ldg(dr + g + 4 + i) : 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (g + i >= g_end) break;
          if (!(ok = __all_sync(0xffffffffu, mbar_wait(acc_full + acc, aph, abort_flag, nullptr)))) break;
          fence_after();
          if (g + i < g1) {   // (the last stage of an odd number of groups: its second one is no group)
#pragma unroll
            for (int b = 0; b < NB; ++b) {
              uint32_t v[16];
              tmem_ld16(lane_d + (uint32_t)(acc * 64 + 16 * b), v);
#pragma unroll
              for (int e = 0; e < 16; ++e) tot[16 * b + e] = fmaf(__uint_as_float(v[e]), d[i], tot[16 * b + e]);
            }
          }
          fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(acc_empty + acc);
          if (++acc == kW4Accs) { acc = 0; aph ^= 1u; }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) d[i] = dn[i];
      }
      if (!ok) break;
      if (a.nsplit > 1) {   // the sums to shared memory, [row][channel]: every load has landed, every MMA read what it needs
        float* red = reinterpret_cast<float*>(smem);
#pragma unroll
        for (int m = 0; m < kRows; ++m) red[m * kW4Tile + r] = tot[m];
        break;              // (one tile a CTA)
      }
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        const int count = a.M - 16 * b;
        if (count <= 0) break;
        float f[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) f[e] = tot[16 * b + e];
        uint16_t res[16];
        if (a.res != nullptr) load_res16(res, a.res, live, (size_t)(16 * b), n, a.N, count);
        store16(f, live, (size_t)(16 * b), n, a.N, count, a.y, a.y_is_f32 != 0, a.res != nullptr, res);
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
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512u) : "memory");
  }
  if (a.nsplit == 1) return;
  // every CTA of the cluster finishes a share of the rows, four channels a lane
  const int per = (a.M + a.nsplit - 1) / a.nsplit, m_end = min(a.M, (split + 1) * per), n = (int)blockIdx.x * kW4Tile + lane * 4;
  const uint32_t red_addr = smem_u32(smem);
  const bool quad = (a.N & 3) == 0;   // (then four channels are inside or outside together, and aligned)
  for (int m = split * per + warp; m < m_end && *abort_flag == 0; m += kW4Threads / 32) {
    const size_t idx = (size_t)m * a.N + n;
    uint2 rr = make_uint2(0, 0);
    if (a.res != nullptr && quad && n < a.N) rr = *reinterpret_cast<const uint2*>(a.res + idx);
    uint4 p[8];
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (k < a.nsplit) p[k] = ld_cluster_v4(cluster_map(red_addr + (uint32_t)(m * kW4Tile + lane * 4) * 4, (uint32_t)k));
    float f[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (k >= a.nsplit) break;
      const uint32_t v[4] = {p[k].x, p[k].y, p[k].z, p[k].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) f[e] = k == 0 ? __uint_as_float(v[e]) : f[e] + __uint_as_float(v[e]);
    }
    auto rounded = [](float v) { return __bfloat162float(__float2bfloat16_rn(v)); };
    if (quad) {
      if (n >= a.N) continue;
      if (a.res != nullptr) {
        f[0] = rounded(f[0]) + __uint_as_float(rr.x << 16);
        f[1] = rounded(f[1]) + __uint_as_float(rr.x & 0xffff0000u);
        f[2] = rounded(f[2]) + __uint_as_float(rr.y << 16);
        f[3] = rounded(f[3]) + __uint_as_float(rr.y & 0xffff0000u);
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
      float o = f[e];
      if (a.res != nullptr) o = rounded(o) + __bfloat162float(a.res[idx + e]);
      if (a.y_is_f32) reinterpret_cast<float*>(a.y)[idx + e] = o;
      else reinterpret_cast<__nv_bfloat16*>(a.y)[idx + e] = __float2bfloat16_rn(o);
    }
  }
  __syncwarp();
  cluster_arrive();   // nobody's shared memory goes away while another CTA may read it
  cluster_wait();
}

// Clusters of s CTAs, one on an SM, that the device holds at once (they lie within a group of SMs, so long ones leave SMs unused).
template <int NB>
int w4_clusters(int s) {
  static std::mutex mu;
  static int seen[9] = {};
  std::lock_guard<std::mutex> lock(mu);
  int& n = seen[s];
  if (n == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1, (unsigned)s);
    cfg.blockDim = dim3(kW4Threads);
    cfg.dynamicSmemBytes = kW4Smem;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 1;
    attr.val.clusterDim.y = (unsigned)s;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, w4_kernel<NB>, &cfg) != cudaSuccess) cudaGetLastError();
    if (n < 1) n = 1;
  }
  return n;
}

template <int NB>
int launch_w4(W4Args a, const uint8_t* w, cudaStream_t stream) {
  static DeviceOnce once;
  int rc = allow_shared_memory(once, kW4Smem, true, {(const void*)w4_kernel<NB>});
  if (rc != QUASAR_OK) return rc;
  constexpr int kStage = kW4Weights + 4 * 16 * NB * 128;
  a.tiles = (a.N + kW4Tile - 1) / kW4Tile;
  a.groups = a.K / kGroup;
  a.stages_k = (a.groups + 1) / 2;
  a.ring = (int)((kW4Smem - kW4Fixed) / kStage);
  if (a.ring > 8) a.ring = 8;
  // Tiles in turn on the SMs, or a tile's ranges in a cluster, all of them at once: by the stages that the longest CTA takes.  The
  // exchange of sums costs about four of them.
  a.nsplit = 1;
  double best = (double)((a.tiles + 147) / 148) * (a.stages_k + 1);
  for (int s = 2; s <= 8 && s <= a.stages_k; ++s) {
    if (a.tiles > w4_clusters<NB>(s)) break;
    const double cost = (a.stages_k + s - 1) / s + 4.0;
    if (cost < best) { best = cost; a.nsplit = s; }
  }
  CUtensorMap map_w;
  rc = make_map_sw128(&map_w, w, (uint64_t)a.N, (uint64_t)a.K / 2, kW4Tile);
  if (rc != QUASAR_OK) return rc;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.nsplit > 1 ? a.tiles : std::min(a.tiles, 148)), (unsigned)a.nsplit);
  cfg.blockDim = dim3(kW4Threads);
  cfg.dynamicSmemBytes = (size_t)a.ring * kStage + kW4Fixed;
  cfg.stream = stream;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = 1;
  attr.val.clusterDim.y = (unsigned)a.nsplit;
  attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = a.nsplit > 1 ? 1 : 0;
  QUASAR_CUDA_CHECK(cudaLaunchKernelEx(&cfg, w4_kernel<NB>, map_w, a));
  count_launch();
  return QUASAR_OK;
}

}  // namespace

int launch_quantize_int4(const __nv_bfloat16* w, int64_t N, int64_t K, uint8_t* packed, float* delta, cudaStream_t stream) {
  if (N == 0) return QUASAR_OK;
  const int64_t nvec = N * (K / 8), per = 256 * kQ4Pieces;
  if ((nvec + per - 1) / per > 0x7fffffffLL) { set_error("quantize_int4: matrix too large"); return QUASAR_ERR_SHAPE; }
  quantize_int4_kernel<<<(unsigned)((nvec + per - 1) / per), 256, 0, stream>>>(w, nvec, reinterpret_cast<uint32_t*>(packed), delta);
  QUASAR_LAUNCH_CHECK();
  return QUASAR_OK;
}

size_t linear_w4_workspace_bytes(int64_t M, int64_t N, int64_t K) {
  (void)M; (void)N; (void)K;
  return 16;   // (nothing is kept there any more)
}

int launch_linear_w4(const __nv_bfloat16* x, const uint8_t* w, const float* delta, int64_t M, int64_t N, int64_t K, void* y,
                     bool y_is_f32, const __nv_bfloat16* residual, void* workspace, size_t workspace_bytes,
                     cudaStream_t stream) {
  if (M <= 0 || N <= 0 || K <= 0 || (K % kGroup) != 0 || N > 0x7fffffff || K > 0x7fffffff) {
    set_error("linear_w4: unsupported sizes M=%lld N=%lld K=%lld (K must be a multiple of %d)", (long long)M, (long long)N,
              (long long)K, kGroup);
    return QUASAR_ERR_SHAPE;
  }
  if (workspace_bytes < linear_w4_workspace_bytes(M, N, K)) {
    set_error("linear_w4: workspace of %zu bytes, need %zu", workspace_bytes, linear_w4_workspace_bytes(M, N, K));
    return QUASAR_ERR_CAPACITY;
  }
  (void)workspace;
  const size_t ybytes = y_is_f32 ? 4 : 2;
  const int64_t blocks = (M + kW4Rows - 1) / kW4Rows, rows = (M + blocks - 1) / blocks;
  for (int64_t m0 = 0; m0 < M; m0 += rows) {
    W4Args a;
    a.M = (int)((M - m0) < rows ? (M - m0) : rows);
    a.N = (int)N; a.K = (int)K;
    a.x = x + m0 * K; a.delta = delta;
    a.y = reinterpret_cast<unsigned char*>(y) + (size_t)m0 * N * ybytes;
    a.res = residual ? residual + m0 * N : nullptr;
    a.y_is_f32 = y_is_f32 ? 1 : 0;
    int rc;
    switch ((a.M + 15) / 16) {
      case 1: rc = launch_w4<1>(a, w, stream); break;
      case 2: rc = launch_w4<2>(a, w, stream); break;
      case 3: rc = launch_w4<3>(a, w, stream); break;
      default: rc = launch_w4<4>(a, w, stream); break;
    }
    if (rc != QUASAR_OK) return rc;
  }
  return QUASAR_OK;
}

}  // namespace quasar
