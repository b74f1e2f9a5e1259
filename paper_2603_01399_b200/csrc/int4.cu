// 4-bit group-wise weights (Section 6, "Ultra-low Bit Verification": weights of 4 bits or fewer, the first
// item of the paper's outlook).  The quantiser is Q of Section 3.2 Eq. 6 with the range [-7, 7] and one
// step size per output channel and group of 128 consecutive input channels; two codes per byte (the even
// input channel in the low nibble, two's complement).  The linear layer is Eq. 8 with one step per group:
//   Y[m][n] = sum_g delta[n][g] * sum_{k in g} X[m][k] * code[n][k]
// The weight stream is a quarter of the bf16 one (Section 3.4's M * bytes / BW term).
//
// Kernel: a CTA of 8 warps owns 128 output channels x a range of groups, a warp 16 channels.  The weights of up to four
// groups are asked for at once, 16 bytes a row and group and lane, before the activations of the chunk are staged in shared
// memory; the groups then run without a barrier between them.  A code becomes a bf16 by placing (code + 8) under the
// exponent of 128 and subtracting 136 (exact), two codes per instruction.  Shifting by 4 bits pairs code i with code
// i + 4, so the activations are staged in that order (0,4,1,5,2,6,3,7 within eight) and the operands of mma.m16n8k16 line
// up without further moves; the contraction index may be permuted freely as long as both operands agree.  fp32
// accumulation per group, folded into the running sum with the group's step size.  The ranges of a channel block form a
// cluster and add their sums through distributed shared memory in the order of the ranges.  What bounds it (16 x 4096 x 12288,
// 17.9 us): waiting for weights - a range of twelve groups asks for four at a time, one after the other; a scheduler has 3.5
// warps and issues in 36 % of its cycles, the integer pipes are 29 % busy, the tensor pipe 14 %, the memory 17 %.
#include <algorithm>

#include "common.cuh"
#include "quant.cuh"
#include "tc_common.cuh"

namespace quasar {

namespace {

constexpr int kGroup = 128;
constexpr int kW4Threads = 256;
constexpr int kW4BlockN = 128;
constexpr int kW4Rows = 64;        // activation rows of a launch
constexpr int kW4Ahead = 4;        // groups whose weights a lane holds at a time

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
  const uint8_t* w;          // [N][K/2]
  const float* delta;        // [N][K/128]
  void* y;
  const __nv_bfloat16* res;
  int M, N, K, nsplit, chunk, y_is_f32;   // chunk: groups whose activations are staged at a time
};

__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

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

__device__ __forceinline__ uint4 ldg_once(const void* p) {
  uint4 r;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p));
  return r;
}

// where piece p (16 bytes: eight elements of the group) of row `row` lies among a row's 16 pieces of a group: lane t reads its
// pieces 4 t .. 4 t + 3 one after the other, and no two of eight neighbouring lanes meet in a bank
__device__ __forceinline__ int piece_at(int p, int row) { return (((p & 3) << 2) | (p >> 2)) ^ ((row & 1) << 2); }

template <int NT>
__global__ void __launch_bounds__(kW4Threads) w4_gemm_kernel(W4Args a) {
  extern __shared__ __align__(16) unsigned char smem[];
  uint4* xs = reinterpret_cast<uint4*>(smem);   // [group of the chunk][NT * 8 rows][16 pieces]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int n0 = blockIdx.x * kW4BlockN + warp * 16;
  const int ngroups = a.K / kGroup;
  const int g_begin = (int)((int64_t)blockIdx.y * ngroups / a.nsplit), g_end = (int)((int64_t)(blockIdx.y + 1) * ngroups / a.nsplit);
  const int r0 = min(n0 + g, a.N - 1), r1 = min(n0 + g + 8, a.N - 1);
  const uint8_t* wrow0 = a.w + (size_t)r0 * (a.K / 2) + t * 16;
  const uint8_t* wrow1 = a.w + (size_t)r1 * (a.K / 2) + t * 16;
  const float* drow0 = a.delta + (size_t)r0 * ngroups;
  const float* drow1 = a.delta + (size_t)r1 * ngroups;
  float tot[NT][4];
#pragma unroll
  for (int i = 0; i < NT; ++i) tot[i][0] = tot[i][1] = tot[i][2] = tot[i][3] = 0.f;

  for (int c0 = g_begin; c0 < g_end; c0 += a.chunk) {
    const int cn = min(a.chunk, g_end - c0);
    uint4 wa[kW4Ahead], wb[kW4Ahead];
    float d0[kW4Ahead], d1[kW4Ahead];
    auto fetch = [&](int from) {
#pragma unroll
      for (int u = 0; u < kW4Ahead; ++u) {
        if (from + u < cn) {
          wa[u] = ldg_once(wrow0 + (size_t)(c0 + from + u) * 64);
          wb[u] = ldg_once(wrow1 + (size_t)(c0 + from + u) * 64);
          d0[u] = __ldg(drow0 + c0 + from + u);
          d1[u] = __ldg(drow1 + c0 + from + u);
        }
      }
    };
    fetch(0);
    if (c0 > g_begin) __syncthreads();   // the chunk before has been read
    // staged four pieces a thread at a time, all of them in flight at once
    const int pieces = NT * 8 * 16 * cn;
    for (int i0 = threadIdx.x; i0 < pieces; i0 += 4 * kW4Threads) {
      uint4 raw[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int i = i0 + j * kW4Threads;
        const int row = (i >> 4) % (NT * 8), gi = (i >> 4) / (NT * 8), pc = i & 15;
        raw[j] = (i < pieces && row < a.M) ? *reinterpret_cast<const uint4*>(a.x + (size_t)row * a.K + (size_t)(c0 + gi) * kGroup + pc * 8)
                                           : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int i = i0 + j * kW4Threads;
        if (i >= pieces) break;
        const int row = (i >> 4) % (NT * 8), gi = (i >> 4) / (NT * 8), pc = i & 15;
        uint4 v;   // halves e0..e7 -> e0,e4,e1,e5,e2,e6,e3,e7
        v.x = __byte_perm(raw[j].x, raw[j].z, 0x5410);
        v.y = __byte_perm(raw[j].x, raw[j].z, 0x7632);
        v.z = __byte_perm(raw[j].y, raw[j].w, 0x5410);
        v.w = __byte_perm(raw[j].y, raw[j].w, 0x7632);
        xs[(gi * NT * 8 + row) * 16 + piece_at(pc, row)] = v;
      }
    }
    __syncthreads();
    for (int from = 0; from < cn; from += kW4Ahead) {
      if (from > 0) fetch(from);
#pragma unroll
      for (int u = 0; u < kW4Ahead; ++u) {
        if (from + u >= cn) break;
        float acc[NT][4];
#pragma unroll
        for (int i = 0; i < NT; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;
        const uint32_t pa[4] = {wa[u].x, wa[u].y, wa[u].z, wa[u].w}, pb[4] = {wb[u].x, wb[u].y, wb[u].z, wb[u].w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {   // eight codes of each row: two MMAs
          uint32_t A[4], B[4];
          nib8_to_bf16(pa[c], A);
          nib8_to_bf16(pb[c], B);
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) {
            const int row = nt * 8 + g;
            const uint4 x = xs[((from + u) * NT * 8 + row) * 16 + piece_at(t * 4 + c, row)];
            mma_bf16(acc[nt], A[0], B[0], A[1], B[1], x.x, x.y);
            mma_bf16(acc[nt], A[2], B[2], A[3], B[3], x.z, x.w);
          }
        }
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          tot[nt][0] = fmaf(acc[nt][0], d0[u], tot[nt][0]);
          tot[nt][1] = fmaf(acc[nt][1], d0[u], tot[nt][1]);
          tot[nt][2] = fmaf(acc[nt][2], d1[u], tot[nt][2]);
          tot[nt][3] = fmaf(acc[nt][3], d1[u], tot[nt][3]);
        }
      }
    }
  }
  // the sums to shared memory, [row][channel of the block]; every CTA of the cluster finishes a share of the rows
  __syncthreads();
  float* red = reinterpret_cast<float*>(smem);
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
    for (int e = 0; e < 4; ++e) red[(nt * 8 + 2 * t + (e & 1)) * kW4BlockN + warp * 16 + g + (e >> 1) * 8] = tot[nt][e];
  }
  if (a.nsplit > 1) {
    tc::cluster_arrive();
    tc::cluster_wait();
  } else {
    __syncthreads();
  }
  const int per = (a.M + a.nsplit - 1) / a.nsplit, m_begin = (int)blockIdx.y * per, m_end = min(a.M, m_begin + per);
  const uint32_t red_addr = tc::smem_u32(red);
  for (int i = threadIdx.x; i < (m_end - m_begin) * kW4BlockN; i += kW4Threads) {
    const int m = m_begin + i / kW4BlockN, c = i % kW4BlockN, n = blockIdx.x * kW4BlockN + c;
    if (n >= a.N) continue;
    const uint32_t off = (uint32_t)(m * kW4BlockN + c) * 4;
    float v;
    if (a.nsplit == 1) {
      v = red[m * kW4BlockN + c];
    } else {
      float p[8];
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (k < a.nsplit) p[k] = tc::ld_cluster_f32(tc::cluster_map(red_addr + off, (uint32_t)k));
      v = p[0];
#pragma unroll
      for (int k = 1; k < 8; ++k)
        if (k < a.nsplit) v += p[k];
    }
    const size_t idx = (size_t)m * a.N + n;
    if (a.res != nullptr) v = __bfloat162float(__float2bfloat16_rn(v)) + __bfloat162float(a.res[idx]);
    if (a.y_is_f32) reinterpret_cast<float*>(a.y)[idx] = v;
    else reinterpret_cast<__nv_bfloat16*>(a.y)[idx] = __float2bfloat16_rn(v);
  }
  if (a.nsplit > 1) {   // nobody's shared memory goes away while another CTA may read it
    tc::cluster_arrive();
    tc::cluster_wait();
  }
}

// Clusters of s CTAs with this much shared memory that the device holds at once (they lie within a group of SMs, so long ones
// leave SMs unused); 1 for a call where that cannot be found out.
template <int NT>
int w4_clusters(int device, int s, int chunk, size_t smem) {
  static DeviceAnswers<9 * 64> kept;
  return std::max(1, clusters_at_once(kept, device, s * 64 + chunk, (const void*)w4_gemm_kernel<NT>, kW4Threads, smem, 1, (unsigned)s));
}

template <int NT>
int launch_w4_nt(W4Args a, cudaStream_t stream) {
  static DeviceOnce once;
  int device = 0;
  const int rc = allow_shared_memory(once, 100 * 1024, false, {(const void*)w4_gemm_kernel<NT>}, &device);
  if (rc != QUASAR_OK) return rc;
  const int nblocks = (a.N + kW4BlockN - 1) / kW4BlockN, ngroups = a.K / kGroup;
  // Ranges: a launch takes the waves of clusters that the device holds at once - where they do not all fit, half a one more, as
  // CTAs follow one another - times the groups of a range and what a range costs besides, about three groups.  No range shorter
  // than three groups.  (us at 1 row by ranges 1 / 2 / 3 / 4 / 5 / 6 / 8: 24,576 x 4096 30 / 28 / 33 / 31 / 33 / 38 / 38; 6144 x 4096
  // 21 / 15 / 15 / 13 / 12 / 15 / 15; 151,936 x 4096 111 / 121 / 146; at 64 rows, one CTA on an SM: 4096 x 4096 52 / 32 / 25 / 19 / 31.)
  constexpr int kGroupBytes = NT * 8 * 256;
  double best = 0;
  size_t smem = 0;
  a.nsplit = 0;
  for (int s = 1; s <= 8 && (s == 1 || ngroups / s >= 3); ++s) {
    const int per = (ngroups + s - 1) / s;
    int chunk = (96 * 1024) / kGroupBytes;
    if (chunk > kW4Ahead) chunk = chunk / kW4Ahead * kW4Ahead;
    chunk = std::min(chunk, per);
    const size_t need = std::max((size_t)chunk * kGroupBytes, (size_t)NT * 8 * kW4BlockN * 4);
    const double waves = (double)nblocks / w4_clusters<NT>(device, s, chunk, need);
    const double cost = (waves > 1 ? waves + 0.5 : 1.0) * (per + 3);
    if (a.nsplit == 0 || cost < best) {
      best = cost;
      a.nsplit = s;
      a.chunk = chunk;
      smem = need;
    }
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)nblocks, (unsigned)a.nsplit);
  cfg.blockDim = dim3(kW4Threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = 1;
  attr.val.clusterDim.y = (unsigned)a.nsplit;
  attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = a.nsplit > 1 ? 1 : 0;
  QUASAR_CUDA_CHECK(cudaLaunchKernelEx(&cfg, w4_gemm_kernel<NT>, a));
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
    a.x = x + m0 * K; a.w = w; a.delta = delta;
    a.y = reinterpret_cast<unsigned char*>(y) + (size_t)m0 * N * ybytes;
    a.res = residual ? residual + m0 * N : nullptr;
    a.y_is_f32 = y_is_f32 ? 1 : 0;
    int rc;
    switch ((a.M + 7) / 8) {
      case 1: rc = launch_w4_nt<1>(a, stream); break;
      case 2: rc = launch_w4_nt<2>(a, stream); break;
      case 3: rc = launch_w4_nt<3>(a, stream); break;
      case 4: rc = launch_w4_nt<4>(a, stream); break;
      case 5: rc = launch_w4_nt<5>(a, stream); break;
      case 6: rc = launch_w4_nt<6>(a, stream); break;
      case 7: rc = launch_w4_nt<7>(a, stream); break;
      default: rc = launch_w4_nt<8>(a, stream); break;
    }
    if (rc != QUASAR_OK) return rc;
  }
  return QUASAR_OK;
}

}  // namespace quasar
