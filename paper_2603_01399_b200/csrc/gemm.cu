// The linear layer  Y[m][n] = delta[n] * sum_k X[m][k] * W[n][k]  (Section 3.2 Eq. 8 / Section 3.3 Eq. 10,
// weight-only form) with int8 or bf16 weights: which kernel runs a call.
//
//  * The tcgen05 kernel (tc_linear.cu), int8 weights behind a pre-pass that writes the activations as digit rows:
//    everything but the next two.
//  * `skinny_gemm_kernel` below, warp-level MMAs on blocks of at most 8 rows whose contraction has at most 512
//    elements: such a call is all latency, and one kernel is shorter than pre-pass and tcgen05 kernel (3.1-3.8 us
//    against 5.8 us at 1024 x 256; from two 512-element pieces on the order turns: 6.3 us against 8.4 us at
//    1024 x 1024, 8 rows).
//  * the same kernel, in groups of 8 rows, where the caller's scratch does not hold even one row of digits.
#include <mutex>

#include "common.cuh"
#include "tc_linear.cuh"
#include "tc_wide.cuh"

namespace quasar {

namespace {

constexpr int kWarps = 4;
constexpr int kThreads = kWarps * 32;
constexpr int kBlockN = kWarps * 16;  // output channels per CTA
constexpr int kSub = 512;             // contraction elements staged in shared memory at a time
constexpr size_t kCounterBytes = 64 * 1024;   // reserved at the start of every workspace (quasar.h)
constexpr int64_t kMaxChannels = (int64_t)(kCounterBytes / sizeof(int)) * kBlockN;

struct GemmArgs {
  const __nv_bfloat16* x;   // [M][K]
  const int8_t* w;          // [N][K]
  const float* delta;       // [N]
  void* y;                  // [M][N] bf16 or fp32
  const __nv_bfloat16* res; // [M][N] or nullptr
  int M, N, K;              // M <= 8
  int y_is_f32;
};

__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Four signed bytes -> four bf16 (exact): byte i becomes the low mantissa byte of 2^23, which
// after the +128 bias flip reads 2^23 + (v + 128); subtracting 2^23 + 128 leaves v.
__device__ __forceinline__ void s8x4_to_bf16x4(uint32_t w, uint32_t& lo, uint32_t& hi) {
  const uint32_t u = w ^ 0x80808080u;
  const float f0 = __uint_as_float(__byte_perm(u, 0x4B000000u, 0x7440)) - 8388736.f;
  const float f1 = __uint_as_float(__byte_perm(u, 0x4B000000u, 0x7441)) - 8388736.f;
  const float f2 = __uint_as_float(__byte_perm(u, 0x4B000000u, 0x7442)) - 8388736.f;
  const float f3 = __uint_as_float(__byte_perm(u, 0x4B000000u, 0x7443)) - 8388736.f;
  __nv_bfloat162 p0 = __floats2bfloat162_rn(f0, f1);
  __nv_bfloat162 p1 = __floats2bfloat162_rn(f2, f3);
  lo = *reinterpret_cast<uint32_t*>(&p0);
  hi = *reinterpret_cast<uint32_t*>(&p1);
}

__device__ __forceinline__ uint4 ldg_stream(const void* p) {
  uint4 r;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p));
  return r;
}

// The weights are the 16-row MMA operand (rows = output channels), the activation rows the 8-wide one, zero-padded.  The
// contraction index may be permuted freely as long as both operands agree, so each thread loads 16 contiguous weight
// bytes of one row and treats them as the k-columns its fragment slots need; the matching activations come from a
// swizzled shared-memory copy.  A CTA of 4 warps owns 64 output channels and the whole contraction.
__global__ void __launch_bounds__(kThreads) skinny_gemm_kernel(GemmArgs a) {
  constexpr int kChunksPerRow = kSub / 8;
  constexpr int kSteps = kSub / 64;   // a warp step covers 64 contraction elements
  constexpr int kUnroll = 4;
  __shared__ uint4 xs[8 * kChunksPerRow];   // 16-byte chunks, swizzled by the row's parity

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  const int n0 = blockIdx.x * kBlockN + warp * 16;
  const int r0 = min(n0 + g, a.N - 1), r1 = min(n0 + g + 8, a.N - 1);
  const int8_t* wrow0 = a.w + (size_t)r0 * a.K;
  const int8_t* wrow1 = a.w + (size_t)r1 * a.K;

  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  for (int kk = 0; kk < a.K; kk += kSub) {
    __syncthreads();
    // stage X[:, kk : kk + kSub) (zero beyond M or K)
    for (int c = threadIdx.x; c < 8 * kChunksPerRow; c += kThreads) {
      const int row = c / kChunksPerRow, ch = c % kChunksPerRow;
      const int k = kk + ch * 8;
      uint4 v = make_uint4(0, 0, 0, 0);
      if (row < a.M && k < a.K) v = *reinterpret_cast<const uint4*>(a.x + (size_t)row * a.K + k);
      xs[row * kChunksPerRow + (ch ^ (row & 1))] = v;
    }
    __syncthreads();
#pragma unroll 1
    for (int s0 = 0; s0 < kSteps; s0 += kUnroll) {
      if (kk + s0 * 64 >= a.K) break;
      uint4 wa[kUnroll], wb[kUnroll];
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        const int k = kk + (s0 + u) * 64 + t * 16;
        wa[u] = k < a.K ? ldg_stream(wrow0 + k) : make_uint4(0, 0, 0, 0);
        wb[u] = k < a.K ? ldg_stream(wrow1 + k) : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        uint32_t A0[4], A1[4], A2[4], A3[4];
        const uint32_t* pa = reinterpret_cast<const uint32_t*>(&wa[u]);
        const uint32_t* pb = reinterpret_cast<const uint32_t*>(&wb[u]);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          s8x4_to_bf16x4(pa[j], A0[j], A2[j]);
          s8x4_to_bf16x4(pb[j], A1[j], A3[j]);
        }
        const int ch = (s0 + u) * 8 + t * 2;
        const uint4 x0 = xs[g * kChunksPerRow + (ch ^ (g & 1))];
        const uint4 x1 = xs[g * kChunksPerRow + ((ch + 1) ^ (g & 1))];
        mma_bf16(acc, A0[0], A1[0], A2[0], A3[0], x0.x, x0.y);
        mma_bf16(acc, A0[1], A1[1], A2[1], A3[1], x0.z, x0.w);
        mma_bf16(acc, A0[2], A1[2], A2[2], A3[2], x1.x, x1.y);
        mma_bf16(acc, A0[3], A1[3], A2[3], A3[3], x1.z, x1.w);
      }
    }
  }
  // acc[0..1]: channel n0+g, rows 2t, 2t+1;  acc[2..3]: channel n0+g+8
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int n = n0 + g + (e >> 1) * 8, m = 2 * t + (e & 1);
    if (n >= a.N || m >= a.M) continue;
    const size_t idx = (size_t)m * a.N + n;
    float v = acc[e] * a.delta[n];
    if (a.res != nullptr) v = __bfloat162float(__float2bfloat16_rn(v)) + __bfloat162float(a.res[idx]);
    if (a.y_is_f32) reinterpret_cast<float*>(a.y)[idx] = v;
    else reinterpret_cast<__nv_bfloat16*>(a.y)[idx] = __float2bfloat16_rn(v);
  }
}

size_t align256g(size_t v) { return (v + 255) / 256 * 256; }

// bytes of M activation rows as digits (behind the reserved start of a workspace)
size_t digit_bytes(int64_t M, int64_t K) { return align256g((size_t)kDigitPlanes * M * K) + align256g((size_t)M * 4); }

}  // namespace

// What this entry point has asked for since its first version - an fp16 copy of up to 80 rows and the partial sums of the
// k-ranges, up to 72 rows at a time.  The built-in scratch of linear_static takes the shapes that fit it by this measure.
static size_t linear_static_need(int64_t M, int64_t N, int64_t K) {
  constexpr int64_t kMaxRowsPerGemm = 72;
  auto ranges = [](int64_t blocks, int64_t pieces, int64_t want) {
    want = want < 1 ? 1 : (want > pieces ? pieces : want);
    want = want > 32 ? 32 : want;
    const int64_t per = (pieces + want - 1) / want;
    return (pieces + per - 1) / per;
  };
  const int64_t rows = M < kMaxRowsPerGemm ? M : kMaxRowsPerGemm, rows_u = M < 80 ? M : 80;
  const int64_t b0 = (N + 63) / 64, b1 = (N + 127) / 128;
  const int64_t s0 = ranges(b0, (K + 511) / 512, (148 * 4 + b0 - 1) / b0);
  size_t need = s0 > 1 ? (size_t)s0 * ((rows + 7) / 8 * 8) * N * 4 : 0;
  if (M > 8) {
    const int64_t s1 = ranges(b1, (K + 127) / 128, 296 / b1);
    const size_t partial = (s1 > 1 || N <= 32768) ? (size_t)s1 * ((rows_u + 15) / 16 * 16) * N * 4 : 0;
    const size_t u = align256g((size_t)rows_u * K * 2) + align256g((size_t)rows_u * 4) + partial;
    need = u > need ? u : need;
  }
  return kCounterBytes + need;
}

// What a call asks its caller for: the digit rows of a block that has them, and never less than it asked for in earlier
// versions, so that sizes worked out then still hold.
size_t linear_workspace_bytes(int64_t M, int64_t N, int64_t K) {
  const size_t digits = kCounterBytes + (tc_wide_better(M, K) ? 0 : digit_bytes(M, K)), before = linear_static_need(M, N, K);
  return digits > before ? digits : before;
}

int launch_linear(const __nv_bfloat16* x, const void* w, const float* delta, int weight_dtype, int64_t M, int64_t N,
                  int64_t K, void* y, bool y_is_f32, const __nv_bfloat16* residual, void* workspace,
                  size_t workspace_bytes, cudaStream_t stream, int32_t* status) {
  if (M <= 0 || N <= 0 || K <= 0 || (K % 16) != 0 || N > kMaxChannels || K > 0x7fffffff) {
    set_error("linear: unsupported sizes M=%lld N=%lld K=%lld (K must be a multiple of 16, N at most %lld)",
              (long long)M, (long long)N, (long long)K, (long long)kMaxChannels);
    return QUASAR_ERR_SHAPE;
  }
  if (workspace_bytes < kCounterBytes) {
    set_error("linear: workspace of %zu bytes, need %zu", workspace_bytes, linear_workspace_bytes(M, N, K));
    return QUASAR_ERR_CAPACITY;
  }
  if (weight_dtype == QUASAR_W_BF16)
    return launch_tc_linear_bf16(x, reinterpret_cast<const __nv_bfloat16*>(w), M, N, K, y, y_is_f32, residual, nullptr, status, false,
                                 stream);
  const int8_t* wq = reinterpret_cast<const int8_t*>(w);
  if (tc_wide_better(M, K)) return launch_tc_wide(x, wq, delta, M, N, K, y, y_is_f32, residual, nullptr, status, false, stream);
  const size_t ybytes = y_is_f32 ? 4 : 2;
  // rows whose digits fit behind the reserved start of the workspace: all of them, unless the workspace is smaller than
  // linear_workspace_bytes reports (the built-in one of linear_static)
  const int64_t room = (int64_t)(workspace_bytes - kCounterBytes);
  const int64_t fit = (int64_t)digit_bytes(M, K) <= room ? M : room > 512 ? (room - 512) / (kDigitPlanes * K + 4) : 0;
  if ((M <= 8 && K <= kSub) || fit < 1) {
    for (int64_t m0 = 0; m0 < M; m0 += 8) {
      GemmArgs a;
      a.M = (int)((M - m0) < 8 ? (M - m0) : 8);
      a.N = (int)N; a.K = (int)K;
      a.x = x + m0 * K; a.w = wq; a.delta = delta;
      a.y = reinterpret_cast<unsigned char*>(y) + (size_t)m0 * N * ybytes;
      a.res = residual ? residual + m0 * N : nullptr;
      a.y_is_f32 = y_is_f32 ? 1 : 0;
      skinny_gemm_kernel<<<(unsigned)((N + kBlockN - 1) / kBlockN), kThreads, 0, stream>>>(a);
      QUASAR_LAUNCH_CHECK();
    }
    return QUASAR_OK;
  }
  bool done = false;
  const int rc = launch_tc_linear_direct(x, wq, delta, M, N, K, y, y_is_f32, residual, status, &done, stream);
  if (rc != QUASAR_OK || done) return rc;
  const int64_t step = fit < M ? fit : M;
  for (int64_t m0 = 0; m0 < M; m0 += step) {
    const int64_t rows = (M - m0) < step ? (M - m0) : step;
    int8_t* xd = reinterpret_cast<int8_t*>(workspace) + kCounterBytes;
    float* scale = reinterpret_cast<float*>(xd + align256g((size_t)kDigitPlanes * rows * K));
    int rc = launch_digit_rows(x + m0 * K, rows, K, xd, scale, stream);
    if (rc != QUASAR_OK) return rc;
    // (the pre-pass starts only when whatever wrote the weights has finished, so they may be read beside it)
    rc = launch_tc_linear_digits(xd, scale, wq, delta, rows, N, K, reinterpret_cast<unsigned char*>(y) + (size_t)m0 * N * ybytes,
                                 y_is_f32, residual ? residual + m0 * N : nullptr, nullptr, status, true, stream);
    if (rc != QUASAR_OK) return rc;
  }
  return QUASAR_OK;
}

// ---- the same linear layer with its scratch inside the library ------------------------------------
// Scratch for callers that cannot hand over a workspace: a fixed array in device memory that every GPU loading the
// library holds until the process exits.
constexpr size_t kStaticScratchBytes = 4u << 20;
static __device__ __align__(256) unsigned char g_linear_scratch[kStaticScratchBytes];

size_t linear_static_scratch_bytes() { return kStaticScratchBytes; }

int launch_linear_static(const __nv_bfloat16* x, const void* w, const float* delta, int weight_dtype, int64_t M,
                         int64_t N, int64_t K, void* y, bool y_is_f32, const __nv_bfloat16* residual,
                         cudaStream_t stream) {
  if (M <= 0 || N <= 0 || K <= 0 || (K % 16) != 0 || N > kMaxChannels || K > 0x7fffffff) {
    set_error("linear_static: unsupported sizes M=%lld N=%lld K=%lld (K must be a multiple of 16, N at most %lld)",
              (long long)M, (long long)N, (long long)K, (long long)kMaxChannels);
    return QUASAR_ERR_SHAPE;
  }
  // Refused: blocks whose fp32 sums would not fit the array (the documented limit), whatever the kernel of today keeps there.
  const size_t need = linear_static_need(M, N, K);
  if (need > kStaticScratchBytes) {
    set_error("linear_static: M=%lld N=%lld K=%lld needs %zu bytes of scratch, the built-in array holds %zu; "
              "use quasar_linear with a workspace",
              (long long)M, (long long)N, (long long)K, need, kStaticScratchBytes);
    return QUASAR_ERR_CAPACITY;
  }
  // In host code the array's name only stands for the symbol; its device address is looked up once per
  // device (with that device current) and kept.  The lookup comes after the argument checks, so a refused
  // call touches nothing; it is the only step that may make the runtime load the module (and with it
  // materialise the array) - hence "first call outside any capture".
  constexpr int kMaxDevices = 64;
  static void* scratch_of_device[kMaxDevices] = {};
  static std::mutex mu;
  int dev = 0;
  QUASAR_CUDA_CHECK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) {
    set_error("linear_static: device ordinal %d not supported (at most %d devices)", dev, kMaxDevices);
    return QUASAR_ERR_CAPACITY;
  }
  void* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lock(mu);
    if (scratch_of_device[dev] == nullptr) {
      void* ptr = nullptr;
      QUASAR_CUDA_CHECK(cudaGetSymbolAddress(&ptr, g_linear_scratch));
      scratch_of_device[dev] = ptr;
    }
    scratch = scratch_of_device[dev];
  }
  return launch_linear(x, w, delta, weight_dtype, M, N, K, y, y_is_f32, residual, scratch, kStaticScratchBytes, stream, nullptr);
}

}  // namespace quasar
