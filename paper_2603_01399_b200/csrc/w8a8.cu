// The paper's W8A8 form of the linear layer (Section 3.2 Eq. 4-8, Section 3.3 Eq. 9-10):
//   offline   s_j (Eq. 5), W~ = W diag(s)^-1 (Eq. 4), W_int8 = Q(W~, delta_w) (Eq. 6)
//   online    X_int8 = Q(X * s, delta_x) per token, fused smoothing + quantisation (Eq. 9)
//             Y_int32 = W_int8 x X_int8 on the integer tensor cores (Eq. 8),  Y = Y_int32 * (delta_w * delta_x) (Eq. 10)
// Q(., delta) is the same operator everywhere: delta = absmax / 127 (fp32 IEEE division, 1 for an all-zero
// row), q = clamp(round_half_even(v / delta), -127, 127).  No fast-math on any of these paths: the integer
// codes, and with them the int32 accumulators, are bit-exact with the definition.
//
// Direction of s: Eq. 4 and Eq. 9 multiply the activations by s and divide the weights by it; for that to
// shrink an outlier channel (the stated purpose) s_j = max|W_j|^(1-alpha) / max|X_j|^alpha, the reciprocal
// of the expression printed as Eq. 5 (which is the factor the activations are divided by).
#include "common.cuh"
#include "tc_linear.cuh"

namespace quasar {

namespace {

// ---- Eq. 5: column maxima of W, then the factors ----------------------------------------------------
// A thread keeps the maxima of 8 neighbouring columns over a strip of 64 rows (16-byte loads, eight rows in flight);
// non-negative floats order like their bit patterns.
__global__ void __launch_bounds__(256) colmax_kernel(const __nv_bfloat16* __restrict__ w, int64_t N, int64_t K,
                                                     unsigned* __restrict__ colmax_bits) {
  const int64_t nvec = K / 8, v = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (v >= nvec) return;
  const int64_t n0 = (int64_t)blockIdx.y * 64;
  const int64_t n1 = n0 + 64 < N ? n0 + 64 : N;
  const uint4* p = reinterpret_cast<const uint4*>(w) + v;
  __nv_bfloat162 m[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) m[e] = __floats2bfloat162_rn(0.f, 0.f);
  auto take = [&](const uint4& r) {   // (NaNs do not enter)
    const uint32_t x[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) m[e] = __hmax2(m[e], __habs2(*reinterpret_cast<const __nv_bfloat162*>(&x[e])));
  };
  int64_t n = n0;
  for (; n + 8 <= n1; n += 8) {
    uint4 r[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) r[i] = __ldg(p + (n + i) * nvec);
#pragma unroll
    for (int i = 0; i < 8; ++i) take(r[i]);
  }
  for (; n < n1; ++n) take(__ldg(p + n * nvec));
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    atomicMax(colmax_bits + v * 8 + 2 * e, __float_as_uint(__low2float(m[e])));
    atomicMax(colmax_bits + v * 8 + 2 * e + 1, __float_as_uint(__high2float(m[e])));
  }
}

// the same for row lengths that are no multiple of 8: a thread per column
__global__ void __launch_bounds__(256) colmax_any_kernel(const __nv_bfloat16* __restrict__ w, int64_t N, int64_t K,
                                                         unsigned* __restrict__ colmax_bits) {
  const int64_t k = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (k >= K) return;
  const int64_t n0 = (int64_t)blockIdx.y * 64;
  const int64_t n1 = n0 + 64 < N ? n0 + 64 : N;
  float m = 0.f;
  for (int64_t n = n0; n < n1; ++n) m = fmaxf(m, fabsf(__bfloat162float(w[n * K + k])));
  atomicMax(colmax_bits + k, __float_as_uint(m));
}

__global__ void smooth_factor_kernel(const float* __restrict__ act_absmax, const unsigned* __restrict__ colmax_bits,
                                     int64_t K, double alpha, float* __restrict__ s) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= K) return;
  const double a = (double)act_absmax[k], wm = (double)__uint_as_float(colmax_bits[k]);
  float out = 1.0f;
  if (a > 0.0 && wm > 0.0) out = (float)(pow(wm, 1.0 - alpha) / pow(a, alpha));
  s[k] = out;
}

// The integer contraction (s8 x s8 -> s32, exact) and Eq. 10 are the tcgen05 kernel of tc_linear.cu.
constexpr size_t kCounterBytes = 64 * 1024;   // reserved at the start of every workspace (quasar.h)
constexpr int64_t kMaxChannels = (int64_t)1 << 20;

size_t align256(size_t v) { return (v + 255) / 256 * 256; }

}  // namespace

int launch_smoothing_factors(const float* act_absmax, const __nv_bfloat16* w, int64_t N, int64_t K, float alpha,
                             float* s_out, cudaStream_t stream) {
  // the column maxima are gathered in the output array itself (as bit patterns); the factor kernel reads
  // entry k and overwrites it
  unsigned* colmax = reinterpret_cast<unsigned*>(s_out);
  QUASAR_CUDA_CHECK(cudaMemsetAsync(colmax, 0, (size_t)K * sizeof(unsigned), stream));
  if (K % 8 == 0)
    colmax_kernel<<<dim3((unsigned)((K / 8 + 255) / 256), (unsigned)((N + 63) / 64)), 256, 0, stream>>>(w, N, K, colmax);
  else
    colmax_any_kernel<<<dim3((unsigned)((K + 255) / 256), (unsigned)((N + 63) / 64)), 256, 0, stream>>>(w, N, K, colmax);
  QUASAR_LAUNCH_CHECK();
  smooth_factor_kernel<<<(unsigned)((K + 255) / 256), 256, 0, stream>>>(act_absmax, colmax, K, (double)alpha, s_out);
  QUASAR_LAUNCH_CHECK();
  return QUASAR_OK;
}

size_t linear_w8a8_workspace_bytes(int64_t M, int64_t N, int64_t K) {
  (void)N;
  return kCounterBytes + align256((size_t)M * K) + align256((size_t)M * sizeof(float));
}

int launch_linear_w8a8(const __nv_bfloat16* x, const float* smooth, const int8_t* w, const float* delta_w, int64_t M,
                       int64_t N, int64_t K, void* y, bool y_is_f32, const __nv_bfloat16* residual, int32_t* acc_out,
                       void* workspace, size_t workspace_bytes, int32_t* status, cudaStream_t stream) {
  if (M <= 0 || N <= 0 || K <= 0 || (K % 16) != 0 || N > kMaxChannels || K > 0x7fffffff) {
    set_error("linear_w8a8: unsupported sizes M=%lld N=%lld K=%lld (K must be a multiple of 16, N at most %lld)",
              (long long)M, (long long)N, (long long)K, (long long)kMaxChannels);
    return QUASAR_ERR_SHAPE;
  }
  if (workspace_bytes < linear_w8a8_workspace_bytes(M, N, K)) {
    set_error("linear_w8a8: workspace of %zu bytes, need %zu", workspace_bytes, linear_w8a8_workspace_bytes(M, N, K));
    return QUASAR_ERR_CAPACITY;
  }
  unsigned char* ws = reinterpret_cast<unsigned char*>(workspace);
  int8_t* xq = reinterpret_cast<int8_t*>(ws + kCounterBytes);
  float* dx = reinterpret_cast<float*>(ws + kCounterBytes + align256((size_t)M * K));
  // Eq. 9: fused smoothing + per-token quantisation of the activations
  const int rc = launch_quantize_smoothed(x, smooth, 2, M, K, xq, dx, stream);
  if (rc != QUASAR_OK) return rc;
  return launch_tc_linear_w8a8(xq, dx, w, delta_w, M, N, K, y, y_is_f32, residual, acc_out, nullptr, status, true, stream);
}

}  // namespace quasar
