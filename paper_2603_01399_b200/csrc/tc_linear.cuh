// Linear layers on the tcgen05 tensor cores (tc_linear.cu).
#pragma once

#include "common.cuh"
#include "rope.cuh"

namespace quasar {

// The launchers below take `pdl`: launched as a dependent of the kernel in front of it on the stream, whose results are waited
// for before the activations, the residual or y are touched; the WEIGHTS may be read before that, so a caller sets it only
// where the kernel in front does not write them and was itself launched behind whatever did.
// y may be nullptr and keys not: then only the rows' arg-max over the output channels is wanted.

int launch_tc_linear_bf16(const __nv_bfloat16* x, const __nv_bfloat16* w, int64_t M, int64_t N, int64_t K, void* y, bool y_is_f32,
                          const __nv_bfloat16* residual, unsigned long long* keys, int32_t* error, bool pdl, cudaStream_t stream);

// int8 weights, bf16 activations as digit rows: xd [kDigitPlanes M][K] int8 and row_scale [M], see write_digits8
constexpr int kDigitPlanes = 4;
constexpr int kDigitRows = 256 / kDigitPlanes;   // rows of a block at most: operand B of an MMA has 256
int launch_digit_rows(const __nv_bfloat16* x, int64_t M, int64_t K, int8_t* xd, float* row_scale, cudaStream_t stream);
int launch_tc_linear_digits(const int8_t* xd, const float* row_scale, const int8_t* w, const float* dw, int64_t M, int64_t N,
                            int64_t K, void* y, bool y_is_f32, const __nv_bfloat16* residual, unsigned long long* keys, int32_t* error, bool pdl,
                            cudaStream_t stream);

// the same on the bf16 rows themselves, in one launch, for blocks of up to 6 rows; *done false: not for this matrix, nothing launched
int launch_tc_linear_direct(const __nv_bfloat16* x, const int8_t* w, const float* dw, int64_t M, int64_t N, int64_t K, void* y, bool y_is_f32,
                            const __nv_bfloat16* residual, int32_t* error, bool* done, cudaStream_t stream);

// int8 weights, int8 activations with their step sizes (Eq. 8, Eq. 10); acc_out: the raw sums, or nullptr
int launch_tc_linear_w8a8(const int8_t* xq, const float* dx, const int8_t* w, const float* dw, int64_t M, int64_t N, int64_t K,
                          void* y, bool y_is_f32, const __nv_bfloat16* residual, int32_t* acc_out, unsigned long long* keys, int32_t* error, bool pdl,
                          cudaStream_t stream);

// Layers of the pass with the step that follows in their epilogue (form: OperandForm, which the operand is in; always
// dependent launches), for blocks that tc_fusable accepts.
// qkv projection: QK-norm, RoPE and KV append; writes q (into rope.qkv) and the cache rows.
bool tc_fusable(int form, int64_t M);
int launch_tc_qkv_rope(int form, const void* x, const float* dx, const void* w, const float* dw, int64_t M, int64_t K, const RopeArgs& rope,
                       int32_t* error, cudaStream_t stream);
// gate+up projection: act = silu(gate) * up, [M][F] bf16; act_max [M] (zero before): bits of each row's largest magnitude,
// times the smoothing factors of the down projection's input if there are any
int launch_tc_gateup_swiglu(int form, const void* x, const float* dx, const void* w, const float* dw, int64_t M, int64_t F, int64_t K,
                            __nv_bfloat16* act, unsigned* act_max, const float* smooth, int32_t* error, cudaStream_t stream);

#ifdef __CUDACC__
// Order-preserving key of a value and its index: the larger key is the larger value and, among equals, the lower index.
__device__ __forceinline__ unsigned long long argmax_key(float x, int idx) {
  x += 0.0f;                                            // -0 -> +0: they compare equal
  uint32_t u = __float_as_uint(x);
  u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
  return ((unsigned long long)u << 32) | (unsigned long long)(0xffffffffu - (uint32_t)idx);
}

// Sixteen rows of a tile whose lanes are 32 neighbouring channels: rows r0 .. r0 + 15 of f, one channel (n) a lane.

// The rows' arg-max over the warp's channels joins what the warp has seen of them so far: best [16] for the rows r0 .. (lane j
// looks after row j, so nothing here is atomic).  NaNs never enter; of equal values the lowest channel does.
__device__ __forceinline__ void best16(const float (&f)[16], bool live, int n, int count, unsigned long long* best) {
  const int lane = threadIdx.x & 31;
  uint32_t mine = 0u, at = 0u;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const uint32_t key = live && f[j] == f[j] ? (uint32_t)(argmax_key(f[j], 0) >> 32) : 0u;
    const uint32_t top = __reduce_max_sync(0xffffffffu, key);
    const unsigned who = __ballot_sync(0xffffffffu, key == top);
    if (lane == j) { mine = top; at = (uint32_t)__ffs(who) - 1u; }
  }
  if (lane < count && mine != 0u) {   // (no value has the key 0: that of a negative NaN)
    const unsigned long long k = ((unsigned long long)mine << 32) | (unsigned long long)(0xffffffffu - ((uint32_t)(n - lane) + at));
    if (k > best[lane]) best[lane] = k;
  }
}

// The rows to their places, y [.][N] from row m on.  (Rows, residual and type are told apart outside the loops: inside, a row
// took a warp 175 cycles of one instruction waiting for another.)
__device__ __forceinline__ void store16(float (&f)[16], bool live, size_t m, int n, int N, int count, void* y, bool f32, bool with_res,
                                        const uint16_t (&res)[16]) {
  if (!live) return;
  if (with_res) {
#pragma unroll
    for (int j = 0; j < 16; ++j) f[j] = __bfloat162float(__float2bfloat16_rn(f[j])) + __uint_as_float((uint32_t)res[j] << 16);
  }
  if (f32) {
    float* p = reinterpret_cast<float*>(y) + m * N + n;
#pragma unroll
    for (int j = 0; j < 16; ++j, p += N)
      if (j < count) *p = f[j];
  } else {
    __nv_bfloat16* p = reinterpret_cast<__nv_bfloat16*>(y) + m * N + n;
#pragma unroll
    for (int j = 0; j < 16; ++j, p += N)
      if (j < count) *p = __float2bfloat16_rn(f[j]);
  }
}

__device__ __forceinline__ void load_res16(uint16_t (&r)[16], const __nv_bfloat16* res, bool live, size_t m, int n, int N, int count) {
  const uint16_t* p = reinterpret_cast<const uint16_t*>(res) + m * N + n;
#pragma unroll
  for (int j = 0; j < 16; ++j, p += N) r[j] = live && j < count ? *p : (uint16_t)0;
}

constexpr int kDigitThreads = 256;

// Magnitudes as bit patterns: they order like the numbers, with infinity above those and NaN above infinity, so that a maximum
// of them (unlike fmaxf's) does not lose a NaN.
__device__ __forceinline__ uint32_t magnitude(float f) { return __float_as_uint(f) & 0x7fffffffu; }
// the larger magnitude of two bf16 in a word
__device__ __forceinline__ uint32_t magnitude2(uint32_t w) { return max((w << 16) & 0x7fffffffu, w & 0x7fff0000u); }

__device__ __forceinline__ uint32_t digit_block_max(uint32_t v, uint32_t* s_max) {
  v = __reduce_max_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = v;
  __syncthreads();
  v = s_max[0];
#pragma unroll
  for (int i = 1; i < kDigitThreads / 32; ++i) v = max(v, s_max[i]);
  return v;
}

// A row as fixed point against a power of two above its largest magnitude (its bits): x = q * 2^(E-31) (up = 2^(31-E), down
// its inverse).  E leaves the largest magnitude 2^-6 of room: four balanced digits end at 0.996 * 2^31, and a maximum taken before
// its element was rounded to bf16 may be short by 2^-9.  A bf16 element within 2^-23 of the maximum is represented exactly, a
// smaller one to 2^-32 of 2^E.  (Three digits, 2^-14 and 2^-22, lost what rows with outliers hold beside them: 4096 x 4096, one
// element of 2^12 that meets weights of zero among normal ones, relative error of the product 8e-4; an fp32 sum 1e-7.)  A row that holds a NaN is NaN times whatever its digits are.  One that holds infinities
// and no NaN (up = 0) has the digits +-1 for them and 0 for the rest, times infinity: the product is the infinity of the sign
// of the weight that meets it, and NaN where that is zero.  (Several infinities that pull apart: the sign of the larger weights.)
__device__ __forceinline__ void digit_scale(uint32_t amax_bits, float& up, float& down) {
  const float amax = __uint_as_float(amax_bits);
  up = 1.f;
  down = 1.f;
  if (amax_bits == 0x7f800000u) {
    up = 0.f;
    down = amax;
  } else if (amax_bits > 0u && amax_bits < 0x7f800000u) {
    int e;
    const float f = frexpf(amax, &e);  // amax = f * 2^e, f in [0.5, 1): |x| < 2^e along the row
    if (f > 0.984375f) ++e;
    e = e < -95 ? -95 : e;             // keeps both factors normal numbers
    up = ldexpf(1.f, 31 - e);
    down = ldexpf(1.f, e - 31);
  } else if (amax_bits > 0x7f800000u) {
    down = __int_as_float(0x7fc00000);
  }
}

// The elements of a row that holds infinities (digit_scale: up = 0): +-1 for those and 0 for the rest, to be taken with up = 1.
// (Apart from digits8, whose loops are on the way of every call: tested there, element by element or eight at a time, it cost the
// one-launch form 1.4 us of 7.4.)
__device__ __forceinline__ float only_infinite(float f) { return magnitude(f) == 0x7f800000u ? copysignf(1.f, f) : 0.f; }
__device__ __forceinline__ uint32_t only_infinite2(uint32_t w) {   // two bf16 in a word
  uint32_t out = 0;
  if ((w & 0x00007fffu) == 0x00007f80u) out |= (w & 0x00008000u) | 0x00003f80u;
  if ((w & 0x7fff0000u) == 0x7f800000u) out |= (w & 0x80000000u) | 0x3f800000u;
  return out;
}

// q as four balanced base-256 digits, q = d0 + 2^8 d1 + 2^16 d2 + 2^24 d3, each an int8: eight elements, digit by digit
__device__ __forceinline__ void digits8(const float (&f)[8], float up, uint2 (&out)[kDigitPlanes]) {
  uint32_t p[kDigitPlanes][2] = {};
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const float v = fminf(fmaxf(f[e] * up, -2139062016.f), 2139062016.f);
    // Balanced digits without a chain from one to the next: the bytes of q + 0x00808080, with the tops of the low three turned,
    // are its digits (a byte b + 128 carries where the digit below it is negative).
    const uint32_t q = ((uint32_t)__float2int_rn(v) + 0x00808080u) ^ 0x00808080u;
#pragma unroll
    for (int d = 0; d < kDigitPlanes; ++d) p[d][e >> 2] |= ((q >> (8 * d)) & 0xffu) << (8 * (e & 3));
  }
#pragma unroll
  for (int d = 0; d < kDigitPlanes; ++d) out[d] = make_uint2(p[d][0], p[d][1]);
}
// eight elements from k on, plane d at d * K (up: as digit_scale gives it)
__device__ __forceinline__ void write_digits8(const float (&x)[8], float up, int8_t* dst, int64_t K, int64_t k) {
  uint2 p[kDigitPlanes];
  float f[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) f[e] = x[e];
  if (up == 0.f) {
    up = 1.f;
#pragma unroll
    for (int e = 0; e < 8; ++e) f[e] = only_infinite(x[e]);
  }
  digits8(f, up, p);
#pragma unroll
  for (int d = 0; d < kDigitPlanes; ++d) *reinterpret_cast<uint2*>(dst + d * K + k) = p[d];
}
#endif

}  // namespace quasar
