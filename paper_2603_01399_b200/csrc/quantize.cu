// Symmetric uniform quantisation of rows, one step size per row (Section 3.2 Eq. 6): offline weight preparation (Section
// 3.3; plain, or of W / s for the W8A8 form, Eq. 4) and the online quantisation of activations X * s (Eq. 9).
//
// 2 B read + 1 B written per element: every row stays in registers between its maximum and its codes, 1 to 8 warps a row so
// that a lane holds up to 4 (12 on the longest rows) 16-byte pieces, all of them in flight at once, and the quotients are
// rounded without a division (quant.cuh).  What bounds it: issuing some 17 instructions an element, 71 % of the slots of the
// whole launch, at half the warps an SM could hold (56 registers); the memory is half busy.  24,576 x 4096 takes 68 us, of which the
// memory needs 47; a CTA per row that read it twice and divided took 88.
#include "common.cuh"
#include "quant.cuh"
#include "tc_common.cuh"

namespace quasar {

namespace {

constexpr int kQuantThreads = 256;
constexpr int kQuantWarps = kQuantThreads / 32;

enum SmoothMode { kPlain = 0, kDivide = 1, kMultiply = 2 };

// the eight values of vector i, smoothed
template <int MODE>
__device__ __forceinline__ void smooth8(float (&f)[8], const float* __restrict__ s, int64_t i) {
  if (MODE == kPlain) return;
  const float4 a = __ldg(reinterpret_cast<const float4*>(s) + 2 * i), b = __ldg(reinterpret_cast<const float4*>(s) + 2 * i + 1);
  const float sv[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
  for (int e = 0; e < 8; ++e) f[e] = MODE == kDivide ? __fdiv_rn(f[e], sv[e]) : __fmul_rn(f[e], sv[e]);
}

// of eight bf16 as they are packed: pairwise, a NaN wins
__device__ __forceinline__ void take_packed(__nv_bfloat162& m, const uint4& v) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int e = 0; e < 4; ++e) m = __hmax2_nan(m, __habs2(*reinterpret_cast<const __nv_bfloat162*>(&w[e])));
}

__device__ __forceinline__ float step_of(float amax) { return amax == 0.f ? 1.0f : __fdiv_rn(amax, 127.0f); }

// V pieces of 8 elements per lane, `wpr` warps per row (V * 32 * wpr pieces >= the row's)
template <int MODE, int V>
__global__ void __launch_bounds__(kQuantThreads)
quantize_rows_kernel(const __nv_bfloat16* __restrict__ w, const float* __restrict__ s, int64_t N, int nvec, int wpr,
                     int8_t* __restrict__ q, float* __restrict__ delta) {
  tc::pdl_trigger();   // (the contraction that follows in quasar_linear_w8a8 asks for its weights meanwhile)
  __shared__ uint2 s_max[kQuantWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t n = (int64_t)blockIdx.x * (kQuantWarps / wpr) + warp / wpr;
  const bool live = n < N;
  const int first = (warp % wpr) * 32 + lane, step = 32 * wpr;
  const uint4* row = reinterpret_cast<const uint4*>(w) + (live ? n : 0) * nvec;
  uint4 raw[V];
#pragma unroll
  for (int j = 0; j < V; ++j) raw[j] = (live && first + j * step < nvec) ? __ldg(row + first + j * step) : make_uint4(0, 0, 0, 0);
  float f[MODE == kPlain ? 1 : V][8];
  AbsMax m;
  if (MODE == kPlain) {
    __nv_bfloat162 pm = __floats2bfloat162_rn(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < V; ++j) take_packed(pm, raw[j]);
    m.take(__low2float(pm));
    m.take(__high2float(pm));
    if (m.has_nan()) {   // the largest of the numbers among them
#pragma unroll
      for (int j = 0; j < V; ++j) {
        unpack_bf16x8(raw[j], f[0]);
#pragma unroll
        for (int e = 0; e < 8; ++e) m.take(f[0][e]);
      }
    }
  } else {
#pragma unroll
    for (int j = 0; j < V; ++j) {
      float (&x)[8] = f[MODE == kPlain ? 0 : j];
      unpack_bf16x8(raw[j], x);
      if (first + j * step < nvec) smooth8<MODE>(x, s, first + j * step);
#pragma unroll
      for (int e = 0; e < 8; ++e) m.take(x[e]);
    }
  }
  m.num = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m.num)));   // (magnitudes order like their bits)
  m.bits = __reduce_max_sync(0xffffffffu, m.bits);
  if (wpr > 1) {
    if (lane == 0) s_max[warp] = make_uint2(__float_as_uint(m.num), m.bits);
    __syncthreads();
    for (int i = 0; i < wpr; ++i) {
      const uint2 o = s_max[warp / wpr * wpr + i];
      m.num = fmaxf(m.num, __uint_as_float(o.x));
      m.bits = max(m.bits, o.y);
    }
  }
  const QuantStep st = quant_step(step_of(m.num), m.has_nan());
  if (!live) return;
  if (first == 0) delta[n] = st.delta;
  uint2* qrow = reinterpret_cast<uint2*>(q) + n * nvec;
#pragma unroll
  for (int j = 0; j < V; ++j) {
    const int i = first + j * step;
    if (i >= nvec) continue;
    float (&x)[8] = f[MODE == kPlain ? 0 : j];
    if (MODE == kPlain) unpack_bf16x8(raw[j], x);
    float c[8];
    quantize8(x, st, 127, c);
    qrow[i] = pack_codes8(c);
  }
}

// rows too long for registers: one CTA per row, read twice
template <int MODE>
__global__ void __launch_bounds__(kQuantThreads)
quantize_long_rows_kernel(const __nv_bfloat16* __restrict__ w, const float* __restrict__ s, int64_t nvec, int8_t* __restrict__ q,
                          float* __restrict__ delta) {
  tc::pdl_trigger();
  __shared__ uint2 s_max[kQuantWarps];
  const int64_t n = blockIdx.x;
  const uint4* row = reinterpret_cast<const uint4*>(w) + n * nvec;
  float f[8];
  AbsMax m;
  for (int64_t i = threadIdx.x; i < nvec; i += kQuantThreads) {
    unpack_bf16x8(__ldg(row + i), f);
    smooth8<MODE>(f, s, i);
#pragma unroll
    for (int e = 0; e < 8; ++e) m.take(f[e]);
  }
  m.num = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m.num)));
  m.bits = __reduce_max_sync(0xffffffffu, m.bits);
  if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = make_uint2(__float_as_uint(m.num), m.bits);
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kQuantWarps; ++i) {
    m.num = fmaxf(m.num, __uint_as_float(s_max[i].x));
    m.bits = max(m.bits, s_max[i].y);
  }
  const QuantStep st = quant_step(step_of(m.num), m.has_nan());
  if (threadIdx.x == 0) delta[n] = st.delta;
  for (int64_t i = threadIdx.x; i < nvec; i += kQuantThreads) {
    unpack_bf16x8(__ldg(row + i), f);
    smooth8<MODE>(f, s, i);
    float c[8];
    quantize8(f, st, 127, c);
    reinterpret_cast<uint2*>(q)[n * nvec + i] = pack_codes8(c);
  }
}

template <int MODE>
int launch_mode(const __nv_bfloat16* w, const float* s, int64_t N, int64_t K, int8_t* q, float* delta, cudaStream_t stream) {
  const int64_t nvec = K / 8;
  int wpr = 1;
  while (wpr < 8 && nvec > (int64_t)4 * 32 * wpr) wpr *= 2;
  const unsigned grid = (unsigned)((N + kQuantWarps / wpr - 1) / (kQuantWarps / wpr));
  if (nvec <= (int64_t)2 * 32 * wpr)
    quantize_rows_kernel<MODE, 2><<<grid, kQuantThreads, 0, stream>>>(w, s, N, (int)nvec, wpr, q, delta);
  else if (nvec <= (int64_t)4 * 32 * wpr)
    quantize_rows_kernel<MODE, 4><<<grid, kQuantThreads, 0, stream>>>(w, s, N, (int)nvec, wpr, q, delta);
  else if (nvec <= (int64_t)8 * 32 * wpr)
    quantize_rows_kernel<MODE, 8><<<grid, kQuantThreads, 0, stream>>>(w, s, N, (int)nvec, wpr, q, delta);
  else if (nvec <= (int64_t)12 * 32 * wpr)
    quantize_rows_kernel<MODE, 12><<<grid, kQuantThreads, 0, stream>>>(w, s, N, (int)nvec, wpr, q, delta);
  else
    quantize_long_rows_kernel<MODE><<<(unsigned)N, kQuantThreads, 0, stream>>>(w, s, nvec, q, delta);
  QUASAR_LAUNCH_CHECK();
  return QUASAR_OK;
}

}  // namespace

int launch_quantize(const __nv_bfloat16* w, int64_t N, int64_t K, int8_t* q, float* delta, cudaStream_t stream) {
  if (N == 0) return QUASAR_OK;
  return launch_mode<kPlain>(w, nullptr, N, K, q, delta, stream);
}

int launch_quantize_smoothed(const __nv_bfloat16* v, const float* s, int mode, int64_t rows, int64_t K, int8_t* q,
                             float* delta, cudaStream_t stream) {
  if (rows == 0) return QUASAR_OK;
  if (s == nullptr) return launch_mode<kPlain>(v, nullptr, rows, K, q, delta, stream);
  if (mode == kDivide) return launch_mode<kDivide>(v, s, rows, K, q, delta, stream);
  return launch_mode<kMultiply>(v, s, rows, K, q, delta, stream);
}

}  // namespace quasar
