// Linear layers on int8 weights and bf16 activations for blocks too wide for digit rows (tc_wide.cu).
#pragma once

#include "common.cuh"
#include "rope.cuh"

namespace quasar {

// Whether a block of M rows with a contraction of K elements is for this kernel rather than for digit rows (see tc_wide.cu).
bool tc_wide_better(int64_t M, int64_t K);

// `pdl` as in tc_linear.cuh.  y may be nullptr and keys not: then only the rows' arg-max over the output channels is wanted.
int launch_tc_wide(const __nv_bfloat16* x, const int8_t* w, const float* dw, int64_t M, int64_t N, int64_t K, void* y, bool y_is_f32,
                   const __nv_bfloat16* residual, unsigned long long* keys, int32_t* error, bool pdl, cudaStream_t stream);
// gate+up projection: act = silu(gate) * up, [M][F] bf16
int launch_tc_wide_swiglu(const __nv_bfloat16* x, const int8_t* w, const float* dw, int64_t M, int64_t F, int64_t K, __nv_bfloat16* act,
                          int32_t* error, bool pdl, cudaStream_t stream);
// qkv projection with QK-norm, RoPE and KV append (a dependent launch), where tc_wide_rope_fits says that the layer runs as k-ranges;
// writes q (into rope.qkv) and the cache rows
bool tc_wide_rope_fits(int64_t M, int64_t N, int64_t K);
int launch_tc_wide_qkv_rope(const __nv_bfloat16* x, const int8_t* w, const float* dw, int64_t M, int64_t K, const RopeArgs& rope, int32_t* error,
                            cudaStream_t stream);

}  // namespace quasar
