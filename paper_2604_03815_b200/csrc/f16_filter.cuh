// Shared pieces of the half-precision prefilter (score_select_f16.cu, f16_convert.cu, refine_f16.cu):
// the per-head statistics, the power-of-two scaling of the fp16 operand copies and the error bound of
// an fp16-accumulated tensor-core score.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

namespace kmip {

// Groups kept per row by the prefilter sweep for 16 < k <= 32 (k + slack, a multiple of 8).
constexpr int kF16List32 = 48;
// ... and for 32 < k <= 103.
constexpr int kF16ListMost = 120;

// Rows whose squared norm reaches this (or is not finite) take no part in the maxima below: their fp16 copies overflow under
// any scale that suits the others.  Such a query row, and every row of a head with such a key, is scored exactly
// (refine_f16.cu).
constexpr float kF16RangeN2 = 1.5e38f;

// Per head: largest squared norm of a query row, of a key row, and of the first 16 elements of a key
// row (the partial sum after the first tensor-core step of a wider head); largest squared norm of what the conversion
// of a key row to fp16 lost (fp32 storage only; bf16 values convert exactly up to underflow).  Float bits, maxima taken
// with integer atomics (the values are non-negative).
struct F16HeadStat {
    float q_n2max;
    float k_n2max;
    float k_first16_n2max;
    float k_lost_n2max;  // of the SCALED row; +infinity: the head has a key beyond kF16RangeN2
};

// Power of two s such that s * sqrt(n2max) lies in [32, 64) (up to the rounding of the square root):
// products of two scaled rows stay below 4096 < 65504, and elements lose bits only below 2^-14.
__host__ __device__ inline float f16_scale_from_n2max(float n2max) {
    if (!(n2max > 0.0f) || !(n2max < 3.0e38f)) return 1.0f;
    int e = 0;
    frexpf(sqrtf(n2max), &e);  // sqrt = m * 2^e, m in [0.5, 1)
    int se = 6 - e;
    se = se < -60 ? -60 : (se > 60 ? 60 : se);
    return ldexpf(1.0f, se);
}

// |fp16 score T - exact scaled score| <= a + r * |T| for every key of the head, given the row's scaled
// norms.  The tensor cores round the fp16 accumulator to nearest once per 16-deep step: the last
// rounding is at most 2^-11 |T|, an earlier one at most 2^-11 times the partial sum, itself at most
// |q[0:16 s]| |k[0:16 s]| (`partial`: the sum of these products over the steps before the last).  2^-18 |q||k| covers
// the internal summation, 2.5e-5 the elements that underflowed in the conversion (scaled norms are below 64) and
// subnormal results; `lost` what rounding fp32 operands to fp16 changed (at most |q| |dk| + |dq| |k|; 0 for bf16).
constexpr float kF16RelErr = 4.8923e-4f;  // 2^-11 (1 + 2^-9)
__host__ __device__ inline float f16_abs_err(float partial, float nq, float nk_max, float lost) {
    return kF16RelErr * partial + 3.8147e-6f * nq * nk_max + 2.5e-5f + lost;
}

}  // namespace kmip
