// FP32 (hi, lo) pair sums of the field diagnostics: about 48-bit arithmetic at
// FP32 speed (FP64 instructions run at a small fraction of the FP32 rate on
// this part), shared by the single-run and the batched reductions.
#pragma once

namespace pic {

// (hi, lo) += a, with the rounding error of the FP32 sum (Knuth's TwoSum,
// exact in round-to-nearest) carried in lo.
__device__ __forceinline__ void ff_add(float &hi, float &lo, float a) {
    const float s = __fadd_rn(hi, a);
    const float bb = __fsub_rn(s, hi);
    const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(a, bb));
    lo = __fadd_rn(lo, err);
    hi = s;
}

// (hi, lo) += x^2: the product x*x is split exactly into its rounded value
// and the FMA residual x*x - fl(x*x) (an FP32 product of FP32 inputs is exact
// in 48 bits)
__device__ __forceinline__ void ff_add_sq(float &hi, float &lo, float x) {
    const float p = __fmul_rn(x, x);
    const float e = __fmaf_rn(x, x, -p);
    ff_add(hi, lo, p);
    lo = __fadd_rn(lo, e);
}

}  // namespace pic
