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

// The block's sums of four such pairs, in out[0..3] as FP64: pairs are added
// across the lanes in FP32 (error terms included), warps in FP64, both in a
// fixed order.  Every thread of the THREADS-thread block calls it.
template <int THREADS>
__device__ __forceinline__ void block_field_sums(float (&hi)[4], float (&lo)[4], double *out) {
    __shared__ double red[4][THREADS / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        for (int o = 16; o > 0; o >>= 1) {
            const float h = __shfl_down_sync(0xffffffffu, hi[q], o);
            const float l = __shfl_down_sync(0xffffffffu, lo[q], o);
            ff_add(hi[q], lo[q], h);
            lo[q] = __fadd_rn(lo[q], l);
        }
        if (lane == 0) red[q][wid] = (double)hi[q] + (double)lo[q];
    }
    __syncthreads();
    if (threadIdx.x < 4) {
        double t = 0.0;
        for (int w = 0; w < THREADS / 32; ++w) t += red[threadIdx.x][w];
        out[threadIdx.x] = t;
    }
}

}  // namespace pic
