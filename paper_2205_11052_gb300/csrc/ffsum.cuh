// FP32 (hi, lo) pair sums of the field diagnostics: about 48-bit arithmetic at
// FP32 speed (FP64 instructions run at a small fraction of the FP32 rate on
// this part), shared by the single-run and the batched reductions.
#pragma once

#include "records.cuh"

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

// A factor and what a product with it and 2^52 + q is off by
struct FixedScale {
    double s, off;
};
inline FixedScale fixed_scale(double s) {
    const double most = 8.4527e270;   // beyond FP32's range with any q but 0, 2^52 s within FP64's
    if (s > most) s = most;
    if (s < -most) s = -most;
    return FixedScale{s, -4503599627370496.0 * s};
}

// Fixed-point sum q (below 2^52: 2^31 particles of 2^20 units fit) times a scale, the
// FP64 product rounded to FP32.  q's bits below an exponent of 2^52 are 2^52 + q, so one
// fused multiply-add gives the product, and the rounding is integer instructions: FP64
// ones run at about two lanes per clock and SM, and with three of them a node (a
// conversion, the product, a conversion) they bound the conversion of a grid: 16.8M
// nodes 92.7 us, now 55.8 (their bytes 50).
__device__ __forceinline__ float fixed_density(unsigned long long q, const FixedScale &f) {
    const double d = fma(__longlong_as_double((long long)(q | 0x4330000000000000ull)), f.s, f.off);
    if (q == 0ull) return __uint_as_float((unsigned)__double2hiint(f.s) & 0x80000000u);   // 0 s
    return narrow(d);
}

}  // namespace pic
