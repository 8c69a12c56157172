// Sums of the field diagnostics: in FP64, and on the grids solved by cuFFT in FP32
// (hi, lo) pairs, about 48-bit arithmetic at FP32 speed (FP64 instructions run at
// a small fraction of the FP32 rate on this part); and the conversion of the
// fixed-point density.
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

// The warp's sums of four totals t of each lane: lane 8 q returns the q-th.  The lanes
// trade halves of the four first: 2 + 1 + 3 FP64 additions instead of 20, at about two
// lanes per clock and SM.
__device__ __forceinline__ double warp_sums(const double (&t)[4]) {
    const bool up = threadIdx.x & 16, odd = threadIdx.x & 8;
    const double a = (up ? t[2] : t[0]) + __shfl_xor_sync(0xffffffffu, up ? t[0] : t[2], 16);
    const double b = (up ? t[3] : t[1]) + __shfl_xor_sync(0xffffffffu, up ? t[1] : t[3], 16);
    double r = (odd ? b : a) + __shfl_xor_sync(0xffffffffu, odd ? a : b, 8);
    for (int o = 4; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    return r;
}

// The block's sums of four totals of each thread, in out[0..3], in a fixed order.
// Every thread of the THREADS-thread block calls it.
template <int THREADS>
__device__ __forceinline__ void block_field_sums(const double (&t)[4], double *out) {
    __shared__ double red[4][THREADS / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const double w4 = warp_sums(t);
    if ((lane & 7) == 0) red[lane >> 3][wid] = w4;
    __syncthreads();
    if (threadIdx.x < 4) {
        double s = 0.0;
        for (int w = 0; w < THREADS / 32; ++w) s += red[threadIdx.x][w];
        out[threadIdx.x] = s;
    }
}
// ... given as pairs
template <int THREADS>
__device__ __forceinline__ void block_field_sums(const float (&hi)[4], const float (&lo)[4], double *out) {
    double t[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) t[q] = widen(hi[q]) + widen(lo[q]);
    block_field_sums<THREADS>(t, out);
}
// s += the squares of e's components and the density r
__device__ __forceinline__ void add_field(double (&s)[4], const float4 &e, float r) {
    const double x = widen(e.x), y = widen(e.y), z = widen(e.z);
    s[0] = fma(x, x, s[0]);
    s[1] = fma(y, y, s[1]);
    s[2] = fma(z, z, s[2]);
    s[3] += widen(r);
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
