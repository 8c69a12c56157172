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

// A factor in FP64 and as an FP32 pair
struct FixedScale {
    double s;
    float hi, lo;
};
inline FixedScale fixed_scale(double s) {
    const float hi = (float)s;
    return FixedScale{s, hi, (float)(s - (double)hi)};
}
// (not inlined: see records.cuh)
static __device__ __noinline__ float fixed_density_any(unsigned long long q, double s) {
    return (float)((double)(long long)q * s);
}

// Fixed-point sum q (below 2^63) times a scale, the FP64 product rounded to FP32.  By
// FP32: q is split into three exactly converted parts whose sum and product carry
// their rounding errors, which gives the product within 2^-20 units in the last place
// beside the rounded result and what that leaves over.  Results closer than 5e-6 units to
// halfway between two floats, powers of two and the smallest and largest exponents
// take the FP64 product (three FP64 instructions for every node bound the conversion
// of a grid: 16.8M nodes took 92.7 us, without any 48.5, as here).
__device__ __forceinline__ float fixed_density(unsigned long long q, const FixedScale &f) {
    constexpr float kMagic = 8388608.0f;   // 2^23: its mantissa bits hold an integer
    auto part = [](unsigned int v) { return __fsub_rn(__uint_as_float(0x4B000000u | v), kMagic); };
    const float a = part((unsigned int)(q >> 40)) * 1099511627776.0f;
    const float b = part((unsigned int)(q >> 20) & 0xFFFFFu) * 1048576.0f;
    const float c = part((unsigned int)q & 0xFFFFFu);
    const float ab = __fadd_rn(a, b);
    float lo = __fsub_rn(b, __fsub_rn(ab, a));
    const float t = __fadd_rn(ab, c);
    lo = __fadd_rn(lo, __fsub_rn(c, __fsub_rn(t, ab)));
    const float p = __fmul_rn(t, f.hi);
    float e = __fmaf_rn(t, f.hi, -p);
    e = __fmaf_rn(t, f.lo, e);
    e = __fmaf_rn(lo, f.hi, e);
    const float r = __fadd_rn(p, e);
    const float rest = __fsub_rn(e, __fsub_rn(r, p));
    const unsigned int bits = __float_as_uint(r) & 0x7fffffffu;
    const float half = __uint_as_float((bits & 0x7f800000u) - (24u << 23));   // of r's last place
    const bool sure = fabsf(rest) < 0.99999f * half && (bits & 0x7fffffu) != 0u &&
                      bits - (64u << 23) < (184u << 23);
    if (q == 0ull) return p;
    return sure ? r : fixed_density_any(q, f.s);
}

}  // namespace pic
