// 32-byte particle records: the readback's scratch between the store's order
// and load order (one aligned sector per particle), and the FP64 helpers of
// the readback kernels.
#pragma once

#include "pic_internal.cuh"

namespace pic {

__device__ __forceinline__ void st_record(float4 *rec, int64_t q, const float4 &a, const float4 &b) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(rec + 2 * q),
                 "f"(a.x), "f"(a.y), "f"(a.z), "f"(a.w), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w)
                 : "memory");
}
__device__ __forceinline__ void ld_record(const float4 *rec, int64_t q, float4 &a, float4 &b) {
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z),
                   "=f"(b.w)
                 : "l"(rec + 2 * q));
}

// (double)f by integer instructions: the exponent is rebiased and the mantissa
// shifted; subnormals are scaled by 2^64 first, infinities and NaNs get the
// top exponent (the FP64 pipe, which conversions also use, runs at about two
// lanes per clock and SM on this part)
__device__ __forceinline__ double widen(float f) {
    const unsigned sign = __float_as_uint(f) & 0x80000000u;
    unsigned b = __float_as_uint(f) & 0x7fffffffu;
    unsigned bias = 0x38000000u;   // (1023 - 127) << 20
    if (b < 0x00800000u) {         // zero or subnormal
        b = __float_as_uint(__uint_as_float(b) * 18446744073709551616.0f);
        bias = b ? 0x34000000u : 0u;   // 2^-64 more
    }
    if (b >= 0x7f800000u) bias = 0x70000000u;   // infinity, NaN
    return __hiloint2double((int)(((b >> 3) + bias) | sign), (int)(b << 29));
}

// (float)x, round to nearest with ties to even, by integer instructions; values
// outside the range of normal floats take the conversion.  (The rare paths here and
// below are calls: predicated instructions would hold the FP64 units all the same.)
static __device__ __noinline__ float narrow_any(double x) { return (float)x; }
__device__ __forceinline__ float narrow(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
    if (b < 0x3810000000000000ull || b >= 0x47E0000000000000ull) return narrow_any(x);
    const unsigned long long r = b + 0x0fffffffull + ((b >> 29) & 1ull);
    return __uint_as_float((unsigned)((r >> 29) - 0x1C0000000ull) |
                           ((unsigned)__double2hiint(x) & 0x80000000u));
}

// Floor of s and the rest rounded to FP32, for |s| < 2^52.  For 2^-26 <= |s| < 2^10
// and a rest of at least 2^-17 by integer instructions: s in units of 2^-53, what lies
// below them kept as the last bit; of the rest's 53 bits the first 23 and the next 23,
// the last seven as one bit, become floats by their bits and are added exactly, so
// that it is rounded once.
struct FloorRest {
    long long whole;
    float rest;
};
static __device__ __noinline__ FloorRest floor_rest_any(double s) {
    const double fl = floor(s);
    return FloorRest{(long long)fl, (float)(s - fl)};
}
__device__ __forceinline__ FloorRest floor_rest(double s) {
    const unsigned es = (unsigned)(__double2hiint(s) >> 20) & 0x7ffu;
    const unsigned long long m =
        ((unsigned long long)__double_as_longlong(s) & 0xfffffffffffffull) | 0x10000000000000ull;
    const int up = min(max((int)es - 1022, -25), 10);   // |s| = m 2^(up - 53)
    unsigned long long u = m << max(up, 0);
    if (up < 0) u = (m >> -up) | ((m & ((1ull << -up) - 1ull)) != 0ull);
    const long long q = __double2hiint(s) < 0 ? -(long long)u : (long long)u;
    const unsigned hi = (unsigned)((unsigned long long)q >> 30) & 0x7fffffu;
    const unsigned lo = (unsigned)q & 0x3fffffffu;
    if (es - (1023u - 26u) >= 36u || hi < 64u) return floor_rest_any(s);
    const float h = __uint_as_float(0x4b000000u | hi) - 8388608.0f;
    const float l = __uint_as_float(0x4b000000u | (lo >> 7) | ((lo & 127u) != 0u)) - 8388608.0f;
    return FloorRest{q >> 53, fmaf(h, 1.1920928955078125e-7f, l * 1.4210854715202004e-14f)};
}

// i + 1/2 in FP64 for 0 <= i < 2^31: 2^51 + (2 i + 1) / 2 built from its bits
__device__ __forceinline__ double half_node(int i) {
    return __hiloint2double(0x43200000, 2 * i + 1) - 2251799813685248.0;
}

// (i + 1/2) + o in FP64 for 0 <= i < 2^10, or i = -1 and o >= 1/2, rounded once.  For 2^-19 <= o < 1 the sum
// is exact, and an integer in units of 2^-42 below 2^53 gives its bits
__device__ __forceinline__ double half_node_plus(int i, float o) {
    const unsigned b = __float_as_uint(o), e = b >> 23;
    if (e - 108u >= 19u) return half_node(i) + widen(o);
    const unsigned long long f = ((unsigned long long)(2 * i + 1) << 41) +
                                 ((unsigned long long)((b & 0x7fffffu) | 0x800000u) << (e - 108u));
    if (f == 0ull) return 0.0;   // i = -1, o = 1/2
    const int z = __clzll((long long)f) - 11;   // to the mantissa's leading bit
    return __longlong_as_double((long long)((f << z) + ((unsigned long long)(1032 - z) << 52)));
}

// whether x lies in [0, L), on the bits: non-negative doubles order like their
// bit patterns, a set sign bit or a NaN compares above
__device__ __forceinline__ bool in_box(double x, double L) {
    return (unsigned long long)__double_as_longlong(x) < (unsigned long long)__double_as_longlong(L);
}

// x folded into [0, L); the FP64 division is for positions more than a box away
__device__ __forceinline__ double wrap_position(double x, double L) {
    if (!in_box(x, L)) {
        x += __double_as_longlong(x) < 0 ? L : -L;
        if (!in_box(x, L)) {
            x -= L * floor(x / L);
            if (x >= L) x -= L;
            if (x < 0.0) x = 0.0;
        }
    }
    return x;
}

}  // namespace pic
