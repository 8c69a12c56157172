// Line transforms in shared memory for the field solve of grids whose axes are
// at most kFftMaxN long and split into the radices below.
//
// Decimation in frequency forward, decimation in time backward, both in place
// with the mirrored stages (Cooley and Tukey, 1965; Gentleman and Sande, 1966):
// the forward transform leaves frequency k at position pos[k], the backward one
// takes it from there, so no stage reorders anything and the operators between
// the two look up the frequency of a position.
#pragma once

#include "pic_internal.cuh"

namespace pic {

namespace fft {

// w / d and w % d for 0 <= w < 2^20 by the reciprocal (the half keeps quotients off
// the integers, and their rounding error is far below 1 / d)
struct FastDiv {
    int d;
    float inv;
    __device__ __forceinline__ explicit FastDiv(int d_) : d(d_), inv(1.0f / (float)d_) {}
    __device__ __forceinline__ int quot(int w) const { return (int)(((float)w + 0.5f) * inv); }
};

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
// multiplication by -i (forward) or +i (backward)
template <bool INV>
__device__ __forceinline__ float2 rot(float2 a) {
    return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

// R-point transform of x in registers, natural order in and out
template <int R, bool INV>
struct Dft;

template <bool INV>
struct Dft<2, INV> {
    static __device__ __forceinline__ void run(float2 (&x)[2]) {
        const float2 a = x[0];
        x[0] = cadd(a, x[1]);
        x[1] = csub(a, x[1]);
    }
};

template <bool INV>
struct Dft<3, INV> {
    static __device__ __forceinline__ void run(float2 (&x)[3]) {
        constexpr float s3 = 0.86602540378443864676f;   // sin(pi/3)
        const float2 t = cadd(x[1], x[2]), d = rot<INV>(csub(x[1], x[2]));
        const float2 m = make_float2(x[0].x - 0.5f * t.x, x[0].y - 0.5f * t.y);
        x[0] = cadd(x[0], t);
        x[1] = make_float2(m.x + s3 * d.x, m.y + s3 * d.y);
        x[2] = make_float2(m.x - s3 * d.x, m.y - s3 * d.y);
    }
};

template <bool INV>
struct Dft<4, INV> {
    static __device__ __forceinline__ void run(float2 (&x)[4]) {
        const float2 a = cadd(x[0], x[2]), b = csub(x[0], x[2]);
        const float2 c = cadd(x[1], x[3]), d = rot<INV>(csub(x[1], x[3]));
        x[0] = cadd(a, c);
        x[1] = cadd(b, d);
        x[2] = csub(a, c);
        x[3] = csub(b, d);
    }
};

// odd primes: pairs x_j +- x_{R-j} against the cosines and sines of 2 pi j k / R
template <int R, bool INV>
struct DftOdd {
    static __device__ __forceinline__ void run(float2 (&x)[R], const float (&c)[R], const float (&s)[R]) {
        constexpr int H = R / 2;
        float2 t[H], d[H], sum = x[0];
#pragma unroll
        for (int j = 0; j < H; ++j) {
            t[j] = cadd(x[j + 1], x[R - 1 - j]);
            d[j] = rot<INV>(csub(x[j + 1], x[R - 1 - j]));
            sum = cadd(sum, t[j]);
        }
        const float2 x0 = x[0];
        x[0] = sum;
#pragma unroll
        for (int k = 1; k <= H; ++k) {
            float2 a = x0, b = make_float2(0.f, 0.f);
#pragma unroll
            for (int j = 1; j <= H; ++j) {
                const int m = (j * k) % R;
                a.x += c[m] * t[j - 1].x;
                a.y += c[m] * t[j - 1].y;
                b.x += s[m] * d[j - 1].x;
                b.y += s[m] * d[j - 1].y;
            }
            x[k] = cadd(a, b);
            x[R - k] = csub(a, b);
        }
    }
};
template <bool INV>
struct Dft<5, INV> {
    static __device__ __forceinline__ void run(float2 (&x)[5]) {
        const float c[5] = {1.f, 0.30901699437494742410f, -0.80901699437494742410f,
                            -0.80901699437494742410f, 0.30901699437494742410f};
        const float s[5] = {0.f, 0.95105651629515357212f, 0.58778525229247312917f,
                            -0.58778525229247312917f, -0.95105651629515357212f};
        DftOdd<5, INV>::run(x, c, s);
    }
};
template <bool INV>
struct Dft<7, INV> {
    static __device__ __forceinline__ void run(float2 (&x)[7]) {
        const float c[7] = {1.f, 0.62348980185873353053f, -0.22252093395631440429f,
                            -0.90096886790241912624f, -0.90096886790241912624f,
                            -0.22252093395631440429f, 0.62348980185873353053f};
        const float s[7] = {0.f, 0.78183148246802980871f, 0.97492791218182360702f,
                            0.43388373911755812048f, -0.43388373911755812048f,
                            -0.97492791218182360702f, -0.78183148246802980871f};
        DftOdd<7, INV>::run(x, c, s);
    }
};

// R1 R2 points as R2 transforms of R1, twiddles, R1 transforms of R2; w[m] =
// exp(-2 pi i m / (R1 R2)) for the m = j2 k1 that occur
template <int R1, int R2, bool INV>
struct DftPair {
    static __device__ __forceinline__ void run(float2 (&x)[R1 * R2], const float2 (&w)[R1 * R2]) {
        float2 y[R2][R1];
#pragma unroll
        for (int j = 0; j < R2; ++j) {
#pragma unroll
            for (int q = 0; q < R1; ++q) y[j][q] = x[q * R2 + j];
            Dft<R1, INV>::run(y[j]);
#pragma unroll
            for (int k = 1; k < R1; ++k)
                if (j > 0) y[j][k] = cmul(y[j][k], INV ? make_float2(w[j * k].x, -w[j * k].y) : w[j * k]);
        }
#pragma unroll
        for (int k = 0; k < R1; ++k) {
            float2 z[R2];
#pragma unroll
            for (int j = 0; j < R2; ++j) z[j] = y[j][k];
            Dft<R2, INV>::run(z);
#pragma unroll
            for (int q = 0; q < R2; ++q) x[k + R1 * q] = z[q];
        }
    }
};
template <bool INV>
struct Dft<6, INV> {
    static __device__ __forceinline__ void run(float2 (&x)[6]) {
        constexpr float h = 0.5f, s = 0.86602540378443864676f;
        const float2 w[6] = {{1.f, 0.f}, {h, -s}, {-h, -s}, {-1.f, 0.f}, {-h, s}, {h, s}};
        DftPair<3, 2, INV>::run(x, w);
    }
};
template <bool INV>
struct Dft<8, INV> {
    static __device__ __forceinline__ void run(float2 (&x)[8]) {
        constexpr float r = 0.70710678118654752440f;
        const float2 w[8] = {{1.f, 0.f}, {r, -r}, {0.f, -1.f}, {-r, -r}, {-1.f, 0.f}, {-r, r}, {0.f, 1.f}, {r, r}};
        DftPair<4, 2, INV>::run(x, w);
    }
};
template <bool INV>
struct Dft<16, INV> {
    static __device__ __forceinline__ void run(float2 (&x)[16]) {
        constexpr float r = 0.70710678118654752440f, c = 0.92387953251128675613f, s = 0.38268343236508977173f;
        const float2 w[16] = {{1.f, 0.f},  {c, -s},  {r, -r},  {s, -c},  {0.f, -1.f}, {-s, -c}, {-r, -r}, {-c, -s},
                              {-1.f, 0.f}, {-c, s},  {-r, r},  {-s, c},  {0.f, 1.f},  {s, c},   {r, r},   {c, s}};
        DftPair<4, 4, INV>::run(x, w);
    }
};

// One stage of radix R over `lines` lines of the axis in shared memory: blocks
// of M elements become R interleaved blocks of M / R (forward) or back.  Lanes
// run over the lines, whose stride is odd or 1, so accesses do not collide.
template <int R, bool INV>
__device__ __forceinline__ void stage(float2 *s, int lines, int line_stride, int elem_stride, int n,
                                      int M, const float2 *tw) {
    const int sub = M / R, per_line = n / R, work = lines * per_line;
    const FastDiv by_lines(lines), by_sub(sub);
    const int tstep = n / M;
    for (int w = threadIdx.x; w < work; w += blockDim.x) {
        const int u = by_lines.quot(w), line = w - u * lines;
        const int b = by_sub.quot(u), j = u - b * sub;
        float2 *p = s + line * line_stride + (b * M + j) * elem_stride;
        const int step = sub * elem_stride;
        float2 x[R];
#pragma unroll
        for (int q = 0; q < R; ++q) x[q] = p[q * step];
        if (INV && sub > 1) {
#pragma unroll
            for (int q = 1; q < R; ++q) {
                const float2 t = tw[tstep * j * q];
                x[q] = cmul(x[q], make_float2(t.x, -t.y));
            }
        }
        Dft<R, INV>::run(x);
        if (!INV && sub > 1) {
#pragma unroll
            for (int q = 1; q < R; ++q) x[q] = cmul(x[q], tw[tstep * j * q]);
        }
#pragma unroll
        for (int q = 0; q < R; ++q) p[q * step] = x[q];
    }
    __syncthreads();
}

// all stages of one axis over `lines` lines in shared memory; every thread of
// the block calls it, with the data written and a barrier passed.  Not inlined:
// one copy of the stages per kernel and direction keeps its code small.
template <bool INV>
__device__ __noinline__ void lines(float2 *s, int nlines, int line_stride, int elem_stride,
                                   const FftAxis &ax, const float2 *tw) {
    int M = INV ? 1 : ax.n;
    for (int i = 0; i < ax.stages; ++i) {
        const int R = ax.radix[INV ? ax.stages - 1 - i : i];
        if (INV) M *= R;
        switch (R) {
        case 2: stage<2, INV>(s, nlines, line_stride, elem_stride, ax.n, M, tw); break;
        case 3: stage<3, INV>(s, nlines, line_stride, elem_stride, ax.n, M, tw); break;
        case 4: stage<4, INV>(s, nlines, line_stride, elem_stride, ax.n, M, tw); break;
        case 5: stage<5, INV>(s, nlines, line_stride, elem_stride, ax.n, M, tw); break;
        case 6: stage<6, INV>(s, nlines, line_stride, elem_stride, ax.n, M, tw); break;
        case 7: stage<7, INV>(s, nlines, line_stride, elem_stride, ax.n, M, tw); break;
        case 8: stage<8, INV>(s, nlines, line_stride, elem_stride, ax.n, M, tw); break;
        case 16: stage<16, INV>(s, nlines, line_stride, elem_stride, ax.n, M, tw); break;
        }
        if (!INV) M /= R;
    }
}

}  // namespace fft
}  // namespace pic
