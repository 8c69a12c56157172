// Field solve (Section 3.1 step 2, Eq. potential; Section 3.2 of
// arXiv 2205.11052) of grids whose three axes are at most kFftMaxN long and products
// of 2, 3, 5 and 7, with (y, z) planes of at most 96^2 nodes (fft_supported), in three
// kernels around the line transforms of fft.cuh:
//   k_fft_x_forward   rows of rho -> spectra over x (two real rows per complex
//                     line), stored by x frequency: rho_hat[kx][z][y]
//   k_fft_yz          one (y, z) plane of one x frequency and one component per
//                     block, in shared memory: forward over y and z, the Green
//                     kernel of k_green, back over z and y
//   k_fft_x_backward  rows of the three components -> the x-paired E8, E4 where the
//                     caller keeps it and, when asked, the block's partial sums
// The adjoint's solve runs the mirrored kernels (three components forward, the
// conjugate symbol, one density backward).
//
// Around cuFFT the same solve took eleven launches: its transforms over one axis
// each (six), the Green kernel, the interleaving, the pairing and the field sums,
// each a pass over memory: 20 steps with records of 16^3 x 8 took 1.95 ms, now 1.47,
// of 64^3 x 16 4.22, now 3.59.
#include <math.h>

#include <algorithm>
#include <vector>

#include "ffsum.cuh"
#include "fft.cuh"
#include "pic_internal.cuh"

namespace pic {

namespace {

using fft::lines;

constexpr int kRowsF = 32;   // rows of one plane per block of the forward x kernel
constexpr int kRowsB = 16;   // of the backward one
constexpr int kXThreads = 128;

__device__ __forceinline__ void load_twiddles(float2 *tw, const FftTables *tab, int axis, int n) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) tw[i] = tab->tw[axis][i];
}

// The spectra of the two real rows packed in a complex line: Z = A + i B, with
// A(k) = (Z(k) + Z*(n - k)) / 2 and B(k) = (Z(k) - Z*(n - k)) / (2 i).
__device__ __forceinline__ void unpack_rows(float2 z, float2 m, float2 &a, float2 &b) {
    a = make_float2(0.5f * (z.x + m.x), 0.5f * (z.y - m.y));
    b = make_float2(0.5f * (z.y + m.y), 0.5f * (m.x - z.x));
}

// COMPS = 1: rows of rho (float).  COMPS = 3: rows of the three components of
// lE4, which is cleared for the next reverse push.
template <int COMPS>
__global__ void __launch_bounds__(kXThreads) k_fft_x_forward(int ny, int nz, int nh, FftAxis ax,
                                                             const FftTables *__restrict__ tab,
                                                             const float *rho,
                                                             float4 *lE4,
                                                             float2 *__restrict__ out, int64_t nhalf) {
    dep_begin(rho, lE4, out);
    if (COMPS == 1) {   // blockIdx.z: one of several grids in a row
        rho += blockIdx.z * ((int64_t)ax.n * ny * nz);
        out += blockIdx.z * nhalf;
    }
    constexpr int ROWS = COMPS == 1 ? kRowsF : kRowsB;
    constexpr int PAIRS = ROWS / 2;
    extern __shared__ float2 sm[];
    const int n = ax.n, pitch = n | 1;
    float2 *s = sm, *tw = sm + COMPS * PAIRS * pitch;
    const int z = blockIdx.y, y0 = blockIdx.x * ROWS, rows = min(ROWS, ny - y0);
    load_twiddles(tw, tab, 0, n);
    float *sf = reinterpret_cast<float *>(s);
    const fft::FastDiv by_n(n), by_nh(nh);
    for (int w = threadIdx.x; w < ROWS * n; w += kXThreads) {
        const int r = by_n.quot(w), x = w - r * n;
        const int64_t g = ((int64_t)z * ny + y0 + r) * n + x;
        float v[3] = {0.f, 0.f, 0.f};
        if (r < rows) {
            if (COMPS == 1) {
                v[0] = rho[g];
            } else {
                const float4 e = lE4[g];
                v[0] = e.x;
                v[1] = e.y;
                v[2] = e.z;
            }
        }
#pragma unroll
        for (int d = 0; d < COMPS; ++d) sf[2 * ((d * PAIRS + (r >> 1)) * pitch + x) + (r & 1)] = v[d];
    }
    __syncthreads();
    if (COMPS == 3) {   // in a loop of its own, so that the loads above overlap
        float4 *row = lE4 + ((int64_t)z * ny + y0) * n;
        for (int w = threadIdx.x; w < rows * n; w += kXThreads) row[w] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    lines<false>(s, COMPS * PAIRS, pitch, 1, ax, tw);
    // lanes over the rows: runs of ROWS values at one frequency
    for (int w = threadIdx.x; w < COMPS * nh * PAIRS; w += kXThreads) {
        const int q = w % PAIRS, u = w / PAIRS;
        const int d = COMPS == 1 ? 0 : by_nh.quot(u), k = u - d * nh;
        const float2 *line = s + (d * PAIRS + q) * pitch;
        float2 a, b;
        unpack_rows(line[tab->pos[0][k]], line[tab->pos[0][k == 0 ? 0 : n - k]], a, b);
        float2 *o = out + d * nhalf + ((int64_t)k * nz + z) * ny + y0;
        if (2 * q < rows) o[2 * q] = a;
        if (2 * q + 1 < rows) o[2 * q + 1] = b;
    }
}

// plane of one x frequency: [z][y] in global memory, pitch ny | 1 in shared
__device__ __forceinline__ void load_plane(float2 *s, const float2 *in, int ny, int nz,
                                           int pitch) {
    const fft::FastDiv by_ny(ny);
    for (int w = threadIdx.x; w < ny * nz; w += blockDim.x) {
        const int z = by_ny.quot(w);
        s[z * pitch + (w - z * ny)] = in[w];
    }
}
__device__ __forceinline__ void store_plane(float2 *__restrict__ out, const float2 *s, int ny, int nz,
                                            int pitch) {
    const fft::FastDiv by_ny(ny);
    for (int w = threadIdx.x; w < ny * nz; w += blockDim.x) {
        const int z = by_ny.quot(w);
        out[w] = s[z * pitch + (w - z * ny)];
    }
}

// out_d = symbol_d(in) over one plane (blockIdx.x: x frequency, blockIdx.y: d,
// blockIdx.z: grid; each grid has its own wavenumbers)
__global__ void __launch_bounds__(512) k_fft_yz(int nx, int ny, int nz, int nh, FftAxis ay, FftAxis az,
                                                const FftTables *__restrict__ tab,
                                                const float *__restrict__ ktab, float inv_ng,
                                                const float2 *in,
                                                float2 *__restrict__ out, int64_t nhalf, int mi, int mj,
                                                int mk, int mode_comp, int mode_conj,
                                                double *__restrict__ mode) {
    dep_begin(in, out, mode);
    in += blockIdx.z * nhalf;
    out += blockIdx.z * 3 * nhalf;
    ktab += blockIdx.z * (nh + 2 * (ny + nz));
    extern __shared__ float2 sm[];
    const int pitch = ny | 1, a = blockIdx.x, d = blockIdx.y;
    float2 *s = sm, *twy = sm + nz * pitch, *twz = twy + ny;
    load_twiddles(twy, tab, 1, ny);
    load_twiddles(twz, tab, 2, nz);
    load_plane(s, in + (int64_t)a * ny * nz, ny, nz, pitch);
    __syncthreads();
    lines<false>(s, nz, pitch, 1, ay, twy);
    lines<false>(s, ny, 1, pitch, az, twz);
    const float *kyp = ktab + nh, *gyp = kyp + ny, *kzp = gyp + ny, *gzp = kzp + nz;
    const float kx = ktab[a];
    const float gx = ((nx & 1) == 0 && a == nx / 2) ? 0.0f : kx;
    const fft::FastDiv by_ny(ny);
    for (int w = threadIdx.x; w < ny * nz; w += blockDim.x) {
        const int pz = by_ny.quot(w), py = w - pz * ny;
        const float ky = kyp[py], kz = kzp[pz];
        float2 &e = s[pz * pitch + py];
        const float2 rh = e;
        float2 v = make_float2(0.f, 0.f);
        if ((a | py | pz) != 0) {   // frequency 0 stays at position 0
            const float sc = inv_ng / (kx * kx + ky * ky + kz * kz) *
                             (d == 0 ? gx : (d == 1 ? gyp[py] : gzp[pz]));
            v = make_float2(sc * rh.y, -sc * rh.x);   // -i g rh
        }
        e = v;
        if (d == mode_comp && a == mi && py == mj && pz == mk) {
            mode[2 * blockIdx.z] = (double)v.x;
            mode[2 * blockIdx.z + 1] = mode_conj ? -(double)v.y : (double)v.y;
        }
    }
    __syncthreads();
    lines<true>(s, ny, 1, pitch, az, twz);
    lines<true>(s, nz, pitch, 1, ay, twy);
    float2 *o = out + d * nhalf + (int64_t)a * ny * nz;
    store_plane(o, s, ny, nz, pitch);
}

// lrho^ = sum_d (+i g_d / |k|^2) lE^_d / N_g of one x frequency, in two kernels: a
// block per component transforms its plane forward in place and applies +i g_d
// (blockIdx.y: d), then a block adds the three, applies 1 / (|k|^2 N_g) and
// transforms back.  One block for all four planes took 43 us at 64^3 (33 blocks),
// the two kernels 27.
__global__ void __launch_bounds__(512) k_fft_yz_adj(int nx, int ny, int nz, int nh, FftAxis ay,
                                                    FftAxis az, const FftTables *__restrict__ tab,
                                                    const float *__restrict__ ktab,
                                                    float2 *lE_hat, int64_t nhalf) {
    dep_begin(lE_hat);
    extern __shared__ float2 sm[];
    const int pitch = ny | 1, a = blockIdx.x, d = blockIdx.y;
    float2 *s = sm, *twy = sm + nz * pitch, *twz = twy + ny;
    float2 *io = lE_hat + d * nhalf + (int64_t)a * ny * nz;
    load_twiddles(twy, tab, 1, ny);
    load_twiddles(twz, tab, 2, nz);
    load_plane(s, io, ny, nz, pitch);
    __syncthreads();
    lines<false>(s, nz, pitch, 1, ay, twy);
    lines<false>(s, ny, 1, pitch, az, twz);
    const float *gyp = ktab + nh + ny, *gzp = gyp + ny + nz;
    const float gx = ((nx & 1) == 0 && a == nx / 2) ? 0.0f : ktab[a];
    const fft::FastDiv by_ny(ny);
    for (int w = threadIdx.x; w < ny * nz; w += blockDim.x) {
        const int pz = by_ny.quot(w), py = w - pz * ny;
        const float g = d == 0 ? gx : (d == 1 ? gyp[py] : gzp[pz]);
        const float2 e = s[pz * pitch + py];
        io[w] = make_float2(-g * e.y, g * e.x);   // +i g e
    }
}

__global__ void __launch_bounds__(512) k_fft_yz_adj_back(int ny, int nz, int nh, FftAxis ay, FftAxis az,
                                                         const FftTables *__restrict__ tab,
                                                         const float *__restrict__ ktab, float inv_ng,
                                                         const float2 *lE_hat,
                                                         float2 *__restrict__ out, int64_t nhalf) {
    dep_begin(lE_hat, out);
    extern __shared__ float2 sm[];
    const int pitch = ny | 1, a = blockIdx.x;
    float2 *s = sm, *twy = sm + nz * pitch, *twz = twy + ny;
    load_twiddles(twy, tab, 1, ny);
    load_twiddles(twz, tab, 2, nz);
    const float2 *in = lE_hat + (int64_t)a * ny * nz;
    const float *kyp = ktab + nh, *kzp = kyp + 2 * ny;
    const float kx = ktab[a];
    const fft::FastDiv by_ny(ny);
    for (int w = threadIdx.x; w < ny * nz; w += blockDim.x) {
        const int pz = by_ny.quot(w), py = w - pz * ny;
        const float ky = kyp[py], kz = kzp[pz];
        const float2 v = fft::cadd(fft::cadd(in[w], in[w + nhalf]), in[w + 2 * nhalf]);
        const float sc = (a | py | pz) != 0 ? inv_ng / (kx * kx + ky * ky + kz * kz) : 0.0f;
        s[pz * pitch + py] = make_float2(sc * v.x, sc * v.y);
    }
    __syncthreads();
    lines<true>(s, ny, 1, pitch, az, twz);
    lines<true>(s, nz, pitch, 1, ay, twy);
    store_plane(out + (int64_t)a * ny * nz, s, ny, nz, pitch);
}

// rows y0.. of plane z of COMPS components, from spectra by x frequency to two
// real rows per complex line in shared memory
template <int COMPS>
__device__ __forceinline__ void rows_backward(float2 *s, float2 *tw, const float2 *in,
                                              int64_t nhalf, int ny, int nz, int nh, int z, int y0,
                                              int rows, const FftAxis &ax,
                                              const FftTables *__restrict__ tab) {
    constexpr int PAIRS = kRowsB / 2;
    const int n = ax.n, pitch = n | 1;
    load_twiddles(tw, tab, 0, n);
    const fft::FastDiv by_nh(nh);
    for (int w = threadIdx.x; w < COMPS * nh * PAIRS; w += kXThreads) {
        const int q = w % PAIRS, u = w / PAIRS;
        const int d = COMPS == 1 ? 0 : by_nh.quot(u), k = u - d * nh;
        const float2 *p = in + d * nhalf + ((int64_t)k * nz + z) * ny + y0;
        float2 a = make_float2(0.f, 0.f), b = a;
        if (2 * q < rows) a = p[2 * q];
        if (2 * q + 1 < rows) b = p[2 * q + 1];
        if (k == 0 || 2 * k == n) a.y = b.y = 0.0f;   // real for a real row
        float2 *line = s + (d * PAIRS + q) * pitch;
        line[tab->pos[0][k]] = make_float2(a.x - b.y, a.y + b.x);   // A + i B
        if (k != 0 && 2 * k != n)
            line[tab->pos[0][n - k]] = make_float2(a.x + b.y, b.x - a.y);   // A* + i B*
    }
    __syncthreads();
    lines<true>(s, COMPS * PAIRS, pitch, 1, ax, tw);
}

// fpart: the block's sums in FP64 (20 steps with records of 64^3 x 16 3.13 ms; in FP32
// pairs, which are off by 8e-16 there, 3.11)
__global__ void __launch_bounds__(kXThreads) k_fft_x_backward(int ny, int nz, int nh, FftAxis ax,
                                                              const FftTables *__restrict__ tab,
                                                              const float2 *in,
                                                              int64_t nhalf, float4 *__restrict__ E4,
                                                              float4 *__restrict__ E8,
                                                              float *__restrict__ rho, bool clear_rho,
                                                              double *__restrict__ fpart, int fstride) {
    dep_begin(in, E4, E8, rho, fpart);
    const int64_t grid0 = blockIdx.z * ((int64_t)ax.n * ny * nz);
    in += blockIdx.z * 3 * nhalf;
    if (E4) E4 += grid0;
    E8 += 2 * grid0;
    rho += grid0;
    constexpr int PAIRS = kRowsB / 2;
    extern __shared__ float2 sm[];
    const int n = ax.n, pitch = n | 1;
    const int z = blockIdx.y, y0 = blockIdx.x * kRowsB, rows = min(kRowsB, ny - y0);
    rows_backward<3>(sm, sm + 3 * PAIRS * pitch, in, nhalf, ny, nz, nh, z, y0, rows, ax, tab);
    const float *sf = reinterpret_cast<const float *>(sm);
    double sums[4] = {0.0, 0.0, 0.0, 0.0};
    const fft::FastDiv by_n(n);
    for (int w = threadIdx.x; w < rows * n; w += kXThreads) {
        const int r = by_n.quot(w), x = w - r * n, x1 = x + 1 == n ? 0 : x + 1;
        const float *f0 = sf + 2 * ((r >> 1) * pitch) + (r & 1);
        const float *f1 = f0 + 2 * PAIRS * pitch, *f2 = f1 + 2 * PAIRS * pitch;
        const float4 e = make_float4(f0[2 * x], f1[2 * x], f2[2 * x], 0.0f);
        const int64_t g = ((int64_t)z * ny + y0 + r) * n + x;
        if (E4) E4[g] = e;
        E8[2 * g] = make_float4(e.x, e.y, f0[2 * x1], f1[2 * x1]);
        E8[2 * g + 1] = make_float4(e.z, f2[2 * x1], 0.0f, 0.0f);
        if (fpart) add_field(sums, e, rho[g]);
        if (clear_rho) rho[g] = 0.0f;
    }
    if (fpart)
        block_field_sums<kXThreads>(sums, fpart + 4 * ((int64_t)blockIdx.z * fstride +
                                                       blockIdx.y * gridDim.x + blockIdx.x));
}

// lrho rows -> the x-paired copy read by the deposit-term gathers; the largest
// |lrho| goes to adj_lrho[par], and the slots of the next reverse push are cleared
__global__ void __launch_bounds__(kXThreads) k_fft_x_backward_adj(int ny, int nz, int nh, FftAxis ax,
                                                                  const FftTables *__restrict__ tab,
                                                                  const float2 *in,
                                                                  float2 *__restrict__ lrho2, Ctrl *ctrl,
                                                                  int par) {
    dep_begin(in, lrho2, ctrl);
    constexpr int PAIRS = kRowsB / 2;
    extern __shared__ float2 sm[];
    const int n = ax.n, pitch = n | 1;
    const int z = blockIdx.y, y0 = blockIdx.x * kRowsB, rows = min(kRowsB, ny - y0);
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
        ctrl->adj_ly[par ^ 1] = 0u;
        ctrl->adj_lv[par ^ 1] = 0u;
    }
    rows_backward<1>(sm, sm + PAIRS * pitch, in, 0, ny, nz, nh, z, y0, rows, ax, tab);
    const float *sf = reinterpret_cast<const float *>(sm);
    float m = 0.0f;
    const fft::FastDiv by_n(n);
    for (int w = threadIdx.x; w < rows * n; w += kXThreads) {
        const int r = by_n.quot(w), x = w - r * n, x1 = x + 1 == n ? 0 : x + 1;
        const float *f = sf + 2 * ((r >> 1) * pitch) + (r & 1);
        lrho2[((int64_t)z * ny + y0 + r) * n + x] = make_float2(f[2 * x], f[2 * x1]);
        m = fmaxf(m, fabsf(f[2 * x]));
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0 && m > 0.0f) atomicMax(&ctrl->adj_lrho[par], __float_as_uint(m));
}

// Split n into the radices of fft.cuh, fewest stages first.  (Stages of larger
// primes as plain sums lost: 78 x 88 x 91 took 139 us against cuFFT's 76.)
void split(int m, int depth, int *cur, int &best, int &best_sum, FftAxis &a) {
    if (m == 1) {
        int sum = 0;
        for (int i = 0; i < depth; ++i) sum += cur[i];
        // a lone 16 leaves one thread a line: two stages of 4 keep more busy
        if (depth == 1 && cur[0] == 16) depth = 2, cur[0] = cur[1] = 4, sum = 8;
        if (depth < best || (depth == best && sum < best_sum)) {
            best = depth;
            best_sum = sum;
            a.stages = depth;
            for (int i = 0; i < depth; ++i) a.radix[i] = cur[i];
        }
        return;
    }
    if (depth >= kFftMaxStages) return;
    for (int r : {16, 8, 7, 6, 5, 4, 3, 2}) {
        if (m % r != 0 || (depth > 0 && r > cur[depth - 1])) continue;
        cur[depth] = r;
        split(m / r, depth + 1, cur, best, best_sum, a);
    }
}

size_t yz_smem(const Geom &g) {
    return sizeof(float2) * ((size_t)g.n[2] * (g.n[1] | 1) + g.n[1] + g.n[2]);
}
size_t x_smem(const Geom &g, int line_count) {
    return sizeof(float2) * ((size_t)line_count * (g.n[0] | 1) + g.n[0]);
}
int yz_threads(const Geom &g) {
    const int pts = g.n[1] * g.n[2];
    return pts >= 2048 ? 512 : (pts >= 1024 ? 256 : 128);
}

}  // namespace

bool fft_axis(int n, FftAxis &a) {
    a = FftAxis{};
    a.n = n;
    if (n < 1 || n > kFftMaxN) return false;
    int best = kFftMaxStages + 1, best_sum = 0, cur[kFftMaxStages];
    split(n, 0, cur, best, best_sum, a);
    return best <= kFftMaxStages;
}

void fft_tables(const FftAxis ax[3], FftTables &t) {
    for (int d = 0; d < 3; ++d) {
        const int n = ax[d].n;
        for (int k = 0; k < n; ++k) {
            const double phi = -2.0 * 3.14159265358979323846 * k / n;
            t.tw[d][k] = make_float2((float)cos(phi), (float)sin(phi));
            int f = k, p = 0, m = n;
            for (int i = 0; i < ax[d].stages; ++i) {
                m /= ax[d].radix[i];
                p += (f % ax[d].radix[i]) * m;
                f /= ax[d].radix[i];
            }
            t.pos[d][k] = p;
        }
    }
}

// Planes of at most 96^2 points: 96^3 solves take 55 us against 63 through cuFFT,
// 64^3 33 against 47, 16^3 23 against 33 (200 in a row); at 128^3 the 195 blocks
// of one per SM make two rounds and take 157 against 102 (with sums, cold caches).
bool fft_supported(const Geom &g, FftAxis ax[3]) {
    for (int d = 0; d < 3; ++d)
        if (!fft_axis(g.n[d], ax[d])) return false;
    return g.n[1] * g.n[2] <= 96 * 96;
}

// x: nh wavenumbers; y and z: those at each position, then the gradient's (zero at
// the Nyquist frequency)
int fft_ktab_size(const Geom &g) { return g.nh + 2 * (g.n[1] + g.n[2]); }
void fft_ktab(const Geom &g, const double *L_d, const FftTables &t, float *out) {
    std::vector<float> k((size_t)(g.nh + g.n[1] + g.n[2]));
    green_table(g, L_d, k.data());
    for (int a = 0; a < g.nh; ++a) out[a] = k[a];
    float *o = out + g.nh;
    int off = g.nh;
    for (int d = 1; d < 3; ++d) {
        const int n = g.n[d];
        for (int f = 0; f < n; ++f) {
            const int p = t.pos[d][f];
            o[p] = k[off + f];
            o[n + p] = (n & 1) == 0 && f == n / 2 ? 0.0f : k[off + f];
        }
        o += 2 * n;
        off += n;
    }
}

int fft_sum_blocks(const Geom &g) { return (g.n[1] + kRowsB - 1) / kRowsB * g.n[2]; }

cudaError_t fft_prepare() {
    cudaError_t e;
    // the largest plane of fft_supported, its rows padded: 128 x (72 | 1) points
    const int most = (int)(sizeof(float2) * (96 * 96 + 128 + 2 * kFftMaxN));
    if ((e = cudaFuncSetAttribute(k_fft_yz, cudaFuncAttributeMaxDynamicSharedMemorySize, most)) != cudaSuccess)
        return e;
    if ((e = cudaFuncSetAttribute(k_fft_yz_adj, cudaFuncAttributeMaxDynamicSharedMemorySize, most)) !=
        cudaSuccess)
        return e;
    return cudaFuncSetAttribute(k_fft_yz_adj_back, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
}

cudaError_t launch_fft_solve(const Geom &g, int m, const FftAxis ax[3], const FftTables *tab,
                             const float *ktab, float *rho, bool clear_rho, float2 *rho_hat, float2 *E_hat,
                             int64_t nhalf, const int *mode_idx, int mode_comp, int mode_conj,
                             double *mode, float4 *E4, float4 *E8, double *fpart, int fstride,
                             LStream st) {
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
    const float inv_ng = (float)(1.0 / ((double)nx * ny * nz));
    launch_dep(k_fft_x_forward<1>, dim3((ny + kRowsF - 1) / kRowsF, nz, m), kXThreads, x_smem(g, kRowsF / 2), st, 
        ny, nz, g.nh, ax[0], tab, rho, nullptr, rho_hat, nhalf);
    launch_dep(k_fft_yz, dim3(g.nh, 3, m), yz_threads(g), yz_smem(g), st, nx, ny, nz, g.nh, ax[1], ax[2], tab, ktab,
                                                                 inv_ng, rho_hat, E_hat, nhalf, mode_idx[0],
                                                                 mode_idx[1], mode_idx[2], mode_comp,
                                                                 mode_conj, mode);
    launch_dep(k_fft_x_backward, dim3((ny + kRowsB - 1) / kRowsB, nz, m), kXThreads, x_smem(g, 3 * kRowsB / 2), st,
               ny, nz, g.nh, ax[0], tab, E_hat, nhalf, E4, E8, rho, clear_rho, fpart, fstride);
    return cudaGetLastError();
}

cudaError_t launch_fft_adj_solve(const Geom &g, const FftAxis ax[3], const FftTables *tab,
                                 const float *ktab, float4 *lE4, float2 *lE_hat, float2 *lrho_hat,
                                 int64_t nhalf, float2 *lrho2, Ctrl *ctrl, int par, LStream st) {
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
    const float inv_ng = (float)(1.0 / ((double)nx * ny * nz));
    const dim3 rows((ny + kRowsB - 1) / kRowsB, nz);
    launch_dep(k_fft_x_forward<3>, rows, kXThreads, x_smem(g, 3 * kRowsB / 2), st, ny, nz, g.nh, ax[0], tab, nullptr,
                                                                           lE4, lE_hat, nhalf);
    launch_dep(k_fft_yz_adj, dim3(g.nh, 3), yz_threads(g), yz_smem(g), st, nx, ny, nz, g.nh, ax[1], ax[2], tab, ktab,
                                                                  lE_hat, nhalf);
    launch_dep(k_fft_yz_adj_back, g.nh, yz_threads(g), yz_smem(g), st, ny, nz, g.nh, ax[1], ax[2], tab, ktab, inv_ng,
                                                              lE_hat, lrho_hat, nhalf);
    launch_dep(k_fft_x_backward_adj, rows, kXThreads, x_smem(g, kRowsB / 2), st, ny, nz, g.nh, ax[0], tab, lrho_hat,
                                                                         lrho2, ctrl, par);
    return cudaGetLastError();
}

}  // namespace pic
