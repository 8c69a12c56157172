// Field solve (Section 3.1 step 2, Eq. potential; Section 3.2 of
// arXiv 2205.11052) and the FP64 diagnostic reductions.
//
// Around cuFFT's R2C / C2R transforms, k_green maps the charge spectrum to
// the three field spectra:  -Lap(phi) = rho - rho_i (eps0 = 1), E = -grad(phi)
//   E^_d(m) = -i k_d rho^(m) / |k|^2 / N_g,   k_d = 2 pi m_d / L_d,
// with |k|^2 over the continuous wavenumbers (m_d in [-N_d/2, N_d/2)), the
// k = 0 mode (the uniform ion background) set to zero and each axis' Nyquist
// component of the gradient set to zero so E stays real.  The 1/N_g of the
// inverse transform is folded in here.  k_pack_E turns what the transform leaves into
// the x-paired field that the gathers read (32 bytes a node).
//
// Diagnostics (figures of Section 4): W_d = h^3 sum_g E_d^2, Q = h^3 sum_g rho,
// per thread in FP32 pairs that carry their rounding errors (ffsum.cuh), from there on
// in FP64, in a fixed order.
#include <math.h>

#include "ffsum.cuh"
#include "pic_internal.cuh"

namespace pic {

namespace {

// One thread per coefficient of an x-row (a) of the half spectrum; the row
// (b, c) comes from the block's y and z indices, so no index is divided.
// ktab holds the FP32 wavenumbers of every FFT index per axis (x: nh
// entries, then y: ny, then z: nz), rounded once from FP64 on the host.
__global__ void __launch_bounds__(128) k_green(int nx, int ny, int nz, int nh,
                                               const float *__restrict__ ktab, float inv_ng,
                                               const float2 *rho_hat,
                                               float2 *__restrict__ E_hat, int64_t nhalf, int mi,
                                               int mj, int mk, int mode_comp, int mode_conj,
                                               Ctrl *ctrl) {
    dep_begin(rho_hat, E_hat, ctrl);
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= nh) return;
    const int b = blockIdx.y, c = blockIdx.z;
    const int64_t q = ((int64_t)c * ny + b) * nh + a;
    const float kx = ktab[a], ky = ktab[nh + b], kz = ktab[nh + ny + c];
    const float gx = ((nx & 1) == 0 && a == nx / 2) ? 0.0f : kx;
    const float gy = ((ny & 1) == 0 && b == ny / 2) ? 0.0f : ky;
    const float gz = ((nz & 1) == 0 && c == nz / 2) ? 0.0f : kz;
    const float k2 = kx * kx + ky * ky + kz * kz;
    float2 ex = make_float2(0.f, 0.f), ey = ex, ez = ex;
    if (q != 0) {
        const float2 rh = rho_hat[q];
        const float sc = inv_ng / k2;
        // -i * g * rh = g * (rh.y, -rh.x)
        ex = make_float2(gx * sc * rh.y, -gx * sc * rh.x);
        ey = make_float2(gy * sc * rh.y, -gy * sc * rh.x);
        ez = make_float2(gz * sc * rh.y, -gz * sc * rh.x);
    }
    E_hat[q] = ex;
    E_hat[q + nhalf] = ey;
    E_hat[q + 2 * nhalf] = ez;
    if (a == mi && b == mj && c == mk) {
        const float2 m = (mode_comp == 0) ? ex : (mode_comp == 1 ? ey : ez);
        ctrl->mode[0] = (double)m.x;
        ctrl->mode[1] = mode_conj ? -(double)m.y : (double)m.y;
    }
}

__global__ void k_diag_finalize(const double *fpart, int fblocks,
                                const double *ppart, int pblocks, double dV,
                                double mp, double dt, Ctrl *ctrl, pic_diag_t *ring,
                                int ring_cap) {
    dep_begin(fpart, ppart, ctrl, ring);
    // one warp per quantity: strided sums per lane, then a fixed tree (a block
    // tree over 256 x 8 FP64 values took 9.6 us, mostly its 64 barriers' adds)
    __shared__ double red[8];
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    const double *part = q < 4 ? fpart + q : ppart + (q - 4);
    const int blocks = q < 4 ? fblocks : pblocks;
    double s = 0.0;
    for (int b = lane; b < blocks; b += 32) s += part[4 * b];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) red[q] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        const long long step = ctrl->step - 1;   // the push already advanced it
        pic_diag_t d;
        d.step = step;
        d.t_field = ((double)step + 0.5) * dt;
        d.Wx = dV * red[0];
        d.Wy = dV * red[1];
        d.Wz = dV * red[2];
        d.Q = dV * red[3];
        d.mode_re = ctrl->mode[0];
        d.mode_im = ctrl->mode[1];
        d.t = ((double)step + 1.0) * dt;
        d.Px = mp * red[4];
        d.Py = mp * red[5];
        d.Pz = mp * red[6];
        d.K = 0.5 * mp * red[7];
        const long long slot = ctrl->diag_written % ring_cap;
        ring[slot] = d;
        ctrl->diag_written += 1;
    }
}

}  // namespace

namespace {
// Field rows (component d of row r from planar + d * dist + r * pitch on, every
// ES-th float) -> the x-paired E8 read by 256-bit loads (the components at q, then those at
// its +x neighbour, periodic: Ex Ey Ex' Ey' | Ez Ez' 0 0) and, with SUMS, the
// block's partial sums of Ex^2, Ey^2, Ez^2 and rho.  Bound by DRAM: 12 bytes read
// and 32 written per node (16.8M nodes: 163 us; with E4 written too 246 us).  With
// the interleaving left to the inverse transform, as the gradient sweeps have it
// (output stride 4: 407 us against 92 planar), a pairing pass (120) and a pass for the
// sums (81), a 256^3 solve with sums took 0.85 ms.
template <int ES, bool SUMS>
__global__ void __launch_bounds__(256) k_pack_E(int nx, int64_t rows, int64_t pitch, int64_t dist,
                                                const float *planar,
                                                float4 *__restrict__ E8,
                                                float *__restrict__ rho, bool clear_rho,
                                                double *__restrict__ part) {
    dep_begin(planar, E8, rho, part);
    float hi[4] = {0.f, 0.f, 0.f, 0.f}, lo[4] = {0.f, 0.f, 0.f, 0.f};
    // one warp per row
    const int lane = threadIdx.x & 31;
    for (int64_t r = blockIdx.x * 8 + (threadIdx.x >> 5); r < rows; r += gridDim.x * 8) {
        const float *p0 = planar + r * pitch, *p1 = p0 + dist, *p2 = p1 + dist;
        for (int x = lane; x < nx; x += 32) {
            const int x1 = x + 1 == nx ? 0 : x + 1;
            const int64_t q = r * nx + x;
            const float4 e = make_float4(p0[ES * x], p1[ES * x], p2[ES * x], 0.0f);
            E8[2 * q] = make_float4(e.x, e.y, p0[ES * x1], p1[ES * x1]);
            E8[2 * q + 1] = make_float4(e.z, p2[ES * x1], 0.0f, 0.0f);
            if (SUMS) {
                ff_add_sq(hi[0], lo[0], e.x);
                ff_add_sq(hi[1], lo[1], e.y);
                ff_add_sq(hi[2], lo[2], e.z);
                ff_add(hi[3], lo[3], rho[q]);
            }
            if (clear_rho) rho[q] = 0.0f;
        }
    }
    if (SUMS) block_field_sums<256>(hi, lo, part + 4 * (int64_t)blockIdx.x);
}
}  // namespace

namespace {
// E8 -> one float4 (Ex, Ey, Ez, 0) per node, the layout of pic_get_field
__global__ void __launch_bounds__(256) k_unpair_E(int64_t ng, const float4 *E8,
                                                  float4 *__restrict__ E4) {
    dep_begin(E8, E4);
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= ng) return;
    const float4 a = E8[2 * q];
    E4[q] = make_float4(a.x, a.y, E8[2 * q + 1].x, 0.0f);
}
}  // namespace

cudaError_t launch_unpair_E(int64_t ng, const float4 *E8, float4 *E4, LStream st) {
    launch_dep(k_unpair_E, (unsigned)((ng + 255) / 256), 256, 0, st, ng, E8, E4);
    return cudaGetLastError();
}

cudaError_t launch_pack_E(const Geom &g, const float *E, bool interleaved, float4 *E8, float *rho,
                          bool clear_rho, double *part, LStream st) {
    const int64_t rows = (int64_t)g.n[1] * g.n[2];
    const int64_t pitch = interleaved ? 4 * (int64_t)g.n[0] : 2 * (int64_t)g.nh;
    const int64_t dist = interleaved ? 1 : pitch * rows;
#define PIC_PACK(ES, SUMS)                                                                          \
    launch_dep(k_pack_E<ES, SUMS>, kDiagFieldBlocks, 256, 0, st, g.n[0], rows, pitch, dist, E, E8, rho, \
               clear_rho, part)
    if (interleaved) { if (part) PIC_PACK(4, true); else PIC_PACK(4, false); }
    else             { if (part) PIC_PACK(1, true); else PIC_PACK(1, false); }
#undef PIC_PACK
    return cudaGetLastError();
}

void green_table(const Geom &g, const double *L_d, float *ktab) {
    const double two_pi = 6.283185307179586476925286766559;
    int o = 0;
    for (int a = 0; a < g.nh; ++a) ktab[o++] = (float)(two_pi / L_d[0] * a);
    for (int b = 0; b < g.n[1]; ++b) {
        const int m = (b <= g.n[1] / 2) ? b : b - g.n[1];
        ktab[o++] = (float)(two_pi / L_d[1] * m);
    }
    for (int c = 0; c < g.n[2]; ++c) {
        const int m = (c <= g.n[2] / 2) ? c : c - g.n[2];
        ktab[o++] = (float)(two_pi / L_d[2] * m);
    }
}

cudaError_t launch_green(const Geom &g, const float *ktab, const float2 *rho_hat, float2 *E_hat,
                         int64_t nhalf, const int *mode_idx, int mode_comp, int mode_conj,
                         Ctrl *ctrl, LStream st) {
    const double ng = (double)g.n[0] * g.n[1] * g.n[2];
    const int T = 128;
    const dim3 grid((unsigned)((g.nh + T - 1) / T), (unsigned)g.n[1], (unsigned)g.n[2]);
    launch_dep(k_green, grid, T, 0, st, g.n[0], g.n[1], g.n[2], g.nh, ktab, (float)(1.0 / ng), rho_hat,
                                E_hat, nhalf, mode_idx[0], mode_idx[1], mode_idx[2], mode_comp,
                                mode_conj, ctrl);
    return cudaGetLastError();
}

cudaError_t launch_diag_finalize(const double *field_part, int field_blocks,
                                 const double *push_part, int push_blocks, double dV, double mp, double dt, Ctrl *ctrl,
                                 pic_diag_t *ring, int ring_cap, LStream st) {
    launch_dep(k_diag_finalize, 1, 256, 0, st, field_part, field_blocks, push_part, push_blocks, dV,
                                       mp, dt, ctrl, ring, ring_cap);
    return cudaGetLastError();
}

}  // namespace pic
