// The per-particle gather + Boris push + drift of Section 3.1 steps 3-4
// (Eq. momentum_eqn) and Section 3.2 of arXiv 2205.11052, shared by the
// single-run and the batched kernels.
//
// E is interpolated to the particle with the CIC weights of the deposit, the
// velocity is advanced by the Boris rotation (exact solution of
// v1 = v0 + dt (q/m) [e + (v0 + v1)/2 x B]) and the position drifts by a full
// step in cell units, carried into the cell index and wrapped periodically.
#pragma once

#include "cic.cuh"
#include "ffsum.cuh"
#include "pic_internal.cuh"
#include "records.cuh"

namespace pic {

__device__ __forceinline__ void advance_cells(const Geom &g, float sx, float sy, float sz, int &i,
                                              int &j, int &k, int32_t &c, float &fx, float &fy,
                                              float &fz, int &bad, int (&step)[3]);

// Velocity moments (sum v, sum |v|^2) are summed per thread in FP32 over a few
// particles (as many as a tile takes without a fold, or one loop iteration), those
// sums in (hi, lo) pairs that carry their rounding errors, and the threads in
// FP64.  (With FP64 totals per thread the folds kept the scarce FP64 units busy:
// 134M particles with records 2.31 ms a push, now 2.28.  The kinetic energy of 33
// thousand to 134M particles is off by 1e-11 to 4e-10 of the FP64 sum of the same
// velocities, with FP64 totals by 1e-11 to 3e-9: the FP32 sums decide.)
struct Moments {
    float a[4] = {0.f, 0.f, 0.f, 0.f};
    float hi[4] = {0.f, 0.f, 0.f, 0.f}, lo[4] = {0.f, 0.f, 0.f, 0.f};
    __device__ __forceinline__ void add(float vx, float vy, float vz) {
        a[0] += vx;
        a[1] += vy;
        a[2] += vz;
        a[3] += vx * vx + vy * vy + vz * vz;
    }
    __device__ __forceinline__ void fold() {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            ff_add(hi[q], lo[q], a[q]);
            a[q] = 0.f;
        }
    }
    __device__ __forceinline__ double total(int q) const { return widen(hi[q]) + widen(lo[q]); }
};

// The warp's sums of the four totals: lane 8 q returns the q-th (each lane's four
// summed over the warp by themselves took 24 FP64 additions and 8 conversions: the push
// of 4.2M particles 90.3 us, so 88.6)
__device__ __forceinline__ double warp_total(const Moments &mo) {
    const double t[4] = {mo.total(0), mo.total(1), mo.total(2), mo.total(3)};
    return warp_sums(t);
}

// One (y, z) row of a stencil: Ex and Ey at its two x corners, and the two Ez
struct ERow {
    float2 a, b, z;
};
__device__ __forceinline__ ERow row_of(const float4 &e0, const float4 &e1) {
    return ERow{make_float2(e0.x, e0.y), make_float2(e1.x, e1.y), make_float2(e0.z, e1.z)};
}

// CIC interpolation of the rows (corner bits b | c<<1).  The roundings are written out, so
// that every kernel that pushes a particle gives the same bits: a step and the split
// calls can be compared exactly.  (In packed pairs of FP32 operations, Ez's two x corners
// side by side, the split push is 4% faster, 8 steps of the split cycle on 64^3 x 64 in
// 4.10 ms and not 4.26, but rounds otherwise; with Ex and Ey alone packed, which does
// not, it gains nothing.)
__device__ __forceinline__ float lerp_x(float gx, float a, float fx, float b) {
    return __fmaf_rn(gx, a, __fmul_rn(fx, b));
}
__device__ __forceinline__ float sum_rows(const float (&w)[4], const float (&v)[4]) {
    return __fmaf_rn(w[3], v[3], __fmaf_rn(w[2], v[2], __fmaf_rn(w[0], v[0], __fmul_rn(w[1], v[1]))));
}
__device__ __forceinline__ void row_weights(float fy, float fz, float (&w)[4]) {
    const float gy = 1.0f - fy, gz = 1.0f - fz;
    w[0] = __fmul_rn(gy, gz);
    w[1] = __fmul_rn(fy, gz);
    w[2] = __fmul_rn(gy, fz);
    w[3] = __fmul_rn(fy, fz);
}
__device__ __forceinline__ void interp_E(const ERow r[4], float fx, float fy, float fz, float &ex,
                                         float &ey, float &ez) {
    const float gx = 1.0f - fx;
    float w[4], vx[4], vy[4], vz[4];
    row_weights(fy, fz, w);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        vx[q] = lerp_x(gx, r[q].a.x, fx, r[q].b.x);
        vy[q] = lerp_x(gx, r[q].a.y, fx, r[q].b.y);
        vz[q] = lerp_x(gx, r[q].z.x, fx, r[q].z.y);
    }
    ex = sum_rows(w, vx);
    ey = sum_rows(w, vy);
    ez = sum_rows(w, vz);
}

// E8 holds, per node q, E at q and (primed) at its +x neighbour (periodic) as Ex
// Ey Ex' Ey' Ez Ez' and two unused floats, so each of the four (y, z) corner rows of the
// stencil is one aligned 256-bit load
__device__ __forceinline__ void ld_pair(const float4 *p, float4 &a, float4 &b) {
    asm("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(a.x), "=f"(a.y), "=f"(b.x), "=f"(b.y), "=f"(a.z), "=f"(b.z), "=f"(a.w), "=f"(b.w)
        : "l"(p));
}

__device__ __forceinline__ void gather_E_pairs(const Geom &g, const float4 *E8, int i,
                                               int j, int k, float fx, float fy, float fz,
                                               float &ex, float &ey, float &ez) {
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
    const int j1 = (j + 1 == ny) ? 0 : j + 1;
    const int k1 = (k + 1 == nz) ? 0 : k + 1;
    const int nxy = nx * ny;
    const int r00 = j * nx + k * nxy + i, r10 = j1 * nx + k * nxy + i;
    const int r01 = j * nx + k1 * nxy + i, r11 = j1 * nx + k1 * nxy + i;
    const int at[4] = {r00, r10, r01, r11};
    ERow r[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float4 e0, e1;
        ld_pair(E8 + 2 * (int64_t)at[q], e0, e1);
        r[q] = row_of(e0, e1);
    }
    interp_E(r, fx, fy, fz, ex, ey, ez);
}

// E at the particle from a copy of the field on a box in shared memory (one
// float4 per slot; s0 is the stencil base's slot, rows S0 slots apart in y,
// planes S01 apart in z)
__device__ __forceinline__ void gather_E_box(const float4 *sE, int s0, int S0, int S01, float fx,
                                             float fy, float fz, float &ex, float &ey,
                                             float &ez) {
    const ERow r[4] = {row_of(sE[s0], sE[s0 + 1]), row_of(sE[s0 + S0], sE[s0 + S0 + 1]),
                       row_of(sE[s0 + S01], sE[s0 + S01 + 1]),
                       row_of(sE[s0 + S01 + S0], sE[s0 + S01 + S0 + 1])};
    interp_E(r, fx, fy, fz, ex, ey, ez);
}

// Boris kick with the interpolated field (plus the external quadrupole), then
// a full drift in cell units carried into the cell index and wrapped; (i, j, k)
// is the particle's stencil base before the step and after it, step the cells it
// moved (before the wrap)
template <bool EXT, bool MAG>
__device__ __forceinline__ void kick_drift(const Geom &g, const PushConst &pc, float ex, float ey,
                                           float ez, int &i, int &j, int &k, int32_t &c, float &fx,
                                           float &fy, float &fz, float &vx, float &vy, float &vz,
                                           int &bad, int (&step)[3]) {
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
    if (EXT) {
        // quadrupole about the box centre at x in [0, L): (x - c)/h = i - N/2 +
        // 1/2 + f, wrapped into [-N/2, N/2) (a particle in [0, h/2) has its
        // stencil base on node N-1, i.e. i + 1/2 + f lies in [N, N + 1/2))
        float ux = (float)i - pc.half_n[0] + 0.5f + fx;
        float uy = (float)j - pc.half_n[1] + 0.5f + fy;
        float uz = (float)k - pc.half_n[2] + 0.5f + fz;
        if (ux >= pc.half_n[0]) ux -= (float)nx;
        if (uy >= pc.half_n[1]) uy -= (float)ny;
        if (uz >= pc.half_n[2]) uz -= (float)nz;
        ex += -0.5f * pc.wz2 * (ux * g.h[0]);
        ey += -0.5f * pc.wz2 * (uy * g.h[1]);
        ez += pc.wz2 * (uz * g.h[2]);
    }
    // Boris: half kick, rotation, half kick
    float mx = vx + pc.qm_half_dt * ex;
    float my = vy + pc.qm_half_dt * ey;
    float mz = vz + pc.qm_half_dt * ez;
    if (MAG) {
        const float px = mx + (my * pc.t[2] - mz * pc.t[1]);
        const float py = my + (mz * pc.t[0] - mx * pc.t[2]);
        const float pz = mz + (mx * pc.t[1] - my * pc.t[0]);
        mx += py * pc.s[2] - pz * pc.s[1];
        my += pz * pc.s[0] - px * pc.s[2];
        mz += px * pc.s[1] - py * pc.s[0];
    }
    vx = mx + pc.qm_half_dt * ex;
    vy = my + pc.qm_half_dt * ey;
    vz = mz + pc.qm_half_dt * ez;

    // drift a full step in cell units, carry into the cell index, wrap
    advance_cells(g, fx + pc.dt_over_h[0] * vx, fy + pc.dt_over_h[1] * vy,
                  fz + pc.dt_over_h[2] * vz, i, j, k, c, fx, fy, fz, bad, step);
}

// New in-cell offsets s (in cell units, relative to the stencil base
// (i, j, k)): carry floor(s) into the cell index, keep the fraction, wrap
// periodically, repack the cell; (i, j, k) become the new stencil base, step the
// carries
__device__ __forceinline__ void advance_cells(const Geom &g, float sx, float sy, float sz, int &i,
                                              int &j, int &k, int32_t &c, float &fx, float &fy,
                                              float &fz, int &bad, int (&step)[3]) {
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
    float flx = floorf(sx), fly = floorf(sy), flz = floorf(sz);
    fx = sx - flx;
    fy = sy - fly;
    fz = sz - flz;
    if (fx >= 1.0f) { fx = 0.0f; flx += 1.0f; }
    if (fy >= 1.0f) { fy = 0.0f; fly += 1.0f; }
    if (fz >= 1.0f) { fz = 0.0f; flz += 1.0f; }
    if (!(fabsf(flx) < 1.0e6f && fabsf(fly) < 1.0e6f && fabsf(flz) < 1.0e6f)) {
        bad |= PIC_FLAG_NONFINITE;
        flx = fly = flz = 0.0f;
        fx = fy = fz = 0.0f;
    }
    step[0] = (int)flx;
    step[1] = (int)fly;
    step[2] = (int)flz;
    i += step[0];
    j += step[1];
    k += step[2];
    if ((unsigned)i >= (unsigned)nx) { i %= nx; if (i < 0) i += nx; }
    if ((unsigned)j >= (unsigned)ny) { j %= ny; if (j < 0) j += ny; }
    if ((unsigned)k >= (unsigned)nz) { k %= nz; if (k < 0) k += nz; }
    c = pack_cell(i, j, k);
}

// stencil base of a packed cell (flagged and clamped to 0 if out of range)
__device__ __forceinline__ void decode_base(const Geom &g, int32_t c, int &i, int &j, int &k,
                                            int &bad) {
    i = cell_i(c);
    j = cell_j(c);
    k = cell_k(c);
    if (i >= g.n[0] || j >= g.n[1] || k >= g.n[2]) {   // never produced by the kernels
        bad |= PIC_FLAG_BAD_CELL;
        i = j = k = 0;
    }
}

// gather from the x-paired grid + kick + drift; (i, j, k) receives the new
// stencil base (the fields of the new packed cell c)
template <bool EXT, bool MAG>
__device__ __forceinline__ void push_one_pairs(const Geom &g, const PushConst &pc,
                                               const float4 *E8, int32_t &c,
                                               float &fx, float &fy, float &fz, float &vx,
                                               float &vy, float &vz, int &bad, int &i, int &j,
                                               int &k) {
    decode_base(g, c, i, j, k, bad);
    float ex, ey, ez;
    gather_E_pairs(g, E8, i, j, k, fx, fy, fz, ex, ey, ez);
    int step[3];
    kick_drift<EXT, MAG>(g, pc, ex, ey, ez, i, j, k, c, fx, fy, fz, vx, vy, vz, bad, step);
}

template <bool EXT, bool MAG>
__device__ __forceinline__ void push_one_pairs(const Geom &g, const PushConst &pc,
                                               const float4 *E8, int32_t &c,
                                               float &fx, float &fy, float &fz, float &vx,
                                               float &vy, float &vz, int &bad) {
    int i, j, k;
    push_one_pairs<EXT, MAG>(g, pc, E8, c, fx, fy, fz, vx, vy, vz, bad, i, j, k);
}

// E at the particle from the x-paired copy of the box (cic::stage_pairs): the
// four (y, z) rows of the stencil cost a 16-byte and an 8-byte shared load each,
// 24 bytes a row against two 16-byte loads of whole nodes.  Lanes at random slots
// collide in the banks, so the wavefronts go with the bytes: about 67 per warp and
// gather, 85 with whole nodes.
template <int B = 0>
__device__ __forceinline__ void gather_E_pair_box(const float4 *sA, const float2 *sB, int s0, int S0r,
                                                  int S01r, float fx, float fy, float fz, float &ex,
                                                  float &ey, float &ez) {
    const int S0 = B > 0 ? B : S0r, S01 = B > 0 ? B * B : S01r;   // B > 0: a constant box
    const int off[4] = {0, S0, S01, S01 + S0};
    ERow r[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float4 a = sA[s0 + off[q]];
        r[q] = ERow{make_float2(a.x, a.y), make_float2(a.z, a.w), sB[s0 + off[q]]};
    }
    interp_E(r, fx, fy, fz, ex, ey, ez);
}

// Gather + kick + drift with E read from sE, the block's shared-memory copy
// of the box of tile t (cic::stage_box), when the particle's stencil lies in
// that box: eight 16-byte shared loads, a few shared wavefronts per warp
// instead of one L1 wavefront per particle and 32-byte global read.  Other
// particles, and every particle when sE is null, read the x-paired grid E8.
// (i, j, k) receives the new stencil base.
template <bool EXT, bool MAG>
__device__ __forceinline__ void push_one_staged(const Geom &g, const PushConst &pc,
                                                const float4 *E8, const float4 *sE,
                                                const cic::Tile &t, int32_t &c, float &fx,
                                                float &fy, float &fz, float &vx, float &vy,
                                                float &vz, int &bad, int &i, int &j, int &k) {
    decode_base(g, c, i, j, k, bad);
    float ex, ey, ez;
    int s0;
    if (sE != nullptr && cic::box_base(t, g, i, j, k, s0))
        gather_E_box(sE, s0, t.S0, t.S01, fx, fy, fz, ex, ey, ez);
    else
        gather_E_pairs(g, E8, i, j, k, fx, fy, fz, ex, ey, ez);
    int step[3];
    kick_drift<EXT, MAG>(g, pc, ex, ey, ez, i, j, k, c, fx, fy, fz, vx, vy, vz, bad, step);
}

}  // namespace pic
