// Particle kernels: load/normalise, readback, and the fused gather + push.
//
// Gather + push follows Section 3.1 steps 3-4 (Eq. momentum_eqn) and
// Section 3.2 of arXiv 2205.11052: E is interpolated to the particle with the
// CIC weights of the deposit, the velocity is advanced by the Boris rotation
// (exact solution of v1 = v0 + dt (q/m) [e + (v0 + v1)/2 x B]), and the
// position drifts by a full step, wrapped periodically.  The device keeps the
// drift-kick-drift state (x_{n+1/2}, v_n), so one pass takes x_{n+1/2} to
// x_{n+3/2} = x_{n+1/2} + dt v_{n+1}.
#include <math.h>

#include <algorithm>

#include "cic.cuh"
#include "push.cuh"
#include "records.cuh"

namespace pic {

namespace {

__device__ __forceinline__ void raise_flag(Ctrl *ctrl, int bit) { atomicOr(&ctrl->flags, bit); }

// ---------------------------------------------------------------------------
// load: FP64 (x_0, v_0) -> x_{1/2} = x_0 + dt/2 v_0 -> (cell, offset, v)
//
// From device memory it was bound by the FP64 units (about two lanes per clock and
// SM, conversions included): 4.2M particles 206 us; with the floor and the roundings
// by integer instructions 80 (its bytes 50).
// ---------------------------------------------------------------------------
constexpr int kLoadThreads = 256;

__global__ void __launch_bounds__(kLoadThreads) k_load(const double *__restrict__ x,
                                                      const double *__restrict__ v, int64_t m,
                                                      int64_t base, Geom g, double ih0,
                                                      double ih1, double ih2, double half_dt,
                                                      Ctrl *ctrl) {
    // the block's 256 (x, y, z) triples of x and of v are read as contiguous
    // runs (every byte once, six independent loads per thread) and staged in
    // shared memory: the source may be host memory read over the chip-to-chip
    // link, where strided 8-byte reads would fetch each line three times
    __shared__ double sx[3 * kLoadThreads], sv[3 * kLoadThreads];
    const ParticleSet ps = ctrl->sets[ctrl->cur];
    const double ih[3] = {ih0, ih1, ih2};
    bool any_bad = false;
    // blocks stride over runs of kLoadThreads particles
    for (int64_t p0 = (int64_t)blockIdx.x * kLoadThreads; p0 < m;
         p0 += (int64_t)gridDim.x * kLoadThreads) {
        const int cnt = (int)(m - p0 < kLoadThreads ? m - p0 : kLoadThreads);
        __syncthreads();   // the previous run's shared values are consumed
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const int j = r * kLoadThreads + threadIdx.x;
            if (j < 3 * cnt) {
                sx[j] = x[3 * p0 + j];
                sv[j] = v[3 * p0 + j];
            }
        }
        __syncthreads();
        if ((int)threadIdx.x >= cnt) continue;
        const int64_t p = p0 + threadIdx.x;
        double xr[3], vr[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            xr[d] = sx[3 * threadIdx.x + d];
            vr[d] = sv[3 * threadIdx.x + d];
        }
        int idx[3];
        float off[3];
        bool ok = true;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            double vd = vr[d];
            double xd = xr[d] + half_dt * vd;
            double s = xd * ih[d] - 0.5;      // node g at (g + 1/2) h
            // finite v and |s| < 2^52, tested on the exponent fields (FP64
            // instructions are scarce on this GPU; integer ones are not)
            const unsigned es =
                (unsigned)((unsigned long long)__double_as_longlong(s) >> 52) & 0x7ffu;
            const unsigned ev =
                (unsigned)((unsigned long long)__double_as_longlong(vd) >> 52) & 0x7ffu;
            if (es >= 1023u + 52u || ev == 0x7ffu) {
                ok = false;
                s = 0.0;
            }
            const FloorRest fr = floor_rest(s);
            long long il = fr.whole;
            float ff = fr.rest;
            if ((unsigned long long)il >= (unsigned long long)g.n[d]) {   // outside: wrap
                il += il < 0 ? g.n[d] : -g.n[d];
                if ((unsigned long long)il >= (unsigned long long)g.n[d]) {   // a box away
                    il %= g.n[d];
                    if (il < 0) il += g.n[d];
                }
            }
            if (ff >= 1.0f) {             // rounding to 1.0f moves to the next node
                ff = 0.0f;
                il += 1;
                if (il == g.n[d]) il = 0;
            }
            idx[d] = (int)il;
            off[d] = ff;
            ps.v[d][base + p] = ok ? narrow(vd) : 0.0f;
        }
        if (!ok) any_bad = true;
        ps.cell[base + p] = pack_cell(idx[0], idx[1], idx[2]);
        ps.o[0][base + p] = off[0];
        ps.o[1][base + p] = off[1];
        ps.o[2][base + p] = off[2];
        ps.pid[base + p] = (int32_t)(base + p);
    }
    if (any_bad) raise_flag(ctrl, PIC_FLAG_NONFINITE);
}

// ---------------------------------------------------------------------------
// synchronised readback x_n = x_{n+1/2} - dt/2 v_n in load order, in two
// passes through 32-byte records in the other particle set (its contents are
// dead between two re-binnings): k_unload_records reads the store in its own
// order and writes record pid, one full sector each; k_unload streams the
// records out as FP64 triples.
//
// Both are bound by DRAM (the first by its scattered sector writes).  Read
// through an inverse permutation, seven scattered 4-byte loads per particle,
// each fetching a 32-byte sector, took 24.1 ms at 134M particles; the two
// passes take 5.3 ms.  Writing the FP64 triples scattered in one pass
// (partial sectors) measured 12.3 ms.
//
// To host memory the link is the bound (193 GB/s, 4 particles per ns, which the
// scattered loads reach), so there the inverse permutation stays: it is the
// shorter pass to wait for (58 against 141 us at 8M particles).
// ---------------------------------------------------------------------------
__global__ void k_invperm(int64_t n, const Ctrl *ctrl, int32_t *inv) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const ParticleSet ps = ctrl->sets[ctrl->cur];
    const int32_t q = ps.pid[p];
    if (is_particle(q, n)) inv[q] = (int32_t)p;
}

__global__ void __launch_bounds__(256) k_unload_records(int64_t n, const Ctrl *ctrl) {
    dep_begin(ctrl);
    const int cur = ctrl->cur;
    const ParticleSet ps = ctrl->sets[cur];
    float4 *rec = reinterpret_cast<float4 *>(ctrl->sets[1 - cur].cell);
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int32_t q = __ldcs(ps.pid + p);
    if (!is_particle(q, n)) return;
    st_record(rec, q,
              make_float4(__int_as_float(__ldcs(ps.cell + p)), __ldcs(ps.o[0] + p),
                          __ldcs(ps.o[1] + p), __ldcs(ps.o[2] + p)),
              make_float4(__ldcs(ps.v[0] + p), __ldcs(ps.v[1] + p), __ldcs(ps.v[2] + p), 0.0f));
}

// Particles [o0, o0 + m) of the load order -> x, v, from their records or
// (GATHER) from the store through inv.  FP64 instructions run at about two lanes
// per clock and SM on this part, so each component costs two: the node positions
// come from a table, floats are widened and the wrap is tested on the bits (with
// conversions and divisions the FP64 pipe was 85% busy: 5.0 ms at 134M).
template <bool GATHER>
__global__ void __launch_bounds__(kLoadThreads) k_unload(int64_t o0, int64_t m, int64_t n,
                                                        const int32_t *inv,
                                                        const double *__restrict__ node_pos,
                                                        double h0, double h1, double h2,
                                                        double L0, double L1, double L2,
                                                        double half_dt, const Ctrl *ctrl,
                                                        double *__restrict__ x,
                                                        double *__restrict__ v) {
    dep_begin(inv, ctrl, x, v);
    // results are staged in shared memory and written as contiguous runs (the
    // destination may be host memory written over the chip-to-chip link)
    __shared__ double sx[3 * kLoadThreads], sv[3 * kLoadThreads];
    const int64_t q0 = (int64_t)blockIdx.x * kLoadThreads;
    const int cnt = (int)(m - q0 < kLoadThreads ? m - q0 : kLoadThreads);
    if ((int)threadIdx.x < cnt) {
        float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f), b = a;
        if (GATHER) {
            const ParticleSet ps = ctrl->sets[ctrl->cur];
            const int32_t p = inv[o0 + q0 + threadIdx.x];
            if (is_particle(p, n)) {
                a = make_float4(__int_as_float(ps.cell[p]), ps.o[0][p], ps.o[1][p], ps.o[2][p]);
                b = make_float4(ps.v[0][p], ps.v[1][p], ps.v[2][p], 0.0f);
            }
        } else {
            ld_record(reinterpret_cast<const float4 *>(ctrl->sets[1 - ctrl->cur].cell),
                      o0 + q0 + threadIdx.x, a, b);
        }
        const int32_t c = __float_as_int(a.x);
        const int idx[3] = {cell_i(c), cell_j(c), cell_k(c)};
        const float o[3] = {a.y, a.z, a.w}, w[3] = {b.x, b.y, b.z};
        const double h[3] = {h0, h1, h2};
        const double L[3] = {L0, L1, L2};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const double vd = widen(w[d]);
            const double pos = fma(widen(o[d]), h[d], __ldg(node_pos + d * kMaxN + idx[d]));
            sx[3 * threadIdx.x + d] = wrap_position(fma(-half_dt, vd, pos), L[d]);
            sv[3 * threadIdx.x + d] = vd;
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const int j = r * kLoadThreads + threadIdx.x;
        if (j < 3 * cnt) {
            x[3 * q0 + j] = sx[j];
            v[3 * q0 + j] = sv[j];
        }
    }
}

// ---------------------------------------------------------------------------
// gather + Boris push + drift + periodic wrap (push_one_pairs in push.cuh)
//
// Each thread owns groups of 4 consecutive particles: the seven SoA streams
// are read and written as 16-byte vectors with evict-first hints (they are
// touched once per step), so that the x-paired field stays cached (64 MiB at
// 128^3, of 129 MB of L2).
// ---------------------------------------------------------------------------
template <bool DIAG, bool EXT, bool MAG>
__global__ void __launch_bounds__(256, 3) k_gather_push(int64_t n, Geom g, PushConst pc, Ctrl *ctrl,
                                                      const float4 *E8,
                                                      double *__restrict__ part) {
    dep_begin(ctrl, E8, part);
    const ParticleSet ps = ctrl->sets[ctrl->cur];
    float a_vx = 0.f, a_vy = 0.f, a_vz = 0.f, a_v2 = 0.f;
    double d_v[4] = {0.0, 0.0, 0.0, 0.0};
    int bad = 0;
    const int64_t ngroups = n >> 2;                      // full groups of 4
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < ngroups; q += stride) {
        int4 c = __ldcs(reinterpret_cast<const int4 *>(ps.cell) + q);
        float4 ox = __ldcs(reinterpret_cast<const float4 *>(ps.o[0]) + q);
        float4 oy = __ldcs(reinterpret_cast<const float4 *>(ps.o[1]) + q);
        float4 oz = __ldcs(reinterpret_cast<const float4 *>(ps.o[2]) + q);
        float4 ux = __ldcs(reinterpret_cast<const float4 *>(ps.v[0]) + q);
        float4 uy = __ldcs(reinterpret_cast<const float4 *>(ps.v[1]) + q);
        float4 uz = __ldcs(reinterpret_cast<const float4 *>(ps.v[2]) + q);
        push_one_pairs<EXT, MAG>(g, pc, E8, c.x, ox.x, oy.x, oz.x, ux.x, uy.x, uz.x, bad);
        push_one_pairs<EXT, MAG>(g, pc, E8, c.y, ox.y, oy.y, oz.y, ux.y, uy.y, uz.y, bad);
        push_one_pairs<EXT, MAG>(g, pc, E8, c.z, ox.z, oy.z, oz.z, ux.z, uy.z, uz.z, bad);
        push_one_pairs<EXT, MAG>(g, pc, E8, c.w, ox.w, oy.w, oz.w, ux.w, uy.w, uz.w, bad);
        __stcs(reinterpret_cast<int4 *>(ps.cell) + q, c);
        __stcs(reinterpret_cast<float4 *>(ps.o[0]) + q, ox);
        __stcs(reinterpret_cast<float4 *>(ps.o[1]) + q, oy);
        __stcs(reinterpret_cast<float4 *>(ps.o[2]) + q, oz);
        __stcs(reinterpret_cast<float4 *>(ps.v[0]) + q, ux);
        __stcs(reinterpret_cast<float4 *>(ps.v[1]) + q, uy);
        __stcs(reinterpret_cast<float4 *>(ps.v[2]) + q, uz);
        if (DIAG) {
            a_vx += (ux.x + ux.y) + (ux.z + ux.w);
            a_vy += (uy.x + uy.y) + (uy.z + uy.w);
            a_vz += (uz.x + uz.y) + (uz.z + uz.w);
            a_v2 += (ux.x * ux.x + uy.x * uy.x + uz.x * uz.x) + (ux.y * ux.y + uy.y * uy.y + uz.y * uz.y) +
                    (ux.z * ux.z + uy.z * uy.z + uz.z * uz.z) + (ux.w * ux.w + uy.w * uy.w + uz.w * uz.w);
            d_v[0] += (double)a_vx;
            d_v[1] += (double)a_vy;
            d_v[2] += (double)a_vz;
            d_v[3] += (double)a_v2;
            a_vx = a_vy = a_vz = a_v2 = 0.f;
        }
    }
    // the n mod 4 particles after the last full group: first threads of block 0
    if (blockIdx.x == 0 && threadIdx.x < (n & 3)) {
        const int64_t p = (ngroups << 2) + threadIdx.x;
        int32_t c = ps.cell[p];
        float fx = ps.o[0][p], fy = ps.o[1][p], fz = ps.o[2][p];
        float vx = ps.v[0][p], vy = ps.v[1][p], vz = ps.v[2][p];
        push_one_pairs<EXT, MAG>(g, pc, E8, c, fx, fy, fz, vx, vy, vz, bad);
        ps.cell[p] = c;
        ps.o[0][p] = fx;
        ps.o[1][p] = fy;
        ps.o[2][p] = fz;
        ps.v[0][p] = vx;
        ps.v[1][p] = vy;
        ps.v[2][p] = vz;
        if (DIAG) {
            a_vx += vx;
            a_vy += vy;
            a_vz += vz;
            a_v2 += vx * vx + vy * vy + vz * vz;
        }
    }
    if (bad) raise_flag(ctrl, bad);
    if (DIAG) {
        // per-thread FP64 totals -> FP64 block sum in a fixed order -> one
        // partial per block (deterministic)
        double d[4] = {d_v[0] + a_vx, d_v[1] + a_vy, d_v[2] + a_vz, d_v[3] + a_v2};
        __shared__ double red[4][8];
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        for (int q = 0; q < 4; ++q) {
            double t = d[q];
            for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
            if (lane == 0) red[q][wid] = t;
        }
        __syncthreads();
        if (threadIdx.x < 4) {
            double t = 0.0;
            const int nw = blockDim.x >> 5;
            for (int w = 0; w < nw; ++w) t += red[threadIdx.x][w];
            part[4 * blockIdx.x + threadIdx.x] = t;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctrl->step += 1;
        ctrl->since_sort += 1;
    }
}


// ---------------------------------------------------------------------------
// fused gather + push + deposit of the new positions (one pass per step)
//
// Scatter of step n+1 needs exactly the positions this push writes, so the
// CTA that pushes a work item's particles also deposits them into the
// item's shared-memory tile (the sort's tile plus guard cells) and flushes
// it at the end: per step the particle store is read and written once (56
// bytes per particle) instead of being read again by a separate deposit.
// ---------------------------------------------------------------------------
// The staged field box of a tile: its guard layers (at most the deposit's) and
// extents.  BE > 0: BE slots on each axis.
struct EBox {
    int guard, row, plane, S;
};
template <int BE>
__device__ __forceinline__ EBox e_box(const Geom &g, int guard) {
    EBox e;
    e.guard = guard;
    e.row = BE > 0 ? BE : g.tile[0] + 2 * guard + 1;
    e.plane = BE > 0 ? BE * BE : e.row * (g.tile[1] + 2 * guard + 1);
    e.S = BE > 0 ? BE * BE * BE : e.plane * (g.tile[2] + 2 * guard + 1);
    return e;
}
// slot of the stencil base with deposit slots (si, sj, sk) in the staged box; false
// if its stencil leaves it
template <int BE>
__device__ __forceinline__ bool e_slot(const Geom &g, const EBox &e, int si, int sj, int sk, int &s) {
    const int dg = g.guard - e.guard;
    const unsigned a = (unsigned)(si - dg), b = (unsigned)(sj - dg), c = (unsigned)(sk - dg);
    s = (int)a + e.row * (int)b + e.plane * (int)c;
    if (BE > 0) return a < (unsigned)(BE - 1) && b < (unsigned)(BE - 1) && c < (unsigned)(BE - 1);
    return a < (unsigned)(g.tile[0] + 2 * e.guard) && b < (unsigned)(g.tile[1] + 2 * e.guard) &&
           c < (unsigned)(g.tile[2] + 2 * e.guard);
}

// One particle of the tile t (or of a sparse segment: everything through the
// grid).  E comes from (sA, sB), the block's copy of the tile's box, when it holds
// one and the stencil lies in it, else from the x-paired grid.  The slots of the
// new stencil base are the old ones plus the cells moved, so the periodic
// folding is done once per particle unless it leaves the box.
template <bool DIAG, bool EXT, bool MAG, bool FIXED, int B, int BE>
__device__ __forceinline__ void pd_one(const Geom &g, const PushConst &pc, const float4 *E8,
                                       const float4 *sA, const float2 *sB, const EBox &eb, bool sparse,
                                       uint32_t *acc, const cic::Tile &t, float *rho,
                                       unsigned long long *rho64, float qscale, int32_t &c, float &fx,
                                       float &fy, float &fz, float &vx, float &vy, float &vz, int &bad,
                                       unsigned long long &strays, Moments &mo) {
    int i, j, k, step[3];
    decode_base(g, c, i, j, k, bad);
    int si = cic::box_slot(i, t.ox, g.n[0], g.guard);
    int sj = cic::box_slot(j, t.oy, g.n[1], g.guard);
    int sk = cic::box_slot(k, t.oz, g.n[2], g.guard);
    float ex, ey, ez;
    int es;
    if (sA != nullptr && e_slot<BE>(g, eb, si, sj, sk, es))
        gather_E_pair_box<BE>(sA, sB, es, eb.row, eb.plane, fx, fy, fz, ex, ey, ez);
    else
        gather_E_pairs(g, E8, i, j, k, fx, fy, fz, ex, ey, ez);
    kick_drift<EXT, MAG>(g, pc, ex, ey, ez, i, j, k, c, fx, fy, fz, vx, vy, vz, bad, step);
    if (DIAG) mo.add(vx, vy, vz);
    if (!sparse) {
        si += step[0];
        sj += step[1];
        sk += step[2];
        int s = si + cic::box_row<B>(t) * sj + cic::box_plane<B>(t) * sk;
        if (cic::in_box_slots<B>(t, g, si, sj, sk) || cic::box_base<B>(t, g, i, j, k, s)) {
            cic::tile_add_at<FIXED, B>(acc, t, s, fx, fy, fz);
            return;
        }
        ++strays;
    }
    float w[8];
    cic::weights(fx, fy, fz, w);
    cic::deposit_global<FIXED>(rho, rho64, g, i, j, k, w, fx, fy, fz, qscale);
}

// staged: the block copies its tile's box of E8 to shared memory at each change
// of tile, with e_guard guard layers, and gathers there (see pd_one).  BE > 0:
// that box is BE slots long on each axis; B > 0: the deposit's is B slots long
// (see cic::box_row).
template <bool DIAG, bool EXT, bool MAG, bool FIXED, int B, int BE>
__global__ void __launch_bounds__(kPushThreadsPerSM / 2, 2) k_push_deposit(Geom g, PushConst pc, Ctrl *ctrl,
                                                          const int4 *items,
                                                          bool staged, int e_guard,
                                                          const float4 *E8,
                                                          float *rho, unsigned long long *rho64,
                                                          float qscale, int sparse_below, int tile_cost,
                                                          double *__restrict__ part,
                                                          SaveY save) {
    dep_begin(ctrl, items, E8, rho, rho64, part);
    extern __shared__ __align__(16) uint32_t acc[];
    const ParticleSet ps = ctrl->sets[ctrl->cur];
    const int n_items = ctrl->n_items;
    Moments mo;
    int bad = 0;
    unsigned long long strays = 0;
    // a contiguous run of work items per block, walked tile by tile
    Segments run = run_segments(items, n_items, tile_cost);
    const int S = cic::tile_of(g, 0).S;
    void *sum = reinterpret_cast<char *>(acc) + cic::sum_offset(S);
    float4 *sA = reinterpret_cast<float4 *>(reinterpret_cast<char *>(acc) + cic::stage_offset(S));
    const EBox eb = e_box<BE>(g, e_guard);
    float2 *sB = reinterpret_cast<float2 *>(sA + eb.S);
    for (int s = threadIdx.x; s < S; s += blockDim.x) {
        acc[s] = 0u;
        if (FIXED) reinterpret_cast<unsigned long long *>(sum)[s] = 0ull;
        else reinterpret_cast<float *>(sum)[s] = 0.0f;
    }
    // t: the tile of the dense segments (sparse ones deposit and gather globally)
    bool any = false, folded = false;
    cic::Tile t = cic::tile_of(g, 0);
    int tile;
    PIndex begin, end;
    while (next_segment(run, tile, begin, end)) {
        const bool sparse = (int)(end - begin) < sparse_below;
        // one particle per thread and iteration (coalesced 4-byte streams);
        // the next iteration's particle is loaded before this one is pushed
        PIndex p = begin + threadIdx.x;
        int32_t nc = 0;
        float nfx = 0.f, nfy = 0.f, nfz = 0.f, nvx = 0.f, nvy = 0.f, nvz = 0.f;
        if (p < end) {
            nc = __ldcs(ps.cell + p);
            nfx = __ldcs(ps.o[0] + p); nfy = __ldcs(ps.o[1] + p); nfz = __ldcs(ps.o[2] + p);
            nvx = __ldcs(ps.v[0] + p); nvy = __ldcs(ps.v[1] + p); nvz = __ldcs(ps.v[2] + p);
        }
        if (!sparse) {
            __syncthreads();   // every add to the tile and read of its box is done
            const cic::Tile tn = cic::tile_of(g, tile);
            if (staged) cic::stage_pairs(sA, sB, E8, cic::tile_of(g, tile, e_guard), g);
            if (any) cic::tile_flush<FIXED>(acc, sum, folded, t, g, rho, rho64, qscale);
            any = true;
            folded = false;
            t = tn;
            cic::stage_wait();
            __syncthreads();
        }
        const float4 *sAi = (staged && !sparse) ? sA : nullptr;
        for (PIndex done = begin;;) {
            // as many particles as the tile takes without a fold
            done += min(end - done, cic::fill_limit() * blockDim.x);
            for (; p < done; p += blockDim.x) {
                int32_t c = nc;
                float fx = nfx, fy = nfy, fz = nfz, vx = nvx, vy = nvy, vz = nvz;
                const PIndex pn = p + blockDim.x;
                if (pn < end) {
                    nc = __ldcs(ps.cell + pn);
                    nfx = __ldcs(ps.o[0] + pn); nfy = __ldcs(ps.o[1] + pn); nfz = __ldcs(ps.o[2] + pn);
                    nvx = __ldcs(ps.v[0] + pn); nvy = __ldcs(ps.v[1] + pn); nvz = __ldcs(ps.v[2] + pn);
                }
                if (save.cell) {
                    __stcs(save.cell + p, c);
                    __stcs(save.o[0] + p, fx);
                    __stcs(save.o[1] + p, fy);
                    __stcs(save.o[2] + p, fz);
                    if (save.v[0]) {
                        __stcs(save.v[0] + p, vx);
                        __stcs(save.v[1] + p, vy);
                        __stcs(save.v[2] + p, vz);
                    }
                }
                pd_one<DIAG, EXT, MAG, FIXED, B, BE>(g, pc, E8, sAi, sB, eb, sparse, acc, t, rho, rho64, qscale,
                                              c, fx, fy, fz, vx, vy, vz, bad, strays, mo);
                __stcs(ps.cell + p, c);
                __stcs(ps.o[0] + p, fx);
                __stcs(ps.o[1] + p, fy);
                __stcs(ps.o[2] + p, fz);
                __stcs(ps.v[0] + p, vx);
                __stcs(ps.v[1] + p, vy);
                __stcs(ps.v[2] + p, vz);
            }
            if (DIAG) mo.fold();
            if (done == end) break;
            __syncthreads();
            cic::tile_fold<FIXED>(acc, sum, S);
            __syncthreads();
            folded = true;
        }
    }
    __syncthreads();
    if (any) cic::tile_flush<FIXED>(acc, sum, folded, t, g, rho, rho64, qscale);
    if (bad) raise_flag(ctrl, bad);
    if (strays) {
        atomicAdd(&ctrl->stray, strays);
        atomicAdd(&ctrl->stray_step, strays);
    }
    if (DIAG) {
        __shared__ double red[4][kPushThreadsPerSM / 64];
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        const double w4 = warp_total(mo);
        if ((lane & 7) == 0) red[lane >> 3][wid] = w4;
        __syncthreads();
        if (threadIdx.x < 4) {
            double tt = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tt += red[threadIdx.x][w];
            part[4 * blockIdx.x + threadIdx.x] = tt;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctrl->step += 1;
        ctrl->since_sort += 1;
    }
}


}  // namespace

cudaError_t launch_load(const double *x, const double *v, int64_t m, int64_t base, const Geom &g,
                        const double *inv_h_d, double dt, Ctrl *ctrl, LStream st,
                        int max_blocks) {
    if (m <= 0) return cudaSuccess;
    const int T = kLoadThreads;
    int64_t B = (m + T - 1) / T;
    if (max_blocks > 0) B = std::min<int64_t>(B, max_blocks);
    k_load<<<(unsigned)B, T, 0, st>>>(x, v, m, base, g, inv_h_d[0], inv_h_d[1], inv_h_d[2],
                                      0.5 * dt,                                      ctrl);
    return cudaGetLastError();
}

// Device-to-device copy of up to 8 arrays in one launch (16-byte vectors; the
// byte tail of each array by the first threads).  Copies inside the arena run
// on the SMs at HBM speed rather than through a copy engine.
__global__ void __launch_bounds__(256) k_copy(CopyList cl) {
    dep_begin();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int a = 0; a < cl.count; ++a) {
        const int64_t n16 = cl.bytes[a] >> 4;
        const uint4 *src = reinterpret_cast<const uint4 *>(cl.src[a]);
        uint4 *dst = reinterpret_cast<uint4 *>(cl.dst[a]);
        for (int64_t q = t0; q < n16; q += stride) dst[q] = src[q];
        const int64_t rem = cl.bytes[a] & 15;
        if (t0 < rem) cl.dst[a][(n16 << 4) + t0] = cl.src[a][(n16 << 4) + t0];
    }
}

cudaError_t launch_copy(const CopyList &cl, LStream st) {
    int64_t total = 0;
    for (int a = 0; a < cl.count; ++a) {
        if ((reinterpret_cast<uintptr_t>(cl.dst[a]) | reinterpret_cast<uintptr_t>(cl.src[a])) & 15)
            return cudaErrorMisalignedAddress;
        total += cl.bytes[a] >> 4;
    }
    if (total == 0 && cl.count == 0) return cudaSuccess;
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((total + 255) / 256, 152 * 8));
    launch_dep(k_copy, blocks, 256, 0, st, cl);
    return cudaGetLastError();
}

__global__ void k_pid_positions(int64_t n, const int32_t *pid, int32_t *pos) {
    dep_begin(pid, pos);
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n && is_particle(pid[p], n)) pos[pid[p]] = (int32_t)p;
}

cudaError_t launch_pid_positions(int64_t n, const int32_t *pid, int32_t *pos, LStream st) {
    if (n <= 0) return cudaSuccess;
    launch_dep(k_pid_positions, (unsigned)((n + 255) / 256), 256, 0, st, n, pid, pos);
    return cudaGetLastError();
}

cudaError_t launch_unload_records(int64_t n, const Ctrl *ctrl, LStream st) {
    if (n <= 0) return cudaSuccess;
    launch_dep(k_unload_records, (unsigned)((n + 255) / 256), 256, 0, st, n, ctrl);
    return cudaGetLastError();
}

cudaError_t launch_invperm(int64_t n, const Ctrl *ctrl, int32_t *inv, LStream st) {
    if (n <= 0) return cudaSuccess;
    k_invperm<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, ctrl, inv);
    return cudaGetLastError();
}

void node_positions(const double *h_d, double *node_pos) {
    for (int d = 0; d < 3; ++d)
        for (int i = 0; i < kMaxN; ++i) node_pos[d * kMaxN + i] = ((double)i + 0.5) * h_d[d];
}

cudaError_t launch_unload(int64_t o0, int64_t m, int64_t n, const int32_t *inv, const double *node_pos,
                          const double *h_d, const double *L_d, double dt, const Ctrl *ctrl,
                          double *x, double *v, LStream st) {
    if (m <= 0) return cudaSuccess;
    const unsigned blocks = (unsigned)((m + kLoadThreads - 1) / kLoadThreads);
#define PIC_UL(G)                                                                            \
    launch_dep(k_unload<G>, blocks, kLoadThreads, 0, st, o0, m, n, inv, node_pos, h_d[0], h_d[1], h_d[2], \
                                                 L_d[0], L_d[1], L_d[2], 0.5 * dt, ctrl, x, v)
    if (inv) PIC_UL(true);
    else PIC_UL(false);
#undef PIC_UL
    return cudaGetLastError();
}

cudaError_t launch_gather_push(int64_t n, const Geom &g, const PushConst &pc, bool diag,
                               Ctrl *ctrl, const float4 *E8, double *part, int blocks,
                               int threads, LStream st) {
    const bool ext = pc.wz2 != 0.0f;
    const bool mag = pc.t[0] != 0.0f || pc.t[1] != 0.0f || pc.t[2] != 0.0f;
#define PIC_GP(D, X, M) launch_dep(k_gather_push<D, X, M>, blocks, threads, 0, st, n, g, pc, ctrl, E8, part)
    if (diag) {
        if (ext) { if (mag) PIC_GP(true, true, true); else PIC_GP(true, true, false); }
        else     { if (mag) PIC_GP(true, false, true); else PIC_GP(true, false, false); }
    } else {
        if (ext) { if (mag) PIC_GP(false, true, true); else PIC_GP(false, true, false); }
        else     { if (mag) PIC_GP(false, false, true); else PIC_GP(false, false, false); }
    }
#undef PIC_GP
    return cudaGetLastError();
}

}  // namespace pic

namespace pic {

// ---------------------------------------------------------------------------
// uniform plasma test (Section 4.4): random displacements instead of the push
// ---------------------------------------------------------------------------

// c-th output (c >= 1) of the SplitMix64 generator seeded with `seed`
__device__ __forceinline__ uint64_t splitmix64(uint64_t seed, uint64_t c) {
    uint64_t z = seed + c * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// displacement along axis d (in cells, in [-1, 1)) of particle pid in step n:
// 2u - 1 with u = the top 24 bits of output ((n 2^32 + pid) 4 + d + 1)
__device__ __forceinline__ float move_cells(uint64_t seed, long long n, int32_t pid, int d) {
    const uint64_t c = (((uint64_t)n << 32) + (uint64_t)(uint32_t)pid) * 4ull + (uint64_t)d + 1ull;
    const uint32_t r = (uint32_t)(splitmix64(seed, c) >> 40);
    return (float)r * (1.0f / 8388608.0f) - 1.0f;   // exact: r < 2^24
}

__device__ __forceinline__ void move_one(const Geom &g, uint64_t seed, long long n, int32_t pid,
                                         int32_t &c, float &fx, float &fy, float &fz, int &bad) {
    int i, j, k;
    decode_base(g, c, i, j, k, bad);
    int step[3];
    advance_cells(g, fx + move_cells(seed, n, pid, 0), fy + move_cells(seed, n, pid, 1),
                  fz + move_cells(seed, n, pid, 2), i, j, k, c, fx, fy, fz, bad, step);
}

template <bool DIAG>
__device__ __forceinline__ void block_moments(const Moments &mo, double *part) {
    if (!DIAG) return;
    __shared__ double red[4][8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const double w4 = warp_total(mo);
    if ((lane & 7) == 0) red[lane >> 3][wid] = w4;
    __syncthreads();
    if (threadIdx.x < 4) {
        double tt = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tt += red[threadIdx.x][w];
        part[4 * blockIdx.x + threadIdx.x] = tt;
    }
}

// the random move of every particle with the deposit of the new positions
// (the work items and shared tiles of k_push_deposit); velocities untouched.
// B > 0: every tile box is B slots long on each axis (see cic::box_row).
template <bool DIAG, bool FIXED, int B>
__global__ void __launch_bounds__(256, PIC_MV_MIN_BLOCKS) k_move_deposit(
    Geom g, uint64_t seed, Ctrl *ctrl, const int4 *items, float *rho,
    unsigned long long *rho64, float qscale, int sparse_below, int tile_cost,
    double *__restrict__ part) {
    dep_begin(ctrl, items, rho, rho64, part);
    extern __shared__ __align__(16) uint32_t acc[];
    const ParticleSet ps = ctrl->sets[ctrl->cur];
    const int n_items = ctrl->n_items;
    const long long n = ctrl->step;   // advanced after this kernel (k_step_inc)
    Moments mo;
    int bad = 0;
    unsigned long long strays = 0;
    Segments run = run_segments(items, n_items, tile_cost);
    const int S = cic::tile_of(g, 0).S;
    void *sum = reinterpret_cast<char *>(acc) + cic::sum_offset(S);
    for (int s = threadIdx.x; s < S; s += blockDim.x) {
        acc[s] = 0u;
        if (FIXED) reinterpret_cast<unsigned long long *>(sum)[s] = 0ull;
        else reinterpret_cast<float *>(sum)[s] = 0.0f;
    }
    // t: the tile of the dense segments (sparse ones deposit globally)
    bool any = false, folded = false;
    cic::Tile t = cic::tile_of(g, 0);
    int tile;
    PIndex begin, end;
    while (next_segment(run, tile, begin, end)) {
        const bool sparse = (int)(end - begin) < sparse_below;
        // the next particle's streams are loaded before the current one moves
        PIndex p = begin + threadIdx.x;
        int32_t nc = 0, npid = 0;
        float nfx = 0.f, nfy = 0.f, nfz = 0.f;
        if (p < end) {
            nc = __ldcs(ps.cell + p);
            nfx = __ldcs(ps.o[0] + p); nfy = __ldcs(ps.o[1] + p); nfz = __ldcs(ps.o[2] + p);
            npid = ps.pid[p];
        }
        if (!sparse) {
            __syncthreads();   // every add to the tile is done
            if (any) cic::tile_flush<FIXED>(acc, sum, folded, t, g, rho, rho64, qscale);
            any = true;
            folded = false;
            t = cic::tile_of(g, tile);
            __syncthreads();
        }
        for (PIndex done = begin;;) {
            done += min(end - done, cic::fill_limit() * blockDim.x);
            for (; p < done; p += blockDim.x) {
                int32_t c = nc;
                float fx = nfx, fy = nfy, fz = nfz;
                const int32_t pid = npid;
                const PIndex pn = p + blockDim.x;
                if (pn < end) {
                    nc = __ldcs(ps.cell + pn);
                    nfx = __ldcs(ps.o[0] + pn); nfy = __ldcs(ps.o[1] + pn); nfz = __ldcs(ps.o[2] + pn);
                    npid = ps.pid[pn];
                }
                move_one(g, seed, n, pid, c, fx, fy, fz, bad);
                const int i = cell_i(c), j = cell_j(c), k = cell_k(c);
                if (sparse) {
                    float w[8];
                    cic::weights(fx, fy, fz, w);
                    cic::deposit_global<FIXED>(rho, rho64, g, i, j, k, w, fx, fy, fz, qscale);
                } else if (!cic::tile_add<FIXED, B>(acc, t, g, i, j, k, fx, fy, fz, rho, rho64, qscale)) {
                    ++strays;
                }
                if (DIAG) mo.add(ps.v[0][p], ps.v[1][p], ps.v[2][p]);
                __stcs(ps.cell + p, c);
                __stcs(ps.o[0] + p, fx);
                __stcs(ps.o[1] + p, fy);
                __stcs(ps.o[2] + p, fz);
            }
            if (DIAG) mo.fold();
            if (done == end) break;
            __syncthreads();
            cic::tile_fold<FIXED>(acc, sum, S);
            __syncthreads();
            folded = true;
        }
    }
    __syncthreads();
    if (any) cic::tile_flush<FIXED>(acc, sum, folded, t, g, rho, rho64, qscale);
    if (bad) raise_flag(ctrl, bad);
    if (strays) {
        atomicAdd(&ctrl->stray, strays);
        atomicAdd(&ctrl->stray_step, strays);
    }
    block_moments<DIAG>(mo, part);
}

// the random move alone (split calls: pic_gather_push)
template <bool DIAG>
__global__ void __launch_bounds__(256) k_move(int64_t np, Geom g, uint64_t seed, Ctrl *ctrl,
                                               double *__restrict__ part) {
    const ParticleSet ps = ctrl->sets[ctrl->cur];
    const long long n = ctrl->step;
    Moments mo;
    int bad = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < np; p += stride) {
        int32_t c = ps.cell[p];
        float fx = ps.o[0][p], fy = ps.o[1][p], fz = ps.o[2][p];
        move_one(g, seed, n, ps.pid[p], c, fx, fy, fz, bad);
        ps.cell[p] = c;
        ps.o[0][p] = fx;
        ps.o[1][p] = fy;
        ps.o[2][p] = fz;
        if (DIAG) {
            mo.add(ps.v[0][p], ps.v[1][p], ps.v[2][p]);
            mo.fold();
        }
    }
    if (bad) raise_flag(ctrl, bad);
    block_moments<DIAG>(mo, part);
}

__global__ void k_step_inc(Ctrl *ctrl) {
    dep_begin(ctrl);
    ctrl->step += 1;
    ctrl->since_sort += 1;
}

bool const_box(const Geom &g) {
    for (int d = 0; d < 3; ++d)
        if (g.tile[d] + 2 * g.guard + 1 != kConstBox) return false;
    return true;
}

cudaError_t launch_move(int64_t np, const Geom &g, uint64_t seed, bool diag, bool fixed, bool deposit,
                        Ctrl *ctrl, const int4 *items, int max_items, float *rho,
                        unsigned long long *rho64, double qscale, int sparse_below, int tile_cost,
                        double *part, int blocks, LStream st) {
    const int nb = std::max(1, std::min(blocks, deposit ? max_items : blocks));
    if (deposit) {
        const size_t smem = tile_deposit_smem(g);
        const float qs = (float)qscale;
        const bool cbox = const_box(g);
#define PIC_MV(D, F, B) \
    launch_dep(k_move_deposit<D, F, B>, nb, 256, smem, st, g, seed, ctrl, items, rho, rho64, qs, sparse_below, \
                                                   tile_cost, part)
        if (diag) {
            if (!fixed) PIC_MV(true, false, 0);
            else if (cbox) PIC_MV(true, true, kConstBox);
            else PIC_MV(true, true, 0);
        } else {
            if (!fixed) PIC_MV(false, false, 0);
            else if (cbox) PIC_MV(false, true, kConstBox);
            else PIC_MV(false, true, 0);
        }
#undef PIC_MV
    } else {
        if (diag) k_move<true><<<nb, 256, 0, st>>>(np, g, seed, ctrl, part);
        else k_move<false><<<nb, 256, 0, st>>>(np, g, seed, ctrl, part);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    launch_dep(k_step_inc, 1, 1, 0, st, ctrl);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return (deposit && fixed) ? launch_rho_finish(g, rho64, rho, qscale, st) : cudaSuccess;
}

// item tile + the block's tile sums
size_t tile_deposit_smem(const Geom &g) {
    const cic::Tile t0 = cic::tile_of(g, 0);
    return cic::sum_offset(t0.S) + 8 * (size_t)t0.S;
}
// Blocks of the fused push + deposit: two of 384 threads per SM with the x-paired
// box (24 bytes a slot after the deposit tiles' 12) while two fit in its 228 KiB
// (plus the kernel's static shared memory and the runtime's 1 KiB per block), else
// three of 256 that read the grid.  13^3 slots (8^3 tiles, two guard layers): 20
// steps of 128^3 x 64 64.1 ms (62.4 since), with whole nodes in the box (16 bytes a
// slot, three blocks of 256) 66.9.  With more guard layers the box takes as many as fit, two at
// least: the Penning bunch's (three, of which the box takes two) 10 steps took 49.8
// ms reading the grid, 46.9 with the box (44.7 since kTileCost); one block of 768 threads with all three 53.7.
PushShape push_shape(const Geom &g) {
    const size_t tiles = cic::stage_offset(cic::tile_of(g, 0).S);
    for (int eg = g.guard; eg >= std::min(g.guard, 2); --eg) {
        const size_t box = tiles + 24 * (size_t)cic::tile_of(g, 0, eg).S;
        if (2 * (box + 2048) <= (size_t)228 * 1024)
            return PushShape{kPushThreadsPerSM / 2, 2, true, eg, box};
    }
    return PushShape{kPushThreadsPerSM / 3, 3, false, 0, tile_deposit_smem(g)};
}
// boxes compiled as constants: the default's, and a three-layer guard's with the
// field box of two
bool const_box15(const Geom &g, const PushShape &ps) {
    for (int d = 0; d < 3; ++d)
        if (g.tile[d] != 8) return false;
    return g.guard == 3 && ps.staged && ps.e_guard == 2;
}

// Allow the fused kernels' shared memory (call outside any stream capture)
cudaError_t push_deposit_prepare(const Geom &g) {
    cudaError_t e = cudaSuccess;
    const size_t tsm = tile_deposit_smem(g), smem = push_shape(g).smem;
#define PIC_MVA(D, F, B) \
    if ((e = allow_smem(k_move_deposit<D, F, B>, tsm)) != cudaSuccess) return e
    PIC_MVA(false, false, 0); PIC_MVA(false, true, 0); PIC_MVA(true, false, 0);
    PIC_MVA(true, true, 0); PIC_MVA(false, true, kConstBox); PIC_MVA(true, true, kConstBox);
#undef PIC_MVA
#define PIC_PDA(D, X, M, F, B, BE) \
    if ((e = allow_smem(k_push_deposit<D, X, M, F, B, BE>, smem)) != cudaSuccess) return e
#define PIC_PDA2(D, X, M) \
    PIC_PDA(D, X, M, false, 0, 0); PIC_PDA(D, X, M, true, 0, 0);          \
    PIC_PDA(D, X, M, true, kConstBox, kConstBox); PIC_PDA(D, X, M, true, 15, kConstBox)
    PIC_PDA2(false, false, false); PIC_PDA2(false, false, true);
    PIC_PDA2(false, true, false);  PIC_PDA2(false, true, true);
    PIC_PDA2(true, false, false);  PIC_PDA2(true, false, true);
    PIC_PDA2(true, true, false);   PIC_PDA2(true, true, true);
#undef PIC_PDA2
#undef PIC_PDA
    return cudaSuccess;
}

cudaError_t launch_push_deposit(const Geom &g, const PushConst &pc, bool diag, bool fixed,
                                Ctrl *ctrl, const int4 *items, int max_items,
                                const float4 *E8, float *rho, unsigned long long *rho64,
                                double qscale, int sparse_below, int tile_cost, double *part,
                                int blocks, const SaveY &save, LStream st) {
    const bool ext = pc.wz2 != 0.0f;
    const bool mag = pc.t[0] != 0.0f || pc.t[1] != 0.0f || pc.t[2] != 0.0f;
    const PushShape ps = push_shape(g);
    const int nb = std::max(1, std::min(blocks, max_items));
    const float qs = (float)qscale;
    cudaError_t e = cudaSuccess;
    const bool cbox = const_box(g) && ps.staged, cbox15 = const_box15(g, ps);
#define PIC_PD(D, X, M, F, B, BE)                                                             \
    launch_dep(k_push_deposit<D, X, M, F, B, BE>, nb, ps.threads, ps.smem, st, g, pc, ctrl, items, \
               ps.staged, ps.e_guard, E8, rho, rho64, qs, sparse_below, tile_cost, part, save)
#define PIC_PD_F(D, X, M)                                            \
    do {                                                             \
        if (!fixed) PIC_PD(D, X, M, false, 0, 0);                    \
        else if (cbox) PIC_PD(D, X, M, true, kConstBox, kConstBox);  \
        else if (cbox15) PIC_PD(D, X, M, true, 15, kConstBox);       \
        else PIC_PD(D, X, M, true, 0, 0);                            \
    } while (0)
    if (diag) {
        if (ext) { if (mag) PIC_PD_F(true, true, true); else PIC_PD_F(true, true, false); }
        else     { if (mag) PIC_PD_F(true, false, true); else PIC_PD_F(true, false, false); }
    } else {
        if (ext) { if (mag) PIC_PD_F(false, true, true); else PIC_PD_F(false, true, false); }
        else     { if (mag) PIC_PD_F(false, false, true); else PIC_PD_F(false, false, false); }
    }
#undef PIC_PD_F
#undef PIC_PD
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return fixed ? launch_rho_finish(g, rho64, rho, qscale, st) : cudaSuccess;
}

}  // namespace pic
