// Batched ensembles: many independent PIC runs (different grids, particle
// counts, charges) advanced by one set of launches per phase.
//
// Every instance keeps the scheme of the single-run path (Section 3.1 steps
// 1-4 and Section 3.2 of arXiv 2205.11052); what changes is only where its
// data lives:
//  * particles of instance i occupy [p0_i, p0_i + np_i) of one shared SoA
//    store (binning keys are global tile ids, tile0_i + local tile, which are
//    ordered by instance, so sorting never moves a particle out of its range);
//  * its grids occupy nodes [g0_i, g0_i + ng_i) of the concatenated rho, rho64
//    and E arrays, instances of equal grid size (a size class) adjacent so a
//    batched cuFFT plan covers the class;
//  * a work item (global tile, particle range) names its instance through the
//    tile -> instance table, so one persistent push + deposit launch walks the
//    work of every instance.
#include <algorithm>

#include "batch.cuh"
#include "cic.cuh"
#include "ffsum.cuh"
#include "push.cuh"
#include "records.cuh"
#include "sort_staged.cuh"

namespace pic {

namespace {

// instance owning particle p: binary search over the particle offsets
__device__ __forceinline__ int inst_of_particle(const long long *__restrict__ p0, int n_inst,
                                                long long p) {
    int lo = 0, hi = n_inst - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (p0[mid] <= p) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

__global__ void k_b_load(const double *__restrict__ x, const double *__restrict__ v, int64_t m,
                         int64_t base, const InstDesc *__restrict__ desc,
                         const long long *__restrict__ p0, int n_inst, double half_dt, Ctrl *ctrl) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= m) return;
    const int64_t p = base + q;
    const InstDesc &D = desc[inst_of_particle(p0, n_inst, p)];
    const ParticleSet ps = ctrl->sets[ctrl->cur];
    int idx[3];
    float off[3];
    bool ok = true;
    for (int d = 0; d < 3; ++d) {
        const double vd = v[3 * q + d];
        double s = (x[3 * q + d] + half_dt * vd) * D.inv_h_d[d] - 0.5;
        if (!isfinite(s) || !isfinite(vd) || fabs(s) > 4.0e15) {
            ok = false;
            s = 0.0;
        }
        const FloorRest fr = floor_rest(s);
        long long il = fr.whole;
        if ((unsigned long long)il >= (unsigned long long)D.g.n[d]) {   // outside: wrap
            il += il < 0 ? D.g.n[d] : -D.g.n[d];
            if ((unsigned long long)il >= (unsigned long long)D.g.n[d]) {   // a box away
                il %= D.g.n[d];
                if (il < 0) il += D.g.n[d];
            }
        }
        float ff = fr.rest;
        if (ff >= 1.0f) {
            ff = 0.0f;
            if (++il == D.g.n[d]) il = 0;
        }
        idx[d] = (int)il;
        off[d] = ff;
        ps.v[d][p] = ok ? narrow(vd) : 0.0f;
    }
    if (!ok) atomicOr(&ctrl->flags, PIC_FLAG_NONFINITE);
    ps.cell[p] = pack_cell(idx[0], idx[1], idx[2]);
    ps.o[0][p] = off[0];
    ps.o[1][p] = off[1];
    ps.o[2][p] = off[2];
    ps.pid[p] = (int32_t)p;
}

// Records [o0, o0 + m) (launch_unload_records over the whole store: pids are
// store slots, instances in internal order) -> x, v.  With c0 the whole store
// goes out in one launch, each instance to its place c0 in the caller's order;
// without, one instance's records go out contiguously.
//
// Bound by FP64 instructions (about two lanes per clock and SM: the product, the
// half step back) and by DRAM.  With a search per thread and (i + 1/2) + o by FP64
// instructions 43M particles took 1.17 ms, without 0.77, and without a wrap for every
// particle of the last half cell 0.71 (the bytes 0.51).  Blocks of several runs, the next one's records loaded
// ahead, measured the same.
__global__ void __launch_bounds__(256) k_b_unload(int64_t o0, int64_t m,
                                                  const InstDesc *__restrict__ desc,
                                                  const long long *__restrict__ p0, int n_inst,
                                                  const long long *__restrict__ c0, double half_dt,
                                                  const Ctrl *ctrl, double *__restrict__ x,
                                                  double *__restrict__ v) {
    dep_begin(ctrl, x, v);
    const float4 *rec = reinterpret_cast<const float4 *>(ctrl->sets[1 - ctrl->cur].cell);
    __shared__ double sx[3 * 256], sv[3 * 256];
    __shared__ long long dst[256];
    __shared__ int first;
    const int64_t q0 = (int64_t)blockIdx.x * 256;
    const int cnt = (int)(m - q0 < 256 ? m - q0 : 256);
    if (threadIdx.x == 0) first = inst_of_particle(p0, n_inst, o0 + q0);   // one search for most
    __syncthreads();
    const bool one = o0 + q0 + cnt <= p0[first + 1];   // the block lies in one instance
    if ((int)threadIdx.x < cnt) {
        const int64_t p = o0 + q0 + threadIdx.x;
        const int inst = one ? first : inst_of_particle(p0, n_inst, p);
        const InstDesc &D = desc[inst];
        dst[threadIdx.x] = c0 ? c0[inst] + (p - p0[inst]) : p - o0;
        float4 a, b;
        ld_record(rec, p, a, b);
        const int32_t c = __float_as_int(a.x);
        const int idx[3] = {cell_i(c), cell_j(c), cell_k(c)};
        const float o[3] = {a.y, a.z, a.w}, w[3] = {b.x, b.y, b.z};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const double vd = widen(w[d]);
            // beyond the last half cell at its place below the first node: no wrap
            const int i = idx[d] == D.g.n[d] - 1 && o[d] >= 0.5f ? -1 : idx[d];
            const double pos = half_node_plus(i, o[d]) * D.h_d[d];
            sx[3 * threadIdx.x + d] = wrap_position(fma(-half_dt, vd, pos), D.L_d[d]);
            sv[3 * threadIdx.x + d] = vd;
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const int j = r * 256 + threadIdx.x;
        if (j < 3 * cnt) {
            const int t = j / 3;
            const int64_t k = 3 * dst[t] + (j - 3 * t);
            x[k] = sx[j];
            v[k] = sv[j];
        }
    }
}

__device__ __forceinline__ int b_key(int32_t c, const InstDesc &D, int &bad) {
    int i = cell_i(c), j = cell_j(c), k = cell_k(c);
    if (i >= D.g.n[0] || j >= D.g.n[1] || k >= D.g.n[2]) {
        bad = 1;
        i = j = k = 0;
    }
    const int ti = tile_div(i, D.g.tdiv[0]), tj = tile_div(j, D.g.tdiv[1]);
    const int tk = tile_div(k, D.g.tdiv[2]);
    return D.tile0 + ti + D.g.ntile[0] * (tj + D.g.ntile[1] * tk);
}

// binning key of particle p: the global tile id of its instance's tile.  A
// thread's copy remembers the particle range of the last instance it looked
// up (a thread meets consecutive particles of one instance), so the binary
// search runs only when p leaves it.
struct BatchKey {
    const InstDesc *desc;
    const long long *p0;
    int n_inst;
    mutable long long lo = 0, hi = 0;
    mutable int inst = 0;
    __device__ __forceinline__ int operator()(int32_t c, int64_t p, int &bad) const {
        if (p < lo || p >= hi) {
            inst = inst_of_particle(p0, n_inst, p);
            lo = p0[inst];
            hi = p0[inst + 1];
        }
        return b_key(c, desc[inst], bad);
    }
};

// Work items (instance tile, particle range) in contiguous runs per block:
// the deposit of the instance's tile and (PUSH) the gather + push before it.
// The tile accumulates in shared memory (u32 fixed point, or FP32 bits), is
// folded into 64-bit per-tile sums before an item that would take it past 4095
// particles, and flushed to the instance's grid when the block moves to another
// tile, so consecutive items of one tile cost one flush.
// (DIAG: the moments of an instance, see emit.)
template <bool PUSH, bool DIAG, bool EXT, bool MAG, bool FIXED>
__global__ void __launch_bounds__(256, PIC_BATCH_PD_MIN_BLOCKS) k_b_push_deposit(
    const InstDesc *__restrict__ desc, const int32_t *__restrict__ tile_inst, Ctrl *ctrl,
    const int4 *items, const float4 *E4, const float4 *E8,
    float *rho, unsigned long long *rho64, int sparse_below, int tile_cost, int max_S,
    double *__restrict__ part) {
    dep_begin(ctrl, items, E4, E8, rho, rho64, part);
    extern __shared__ __align__(16) uint32_t acc[];
    __shared__ double red[4][8];
    void *sum = reinterpret_cast<char *>(acc) + cic::sum_offset(max_S);
    float4 *sE = reinterpret_cast<float4 *>(reinterpret_cast<char *>(acc) + cic::stage_offset(max_S));
    const ParticleSet ps = ctrl->sets[ctrl->cur];
    const int n_items = ctrl->n_items;
    int it0, it1;
    item_run(items, n_items, tile_cost, it0, it1);
    for (int s = threadIdx.x; s < max_S; s += blockDim.x) {
        acc[s] = 0u;
        if (FIXED) reinterpret_cast<unsigned long long *>(sum)[s] = 0ull;
        else reinterpret_cast<float *>(sum)[s] = 0.0f;
    }
    int bad = 0;
    int cur_tile = -1, filled = 0;
    bool folded = false;
    const InstDesc *Dc = desc;
    cic::Tile t{};   // the tile of the dense items
    // DIAG: the block's moments of one instance, over all of its items in the run,
    // go to the last of them, zeros to the others (a block sum in FP64 after every
    // item: push 801 us on 24 instances of up to 48^3 cells, now 771)
    Moments mo;
    const InstDesc *Dm = nullptr;
    auto emit = [&](int it) {
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        __syncthreads();
        const double w4 = warp_total(mo);
        if ((lane & 7) == 0) red[lane >> 3][wid] = w4;
        __syncthreads();
        if (threadIdx.x < 4) {
            double t = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[threadIdx.x][w];
            part[4 * (int64_t)it + threadIdx.x] = t;
        }
        mo = Moments{};
    };
    for (int it = it0; it < it1; ++it) {
        int4 item = items[it];   // z: end of its tile
        if (it + 1 < item.w) item.z = items[it + 1].y;
        const InstDesc &D = desc[tile_inst[item.x]];
        if (DIAG) {
            if (Dm == &D) {
                if (threadIdx.x < 4) part[4 * (int64_t)(it - 1) + threadIdx.x] = 0.0;
            } else if (Dm != nullptr) {
                emit(it - 1);
            }
            Dm = &D;
        }
        const Geom g = D.g;
        const PushConst pc = D.pc;
        const float4 *Ei = E8 + 2 * D.g0;
        float *rhoi = rho + D.g0;
        unsigned long long *rho64i = rho64 + D.g0;
        const float qscale = D.qscale;
        const bool sparse = item.z - item.y < sparse_below;
        if (!sparse) {
            if (item.x != cur_tile) {
                __syncthreads();   // every add to the tile and read of its box is done
                if (cur_tile >= 0)
                    cic::tile_flush<FIXED>(acc, sum, folded, t, Dc->g, rho + Dc->g0, rho64 + Dc->g0,
                                           Dc->qscale);
                cur_tile = item.x;
                filled = 0;
                folded = false;
                t = cic::tile_of(g, item.x - D.tile0);
                Dc = &D;
                if (PUSH && E4 != nullptr) cic::stage_box(sE, E4 + D.g0, t, g);
                cic::stage_wait();
                __syncthreads();
            } else if (filled + (item.z - item.y) > kMaxChunk) {
                __syncthreads();
                cic::tile_fold<FIXED>(acc, sum, t.S);
                __syncthreads();
                filled = 0;
                folded = true;
            }
            filled += item.z - item.y;
        }
        const float4 *sEi = (PUSH && E4 != nullptr && !sparse) ? sE : nullptr;
        // the next particle's streams are loaded before the current one is pushed
        const PIndex end = item.z;
        PIndex p = item.y + threadIdx.x;
        int32_t nc = 0;
        float nfx = 0.f, nfy = 0.f, nfz = 0.f, nvx = 0.f, nvy = 0.f, nvz = 0.f;
        if (p < end) {
            nc = __ldcs(ps.cell + p);
            nfx = __ldcs(ps.o[0] + p); nfy = __ldcs(ps.o[1] + p); nfz = __ldcs(ps.o[2] + p);
            if (PUSH) {
                nvx = __ldcs(ps.v[0] + p); nvy = __ldcs(ps.v[1] + p); nvz = __ldcs(ps.v[2] + p);
            }
        }
        for (; p < end; p += blockDim.x) {
            int32_t c = nc;
            float fx = nfx, fy = nfy, fz = nfz;
            const float cvx = nvx, cvy = nvy, cvz = nvz;
            {
                const PIndex pn = p + blockDim.x;
                if (pn < end) {
                    nc = __ldcs(ps.cell + pn);
                    nfx = __ldcs(ps.o[0] + pn); nfy = __ldcs(ps.o[1] + pn); nfz = __ldcs(ps.o[2] + pn);
                    if (PUSH) {
                        nvx = __ldcs(ps.v[0] + pn); nvy = __ldcs(ps.v[1] + pn);
                        nvz = __ldcs(ps.v[2] + pn);
                    }
                }
            }
            int i, j, k;
            if (PUSH) {
                float vx = cvx, vy = cvy, vz = cvz;
                push_one_staged<EXT, MAG>(g, pc, Ei, sEi, t, c, fx, fy, fz, vx, vy, vz, bad, i, j,
                                          k);
                __stcs(ps.cell + p, c);
                __stcs(ps.o[0] + p, fx);
                __stcs(ps.o[1] + p, fy);
                __stcs(ps.o[2] + p, fz);
                __stcs(ps.v[0] + p, vx);
                __stcs(ps.v[1] + p, vy);
                __stcs(ps.v[2] + p, vz);
                if (DIAG) mo.add(vx, vy, vz);
            }
            if (!PUSH && !cic::decode_cell(c, g, i, j, k)) bad |= PIC_FLAG_BAD_CELL;
            if (sparse) {
                float w[8];
                cic::weights(fx, fy, fz, w);
                cic::deposit_global<FIXED>(rhoi, rho64i, g, i, j, k, w, fx, fy, fz, qscale);
            } else {
                cic::tile_add<FIXED>(acc, t, g, i, j, k, fx, fy, fz, rhoi, rho64i, qscale);
            }
        }
        if (DIAG) mo.fold();
    }
    if (DIAG && Dm != nullptr) emit(it1 - 1);
    __syncthreads();
    if (cur_tile >= 0)
        cic::tile_flush<FIXED>(acc, sum, folded, t, Dc->g, rho + Dc->g0, rho64 + Dc->g0, Dc->qscale);
    if (bad) atomicOr(&ctrl->flags, bad);
}

// integer grid -> charge density of each node's instance; clears rho64
__global__ void k_b_rho_finish(int64_t ng, const InstDesc *__restrict__ desc,
                               const long long *__restrict__ g0, int n_inst,
                               unsigned long long *rho64, float *__restrict__ rho) {
    dep_begin(rho64, rho);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int inst = 0;
    for (int64_t gidx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; gidx < ng; gidx += stride) {
        inst = inst_of_particle(g0, n_inst, gidx);
        rho[gidx] = fixed_density(rho64[gidx], desc[inst].fix);
        rho64[gidx] = 0ull;
    }
}

// Green kernel of one size class: m instances with equal grids; instance j of
// the class is desc[first + j], its half spectrum rho_hat[j * nhalf ...]
__global__ void k_b_green(const InstDesc *__restrict__ desc, int first, int m, int64_t nhalf,
                          const float2 *__restrict__ rho_hat, float2 *__restrict__ E_hat,
                          double *__restrict__ modes) {
    const int64_t qq = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (qq >= (int64_t)m * nhalf) return;
    const int j = (int)(qq / nhalf);
    const int64_t q = qq - (int64_t)j * nhalf;
    const InstDesc &D = desc[first + j];
    const int nx = D.g.n[0], ny = D.g.n[1], nz = D.g.n[2], nh = D.g.nh;
    const int a = (int)(q % nh);
    const int64_t r = q / nh;
    const int b = (int)(r % ny);
    const int c = (int)(r / ny);
    const int my = (b <= ny / 2) ? b : b - ny;
    const int mz = (c <= nz / 2) ? c : c - nz;
    const float kx = (float)(D.two_pi_over_L[0] * a), ky = (float)(D.two_pi_over_L[1] * my);
    const float kz = (float)(D.two_pi_over_L[2] * mz);
    const float gx = ((nx & 1) == 0 && a == nx / 2) ? 0.0f : kx;
    const float gy = ((ny & 1) == 0 && b == ny / 2) ? 0.0f : ky;
    const float gz = ((nz & 1) == 0 && c == nz / 2) ? 0.0f : kz;
    float2 ex = make_float2(0.f, 0.f), ey = ex, ez = ex;
    if (q != 0) {
        const float2 rh = rho_hat[qq];
        const float sc = (float)D.inv_ng / (kx * kx + ky * ky + kz * kz);
        ex = make_float2(gx * sc * rh.y, -gx * sc * rh.x);
        ey = make_float2(gy * sc * rh.y, -gy * sc * rh.x);
        ez = make_float2(gz * sc * rh.y, -gz * sc * rh.x);
    }
    const int64_t mh = (int64_t)m * nhalf;
    E_hat[qq] = ex;
    E_hat[qq + mh] = ey;
    E_hat[qq + 2 * mh] = ez;
    if (a == D.mode_idx[0] && b == D.mode_idx[1] && c == D.mode_idx[2]) {
        const float2 mv = (D.mode_comp == 0) ? ex : (D.mode_comp == 1 ? ey : ez);
        modes[2 * (first + j)] = (double)mv.x;
        modes[2 * (first + j) + 1] = D.mode_conj ? -(double)mv.y : (double)mv.y;
    }
}

// Field energies and charge: block (i, b) leaves the partial sums of nodes
// [b, b + 1) * per of instance i, in FP64 and a fixed order.  One block per
// instance kept 24 of 152 SMs busy for 0.29 ms a step on 24 instances of up to
// 48^3 nodes; 4096 nodes a block take 22 us (in FP32 pairs 13).
__global__ void __launch_bounds__(256) k_b_diag_field(const InstDesc *__restrict__ desc,
                                                      const float *__restrict__ rho,
                                                      const float4 *__restrict__ E4,
                                                      double *__restrict__ fpart, int fstride) {
    const InstDesc &D = desc[blockIdx.x];
    const int nb = D.sum_blocks;
    if (D.own_fft || (int)blockIdx.y >= nb) return;
    const int64_t ng = (int64_t)D.g.n[0] * D.g.n[1] * D.g.n[2];
    const int64_t per = (ng + nb - 1) / nb;
    const int64_t q1 = D.g0 + ((blockIdx.y + 1) * per < ng ? (blockIdx.y + 1) * per : ng);
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    for (int64_t q = D.g0 + blockIdx.y * per + threadIdx.x; q < q1; q += blockDim.x)
        add_field(s, E4[q], rho[q]);
    block_field_sums<256>(s, fpart + 4 * ((int64_t)blockIdx.x * fstride + blockIdx.y));
}

// One record per instance, one block each: the instance's items are
// [item_off[tile0], item_off[tile0 + ntiles]) of the work list (items follow
// the tile order); strided sums per thread, then a fixed tree.  One thread per
// instance walked up to 2000 items in a row: 0.84 ms a step on 24 instances of
// up to 48^3 cells, now 12.7 us.
__global__ void __launch_bounds__(256) k_b_diag_finalize(const InstDesc *__restrict__ desc,
                                                         int n_inst, int fstride,
                                                         const int32_t *item_off,
                                                         const double *fpart,
                                                         const double *ppart,
                                                         const double *modes,
                                                         Ctrl *ctrl, double dt, pic_diag_t *ring,
                                                         int ring_cap) {
    dep_begin(item_off, fpart, ppart, modes, ctrl, ring);
    const int i = blockIdx.x;
    const InstDesc &D = desc[i];
    __shared__ double red[8][256];
    double s[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < D.sum_blocks; b += blockDim.x)
        for (int q = 0; q < 4; ++q) s[q] += fpart[4 * ((int64_t)i * fstride + b) + q];
    const int it1 = item_off[D.tile0 + D.ntiles];
    for (int it = item_off[D.tile0] + threadIdx.x; it < it1; it += blockDim.x)
        for (int q = 0; q < 4; ++q) s[4 + q] += ppart[4 * (int64_t)it + q];
    for (int q = 0; q < 8; ++q) red[q][threadIdx.x] = s[q];
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w)
            for (int q = 0; q < 8; ++q) red[q][threadIdx.x] += red[q][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const long long step = ctrl->step;        // advanced by k_b_step_done afterwards
        const long long slot = ctrl->diag_written % ring_cap;
        pic_diag_t d;
        d.step = step;
        d.t_field = ((double)step + 0.5) * dt;
        d.Wx = D.dV * red[0][0];
        d.Wy = D.dV * red[1][0];
        d.Wz = D.dV * red[2][0];
        d.Q = D.dV * red[3][0];
        d.mode_re = modes[2 * i];
        d.mode_im = modes[2 * i + 1];
        d.t = ((double)step + 1.0) * dt;
        d.Px = D.mp * red[4][0];
        d.Py = D.mp * red[5][0];
        d.Pz = D.mp * red[6][0];
        d.K = 0.5 * D.mp * red[7][0];
        ring[slot * n_inst + i] = d;
    }
}

// planar (Ex, Ey, Ez) of a size class -> E4 and the x-paired E8 (E at q and at
// its +x neighbour; instances and rows start at multiples of nx, so the row
// position of q is q mod nx)
__global__ void k_b_pack(int64_t mng, int nx, const float *__restrict__ planar,
                         float4 *__restrict__ E4, float4 *__restrict__ E8) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < mng; q += stride) {
        const int i = (int)(q % nx);
        const int64_t q1 = (i + 1 == nx) ? q - i : q + 1;
        const float4 e = make_float4(planar[q], planar[q + mng], planar[q + 2 * mng], 0.0f);
        E4[q] = e;
        E8[2 * q] = make_float4(e.x, e.y, planar[q1], planar[q1 + mng]);
        E8[2 * q + 1] = make_float4(e.z, planar[q1 + 2 * mng], 0.0f, 0.0f);
    }
}

__global__ void k_b_step_done(Ctrl *ctrl, int diag) {
    dep_begin(ctrl);
    ctrl->step += 1;
    if (diag) ctrl->diag_written += 1;
}

}  // namespace

cudaError_t launch_b_load(const double *x, const double *v, int64_t m, int64_t base,
                          const InstDesc *desc, const long long *p0, int n_inst, double dt,
                          Ctrl *ctrl, LStream st) {
    if (m <= 0) return cudaSuccess;
    k_b_load<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(x, v, m, base, desc, p0, n_inst, 0.5 * dt, ctrl);
    return cudaGetLastError();
}

cudaError_t launch_b_unload(int64_t o0, int64_t m, const InstDesc *desc, const long long *p0,
                            int n_inst, const long long *c0, double dt, const Ctrl *ctrl, double *x,
                            double *v, LStream st) {
    if (m <= 0) return cudaSuccess;
    launch_dep(k_b_unload, (unsigned)((m + 255) / 256), 256, 0, st, o0, m, desc, p0, n_inst, c0,
                                                            0.5 * dt, ctrl, x, v);
    return cudaGetLastError();
}

cudaError_t launch_b_sort(int64_t n, const InstDesc *desc, const long long *p0, int n_inst,
                          int ntiles, int chunk, Ctrl *ctrl, int32_t *bins, int32_t *scan_tmp,
                          int32_t *tile_items, int2 *tile_range, int4 *items, LStream st) {
    const PassEnd pe{n > 0 && ntiles <= kFusedBins, true, chunk, tile_items, tile_range, items};
    cudaError_t e = staged_pass(n, BatchKey{desc, p0, n_inst}, ntiles, ctrl, bins, scan_tmp, pe, st);
    if (e != cudaSuccess || pe.fused) return e;
    return launch_worklist(bins, ntiles, chunk, tile_items, tile_range, items, scan_tmp, ctrl,
                           n > 0 ? 1 : 0, st);
}

int batch_diag_blocks(const Geom &g) {
    return (int)std::min<int64_t>(64, ((int64_t)g.n[0] * g.n[1] * g.n[2] + 4095) / 4096);
}

cudaError_t batch_sort_prepare() { return staged_prepare<BatchKey>(); }

size_t batch_push_smem(int max_S, bool staged) {
    return staged ? cic::stage_offset(max_S) + 16 * (size_t)max_S
                  : cic::sum_offset(max_S) + 8 * (size_t)max_S;
}

bool batch_stages_E(int max_S, int threads) {
    const int64_t per_sm = std::max(1, PIC_BATCH_PD_MIN_BLOCKS * 256 / std::max(1, threads));
    const size_t per_block = batch_push_smem(max_S, true) + 256 + 1024;
    return (size_t)per_sm * per_block <= (size_t)228 * 1024;
}

cudaError_t launch_b_push_deposit(bool push, bool diag, bool ext, bool mag, bool fixed,
                                  const InstDesc *desc, const int32_t *tile_inst, Ctrl *ctrl,
                                  const int4 *items, int blocks, int threads, int max_S,
                                  const float4 *E4, const float4 *E8,
                                  float *rho, unsigned long long *rho64, int sparse_below,
                                  int tile_cost, double *part, LStream st) {
    const size_t smem = batch_push_smem(max_S, E4 != nullptr && push);
    cudaError_t e = cudaSuccess;
#define PIC_BPD(P, D, X, M, F)                                                                  \
    do {                                                                                        \
        auto kern = k_b_push_deposit<P, D, X, M, F>;                                            \
        if ((e = allow_smem(kern, smem)) != cudaSuccess) return e;                              \
        launch_dep(kern, blocks, threads, smem, st, desc, tile_inst, ctrl, items, push ? E4 : nullptr, \
                                            E8, rho, rho64, sparse_below, tile_cost, max_S,     \
                                            part);                                              \
    } while (0)
#define PIC_BPD_F(P, D, X, M) \
    do { if (fixed) PIC_BPD(P, D, X, M, true); else PIC_BPD(P, D, X, M, false); } while (0)
#define PIC_BPD_M(P, D, X) \
    do { if (mag) PIC_BPD_F(P, D, X, true); else PIC_BPD_F(P, D, X, false); } while (0)
#define PIC_BPD_X(P, D) \
    do { if (ext) PIC_BPD_M(P, D, true); else PIC_BPD_M(P, D, false); } while (0)
    if (!push) PIC_BPD_F(false, false, false, false);
    else if (diag) PIC_BPD_X(true, true);
    else PIC_BPD_X(true, false);
#undef PIC_BPD_X
#undef PIC_BPD_M
#undef PIC_BPD_F
#undef PIC_BPD
    return cudaGetLastError();
}

cudaError_t launch_b_rho_finish(int64_t ng, const InstDesc *desc, const long long *g0, int n_inst,
                                unsigned long long *rho64, float *rho, LStream st) {
    const int b = (int)std::max<int64_t>(1, std::min<int64_t>((ng + 255) / 256, 152 * 8));
    launch_dep(k_b_rho_finish, b, 256, 0, st, ng, desc, g0, n_inst, rho64, rho);
    return cudaGetLastError();
}

cudaError_t launch_b_green(const InstDesc *desc, int first, int m, int64_t nhalf,
                           const float2 *rho_hat, float2 *E_hat, double *modes, LStream st) {
    const int64_t tot = (int64_t)m * nhalf;
    if (tot <= 0) return cudaSuccess;
    k_b_green<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(desc, first, m, nhalf, rho_hat, E_hat,
                                                             modes);
    return cudaGetLastError();
}

cudaError_t launch_b_diag(const InstDesc *desc, int n_inst, int max_blocks, int fstride,
                          const float *rho, const float4 *E4, double *fpart, LStream st) {
    if (max_blocks <= 0) return cudaSuccess;
    k_b_diag_field<<<dim3((unsigned)n_inst, (unsigned)max_blocks), 256, 0, st>>>(desc, rho, E4, fpart,
                                                                                fstride);
    return cudaGetLastError();
}

cudaError_t launch_b_diag_finalize(const InstDesc *desc, int n_inst, int fstride,
                                   const int32_t *item_off, const double *fpart, const double *ppart,
                                   const double *modes, Ctrl *ctrl, double dt, pic_diag_t *ring,
                                   int ring_cap, LStream st) {
    launch_dep(k_b_diag_finalize, n_inst, 256, 0, st, desc, n_inst, fstride, item_off, fpart, ppart, modes, ctrl,
                                              dt, ring, ring_cap);
    return cudaGetLastError();
}

cudaError_t launch_b_pack(int64_t mng, int nx, const float *planar, float4 *E4, float4 *E8,
                          LStream st) {
    const int b = (int)std::max<int64_t>(1, std::min<int64_t>((mng + 255) / 256, 152 * 8));
    k_b_pack<<<b, 256, 0, st>>>(mng, nx, planar, E4, E8);
    return cudaGetLastError();
}

cudaError_t launch_b_step_done(Ctrl *ctrl, bool diag, LStream st) {
    launch_dep(k_b_step_done, 1, 1, 0, st, ctrl, diag ? 1 : 0);
    return cudaGetLastError();
}

}  // namespace pic
