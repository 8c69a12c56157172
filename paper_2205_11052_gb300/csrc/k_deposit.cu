// Scatter (Section 3.1 step 1 of arXiv 2205.11052) with the cloud-in-cell
// shape on the cell-centred grid of Section 3.2:
//   rho_g = sum_p q_p W(x_g - x_p) / h^3,  W = prod_d (1 - |dx_d| / h_d)_+ .
// A particle with stencil base (i, j, k) and offsets (fx, fy, fz) adds
// q_p / h^3 * w_a(fx) w_b(fy) w_c(fz) to node (i + a, j + b, k + c), a, b, c
// in {0, 1}, with w_0(f) = 1 - f and w_1(f) = f (periodic wrap).
//
// Tiled kernel: each CTA takes a contiguous run of work items (ranges of
// binned particles whose stencil base was inside one tile at the last sort;
// consecutive items share tiles) and accumulates the unscaled weights in a
// shared-memory copy of the tile plus `guard` cells on each side (plus the +1
// stencil layer), folded into per-tile sums every 4095 particles at most; both
// go to the grid with one global atomic per touched node when the run moves to
// another tile.  Particles that drifted beyond the guard since the
// last sort go straight to the grid with global atomics, so the result never
// depends on the sort cadence.  Each thread loads its next particle before
// depositing the current one.
//
// Two accumulators:
//  * FP32: float shared tile, float global atomics into rho.
//  * fixed point: the particle's 2^20 units split over its eight corners by
//    nested rounding (cic::fixed_split: they sum exactly to 2^20, none is
//    negative), u32 shared atomics (at most 4095 particles per work item, so
//    a slot cannot reach 2^32) and u64
//    global atomics into an integer grid that k_rho_finish scales into rho.
//    Integer addition is associative, so this deposit is deterministic and
//    conserves the particles' total weight exactly.
#include <algorithm>

#include "cic.cuh"
#include "ffsum.cuh"

namespace pic {

namespace {

using namespace cic;

// B > 0: every tile box is B slots long on each axis (cic::box_row)
template <bool FIXED, int B>
__global__ void __launch_bounds__(256, PIC_DEP_MIN_BLOCKS) k_deposit_tiles(Geom g, const Ctrl *ctrl,
                                                           const int4 *items,
                                                           float qscale, float *rho,
                                                           unsigned long long *rho64, Ctrl *ctrl_w,
                                                           int sparse_below, int tile_cost) {
    dep_begin(ctrl, items, rho, rho64, ctrl_w);
    extern __shared__ __align__(16) uint32_t acc[];
    const ParticleSet ps = ctrl->sets[ctrl->cur];
    const int n_items = ctrl->n_items;
    unsigned long long strays = 0;
    int bad = 0;
    Segments run = run_segments(items, n_items, tile_cost);
    const int S = tile_of(g, 0).S;
    void *sum = reinterpret_cast<char *>(acc) + sum_offset(S);
    for (int s = threadIdx.x; s < S; s += blockDim.x) {
        acc[s] = 0u;
        if (FIXED) reinterpret_cast<unsigned long long *>(sum)[s] = 0ull;
        else reinterpret_cast<float *>(sum)[s] = 0.0f;
    }
    // t: the tile of the dense segments (sparse ones go straight to the grid)
    bool any = false, folded = false;
    Tile t = tile_of(g, 0);
    int tile;
    PIndex begin, end;
    while (next_segment(run, tile, begin, end)) {
        if ((int)(end - begin) < sparse_below) {
            // few particles: skip the shared tile, add straight to the grid
            for (PIndex p = begin + threadIdx.x; p < end; p += blockDim.x) {
                int i, j, k;
                if (!decode_cell(ps.cell[p], g, i, j, k)) bad = 1;
                const float fx = ps.o[0][p], fy = ps.o[1][p], fz = ps.o[2][p];
                float w[8];
                weights(fx, fy, fz, w);
                deposit_global<FIXED>(rho, rho64, g, i, j, k, w, fx, fy, fz, qscale);
            }
            continue;
        }
        PIndex p = begin + threadIdx.x;
        int32_t nc = 0;
        float nfx = 0.f, nfy = 0.f, nfz = 0.f;
        if (p < end) {
            nc = __ldcs(ps.cell + p);
            nfx = __ldcs(ps.o[0] + p);
            nfy = __ldcs(ps.o[1] + p);
            nfz = __ldcs(ps.o[2] + p);
        }
        __syncthreads();   // every add to the tile is done
        if (any) tile_flush<FIXED>(acc, sum, folded, t, g, rho, rho64, qscale);
        any = true;
        folded = false;
        t = tile_of(g, tile);
        __syncthreads();
        for (PIndex done = begin;;) {
            done += min(end - done, fill_limit() * blockDim.x);
            for (; p < done; p += blockDim.x) {
                const int32_t c = nc;
                const float fx = nfx, fy = nfy, fz = nfz;
                const PIndex pn = p + blockDim.x;
                if (pn < end) {
                    nc = __ldcs(ps.cell + pn);
                    nfx = __ldcs(ps.o[0] + pn);
                    nfy = __ldcs(ps.o[1] + pn);
                    nfz = __ldcs(ps.o[2] + pn);
                }
                int i, j, k;
                if (!decode_cell(c, g, i, j, k)) bad = 1;
                if (!tile_add<FIXED, B>(acc, t, g, i, j, k, fx, fy, fz, rho, rho64, qscale)) ++strays;
            }
            if (done == end) break;
            __syncthreads();
            tile_fold<FIXED>(acc, sum, S);
            __syncthreads();
            folded = true;
        }
    }
    __syncthreads();
    if (any) tile_flush<FIXED>(acc, sum, folded, t, g, rho, rho64, qscale);
    if (bad) atomicOr(&ctrl_w->flags, PIC_FLAG_BAD_CELL);
    if (strays) atomicAdd(&ctrl_w->stray, strays);
}

// integer grid -> charge density, and clear the integer grid for next time;
// two nodes per thread and iteration (16-byte loads and stores of the 8-byte
// words, 8-byte stores of the densities), the odd last node by thread 0
__global__ void __launch_bounds__(256) k_rho_finish(int64_t ng, unsigned long long *rho64,
                                                    float *__restrict__ rho, FixedScale f) {
    dep_begin(rho64, rho);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t n2 = ng >> 1;
    ulonglong2 *r2 = reinterpret_cast<ulonglong2 *>(rho64);
    float2 *f2 = reinterpret_cast<float2 *>(rho);
    // two loads in flight
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n2; q += 2 * stride) {
        const bool two = q + stride < n2;
        const ulonglong2 v = __ldcs(r2 + q);
        const ulonglong2 w = two ? __ldcs(r2 + q + stride) : make_ulonglong2(0ull, 0ull);
        __stcs(f2 + q, make_float2(fixed_density(v.x, f), fixed_density(v.y, f)));
        __stcs(r2 + q, make_ulonglong2(0ull, 0ull));
        if (two) {
            __stcs(f2 + q + stride, make_float2(fixed_density(w.x, f), fixed_density(w.y, f)));
            __stcs(r2 + q + stride, make_ulonglong2(0ull, 0ull));
        }
    }
    if ((ng & 1) && blockIdx.x == 0 && threadIdx.x == 0) {
        rho[ng - 1] = fixed_density(rho64[ng - 1], f);
        rho64[ng - 1] = 0ull;
    }
}

}  // namespace

cudaError_t launch_rho_finish(const Geom &g, unsigned long long *rho64, float *rho, double qscale,
                              LStream st) {
    const int64_t ng = (int64_t)g.n[0] * g.n[1] * g.n[2];
    const int fb = (int)std::max<int64_t>(1, std::min<int64_t>((ng / 2 + 255) / 256, 152 * 8));
    launch_dep(k_rho_finish, fb, 256, 0, st, ng, rho64, rho, fixed_scale(qscale / (double)kFixOne));
    return cudaGetLastError();
}

cudaError_t deposit_prepare(const Geom &g) {
    const size_t smem = tile_deposit_smem(g);
    cudaError_t e;
    if ((e = allow_smem(k_deposit_tiles<false, 0>, smem)) != cudaSuccess ||
        (e = allow_smem(k_deposit_tiles<true, 0>, smem)) != cudaSuccess)
        return e;
    return allow_smem(k_deposit_tiles<true, kConstBox>, smem);
}

cudaError_t launch_deposit(int64_t n, const Geom &g, const Ctrl *ctrl, const int4 *items,
                           int max_items, double qscale_d, float *rho, unsigned long long *rho64,
                           bool fixed, Ctrl *ctrl_w, int grid_blocks, int sparse_below,
                           int tile_cost, LStream st) {
    (void)n;
    const float qscale = (float)qscale_d;
    const size_t smem = tile_deposit_smem(g);   // item tile + the block's tile sums
    const int blocks = grid_blocks < max_items ? grid_blocks : (max_items > 0 ? max_items : 1);
    cudaError_t e;
    const bool cbox = const_box(g);
#define PIC_DT(F, B)                                                                              \
    launch_dep(k_deposit_tiles<F, B>, blocks, 256, smem, st, g, ctrl, items, qscale, rho, rho64, ctrl_w, \
               sparse_below, tile_cost)
    if (fixed) {
        if (cbox) PIC_DT(true, kConstBox);
        else PIC_DT(true, 0);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        return launch_rho_finish(g, rho64, rho, qscale_d, st);
    }
    PIC_DT(false, 0);
#undef PIC_DT
    return cudaGetLastError();
}

}  // namespace pic
