// Internal declarations of the GB300 PIC library: device data layout,
// kernel launchers and the handle.  Not part of the C ABI (see pic.h).
#pragma once

#include <cuda_runtime.h>
#include <cufft.h>
#include <stdint.h>

#include "pic.h"

namespace pic {

// ----------------------------------------------------------------------------
// Dependent launches.  A kernel launched by launch_dep on a stream with dep set may
// be put on the SMs while the kernel before it in the stream still runs
// (programmatic dependent launch); its first statement, dep_begin, lets the kernel
// after it do the same and waits until the one before has finished, its writes
// visible.  A kernel that begins so may also be launched plainly.
//
// Such a kernel runs while the one before writes what it is going to read, so none of
// that may be declared constant for the kernel: dep_begin takes its pointers (all but
// those of tables written at bind) and hands them back through an addition that the
// compiler cannot look through, so that no access moves above the wait, and those that
// are only read carry no __restrict__, which allows loads past the coherent cache.
//
// Small runs spend a quarter of their time between kernels: 20 steps of 16^3 x 8
// took 1.41 ms, now 1.08; a gradient in a 24^3 trap 2.74, now 2.26.  Large ones lose:
// the waiting blocks' shared memory is taken from the L1 that gathers rely on (the
// split cycle at 16.8M particles went from 4.06 to 6.25 ms, the 130M Penning bunch
// from 49.8 to 51.4), so only whole steps of at most kDepMaxParticles set it.
// ----------------------------------------------------------------------------
struct LStream {
    cudaStream_t s;
    bool dep;
    LStream(cudaStream_t s_ = nullptr, bool dep_ = false) : s(s_), dep(dep_) {}
    operator cudaStream_t() const { return s; }
};
constexpr int64_t kDepMaxParticles = (int64_t)1 << 23;
// dependent launches on `st` within a scope
struct DepScope {
    LStream &st;
    DepScope(LStream &st_, bool on) : st(st_) { st.dep = on; }
    ~DepScope() { st.dep = false; }
};
template <class... P>
__device__ __forceinline__ void dep_begin(P &...p) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if constexpr (sizeof...(P) > 0) {
        long long zero;
        asm volatile("mov.b64 %0, 0;" : "=l"(zero)::"memory");
        ((p += zero), ...);
    }
}
template <class... P, class... A>
inline cudaError_t launch_dep(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, const LStream &st,
                              A... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st.s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = st.dep ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// ----------------------------------------------------------------------------
// Particle store: structure of arrays, 32 bytes per particle.
//   cell  packed stencil-base cell (i | j << 10 | k << 20), i.e. the node
//         index of the lower corner of the particle's CIC stencil
//   o[3]  FP32 offset in [0, 1) of the position from that node, in cells
//   v[3]  FP32 velocity
//   pid   load-order index (touched only by the sort and the readback)
// Two sets exist; the sort scatters from the current one into the other and
// flips Ctrl::cur on the device, so captured CUDA graphs stay valid.
// ----------------------------------------------------------------------------
struct ParticleSet {
    int32_t *cell;
    float *o[3];
    float *v[3];
    int32_t *pid;
};

// Device control block (lives in the arena).  Everything before `cur` is
// cleared when particles are loaded.
struct Ctrl {
    int32_t flags;          // PIC_FLAG_* bits, OR-ed by kernels
    int32_t n_items;        // deposit work items built by the last sort
    unsigned long long stray;   // particles deposited outside their tile (stat)
    long long step;         // steps since the last load
    long long diag_written; // diagnostic records written since the load
    double mode[2];         // tracked Fourier coefficient of the last solve
    double scalar[2];       // objective and dot-product results
    // adjoint sweep: bit patterns of non-negative float maxima (atomicMax on
    // the bits orders them), double-buffered by step parity: |ly|, |lv| of
    // the multipliers and |lrho| of the last adjoint solve
    unsigned int adj_ly[2], adj_lv[2], adj_lrho[2];
    // stray-triggered re-binning: strays of the last push (summed by the push
    // kernels, cleared by each re-binning decision and each re-binning), the
    // pushes since the last re-binning, re-binnings since the load, and the
    // gate the decision sets for the sort kernels of the current step
    unsigned long long stray_step;
    long long rebins;
    int32_t since_sort;
    int32_t rebin;
    unsigned int done[2];   // blocks done, of the histogram and the scatter (0 between launches)
    int32_t cur;            // which ParticleSet holds the particles
    int32_t pad0;
    ParticleSet sets[2];
};

constexpr int kCellBits = 10;
constexpr int kCellMask = (1 << kCellBits) - 1;
constexpr int kMaxN = 1 << kCellBits;      // 1024 nodes per axis

__host__ __device__ __forceinline__ int32_t pack_cell(int i, int j, int k) {
    return i | (j << kCellBits) | (k << (2 * kCellBits));
}
__host__ __device__ __forceinline__ int cell_i(int32_t c) { return c & kCellMask; }
__host__ __device__ __forceinline__ int cell_j(int32_t c) { return (c >> kCellBits) & kCellMask; }
__host__ __device__ __forceinline__ int cell_k(int32_t c) { return (c >> (2 * kCellBits)) & kCellMask; }

// Whether q names one of n particles.  A re-binning that gave up (PIC_FLAG_TIMEOUT)
// leaves slots that it did not write, in which the other set's former contents, a
// readback's records among them, stand for load indices, and an index that no slot holds
// keeps whatever an inverse of the order had there: what follows such an index asks first.
__device__ __forceinline__ bool is_particle(int32_t q, int64_t n) {
    return (uint64_t)(int64_t)q < (uint64_t)n;
}

// Grid geometry passed by value to kernels.
struct Geom {
    int n[3];          // nodes per axis
    int nh;            // Nx/2 + 1 (R2C innermost length)
    int tile[3];       // deposit tile (cells per axis)
    int ntile[3];      // tiles per axis = ceil(n / tile)
    int guard;         // guard layers around a tile
    int tvol;          // tile[0]*tile[1]*tile[2]
    unsigned tdiv[3];  // ceil(2^32 / tile[d]), 0 for a tile of 1 (see tile_div)
    float h[3];        // cell size
    float inv_h[3];
};

// a / tile[d] for 0 <= a < 1024 by a multiply-high (exact: the rounding of the
// reciprocal adds less than 2^-22 to a quotient whose fraction is <= 1 - 1/1024)
__device__ __forceinline__ int tile_div(int a, unsigned tdiv) {
    return tdiv ? (int)__umulhi((unsigned)a, tdiv) : a;
}

// Per-step push constants (FP32, precomputed on the host in FP64).
struct PushConst {
    float qm_half_dt;      // (q/m) dt / 2
    float dt_over_h[3];    // dt / h_d
    float t[3];            // (q/m) B dt / 2
    float s[3];            // 2 t / (1 + |t|^2)
    float wz2;             // quadrupole strength
    float half_n[3];       // N_d / 2 (box centre in cells)
};

// Diagnostic partial layout: 4 doubles per block.
constexpr int kDiagFieldBlocks = 152 * 8;
constexpr int kNumSMs = 152;   // streaming multiprocessors of the GPU (two dies of 76)
constexpr int kMaxPushBlocks = kNumSMs * 8;
constexpr int kMaxSmemPerBlock = 227 * 1024;   // opt-in shared memory per block
// Lets a kernel be launched with `need` bytes of dynamic shared memory.  The limit belongs
// to the function, which every handle of the process shares, so it is always set to all
// that its static memory leaves: set to a handle's own need, it would be lowered under
// another handle (or a captured graph) that needs more.
template <class K>
inline cudaError_t allow_smem(K *kernel, size_t need) {
    if (need <= 48 * 1024) return cudaSuccess;
    cudaFuncAttributes a;
    const cudaError_t e = cudaFuncGetAttributes(&a, kernel);
    if (e != cudaSuccess) return e;
    const size_t most = kMaxSmemPerBlock - a.sharedSizeBytes;
    if (need > most) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}
// threads per SM the fused push + deposit kernel is compiled for (80 registers)
constexpr int kPushThreadsPerSM = 768;
// resident blocks per SM of the uniform-plasma move + deposit
#ifndef PIC_MV_MIN_BLOCKS
#define PIC_MV_MIN_BLOCKS 4
#endif
// resident blocks per SM of the split-call deposit
#ifndef PIC_DEP_MIN_BLOCKS
#define PIC_DEP_MIN_BLOCKS 4
#endif
// read and write page-locked host particle arrays in place (no staging copies)
#ifndef PIC_ZERO_COPY
#define PIC_ZERO_COPY 1
#endif
constexpr int kMaxChunk = 4095;   // fixed-point tile slots stay below 2^32

// Set the thread-local message returned by pic_last_error(); returns `code`.
int record_error(int code, const char *fmt, ...);

// Work items: int4 (tile, begin, end of its tile, first item of the next tile).  A tile of
// cnt particles is split into ceil(cnt / chunk) items of equal size; items only
// say where a block's run may begin and end, and a block walks the particles of
// its run tile by tile (next_segment), so small items cost it nothing.
//
// The run of work items [it0, it1) of this block.  Items cover the particles
// [0, P) in order; a tile costs its particles plus tile_cost for its staging and
// flush, so the cost before item i is y_i + tile_cost r_i with r_i the tiles with
// particles before the item's (kept below the items, see item_rank), and the block
// takes the items that start within its equal share of the total (with fewer items
// than blocks, block b takes item b).
//
// With at most 4095 particles an item, 4.2M particles on 512 tiles of 8192 gave
// a block two or three items (9200 particles), and 33k particles on 8 tiles kept
// 9 of 456 blocks busy; sixteen items a block (256..4095 particles) keep the
// shares within a few percent (push 110 -> 101 us and 40.6 -> 17.4 us).
//
// A tile's cost in particles (kTileCost) shows where tiles differ: with an item's
// cost instead, a quarter of its size, blocks among the thin tiles at the end of a
// 41^3 grid or around a bunch switched tiles up to eighteen times while the others
// did not (14 steps of 2.5M particles 2.25 ms, now 1.73; the Penning bunch in 256^3,
// 10 steps, 45.2 -> 44.7; with a cost of 512 1.92
// and 46.1, of 4096 1.79 and 45.7).  It is at most half a block's particles, as every
// block stages one tile whatever its share.
constexpr int kItemsPerBlock = 16;
constexpr int kTileCost = 2048;
inline int tile_cost_of(int64_t n, int64_t blocks) {
    return (int)std::max<int64_t>(1, std::min<int64_t>(kTileCost, n / (2 * blocks)));
}
constexpr int kMinChunk = 256;
// Called by every thread of the block (it synchronises): the two item
// indices are found by a two-level search in which each thread tests one
// sample per round, so a block start costs a few dependent loads (two while
// n_items <= blockDim^2), not log2(n_items).
// The rank of item i, kept before the items in falling order
__device__ __forceinline__ int32_t *item_rank(int4 *items, int i) {
    return reinterpret_cast<int32_t *>(items) - 1 - i;
}
__device__ __forceinline__ int item_rank(const int4 *items, int i) {
    return reinterpret_cast<const int32_t *>(items)[-1 - i];
}
// bytes of the ranks before the items
inline size_t rank_bytes(int64_t max_items) { return ((size_t)max_items * 4 + 255) / 256 * 256; }

__device__ __forceinline__ void item_run(const int4 *items, int n_items,
                                         long long tile_cost, int &it0, int &it1) {
    if (n_items <= (int)gridDim.x) {
        // at most one item per block: consecutive blocks (spread over the SMs)
        // take consecutive items, however large
        it0 = min((int)blockIdx.x, n_items);
        it1 = min((int)blockIdx.x + 1, n_items);
        return;
    }
    const long long total =
        n_items > 0 ? (long long)items[n_items - 1].z + tile_cost * (item_rank(items, n_items - 1) + 1) : 0;
    const long long c0 = total * blockIdx.x / gridDim.x;
    const long long c1 = total * (blockIdx.x + 1) / gridDim.x;
    auto cost = [&](int i) { return (long long)items[i].y + tile_cost * item_rank(items, i); };
    // level 1: sample i_t = (t + 1) * step - 1; the first index with cost >= c lies
    // in the step-wide bucket after the last sample below c
    const int nt = (int)blockDim.x;
    const int step = (n_items + nt - 1) / nt;   // >= 1 when n_items > 0
    const int t = (int)threadIdx.x;
    const int si = min((t + 1) * step, n_items) - 1;
    const long long cs = (n_items > 0 && si >= 0) ? cost(si) : 0;
    const int b0 = __syncthreads_count(n_items > 0 && si >= 0 && cs < c0 && (t + 1) * step <= n_items);
    const int b1 = __syncthreads_count(n_items > 0 && si >= 0 && cs < c1 && (t + 1) * step <= n_items);
    // level 2: the first index with cost >= c lies in [b * step, min(n, (b + 1) * step)):
    // count the costs below c there, blockDim at a time
    const int lo0 = b0 * step, lo1 = b1 * step;
    const int hi0 = min(n_items, lo0 + step), hi1 = min(n_items, lo1 + step);
    int r0 = 0, r1 = 0;
    for (int k = 0; k < step; k += nt) {
        const int j0 = lo0 + k + t, j1 = lo1 + k + t;
        r0 += __syncthreads_count(j0 < hi0 && cost(j0) < c0);
        r1 += __syncthreads_count(j1 < hi1 && cost(j1) < c1);
    }
    it0 = min(n_items, lo0 + r0);
    it1 = blockIdx.x + 1 == gridDim.x ? n_items : min(n_items, lo1 + r1);
}

// Index of a particle in the walk over a tile.  Unsigned: a stride past the last of
// 2^31 - 1 particles stays above it (as an int it would be negative, and so below).
using PIndex = uint32_t;

// The particles [begin, end) of one tile, of a block's run [it, it1) of items;
// next_segment moves on to the next tile.  Its item is loaded there: neighbours share a
// line, and held over a tile's particles it costs the push, at its register limit, more
// than the wait (256^3 x 8, four steps: 13.3 ms of pushes, so 12.85).
struct Segments {
    const int4 *items;
    int it, it1, pb;   // pb: the run's last particle + 1
};
__device__ __forceinline__ Segments run_segments(const int4 *items, int n_items,
                                                 long long tile_cost) {
    Segments r;
    r.items = items;
    item_run(items, n_items, tile_cost, r.it, r.it1);
    r.pb = 0;
    if (r.it < r.it1) r.pb = r.it1 < n_items ? items[r.it1].y : items[n_items - 1].z;
    return r;
}
__device__ __forceinline__ bool next_segment(Segments &r, int &tile, PIndex &begin, PIndex &end) {
    if (r.it >= r.it1) return false;
    const int4 i = r.items[r.it];
    tile = i.x;
    begin = i.y;
    end = min(i.z, r.pb);
    r.it = i.w;
    return true;
}

// ----------------------------------------------------------------------------
// kernel launchers (defined in the k_*.cu files); all enqueue on `st`.
// ----------------------------------------------------------------------------
// max_blocks > 0 caps the grid (blocks then stride over the particles)
cudaError_t launch_load(const double *x, const double *v, int64_t m, int64_t base,
                        const Geom &g, const double *inv_h_d, double dt, Ctrl *ctrl,
                        LStream st, int max_blocks = 0);
// readback in load order: the current set's particles as 32-byte records (by
// pid) in the other set, or the inverse of the store's order (inv[pid]); then
// particles [o0, o0 + m) of n as FP64 triples from the records (inv null) or through
// inv; node_pos: kMaxN node positions (i + 1/2) h per axis
cudaError_t launch_unload_records(int64_t n, const Ctrl *ctrl, LStream st);
cudaError_t launch_invperm(int64_t n, const Ctrl *ctrl, int32_t *inv, LStream st);
void node_positions(const double *h_d, double *node_pos);
cudaError_t launch_unload(int64_t o0, int64_t m, int64_t n, const int32_t *inv, const double *node_pos,
                          const double *h_d, const double *L_d, double dt, const Ctrl *ctrl,
                          double *x, double *v, LStream st);

cudaError_t exclusive_scan(int32_t *data, int64_t n, int32_t *tmp, LStream st,
                           const int32_t *gate = nullptr);
cudaError_t sort_prepare();   // kernel attributes; call once per device outside capture
cudaError_t launch_worklist(const int32_t *bin_end, int ntiles, int chunk, int32_t *tile_items,
                            int2 *tile_range, int4 *items, int32_t *scan_tmp, Ctrl *ctrl, int flip,
                            LStream st);
// presort: the particles are in arbitrary order (just loaded); coarse passes
// by tile key >> shift run first so that no slice overflows the staged table
// gate != nullptr: every kernel of the sort returns at once unless *gate is
// nonzero on the device (the stray-triggered re-binning of pic_step)
cudaError_t launch_sort(int64_t n, const Geom &g, int chunk, Ctrl *ctrl, int32_t *bins,
                        int64_t nbins, int32_t *scan_tmp, int32_t *tile_items,
                        int2 *tile_range, int4 *items, bool presort, LStream st,
                        const int32_t *gate = nullptr);
// ctrl->rebin = (period > 0 and ctrl->since_sort >= period) or
// ctrl->stray_step > max_strays; clears ctrl->stray_step
cudaError_t launch_rebin_decide(Ctrl *ctrl, long long max_strays, int period, LStream st);
// kernels launch_sort issues
int sort_launches(int64_t n, int64_t ntiles, bool presort);
int presort_passes(int64_t ntiles);   // coarse passes of a presort
// coarse passes + full-key pass over particles [o, o + n) of the current set
// (which stays unchanged); the range ends in set cur ^ (*passes & 1)
cudaError_t launch_sort_range(int64_t n, int64_t o, const Geom &g, Ctrl *ctrl, int32_t *bins,
                              int64_t nbins, int32_t *scan_tmp, int *passes, int *kernels,
                              LStream st);
cudaError_t launch_flip(Ctrl *ctrl, LStream st);   // ctrl->cur = 1 - ctrl->cur
// one bounded wait that nothing completes: raises PIC_FLAG_TIMEOUT (pic_selftest_timeout)
cudaError_t launch_timeout_selftest(Ctrl *ctrl, LStream st);

cudaError_t launch_deposit(int64_t n, const Geom &g, const Ctrl *ctrl, const int4 *items,
                           int max_items, double qscale, float *rho, unsigned long long *rho64,
                           bool fixed, Ctrl *ctrl_w, int grid_blocks, int sparse_below,
                           int tile_cost, LStream st);

cudaError_t launch_rho_finish(const Geom &g, unsigned long long *rho64, float *rho, double qscale,
                              LStream st);
// the uniform-plasma random move (PIC_OPT_UNIFORM_MOVE) of every particle,
// with the deposit of the new positions when `deposit` (then over the work
// items, like launch_push_deposit); advances the device step counter
cudaError_t launch_move(int64_t np, const Geom &g, uint64_t seed, bool diag, bool fixed, bool deposit,
                        Ctrl *ctrl, const int4 *items, int max_items, float *rho,
                        unsigned long long *rho64, double qscale, int sparse_below, int tile_cost,
                        double *part, int blocks, LStream st);
// block size, blocks per SM, whether the blocks stage E, and the dynamic shared
// memory of the fused push + deposit kernel for geometry g; the one-time
// attribute setting it needs above 48 KiB
struct PushShape {
    int threads, per_sm;
    bool staged;
    int e_guard;   // guard layers of the staged box
    size_t smem;
};
PushShape push_shape(const Geom &g);
size_t tile_deposit_smem(const Geom &g);   // the deposit tiles alone (unstaged kernels)
// the box edge compiled as a constant into the tiled kernels: 8^3 tiles with two
// guard layers (the default geometry)
constexpr int kConstBox = 13;
bool const_box(const Geom &g);
cudaError_t push_deposit_prepare(const Geom &g);
cudaError_t deposit_prepare(const Geom &g);
cudaError_t adj_prepare(const Geom &g);
// Optional copy of the positions a push starts from (cell, o[3]), written by
// the fused kernel as it reads them (the adjoint keeps each step's y).
struct SaveY {
    int32_t *cell;
    float *o[3];
    float *v[3];   // also the velocities before the kick (null: not saved)
};
// E8: the x-paired field (launch_pack_E), 2 float4 per node
cudaError_t launch_push_deposit(const Geom &g, const PushConst &pc, bool diag, bool fixed,
                                Ctrl *ctrl, const int4 *items, int max_items, const float4 *E8,
                                float *rho, unsigned long long *rho64, double qscale,
                                int sparse_below, int tile_cost, double *part, int blocks,
                                const SaveY &save, LStream st);
cudaError_t launch_gather_push(int64_t n, const Geom &g, const PushConst &pc, bool diag,
                               Ctrl *ctrl, const float4 *E8, double *part, int blocks,
                               int threads, LStream st);
// E as cuFFT left it, one float4 per node (interleaved) or planar in the place of its
// spectra, -> the x-paired E8 (Ex Ey Ex' Ey' Ez Ez' 0 0 per node, primed at q + x, periodic),
// and unless null the partial field sums of kDiagFieldBlocks blocks
cudaError_t launch_pack_E(const Geom &g, const float *E, bool interleaved, float4 *E8, float *rho,
                          bool clear_rho, double *part, LStream st);
// E8 -> (Ex, Ey, Ez, 0) per node
cudaError_t launch_unpair_E(int64_t ng, const float4 *E8, float4 *E4, LStream st);

// FP32 wavenumbers of every FFT index per axis (x: nh, y: ny, z: nz entries)
void green_table(const Geom &g, const double *L_d, float *ktab);
cudaError_t launch_green(const Geom &g, const float *ktab, const float2 *rho_hat,
                         float2 *E_hat, int64_t nhalf, const int *mode_idx, int mode_comp,
                         int mode_conj, Ctrl *ctrl, LStream st);
cudaError_t launch_diag_finalize(const double *field_part, int field_blocks,
                                 const double *push_part, int push_blocks, double dV, double mp, double dt,
                                 Ctrl *ctrl, pic_diag_t *ring, int ring_cap, LStream st);

// Field solve by the library's own line transforms (k_fft.cu), for grids whose
// axes are at most kFftMaxN long with no prime factor above 7 and whose (y, z)
// planes fit (fft_supported); others go through cuFFT.
constexpr int kFftMaxN = 128;
constexpr int kFftMaxStages = 4;
struct FftAxis {
    int n, stages;
    int radix[kFftMaxStages];   // forward order
};
// per axis: exp(-2 pi i k / n) and the position of frequency k after a forward
// transform
struct FftTables {
    float2 tw[3][kFftMaxN];
    int pos[3][kFftMaxN];
};
bool fft_axis(int n, FftAxis &a);   // false: not supported
bool fft_supported(const Geom &g, FftAxis ax[3]);
int fft_ktab_size(const Geom &g);   // wavenumber table of one grid for these kernels
void fft_ktab(const Geom &g, const double *L_d, const FftTables &t, float *out);
void fft_tables(const FftAxis ax[3], FftTables &t);
int fft_sum_blocks(const Geom &g);   // blocks that leave partial field sums
cudaError_t fft_prepare();           // kernel attributes; outside any stream capture
// rho (cleared on the way for an FP32 deposit with clear_rho) -> E8 (and E4 and
// fpart, 4 doubles per block, unless null) of m <= 65535
// grids of one size in a row, spectra in a row too; mode_idx are positions in y
// and z; grid j has the wavenumbers
// ktab + j fft_ktab_size, leaves its tracked mode in mode[2 j] and [2 j + 1] and its
// sums from fpart + 4 j fstride on
cudaError_t launch_fft_solve(const Geom &g, int m, const FftAxis ax[3], const FftTables *tab,
                             const float *ktab, float *rho, bool clear_rho, float2 *rho_hat, float2 *E_hat,
                             int64_t nhalf, const int *mode_idx, int mode_comp, int mode_conj,
                             double *mode, float4 *E4, float4 *E8, double *fpart, int fstride,
                             LStream st);
// lE4 (cleared) -> lrho2, with the bound bookkeeping of launch_adj_pair_rho
cudaError_t launch_fft_adj_solve(const Geom &g, const FftAxis ax[3], const FftTables *tab,
                                 const float *ktab, float4 *lE4, float2 *lE_hat, float2 *lrho_hat,
                                 int64_t nhalf, float2 *lrho2, Ctrl *ctrl, int par, LStream st);

// adjoint (k_adjoint.cu)
cudaError_t launch_adj_seed(int64_t ng, const float4 *E8, float4 *lE4, const double *scale3,
                            LStream st);
// up to 8 device-to-device copies in one launch (pointers 16-byte aligned)
struct CopyList {
    int count;
    char *dst[8];
    const char *src[8];
    int64_t bytes[8];
};
cudaError_t launch_copy(const CopyList &cl, LStream st);

// The deposit term of the adjoint of one step, (dD/dy)^T lrho evaluated at
// that step's positions (cell, o) and scaled by q/h_d, folded into the
// reverse push of the step before it (cell == nullptr: no such term).
// Per-step constants of the reverse push of step n: the step's parity and the
// constants of the bound on |le| that scales the integer accumulation of
// G^T le (c = dt q/m; kb = 2 max_d |q / h_d| bounds the deposit term per unit
// |lrho|; with B, |le_d| <= (1 + sqrt 3)/2 |c| max|lv_tot|); with mag set, the
// Boris rotation R (row-major) of v' = R v + (c/2)(R + I) e.
struct AdjBound {
    int par;
    float c_abs, dt, kb;
    int mag;
    float R[9];
};
struct AdjRhoTerm {
    const int32_t *cell;
    const float *o[3];
    const float2 *lrho2;   // x-paired lrho (launch_pair_scalar)
    float sx, sy, sz;
};
// Parameter-gradient sums of one reverse step (part == nullptr: off): per
// block, A_ij = sum_p lv_tot_i vm_j (9, row-major) and sum_p le . Q(y_p)
// (Q the quadrupole direction field), from the saved velocities yv before the
// kick; half_n and h give the box centre in cells and the spacing.
struct PGrad {
    const float *yv[3];
    double *part;   // kPGradTerms doubles per block
    float half_n[3], h[3];
};
constexpr int kPGradTerms = 10;
// threads per SM the reverse push is compiled for (80 registers), its blocks for
// geometry g (see k_adjoint.cu)
constexpr int kAdjThreadsPerSM = 768;
// room in the caller's buffer, whose size is part of the interface; at most half of
// it is launched (adj_blocks)
constexpr int kAdjPushMaxBlocks = kNumSMs * 3 * 2;
struct AdjShape {
    int threads, per_sm;
    bool staged;
    size_t smem;
};
AdjShape adj_shape(const Geom &g);
int adj_blocks(const Geom &g, int max_items);
cudaError_t launch_adj_push(const Geom &g, const Ctrl *ctrl, const int4 *items, int max_items,
                            int tile_cost, const int32_t *ycell, const float *const yo[3], const float4 *E8,
                            float4 *lE4, float c_kick, float dt, float wz2, const AdjRhoTerm &rt,
                            const AdjBound &ab, const PGrad &pg, Ctrl *ctrl_w, LStream st);
// acc[q] += the fixed-order sum of the kPGradTerms partials of the blocks the
// last launch_adj_push used (max_items caps them as there)
cudaError_t launch_pgrad_acc(const Geom &g, const double *part, int max_items, double *acc,
                             LStream st);
cudaError_t launch_green_adj(const Geom &g, const double *L_d, const float2 *lE_hat,
                             float2 *lrho_hat, int64_t nhalf, LStream st);
// where k_adj_rho writes the updated multipliers (o[0] == nullptr: in place)
struct LamOut {
    float *o[3];
    float *v[3];
};
cudaError_t launch_adj_rho(int64_t n, const Geom &g, Ctrl *ctrl, const int32_t *ycell,
                           const float *const yo[3], const float2 *lrho2, float qscale,
                           const LamOut &out, int par, LStream st);
// lrho2[q] = (lrho[q], lrho[q + x (periodic)]); lE4 cleared
cudaError_t launch_adj_pair_rho(const Geom &g, const float *lrho, float2 *lrho2, float4 *lE4,
                                Ctrl *ctrl, int par, LStream st);
cudaError_t launch_adj_zero(int64_t n, const Ctrl *ctrl, LStream st);
struct ReorderArgs {
    const float *in_o[3];
    const float *in_v[3];
    float *out_o[3];
    float *out_v[3];
};
cudaError_t launch_adj_reorder(int64_t n, const int32_t *pos, const int32_t *pid_prev,
                               const float *const in_o[3], const float *const in_v[3],
                               float *const out_o[3], float *const out_v[3], LStream st);
// pos[pid[j]] = j for j < n (the inverse of a particle order)
cudaError_t launch_pid_positions(int64_t n, const int32_t *pid, int32_t *pos, LStream st);
// the multipliers in load order: records (by pid) in `rec` (32 bytes per
// particle, caller's scratch), then records [o0, o0 + m) as the gradients
cudaError_t launch_adj_unload_records(int64_t n, const Ctrl *ctrl, float4 *rec, LStream st);
cudaError_t launch_adj_unload(int64_t o0, int64_t m, const float4 *rec, double half_dt,
                              double scale, double *gx, double *gv, LStream st);
cudaError_t launch_objective(const double *fpart, int nb, double dV, const double *w,
                             double *out, LStream st);
cudaError_t launch_dot(int64_t n, const double *a, const double *b, double *part, int max_part,
                       double *out, LStream st);

}  // namespace pic
