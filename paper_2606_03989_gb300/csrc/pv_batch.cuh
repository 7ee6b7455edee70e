// Batched sweeps: many sequences (each its own image size and state) processed
// by one launch over a work list of (sequence, tile) items. The per-pixel and
// per-tile code is the single-sequence code, so each sequence's result does not
// depend on how the work is scheduled.
#pragma once

#include "pv_kernels.cuh"

namespace pv {

// Per-sequence descriptor in device memory.
template <typename T>
struct SeqDesc {
    Geometry<T> g;
    // factor weights (the same for every sequence of a batch); read per work item
    // so that nothing in the tile arithmetic is loop-invariant in the persistent
    // kernel, which keeps its code generation (and rounding) that of one tile
    Factors<T> f;
    T* state[2];
    T* in_planes[N_INPUT_PLANES];  // I_s, I_t, g_x, g_y, m_x, m_y
    Scalars* sc;
    double* partials;
    const float* frame;    // registered input buffers
    const float* normals;
    unsigned char* br;     // decisions of the sweep, recorded for the adjoint (or null)
    int n_tiles;
};

// The sweep kernel of a launch over n_tiles tiles (of one image, or of a batch
// together) on num_sms SMs. The limits in tiles are those of the 152 SMs measured.
//  - FP32, up to 3/4 tile per SM (114): rows whose blocks all fit on the SMs at three a
//    piece get the registers of three (64x48 5.9 -> 5.5 us a sweep, 128x96 8.2 -> 6.9;
//    where they no longer fit, 160x120 went 8.6 -> 11.7);
//  - up to 2 tiles per SM (304), in FP64 half a tile (76: the rows then fit on the SMs
//    at once): rows (sweep_row). FP32 measured faster at 280 tiles, slower at 384; FP64
//    faster at 24 and 48, slower at 96;
//  - FP32, above 4 tiles per SM (608): tiles whose plane stores are marked to leave L2
//    first. Up to there, one wave of 4 blocks per SM, the two buffers (94 MB) are still
//    in L2 in the next sweep. Larger states do not stay anyway, and what is evicted is
//    then rather the output than the neighbours' planes still to be read: a sweep at
//    320x240 20.5 and 21.1 us without and with, 333x251 30.9 and 30.5, 512x384 58.7 and
//    57.4, 640x480 86.5 and 85.2, 2048x1536 821 and 796 (FP64 the same to 0.2 %).
enum SweepMode { SWEEP_TILES, SWEEP_STREAM, SWEEP_ROWS, SWEEP_ROWS_FEW };
template <typename T>
inline SweepMode sweep_mode(int n_tiles, int num_sms) {
    if (sizeof(T) == 8) return 2 * n_tiles <= num_sms ? SWEEP_ROWS : SWEEP_TILES;
    if (n_tiles * TILE_H <= 3 * num_sms) return SWEEP_ROWS_FEW;
    if (n_tiles <= 2 * num_sms) return SWEEP_ROWS;
    return n_tiles > 4 * num_sms ? SWEEP_STREAM : SWEEP_TILES;
}
template <typename T, SweepMode MODE>
constexpr int sweep_min_blocks() {
    return sizeof(T) == 8 ? 2 : (MODE == SWEEP_ROWS_FEW ? 3 : 4);
}

struct Work {
    int seq;
    int tile;
};

template <typename T>
__device__ __forceinline__ SweepArgs<T> seq_args(const SeqDesc<T>& d, int cur) {
    SweepArgs<T> a;
    a.g = d.g;
    a.f = d.f;
    a.in = d.state[cur];
    a.out = d.state[cur ^ 1];
    a.I_s = d.in_planes[0];
    a.I_t = d.in_planes[1];
    a.g_x = d.in_planes[2];
    a.g_y = d.in_planes[3];
    a.m_x = d.in_planes[4];
    a.m_y = d.in_planes[5];
    a.sc = d.sc;
    a.br = d.br;
    return a;
}

// Grid-wide barrier for a cooperative launch (all blocks resident). The wait is
// bounded: after `limit` polls (each followed by a short sleep) the block sets
// FLAG_TIMEOUT in *flags and gets false.
constexpr long long GRID_SYNC_DEFAULT_LIMIT = 1ll << 24;
struct GridSync {
    unsigned* count;
    unsigned* gen;
    unsigned* flags;
    long long limit;
};

__device__ __forceinline__ bool grid_sync(const GridSync& gs) {
    __shared__ int ok_sh;
    __syncthreads();
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        volatile unsigned* gen = gs.gen;
        const unsigned g0 = *gen;
        __threadfence();
        int ok = 1;
        if (atomicAdd(gs.count, 1u) + 1u == gridDim.x) {
            *gs.count = 0u;
            __threadfence();
            atomicAdd(gs.gen, 1u);
        } else {
            long long spins = 0;
            while (*gen == g0) {
                if (++spins > gs.limit) {
                    ok = 0;
                    atomicOr(gs.flags, FLAG_TIMEOUT);
                    break;
                }
                __nanosleep(64);
            }
        }
        __threadfence();
        ok_sh = ok;
    }
    __syncthreads();
    return ok_sh != 0;
}

// Synchronous sweeps over a list of (sequence, tile) work items; with ROWS each item
// is cut into its TILE_H rows, a block each. A pixel is computed by the same functions
// in the same order either way, and each kernel serves every schedule, so the
// results do not depend on how the work is launched:
//  - one sweep per launch, one block per tile or row (n_iters == 1);
//  - n_iters sweeps in one cooperative launch: blocks stride over the work list
//    and meet at a grid barrier between sweeps. A sweep's stores (generic proxy)
//    are then read by the next sweep's bulk copies (async proxy) on other SMs, so
//    every thread fences the two proxies after its tile, before the barrier
//    publishes the stores.
// work == nullptr stands for the tiles of sequence 0 in order. ROWS is a kernel of its
// own: with both paths in one, 256x256 took 19.3 us a sweep instead of 18.9 and
// 2048x1536 837 instead of 821.
template <typename T, SweepMode MODE>
__global__ void __launch_bounds__(SWEEP_THREADS, sweep_min_blocks<T, MODE>()) k_sweeps(const SeqDesc<T>* __restrict__ seqs,
                                                             const Work* __restrict__ work, int n_tiles,
                                                             int n_iters, int cur0, int flip0,
                                                             GridSync gs) {
    // msg[p * TILE_PX + tid]: a tile's 84 message Lambda planes, bulk-copied in at the
    // start of the tile (the old messages), overwritten in place by the damped new
    // ones; by rows, the four directions' messages of the row
    constexpr bool ROWS = MODE == SWEEP_ROWS || MODE == SWEEP_ROWS_FEW;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bar;
    if (!ROWS) {
        if (threadIdx.x == 0 && threadIdx.y == 0) mbar_init(&bar, 1);
        __syncthreads();
    }
    pdl_wait();
    T* msg = reinterpret_cast<T*>(smem_raw);
    unsigned parity = 0;
    const int n_work = ROWS ? n_tiles * TILE_H : n_tiles;
    for (int it = 0; it < n_iters; ++it) {
        const int cur = (cur0 + it) & 1;
        // every other sweep takes the work from its end: what the previous sweep wrote
        // last is what L2 still holds
        const bool flip = (flip0 + it) & 1;
        for (int k = blockIdx.x; k < n_work; k += gridDim.x) {
            const int w = flip ? n_work - 1 - k : k, item = ROWS ? w / TILE_H : w;
            const Work wk = work ? work[item] : Work{0, item};
            const SweepArgs<T> a = seq_args(seqs[wk.seq], cur);
            const int tx = wk.tile % a.g.tiles_x, ty = wk.tile / a.g.tiles_x;
            if (ROWS) {
                sweep_row(a, tx, ty, w % TILE_H, msg, it + 1 == n_iters);
            } else {
                // a tile whose bulk copy never arrived ends the block's work for the
                // launch: the mbarrier's phase no longer matches `parity`, and the copy
                // may still be writing `msg`
                if (!sweep_tile<MODE == SWEEP_STREAM>(a, tx, ty, msg, &bar, parity, it + 1 == n_iters)) return;
                parity ^= 1u;
                if (n_iters > 1) asm volatile("fence.proxy.async.global;" ::: "memory");
            }
            __syncthreads();
        }
        if (it + 1 < n_iters && !grid_sync(gs)) return;
    }
}

// pixel of a work item's tile handled by this thread (block = 32 x 4 threads)
template <typename T>
__device__ __forceinline__ bool work_pixel(const SeqDesc<T>& d, const Work& wk, int* u, int* v) {
    *u = (wk.tile % d.g.tiles_x) * TILE_W + threadIdx.x;
    *v = (wk.tile / d.g.tiles_x) * TILE_H + threadIdx.y;
    return *u < d.g.W && *v < d.g.H;
}

template <typename T>
__global__ void k_batch_ingest_target(const SeqDesc<T>* __restrict__ seqs, const Work* __restrict__ work) {
    const Work wk = work[blockIdx.x];
    const SeqDesc<T>& d = seqs[wk.seq];
    int u, v;
    if (work_pixel(d, wk, &u, &v)) ingest_target_px(d.g, d.frame, d.in_planes[1], d.in_planes[2], d.in_planes[3], u, v);
}

template <typename T>
__global__ void k_batch_keyframe(const SeqDesc<T>* __restrict__ seqs, const Work* __restrict__ work, int cur) {
    const Work wk = work[blockIdx.x];
    const SeqDesc<T>& d = seqs[wk.seq];
    int u, v;
    if (!work_pixel(d, wk, &u, &v)) return;
    ingest_keyframe_px(d.g, d.frame, d.normals, d.in_planes[0], d.in_planes[4], d.in_planes[5], u, v);
    reset_px(d.g, d.f, d.state[cur], d.sc, u, v);
}

template <typename T>
__global__ void __launch_bounds__(RED_THREADS) k_batch_reduce(const SeqDesc<T>* __restrict__ seqs,
                                                              const Work* __restrict__ work, int cur,
                                                              int anchor) {
    const Work wk = work[blockIdx.x];
    const SeqDesc<T>& d = seqs[wk.seq];
    const int per = reduce_group(d.n_tiles);
    if (wk.tile % per == 0) reduce_tiles(d.g, d.state[cur], d.partials, d.sc, anchor, wk.tile / per, d.n_tiles);
}

}  // namespace pv
