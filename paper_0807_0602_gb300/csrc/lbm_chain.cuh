// Chained steps (LBM_KERNEL_CHAIN, FP64): many time steps in one launch.  The
// work items are (step, tile) pairs in step order; the CTAs draw them one by one
// from a counter.  An item waits only for the tiles of the step before whose
// nodes it reads or overwrites (its own tile and its neighbours, at most 32:
// `deps`), so no step waits for the slowest tile of the whole grid, and neither
// launches nor empty SMs separate the steps.
//
// Why it cannot deadlock: an item depends on items with lower numbers only,
// and a CTA works its items off in ascending order (it draws the next one
// while it waits for the current one's neighbours), so the lowest unfinished
// item can always proceed, however many of the CTAs are resident.  Every wait
// is bounded all the same: a CTA that gives up sets the error bit and the
// abort word, which ends the others' waits, and the launch returns.
//
// Order of the items: every step starts `rot` tiles further on in each run's
// list than the step before (the list runs down the columns of tiles), so that
// with periodic sides too almost a whole step lies between an item and the
// items it waits for.
//
// Where it pays: the FP64 step is bound by the FP64 pipe, so a tile is long (some
// 20 us for 4 rows) and a grid of a few hundred thousand nodes is one or two
// waves of them; launched step by step, most SMs idle in the last wave.  GB300,
// us per step, single steps (best tiling) / chained: 2048 x 130 124 / 103,
// nine 128 x 80 droplets 72 / 54, 256 x 32 20.5 / 26 (too few tiles: the flags'
// round trips through L2 cost more than launches).  FP32 and FP16S keep single
// steps: an acquire drops the SM's L1 lines, which their shifted loads live on
// (64 uneven capillaries FP32: 506 single, 553 chained; 8192 x 160: 37.4, 37.7).
//
// Memory: an item's stores are released at GPU scope when its flag is set
// (thread 0, after the CTA's barrier) and acquired by the threads that poll
// the flags; the populations are read by plain loads, not through the
// read-only path, because other SMs write them within the launch.
#pragma once

#include "lbm_chain_items.h"
#include "lbm_kernels.cuh"

namespace sc {

__device__ __forceinline__ int ld_acquire(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(int* p, int v) {
    asm volatile("st.release.gpu.global.s32 [%0], %1;\n" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_relaxed(const int* p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ int chain_item(const ChainTiles& ct, int item, int nsteps, int rot, int& step) {
    return chain_item_tile(
        item, ct.ntiles, nsteps, rot,
        [&](int i, int& first, int& count) {
            const int2 sp = __ldg(&ct.span[i]);
            first = sp.x;
            count = sp.y;
        },
        step);
}

// tile_fn(tile, parity, ready): advances one tile; calls ready() from every
// thread before it reads any population.  limit: SM cycles after which a wait
// gives up.
template <int THREADS, typename TileFn>
__device__ __forceinline__ void chain_run(const ChainTiles& ct, int nsteps, int parity0, int rot, uint32_t* err,
                                          TileFn tile_fn, long long limit = kWaitCycles) {
    // s_stop: a wait of this item gave up.  Items alternate between its two
    // words, so that no wait writes the word that the threads are still reading:
    // all of them leave the loop at the same item, or none (tile_fn and ready
    // hold barriers of the whole CTA).
    __shared__ int s_tile, s_step, s_stop[2], s_last;
    const int t = threadIdx.x;
    if (t == 0) {
        int st = 0;
        s_tile = chain_item(ct, atomicAdd(&ct.ctl->next, 1), nsteps, rot, st);
        s_step = st;
        s_stop[0] = s_stop[1] = 0;
    }
    __syncthreads();
    bool stop = false;
    for (int word = 0;; word ^= 1) {
        const int tile = s_tile, step = s_step;
        if (tile < 0 || stop) break;
        int ntile = -1, nstep = 0;
        tile_fn(tile, (parity0 + step) & 1, [&] {
            if (t < 32) {
                const int d = step > 0 ? __ldg(&ct.deps[tile * kChainDeps + t]) : -1;
                if (d >= 0 && ld_acquire(&ct.flags[d]) < step) {
                    const long long start = clock64();
                    while (ld_acquire(&ct.flags[d]) < step) {
                        if (clock64() - start > limit || ld_relaxed(&ct.ctl->abort)) {
                            atomicOr(err, ERR_TIMEOUT);
                            atomicExch(&ct.ctl->abort, 1);
                            s_stop[word] = 1;
                            break;
                        }
                    }
                }
            } else if (t == 32) {   // meanwhile: this CTA's next item
                ntile = chain_item(ct, atomicAdd(&ct.ctl->next, 1), nsteps, rot, nstep);
            }
            __syncthreads();
            // (every thread has read s_tile and s_step)
            if (t == 32) {
                s_tile = ntile;
                s_step = nstep;
            }
        });
        __syncthreads();
        stop = s_stop[word] != 0;   // (written again two items on at the earliest)
        if (t == 0 && !stop) st_release(&ct.flags[tile], step + 1);
    }
    // the last CTA leaves the control words and flags zero for the next launch
    if (t == 0) {
        __threadfence();
        s_last = atomicAdd(&ct.ctl->done, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (s_last) {
        __threadfence();
        for (int i = t; i < ct.ntiles; i += THREADS) ct.flags[i] = 0;
        if (t == 0) *ct.ctl = ChainCtl{0, 0, 0, 0};
    }
}

template <typename S, int W, bool G>
__global__ void __launch_bounds__(2 * W, (kBidirMinBlocks<S, W>)) k_chain_bidir(const RunDesc* __restrict__ runs,
                                                                               ChainTiles ct, int nsteps, int parity,
                                                                               int rot, uint32_t* err) {
    chain_run<2 * W>(ct, nsteps, parity, rot, err, [&](int tile, int par, auto ready) {
        bidir_tile<S, W, G, false>(runs, ct.tiles, tile, par, Shape{}, ready);
    });
}

}  // namespace sc
