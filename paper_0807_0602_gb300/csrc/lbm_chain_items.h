// Work items of a chained launch (lbm_chain.cuh): their numbers, and how many
// steps one launch may take.  Plain C++ beside the kernel, so that it can be
// tested on any machine.
#pragma once

#ifdef __CUDACC__
#define LBM_HD_ITEMS __host__ __device__ inline
#else
#define LBM_HD_ITEMS inline
#endif

namespace sc {

// Items are numbered step * ntiles + i in 32-bit integers, and every CTA draws
// one number beyond the last item.
constexpr long long kChainItems = 1LL << 30;

// A launch keeps most of every SM's shared memory from other streams' work until
// it ends, so its length is bounded, too: 2^25 nodes times steps are 13 ms on a
// GB300 (2048 x 130: 126 steps; 30 000 nodes, where steps are longer than their
// nodes ask for: 1100 steps, some 22 ms).  Between launches the tiles drain,
// about a wave of them, below a hundredth of that.  Never less than 8 steps: on
// larger grids a single step takes milliseconds.
constexpr long long kChainNodeSteps = 1LL << 25, kChainMinSteps = 8;

// Steps of the next chained launch of n steps (n >= 1) over ntiles tiles of
// `nodes` nodes in all.
LBM_HD_ITEMS long long chain_launch_steps(long long n, long long ntiles, long long nodes) {
    const long long items = ntiles < kChainItems ? kChainItems / (ntiles > 0 ? ntiles : 1) : 1;
    const long long work = nodes > 0 ? kChainNodeSteps / nodes : n;
    long long most = work > kChainMinSteps ? work : kChainMinSteps;
    if (most > items) most = items;
    return n < most ? n : most;
}

// Tile of item `item` (-1 after the last step) and its step.  span(i, first,
// count): the tiles of tile i's run.  Every step runs through the run's list
// rotated by rot more tiles than the step before (rot < 2^10; with steps times
// count at most 2^30, step % count is at most 2^15, so the product fits).
template <typename Span>
LBM_HD_ITEMS int chain_item_tile(int item, int ntiles, int nsteps, int rot, Span span, int& step) {
    step = item / ntiles;
    if (step >= nsteps) return -1;
    const int i = item - step * ntiles;
    int first = 0, count = 1;
    span(i, first, count);
    const unsigned off = (unsigned)(step % count) * (unsigned)(rot < count ? rot : count) + (unsigned)(i - first);
    return first + (int)(off % (unsigned)count);
}

}  // namespace sc
