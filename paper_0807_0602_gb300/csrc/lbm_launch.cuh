// Launchers of the kernels in lbm_kernels.cuh; Launch<S> is instantiated per
// storage type by kernels_f64.cu, kernels_f32.cu and kernels_f16.cu, and
// Step<S, GEN> by those and by the kernels_gen_*.cu units (GEN = true).
#pragma once

#include <atomic>

#include "lbm_chain.cuh"
#include "lbm_kernels.cuh"
#include "lbm_ring.cuh"

namespace sc {

// Raises the dynamic shared-memory limit of kernel `fn` to `bytes` once per
// device (one bit per device in `done`); two threads racing on a first launch
// both set the same attribute, which is harmless.
static inline cudaError_t ensure_dynamic_smem(const void* fn, int bytes, std::atomic<unsigned long long>& done) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = dev < 64 ? (1ull << dev) : 0ull;
    if (bit && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess && bit) done.fetch_or(bit, std::memory_order_release);
    return e;
}

// Launches a step kernel so that its CTAs may start while the kernel before it
// on the stream ends (it waits itself, step_ready).
template <typename... P, typename... Q>
static cudaError_t launch_step_dyn(void (*fn)(P...), int grid, int threads, int smem, cudaStream_t s, Q... args) {
    cudaLaunchConfig_t cfg{};
    cfg.dynamicSmemBytes = smem;
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, P(args)...);
}

template <typename... P, typename... Q>
static cudaError_t launch_step(void (*fn)(P...), int grid, int threads, cudaStream_t s, Q... args) {
    return launch_step_dyn(fn, grid, threads, 0, s, args...);
}

static inline int clamp_grid(long long want, int cap) {
    if (want < 1) return 1;
    return want > cap ? cap : (int)want;
}

template <typename S>
cudaError_t Launch<S>::init(const RunDesc* d_runs, int nruns, int max_nodes, cudaStream_t s) {
    if (nruns <= 0) return cudaSuccess;
    dim3 grid(clamp_grid((max_nodes + 255) / 256, 2048), nruns);
    k_init<S><<<grid, 256, 0, s>>>(d_runs);
    return cudaGetLastError();
}

template <typename S, bool G>
cudaError_t Step<S, G>::step(int W, const RunDesc* d_runs, const Tile* d_tiles, int ntiles, int parity,
                            cudaStream_t s) {
    if (ntiles <= 0) return cudaSuccess;
    MomOut none{nullptr, nullptr, 0};
    switch (W) {
        case 64: k_step<S, 64, 0, false, G><<<ntiles, 64, 0, s>>>(d_runs, d_tiles, parity, none); break;
        case 128: k_step<S, 128, 0, false, G><<<ntiles, 128, 0, s>>>(d_runs, d_tiles, parity, none); break;
        case 256: k_step<S, 256, 0, false, G><<<ntiles, 256, 0, s>>>(d_runs, d_tiles, parity, none); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <typename S, int W, int D, bool G>
static cudaError_t launch_async(const RunDesc* d_runs, const Tile* d_tiles, int ntiles, int parity, cudaStream_t s) {
    constexpr size_t smem = async_smem_bytes<S, W, D>();
    static std::atomic<unsigned long long> configured{0};   // per instantiation, one bit per device
    const cudaError_t e = ensure_dynamic_smem((const void*)k_step_async<S, W, D, G>, (int)smem, configured);
    if (e != cudaSuccess) return e;
    k_step_async<S, W, D, G><<<ntiles, W, smem, s>>>(d_runs, d_tiles, parity);
    return cudaGetLastError();
}

template <typename S, bool G>
cudaError_t Step<S, G>::step_async(int W, int D, const RunDesc* d_runs, const Tile* d_tiles, int ntiles, int parity,
                                  cudaStream_t s) {
    if (ntiles <= 0) return cudaSuccess;
    if constexpr (sizeof(S) == 2) {
        return cudaErrorInvalidValue;   // cp.async moves 4 or 8 bytes: FP16 storage uses k_step
    } else {
        const int key = W * 10 + D;
        switch (key) {
            case 643: return launch_async<S, 64, 3, G>(d_runs, d_tiles, ntiles, parity, s);
            case 644: return launch_async<S, 64, 4, G>(d_runs, d_tiles, ntiles, parity, s);
            case 1283: return launch_async<S, 128, 3, G>(d_runs, d_tiles, ntiles, parity, s);
            case 1284: return launch_async<S, 128, 4, G>(d_runs, d_tiles, ntiles, parity, s);
            case 2563: return launch_async<S, 256, 3, G>(d_runs, d_tiles, ntiles, parity, s);
            case 2564: return launch_async<S, 256, 4, G>(d_runs, d_tiles, ntiles, parity, s);
            default: return cudaErrorInvalidValue;
        }
    }
}

template <typename S, int W, int D, bool G>
static cudaError_t launch_tma(const RunDesc* d_runs, const Tile* d_tiles, int ntiles, int parity, uint32_t* err,
                              cudaStream_t s) {
    constexpr size_t smem = TmaGeom<S, W, D>::smem_bytes();
    if constexpr (smem > kMaxSmemPerCta) {
        return cudaErrorInvalidValue;
    } else {
        static std::atomic<unsigned long long> configured{0};   // per instantiation, one bit per device
        const cudaError_t e = ensure_dynamic_smem((const void*)k_step_tma<S, W, D, G>, (int)smem, configured);
        if (e != cudaSuccess) return e;
        k_step_tma<S, W, D, G><<<ntiles, W, smem, s>>>(d_runs, d_tiles, parity, err);
        return cudaGetLastError();
    }
}

template <typename S, bool G>
cudaError_t Step<S, G>::step_tma(int W, int D, const RunDesc* d_runs, const Tile* d_tiles, int ntiles, int parity,
                                uint32_t* err, cudaStream_t s) {
    if (ntiles <= 0) return cudaSuccess;
    switch (W * 10 + D) {
        case 644: return launch_tma<S, 64, 4, G>(d_runs, d_tiles, ntiles, parity, err, s);
        case 646: return launch_tma<S, 64, 6, G>(d_runs, d_tiles, ntiles, parity, err, s);
        case 648: return launch_tma<S, 64, 8, G>(d_runs, d_tiles, ntiles, parity, err, s);
        case 1284: return launch_tma<S, 128, 4, G>(d_runs, d_tiles, ntiles, parity, err, s);
        case 1286: return launch_tma<S, 128, 6, G>(d_runs, d_tiles, ntiles, parity, err, s);
        case 1288: return launch_tma<S, 128, 8, G>(d_runs, d_tiles, ntiles, parity, err, s);
        case 2564: return launch_tma<S, 256, 4, G>(d_runs, d_tiles, ntiles, parity, err, s);
        case 2566: return launch_tma<S, 256, 6, G>(d_runs, d_tiles, ntiles, parity, err, s);
        default: return cudaErrorInvalidValue;
    }
}

template <typename S, bool G>
cudaError_t Step<S, G>::step_pf(int W, const RunDesc* d_runs, const Tile* d_tiles, int ntiles, int parity,
                               cudaStream_t s) {
    if (ntiles <= 0) return cudaSuccess;
    switch (W) {
        case 64: k_step_pf<S, 64, G><<<ntiles, 64, 0, s>>>(d_runs, d_tiles, parity); break;
        case 128:
            if constexpr (sizeof(typename Prec<S>::C) == 8) return cudaErrorInvalidValue;
            else k_step_pf<S, 128, G><<<ntiles, 128, 0, s>>>(d_runs, d_tiles, parity);
            break;

        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <typename S, bool G>
cudaError_t Step<S, G>::step_split(int W, const RunDesc* d_runs, const Tile* d_tiles, int ntiles, int parity,
                                  cudaStream_t s) {
    if (ntiles <= 0) return cudaSuccess;
    switch (W) {
        case 64: k_step_split<S, 64, G><<<ntiles, 128, 0, s>>>(d_runs, d_tiles, parity); break;
        case 128: k_step_split<S, 128, G><<<ntiles, 256, 0, s>>>(d_runs, d_tiles, parity); break;
        case 256: k_step_split<S, 256, G><<<ntiles, 512, 0, s>>>(d_runs, d_tiles, parity); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <typename S, bool G>
cudaError_t Step<S, G>::step_l2pf(int W, const RunDesc* d_runs, const Tile* d_tiles, int ntiles, int parity,
                                 cudaStream_t s) {
    if (ntiles <= 0) return cudaSuccess;
    MomOut none{nullptr, nullptr, 0};
    switch (W) {
        case 64: k_step<S, 64, 0, true, G><<<ntiles, 64, 0, s>>>(d_runs, d_tiles, parity, none); break;
        case 128: k_step<S, 128, 0, true, G><<<ntiles, 128, 0, s>>>(d_runs, d_tiles, parity, none); break;
        case 256: k_step<S, 256, 0, true, G><<<ntiles, 256, 0, s>>>(d_runs, d_tiles, parity, none); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <typename S, bool G>
cudaError_t Step<S, G>::step_smem(int W, const RunDesc* d_runs, const Tile* d_tiles, int ntiles, int parity,
                                 cudaStream_t s) {
    if (ntiles <= 0) return cudaSuccess;
    switch (W) {
        case 64: k_step_smem<S, 64, G><<<ntiles, 64, 0, s>>>(d_runs, d_tiles, parity); break;
        case 128: k_step_smem<S, 128, G><<<ntiles, 128, 0, s>>>(d_runs, d_tiles, parity); break;
        case 256:
            if constexpr (sizeof(typename Prec<S>::C) == 8) return cudaErrorInvalidValue;
            else k_step_smem<S, 256, G><<<ntiles, 256, 0, s>>>(d_runs, d_tiles, parity);
            break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <typename S, bool G>
cudaError_t Step<S, G>::step_pair(int W, const RunDesc* d_runs, const Tile* d_tiles, int ntiles, int parity,
                                 cudaStream_t s) {
    if (ntiles <= 0) return cudaSuccess;
    switch (W) {
        case 64: k_step_pair<S, 64, G><<<ntiles, 64, 0, s>>>(d_runs, d_tiles, parity); break;
        case 128:
            if constexpr (sizeof(typename Prec<S>::C) == 8) return cudaErrorInvalidValue;
            else k_step_pair<S, 128, G><<<ntiles, 128, 0, s>>>(d_runs, d_tiles, parity);
            break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <typename S, bool G>
cudaError_t Step<S, G>::step_tile(int W, int R, const RunDesc* d_runs, const Tile* d_tiles, int ntiles, int parity,
                                 cudaStream_t s) {
    if (ntiles <= 0) return cudaSuccess;
    // R = collided rows per tile: TY = R + 2 thread rows
    switch (W * 100 + R) {
        case 3206: return launch_step(k_step_tile<S, 32, 8, G>, ntiles, 256, s, d_runs, d_tiles, parity);
        case 3214: return launch_step(k_step_tile<S, 32, 16, G>, ntiles, 512, s, d_runs, d_tiles, parity);
        case 3230: return launch_step(k_step_tile<S, 32, 32, G>, ntiles, 1024, s, d_runs, d_tiles, parity);
        case 6406: return launch_step(k_step_tile<S, 64, 8, G>, ntiles, 512, s, d_runs, d_tiles, parity);
        case 6414: return launch_step(k_step_tile<S, 64, 16, G>, ntiles, 1024, s, d_runs, d_tiles, parity);
        default: return cudaErrorInvalidValue;
    }
}

// Raises the shared memory limit of the FP64 marches (47 KB static and the products).
template <typename S, bool G>
static cudaError_t bidir_smem() {
    if constexpr (kBidirDynSmem<S, 64> == 0) {
        return cudaSuccess;
    } else {
        static std::atomic<unsigned long long> step{0}, chain{0};
        const cudaError_t e = ensure_dynamic_smem((const void*)k_step_bidir<S, 64, G>, kBidirDynSmem<S, 64>, step);
        if (e != cudaSuccess) return e;
        return ensure_dynamic_smem((const void*)k_chain_bidir<S, 64, G>, kBidirDynSmem<S, 64>, chain);
    }
}

template <typename S, bool G>
cudaError_t Step<S, G>::step_bidir(int W, const RunDesc* d_runs, const Tile* d_tiles, int ntiles, int parity,
                                  const Shape& shape, cudaStream_t s) {
    if (ntiles <= 0) return cudaSuccess;
    if constexpr (sizeof(typename Prec<S>::C) == 4) {
        if (shape.nx > 0 && W == 64)
            return launch_step(k_step_bidir_alike<S, 64, G>, ntiles, 128, s, d_runs, d_tiles, parity, shape);
        if (shape.nx > 0 && W == 128)
            return launch_step(k_step_bidir_alike<S, 128, G>, ntiles, 256, s, d_runs, d_tiles, parity, shape);
    }
    switch (W) {
        case 64: {
            const cudaError_t e = bidir_smem<S, G>();
            if (e != cudaSuccess) return e;
            return launch_step_dyn(k_step_bidir<S, 64, G>, ntiles, 128, kBidirDynSmem<S, 64>, s, d_runs, d_tiles, parity);
        }
        case 128:
            if constexpr (sizeof(typename Prec<S>::C) == 8) return cudaErrorInvalidValue;
            else return launch_step(k_step_bidir<S, 128, G>, ntiles, 256, s, d_runs, d_tiles, parity);
        default: return cudaErrorInvalidValue;
    }
}

template <typename S, int D, bool G>
static cudaError_t ring_fn(const void** fn, int* smem, int* threads) {
    if constexpr (sizeof(S) == 8) {
        return cudaErrorInvalidValue;   // FP64 is arithmetic-bound: it keeps the register kernels
    } else {
        using RG = RingGeom<S, D>;
        constexpr size_t bytes = RG::smem_bytes();
        static_assert(bytes <= kMaxSmemPerCta, "ring slots exceed the shared memory of a CTA");
        static std::atomic<unsigned long long> configured{0};   // per instantiation, one bit per device
        const cudaError_t e = ensure_dynamic_smem((const void*)k_step_ring<S, D, G>, (int)bytes, configured);
        if (e != cudaSuccess) return e;
        *fn = (const void*)k_step_ring<S, D, G>;
        *smem = (int)bytes;
        *threads = RG::THREADS;
        return cudaSuccess;
    }
}

template <typename S, bool G>
static cudaError_t ring_lookup(int D, const void** fn, int* smem, int* threads) {
    switch (D) {
        case 3: return ring_fn<S, 3, G>(fn, smem, threads);
        case 4: return ring_fn<S, 4, G>(fn, smem, threads);
        case 5: return ring_fn<S, 5, G>(fn, smem, threads);
        default: return cudaErrorInvalidValue;
    }
}

template <typename S, bool G>
cudaError_t Step<S, G>::ring_ctas_per_sm(int D, int* out) {
    *out = 0;
    const void* fn = nullptr;
    int smem = 0, threads = 0;
    cudaError_t e = ring_lookup<S, G>(D, &fn, &smem, &threads);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, fn, threads, (size_t)smem);
}

template <typename S, bool G>
cudaError_t Step<S, G>::bidir_ctas_per_sm(int W, int* out) {
    *out = 0;
    switch (W) {
        case 64: {
            const cudaError_t e = bidir_smem<S, G>();
            if (e != cudaSuccess) return e;
            return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k_step_bidir<S, 64, G>, 128, kBidirDynSmem<S, 64>);
        }
        case 128:
            if constexpr (sizeof(typename Prec<S>::C) == 8) return cudaErrorInvalidValue;
            else return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k_step_bidir<S, 128, G>, 256, 0);
        default: return cudaErrorInvalidValue;
    }
}

template <typename S, bool G>
cudaError_t Step<S, G>::two_steps(const RunDesc* d_runs, const Tile* d_tiles, int ntiles, int parity, cudaStream_t s) {
    if constexpr (sizeof(S) == 8) {
        return cudaErrorInvalidValue;   // FP64 is bound by its pipe: no redundant work
    } else {
        if (ntiles <= 0) return cudaSuccess;
        return launch_step(k_two_steps<S, G>, ntiles, 512, s, d_runs, d_tiles, parity);
    }
}

template <typename S, bool G>
cudaError_t Step<S, G>::chain(const RunDesc* d_runs, const ChainTiles& ct, int nsteps, int parity, int rot, int grid,
                              uint32_t* err, cudaStream_t s) {
    if constexpr (sizeof(S) != 8) {
        return cudaErrorInvalidValue;   // FP64 only (lbm_chain.cuh)
    } else {
        if (ct.ntiles <= 0 || nsteps <= 0 || grid <= 0) return cudaSuccess;
        const cudaError_t e = bidir_smem<S, G>();
        if (e != cudaSuccess) return e;
        k_chain_bidir<S, 64, G><<<grid, 128, kBidirDynSmem<S, 64>, s>>>(d_runs, ct, nsteps, parity, rot, err);
        return cudaGetLastError();
    }
}

template <typename S, bool G>
cudaError_t Step<S, G>::chain_ctas_per_sm(int* out) {
    *out = 0;
    if constexpr (sizeof(S) != 8) {
        return cudaErrorInvalidValue;
    } else {
        const cudaError_t e = bidir_smem<S, G>();
        if (e != cudaSuccess) return e;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k_chain_bidir<S, 64, G>, 128, kBidirDynSmem<S, 64>);
    }
}

template <typename S, bool G>
cudaError_t Step<S, G>::step_ring(int D, const RunDesc* d_runs, const Tile* d_tiles, int ntiles, int* queue,
                                  int grid, int parity, uint32_t* err, cudaStream_t s) {
    if (grid <= 0 || ntiles <= 0) return cudaSuccess;
    const void* fn = nullptr;
    int smem = 0, threads = 0;
    cudaError_t e = ring_lookup<S, G>(D, &fn, &smem, &threads);
    if (e != cudaSuccess) return e;
    void* args[] = {(void*)&d_runs, (void*)&d_tiles, (void*)&ntiles, (void*)&queue, (void*)&parity, (void*)&err};
    return cudaLaunchKernel(fn, dim3(grid), dim3(threads), args, (size_t)smem, s);
}

template <typename S, bool G>
cudaError_t Step<S, G>::moments(int W, const RunDesc* d_runs, const Tile* d_tiles, int ntiles, int parity,
                               MomOut out, cudaStream_t s) {
    if (ntiles <= 0) return cudaSuccess;
    switch (W) {
        case 32: k_step<S, 32, 1, false, G><<<ntiles, 32, 0, s>>>(d_runs, d_tiles, parity, out); break;
        case 64: k_step<S, 64, 1, false, G><<<ntiles, 64, 0, s>>>(d_runs, d_tiles, parity, out); break;
        case 128: k_step<S, 128, 1, false, G><<<ntiles, 128, 0, s>>>(d_runs, d_tiles, parity, out); break;
        case 256: k_step<S, 256, 1, false, G><<<ntiles, 256, 0, s>>>(d_runs, d_tiles, parity, out); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <typename S>
cudaError_t Launch<S>::densities(const RunDesc* d_runs, int run, int parity, int nx, int ny, double* nA, double* nB,
                                 cudaStream_t s) {
    const int threads = nx <= 128 ? 128 : 256;
    k_densities<S><<<dim3((nx + threads - 1) / threads, ny < 65535 ? ny : 65535), threads, 0, s>>>(d_runs, run, parity,
                                                                                                 nA, nB);
    return cudaGetLastError();
}

// CTAs of a front scan over the longest capillary
static inline int track_chunks(int max_cap) { return (max_cap + kTrackCols - 1) / kTrackCols; }

template <typename S>
cudaError_t Launch<S>::track(const RunDesc* d_runs, int nruns, int max_cap, int parity, int* first, double* zout,
                             cudaStream_t s) {
    if (nruns <= 0) return cudaSuccess;
    if (max_cap > 0) {
        k_track_scan<S><<<dim3(track_chunks(max_cap), nruns), kTrackThreads, 0, s>>>(d_runs, parity, first);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return launch_step(k_track_final<S>, nruns, 32, s, d_runs, parity, first, zout);
}

template <typename S>
cudaError_t Launch<S>::mass(const RunDesc* d_runs, int nruns, const int2* d_rows, int nrows, int parity,
                            double* d_partials, double* d_mass, uint32_t* d_err, cudaStream_t s) {
    if (nruns <= 0) return cudaSuccess;
    k_mass_rows<S><<<dim3(nrows, kMassChunks), kMassThreads, 0, s>>>(d_runs, d_rows, parity, d_partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_mass_final<<<nruns, kMassThreads, 0, s>>>(d_runs, d_partials, d_mass, d_err);
    return cudaGetLastError();
}

template <typename S>
cudaError_t Launch<S>::log(const RunDesc* d_runs, int nruns, const int2* d_rows, int nrows, int max_cap, int parity,
                           double* d_partials, int* first, LogCtl lc, uint32_t* d_err, cudaStream_t s) {
    if (nruns <= 0) return cudaSuccess;
    const int chunks = max_cap > 0 ? track_chunks(max_cap) : 0;
    const long long grid = (long long)nrows * kMassChunks + (long long)chunks * nruns;
    if (grid > 0x7fffffffLL) return cudaErrorInvalidValue;
    cudaError_t e = launch_step(k_log_rows<S>, (int)grid, kMassThreads, s, d_runs, d_rows, nrows, chunks, parity,
                                d_partials, first);
    if (e != cudaSuccess) return e;
    return launch_step(k_log_final<S>, nruns, kMassThreads, s, d_runs, parity, d_partials, first, lc, d_err);
}

template <typename S>
cudaError_t Launch<S>::export_pops(const RunDesc* d_runs, int run, int parity, int nx, int ny, void* out,
                                   cudaStream_t s) {
    const long long total = 18LL * nx * ny;
    k_export<S><<<clamp_grid((total + 255) / 256, 8192), 256, 0, s>>>(d_runs, run, parity, static_cast<S*>(out));
    return cudaGetLastError();
}

template <typename S>
cudaError_t Launch<S>::import_pops(const RunDesc* d_runs, int run, int parity, int nx, int ny, const void* in,
                                   cudaStream_t s) {
    const long long total = 18LL * nx * ny;
    k_import<S><<<clamp_grid((total + 255) / 256, 8192), 256, 0, s>>>(d_runs, run, parity,
                                                                      static_cast<const S*>(in));
    return cudaGetLastError();
}

// Thread block of a column copy: as many threads along a row as it has
// accesses (at most 256), the rest of 256 threads along the rows.
static inline dim3 cols_block(int accesses) {
    int tx = 1;
    while (tx < accesses && tx < 256) tx *= 2;
    return dim3(tx, 256 / tx);
}

template <typename S>
cudaError_t Launch<S>::get_cols(const RunDesc* d_runs, int run, int parity, int ny, int x0, int ncols, void* out,
                                cudaStream_t s) {
    // 16-byte accesses where every row of the window and of the buffer starts
    // on one (rows of the populations start LBM_COL0 elements into a row of a
    // multiple of 64)
    constexpr int V = 16 / (int)sizeof(S);
    S* o = static_cast<S*>(out);
    const bool wide = x0 % V == 0 && ncols % V == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0;
    const dim3 block = cols_block(wide ? ncols / V : ncols);
    const int grid = clamp_grid((18LL * ny + block.y - 1) / block.y, 8192);
    if (wide) k_get_cols<S, V><<<grid, block, 0, s>>>(d_runs, run, parity, x0, ncols, o);
    else k_get_cols<S, 1><<<grid, block, 0, s>>>(d_runs, run, parity, x0, ncols, o);
    return cudaGetLastError();
}

template <typename S>
cudaError_t Launch<S>::slab_halos(const SlabHalos& h, int ny, cudaStream_t s) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((36 * ny + 127) / 128, 2 * h.n);
    cfg.blockDim = dim3(128);
    cfg.stream = s;
    cudaLaunchAttribute at{};   // as launch_step
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_slab_halos<S>, h);
}

template <typename S>
cudaError_t Launch<S>::set_cols(const RunDesc* d_runs, int run, int parity, int ny, int x0, int ncols,
                                const void* in, cudaStream_t s) {
    const dim3 block = cols_block(ncols);
    k_set_cols<S><<<clamp_grid((18LL * ny + block.y - 1) / block.y, 8192), block, 0, s>>>(
        d_runs, run, parity, x0, ncols, static_cast<const S*>(in));
    return cudaGetLastError();
}

}  // namespace sc
