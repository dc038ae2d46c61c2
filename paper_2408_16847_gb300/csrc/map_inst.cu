// Per-M instantiation of the map kernels.  The build compiles this file once for
// every multipole limit TPCF_M = 0..TPCF_MAX_M and links the objects together.
#include "cat_kernels.cuh"

#ifndef TPCF_M
#error "compile with -DTPCF_M=<m_max>"
#endif

#define TPCF_CAT2(a, b) a##b
#define TPCF_CAT(a, b) TPCF_CAT2(a, b)

namespace tpcf {

// Kernels that keep their tile in shared memory ask for the largest carveout: they are sized to
// fit 2-3 CTAs per SM only with it (the occupancy queries below assume it as well).  The
// block kernels (BT threads, four CTAs per SM) ask for what they use and leave the rest to L1,
// which serves their pixel loads.
template <class Kern>
static cudaError_t prefer_shared(Kern* k, size_t smem, int threads = NTHREADS) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int carve = (int)cudaSharedmemCarveoutMaxShared;
    if (threads == BT) carve = (int)((4 * (smem + 2048) * 100 + 233471) / 233472);
    return cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, carve > 100 ? 100 : carve);
}

// Launch the pair kernel `k` with `smem` bytes of dynamic shared memory.
template <class Kern>
static cudaError_t launch(Kern* k, size_t smem, int grid, const MapDev& g, const MapCall& c, cudaStream_t s,
                          int threads = NTHREADS) {
    cudaError_t e = prefer_shared(k, smem, threads);
    if (e != cudaSuccess) return e;
    k<<<grid, threads, smem, s>>>(g, c);
    return cudaGetLastError();
}

template <class Kern>
static int occupancy(Kern* k, size_t smem, int threads = NTHREADS) {
    int nb = 0;
    if (prefer_shared(k, smem, threads) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, threads, smem) != cudaSuccess) return 0;
    return nb;
}

// The forward pair kernel.
cudaError_t TPCF_CAT(map_fwd_launch_m, TPCF_M)(const MapDev& g, const MapCall& c, int grid, cudaStream_t s) {
    const size_t smem = block_smem_bytes(TPCF_M);
    if (c.group > 1)  // shared neighbour lists (self pairs kept)
        return launch(map_fwd_kernel<TPCF_M, false, true>, smem, grid, g, c, s, BT);
    return c.self_subtract ? launch(map_fwd_kernel<TPCF_M, true>, smem, grid, g, c, s, BT)
                           : launch(map_fwd_kernel<TPCF_M, false>, smem, grid, g, c, s, BT);
}

cudaError_t TPCF_CAT(map_bwd_launch_m, TPCF_M)(const MapDev& g, const MapCall& c, int grid, cudaStream_t s) {
    const size_t smem = adj_smem_bytes(TPCF_M);
    return c.self_subtract ? launch(map_bwd_kernel<TPCF_M, true>, smem, grid, g, c, s, BT)
                           : launch(map_bwd_kernel<TPCF_M, false>, smem, grid, g, c, s, BT);
}

// Resident CTAs per SM of the forward (either self-pair mode).
int TPCF_CAT(map_fwd_occupancy_m, TPCF_M)() {
    const int a = occupancy(map_fwd_kernel<TPCF_M, false>, block_smem_bytes(TPCF_M), BT);
    const int b = occupancy(map_fwd_kernel<TPCF_M, true>, block_smem_bytes(TPCF_M), BT);
    return a < b ? a : b;
}

// Resident CTAs per SM of the adjoint (either self-pair mode).
int TPCF_CAT(map_bwd_occupancy_m, TPCF_M)() {
    const int a = occupancy(map_bwd_kernel<TPCF_M, false>, adj_smem_bytes(TPCF_M), BT);
    const int b = occupancy(map_bwd_kernel<TPCF_M, true>, adj_smem_bytes(TPCF_M), BT);
    return a < b ? a : b;
}

// Forward with the split-precision tensor-core contraction.
cudaError_t TPCF_CAT(map_fwd_tc_launch_m, TPCF_M)(const MapDev& g, const MapCall& c, int grid, cudaStream_t s) {
    const size_t smem = tc_smem_bytes(g.K, TPCF_M, c.self_subtract != 0);
    if (c.self_subtract) {
        auto* k = map_fwd_tc_kernel<TPCF_M, true>;
        cudaError_t e = prefer_shared(k, smem);
        if (e != cudaSuccess) return e;
        k<<<grid, BT, smem, s>>>(g, c);
    } else {
        auto* k = map_fwd_tc_kernel<TPCF_M, false>;
        cudaError_t e = prefer_shared(k, smem);
        if (e != cudaSuccess) return e;
        k<<<grid, BT, smem, s>>>(g, c);
    }
    return cudaGetLastError();
}

// Resident CTAs per SM from the SM's register file and shared memory.  Used for the
// tensor-core kernel, for which cudaOccupancyMaxActiveBlocksPerMultiprocessor answers 1
// although 3 CTAs fit by registers and shared memory (and the profiler's occupancy
// limits agree); the CTAs are persistent and never wait on each other, so a grid
// larger than what is resident is still correct.
template <class Kern>
static int occupancy_by_resources(Kern* k, size_t smem, int threads) {
    if (prefer_shared(k, smem) != cudaSuccess) return 0;
    cudaFuncAttributes a;
    int dev = 0, smem_sm = 0, reserved = 0, regs_sm = 0;
    if (cudaFuncGetAttributes(&a, k) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev) != cudaSuccess)
        return 0;
    const size_t per_cta_smem = smem + a.sharedSizeBytes + (size_t)reserved;
    const int warps = threads / 32;
    const int regs_warp = (a.numRegs * 32 + 255) / 256 * 256;  // allocated per warp in units of 256
    const int by_smem = (int)((size_t)smem_sm / per_cta_smem);
    const int by_regs = regs_warp > 0 ? regs_sm / (regs_warp * warps) : 0;
    return by_smem < by_regs ? by_smem : by_regs;
}

int TPCF_CAT(map_fwd_tc_occupancy_m, TPCF_M)(int K, int self_subtract) {
    const size_t smem = tc_smem_bytes(K, TPCF_M, self_subtract != 0);
    const int nb = self_subtract ? occupancy_by_resources(map_fwd_tc_kernel<TPCF_M, true>, smem, BT)
                                 : occupancy_by_resources(map_fwd_tc_kernel<TPCF_M, false>, smem, BT);
    // at most 512 / TC_TMEM_COLS accumulators per SM; more resident CTAs would wait in tcgen05.alloc
    return nb < 512 / TC_TMEM_COLS ? nb : 512 / TC_TMEM_COLS;
}

// The tile kernels (map_tile.cuh): launch, and resident CTAs per SM; variant 3 or 2 = CTAs per SM
// that the registers are sized for.
template <int OCC>
static cudaError_t tile_launch(const MapDev& g, const MapCall& c, int what, int grid, cudaStream_t s) {
    const bool self = c.self_subtract != 0;
    if (what == TILE_BWD) {
        const size_t smem = bwd_tile_floats_rt(g.K, TPCF_M) * sizeof(float);
        return self ? launch(map_tile_bwd_kernel<TPCF_M, true, OCC>, smem, grid, g, c, s)
                    : launch(map_tile_bwd_kernel<TPCF_M, false, OCC>, smem, grid, g, c, s);
    }
    const size_t smem = tile_floats_rt(g.K, TPCF_M) * sizeof(float);
    return self ? launch(map_tile_fwd_kernel<TPCF_M, true, false, OCC>, smem, grid, g, c, s)
                : launch(map_tile_fwd_kernel<TPCF_M, false, false, OCC>, smem, grid, g, c, s);
}

template <int OCC>
static int tile_occupancy(int what, int K, bool self) {
    if (what == TILE_BWD) {
        const size_t smem = bwd_tile_floats_rt(K, TPCF_M) * sizeof(float);
        return self ? occupancy(map_tile_bwd_kernel<TPCF_M, true, OCC>, smem)
                    : occupancy(map_tile_bwd_kernel<TPCF_M, false, OCC>, smem);
    }
    const size_t smem = tile_floats_rt(K, TPCF_M) * sizeof(float);
    return self ? occupancy(map_tile_fwd_kernel<TPCF_M, true, false, OCC>, smem)
                : occupancy(map_tile_fwd_kernel<TPCF_M, false, false, OCC>, smem);
}

cudaError_t TPCF_CAT(map_tile_launch_m, TPCF_M)(const MapDev& g, const MapCall& c, int what, int variant, int grid,
                                                cudaStream_t s) {
    const bool self = c.self_subtract != 0;
    const size_t smem = tile_floats_rt(g.K, TPCF_M) * sizeof(float);
    if (what == TILE_TC) {
        const size_t tcs = tc_tile_bytes(g.K, TPCF_M, self);
        return self ? launch(map_tile_tc_kernel<TPCF_M, true>, tcs, grid, g, c, s)
                    : launch(map_tile_tc_kernel<TPCF_M, false>, tcs, grid, g, c, s);
    }
    if (what == TILE_GROUPED)  // (self pairs kept)
        return launch(map_tile_fwd_kernel<TPCF_M, false, false, 3, true>, smem, grid, g, c, s);
    if (what == TILE_DIRECT)  // the caller's delta and w, no packed copy
        return launch(map_tile_fwd_kernel<TPCF_M, false, true>, smem, grid, g, c, s);
    return variant == 2 ? tile_launch<2>(g, c, what, grid, s) : tile_launch<3>(g, c, what, grid, s);
}

int TPCF_CAT(map_tile_occupancy_m, TPCF_M)(int what, int variant, int K, int self) {
    if (what == TILE_TC) {
        const size_t smem = tc_tile_bytes(K, TPCF_M, self != 0);
        const int nb = self ? occupancy_by_resources(map_tile_tc_kernel<TPCF_M, true>, smem, NTHREADS)
                            : occupancy_by_resources(map_tile_tc_kernel<TPCF_M, false>, smem, NTHREADS);
        return nb < 512 / TC_TMEM_COLS ? nb : 512 / TC_TMEM_COLS;
    }
    return variant == 2 ? tile_occupancy<2>(what, K, self != 0) : tile_occupancy<3>(what, K, self != 0);
}

cudaError_t TPCF_CAT(map_tile_multi_launch_m, TPCF_M)(const MapDev& g, const MapCall& c, const float2* wdwB,
                                                      const float2* wdwC, int grid, cudaStream_t s) {
    const size_t smem = multi_tile_floats(g.K, TPCF_M) * sizeof(float);
    auto* k = map_tile_multi_kernel<TPCF_M>;
    cudaError_t e = prefer_shared(k, smem);
    if (e != cudaSuccess) return e;
    k<<<grid, NTHREADS, smem, s>>>(g, c, wdwB, wdwC);
    return cudaGetLastError();
}

int TPCF_CAT(map_tile_multi_occupancy_m, TPCF_M)(int K) {
    return occupancy(map_tile_multi_kernel<TPCF_M>, multi_tile_floats(K, TPCF_M) * sizeof(float));
}

// Multi-field forward (three fields on the same pixels).
cudaError_t TPCF_CAT(map_fwd_multi_launch_m, TPCF_M)(const MapDev& g, const MapCall& c, const float2* wdwB,
                                                     const float2* wdwC, int grid, cudaStream_t s) {
    const size_t smem = block_smem_bytes(TPCF_M);
    auto* k = map_fwd_multi_kernel<TPCF_M>;
    cudaError_t e = prefer_shared(k, smem, BT);
    if (e != cudaSuccess) return e;
    k<<<grid, BT, smem, s>>>(g, c, wdwB, wdwC);
    return cudaGetLastError();
}

int TPCF_CAT(map_fwd_multi_occupancy_m, TPCF_M)() {
    return occupancy(map_fwd_multi_kernel<TPCF_M>, block_smem_bytes(TPCF_M), BT);
}

// Multi-field forward on a catalogue.
cudaError_t TPCF_CAT(cat_fwd_multi_launch_m, TPCF_M)(const CatDev& g, const MapCall& c, const float2* wdwB,
                                                     const float2* wdwC, int grid, cudaStream_t s) {
    const size_t smem = cat_fwd_bytes<TPCF_M>(g.K);
    auto* k = cat_fwd_multi_kernel<TPCF_M>;
    cudaError_t e = prefer_shared(k, smem, BT);
    if (e != cudaSuccess) return e;
    k<<<grid, BT, smem, s>>>(g, c, wdwB, wdwC);
    return cudaGetLastError();
}

int TPCF_CAT(cat_fwd_multi_occupancy_m, TPCF_M)(int K) {
    return occupancy(cat_fwd_multi_kernel<TPCF_M>, cat_fwd_bytes<TPCF_M>(K), BT);
}

// Batched forward / adjoint over all the plans of a batch whose largest m_max is this
// M, by tiles or by blocks (the dynamic shared memory is the largest any of them needs).
template <class Kern>
static cudaError_t launch_batch(Kern* k, const BatchItem* items, int n, long long total, unsigned long long* counter,
                                size_t smem, int grid, int threads, cudaStream_t s) {
    cudaError_t e = prefer_shared(k, smem, threads);
    if (e != cudaSuccess) return e;
    k<<<grid, threads, smem, s>>>(items, n, total, counter);
    return cudaGetLastError();
}

cudaError_t TPCF_CAT(batch_fwd_launch_m, TPCF_M)(const BatchItem* items, int n, long long total,
                                                 unsigned long long* counter, size_t smem, int grid, bool tiles,
                                                 cudaStream_t s) {
    return tiles ? launch_batch(batch_tile_fwd_kernel<TPCF_M>, items, n, total, counter, smem, grid, NTHREADS, s)
                 : launch_batch(batch_fwd_kernel<TPCF_M>, items, n, total, counter, smem, grid, BT, s);
}

cudaError_t TPCF_CAT(batch_bwd_launch_m, TPCF_M)(const BatchItem* items, int n, long long total,
                                                 unsigned long long* counter, size_t smem, int grid, bool tiles,
                                                 cudaStream_t s) {
    return tiles ? launch_batch(batch_tile_bwd_kernel<TPCF_M>, items, n, total, counter, smem, grid, NTHREADS, s)
                 : launch_batch(batch_bwd_kernel<TPCF_M>, items, n, total, counter, smem, grid, BT, s);
}

int TPCF_CAT(batch_fwd_occupancy_m, TPCF_M)(size_t smem, bool tiles) {
    return tiles ? occupancy(batch_tile_fwd_kernel<TPCF_M>, smem) : occupancy(batch_fwd_kernel<TPCF_M>, smem, BT);
}

int TPCF_CAT(batch_bwd_occupancy_m, TPCF_M)(size_t smem, bool tiles) {
    return tiles ? occupancy(batch_tile_bwd_kernel<TPCF_M>, smem) : occupancy(batch_bwd_kernel<TPCF_M>, smem, BT);
}

// Catalogue forward.
cudaError_t TPCF_CAT(cat_fwd_launch_m, TPCF_M)(const CatDev& g, const MapCall& c, int grid, cudaStream_t s) {
    const size_t smem = cat_fwd_bytes<TPCF_M>(g.K);
    if (c.self_subtract) {
        auto* k = cat_fwd_kernel<TPCF_M, true>;
        cudaError_t e = prefer_shared(k, smem, BT);
        if (e != cudaSuccess) return e;
        k<<<grid, BT, smem, s>>>(g, c);
    } else {
        auto* k = cat_fwd_kernel<TPCF_M, false>;
        cudaError_t e = prefer_shared(k, smem, BT);
        if (e != cudaSuccess) return e;
        k<<<grid, BT, smem, s>>>(g, c);
    }
    return cudaGetLastError();
}

int TPCF_CAT(cat_fwd_occupancy_m, TPCF_M)(int K, int self_subtract) {
    const size_t smem = cat_fwd_bytes<TPCF_M>(K);
    return self_subtract ? occupancy(cat_fwd_kernel<TPCF_M, true>, smem, BT) : occupancy(cat_fwd_kernel<TPCF_M, false>, smem, BT);
}

// Catalogue adjoint.
cudaError_t TPCF_CAT(cat_bwd_launch_m, TPCF_M)(const CatDev& g, const MapCall& c, int grid, cudaStream_t s) {
    const size_t smem = cat_bwd_bytes<TPCF_M>(g.K);
    auto* k = cat_bwd_kernel<TPCF_M>;
    cudaError_t e = prefer_shared(k, smem, BT);
    if (e != cudaSuccess) return e;
    k<<<grid, BT, smem, s>>>(g, c);
    return cudaGetLastError();
}

int TPCF_CAT(cat_bwd_occupancy_m, TPCF_M)(int K) {
    const size_t smem = cat_bwd_bytes<TPCF_M>(K);
    return occupancy(cat_bwd_kernel<TPCF_M>, smem, BT);
}

#if TPCF_M == 0
cudaError_t cat_count_launch(const CatDev& g, const float2* wdw, long long lo, long long hi, int* counter,
                             unsigned long long* counts, int grid, cudaStream_t s) {
    const size_t smem = cat_smem_bytes(g.K, false, 0);
    cudaError_t e = prefer_shared(cat_count_kernel, smem, BT);
    if (e != cudaSuccess) return e;
    cat_count_kernel<<<grid, BT, smem, s>>>(g, wdw, lo, hi, counter, counts);
    return cudaGetLastError();
}

cudaError_t map_count_launch(const MapDev& g, const float2* wdw, long long lo, long long hi, long long tlo,
                             long long thi, unsigned long long* counts, int grid, cudaStream_t s) {
    map_count_kernel<<<grid, NTHREADS, 0, s>>>(g, wdw, lo, hi, tlo, thi, counts);
    return cudaGetLastError();
}
#endif

}  // namespace tpcf
