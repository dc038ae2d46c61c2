// The plan object and the error helpers shared by the host translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdio.h>

#include <vector>

#include "tpcf_internal.cuh"

namespace tpcf {
// Records a message for tpcf_last_error() and maps a CUDA error to a status.
tpcf_status cuda_fail(cudaError_t e, const char* where);
// Records a message for tpcf_last_error().
void set_error(const char* msg);
// Every device allocation of the library goes through these two (api.cu): they keep
// the count of live allocations and honour tpcf_test_fail_allocation().
cudaError_t dev_malloc(void** p, size_t bytes);
void dev_free(void* p);
}  // namespace tpcf

#define TRY_CUDA(call)                                                   \
    do {                                                                 \
        cudaError_t _e = (call);                                         \
        if (_e != cudaSuccess) return tpcf::cuda_fail(_e, #call);        \
    } while (0)

enum PlanKind { PLAN_MAP = 1, PLAN_CATALOG = 2 };

struct tpcf_plan_s {
    using MapDev = tpcf::MapDev;
    int kind = 0;
    int device = 0;
    int num_sms = 0;
    int64_t npoints = 0;
    int K = 0, M = 0;
    uint32_t flags = 0;
    std::vector<double> edges;
    std::vector<void*> allocs;  // everything freed by destroy
    MapDev map{};
    tpcf::CatDev cat{};
    std::vector<int64_t> tile_off_h;   // map plans: first tile of each ring (host copy)
    // map plans: first linear block and first warp tile of each ring (and the totals), whether the
    // ring has linear blocks (map_block.cuh)
    std::vector<int64_t> lin_off_h, orb_off_h;
    std::vector<unsigned char> lin_h;
    size_t ws_floats = 0;   // workspace of a block (catalogue plans: of a CTA), see ws_take
    int max_blocks = 0;     // blocks that a call may split into parts
    float* ws_graph = nullptr;  // workspace of calls that were captured into graphs
    size_t ws_graph_floats = 0;
    bool counted = false;   // among the plans that keep the workspaces' pool
    // launch configuration of the map pair kernels (defaults, or picked by the autotuner).  Tile
    // kernels: register variant (sized for 3 or 2 CTAs per SM), CTAs per SM launched, rings summed in
    // registers before a shared-memory flush, and for the forward the tile layout (1: quarter-turn
    // runs).  Block kernels: the same share of their own CTAs, and the flush in units of 32 entries.
    struct Tune {
        int variant = 3, ctas = 0, flush = 8, quad = 0;
    } tune_fwd, tune_bwd;
    bool tuned = false;
    // tile kernels of the map pair passes (map_tile.cuh): resident CTAs per SM by TileKernel and register
    // variant (2, 3); the largest share of the bins' area in one bin, and whether the rule of
    // takes_blocks is overridden (1 tiles, 2 blocks)
    int tile_occ[4][2] = {};
    int occ(int what, int variant) const { return tile_occ[what][variant - 2]; }
    double bin_share = 1.0;
    int route = 0;
    // per-call scratch
    float2* wdw = nullptr;
    double* slots = nullptr;
    int fwd_grid = 0, bwd_grid = 0;
    int nslots = 0;  // CTA slots: the largest grid of a forward by tiles
    int nent = 0;
    double* sums = nullptr;
    int* counter = nullptr;
    int* status = nullptr;
    float* H = nullptr;
    // multi-field forward (allocated on its first call): packed fields B and C, slots
    float2* wdw_b = nullptr;
    float2* wdw_c = nullptr;
    double* mslots = nullptr;
    double* msums = nullptr;
    int multi_grid = 0, multi_ctas = 0;
    // shared-neighbour-list forward: tile list of the last group size used
    int2* gtiles = nullptr;  // linear blocks, then warp tiles of the other rings and of the linear ones
    int64_t nglin = 0, ngorb = 0, ngtile = 0, gtiles_cap = 0;
    double gused = 1.0;  // share of the linear blocks' lanes that stand for a run
    int ggroup = 0;
    // staging for tpcf_run_host
    float* st_delta = nullptr;
    float* st_w = nullptr;
    double* st_dL = nullptr;
    double* st_zeta = nullptr;
    double* st_norm = nullptr;
    float* st_grad = nullptr;
    cudaStream_t last_stream = nullptr;
    long long launches = 0;  // kernels this plan has launched (bookkeeping for benchmarks)

    template <typename T>
    cudaError_t alloc(T** p, size_t count) {
        void* q = nullptr;
        cudaError_t e = tpcf::dev_malloc(&q, count * sizeof(T) > 0 ? count * sizeof(T) : 16);
        if (e != cudaSuccess) return e;
        allocs.push_back(q);
        *p = (T*)q;
        return cudaSuccess;
    }
    // Several arrays from one allocation (each cudaMalloc and cudaFree costs tens of us): add()
    // each, then take().
    struct Arrays {
        std::vector<std::pair<void**, size_t>> parts;  // pointer to set, offset
        size_t bytes = 0;
        template <typename T>
        void add(T** p, size_t count) {
            parts.push_back({(void**)p, bytes});
            bytes += (count * sizeof(T) + 255) / 256 * 256;
        }
        cudaError_t take(tpcf_plan_s* P) {
            char* q = nullptr;
            cudaError_t e = P->alloc(&q, bytes);
            if (e == cudaSuccess)
                for (auto& t : parts) *t.first = q + t.second;
            return e;
        }
    };
    ~tpcf_plan_s();
};

namespace tpcf {
// A call's workspace; given back, in stream order, when the call has enqueued its work.
struct WsLease {
    float* p = nullptr;
    cudaStream_t s = nullptr;
    bool pooled = false;
    WsLease() = default;
    WsLease(const WsLease&) = delete;
    ~WsLease() {
        if (pooled) cudaFreeAsync(p, s);
    }
};
cudaError_t ws_take(tpcf_plan_s* P, size_t floats, cudaStream_t s, WsLease* w);
// counts a new plan among those that keep the pool
void ws_count(tpcf_plan_s* P);
}  // namespace tpcf
