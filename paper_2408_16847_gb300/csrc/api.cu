// Host side of the C ABI declared in include/tpcf.h: plan objects, validation,
// launch sequencing and error reporting.  Every numerical step runs in the
// kernels of geometry.cu, small_kernels.cu and map_kernels.cuh.
#include <cuda_runtime.h>
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <atomic>
#include <mutex>
#include <new>
#include <vector>

#include "geometry.cuh"
#include "plan.cuh"

using namespace tpcf;

namespace tpcf {
// per-M launchers (map_inst.cu)
#define TPCF_DECL_MULTI(m)                                                                                    \
    cudaError_t map_fwd_multi_launch_m##m(const MapDev&, const MapCall&, const float2*, const float2*, int, \
                                          cudaStream_t);                                                  \
    int map_fwd_multi_occupancy_m##m();                                                                   \
    cudaError_t map_tile_multi_launch_m##m(const MapDev&, const MapCall&, const float2*, const float2*, int, \
                                           cudaStream_t);                                                 \
    int map_tile_multi_occupancy_m##m(int);
TPCF_DECL_MULTI(0) TPCF_DECL_MULTI(1) TPCF_DECL_MULTI(2) TPCF_DECL_MULTI(3) TPCF_DECL_MULTI(4) TPCF_DECL_MULTI(5)
TPCF_DECL_MULTI(6) TPCF_DECL_MULTI(7) TPCF_DECL_MULTI(8) TPCF_DECL_MULTI(9) TPCF_DECL_MULTI(10)
TPCF_DECL_MULTI(11) TPCF_DECL_MULTI(12) TPCF_DECL_MULTI(13) TPCF_DECL_MULTI(14) TPCF_DECL_MULTI(15)
TPCF_DECL_MULTI(16)
#undef TPCF_DECL_MULTI
struct MultiLaunch {
    cudaError_t (*blocks)(const MapDev&, const MapCall&, const float2*, const float2*, int, cudaStream_t);
    int (*blocks_occ)();
    cudaError_t (*tiles)(const MapDev&, const MapCall&, const float2*, const float2*, int, cudaStream_t);
    int (*tiles_occ)(int);
};
#define TPCF_ROW_MULTI(m) \
    {map_fwd_multi_launch_m##m, map_fwd_multi_occupancy_m##m, map_tile_multi_launch_m##m, map_tile_multi_occupancy_m##m}
static const MultiLaunch kMulti[TPCF_MAX_M + 1] = {
    TPCF_ROW_MULTI(0),  TPCF_ROW_MULTI(1),  TPCF_ROW_MULTI(2),  TPCF_ROW_MULTI(3),  TPCF_ROW_MULTI(4),
    TPCF_ROW_MULTI(5),  TPCF_ROW_MULTI(6),  TPCF_ROW_MULTI(7),  TPCF_ROW_MULTI(8),  TPCF_ROW_MULTI(9),
    TPCF_ROW_MULTI(10), TPCF_ROW_MULTI(11), TPCF_ROW_MULTI(12), TPCF_ROW_MULTI(13), TPCF_ROW_MULTI(14),
    TPCF_ROW_MULTI(15), TPCF_ROW_MULTI(16)};
#undef TPCF_ROW_MULTI
#define TPCF_DECL_M(m)                                                                         \
    cudaError_t map_fwd_launch_m##m(const MapDev&, const MapCall&, int, cudaStream_t);         \
    cudaError_t map_fwd_tc_launch_m##m(const MapDev&, const MapCall&, int, cudaStream_t);      \
    int map_fwd_tc_occupancy_m##m(int, int);                                                  \
    cudaError_t map_bwd_launch_m##m(const MapDev&, const MapCall&, int, cudaStream_t);         \
    int map_fwd_occupancy_m##m();                                                             \
    int map_bwd_occupancy_m##m();                                                             \
    cudaError_t map_tile_launch_m##m(const MapDev&, const MapCall&, int, int, int, cudaStream_t); \
    int map_tile_occupancy_m##m(int, int, int, int);
TPCF_DECL_M(0) TPCF_DECL_M(1) TPCF_DECL_M(2) TPCF_DECL_M(3) TPCF_DECL_M(4) TPCF_DECL_M(5)
TPCF_DECL_M(6) TPCF_DECL_M(7) TPCF_DECL_M(8) TPCF_DECL_M(9) TPCF_DECL_M(10) TPCF_DECL_M(11)
TPCF_DECL_M(12) TPCF_DECL_M(13) TPCF_DECL_M(14) TPCF_DECL_M(15) TPCF_DECL_M(16)
#undef TPCF_DECL_M
cudaError_t map_count_launch(const MapDev& g, const float2* wdw, long long lo, long long hi, long long tlo,
                             long long thi, unsigned long long* counts, int grid, cudaStream_t s);
// catalogue plans (catalog.cu)
tpcf_status build_catalog(tpcf_plan_s* P, const double* d_xyz, int64_t n, cudaStream_t s);
tpcf_status catalog_count(tpcf_plan_s* P, const float* d_w, int64_t lo, int64_t hi, int64_t* d_counts,
                          cudaStream_t s);
tpcf_status catalog_backward(tpcf_plan_s* P, const float* d_delta, const float* d_w, int64_t lo, int64_t hi,
                             const double* d_norm, const double* d_dL, float* d_grad, cudaStream_t s);
tpcf_status catalog_forward(tpcf_plan_s* P, const float* d_delta, const float* d_w, int64_t lo, int64_t hi,
                            double* d_zeta, double* d_norm, double* d_sums, cudaStream_t s);
tpcf_status catalog_forward_multi(tpcf_plan_s* P, const float* const* d_delta, const float* const* d_w, int64_t lo,
                                  int64_t hi, double* d_zeta, double* d_norm, double* d_sums, cudaStream_t s);
// loads the allocation-free forward's scratch array on a device (noalloc.cu)
tpcf_status noalloc_prepare(int dev);

struct MLaunch {
    cudaError_t (*fwd)(const MapDev&, const MapCall&, int, cudaStream_t);
    cudaError_t (*fwd_tc)(const MapDev&, const MapCall&, int, cudaStream_t);
    int (*fwd_tc_occ)(int, int);
    cudaError_t (*bwd)(const MapDev&, const MapCall&, int, cudaStream_t);
    int (*fwd_occ)();
    int (*bwd_occ)();
    cudaError_t (*tile)(const MapDev&, const MapCall&, int, int, int, cudaStream_t);  // TileKernel, variant, grid
    int (*tile_occ)(int, int, int, int);                                            // TileKernel, variant, K, self
};
#define TPCF_ROW_M(m) \
    {map_fwd_launch_m##m,    map_fwd_tc_launch_m##m,  map_fwd_tc_occupancy_m##m, map_bwd_launch_m##m, \
     map_fwd_occupancy_m##m, map_bwd_occupancy_m##m, map_tile_launch_m##m,      map_tile_occupancy_m##m}
static const MLaunch kLaunch[TPCF_MAX_M + 1] = {
    TPCF_ROW_M(0),  TPCF_ROW_M(1),  TPCF_ROW_M(2),  TPCF_ROW_M(3),  TPCF_ROW_M(4),  TPCF_ROW_M(5),
    TPCF_ROW_M(6),  TPCF_ROW_M(7),  TPCF_ROW_M(8),  TPCF_ROW_M(9),  TPCF_ROW_M(10), TPCF_ROW_M(11),
    TPCF_ROW_M(12), TPCF_ROW_M(13), TPCF_ROW_M(14), TPCF_ROW_M(15), TPCF_ROW_M(16)};
#undef TPCF_ROW_M

// applies a configuration cached by the autotuner (tune.cu)
void tune_from_cache(tpcf_plan_s* P);
}  // namespace tpcf

static thread_local char g_last_error[256] = "";

// Allocation bookkeeping: live device allocations, and the test hook that makes the
// n-th next allocation fail as if the device were out of memory.
static std::atomic<long long> g_live_allocs{0};
static std::atomic<long long> g_fail_countdown{0};

namespace tpcf {
static bool injected_failure() {
    long long c = g_fail_countdown.load();
    while (c > 0)
        if (g_fail_countdown.compare_exchange_weak(c, c - 1)) return c == 1;
    return false;
}

cudaError_t dev_malloc(void** p, size_t bytes) {
    if (injected_failure()) {
        *p = nullptr;
        return cudaErrorMemoryAllocation;
    }
    cudaError_t e = cudaMalloc(p, bytes);
    if (e == cudaSuccess) ++g_live_allocs;
    return e;
}
void dev_free(void* p) {
    if (!p) return;
    cudaFree(p);
    --g_live_allocs;
}

// Workspaces of the block and catalogue kernels (up to 0.5 MB per CTA at 20 bins and m_max 10, 0.3 GB
// in all).  A call takes one for the time its kernels run, from a pool per device that all plans
// share: allocated and freed in stream order, so calls on other streams get memory of their own.
// The pool keeps POOL_BYTES when idle and goes with the device's last plan.  A call that is being
// captured into a graph, which may be replayed on any stream, uses memory that its plan keeps.
// (With a workspace in every plan, 64 plans at 20 bins held 36 GB that only one call at a time used.)
constexpr uint64_t POOL_BYTES = uint64_t(1) << 30;
constexpr int POOL_DEVICES = 64;
static std::mutex g_pool_mu;
static cudaMemPool_t g_pool[POOL_DEVICES];
static int g_pool_plans[POOL_DEVICES];

static cudaError_t ws_pool(int dev, cudaMemPool_t* out) {
    std::lock_guard<std::mutex> lock(g_pool_mu);
    if (!g_pool[dev]) {
        cudaMemPoolProps pr;
        memset(&pr, 0, sizeof(pr));
        pr.allocType = cudaMemAllocationTypePinned;
        pr.location.type = cudaMemLocationTypeDevice;
        pr.location.id = dev;
        cudaMemPool_t pool = nullptr;
        cudaError_t e = cudaMemPoolCreate(&pool, &pr);
        if (e != cudaSuccess) return e;
        uint64_t keep = POOL_BYTES;
        int off = 0;
        e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
        // (otherwise a stream's call could be made to wait for another stream's)
        if (e == cudaSuccess) e = cudaMemPoolSetAttribute(pool, cudaMemPoolReuseAllowInternalDependencies, &off);
        if (e != cudaSuccess) {
            cudaMemPoolDestroy(pool);
            return e;
        }
        g_pool[dev] = pool;
    }
    *out = g_pool[dev];
    return cudaSuccess;
}

void ws_count(tpcf_plan_s* P) {
    if (P->device < 0 || P->device >= POOL_DEVICES) return;
    std::lock_guard<std::mutex> lock(g_pool_mu);
    ++g_pool_plans[P->device];
    P->counted = true;
}

cudaError_t ws_take(tpcf_plan_s* P, size_t floats, cudaStream_t s, WsLease* w) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(s, &cap);
    if (e != cudaSuccess) return e;
    if (cap == cudaStreamCaptureStatusNone && P->counted) {
        cudaMemPool_t pool;
        e = ws_pool(P->device, &pool);
        if (e != cudaSuccess) return e;
        if (injected_failure()) return cudaErrorMemoryAllocation;
        void* q = nullptr;
        e = cudaMallocFromPoolAsync(&q, floats * sizeof(float), pool, s);
        if (e != cudaSuccess) return e;
        w->p = (float*)q;
        w->s = s;
        w->pooled = true;
        return cudaSuccess;
    }
    if (P->ws_graph_floats < floats) {  // (an earlier, smaller one stays: a graph may hold it)
        cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;  // a plain allocation is no part of the graph
        cudaThreadExchangeStreamCaptureMode(&mode);
        float* q = nullptr;
        e = P->alloc(&q, floats);
        cudaThreadExchangeStreamCaptureMode(&mode);
        if (e != cudaSuccess) return e;
        P->ws_graph = q;
        P->ws_graph_floats = floats;
    }
    w->p = P->ws_graph;
    return cudaSuccess;
}
}  // namespace tpcf

tpcf_plan_s::~tpcf_plan_s() {
    for (void* p : allocs) tpcf::dev_free(p);
    if (!counted) return;
    std::lock_guard<std::mutex> lock(tpcf::g_pool_mu);
    if (--tpcf::g_pool_plans[device] == 0 && tpcf::g_pool[device]) {
        cudaMemPoolDestroy(tpcf::g_pool[device]);
        tpcf::g_pool[device] = nullptr;
    }
}

extern "C" void tpcf_test_fail_allocation(int64_t n) { g_fail_countdown.store(n > 0 ? n : 0); }

extern "C" int64_t tpcf_test_live_allocations(void) { return g_live_allocs.load(); }

extern "C" tpcf_status tpcf_test_route(tpcf_plan plan, int32_t route) {
    if (!plan || route < 0 || route > 2) return TPCF_ERR_INVALID_ARG;
    plan->route = route;
    return TPCF_OK;
}

namespace tpcf {
tpcf_status cuda_fail(cudaError_t e, const char* where) {
    snprintf(g_last_error, sizeof(g_last_error), "%s: %s", where, cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? TPCF_ERR_OOM : TPCF_ERR_CUDA;
}
void set_error(const char* msg) { snprintf(g_last_error, sizeof(g_last_error), "%s", msg); }
}  // namespace tpcf

extern "C" const char* tpcf_status_string(tpcf_status s) {
    switch (s) {
        case TPCF_OK: return "TPCF_OK";
        case TPCF_ERR_INVALID_ARG: return "TPCF_ERR_INVALID_ARG";
        case TPCF_ERR_CUDA: return "TPCF_ERR_CUDA";
        case TPCF_ERR_OOM: return "TPCF_ERR_OOM";
        case TPCF_ERR_TIMEOUT: return "TPCF_ERR_TIMEOUT";
        case TPCF_ERR_UNSUPPORTED: return "TPCF_ERR_UNSUPPORTED";
        case TPCF_ERR_DEVICE: return "TPCF_ERR_DEVICE";
    }
    return "TPCF_ERR_UNKNOWN";
}

extern "C" const char* tpcf_last_error(void) { return g_last_error; }

static tpcf_status check_bins(const tpcf_bins* b) {
    if (!b || !b->theta_edges_rad) return TPCF_ERR_INVALID_ARG;
    if (b->nbins < 1 || b->nbins > TPCF_MAX_BINS) return TPCF_ERR_INVALID_ARG;
    if (b->m_max < 0 || b->m_max > TPCF_MAX_M) return TPCF_ERR_INVALID_ARG;
    if (b->flags & ~(uint32_t)(TPCF_SELF_PAIRS_SUBTRACT | TPCF_CONTRACT_TC | NORM_FLAGS)) return TPCF_ERR_INVALID_ARG;
    if ((b->flags & NORM_FLAGS) == NORM_FLAGS) return TPCF_ERR_INVALID_ARG;
    const double* t = b->theta_edges_rad;
    if (!(t[0] > 0.0)) return TPCF_ERR_INVALID_ARG;
    for (int e = 0; e < b->nbins; ++e)
        if (!(t[e + 1] > t[e])) return TPCF_ERR_INVALID_ARG;
    if (!(t[b->nbins] < 0.5 * M_PI)) return TPCF_ERR_INVALID_ARG;
    return TPCF_OK;
}

// Flag combinations the kernels do not implement: a per-pivot normalisation with
// self-pair subtraction or the tensor-core contraction.
static tpcf_status check_norm(const tpcf_bins* b) {
    if ((b->flags & NORM_FLAGS) && (b->flags & (TPCF_SELF_PAIRS_SUBTRACT | TPCF_CONTRACT_TC))) {
        set_error("per-pivot normalisation with self-pair subtraction or the TC contraction");
        return TPCF_ERR_UNSUPPORTED;
    }
    return TPCF_OK;
}

static int n_blocks(int64_t n, int bs) { return (int)((n + bs - 1) / bs); }

static tpcf_status build_map(tpcf_plan_s* P, int64_t nside, cudaStream_t s) {
    MapDev& g = P->map;
    const int nrings = (int)(4 * nside - 1);
    const int K = P->K;
    g.nside = (int)nside;
    g.nrings = nrings;
    g.K = K;
    g.M = P->M;
    g.npix = 12 * nside * nside;
    int64_t *first, *pair_off, *tile_off, *lin_off, *orb_off, *npairs_r, *ntiles_r, *nlin_r, *norb_r, *tot;
    int *npr, *shift;
    double *z, *sd, *th, *E, *theta;
    float *zf, *sf, *sf_lo, *rstep, *rstep_lo, *rinvn, *rinvn_lo;
    int2 *ring_range, *bin_range;
    unsigned char* lin;  // ring classes (map_block.cuh)
    int* reach;
    float4* rc;
    tpcf_plan_s::Arrays rings, pairs, scratch;
    rings.add(&first, nrings);
    rings.add(&npr, nrings);
    rings.add(&shift, nrings);
    rings.add(&z, nrings);
    rings.add(&sd, nrings);
    rings.add(&th, nrings);
    rings.add(&zf, nrings);
    rings.add(&sf, nrings);
    rings.add(&rstep, nrings);
    rings.add(&rinvn, nrings);
    rings.add(&sf_lo, nrings);
    rings.add(&rstep_lo, nrings);
    rings.add(&rinvn_lo, nrings);
    rings.add(&ring_range, nrings);
    rings.add(&bin_range, (size_t)nrings * K);
    rings.add(&pair_off, nrings);
    rings.add(&tile_off, nrings);
    rings.add(&npairs_r, nrings);
    rings.add(&ntiles_r, nrings);
    rings.add(&lin_off, nrings);
    rings.add(&orb_off, nrings);
    rings.add(&nlin_r, nrings);
    rings.add(&norb_r, nrings);
    rings.add(&lin, nrings);
    rings.add(&reach, nrings);
    rings.add(&rc, 2 * (size_t)nrings);
    rings.add(&tot, 4);
    rings.add(&E, K + 1);
    rings.add(&theta, K + 1);
    TRY_CUDA(rings.take(P));
    TRY_CUDA(cudaMemcpyAsync(theta, P->edges.data(), sizeof(double) * (K + 1), cudaMemcpyHostToDevice, s));
    edges_kernel<<<1, 64, 0, s>>>(K, theta, E);
    ring_table_kernel<<<n_blocks(nrings, 128), 128, 0, s>>>((int)nside, nrings, first, npr, shift, z, sd, th,
                                                            zf, sf, sf_lo, rstep, rstep_lo, rinvn, rinvn_lo, rc);
    const int np = walk_np(P->M);
    ring_range_kernel<<<n_blocks(nrings, 128), 128, 0, s>>>(nrings, K, th, sd, E, npr, ring_range, bin_range,
                                                            npairs_r, ntiles_r, nlin_r, norb_r, np, lin, reach);
    exclusive_scan_kernel<<<1, 1024, 0, s>>>(npairs_r, pair_off, nrings, tot);
    exclusive_scan_kernel<<<1, 1024, 0, s>>>(ntiles_r, tile_off, nrings, tot + 1);
    exclusive_scan_kernel<<<1, 1024, 0, s>>>(nlin_r, lin_off, nrings, tot + 2);
    exclusive_scan_kernel<<<1, 1024, 0, s>>>(norb_r, orb_off, nrings, tot + 3);
    TRY_CUDA(cudaGetLastError());
    int64_t totals[4];
    TRY_CUDA(cudaMemcpyAsync(totals, tot, sizeof(totals), cudaMemcpyDeviceToHost, s));
    TRY_CUDA(cudaStreamSynchronize(s));
    const int64_t npairs = totals[0], ntiles = totals[1], nlin = totals[2], norb = totals[3];
    P->tile_off_h.resize(nrings);
    P->lin_off_h.resize(nrings + 1);
    P->orb_off_h.resize(nrings + 1);
    P->lin_h.resize(nrings);
    TRY_CUDA(cudaMemcpyAsync(P->tile_off_h.data(), tile_off, sizeof(int64_t) * nrings, cudaMemcpyDeviceToHost, s));
    TRY_CUDA(cudaMemcpyAsync(P->lin_off_h.data(), lin_off, sizeof(int64_t) * nrings, cudaMemcpyDeviceToHost, s));
    TRY_CUDA(cudaMemcpyAsync(P->orb_off_h.data(), orb_off, sizeof(int64_t) * nrings, cudaMemcpyDeviceToHost, s));
    P->lin_off_h[nrings] = nlin;
    P->orb_off_h[nrings] = norb;
    TRY_CUDA(cudaMemcpyAsync(P->lin_h.data(), lin, nrings, cudaMemcpyDeviceToHost, s));
    float2* pair_A;
    int2 *pair_T, *tiles, *lin_list, *orb_list;
    pairs.add(&pair_A, npairs);
    pairs.add(&pair_T, (size_t)npairs * (K + 1));
    pairs.add(&tiles, ntiles);
    pairs.add(&lin_list, nlin);
    pairs.add(&orb_list, norb);
    TRY_CUDA(pairs.take(P));
    pair_table_kernel<<<n_blocks(npairs, 128), 128, 0, s>>>(nrings, K, pair_off, npairs, ring_range, th, sd,
                                                            npr, E, pair_A, pair_T);
    tile_list_kernel<<<nrings, 128, 0, s>>>(nrings, tile_off, ntiles_r, TILE, tiles);
    tile_list_kernel<<<nrings, 128, 0, s>>>(nrings, lin_off, nlin_r, BT * np, lin_list);
    tile_list_kernel<<<nrings, 128, 0, s>>>(nrings, orb_off, norb_r, TILE, orb_list);
    TRY_CUDA(cudaGetLastError());
    g.ring_reach = reach;
    g.rc = rc;
    g.lin_list = lin_list;
    g.orb_list = orb_list;
    g.ring_first = first;
    g.ring_n = npr;
    g.ring_shift = shift;
    g.ring_zf = zf;
    g.ring_sf = sf;
    g.ring_sf_lo = sf_lo;
    g.ring_step_lo = rstep_lo;
    g.ring_invn_lo = rinvn_lo;
    g.ring_step = rstep;
    g.ring_invn = rinvn;
    g.ring_th = th;
    g.ring_s = sd;
    g.ring_range = ring_range;
    g.bin_range = bin_range;
    g.pair_off = pair_off;
    g.pair_A = pair_A;
    g.pair_T = pair_T;
    g.tiles = tiles;
    g.ntiles = ntiles;
    g.E = E;
    // per-call scratch, sized once so calls allocate nothing
    const MLaunch& L = kLaunch[P->M];
    const int self = (P->flags & TPCF_SELF_PAIRS_SUBTRACT) ? 1 : 0;
    const bool tc = (P->flags & TPCF_CONTRACT_TC) != 0;
    const int occ_f = tc ? L.fwd_tc_occ(K, self) : L.fwd_occ();
    const int occ_b = L.bwd_occ();
    if (occ_f < 1 || occ_b < 1) {
        snprintf(g_last_error, sizeof(g_last_error), "kernel does not fit (K=%d, M=%d)", K, P->M);
        return TPCF_ERR_UNSUPPORTED;
    }
    // slots for the largest grid any configuration launches
    P->fwd_grid = P->num_sms * ((occ_f + 1) / 2 * 2);
    P->bwd_grid = P->num_sms * ((occ_b + 1) / 2 * 2);
    P->max_blocks = (int)std::max<int64_t>(1, std::min<int64_t>(2 * std::max(P->fwd_grid, P->bwd_grid), nlin + norb));
    P->fwd_grid = (int)std::min<int64_t>(P->fwd_grid, 8 * (int64_t)P->max_blocks);
    P->ws_floats = block_floats(K, P->M, P->M, self != 0);
    for (int t = TILE_FWD; t <= TILE_BWD; ++t)
        for (int v = 2; v <= 3; ++v)
            if (t != TILE_GROUPED && t != (tc ? TILE_FWD : TILE_TC)) P->tile_occ[t][v - 2] = L.tile_occ(t, v, K, self);
    cudaGetLastError();  // (a kernel that does not fit leaves its calls to the blocks)
    const int fwd = tc ? TILE_TC : TILE_FWD;
    auto widest = [&](tpcf_plan_s::Tune& t, int what) {
        t.variant = P->occ(what, 3) > 0 ? 3 : 2;
        t.ctas = std::max(1, P->occ(what, t.variant));
    };
    widest(P->tune_fwd, fwd);
    widest(P->tune_bwd, TILE_BWD);
    P->nslots = (int)std::max<int64_t>(
        1, std::min<int64_t>(ntiles, (int64_t)P->num_sms * std::max(P->occ(fwd, 2), P->occ(fwd, 3))));
    P->bin_share = 0.0;
    auto area = [&](int e) { return pow(sin(0.5 * P->edges[e]), 2); };
    for (int k = 0; k < K; ++k) P->bin_share = std::max(P->bin_share, (area(k + 1) - area(k)) / (area(K) - area(0)));
    P->nent = n_entries(K, P->M);
    TRY_CUDA(P->alloc(&P->wdw, g.npix + 1));  // and a zero after the last pixel
    TRY_CUDA(P->alloc(&P->slots, (size_t)P->nslots * P->nent));
    scratch.add(&P->sums, P->nent);
    scratch.add(&P->status, 4);
    scratch.add(&P->H, (size_t)(P->M + 1) * K * K * 2 + K);  // H, then cdiag (self-pair mode)
    TRY_CUDA(scratch.take(P));
    TRY_CUDA(P->alloc(&P->counter, 4 + P->max_blocks));  // work counter (4 words), then finished parts per block
    TRY_CUDA(cudaMemsetAsync(P->status, 0, sizeof(int) * 4, s));
    TRY_CUDA(cudaStreamSynchronize(s));
    return TPCF_OK;
}

extern "C" tpcf_status tpcf_plan_create_map(tpcf_plan* out, int64_t nside, const tpcf_bins* bins, void* stream) {
    if (!out) return TPCF_ERR_INVALID_ARG;
    *out = nullptr;
    if (nside < 1 || nside > 8192) return TPCF_ERR_INVALID_ARG;
    tpcf_status st = check_bins(bins);
    if (st == TPCF_OK) st = check_norm(bins);
    if (st != TPCF_OK) return st;
    tpcf_plan_s* P = new (std::nothrow) tpcf_plan_s();
    if (!P) return TPCF_ERR_OOM;
    P->kind = PLAN_MAP;
    P->K = bins->nbins;
    P->M = bins->m_max;
    P->flags = bins->flags;
    P->edges.assign(bins->theta_edges_rad, bins->theta_edges_rad + bins->nbins + 1);
    P->npoints = 12 * nside * nside;
    cudaError_t e = cudaGetDevice(&P->device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&P->num_sms, cudaDevAttrMultiProcessorCount, P->device);
    if (e != cudaSuccess) {
        delete P;
        return cuda_fail(e, "device query");
    }
    cudaStream_t s = (cudaStream_t)stream;
    st = build_map(P, nside, s);
    if (st != TPCF_OK) {
        cudaStreamSynchronize(s);
        delete P;
        return st;
    }
    ws_count(P);
    tune_from_cache(P);
    // place tpcf_forward_noalloc's fixed scratch on this device now, during set-up;
    // on failure that call reports it, so clear the runtime's last-error state here
    if (noalloc_prepare(P->device) != TPCF_OK) cudaGetLastError();
    P->last_stream = s;
    *out = P;
    return TPCF_OK;
}

extern "C" tpcf_status tpcf_plan_create_catalog(tpcf_plan* out, const double* d_xyz, int64_t n,
                                                const tpcf_bins* bins, void* stream) {
    if (!out) return TPCF_ERR_INVALID_ARG;
    *out = nullptr;
    if (!d_xyz || n < 1 || n > 0x7fffffffLL) return TPCF_ERR_INVALID_ARG;
    tpcf_status st = check_bins(bins);
    if (st == TPCF_OK && (bins->flags & TPCF_CONTRACT_TC)) {
        set_error("catalogue plans use the FP32 contraction");
        return TPCF_ERR_UNSUPPORTED;
    }
    if (st == TPCF_OK) st = check_norm(bins);
    if (st != TPCF_OK) return st;
    tpcf_plan_s* P = new (std::nothrow) tpcf_plan_s();
    if (!P) return TPCF_ERR_OOM;
    P->kind = PLAN_CATALOG;
    P->K = bins->nbins;
    P->M = bins->m_max;
    P->flags = bins->flags;
    P->edges.assign(bins->theta_edges_rad, bins->theta_edges_rad + bins->nbins + 1);
    P->npoints = n;
    cudaError_t e = cudaGetDevice(&P->device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&P->num_sms, cudaDevAttrMultiProcessorCount, P->device);
    if (e != cudaSuccess) {
        delete P;
        return cuda_fail(e, "device query");
    }
    cudaStream_t s = (cudaStream_t)stream;
    st = build_catalog(P, d_xyz, n, s);
    if (st != TPCF_OK) {
        cudaStreamSynchronize(s);
        delete P;
        return st;
    }
    ws_count(P);
    P->last_stream = s;
    *out = P;
    return TPCF_OK;
}

extern "C" int64_t tpcf_plan_npoints(tpcf_plan plan) { return plan ? plan->npoints : -1; }

extern "C" int64_t tpcf_plan_kernel_launches(tpcf_plan plan) { return plan ? plan->launches : -1; }

// 0-based ring of RING-order pixel p (HEALPix, Gorski et al. 2005).
static int64_t ring_of_pixel(int64_t nside, int64_t p) {
    const int64_t ncap = 2 * nside * (nside - 1), npix = 12 * nside * nside;
    auto cap_ring = [](int64_t q) {  // 1-based ring r of the north cap holding q: 2r(r-1) <= q
        int64_t r = (int64_t)((1.0 + sqrt(1.0 + 2.0 * (double)q)) * 0.5);
        while (2 * r * (r - 1) > q) --r;
        while (2 * (r + 1) * r <= q) ++r;
        return r;
    };
    if (p < ncap) return cap_ring(p) - 1;
    if (p < npix - ncap) return (p - ncap) / (4 * nside) + nside - 1;
    return 4 * nside - 1 - cap_ring(npix - 1 - p);
}

static int64_t ring_first_pixel(int64_t nside, int64_t ri) {  // 0-based ring
    const int64_t r = ri + 1;
    if (r < nside) return 2 * r * (r - 1);
    if (r <= 3 * nside) return 2 * nside * (nside - 1) + 4 * nside * (r - nside);
    const int64_t rr = 4 * nside - r;
    return 12 * nside * nside - 2 * rr * (rr + 1);
}

// Tiles [*tlo, *thi) of 32 pivots that can hold one of [lo, hi): those of the range's pixels, in the
// quarter-turn layout those of its rings (a ring's pivots are spread over all of its tiles).
static void tile_range(const tpcf_plan_s* P, int64_t lo, int64_t hi, int64_t* tlo, int64_t* thi, bool quad = false) {
    if (hi <= lo) {
        *tlo = *thi = 0;
        return;
    }
    const int64_t nside = P->map.nside;
    const int64_t ra = ring_of_pixel(nside, lo), rb = ring_of_pixel(nside, hi - 1);
    if (quad) {
        *tlo = P->tile_off_h[ra];
        *thi = rb + 1 < (int64_t)P->tile_off_h.size() ? P->tile_off_h[rb + 1] : P->map.ntiles;
        return;
    }
    *tlo = P->tile_off_h[ra] + (lo - ring_first_pixel(nside, ra)) / TILE;
    *thi = P->tile_off_h[rb] + (hi - 1 - ring_first_pixel(nside, rb)) / TILE + 1;
}

// Blocks and parts of a pass over lin_list [lin_lo, lin_lo + nlin) and orb_list [orb_lo, orb_lo + norb)
// (map_block.cuh) for `fields` fields; returns the grid.  Warp tiles go four to a block (one
// per warp), or two if that leaves fewer than four blocks per CTA of a full grid; a call with
// fewer than three blocks per CTA splits each by bins.  The workspace then holds every block
// at once: not beyond WS_PARTS bytes (1216 blocks at 20 bins and m_max 10 take 0.57 GB).
constexpr double WS_PARTS = 1 << 30;

static int block_shape(const tpcf_plan_s* P, const tpcf_plan_s::Tune& t, int occ, int cap, MapCall* c, int fields = 1) {
    // four CTAs of BT threads fit an SM; of `occ` tiles the configuration launches t.ctas
    const int64_t full = (int64_t)P->num_sms * std::max(1, std::min(4, (4 * t.ctas + occ - 1) / std::max(1, occ)));
    auto blocks = [&](int tiles) { return c->nlin + (c->norb + tiles - 1) / tiles; };
    c->tiles = BW;
    while (c->tiles > 2 && blocks(c->tiles) < 4 * full) c->tiles /= 2;
    c->slices = 1;
    if (few_tiles(c->norb, P->K, P->num_sms)) {
        c->tiles = 1;
        c->slices = 4;
    }
    c->ws_floats = fields * P->ws_floats;
    const int64_t n = blocks(c->tiles);
    c->parts = 1;
    if (n < 3 * full && n <= P->max_blocks && n > 0 && (double)n * c->ws_floats * sizeof(float) <= WS_PARTS)
        c->parts = (int)std::min<int64_t>(std::min(8, P->K), (4 * full + n - 1) / n);
    c->done = P->counter + 4;
    return (int)std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(n * c->parts, full), cap));
}

// Takes the workspace of a pass by blocks and sets it in the call: `nent` sums per CTA (a forward's
// slots), then a block per CTA, or one per block where blocks are split.
static cudaError_t blocks_ws(tpcf_plan_s* P, MapCall* c, int grid, int nent, cudaStream_t s, WsLease* w) {
    const int64_t blocks = c->parts > 1 ? c->nlin + (c->norb + c->tiles - 1) / c->tiles : grid;
    const size_t slots = ((size_t)grid * nent * 2 + 63) / 64 * 64;  // floats
    cudaError_t e = ws_take(P, slots + c->ws_floats * (size_t)blocks, s, w);
    if (e != cudaSuccess) return e;
    if (nent) c->slots = reinterpret_cast<double*>(w->p);
    c->ws = w->p + slots;
    return cudaSuccess;
}

// Whether a call goes to the block kernels (map_block.cuh) or to the tile kernels (map_tile.cuh), from
// the call's block_shape.  The blocks evaluate an angle once for several pivots, but give the
// entries of one (warp tile, bin, slice) to one warp and those of one (linear block, part) to one CTA.
// They win where that longest item is short beside the call: `fill` is how many times the longest
// items of all warp tiles would fill the GPU's warps, plus four times the same for the linear blocks and
// the GPU's CTAs (a linear block shares its angles among 256 pivots, so it pays at a quarter of the filling).
// With fewer, most warps wait for a few, and a tile, whose rings eight warps share, is sooner done.
// Shared lists: `share` of the list has pivots in range, and `used` of the linear blocks' lanes have a run.
// Measured on a GB300 over 1,100 calls (Nside 8 to 1200, 1 to 24 bins, m <= 16): below the limits the
// blocks took up to 2.4 times the tiles' time (forward, Nside 200, 1 bin, a slice of 960 pivots: 211 against
// 90 us; three fields, Nside 16, 2 bins: 222 against 110; shared lists of 12, Nside 91: 241 against 197),
// above them 0.3 to 1.03 times (Nside 128, 8 bins: 283 against 555 us).
constexpr double FILL_FWD = 4.5, FILL_MULTI = 4.0, FILL_TC = 5.0, FILL_BWD = 5.0, FILL_GROUPED = 6.0;

static bool takes_blocks(const tpcf_plan_s* P, const MapCall& c, double need, int tile_occ, double share = 1.0,
                         double used = 1.0) {
    if (tile_occ < 1) return true;
    if (P->route) return P->route == 2;
    // shared lists have no images to pair, so one dominant bin leaves the blocks no gain
    if (c.group > 1 && P->bin_share > 0.5) return false;
    const double ctas = 4.0 * P->num_sms, warps = BW * ctas, f = P->bin_share;
    const double fill = c.norb * share * c.slices / (f * warps) +
                        4.0 * c.nlin * share * used / (std::max(f, 1.0 / c.parts) * ctas);
    return fill >= need;
}

static int tile_grid(const tpcf_plan_s* P, int64_t ntiles, int ctas, int cap) {
    const int64_t g = std::min<int64_t>(ntiles, (int64_t)P->num_sms * ctas);
    return (int)std::max<int64_t>(1, std::min<int64_t>(g, cap));
}

static void block_range(const tpcf_plan_s* P, int64_t lo, int64_t hi, MapCall* c) {
    c->lin_list = P->map.lin_list;
    c->orb_list = P->map.orb_list;
    c->lin_lo = c->nlin = c->orb_lo = c->norb = 0;
    if (hi <= lo) return;
    const int64_t nside = P->map.nside, per = (int64_t)BT * walk_np(P->M);
    const int64_t ra = ring_of_pixel(nside, lo), rb = ring_of_pixel(nside, hi - 1);
    c->lin_lo = P->lin_off_h[ra] + (P->lin_h[ra] ? (lo - ring_first_pixel(nside, ra)) / per : 0);
    const int64_t end = P->lin_h[rb] ? P->lin_off_h[rb] + (hi - 1 - ring_first_pixel(nside, rb)) / per + 1
                                     : P->lin_off_h[rb];
    c->nlin = std::max<int64_t>(0, end - c->lin_lo);
    c->orb_lo = P->orb_off_h[ra];  // a partial ring's pivots are spread over all of its warp tiles
    c->norb = P->orb_off_h[rb + 1] - c->orb_lo;
}

// Ints of P->counter a launch needs zeroed: the work counter, and the blocks' finished parts.
static int n_counters(const tpcf_plan_s* P, const MapCall& c) { return 4 + (c.parts > 1 ? P->max_blocks : 0); }

namespace tpcf {
// The kernels that a pass over the whole map takes (1 tiles, 2 blocks), for the autotuner (tune.cu).
int map_route(const tpcf_plan_s* P, bool bwd) {
    const int occ = P->occ(bwd ? TILE_BWD : TILE_FWD, 3);
    const tpcf_plan_s::Tune t{3, occ, 8, 0};  // (not the plan's, which tuning changes)
    MapCall c{};
    block_range(P, 0, P->npoints, &c);
    block_shape(P, t, occ, bwd ? P->bwd_grid : P->fwd_grid, &c);
    return takes_blocks(P, c, bwd ? FILL_BWD : FILL_FWD, occ) ? 2 : 1;
}
}  // namespace tpcf

// group > 1: shared neighbour lists over P->gtiles (tpcf_forward_grouped).
static tpcf_status map_forward(tpcf_plan_s* P, const float* d_delta, const float* d_w, int64_t lo, int64_t hi,
                               double* d_zeta, double* d_norm, double* d_sums, cudaStream_t s, int group = 1) {
    const MapDev& g = P->map;
    P->launches += 4;  // prep, forward, reduce, finalize
    MapCall c{};
    c.wdw = P->wdw;
    c.piv_lo = lo;
    c.piv_hi = hi;
    c.slots = P->slots;
    c.counter = P->counter;
    c.status = P->status;
    c.self_subtract = (P->flags & TPCF_SELF_PAIRS_SUBTRACT) ? 1 : 0;
    c.norm = norm_of_flags(P->flags);
    c.flush = P->tune_fwd.flush;
    c.cells = LIN_CELLS;
    if (group > 1) {  // every run's block; those without a pivot in range return at once
        c.group = group;
        c.lin_list = P->gtiles;
        c.orb_list = P->gtiles + P->nglin;
        c.nlin = P->nglin;
        c.norb = P->ngorb;
    } else {
        block_range(P, lo, hi, &c);
    }
    const tpcf_plan_s::Tune& t = P->tune_fwd;
    const bool tc = (P->flags & TPCF_CONTRACT_TC) != 0;
    const int what = group > 1 ? TILE_GROUPED : (tc ? TILE_TC : TILE_FWD), occ = P->occ(tc ? TILE_TC : TILE_FWD, t.variant);
    int grid = block_shape(P, t, occ, P->fwd_grid, &c);
    const bool blocks = takes_blocks(P, c, group > 1 ? FILL_GROUPED : (tc ? FILL_TC : FILL_FWD), occ,
                                     group > 1 ? (double)(hi - lo) / g.npix : 1.0, group > 1 ? P->gused : 1.0);
    if (!blocks) {
        c.parts = 1;
        if (group > 1) {
            c.gtiles = P->gtiles + P->nglin;
            c.tile_hi = P->ngorb + P->ngtile;
        } else {
            c.quad = t.quad;
            tile_range(P, lo, hi, &c.tile_lo, &c.tile_hi, c.quad != 0);
        }
        grid = tile_grid(P, c.tile_hi - c.tile_lo, t.ctas, P->nslots);
    }
    WsLease ws;
    if (blocks) TRY_CUDA(blocks_ws(P, &c, grid, P->nent, s, &ws));
    fwd_prep_kernel<<<P->num_sms * 8, 256, 0, s>>>(d_delta, d_w, P->wdw, g.npix, c.slots, (int64_t)grid * P->nent,
                                                   P->counter, n_counters(P, c));
    if (!blocks)
        TRY_CUDA(kLaunch[P->M].tile(g, c, what, t.variant, grid, s));
    else if (tc)
        TRY_CUDA(kLaunch[P->M].fwd_tc(g, c, grid, s));
    else
        TRY_CUDA(kLaunch[P->M].fwd(g, c, grid, s));
    reduce_slots_kernel<<<n_blocks(P->nent, 32), REDUCE_THREADS, 0, s>>>(c.slots, grid, P->nent, P->sums);
    const int nout = (P->M + 1) * P->K * P->K;
    finalize_kernel<<<n_blocks(nout, 128), 128, 0, s>>>(P->sums, P->K, P->M, c.self_subtract, 1.0, d_zeta,
                                                        d_norm, d_sums);
    TRY_CUDA(cudaGetLastError());
    return TPCF_OK;
}

extern "C" tpcf_status tpcf_forward_grouped(tpcf_plan plan, const float* d_delta, const float* d_w, int32_t group,
                                            int64_t pivot_begin, int64_t pivot_end, double* d_zeta, double* d_norm,
                                            double* d_sums, void* stream) {
    if (!plan || !d_delta || !d_w || !d_zeta || !d_norm) return TPCF_ERR_INVALID_ARG;
    if (pivot_begin < 0 || pivot_end < pivot_begin || pivot_end > plan->npoints) return TPCF_ERR_INVALID_ARG;
    if (group < 1 || group > 4096) return TPCF_ERR_INVALID_ARG;
    if (plan->kind != PLAN_MAP || (plan->flags & (TPCF_CONTRACT_TC | TPCF_SELF_PAIRS_SUBTRACT | NORM_FLAGS))) {
        set_error("tpcf_forward_grouped: map plans with the default flags only");
        return TPCF_ERR_UNSUPPORTED;
    }
    cudaStream_t s = (cudaStream_t)stream;
    plan->last_stream = s;
    if (group == 1) return map_forward(plan, d_delta, d_w, pivot_begin, pivot_end, d_zeta, d_norm, d_sums, s);
    tpcf_plan_s* P = plan;
    if (P->ggroup != group) {  // the blocks of this run length
        const int64_t nside = P->map.nside;
        std::vector<int2> t, orb, lin_tiles;
        int64_t lin_runs = 0;
        for (int r = 0; r < P->map.nrings; ++r) {
            const int64_t ri = r + 1;
            const int64_t n = ri < nside ? 4 * ri : (ri <= 3 * nside ? 4 * nside : 4 * (4 * nside - ri));
            const int64_t ng = (n + group - 1) / group;
            if (P->lin_h[r]) {
                lin_runs += ng;
                for (int64_t f = 0; f < ng; f += BT * walk_np(P->M)) t.push_back(make_int2(r, (int)f));
            }
            for (int64_t f = 0; f < ng; f += TILE) (P->lin_h[r] ? lin_tiles : orb).push_back(make_int2(r, (int)f));
        }
        const int64_t nglin = (int64_t)t.size(), ngorb = (int64_t)orb.size();
        t.insert(t.end(), orb.begin(), orb.end());
        t.insert(t.end(), lin_tiles.begin(), lin_tiles.end());
        if ((int64_t)t.size() > P->gtiles_cap) {
            int2* buf = nullptr;
            TRY_CUDA(P->alloc(&buf, t.size()));
            P->gtiles = buf;
            P->gtiles_cap = (int64_t)t.size();
        }
        TRY_CUDA(cudaMemcpyAsync(P->gtiles, t.data(), sizeof(int2) * t.size(), cudaMemcpyHostToDevice, s));
        TRY_CUDA(cudaStreamSynchronize(s));
        P->nglin = nglin;
        P->ngorb = ngorb;
        P->ngtile = (int64_t)lin_tiles.size();
        P->gused = nglin ? (double)lin_runs / (nglin * BT * walk_np(P->M)) : 1.0;
        P->ggroup = group;
    }
    return map_forward(P, d_delta, d_w, pivot_begin, pivot_end, d_zeta, d_norm, d_sums, s, group);
}

extern "C" tpcf_status tpcf_forward(tpcf_plan plan, const float* d_delta, const float* d_w, int64_t pivot_begin,
                                    int64_t pivot_end, double* d_zeta, double* d_norm, double* d_sums,
                                    void* stream) {
    if (!plan || !d_delta || !d_w || !d_zeta || !d_norm) return TPCF_ERR_INVALID_ARG;
    if (pivot_begin < 0 || pivot_end < pivot_begin || pivot_end > plan->npoints) return TPCF_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    plan->last_stream = s;
    if (plan->kind == PLAN_MAP) return map_forward(plan, d_delta, d_w, pivot_begin, pivot_end, d_zeta, d_norm,
                                                   d_sums, s);
    if (plan->kind == PLAN_CATALOG)
        return catalog_forward(plan, d_delta, d_w, pivot_begin, pivot_end, d_zeta, d_norm, d_sums, s);
    return TPCF_ERR_UNSUPPORTED;
}

extern "C" tpcf_status tpcf_forward_multi(tpcf_plan plan, const float* d_delta_a, const float* d_w_a,
                                          const float* d_delta_b, const float* d_w_b, const float* d_delta_c,
                                          const float* d_w_c, int64_t pivot_begin, int64_t pivot_end, double* d_zeta,
                                          double* d_norm, double* d_sums, void* stream) {
    if (!plan || !d_delta_a || !d_w_a || !d_delta_b || !d_w_b || !d_delta_c || !d_w_c || !d_zeta || !d_norm)
        return TPCF_ERR_INVALID_ARG;
    if (pivot_begin < 0 || pivot_end < pivot_begin || pivot_end > plan->npoints) return TPCF_ERR_INVALID_ARG;
    tpcf_plan_s* P = plan;
    if (P->flags & (TPCF_CONTRACT_TC | TPCF_SELF_PAIRS_SUBTRACT | NORM_FLAGS)) {
        set_error("tpcf_forward_multi: plans with the FP32 contraction, self pairs kept, default normalisation");
        return TPCF_ERR_UNSUPPORTED;
    }
    cudaStream_t s = (cudaStream_t)stream;
    P->last_stream = s;
    if (P->kind == PLAN_CATALOG) {
        const float* dd[3] = {d_delta_a, d_delta_b, d_delta_c};
        const float* ww[3] = {d_w_a, d_w_b, d_w_c};
        return catalog_forward_multi(P, dd, ww, pivot_begin, pivot_end, d_zeta, d_norm, d_sums, s);
    }
    if (P->kind != PLAN_MAP) return TPCF_ERR_UNSUPPORTED;
    const MapDev& g = P->map;
    const int K = P->K, M = P->M;
    const int nent = n_entries_multi(K, M);
    if (!P->wdw_b) {
        // the three fields' moments of one tile have to fit an SM: the tile kernel's limit, and so the
        // call's at every size (the blocks would take more)
        if (((size_t)3 * (K * (M + 1) * 2 + K) * TILE + 6 * TILE) * sizeof(float) > 232448 || kMulti[M].blocks_occ() < 1) {
            snprintf(g_last_error, sizeof(g_last_error),
                     "tpcf_forward_multi: three fields' moments (K=%d, m_max=%d) do not fit in shared memory", K, M);
            return TPCF_ERR_UNSUPPORTED;
        }
        P->multi_ctas = kMulti[M].tiles_occ(K);
        const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(g.ntiles, (int64_t)P->num_sms * P->multi_ctas));
        float2 *b, *c;
        double *sl, *su;
        TRY_CUDA(P->alloc(&b, g.npix + 1));
        TRY_CUDA(P->alloc(&c, g.npix + 1));
        TRY_CUDA(P->alloc(&sl, (size_t)grid * nent));
        TRY_CUDA(P->alloc(&su, (size_t)nent));
        P->wdw_c = c;
        P->mslots = sl;
        P->msums = su;
        P->multi_grid = grid;
        P->wdw_b = b;
    }
    pack_kernel<<<P->num_sms * 8, 256, 0, s>>>(d_delta_b, d_w_b, P->wdw_b, g.npix);
    pack_kernel<<<P->num_sms * 8, 256, 0, s>>>(d_delta_c, d_w_c, P->wdw_c, g.npix);
    MapCall c{};
    c.wdw = P->wdw;
    c.piv_lo = pivot_begin;
    c.piv_hi = pivot_end;
    c.slots = P->mslots;
    c.counter = P->counter;
    c.status = P->status;
    c.flush = P->tune_fwd.flush;
    c.cells = LIN_CELLS;
    block_range(P, pivot_begin, pivot_end, &c);
    int grid = block_shape(P, P->tune_fwd, P->occ(TILE_FWD, P->tune_fwd.variant), P->fwd_grid, &c, 3);
    const bool blocks = takes_blocks(P, c, FILL_MULTI, P->multi_ctas);
    if (!blocks) {
        c.parts = 1;
        tile_range(P, pivot_begin, pivot_end, &c.tile_lo, &c.tile_hi, true);
        grid = tile_grid(P, c.tile_hi - c.tile_lo, P->multi_ctas, P->multi_grid);
    }
    WsLease ws;
    if (blocks) TRY_CUDA(blocks_ws(P, &c, grid, nent, s, &ws));
    fwd_prep_kernel<<<P->num_sms * 8, 256, 0, s>>>(d_delta_a, d_w_a, P->wdw, g.npix, c.slots, (int64_t)grid * nent,
                                                   P->counter, n_counters(P, c));
    TRY_CUDA((blocks ? kMulti[M].blocks : kMulti[M].tiles)(g, c, P->wdw_b, P->wdw_c, grid, s));
    reduce_slots_kernel<<<n_blocks(nent, 32), REDUCE_THREADS, 0, s>>>(c.slots, grid, nent, P->msums);
    const int nout = (M + 1) * K * K;
    finalize_full_kernel<<<n_blocks(nout, 128), 128, 0, s>>>(P->msums, K, M, d_zeta, d_norm, d_sums);
    P->launches += 6;  // prep and two packs, the pair kernel, reduce, finalize
    TRY_CUDA(cudaGetLastError());
    return TPCF_OK;
}

extern "C" tpcf_status tpcf_count_pairs(tpcf_plan plan, const float* d_w, int64_t pivot_begin,
                                        int64_t pivot_end, int64_t* d_counts, void* stream) {
    if (!plan || !d_w || !d_counts) return TPCF_ERR_INVALID_ARG;
    if (pivot_begin < 0 || pivot_end < pivot_begin || pivot_end > plan->npoints) return TPCF_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    plan->last_stream = s;
    if (plan->kind == PLAN_CATALOG) return catalog_count(plan, d_w, pivot_begin, pivot_end, d_counts, s);
    if (plan->kind != PLAN_MAP) return TPCF_ERR_UNSUPPORTED;
    const MapDev& g = plan->map;
    // only the weights matter: pack them with a zero field
    pack_kernel<<<plan->num_sms * 8, 256, 0, s>>>(d_w, d_w, plan->wdw, g.npix);
    plan->launches += 2;
    TRY_CUDA(cudaMemsetAsync(d_counts, 0, 3 * sizeof(int64_t), s));
    int64_t tlo, thi;
    tile_range(plan, pivot_begin, pivot_end, &tlo, &thi);
    TRY_CUDA(map_count_launch(g, plan->wdw, pivot_begin, pivot_end, tlo, thi, (unsigned long long*)d_counts,
                              plan->num_sms * 4, s));
    return TPCF_OK;
}

static tpcf_status map_backward(tpcf_plan_s* P, const float* d_delta, const float* d_w, int64_t lo, int64_t hi,
                                const double* d_norm, const double* d_dL, float* d_grad, cudaStream_t s) {
    const MapDev& g = P->map;
    const int self = (P->flags & TPCF_SELF_PAIRS_SUBTRACT) ? 1 : 0;
    P->launches += 2;  // prep, adjoint
    MapCall c{};
    c.wdw = P->wdw;
    c.piv_lo = lo;
    c.piv_hi = hi;
    c.counter = P->counter;
    c.status = P->status;
    c.H = P->H;
    c.grad = d_grad;
    c.self_subtract = self;
    c.flush = P->tune_bwd.flush;
    c.cells = LIN_CELLS;
    block_range(P, lo, hi, &c);
    const tpcf_plan_s::Tune& t = P->tune_bwd;
    const int occ = P->occ(TILE_BWD, t.variant);
    int grid = block_shape(P, t, occ, P->bwd_grid, &c);
    const bool blocks = takes_blocks(P, c, FILL_BWD, occ);
    if (!blocks) {
        c.parts = 1;
        tile_range(P, lo, hi, &c.tile_lo, &c.tile_hi);
        grid = tile_grid(P, c.tile_hi - c.tile_lo, t.ctas, P->num_sms * t.ctas);
    }
    WsLease ws;
    if (blocks) TRY_CUDA(blocks_ws(P, &c, grid, 0, s, &ws));
    bwd_prep_kernel<<<P->num_sms * 8, 256, 0, s>>>(d_delta, d_w, P->wdw, d_grad, g.npix, d_dL, d_norm, P->K, P->M, P->H,
                                                   self, P->counter, n_counters(P, c));
    if (!blocks) {
        TRY_CUDA(kLaunch[P->M].tile(g, c, TILE_BWD, t.variant, grid, s));
        return TPCF_OK;
    }
    c.step = c.parts > 1 ? 1 : 0;
    TRY_CUDA(kLaunch[P->M].bwd(g, c, grid, s));
    if (c.step == 1) {  // the blocks' h are in the workspace: the neighbour legs, again in parts
        TRY_CUDA(cudaMemsetAsync(P->counter, 0, sizeof(int), s));
        c.step = 2;
        TRY_CUDA(kLaunch[P->M].bwd(g, c, grid, s));
        P->launches += 1;
    }
    return TPCF_OK;
}

extern "C" tpcf_status tpcf_backward(tpcf_plan plan, const float* d_delta, const float* d_w, int64_t pivot_begin,
                                     int64_t pivot_end, const double* d_norm, const double* d_dL_dzeta,
                                     float* d_grad, void* stream) {
    if (!plan || !d_delta || !d_w || !d_norm || !d_dL_dzeta || !d_grad) return TPCF_ERR_INVALID_ARG;
    if (pivot_begin < 0 || pivot_end < pivot_begin || pivot_end > plan->npoints) return TPCF_ERR_INVALID_ARG;
    if (plan->flags & NORM_FLAGS) {
        set_error("tpcf_backward: plans with a per-pivot normalisation have no adjoint");
        return TPCF_ERR_UNSUPPORTED;
    }
    cudaStream_t s = (cudaStream_t)stream;
    plan->last_stream = s;
    if (plan->kind == PLAN_MAP)
        return map_backward(plan, d_delta, d_w, pivot_begin, pivot_end, d_norm, d_dL_dzeta, d_grad, s);
    if (plan->kind == PLAN_CATALOG)
        return catalog_backward(plan, d_delta, d_w, pivot_begin, pivot_end, d_norm, d_dL_dzeta, d_grad, s);
    return TPCF_ERR_UNSUPPORTED;
}

extern "C" tpcf_status tpcf_plan_halo(tpcf_plan plan, int64_t begin, int64_t end, int64_t* halo_begin,
                                      int64_t* halo_end) {
    if (!plan || !halo_begin || !halo_end) return TPCF_ERR_INVALID_ARG;
    if (begin < 0 || end < begin || end > plan->npoints) return TPCF_ERR_INVALID_ARG;
    if (plan->kind != PLAN_MAP) {
        set_error("tpcf_plan_halo: map plans only");
        return TPCF_ERR_UNSUPPORTED;
    }
    if (begin == end) {
        *halo_begin = *halo_end = begin;
        return TPCF_OK;
    }
    const int64_t nside = plan->map.nside;
    const int64_t ra = ring_of_pixel(nside, begin), rb = ring_of_pixel(nside, end - 1);
    int2 wa, wb;
    // ring windows are symmetric (ring r is in reach of ring i iff i is in reach of r)
    // and monotone in the ring index, so the halo rings are those of the end rings
    TRY_CUDA(cudaMemcpy(&wa, plan->map.ring_range + ra, sizeof(int2), cudaMemcpyDeviceToHost));
    TRY_CUDA(cudaMemcpy(&wb, plan->map.ring_range + rb, sizeof(int2), cudaMemcpyDeviceToHost));
    *halo_begin = ring_first_pixel(nside, wa.x);
    *halo_end = ring_first_pixel(nside, (int64_t)wb.y + 1);
    return TPCF_OK;
}

extern "C" tpcf_status tpcf_run_host(tpcf_plan plan, const float* h_delta, const float* h_w,
                                     const double* h_dL_dzeta, double* h_zeta, double* h_norm, float* h_grad,
                                     void* stream) {
    if (!plan || !h_delta || !h_w || !h_zeta || !h_norm) return TPCF_ERR_INVALID_ARG;
    if (h_dL_dzeta && !h_grad) return TPCF_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    tpcf_plan_s* P = plan;
    const int64_t n = P->npoints;
    const size_t nz = (size_t)(P->M + 1) * P->K * P->K * 2;
    if (!P->st_delta) {
        // staging buffers, kept by the plan; published together so that a failed
        // allocation leaves the plan as it was (what was allocated is freed with it)
        float *sd, *sw, *sg;
        double *sdl, *sz, *sn;
        TRY_CUDA(P->alloc(&sd, n));
        TRY_CUDA(P->alloc(&sw, n));
        TRY_CUDA(P->alloc(&sdl, nz));
        TRY_CUDA(P->alloc(&sz, nz));
        TRY_CUDA(P->alloc(&sn, (size_t)P->K * P->K));
        TRY_CUDA(P->alloc(&sg, n));
        P->st_w = sw;
        P->st_dL = sdl;
        P->st_zeta = sz;
        P->st_norm = sn;
        P->st_grad = sg;
        P->st_delta = sd;
    }
    TRY_CUDA(cudaMemcpyAsync(P->st_delta, h_delta, sizeof(float) * n, cudaMemcpyHostToDevice, s));
    TRY_CUDA(cudaMemcpyAsync(P->st_w, h_w, sizeof(float) * n, cudaMemcpyHostToDevice, s));
    tpcf_status st = tpcf_forward(P, P->st_delta, P->st_w, 0, n, P->st_zeta, P->st_norm, nullptr, stream);
    if (st != TPCF_OK) return st;
    if (h_dL_dzeta) {
        TRY_CUDA(cudaMemcpyAsync(P->st_dL, h_dL_dzeta, sizeof(double) * nz, cudaMemcpyHostToDevice, s));
        st = tpcf_backward(P, P->st_delta, P->st_w, 0, n, P->st_norm, P->st_dL, P->st_grad, stream);
        if (st != TPCF_OK) return st;
        TRY_CUDA(cudaMemcpyAsync(h_grad, P->st_grad, sizeof(float) * n, cudaMemcpyDeviceToHost, s));
    }
    TRY_CUDA(cudaMemcpyAsync(h_zeta, P->st_zeta, sizeof(double) * nz, cudaMemcpyDeviceToHost, s));
    TRY_CUDA(cudaMemcpyAsync(h_norm, P->st_norm, sizeof(double) * P->K * P->K, cudaMemcpyDeviceToHost, s));
    TRY_CUDA(cudaStreamSynchronize(s));
    return tpcf_plan_sync(P);
}

extern "C" tpcf_status tpcf_plan_sync(tpcf_plan plan) {
    if (!plan) return TPCF_ERR_INVALID_ARG;
    TRY_CUDA(cudaStreamSynchronize(plan->last_stream));
    int st = 0;
    TRY_CUDA(cudaMemcpy(&st, plan->status, sizeof(int), cudaMemcpyDeviceToHost));
    if (st & ST_TC_TIMEOUT_BIT) {
        snprintf(g_last_error, sizeof(g_last_error), "device status 0x%x (tensor-core wait timed out)", st);
        return TPCF_ERR_TIMEOUT;
    }
    if (st & ST_BAD_TILE) {
        snprintf(g_last_error, sizeof(g_last_error), "device status 0x%x (bad tile table)", st);
        return TPCF_ERR_DEVICE;
    }
    return TPCF_OK;
}

extern "C" void tpcf_plan_destroy(tpcf_plan plan) {
    if (!plan) return;
    cudaStreamSynchronize(plan->last_stream);
    delete plan;
}
