// Internal declarations shared by the translation units of libtpcf.
// Device views of plans, launch argument blocks and the per-M launcher table.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/tpcf.h"

namespace tpcf {

constexpr int TILE = 32;     // pivots per tile: one pivot per lane
constexpr int NWARPS = 8;    // warps per CTA of the tile kernels (map_tile.cuh); they split a tile's neighbour rings
constexpr int NTHREADS = TILE * NWARPS;
constexpr int BW = 4;        // warps per CTA of the block kernels (map_block.cuh), four CTAs per SM
constexpr int BT = TILE * BW;

// Threshold encoding of pair_T entries (see geometry.cu).
constexpr int T_ZERO = -1;          // every pixel of ring r is at or beyond the edge
constexpr int T_INF = 0x7fffffff;   // every pixel of ring r is inside the edge

// Read-only device view of a map plan (kernels take it by value).
struct MapDev {
    int nside, nrings, K, M;
    int64_t npix;
    const int64_t* ring_first;  // [nrings] first pixel of ring
    const int* ring_n;          // [nrings] pixels in ring (always even)
    const int* ring_shift;      // [nrings] pixel p of the ring sits at phi = pi (2p + shift) / n
    const float* ring_zf;       // [nrings] cos(colatitude), fp32
    const float* ring_sf;       // [nrings] sin(colatitude), fp32 (rounded)
    const float* ring_sf_lo;    // [nrings] sin(colatitude) - ring_sf
    const float* ring_step;     // [nrings] pi / n (half longitude step), fp32
    const float* ring_step_lo;  // [nrings] pi / n - ring_step
    const float* ring_invn;     // [nrings] 1 / n, fp32
    const float* ring_invn_lo;  // [nrings] 1 / n - ring_invn
    const double* ring_th;      // [nrings] colatitude, fp64
    const double* ring_s;       // [nrings] sin(colatitude), fp64
    const int2* ring_range;     // [nrings] neighbour rings (rlo, rhi) of pivot ring i
    const int2* bin_range;      // [nrings * K] rings of pivot ring i that may hold bin-k pixels
    const int64_t* pair_off;    // [nrings] first (i, r) pair index of pivot ring i
    const float2* pair_A;       // [npairs] sin(theta_i - theta_r) as fp32 (hi, lo) from fp64
    const int2* pair_T;         // [npairs * (K+1)] edge offsets T_e in ring-r pixels
    const int2* tiles;          // [ntiles] (ring, first pivot index in ring): 32 consecutive pivots
    int64_t ntiles;
    const int2* lin_list;       // linear blocks (ring, first pivot): BT walk_np consecutive pivots (map_block.cuh)
    const int2* orb_list;       // warp tiles (ring, first position) of the other rings: 32 positions and their turned images
    const int* ring_reach;      // [nrings] pixels that a linear tile's rows reach beyond a pivot
    const float4* rc;           // [2 * nrings] (s, s_lo, step, step_lo), (1/n, its lo, 2 n + shift, first)
    const double* E;            // [K+1] sin^2(theta_e / 2)
};

// Read-only device view of a catalogue plan: the points sorted into a sphere grid
// of colatitude bands, each cut into equal longitude sectors (cells).  Points of a
// cell are contiguous, cells are ordered band by band, sectors by longitude.
constexpr int CAT_LUT = 1024;  // entries of the bin lookup table (uniform in the bits of fp32 chord^2)
struct CatDev {
    int64_t n;
    int K, M;
    const float4* p_hi;          // [n] sorted unit vectors, fp32 part (x, y, z, 0)
    const float4* p_lo;          // [n] fp64 - fp32 remainders (x, y, z), w = sorted index bits
    const double* xyz;           // [3n] sorted unit vectors, fp64
    const int64_t* orig;         // [n] caller's index of each sorted point
    const int64_t* cell_start;   // [ncells + 1] first sorted point of each cell
    const int64_t* band_first;   // [nbands + 1] first cell of each band
    const int64_t* band_ns;      // [nbands] sectors in each band
    int nbands;
    double hband;                // band height (rad)
    double theta_max;            // outer bin edge (rad)
    const float* E2;             // [K+1] chord^2 of the edges, fp32
    const double* Ed2;           // [K+1] chord^2 of the edges, fp64
    const unsigned char* lut;    // [CAT_LUT] first edge above each table cell's lower end (cat_edges_kernel)
    int lut_base, lut_shift;     // bits of the table's origin, and their right shift to a cell
    int64_t ntiles;              // ceil(n / TILE)
};

// Per-call arguments of the map kernels.
struct MapCall {
    const float2* wdw;      // [npix] (w * delta, w)
    const float* delta;     // [npix] caller's delta (kernels that read it directly)
    const float* w;         // [npix] caller's weights (idem)
    int64_t piv_lo, piv_hi; // pivot pixel range
    double* slots;          // [grid * nentries] per-CTA fp64 partial sums
    int* counter;           // work counter (zeroed before launch)
    int* status;            // latched device error flags
    const float* H;         // backward: [(M+1) * K * K * 2] fp32, conj(C(k,k')) + C(k',k)
    float* grad;            // backward: [npix]
    int self_subtract;      // subtract the j = k self term
    int flush;              // register sums go on after so many rings (tiles) or 32 entries (blocks); tuned
    int64_t tile_lo, tile_hi;  // tile kernels: tiles that can hold a pivot of [piv_lo, piv_hi)
    int quad;               // tile kernels: tiles in the quarter-turn layout (tile_pivot)
    int norm;               // NORM_*: per-pivot normalisation of the moments before the contraction
    // blocks of the call (map_block.cuh): nlin of lin_list from lin_lo, then norb warp tiles of
    // orb_list from orb_lo, `tiles` to a block; each block in `parts` by bins
    const int2 *lin_list, *orb_list;
    long long lin_lo, nlin, orb_lo, norb;
    int tiles, parts;
    int slices;             // 1, or (tiles = 1) slices of the rings of a bin that go to warps of their own
    int* done;              // parts > 1: [blocks] finished parts (zeroed before launch)
    int step;               // adjoint: phases of this launch (bwd_block)
    float* ws;              // workspace: per block (parts > 1) or per CTA
    size_t ws_floats;       // floats of a block's workspace
    int cells;              // cells listed at a time on linear rings
    int group;              // > 1: shared neighbour lists, one lane per run of `group` ring pixels
    const int2* gtiles;     // tile kernels, group > 1: tiles (ring, first run of the tile)
};

// One plan of a batch (device-resident): its geometry, its per-call arguments and
// the index of its first tile in the batch's concatenated work queue.
// Per-pivot normalisation of the moments (MapCall::norm): none (zeta = S / D), each
// bin by its own weight W^k(i), or every bin by the pivot's total sum_k W^k(i).
constexpr int NORM_NONE = 0;
constexpr int NORM_BIN_MEAN = 1;
constexpr int NORM_PIVOT_TOTAL = 2;
constexpr uint32_t NORM_FLAGS = TPCF_NORM_BIN_MEAN | TPCF_NORM_PIVOT_TOTAL;
inline int norm_of_flags(uint32_t flags) {
    return (flags & TPCF_NORM_BIN_MEAN) ? NORM_BIN_MEAN : ((flags & TPCF_NORM_PIVOT_TOTAL) ? NORM_PIVOT_TOTAL : NORM_NONE);
}

constexpr int TPCF_MAX_BATCH = 256;
struct BatchItem {
    MapDev g;
    MapCall c;
    long long tile0;
};

// Entries of the per-tile partial sums: S for k1 <= k2 (complex), then D (k1 <= k2),
// then, with self-pair subtraction, the two diagonals sum w d Q and sum w QW.
inline __host__ __device__ int n_pairs_tri(int K) { return K * (K + 1) / 2; }
inline __host__ __device__ int n_entries(int K, int M) {
    return 2 * (M + 1) * n_pairs_tri(K) + n_pairs_tri(K) + 2 * K;
}
// Entries of the multi-field partial sums: full K x K matrices, S (complex) per m, then D.
inline __host__ __device__ int n_entries_multi(int K, int M) { return 2 * (M + 1) * K * K + K * K; }

// The tile kernels (map_tile.cuh) that a call can take.
enum TileKernel { TILE_FWD, TILE_GROUPED, TILE_TC, TILE_BWD, TILE_DIRECT };
constexpr int ROW = 512;  // floats per warp row buffer of the tile adjoint (wider rows: whole-ring or global adds)
// Shared memory (floats) of a forward tile with runtime m_max mr: moments A[k][m][re/im][32],
// W, Q, QW [k][32], the pivots' (w d, w).
__host__ __device__ inline size_t tile_floats_rt(int K, int mr) {
    return (size_t)K * (mr + 1) * 2 * TILE + 3 * (size_t)K * TILE + 2 * TILE;
}
// Shared memory (floats) of an adjoint tile: phases 1-2 use the moments, W, Q, QW, the pivots, the
// primary-term sums and one m of H; phase 3 keeps the moments (then h) and the warps' row buffers.
__host__ __device__ inline size_t bwd_tile_floats_rt(int K, int mr) {
    const size_t a = (size_t)K * (mr + 1) * 2 * TILE;
    const size_t p12 = a + 3 * (size_t)K * TILE + 2 * TILE + TILE + (size_t)K * K * 2;
    const size_t p3 = a + (size_t)NWARPS * ROW;
    return p12 > p3 ? p12 : p3;
}

// Pivots per lane of the block kernels (map_block.cuh): 2 bins' sums of M + 1 multipoles each
// take 4 (M + 1) registers.
__host__ __device__ constexpr int walk_np(int M) { return 2; }
// Floats of 32 pivots' moments in the workspace: A[m][k][re/im][32], W[k][32], and Q, QW with
// self-pair subtraction; and of a block's.
__host__ __device__ inline size_t sub_floats_rt(int K, int mr, bool self) {
    return (size_t)K * (mr + 1) * 2 * TILE + (self ? 3 : 1) * (size_t)K * TILE;
}
inline size_t block_floats(int K, int mr, int M, bool self) { return (size_t)BW * walk_np(M) * sub_floats_rt(K, mr, self); }
// Slices of a batch's words that go to warps of their own in pass 2 where there are few bins for the four
// warps; each has a subtile of its own, which cat_tile_moments adds up.  (A bin per warp leaves three of four warps idle at
// one bin.  3,000 points: 131 us at 1 bin, 156 us at 12, against 236 and 334 with 8 warps and atomics.)
__host__ __device__ inline int cat_slices(int K) { return K >= 8 ? 1 : (K >= 4 ? 2 : 4); }
// Calls whose (warp tile, bin) items would leave most warps of the GPU without two: tiles then go one
// to a block and a bin's rings to four warps.
__host__ __device__ inline bool few_tiles(long long norb, int K, int num_sms) {
    return norb * K < (long long)2 * 4 * BW * num_sms;
}
constexpr int LIN_MIN = 256;  // smallest ring that is worth a linear block
constexpr int LIN_CELLS = 1024;       // (bin, ring) cells listed at a time (6 bytes each)
constexpr int LIN_CHUNK = BT;         // entries staged at a time, one per thread
constexpr int LIN_HEAD = 512;         // small tables
// Bytes of moments staged by the contraction: three fields at the most bins, one multipole and W, need
// 3 x 3 x 32 x 32 words.
constexpr int CON_STAGE = 36 * 1024;
static_assert(CON_STAGE >= 3 * 3 * TPCF_MAX_BINS * TILE * 4, "three fields' stage");
// Bytes of a staged entry of the linear walk: two pixel offsets and a weight, then 8 bytes per
// multipole; an odd number of 16-byte words against bank conflicts of the staging stores.
__host__ __device__ constexpr int lin_stride(int M) { return 16 * (((M + 1) / 2 + 1) | 1); }
constexpr int ORB_STRIDE = 80;        // bytes of a staged ring of the other rings' walk (64, odd in 16-byte words)
// Shared memory (bytes) of a block kernel: the linear walk's tables and two chunks, or each warp's
// staged rings, or the contraction's stage with the pivots' values of up to three fields.
__host__ __device__ constexpr size_t block_smem_bytes(int M) {
    const size_t a = LIN_HEAD + (size_t)2 * LIN_CHUNK * lin_stride(M) + (LIN_CELLS + 4) * 4 + LIN_CELLS * 2;
    const size_t b = CON_STAGE + 6 * TILE * 4, c = (size_t)BW * 32 * ORB_STRIDE;
    return a > b ? (a > c ? a : c) : (b > c ? b : c);
}

// The adjoint's phase 3 on linear rings (map_block_bwd.cuh): two chunks of staged entries and the
// cell table, then each warp's rows; phase 2's stage is smaller.
constexpr int ADJ_CHUNK = 64;          // entries staged at a time
constexpr int ADJ_CELLS = 1024;        // cells listed at a time
constexpr int ADJ_ROW_FLOATS = 2048;   // words of a warp's rows
__host__ __device__ constexpr size_t adj_head_bytes(int M) {
    return LIN_HEAD + (size_t)2 * ADJ_CHUNK * lin_stride(M) + (ADJ_CELLS + 4) * 4 + ADJ_CELLS * 2;
}
__host__ __device__ constexpr size_t adj_smem_bytes(int M) {
    const size_t a = adj_head_bytes(M) + (size_t)BW * ADJ_ROW_FLOATS * 4;
    const size_t b = (size_t)4 * TPCF_MAX_BINS * 2 * TILE * 4 + (size_t)TPCF_MAX_BINS * TPCF_MAX_BINS * 8 + 3 * 4 * TILE * 4;
    const size_t c = LIN_HEAD + (size_t)2 * LIN_CHUNK * lin_stride(M) + (LIN_CELLS + 4) * 4 + LIN_CELLS * 2;
    const size_t d = a > b ? a : b;
    return d > c ? d : c;
}

// Device status bits.
constexpr int ST_BAD_TILE = 1;
constexpr int ST_ROW_OVERFLOW = 2;    // informational: a row wider than the warp's buffer used direct global adds
constexpr int ST_TC_TIMEOUT_BIT = 4;  // a tensor-core completion wait gave up

}  // namespace tpcf
