// Catalogue kernels: the estimator of Sec. 3.1 (eqs. Xm.binned, zetamEst) for points at
// arbitrary positions, found through the plan's sphere grid.
//
// A tile is 32 consecutive points of the grid order (spatially compact), one pivot
// per lane.  Warp 0 bounds the tile's live pivots by a cap (centre, radius R); every
// point within R + theta_max of the centre lies in the cells the cap overlaps, which
// are a handful of contiguous index ranges per colatitude band.  The CTA stages those of these
// candidates that are close enough to the centre, up to 512 at a time, as fp32 hi/lo offsets
// from it, and makes two passes:
//   1. a warp takes 32 candidates (a word) and bins each for its 32 pivots, from one broadcast
//      read and a table over the bits of chord^2.  Bin k of pivot `lane` is one bit in the word's
//      mask [k][lane];
//   2. a warp takes a bin: each lane goes through the candidates in its own masks of that bin, so
//      every lane's sums stay in registers for the whole batch and go to the CTA's workspace in
//      global memory once per bin and batch, without atomics.
// Pass 2 has no bin decision and pass 1 no angle; neither diverges but for the lanes' different
// numbers of candidates in a bin.  Candidates whose chord^2 is too close to an edge for the table
// go a slower way (cat_near_edge), down to FP64 within CAT_AMB of the edge.  The contraction of a
// tile is that of the map blocks (block_contract).
// Bound: instruction issue.  Before (chunks of 32 candidates, shared-memory atomics) and now: 8 x 10^6
// points, 16 bins, m <= 10: 457 -> 200 ms; 5 x 10^4 points with gradient: 2.03 -> 0.58 ms.
#pragma once

#include "map_kernels.cuh"

namespace tpcf {

constexpr float CAT_AMB = 2.0e-6f;  // relative margin of fp32 chord^2 to an edge (error ~3e-7)
constexpr float CAT_MARGIN = 8.0e-6f;  // angular margin of the fp32 cell query (rad)
constexpr float CAT_FAR = 1.0e3f;      // where lanes and slots that are not in use are placed

// Bin of chord^2 in fp64 over the edges (ties to the upper bin) for sorted points j
// (candidate) and si (pivot): -1 below the first edge, K at or beyond the last.
static __device__ __noinline__ int cat_exact_bin(const double* __restrict__ Ed2, int K, const double* __restrict__ xyz,
                                          int64_t j, int64_t si) {
    const double dx = xyz[3 * j] - xyz[3 * si], dy = xyz[3 * j + 1] - xyz[3 * si + 1],
                 dz = xyz[3 * j + 2] - xyz[3 * si + 2];
    const double c2 = dx * dx + dy * dy + dz * dz;
    int k = -1;
    while (k < K && c2 >= Ed2[k + 1]) ++k;
    return k;
}

// The bin of a candidate near an edge, or where the table's cells hold several edges: from
// chord^2 to full fp32 precision (c2), in FP64 within CAT_AMB of an edge.
static __device__ __noinline__ int cat_near_edge(const CatDev& g, float c2, int64_t j, int64_t si) {
    int k = -1;
    bool near = false;
    for (int e = 0; e <= g.K; ++e) {
        const float E = __ldg(g.E2 + e);
        k += c2 >= E ? 1 : 0;
        near = near || fabsf(c2 - E) <= CAT_AMB * E;
    }
    return near && si >= 0 ? cat_exact_bin(g.Ed2, g.K, g.xyz, j, si) : k;
}

// The lane's pivot: fp32 hi/lo position (of the unit vector; cat_place moves it to the cap's
// centre), local north / east basis and its sorted index (the FP64 position is read only for
// the rare exact bin decisions).
struct CatPivot {
    float hx, hy, hz, lx, ly, lz;
    float nx, ny, nz, ex, ey;
    int64_t si;
};

// si < 0: a padding lane, placed at (0, 0, 1).
__device__ __forceinline__ CatPivot cat_pivot(const CatDev& g, int64_t si) {
    CatPivot P;
    P.si = si;
    float4 h = make_float4(0.0f, 0.0f, 1.0f, 0.0f), l = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (si >= 0) {
        h = g.p_hi[si];
        l = g.p_lo[si];
    }
    P.hx = h.x;
    P.hy = h.y;
    P.hz = h.z;
    P.lx = l.x;
    P.ly = l.y;
    P.lz = l.z;
    // the basis in fp32 (its rounding is a fixed rotation of the pivot's frame, which
    // cancels in a conj(a), plus ~1e-7 of non-orthogonality)
    const float s2 = fmaf(P.hx, P.hx, P.hy * P.hy);
    if (s2 > 1e-12f) {
        const float is = rsqrtf(s2);
        P.ex = -P.hy * is;  // east = z x n / |z x n|
        P.ey = P.hx * is;
        P.nx = -P.hz * P.hx * is;  // north = n x east
        P.ny = -P.hz * P.hy * is;
        P.nz = s2 * is;
    } else {  // on the axis: any tangent basis of the same handedness
        P.ex = 0.0f;
        P.ey = 1.0f;
        P.nx = -P.hz;
        P.ny = 0.0f;
        P.nz = 0.0f;
    }
    return P;
}

// Warp 0: a cap holding every live pivot of the tile together with its neighbours
// (radius theta_max), as a range of cell bands and a longitude half-width about the
// cap's centre: s_cap = (phi_c, dphi, first band, last band, full, centre x, y, z).  All in fp32:
// CAT_MARGIN (rad) exceeds every rounding of the centre, radius, colatitude and band
// division (each below ~1e-6 rad), and the sine ratio is rounded up, so the cells are
// a superset of the exact cap; bins are then decided per candidate.  The caller
// synchronises afterwards.
__device__ __forceinline__ void cat_tile_cap(const CatDev& g, bool live, const CatPivot& P, float* s_cap) {
    const float px = P.hx + P.lx, py = P.hy + P.ly, pz = P.hz + P.lz;
    float sx = live ? px : 0.0f, sy = live ? py : 0.0f, sz = live ? pz : 0.0f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sx += __shfl_xor_sync(0xffffffffu, sx, o);
        sy += __shfl_xor_sync(0xffffffffu, sy, o);
        sz += __shfl_xor_sync(0xffffffffu, sz, o);
    }
    float nrm = sqrtf(fmaf(sx, sx, fmaf(sy, sy, sz * sz)));
    if (!(nrm > 1e-6f)) {  // live pivots cancel out: any centre will do (r is measured from it)
        sx = 0.0f;
        sy = 0.0f;
        sz = 1.0f;
        nrm = 1.0f;
    }
    const float cx = sx / nrm, cy = sy / nrm, cz = sz / nrm;
    float r = 0.0f;
    if (live) {
        const float dx = px - cx, dy = py - cy, dz = pz - cz;
        const float ch = sqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
        r = 2.0f * asinf(fminf(1.0f, 0.5f * ch));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r = fmaxf(r, __shfl_xor_sync(0xffffffffu, r, o));
    if ((threadIdx.x & 31) == 0) {
        const float PI_F = 3.14159265f;
        const float Q = r + (float)g.theta_max + CAT_MARGIN;
        const float thc = atan2f(sqrtf(fmaf(cx, cx, cy * cy)), cz);
        float phc = atan2f(cy, cx);
        if (phc < 0.0f) phc += 2.0f * PI_F;
        int b0 = 0, b1 = g.nbands - 1;
        float full = 1.0f, dphi = PI_F;
        const float lo = thc - Q - CAT_MARGIN, hi = thc + Q + CAT_MARGIN;
        if (Q < PI_F) {
            const float hb = (float)g.hband;
            b0 = max(0, (int)floorf(lo / hb));
            b1 = min(g.nbands - 1, (int)floorf(hi / hb));
            if (lo > 0.0f && hi < PI_F) {  // no pole inside: then Q < pi / 2, sin rises with Q
                // sin is concave on [0, pi]: its least value over thc +- margin is at an end
                const float st = fminf(sinf(thc - CAT_MARGIN), sinf(thc + CAT_MARGIN));
                const float x = sinf(Q) / st * (1.0f + 1.0e-6f);
                if (x < 1.0f) {
                    full = 0.0f;
                    dphi = asinf(x) + CAT_MARGIN;
                }
            }
        }
        s_cap[0] = phc;
        s_cap[1] = dphi;
        s_cap[2] = (float)b0;
        s_cap[3] = (float)b1;
        s_cap[4] = full;
        s_cap[5] = cx;
        s_cap[6] = cy;
        s_cap[7] = cz;
    }
}

// Coordinate h + l relative to c, again as hi/lo (Knuth's two-sum: no digit of the pair is lost).
__device__ __forceinline__ void cat_rel(float h, float l, float c, float& H, float& L) {
    const float s = h - c, b = s - h;
    const float t = ((h - (s - b)) + (-c - b)) + l;
    H = s + t;
    L = t - (H - s);
}

// Shared memory of a catalogue CTA.  The union is the candidates and their masks, the
// contraction's stage, or the adjoint's phase 2.
struct CatShared {
    unsigned char* lut;  // [CAT_LUT] next edge above a cell of chord^2 (see cat_edges_kernel)
    float2* edge;        // [K + 3] chord^2 of the edge, margin below which cat_near_edge decides
    float* cap;          // [9]: cat_tile_cap, then the largest chord from the cap's centre to a live pivot
    int* item;           // next bin of the batch
    int* cnt;            // [BW] candidates staged by a warp
    int* wsum;           // [BW]
    int* pre;            // [2 BT + 1] candidates before a cell range of the band group
    int* start;          // [2 BT] first candidate of the range
    char* stage;         // the union
    int words;           // words of 32 candidates a warp stages at a time; BW words of them in all
    float4 *hi, *lo;     // [32 BW words] offset from the cap's centre and w d; its remainder and w
    int* idx;            // [32 BW words] sorted index
    unsigned* mask;      // [K + 1][BW words][32]; row K takes the candidates outside the bins
    float* leg;          // [32 BW words] adjoint only: sums of the legs to a candidate
};

constexpr size_t CAT_HEAD = CAT_LUT + 8 * 40 + 4 * 16 + 4 * 16 + 4 * (4 * BT + 16);

// Words a warp stages at a time: as many as leave room for four CTAs on an SM (57,000 bytes each), at
// most 4.  More candidates to a batch mean fewer trips of the sums to the workspace and lanes
// with more equal numbers of candidates in a bin.
__host__ __device__ inline size_t cat_word_bytes(int K, bool legs) {
    return BW * (32 * (2 * sizeof(float4) + (legs ? 2 : 1) * sizeof(int)) + (size_t)(K + 1) * TILE * 4);
}
__host__ __device__ inline int cat_words(int K, bool legs) {
    const int w = (int)((57000 - CAT_HEAD) / cat_word_bytes(K, legs));
    return w > 4 ? 4 : w;
}
__host__ __device__ inline size_t cat_smem_bytes(int K, bool legs, size_t other) {
    const size_t b = cat_words(K, legs) * cat_word_bytes(K, legs);
    return CAT_HEAD + (b > other ? b : other);
}
// forward (6 TILE floats of pivot values, as for three fields), adjoint
template <int M>
__host__ __device__ inline size_t cat_fwd_bytes(int K) {
    return cat_smem_bytes(K, false, CON_STAGE + 6 * TILE * sizeof(float));
}
template <int M>
__host__ __device__ inline size_t cat_bwd_bytes(int K) { return cat_smem_bytes(K, true, adj_smem_bytes(M)); }

__device__ __forceinline__ CatShared cat_shared(char* smem, int K, bool legs) {
    CatShared S;
    S.lut = reinterpret_cast<unsigned char*>(smem);
    S.edge = reinterpret_cast<float2*>(smem + CAT_LUT);
    S.cap = reinterpret_cast<float*>(S.edge + 40);
    S.item = reinterpret_cast<int*>(S.cap + 16);
    S.cnt = S.item + 4;
    S.wsum = S.item + 8;
    S.pre = S.item + 16;
    S.start = S.pre + 2 * BT + 16;
    S.stage = smem + CAT_HEAD;
    S.words = cat_words(K, legs);
    const int n = BW * 32 * S.words;
    S.hi = reinterpret_cast<float4*>(S.stage);
    S.lo = S.hi + n;
    S.idx = reinterpret_cast<int*>(S.lo + n);
    S.mask = reinterpret_cast<unsigned*>(S.idx + n);
    S.leg = reinterpret_cast<float*>(S.mask + (K + 1) * n);
    return S;
}

__device__ __forceinline__ void cat_load_lut(const CatDev& g, const CatShared& S) {
    for (int e = threadIdx.x; e < CAT_LUT / 4; e += BT)
        reinterpret_cast<unsigned*>(S.lut)[e] = __ldg(reinterpret_cast<const unsigned*>(g.lut) + e);
}

// (w d, w) of pivot `lane` of a tile; zero outside the call's pivot range and where w = 0.
__device__ __forceinline__ float2 cat_value(const CatDev& g, const float2* __restrict__ wdw, int64_t lo, int64_t hi,
                                            int64_t tile, int lane) {
    const int64_t si = tile * TILE + lane;
    float2 v = make_float2(0.0f, 0.0f);
    if (si < g.n) {
        const int64_t o = g.orig[si];
        if (o >= lo && o < hi) v = wdw[si];
    }
    return v.y != 0.0f ? v : make_float2(0.0f, 0.0f);
}

// Prepares a tile: its cap, the margins of the edges and the lane's pivot relative to the cap's
// centre; lanes that are not live are moved away from every candidate.  Called by every thread.
//
// Pass 1 uses the offsets' fp32 high parts alone.  With p, q the offsets of pivot and candidate,
// each rounded to 2^-24 of itself, and d = q - p, |q| <= |d| + |p|: chord^2 is off by at most
// 2^-24 (7 d^2 + 8 |d| |p|), a quarter of the margin 2e-6 (E + rho sqrt(E)) at an edge.  A
// table cell only knows the one edge within a cell's width, so margins stay below that width (2^(shift - 24)
// of E at least); where a wide tile's margin at small edges is larger, cat_near_edge decides the candidates
// nearer than these.  (When it decided all candidates of such a tile, 5 x 10^5 clustered points with bins from
// 0.001 to 1 degree took 14.0 ms, now 3.6; chunks of candidates with a bin search each took 6.5.)
__device__ __forceinline__ CatPivot cat_place(const CatDev& g, const CatShared& S, int64_t tile, bool live) {
    const int lane = threadIdx.x & 31;
    const int64_t si = tile * TILE + lane;
    CatPivot P = cat_pivot(g, si < g.n ? si : -1);
    if ((threadIdx.x >> 5) == 0) cat_tile_cap(g, live, P, S.cap);
    __syncthreads();
    cat_rel(P.hx, P.lx, S.cap[5], P.hx, P.lx);
    cat_rel(P.hy, P.ly, S.cap[6], P.hy, P.ly);
    cat_rel(P.hz, P.lz, S.cap[7], P.hz, P.lz);
    if ((threadIdx.x >> 5) == 0) {
        // from the offsets, which are good to 2^-24 of themselves: the unit vectors' fp32 parts
        // are off by 6e-8, which is more than the relative margins of cat_batches where theta_max is small
        float d2 = live ? fmaf(P.hx, P.hx, fmaf(P.hy, P.hy, P.hz * P.hz)) : 0.0f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) d2 = fmaxf(d2, __shfl_xor_sync(0xffffffffu, d2, o));
        const float rho = sqrtf(d2) * (1.0f + 1.0e-6f);
        if (lane == 0) S.cap[8] = rho;
        const float cell = exp2f((float)(g.lut_shift - 24)) * 0.99f;
        float lim = 0.0f;  // chord^2 up to which an edge's margin reaches beyond a cell's width
        for (int e = lane; e < g.K + 3; e += 32) {
            const float E = e <= g.K ? g.E2[e] : 0.0f;
            const float amb = 2.0e-6f * fmaf(rho, sqrtf(E), E);
            if (amb > cell * E) lim = fmaxf(lim, E + amb);
            S.edge[e] = e <= g.K ? make_float2(E, amb)
                                 : (e == g.K + 1 ? make_float2(INFINITY, 0.0f) : make_float2(0.0f, INFINITY));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) lim = fmaxf(lim, __shfl_xor_sync(0xffffffffu, lim, o));
        // the next edge above such a chord^2 is edge e at most where edge e - 1 lies below lim
        if (lim > 0.0f)
            for (int e = lane; e < g.K + 2; e += 32)
                if (e == 0 || g.E2[e - 1] < lim) S.edge[e].y = INFINITY;
    }
    __syncthreads();
    if (!live) {
        P.hx = CAT_FAR;
        P.si = -1;
    }
    return P;
}

// The candidates of the cap, staged a batch at a time: batch(first) for each, between barriers; at
// least once.  A candidate is kept if it can be in a bin of a live pivot, all of which are within
// rho of the centre.  Each warp fills words of its own (the order of a sum stays the same from run
// to run), the rest of its last word with points far away; S.cnt says how many.  Called by every thread.
template <class F>
__device__ __forceinline__ void cat_batches(const CatDev& g, const float2* __restrict__ wdw, const CatShared& S,
                                            F&& batch) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // sector bounds in fp32: the extra 4e-6 rad covers its rounding (phi < 2 pi), so the
    // cell ranges stay a superset of the cap
    const float phc = S.cap[0], dphi = S.cap[1] + 4.0e-6f;
    const int b0 = (int)S.cap[2], b1 = (int)S.cap[3];
    const bool full = S.cap[4] != 0.0f;
    const float rho = S.cap[8], rlo = sqrtf(__ldg(g.E2)), rhi = sqrtf(__ldg(g.E2 + g.K));
    const float far = (rhi + rho) * (1.0f + 1.0e-5f), nearby = fmaxf(rlo - rho - 1.0e-5f * (rlo + rho), 0.0f);
    const float far2 = far * far, near2 = nearby * nearby;
    bool first = true;
    int c = 0;  // candidates staged by this warp
    const int w0 = 32 * S.words * warp, cap = 32 * S.words;
    for (int bg = b0; bg <= b1; bg += BT) {
        // a band per thread: at most two cell ranges (the sector range may wrap around phi = 0)
        int64_t pa0 = 0, pa1 = 0, pb0 = 0, pb1 = 0;
        if (bg + tid <= b1) {
            const int64_t ns = g.band_ns[bg + tid], cf = g.band_first[bg + tid];
            int64_t ca0 = cf, ca1 = cf + ns, cb1 = cf;
            if (!full) {
                const float scale = (float)ns * (float)(0.5 / M_PI);
                const int64_t sa = (int64_t)floorf((phc - dphi) * scale);
                const int64_t sb = (int64_t)floorf((phc + dphi) * scale);
                const int64_t len = sb - sa + 1;
                if (len < ns) {
                    int64_t s0 = sa % ns;
                    if (s0 < 0) s0 += ns;
                    ca0 = cf + s0;
                    if (s0 + len <= ns) {
                        ca1 = ca0 + len;
                    } else {
                        cb1 = cf + (s0 + len - ns);
                    }
                }
            }
            pa0 = g.cell_start[ca0];
            pa1 = g.cell_start[ca1];
            if (cb1 > cf) {
                pb0 = g.cell_start[cf];
                pb1 = g.cell_start[cb1];
            }
        }
        const int na = (int)(pa1 - pa0), s = na + (int)(pb1 - pb0);
        int inc = s;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, d);
            if (lane >= d) inc += v;
        }
        if (lane == 31) S.wsum[warp] = inc;
        __syncthreads();
        int base = inc - s;
        for (int w = 0; w < warp; ++w) base += S.wsum[w];
        S.pre[2 * tid] = base;
        S.pre[2 * tid + 1] = base + na;
        S.start[2 * tid] = (int)pa0;
        S.start[2 * tid + 1] = (int)pb0;
        if (tid == BT - 1) S.pre[2 * BT] = base + s;
        __syncthreads();
        const int total = S.pre[2 * BT];
        const bool last = bg + BT > b1;
        for (int x = 32 * warp;;) {
            for (; x < total && c <= cap - 32; x += BT) {
                const int e = x + lane;
                bool keep = false;
                float4 H, L;
                int j = 0;
                if (e < total) {
                    int lo = 0, hi = 2 * BT - 1;  // the last range that starts at or before e
                    while (lo < hi) {
                        const int mid = (lo + hi + 1) >> 1;
                        if (S.pre[mid] <= e) lo = mid; else hi = mid - 1;
                    }
                    j = S.start[lo] + (e - S.pre[lo]);
                    const float4 h = g.p_hi[j], l = g.p_lo[j];
                    const float2 v = wdw[j];
                    cat_rel(h.x, l.x, S.cap[5], H.x, L.x);
                    cat_rel(h.y, l.y, S.cap[6], H.y, L.y);
                    cat_rel(h.z, l.z, S.cap[7], H.z, L.z);
                    H.w = v.x;
                    L.w = v.y;
                    const float d2 = fmaf(H.x, H.x, fmaf(H.y, H.y, H.z * H.z));
                    keep = d2 <= far2 && d2 >= near2;
                }
                const unsigned kept = __ballot_sync(0xffffffffu, keep);
                if (keep) {
                    const int at = w0 + c + __popc(kept & ((1u << lane) - 1u));
                    S.hi[at] = H;
                    S.lo[at] = L;
                    S.idx[at] = j;
                }
                c += __popc(kept);
            }
            const bool more = __syncthreads_or(x < total) != 0;
            if (!more && !last) break;  // the next group of bands fills up
            // (a warp without a candidate fills its first word: lanes of pass 2 that have none read slot 0,
            // which must hold numbers)
            if (lane < (c ? (32 - c) & 31 : 32)) {
                S.hi[w0 + c + lane] = make_float4(-CAT_FAR, 0.0f, 0.0f, 0.0f);
                S.lo[w0 + c + lane] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            }
            if (lane == 0) S.cnt[warp] = c;
            if (tid == 0) *S.item = 0;
            __syncwarp();
            batch(first);
            __syncthreads();
            first = false;
            c = 0;
            if (!more) break;
        }
    }
}

// Pass 1 for J of the warp's words at once, from word w on: a candidate of each, so that their chains of
// loads and the updates of their masks, which are in different words, overlap.
template <int J>
__device__ __forceinline__ void cat_bin_words(const CatDev& g, const CatShared& S, const CatPivot& P, int w) {
    const int lane = threadIdx.x & 31;
    const int base = g.lut_base, shift = g.lut_shift, row = BW * S.words * TILE;
    unsigned* mw = S.mask + w * TILE + lane;
    const float4* q = S.hi + w * 32;
#pragma unroll 1
    for (int u = 0; u < 32; ++u) {
        float3 d[J];
        float c2[J], x[J], amb[J];
        int k[J];
        bool near = false;
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const float4 qh = q[j * 32 + u];
            d[j] = make_float3(qh.x - P.hx, qh.y - P.hy, qh.z - P.hz);
            c2[j] = fmaf(d[j].x, d[j].x, fmaf(d[j].y, d[j].y, d[j].z * d[j].z));
            k[j] = S.lut[min((max(__float_as_int(c2[j]), base) - base) >> shift, CAT_LUT - 1)];
        }
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const float2 e = S.edge[k[j]];
            x[j] = c2[j] - e.x;
            amb[j] = e.y;
            if (x[j] < 0.0f) --k[j];
            near = near || fabsf(x[j]) <= amb[j];
        }
        if (near) {
#pragma unroll
            for (int j = 0; j < J; ++j)
                if (fabsf(x[j]) <= amb[j]) {
                    const int at = (w + j) * 32 + u;
                    const float4 ql = S.lo[at];
                    const float ex = d[j].x + (ql.x - P.lx), ey = d[j].y + (ql.y - P.ly), ez = d[j].z + (ql.z - P.lz);
                    k[j] = cat_near_edge(g, fmaf(ex, ex, fmaf(ey, ey, ez * ez)), S.idx[at], P.si);
                }
        }
        unsigned m[J];
#pragma unroll
        for (int j = 0; j < J; ++j) {
            k[j] = (int)min((unsigned)k[j], (unsigned)g.K) * row + j * TILE;
            m[j] = mw[k[j]];
        }
#pragma unroll
        for (int j = 0; j < J; ++j) mw[k[j]] = m[j] | (1u << u);
    }
}

// Pass 1 of a batch: the masks of the warp's own candidates.  The masks are zero on entry.
__device__ __forceinline__ void cat_bins(const CatDev& g, const CatShared& S, const CatPivot& P) {
    const int warp = threadIdx.x >> 5;
    int w = S.words * warp;
    const int we = w + ((S.cnt[warp] + 31) >> 5);
    for (; w + 3 < we; w += 4) cat_bin_words<4>(g, S, P, w);
    for (; w + 1 < we; w += 2) cat_bin_words<2>(g, S, P, w);
    if (w < we) cat_bin_words<1>(g, S, P, w);
}

// Position angle of a candidate: the lane's pivot sees the offset (hi, lo) under this folded angle.
__device__ __forceinline__ Fold cat_angle(const CatPivot& P, const float4& qh, const float4& ql) {
    const float dx = (qh.x - P.hx) + (ql.x - P.lx);
    const float dy = (qh.y - P.hy) + (ql.y - P.ly);
    const float dz = (qh.z - P.hz) + (ql.z - P.lz);
    const float N = fmaf(dx, P.nx, fmaf(dy, P.ny, dz * P.nz));
    const float E = fmaf(dx, P.ex, dy * P.ey);
    const float rinv = rsqrtf(fmaxf(fmaf(N, N, E * E), 1e-30f));
    return fold_angle(N * rinv, E * rinv);
}

// Pass 2 over bin k and slice sl of a batch: f(on, u, hi, lo) for each candidate u of the lane (on false
// where other lanes have more), two at a time.  Leaves the bin's masks zero.
template <class FB, class F>
__device__ __forceinline__ void cat_bin_pairs(const CatShared& S, int k, int sl, int slices, FB&& begin, F&& f) {
    const int lane = threadIdx.x & 31, nw = BW * S.words / slices, base0 = sl * nw * 32;
    unsigned* mk = S.mask + ((size_t)k * BW * S.words + sl * nw) * TILE + lane;
    unsigned words = 0u;
    int cnt = 0;
#pragma unroll 4
    for (int w = 0; w < nw; ++w) {  // (words that were not filled are zero)
        const unsigned m = mk[w * TILE];
        cnt += __popc(m);
        words |= (m != 0u ? 1u : 0u) << w;
    }
    const int most = __reduce_max_sync(0xffffffffu, cnt);
    if (!begin(most)) return;
    unsigned m = 0u;
    int base = base0;
    auto next = [&]() {  // the lane's next candidate, or some candidate
        if (m == 0u && words != 0u) {
            const int w = __ffs(words) - 1;
            words &= words - 1u;
            m = mk[w * TILE];
            mk[w * TILE] = 0u;
            base = base0 + w * 32;
        }
        const int u = base + max(__ffs(m) - 1, 0);
        m &= m - 1u;
        return u;
    };
#pragma unroll 1
    for (int i = 0; i < most; i += 2) {
        const int u0 = next(), u1 = next();
        const float4 h0 = S.hi[u0], l0 = S.lo[u0], h1 = S.hi[u1], l1 = S.lo[u1];
        f(i < cnt, u0, h0, l0);
        f(i + 1 < cnt, u1, h1, l1);
    }
}

__device__ __forceinline__ int cat_next_bin(const CatShared& S) {
    int k = 0;
    if ((threadIdx.x & 31) == 0) k = atomicAdd(S.item, 1);
    return __shfl_sync(0xffffffffu, k, 0);
}

__device__ __forceinline__ void cat_zero_masks(const CatShared& S, int K) {
    for (int e = threadIdx.x; e < K * BW * S.words * TILE; e += BT) S.mask[e] = 0u;
}

// The moments of a tile with the neighbour values `wdw`, into its subtile of the workspace.
// Called by every thread; complete after the caller's barrier.
template <int M, bool SELF>
__device__ __forceinline__ void cat_tile_moments(const CatDev& g, const float2* __restrict__ wdw, const CatShared& S,
                                                 const CatPivot& P, float* ws, size_t sub_floats) {
    const int K = g.K;
    const int slices = cat_slices(K);
    cat_zero_masks(S, K);  // the union held other things
    cat_batches(g, wdw, S, [&](bool first) {
        cat_bins(g, S, P);
        __syncthreads();
        BinAcc<M, 1, SELF> A;
        A.zero();
        for (int it = cat_next_bin(S); it < K * slices; it = cat_next_bin(S)) {
            const int k = it / slices, sl = it - k * slices;
            bool any = false;
            cat_bin_pairs(
                S, k, sl, slices,
                [&](int most) {
                    any = most > 0;
                    return any;
                },
                [&](bool on, int, const float4& qh, const float4& ql) {
                    const float wd = on ? qh.w : 0.0f, w = on ? ql.w : 0.0f;
                    harmonicsf<M>(A.a[0], cat_angle(P, qh, ql), wd, wd);
                    A.a[0][0].y += w;
                    if (SELF) A.q[0] = __ffma2_rn(make_float2(wd, w), make_float2(wd, w), A.q[0]);
                });
            if (any || first) A.flush(ws + sl * sub_floats, sub_floats, K, k, first, M);
        }
    });
    if (slices > 1) {  // (cat_batches ends with a barrier)
        const int n = (int)(sub_floats / 4);
        float4* w = reinterpret_cast<float4*>(ws);
        for (int e = threadIdx.x; e < n; e += BT) {
            float4 v = __ldcg(w + e);
            for (int s = 1; s < slices; ++s) {
                const float4 u = __ldcg(w + s * n + e);
                v = make_float4(v.x + u.x, v.y + u.y, v.z + u.z, v.w + u.w);
            }
            __stcg(w + e, v);
        }
        __syncthreads();
    }
}

// Forward: persistent CTAs draw tiles.
template <int M, bool SELF>
__global__ void __launch_bounds__(BT, 4) cat_fwd_kernel(CatDev g, MapCall c) {
    extern __shared__ __align__(16) float smem[];
    __shared__ int s_tile;
    const CatShared S = cat_shared(reinterpret_cast<char*>(smem), g.K, false);
    const int lane = threadIdx.x & 31;
    const size_t sub_floats = sub_floats_rt(g.K, M, SELF);
    float* ws = c.ws + (size_t)blockIdx.x * c.ws_floats;
    double* slot = c.slots + (size_t)blockIdx.x * n_entries(g.K, M);
    cat_load_lut(g, S);
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(c.counter, 1);
        __syncthreads();
        const int64_t tile = s_tile;
        if (tile >= g.ntiles) break;
        const bool live = cat_value(g, c.wdw, c.piv_lo, c.piv_hi, tile, lane).y != 0.0f;
        if (!__syncthreads_or(live)) continue;
        const CatPivot P = cat_place(g, S, tile, live);
        cat_tile_moments<M, SELF>(g, c.wdw, S, P, ws, sub_floats);
        block_contract<SELF>(
            g.K, M, ws, sub_floats, 1, 1u,
            [&](int, int l) { return cat_value(g, c.wdw, c.piv_lo, c.piv_hi, tile, l); }, S.stage, slot, SELF, c.norm);
        __syncthreads();
    }
}

// Multi-field forward on a catalogue (tpcf_forward_multi): three fields on the same
// points, each with its own weights.  The tile's candidates are gone through once per field (the
// moments of the neighbour fields A, B, C), and block_contract_multi forms the cyclic
// sum over the pivot field.
template <int M>
__global__ void __launch_bounds__(BT, 4) cat_fwd_multi_kernel(CatDev g, MapCall c, const float2* __restrict__ wdwB,
                                                              const float2* __restrict__ wdwC) {
    extern __shared__ __align__(16) float smem[];
    __shared__ int s_tile;
    const CatShared S = cat_shared(reinterpret_cast<char*>(smem), g.K, false);
    const int lane = threadIdx.x & 31;
    const size_t sub_floats = sub_floats_rt(g.K, M, false), field_ws = c.ws_floats / 3;
    float* ws = c.ws + (size_t)blockIdx.x * c.ws_floats;
    double* slot = c.slots + (size_t)blockIdx.x * n_entries_multi(g.K, M);
    const float2* arr[3] = {c.wdw, wdwB, wdwC};
    cat_load_lut(g, S);
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(c.counter, 1);
        __syncthreads();
        const int64_t tile = s_tile;
        if (tile >= g.ntiles) break;
        bool live = false;
#pragma unroll
        for (int f = 0; f < 3; ++f)
            live = live || cat_value(g, arr[f], c.piv_lo, c.piv_hi, tile, lane).y != 0.0f;
        if (!__syncthreads_or(live)) continue;
        const CatPivot P = cat_place(g, S, tile, live);
#pragma unroll 1
        for (int f = 0; f < 3; ++f) cat_tile_moments<M, false>(g, arr[f], S, P, ws + f * field_ws, sub_floats);
        block_contract_multi(
            g.K, M, ws, field_ws, sub_floats, 1, 1u,
            [&](int f, int, int l) { return cat_value(g, arr[f], c.piv_lo, c.piv_hi, tile, l); }, S.stage, slot);
        __syncthreads();
    }
}

// Catalogue adjoint, dL/d(delta_p) (the map adjoint's three phases on the catalogue
// walk): phase 1 recomputes the tile's moments, phase 2 (block_h) forms w d H conj(a) in place
// and the primary term, phase 3 goes through the batches again and adds
// w_j w_i d_i sum_m (cos(m phi) Re h_m^k + sin(m phi) Im h_m^k) for every in-bin pair;
// the 32 pivots' contributions to a candidate are summed in shared memory before one
// atomic add to its gradient.
template <int M>
__global__ void __launch_bounds__(BT, 4) cat_bwd_kernel(CatDev g, MapCall c) {
    extern __shared__ __align__(16) float smem[];
    __shared__ int s_tile;
    const int K = g.K;
    const CatShared S = cat_shared(reinterpret_cast<char*>(smem), K, true);
    const int lane = threadIdx.x & 31, slices = cat_slices(K);
    const size_t sub_floats = sub_floats_rt(K, M, false);
    float* ws = c.ws + (size_t)blockIdx.x * c.ws_floats;
    cat_load_lut(g, S);
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(c.counter, 1);
        __syncthreads();
        const int64_t tile = s_tile;
        if (tile >= g.ntiles) break;
        const bool live = cat_value(g, c.wdw, c.piv_lo, c.piv_hi, tile, lane).y != 0.0f;
        if (!__syncthreads_or(live)) continue;
        const CatPivot P = cat_place(g, S, tile, live);
        cat_tile_moments<M, false>(g, c.wdw, S, P, ws, sub_floats);
        block_h<M, false>(
            c, K, M, ws, sub_floats, 1, 1u,
            [&](int s, int l) {
                return s == 0 ? cat_value(g, c.wdw, c.piv_lo, c.piv_hi, tile, l) : make_float2(0.0f, 0.0f);
            },
            [&](int, int l) { return g.orig[tile * TILE + l]; }, S.stage);
        __syncthreads();
        cat_zero_masks(S, K);
        for (int e = threadIdx.x; e < 32 * BW * S.words; e += BT) S.leg[e] = 0.0f;
        cat_batches(g, c.wdw, S, [&](bool) {
            cat_bins(g, S, P);
            __syncthreads();
            for (int it = cat_next_bin(S); it < K * slices; it = cat_next_bin(S)) {
                const int k = it / slices, sl = it - k * slices;
                float2 h[1][M + 1];
                cat_bin_pairs(
                    S, k, sl, slices,
                    [&](int most) {
                        if (most > 0) load_h<M, 1>(h, ws, sub_floats, K, k, 1u, M);
                        return most > 0;
                    },
                    [&](bool on, int u, const float4& qh, const float4& ql) {
                        float X, Y;
                        adj_harmonicsf<M>(h[0], cat_angle(P, qh, ql), X, Y);
                        if (on) atomicAdd(S.leg + u, X + Y);
                    });
            }
            __syncthreads();
            for (int e = threadIdx.x; e < 32 * BW * S.words; e += BT) {
                if (e % (32 * S.words) >= S.cnt[e / (32 * S.words)]) continue;
                const float v = S.lo[e].w * S.leg[e];
                S.leg[e] = 0.0f;
                if (v != 0.0f) atomicAdd(c.grad + g.orig[S.idx[e]], v);
            }
        });
        __syncthreads();
    }
}

#if defined(TPCF_M) && TPCF_M == 0  // one definition, in the M = 0 object
// Exact number of in-bin ordered pairs (i, j) with w_i != 0 and caller index of i in
// [lo, hi): counts[0] += total.  Same tiles and candidates as the forward.
__global__ void __launch_bounds__(BT) cat_count_kernel(CatDev g, const float2* __restrict__ wdw, long long lo,
                                                       long long hi, int* counter, unsigned long long* counts) {
    extern __shared__ __align__(16) float smem[];
    __shared__ int s_tile;
    const CatShared S = cat_shared(reinterpret_cast<char*>(smem), g.K, false);
    const int lane = threadIdx.x & 31;
    cat_load_lut(g, S);
    cat_zero_masks(S, g.K);
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(counter, 1);
        __syncthreads();
        const int64_t tile = s_tile;
        if (tile >= g.ntiles) break;
        const bool live = cat_value(g, wdw, lo, hi, tile, lane).y != 0.0f;
        if (!__syncthreads_or(live)) continue;
        const CatPivot P = cat_place(g, S, tile, live);
        unsigned long long cnt = 0;
        cat_batches(g, wdw, S, [&](bool) {
            cat_bins(g, S, P);
            __syncthreads();
            for (int e = threadIdx.x; e < g.K * BW * S.words * TILE; e += BT) {
                cnt += __popc(S.mask[e]);  // lanes that are not live are in no bin
                S.mask[e] = 0u;
            }
        });
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
        if (lane == 0 && cnt) atomicAdd(counts, cnt);
        __syncthreads();
    }
}
#endif

}  // namespace tpcf
