// Moments of a block of pivots, and their contraction.
//
// The pivots of a ring see common position angles, so an angle is worth evaluating once
// for many pivots.  Rings fall in two classes:
//   * linear: all neighbour rings have the ring's own pixel count (the equatorial belt).
//     Every pivot of the ring sees a neighbour at pixel offset t under the same angle, and
//     the pixels at +t and -t are mirror images.  A block is 128 P consecutive pivots, P per
//     lane; the CTA lists the (ring, offset) entries bin by bin, each thread stages the
//     harmonics cos(m phi), sin(m phi) of one entry, and every warp sweeps the staged
//     entries for its own pivots: two pixels and one packed FMA per multipole and entry;
//   * others: every HEALPix ring is invariant under quarter and half turns, so pivots a turn
//     apart see the same neighbours turned.  A warp tile is 32 consecutive positions in the
//     first 1 / NP of a ring, one per lane, with their NP turned images: the lane evaluates an
//     angle and runs the harmonic recurrence once for its images.
//     A block is several warp tiles; its warps draw (tile, bin) items.
// The sums of one bin stay in registers and go to the block's workspace in global memory
// (471 KB per CTA at 20 bins and m_max 10, 286 MB in flight, so through HBM: 12.4 GB in 11.7 ms at Nside 512, a
// sixth of the card's rate): no shared-memory atomics, no barrier per ring or bin.
// Then the CTA stages the workspace 32 pivots at a time and contracts it.  Calls with too little work for
// this split go to map_tile.cuh (takes_blocks in api.cu).
//
// A call with few blocks splits each into parts by bins, so that it still fills the GPU; the
// part that finishes last contracts.
//
// Bound: FP32 and load/store issue.  Per call on a GB300, by tiles (a ring at a time per pivot, sums by
// shared-memory atomics) and by blocks: Nside 512, 20 bins to 2 deg, m <= 10: 33.3 -> 11.8 ms; Nside 4096
// polar slice (2 x 10^-3 of the pixels): 71.9 -> 46.9 ms; Nside 64, 10 bins: 328 -> 217 us.
#pragma once

namespace tpcf {

// Middle pixel of run gi of the shared neighbour lists.
__device__ __forceinline__ int group_middle(int gi, int ng, int group, int n) {
    const int s0 = min(gi, ng - 1) * group;
    return s0 + (min(group, n - s0) - 1) / 2;
}

// (w d, w) of the pivots at ring position x (a pixel, or a run of pixels), zero where the
// call's pivot range or the ring ends.
template <class L>
__device__ __forceinline__ float2 pivot_value(const L& ld, const MapCall& c, long long first, int n, int group, int ng,
                                              int x) {
    float2 v = make_float2(0.0f, 0.0f);
    if (group > 1) {
        if (x < ng) {
            const int s0 = x * group, ln = min(group, n - s0);
            for (int u = 0; u < ln; ++u) {
                const long long pix = first + s0 + u;
                if (pix >= c.piv_lo && pix < c.piv_hi) {
                    const float2 t = ld(pix);
                    v.x += t.x;
                    v.y += t.y;
                }
            }
        }
        return v;
    }
    const long long pix = first + x;
    if (x < n && pix >= c.piv_lo && pix < c.piv_hi) v = ld(pix);
    return v;
}

// A subtile of the workspace: A[m][k][re/im][32], W[k][32], with SELF Q[k][32], QW[k][32].
__device__ __forceinline__ float* sub_a(float* sub, int K, int m, int k) { return sub + (size_t)(m * K + k) * 2 * TILE; }

// Register sums of one bin for a lane's NP pivots: index 0 of a holds (a_0, W).
template <int M, int NP, bool SELF>
struct BinAcc {
    float2 a[NP][M + 1];
    float2 q[SELF ? NP : 1];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int j = 0; j < NP; ++j)
#pragma unroll
            for (int m = 0; m <= M; ++m) a[j][m] = make_float2(0.0f, 0.0f);
        if (SELF)
#pragma unroll
            for (int j = 0; j < NP; ++j) q[j] = make_float2(0.0f, 0.0f);
    }
    // Stores (first) or adds the sums of bin k to the NP subtiles from ws on; every value is
    // only touched by its own thread.  Then zeroes them.
    __device__ __forceinline__ void flush(float* ws, size_t sub_floats, int K, int k, bool first, int mr) {
        const int lane = threadIdx.x & 31;
        float* wk = ws + (size_t)(mr + 1) * K * 2 * TILE + k * TILE + lane;
        auto put = [&](float* p, float v) { __stcg(p, first ? v : __ldcg(p) + v); };
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            float* p = ws + j * sub_floats + k * 2 * TILE + lane;
            put(p, a[j][0].x);
            if (first) __stcg(p + TILE, 0.0f);
            put(wk + j * sub_floats, a[j][0].y);
            if (SELF) {
                put(wk + j * sub_floats + K * TILE, q[j].x);
                put(wk + j * sub_floats + 2 * K * TILE, q[j].y);
            }
#pragma unroll
            for (int m = 1; m <= M; ++m) {
                if (m > mr) break;
                p += (size_t)K * 2 * TILE;
                put(p, a[j][m].x);
                put(p + TILE, a[j][m].y);
            }
        }
        zero();
    }
};

// ------------------------------------------------------------------ linear rings

// Position of bin edge e on a ring, in pixels relative to the pivot's cint: the first
// pixel p at or beyond the edge on the + side (linear rings: the edge cuts every ring).
struct EdgePos {
    bool zero;  // every pixel is at or beyond the edge
    int p;
};

__device__ __forceinline__ EdgePos edge_pos(const LaneC& c, int2 T, const LazyEdge& x) {
    EdgePos e;
    e.zero = T.x == T_ZERO;
    e.p = e.zero ? 0 : pos_edge(c, T, x, 0) - c.cint;
    return e;
}

// Cell of a linear block: pairs at offsets a .. a + n - 1 (offset 0 with no fraction is
// the single pixel on the pivot's meridian).
__device__ __forceinline__ void cell_lin(const EdgePos& lo, const EdgePos& hi, int crem, int& a, int& n) {
    const int none = crem == 0 ? 0 : 1;
    a = lo.zero ? none : lo.p;
    n = max(0, (hi.zero ? none : hi.p) - a);
}

// The ring of an entry from its packed record.
struct WalkRing {
    int n, shift, first;
};

__device__ __forceinline__ WalkRing walk_ring(const MapDev& g, const PivotRing& P, int r, RingCtx& R) {
    const float4 c0 = __ldg(g.rc + 2 * r), c1 = __ldg(g.rc + 2 * r + 1);
    const float2 A = __ldg(g.pair_A + P.pair0 + (r - P.rlo));
    WalkRing w;
    const int ns = __float_as_int(c1.z);
    w.n = ns >> 1;
    w.shift = ns & 1;
    w.first = __float_as_int(c1.w);
    R.s_r = c0.x;
    R.s_lo = c0.y;
    R.step = c0.z;
    R.step_lo = c0.w;
    R.inv_n = c1.x;
    R.invn_lo = c1.y;
    R.A = A.x;
    R.A_lo = A.y;
    R.B = 2.0f * P.z_i * c0.x;
    return w;
}

// The position angle of the entry at offset fi - cfrac, folded (see pixel_dir, fold_angle).
__device__ __forceinline__ float4 entry_angle(const RingCtx& R, int fi, float cfrac) {
    const float ft = (float)fi;
    const float xneg = -cfrac * R.step, uneg = -cfrac * R.inv_n;
    float cph, sph;
    if (fabsf(ft - cfrac) * R.step <= FAST_XMAX)
        pixel_dir<true>(ft, xneg, uneg, R, cph, sph);
    else
        pixel_dir<false>(ft, xneg, uneg, R, cph, sph);
    const Fold f = fold_angle(cph, sph);
    return make_float4(f.ac, f.ss, f.sg, f.lam);
}


// Sweep of staged entries [e0, e1) for the lane's P pivots at ring pixels q[j] (consecutive
// blocks of 32 unless GEN).  WRAP: a row may wrap around the ring.
template <int M, int P, bool SELF, bool WRAP, bool GEN, class L>
__device__ __forceinline__ void lin_sweep(const char* stage, int e0, int e1, const L& ld, int nring, const int (&q)[P],
                                          BinAcc<M, P, SELF>& A, int mr) {
    constexpr int STR = lin_stride(M);
    const char* row = stage + (ptrdiff_t)e0 * STR;
    const char* const last = stage + (ptrdiff_t)(e1 - 1) * STR;
    auto next = [&](const char* r) { return r == last ? r : r + STR; };
    auto head = [&](const char* r) { return *reinterpret_cast<const int4*>(r); };
    auto fetch = [&](const int4& f, float2 (&p)[P], float2 (&m)[P]) {
#pragma unroll
        for (int j = 0; j < P; ++j) {
            int ip, im;
            if (WRAP) {
                ip = wrap_idx(q[j] + f.x, nring) + f.w;
                im = wrap_idx(q[j] + f.y, nring) + f.w;
            } else {
                ip = (GEN ? q[j] : q[0] + 32 * j) + f.x;
                im = (GEN ? q[j] : q[0] + 32 * j) + f.y;
            }
            p[j] = ld(ip);
            m[j] = ld(im);
        }
    };
    // the pixels of the next entry are loaded while this one is summed; its offsets came one
    // entry earlier still
    int4 f0 = head(row);
    const char* row1 = next(row);
    int4 f1 = head(row1);
    float2 p[P], m[P];
    fetch(f0, p, m);
#pragma unroll 2
    for (int e = e0; e < e1; ++e) {
        float2 pn[P], mn[P];
        fetch(f1, pn, mn);
        const char* row2 = next(row1);
        const int4 f2 = head(row2);
        const float h = __int_as_float(f0.z);  // 1/2 for the single pixel on the meridian, which is read twice
        float2 cs[P];
#pragma unroll
        for (int j = 0; j < P; ++j) {
            A.a[j][0] = __ffma2_rn(__fadd2_rn(p[j], m[j]), make_float2(h, h), A.a[j][0]);
            if (SELF)
                A.q[j] = __ffma2_rn(__ffma2_rn(p[j], p[j], __fmul2_rn(m[j], m[j])), make_float2(h, h), A.q[j]);
            cs[j] = make_float2(p[j].x + m[j].x, p[j].x - m[j].x);
        }
        const float4* co = reinterpret_cast<const float4*>(row) + 1;
#pragma unroll
        for (int i = 0; i < (M + 1) / 2; ++i) {
            const int mm = 2 * i + 1;
            if (mm > mr) break;
            const float4 v = co[i];
#pragma unroll
            for (int j = 0; j < P; ++j) A.a[j][mm] = __ffma2_rn(cs[j], make_float2(v.x, v.y), A.a[j][mm]);
            if (mm + 1 <= M) {
                if (mm + 1 > mr) break;
#pragma unroll
                for (int j = 0; j < P; ++j) A.a[j][mm + 1] = __ffma2_rn(cs[j], make_float2(v.z, v.w), A.a[j][mm + 1]);
            }
        }
        row = row1;
        row1 = row2;
        f0 = f1;
        f1 = f2;
#pragma unroll
        for (int j = 0; j < P; ++j) {
            p[j] = pn[j];
            m[j] = mn[j];
        }
    }
}

// Tables of the linear walk in shared memory.
struct LinTables {
    int *rlo, *cum, *ws;  // first ring of a bin; first cell of a bin; warp sums of the scan
    int* pre;             // [cells + 1] entry counts of the cells, then their prefix sums
    short* a0;            // [cells] first offset of a cell's run
    char* stage;          // 2 x chunk entries
    int cells;
};

__device__ __forceinline__ LinTables lin_tables(char* smem, int M, int chunk, int cells) {
    LinTables t;
    t.rlo = reinterpret_cast<int*>(smem);
    t.cum = t.rlo + 32;
    t.ws = t.cum + 40;
    t.stage = smem + LIN_HEAD;
    t.pre = reinterpret_cast<int*>(t.stage + (size_t)2 * chunk * lin_stride(M));
    t.a0 = reinterpret_cast<short*>(t.pre + cells + 4);
    t.cells = cells;
    return t;
}

// Bin ranges of pivot ring i within rings [ra, rb]: rlo[k], cum[k].  Called by warp 0.
__device__ __forceinline__ void bin_cells(const MapDev& g, int i, int K, int ra, int rb, int* rlo, int* cum) {
    const int lane = threadIdx.x & 31;
    int n = 0;
    if (lane < K) {
        const int2 br = g.bin_range[(long long)i * K + lane];
        rlo[lane] = max(br.x, ra);
        n = max(0, min(br.y, rb) - max(br.x, ra) + 1);
    }
    int s = n;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, s, d);
        if (lane >= d) s += v;
    }
    if (lane < K) cum[lane + 1] = s;
    if (lane == 0) cum[0] = 0;
}

// Builds cells [x0, x0 + nx) of the flattened (bin, ring) order and scans their counts.
// Called by every thread (contains barriers, one at the end).
__device__ __forceinline__ void lin_cells(const MapDev& g, const PivotRing& P, const LinTables& t, int ka, int kb, int x0,
                                          int nx) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int K = g.K;
    // a thread takes four bins of one ring, so that an edge serves as the upper end of a
    // bin and the lower end of the next
    const int nkc = (kb - ka + 4) >> 2, rb = t.rlo[kb];
    const int tasks = (t.cum[kb + 1] - t.cum[kb]) * nkc;
    for (int e = tid; e < tasks; e += BT) {
        const int r = rb + e / nkc, k0 = ka + 4 * (e % nkc), k1 = min(k0 + 4, kb + 1);
        const LaneC c = lane_c(0, P.s_i, P.n_i, g.ring_shift[r], P.n_i);
        const int2* T = g.pair_T + (P.pair0 + (r - P.rlo)) * (K + 1);
        EdgePos lo = edge_pos(c, T[k0], LazyEdge{g, P.i, r, k0});
        for (int k = k0; k < k1; ++k) {
            const EdgePos hi = edge_pos(c, T[k + 1], LazyEdge{g, P.i, r, k + 1});
            const int in = r - t.rlo[k], xi = t.cum[k] + in - x0;
            if (in >= 0 && in < t.cum[k + 1] - t.cum[k] && xi >= 0 && xi < nx) {
                int a0, n0;
                cell_lin(lo, hi, c.crem, a0, n0);
                t.pre[xi] = n0;
                t.a0[xi] = (short)a0;
            }
            lo = hi;
        }
    }
    __syncthreads();
    const int per = (nx + BT - 1) / BT;
    const int b = min(nx, tid * per), e = min(nx, b + per);
    int s = 0;
    for (int i = b; i < e; ++i) s += t.pre[i];
    int inc = s;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += v;
    }
    if (lane == 31) t.ws[warp] = inc;
    __syncthreads();
    int base = inc - s;
    for (int w = 0; w < warp; ++w) base += t.ws[w];
    for (int i = b; i < e; ++i) {
        const int v = t.pre[i];
        t.pre[i] = base;
        base += v;
    }
    if (tid == BT - 1) t.pre[nx] = base;
    __syncthreads();
}

// What the offsets of a staged entry are: relative to the ring (the row may wrap: offsets, weight,
// first pixel of the ring), absolute (offsets from the pivot's ring pixel, weight), or relative
// with the number of the ring in the row block (the adjoint's rows).
enum LinHead { HEAD_WRAP, HEAD_ABS, HEAD_ROW };

// Stages one entry per thread: entries [CH c, CH c + CH) of the group's list.
template <int M, int CH>
__device__ __forceinline__ void lin_stage(const MapDev& g, const PivotRing& P, const LinTables& t, int ka, int kb, int x0,
                                          int nx, int total, int c, int head, int ra, int mr) {
    const int ent = c * CH + threadIdx.x;
    if (threadIdx.x >= CH || ent >= total) return;
    int lo = 0, hi = nx - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (t.pre[mid] <= ent) lo = mid; else hi = mid - 1;
    }
    int k = ka;
    while (k < kb && t.cum[k + 1] <= x0 + lo) ++k;
    const int r = t.rlo[k] + x0 + lo - t.cum[k];
    const int fi = t.a0[lo] + (ent - t.pre[lo]);
    RingCtx R;
    const WalkRing w = walk_ring(g, P, r, R);
    const int d = P.s_i - w.shift, dq = d < 0 ? -1 : 0, half = d != 0 ? 1 : 0;
    const float h = half == 0 && fi == 0 ? 0.5f : 1.0f;
    const int rp = dq + fi, rm = dq + half - fi;
    char* row = t.stage + (size_t)((c & 1) * CH + threadIdx.x) * lin_stride(M);
    *reinterpret_cast<int4*>(row) = head == HEAD_ABS ? make_int4(w.first + rp, w.first + rm, __float_as_int(h), 0)
                                                     : make_int4(rp, rm, __float_as_int(h), head == HEAD_ROW ? r - ra : w.first);
    if constexpr (M >= 1) {
        const float4 f = entry_angle(R, fi, half ? 0.5f : 0.0f);
        float4* co = reinterpret_cast<float4*>(row) + 1;
        float2 X = make_float2(h * f.x, h * f.y), D = make_float2(0.5f * f.w * h, h * f.y);
        const float2 L2 = make_float2(f.w, f.w);
        float2 odd = make_float2(f.z * X.x, f.z * X.y);
#pragma unroll
        for (int m = 2; m <= M; ++m) {
            if (m > mr + 1) break;  // (the second of a stored pair may lie one above mr)
            D = __ffma2_rn(L2, X, D);
            X = __fadd2_rn(X, D);
            if (m & 1)
                odd = make_float2(f.z * X.x, f.z * X.y);
            else
                co[m / 2 - 1] = make_float4(odd.x, odd.y, X.x, X.y);
        }
        if constexpr (M & 1) co[M / 2] = make_float4(odd.x, odd.y, 0.0f, 0.0f);
    }
}

// Moments of bins [k0, k1) of a linear block into the warp's P subtiles (ws).  Every thread
// calls it; warps without a live pivot only help to stage.
template <int M, int P, bool SELF, bool GEN, class L>
__device__ __forceinline__ void lin_moments(const MapDev& g, const PivotRing& PR, const int (&q)[P], bool live, int k0,
                                            int k1, const L& ld, float* ws, size_t sub_floats, char* smem, int cells,
                                            int flush, int mr) {
    const LinTables t = lin_tables(smem, M, LIN_CHUNK, cells);
    const int K = g.K;
    const int reach = g.ring_reach[PR.i];
    int qmin = q[0], qmax = q[0];
#pragma unroll
    for (int j = 1; j < P; ++j) {
        qmin = min(qmin, q[j]);
        qmax = max(qmax, q[j]);
    }
    // the staged offsets are relative to the ring or absolute, for the whole CTA
    const bool wrap = __syncthreads_or(qmin - reach < 0 || qmax + reach >= PR.n_i);
    const int head = wrap ? HEAD_WRAP : HEAD_ABS;
    if ((threadIdx.x >> 5) == 0) bin_cells(g, PR.i, K, 0, g.nrings - 1, t.rlo, t.cum);
    __syncthreads();
    const int xb = t.cum[k0], xe = t.cum[k1];
    BinAcc<M, P, SELF> A;
    A.zero();
    int k = k0, done = 0;  // current bin; entries summed in registers
    bool first = true;     // nothing of bin k written yet
    for (int x0 = xb; x0 < xe; x0 += cells) {
        const int nx = min(cells, xe - x0);
        int ka = k0;
        while (t.cum[ka + 1] <= x0) ++ka;
        int kb = ka;
        while (t.cum[kb + 1] < x0 + nx) ++kb;
        lin_cells(g, PR, t, ka, kb, x0, nx);
        const int total = t.pre[nx];
        lin_stage<M, LIN_CHUNK>(g, PR, t, ka, kb, x0, nx, total, 0, head, 0, mr);
        __syncthreads();
        int pos = 0;
        for (int c = 0; c * LIN_CHUNK < total || c == 0; ++c) {
            lin_stage<M, LIN_CHUNK>(g, PR, t, ka, kb, x0, nx, total, c + 1, head, 0, mr);
            if (live) {
                const int cend = min(total, (c + 1) * LIN_CHUNK);
                const char* st = t.stage + (ptrdiff_t)((c & 1) - c) * LIN_CHUNK * lin_stride(M);
                for (;;) {
                    const int xk = t.cum[k + 1] - x0;  // end of bin k in the group's cells
                    const int bend = xk <= nx ? t.pre[xk] : total, e = min(bend, cend);
                    if (e > pos) {
                        if (wrap)
                            lin_sweep<M, P, SELF, true, GEN>(st, pos, e, ld, PR.n_i, q, A, mr);
                        else
                            lin_sweep<M, P, SELF, false, GEN>(st, pos, e, ld, PR.n_i, q, A, mr);
                        done += e - pos;
                        pos = e;
                    }
                    if (pos < bend || xk > nx) break;  // the bin goes on in the next chunk or group
                    A.flush(ws, sub_floats, K, k, first, mr);
                    first = true;
                    done = 0;
                    if (++k == k1) break;
                    if (t.cum[k] - x0 >= nx) break;  // bin k starts in the next group
                }
                if (done >= 32 * flush) {  // blocked summation: short running sums
                    A.flush(ws, sub_floats, K, k, first, mr);
                    first = false;
                    done = 0;
                }
            }
            __syncthreads();
        }
    }
}

// ------------------------------------------------------------------ other rings

// Cursor over the lane's two runs (pixels a0 .. a0 + n0 - 1, then a1 .. a1 + n1 - 1) of a ring and
// their IM images, 1 / IM of the ring apart.  WRAP: some run or image wraps around the ring.
template <int IM, bool WRAP>
struct RunCursor {
    int i0[IM], i1[IM];  // first pixel of each run, the second less the length of the first
    float f0, f1;
    int n0, tot, n, first;
    __device__ __forceinline__ RunCursor(const WalkRing& w, const LaneC& c, const BinRuns& b) {
        n0 = b.n0;
        tot = b.n0 + b.n1;
        n = w.n;
        first = w.first;
        i0[0] = wrap_idx(b.a0, n);
        i1[0] = wrap_idx(b.a1, n);
#pragma unroll
        for (int j = 1; j < IM; ++j) {
            i0[j] = wrap_idx(i0[j - 1] + n / IM, n);
            i1[j] = wrap_idx(i1[j - 1] + n / IM, n);
        }
#pragma unroll
        for (int j = 0; j < IM; ++j) {
            i0[j] += WRAP ? 0 : first;
            i1[j] += (WRAP ? 0 : first) - n0;
        }
        f0 = (float)(b.a0 - c.cint);
        f1 = (float)(b.a1 - c.cint - b.n0);
    }
    __device__ __forceinline__ int pixel(int t, int j) const {
        const int x = (t < n0 ? i0[j] : i1[j]) + t;
        return WRAP ? (x >= n ? x - n : x) + first : x;
    }
    __device__ __forceinline__ float offset(int t) const { return (t < n0 ? f0 : f1) + (float)t; }
};

// Adds one entry (position angle from offset fi) to the sums of the lane's IM images.
template <int M, int IM, bool FAST, bool SELF>
__device__ __forceinline__ void orbit_add(const RingCtx& R, float fi, float xneg, float uneg, const float2 (&v)[IM],
                                          BinAcc<M, IM, SELF>& A, int mr) {
    float cph, sph;
    pixel_dir<FAST>(fi, xneg, uneg, R, cph, sph);
#pragma unroll
    for (int j = 0; j < IM; ++j) {
        A.a[j][0] = __fadd2_rn(A.a[j][0], v[j]);
        if (SELF) A.q[j] = __ffma2_rn(v[j], v[j], A.q[j]);
    }
    if constexpr (M >= 1) {
        if (mr < 1) return;
        const Fold f = fold_angle(cph, sph);
        float2 X = make_float2(f.ac, f.ss), D = make_float2(0.5f * f.lam, f.ss);
        const float2 L2 = make_float2(f.lam, f.lam);
        float o[IM];  // odd multipoles take the fold's sign
#pragma unroll
        for (int j = 0; j < IM; ++j) {
            o[j] = f.sg * v[j].x;
            A.a[j][1] = __ffma2_rn(make_float2(o[j], o[j]), X, A.a[j][1]);
        }
#pragma unroll
        for (int m = 2; m <= M; ++m) {
            if (m > mr) break;
            D = __ffma2_rn(L2, X, D);
            X = __fadd2_rn(X, D);
#pragma unroll
            for (int j = 0; j < IM; ++j) {
                const float u = (m & 1) ? o[j] : v[j].x;
                A.a[j][m] = __ffma2_rn(make_float2(u, u), X, A.a[j][m]);
            }
        }
    }
}

// Walk of the lane's two runs of ring R for its IM images.  Where nothing wraps, the part of
// each run that all lanes have goes without predicates; the rest of both runs together.
template <int M, int IM, bool FAST, bool WRAP, bool SELF, class L>
__device__ __forceinline__ void orbit_runs(const RingCtx& R, const WalkRing& w, const L& ld, const LaneC& c, BinRuns b,
                                           BinAcc<M, IM, SELF>& A, int mr) {
    const float xneg = -c.cfrac * R.step, uneg = -c.cfrac * R.inv_n;
    if (!WRAP) {
#pragma unroll 1
        for (int s = 0; s < 2; ++s) {
            const int a = s ? b.a1 : b.a0, len = __reduce_min_sync(0xffffffffu, s ? b.n1 : b.n0);
            if (len < 2) continue;
            int x0 = wrap_idx(a, w.n);
            float2 v[IM];
            int x[IM];
#pragma unroll
            for (int j = 0; j < IM; ++j) {
                x[j] = x0 + w.first;
                v[j] = ld(x[j]);
                x0 = wrap_idx(x0 + w.n / IM, w.n);
            }
            float fi = (float)(a - c.cint);
#pragma unroll 2
            for (int t = 0; t < len; ++t, fi += 1.0f) {
                float2 vn[IM];  // the next pixels (the one after the last is read and not used)
#pragma unroll
                for (int j = 0; j < IM; ++j) vn[j] = ld(x[j] + t + 1);
                orbit_add<M, IM, FAST, SELF>(R, fi, xneg, uneg, v, A, mr);
#pragma unroll
                for (int j = 0; j < IM; ++j) v[j] = vn[j];
            }
            if (s) {
                b.a1 += len;
                b.n1 -= len;
            } else {
                b.a0 += len;
                b.n0 -= len;
            }
        }
    }
    const int maxt = __reduce_max_sync(0xffffffffu, b.n0 + b.n1);
    const RunCursor<IM, WRAP> cur(w, c, b);
    auto fetch = [&](int t, float2 (&v)[IM]) {
#pragma unroll
        for (int j = 0; j < IM; ++j) v[j] = t < cur.tot ? ld(cur.pixel(t, j)) : make_float2(0.0f, 0.0f);
    };
    float2 v[IM];
    fetch(0, v);
#pragma unroll 1
    for (int t = 0; t < maxt; ++t) {
        float2 vn[IM];
        fetch(t + 1, vn);  // the next pixels, while these are summed
        orbit_add<M, IM, FAST, SELF>(R, cur.offset(t), xneg, uneg, v, A, mr);
#pragma unroll
        for (int j = 0; j < IM; ++j) v[j] = vn[j];
    }
}

// Calls f(R, w, c, runs, fast, flat) for every ring with bin-k pixels, for the lane's pivot at ring
// position q of ring i.  fast: the polynomial covers the runs' offsets; flat: no run or
// image wraps.  The rings' constants are loaded 32 at a time, a ring per lane, and read back
// from the warp's stage in shared memory.
template <int IM, class F>
__device__ __forceinline__ void orbit_rings(const MapDev& g, const PivotRing& P, int q, int k, int sl, int S, char* stage,
                                            F&& f) {
    const int lane = threadIdx.x & 31;
    const int2 all = g.bin_range[(long long)P.i * g.K + k];
    const int nr = all.y - all.x + 1;
    const int2 br = make_int2(all.x + nr * sl / S, all.x + nr * (sl + 1) / S - 1);  // slice sl of S
    for (int r0 = br.x; r0 <= br.y; r0 += 32) {
        __syncwarp();
        bool on = false;
        if (r0 + lane <= br.y) {
            const int r = r0 + lane;
            const int2* T = g.pair_T + (P.pair0 + (r - P.rlo)) * (g.K + 1) + k;
            const int2 Tk = T[0], Tk1 = T[1];
            on = Tk.x != T_INF && Tk1.x != T_ZERO;  // the ring has bin-k pixels
            const float4 c0 = __ldg(g.rc + 2 * r), c1 = __ldg(g.rc + 2 * r + 1);
            const float2 Ap = __ldg(g.pair_A + P.pair0 + (r - P.rlo));
            float4* row = reinterpret_cast<float4*>(stage + lane * ORB_STRIDE);
            row[0] = c0;
            row[1] = c1;
            row[2] = make_float4(Ap.x, Ap.y, 2.0f * P.z_i * c0.x, 0.0f);
            row[3] = make_float4(__int_as_float(Tk.x), __int_as_float(Tk.y), __int_as_float(Tk1.x),
                                 __int_as_float(Tk1.y));
        }
        unsigned todo = __ballot_sync(0xffffffffu, on);
        __syncwarp();
        while (todo) {
            const int u = __ffs(todo) - 1;
            todo &= todo - 1u;
            const float4* row = reinterpret_cast<const float4*>(stage + u * ORB_STRIDE);
            const float4 c0 = row[0], c1 = row[1], c2 = row[2];
            const int4 T = *reinterpret_cast<const int4*>(row + 3);
            RingCtx R;
            R.s_r = c0.x;
            R.s_lo = c0.y;
            R.step = c0.z;
            R.step_lo = c0.w;
            R.inv_n = c1.x;
            R.invn_lo = c1.y;
            R.A = c2.x;
            R.A_lo = c2.y;
            R.B = c2.z;
            WalkRing w;
            w.n = __float_as_int(c1.z) >> 1;
            w.shift = __float_as_int(c1.z) & 1;
            w.first = __float_as_int(c1.w);
            const LaneC c = IM > 1 ? lane_c32(q, P.s_i, P.n_i, w.shift, w.n) : lane_c(q, P.s_i, P.n_i, w.shift, w.n);
            const BinRuns b = bin_runs(c, make_int2(T.x, T.y), make_int2(T.z, T.w), LazyEdge{g, P.i, r0 + u, k}, w.n);
            const float om = fmaxf(run_omax(c, b.a0, b.n0), run_omax(c, b.a1, b.n1));
            // no run leaves its 1 / IM of the ring, so none of its images wraps
            const int span = w.n / IM;
            int y0 = wrap_idx(b.a0, w.n), y1 = wrap_idx(b.a1, w.n);
            if (IM > 1) {
                y0 -= y0 >= span ? span : 0;
                y1 -= y1 >= span ? span : 0;
            }
            const bool flat = y0 + b.n0 <= span && y1 + b.n1 <= span;
            f(R, w, c, b, __all_sync(0xffffffffu, om * R.step <= FAST_XMAX), __all_sync(0xffffffffu, flat));
        }
    }
}

// One (warp tile, bin, slice of the rings) item: the moments of bin k for pivots at ring position
// q of ring i and its turned images, into IM subtiles.
template <int M, int IM, bool SELF, class L>
__device__ __forceinline__ void orbit_bin(const MapDev& g, const PivotRing& P, int q, int k, int sl, int S, const L& ld, float* ws,
                                          size_t sub_floats, char* stage, int flush, int mr) {
    BinAcc<M, IM, SELF> A;
    A.zero();
    bool first = true;
    int done = 0;  // entries summed in registers
    orbit_rings<IM>(g, P, q, k, sl, S, stage, [&](const RingCtx& R, const WalkRing& w, const LaneC& c, const BinRuns& b, bool fast,
                                           bool flat) {
        if (!fast)
            orbit_runs<M, IM, false, true, SELF>(R, w, ld, c, b, A, mr);
        else if (flat)
            orbit_runs<M, IM, true, false, SELF>(R, w, ld, c, b, A, mr);
        else
            orbit_runs<M, IM, true, true, SELF>(R, w, ld, c, b, A, mr);
        done += __reduce_max_sync(0xffffffffu, b.n0 + b.n1);
        if (done >= 32 * flush) {  // blocked summation
            A.flush(ws, sub_floats, g.K, k, first, mr);
            first = false;
            done = 0;
        }
    });
    if (first || done) A.flush(ws, sub_floats, g.K, k, first, mr);
}

// ------------------------------------------------------------------- contraction

// Per-block partial sums into the CTA's FP64 slot (eq. zetamEst2 summed over pivots).  Slot
// layout: for m, for pair (k1 <= k2): (Re S, Im S); then D for pairs; then the self-pair
// diagonals sum_i w_i d_i Q^k(i) and sum_i w_i QW^k(i).
//
// The subtiles are staged one at a time, a group of multipoles at once (all of them at 20
// bins and m_max 10).  A thread takes a 4 x 4 block of bin pairs of one multipole: 17
// shared-memory words feed 64 multiply-adds.  fp32 sums run over two subtiles
// (64 pivots; three fields: over the three products of two), then go through shared memory to the slot, in
// order.
constexpr int CON_RUN = 2;            // subtiles summed in fp32
// Pivots summed at a time before they are added to the run's sum.  The two multiply-adds of a pivot both
// round at the size of the sum, and the weight rounds before them; short first sums keep the error of a slot
// below that of a chain of 32 with the finished products (map_tile.cuh).  Emulated, relative to the sum of
// 128 pivots, for random moments and for moments of one sign: chain 1.07e-7 and 4.4e-8; runs of 64 with
// first sums of 8 9.7e-8 and 3.8e-8 (of 16: 1.15e-7 and 4.2e-8); runs of 128 with first sums of 16,
// as it was, 1.21e-7 and 5.8e-8.
constexpr int CON_FOLD = 8;

// Multipoles staged at once: the groups are of equal size, fit the stage and leave threads for D.
__host__ __device__ inline int con_group(int K, int mr, int slices) {
    const int nb = (K + CB - 1) / CB, nbp = nb * (nb + 1) / 2;
    int g = (CON_STAGE - slices * K * TILE * 4) / (K * 2 * TILE * 4);
    const int h = BT / nbp - 1;
    g = g < h ? g : h;
    g = g < 1 ? 1 : g;
    const int rounds = (mr + 1 + g - 1) / g;
    return (mr + 1 + rounds - 1) / rounds;
}

// Copies n floats (a multiple of 4; 16-byte aligned) from the workspace.
__device__ __forceinline__ void stage_copy(float* dst, const float* src, int n) {
    for (int e = threadIdx.x * 4; e < n; e += BT * 4) {
        const unsigned d = (unsigned)__cvta_generic_to_shared(dst + e);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src + e) : "memory");
    }
}
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Scales the staged moments by 1 / W^k or 1 / sum_k W^k of their pivot (0 where that is 0) and
// sets the staged W to 1 (per-pivot normalisation, Sec. 3.1).  The caller synchronises before.
__device__ __forceinline__ void stage_normalize(int K, int nm, float* sA, float* sW, int norm) {
    constexpr int PER = (TPCF_MAX_BINS * TILE + BT - 1) / BT;
    float inv[PER];
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int e = threadIdx.x + u * BT;
        float W = 0.0f;
        if (e < K * TILE) {
            if (norm == NORM_BIN_MEAN) {
                W = sW[e];
            } else {
                for (int k = 0; k < K; ++k) W += sW[k * TILE + (e & (TILE - 1))];
            }
        }
        inv[u] = W > 0.0f ? 1.0f / W : 0.0f;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int e = threadIdx.x + u * BT;
        if (e < K * TILE) {
            float* a = sA + (size_t)(e / TILE) * 2 * TILE + (e & (TILE - 1));
            for (int m = 0; m < nm; ++m, a += (size_t)K * 2 * TILE) {
                a[0] *= inv[u];
                a[TILE] *= inv[u];
            }
            sW[e] = 1.0f;
        }
    }
    __syncthreads();
}

// smem: CON_STAGE bytes and 2 TILE floats of pivot values.  value(s, lane): (w d, w) of pivot
// `lane` of subtile s.  Called by every thread.
template <bool SELF, class V>
__device__ __forceinline__ void block_contract(int K, int mr, const float* ws, size_t sub_floats, int nsub,
                                               unsigned live, V&& value, char* smem, double* slot, bool self, int norm) {
    float* sA = reinterpret_cast<float*>(smem);
    float* sPiv = reinterpret_cast<float*>(smem + CON_STAGE);
    const int P = n_pairs_tri(K), nS = (mr + 1) * P;
    const int nb = (K + CB - 1) / CB, nbp = nb * (nb + 1) / 2;
    const int tid = threadIdx.x, lane = tid & 31;
    const int slices = SELF ? 3 : 1;
    const int mg = con_group(K, mr, slices);
    for (int m0 = 0; m0 <= mr; m0 += mg) {
        const int nm = min(mg, mr + 1 - m0);
        float* sW = sA + (size_t)nm * K * 2 * TILE;
        const bool withW = m0 == 0 || norm != NORM_NONE;
        // this thread's block: of multipole m0 + ml, or of D (ml = nm), or none
        const int ml = tid / nbp;
        const bool isS = ml < nm, isD = m0 == 0 && ml == nm;
        int b1 = 0, b2 = 0;
        tri_block(tid - ml * nbp, b1, b2);
        int o1[CB], o2[CB];  // offsets of the rows; bins past the last one repeat it and are not written
#pragma unroll
        for (int i = 0; i < CB; ++i) {
            const int k1 = min(CB * b1 + i, K - 1), k2 = min(CB * b2 + i, K - 1);
            o1[i] = isD ? nm * K * 2 * TILE + k1 * TILE : (ml * K + k1) * 2 * TILE;
            o2[i] = isD ? nm * K * 2 * TILE + k2 * TILE : (ml * K + k2) * 2 * TILE;
        }
        float2 tot[CB][CB], acc[CB][CB];
#pragma unroll
        for (int i = 0; i < CB; ++i)
#pragma unroll
            for (int j = 0; j < CB; ++j) tot[i][j] = make_float2(0.0f, 0.0f);
        int run = 0;
        for (int s = 0; s < nsub; ++s) {
            if ((live >> s) & 1u) {
                const float* sub = ws + (size_t)s * sub_floats;
                stage_copy(sA, sub + (size_t)m0 * K * 2 * TILE, nm * K * 2 * TILE);
                if (withW) stage_copy(sW, sub + (size_t)(mr + 1) * K * 2 * TILE, slices * K * TILE);
                if (tid < TILE) {
                    const float2 v = value(s, lane);
                    sPiv[lane] = v.x;
                    sPiv[TILE + lane] = v.y;
                }
                stage_wait();
                __syncthreads();
                if (norm != NORM_NONE) stage_normalize(K, nm, sA, sW, norm);
#pragma unroll 1
                for (int t0 = 0; t0 < TILE; t0 += CON_FOLD) {
#pragma unroll
                    for (int i = 0; i < CB; ++i)
#pragma unroll
                        for (int j = 0; j < CB; ++j) acc[i][j] = make_float2(0.0f, 0.0f);
                    if (isS) {
#pragma unroll 2
                        for (int t = t0; t < t0 + CON_FOLD; ++t) {
                            const int l = (t + lane) & (TILE - 1);  // a warp's 32 reads of a word hit 32 banks
                            const float w = sPiv[l];
                            float2 x[CB], y[CB];
#pragma unroll
                            for (int i = 0; i < CB; ++i) {
                                x[i] = make_float2(w * sA[o1[i] + l], w * sA[o1[i] + TILE + l]);
                                y[i] = make_float2(sA[o2[i] + l], sA[o2[i] + TILE + l]);
                            }
#pragma unroll
                            for (int j = 0; j < CB; ++j) {
                                const float2 z = make_float2(y[j].y, -y[j].x);
#pragma unroll
                                for (int i = 0; i < CB; ++i)  // (a c + b d, a d - b c)
                                    acc[i][j] = __ffma2_rn(make_float2(x[i].x, x[i].x), y[j],
                                                           __ffma2_rn(make_float2(x[i].y, x[i].y), z, acc[i][j]));
                            }
                        }
                    } else if (isD) {
                        for (int t = t0; t < t0 + CON_FOLD; ++t) {
                            const int l = (t + lane) & (TILE - 1);
                            const float w = sPiv[TILE + l];
#pragma unroll
                            for (int i = 0; i < CB; ++i)
#pragma unroll
                                for (int j = 0; j < CB; ++j)
                                    acc[i][j].x = fmaf(w, sA[o1[i] + l] * sA[o2[j] + l], acc[i][j].x);
                        }
                    }
#pragma unroll
                    for (int i = 0; i < CB; ++i)
#pragma unroll
                        for (int j = 0; j < CB; ++j) tot[i][j] = __fadd2_rn(tot[i][j], acc[i][j]);
                }
                if (SELF && self && m0 == 0 && tid < K) {
                    const float* Q = sW + (K + tid) * TILE;
                    float q1 = 0.0f, q2 = 0.0f;
                    for (int t = 0; t < TILE; ++t) {
                        const int l = (t + lane) & (TILE - 1);
                        q1 = fmaf(sPiv[l], Q[l], q1);
                        q2 = fmaf(sPiv[TILE + l], Q[K * TILE + l], q2);
                    }
                    red_add_f32(slot + 2 * nS + P + tid, q1);
                    red_add_f32(slot + 2 * nS + P + K + tid, q2);
                }
                ++run;
            }
            __syncthreads();  // the stage is free again
            if (run == CON_RUN || (s == nsub - 1 && run)) {
                run = 0;
                // through shared memory, so that the reductions to the slot are in order
                float* out = sA;
                if (isS || isD) {
                    const int base = isD ? 2 * nm * P : 2 * ml * P;
#pragma unroll
                    for (int i = 0; i < CB; ++i)
#pragma unroll
                        for (int j = 0; j < CB; ++j) {
                            const int k1 = CB * b1 + i, k2 = CB * b2 + j, pi = k2 * (k2 + 1) / 2 + k1;
                            if (k1 <= k2 && k2 < K) {
                                if (isD) {
                                    out[base + pi] = tot[i][j].x;
                                } else {
                                    out[base + 2 * pi] = tot[i][j].x;
                                    out[base + 2 * pi + 1] = tot[i][j].y;
                                }
                            }
                            tot[i][j] = make_float2(0.0f, 0.0f);
                        }
                }
                __syncthreads();
                for (int e = tid; e < 2 * nm * P; e += BT) red_add_f32(slot + 2 * m0 * P + e, out[e]);
                if (m0 == 0)
                    for (int e = tid; e < P; e += BT) red_add_f32(slot + 2 * nS + e, out[2 * nm * P + e]);
                __syncthreads();
            }
        }
    }
}

// Contraction of three fields (tpcf_forward_multi), the same way: the cyclic sums over
// (P, X, Y) of (A, B, C) into full K x K matrices (slot: for m, for (k1, k2): (Re S, Im S); then
// D).  field_ws: floats between the fields' workspaces; value(f, s, lane): pivots of field f.
__host__ __device__ inline int con_group_multi(int K, int mr) {
    const int nb = (K + CB - 1) / CB;
    int g = (CON_STAGE - 3 * K * TILE * 4) / (3 * K * 2 * TILE * 4);
    const int h = BT / (nb * nb) - 1;
    g = g < h ? g : h;
    g = g < 1 ? 1 : g;
    const int rounds = (mr + 1 + g - 1) / g;
    return (mr + 1 + rounds - 1) / rounds;
}

template <class V>
__device__ __forceinline__ void block_contract_multi(int K, int mr, const float* ws, size_t field_ws, size_t sub_floats,
                                                     int nsub, unsigned live, V&& value, char* smem, double* slot) {
    float* sA = reinterpret_cast<float*>(smem);
    float* sPiv = reinterpret_cast<float*>(smem + CON_STAGE);  // [field][w d, w][32]
    const int KK = K * K, nS = (mr + 1) * KK;
    const int nb = (K + CB - 1) / CB, nbp = nb * nb;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int mg = con_group_multi(K, mr);
    for (int m0 = 0; m0 <= mr; m0 += mg) {
        const int nm = min(mg, mr + 1 - m0);
        const int fstr = nm * K * 2 * TILE + K * TILE;  // floats of a field's staged part
        const int ml = tid / nbp;
        const bool isS = ml < nm, isD = m0 == 0 && ml == nm;
        const int b1 = (tid - ml * nbp) / nb, b2 = (tid - ml * nbp) % nb;
        int o1[CB], o2[CB];
#pragma unroll
        for (int i = 0; i < CB; ++i) {
            const int k1 = min(CB * b1 + i, K - 1), k2 = min(CB * b2 + i, K - 1);
            o1[i] = isD ? nm * K * 2 * TILE + k1 * TILE : (ml * K + k1) * 2 * TILE;
            o2[i] = isD ? nm * K * 2 * TILE + k2 * TILE : (ml * K + k2) * 2 * TILE;
        }
        float2 tot[CB][CB], acc[CB][CB];
#pragma unroll
        for (int i = 0; i < CB; ++i)
#pragma unroll
            for (int j = 0; j < CB; ++j) tot[i][j] = make_float2(0.0f, 0.0f);
        int run = 0;
        for (int s = 0; s < nsub; ++s) {
            if ((live >> s) & 1u) {
                for (int f = 0; f < 3; ++f) {
                    const float* sub = ws + f * field_ws + (size_t)s * sub_floats;
                    stage_copy(sA + f * fstr, sub + (size_t)m0 * K * 2 * TILE, nm * K * 2 * TILE);
                    stage_copy(sA + f * fstr + nm * K * 2 * TILE, sub + (size_t)(mr + 1) * K * 2 * TILE, K * TILE);
                }
                if (warp < 3) {
                    const float2 v = value(warp, s, lane);
                    sPiv[warp * 2 * TILE + lane] = v.x;
                    sPiv[warp * 2 * TILE + TILE + lane] = v.y;
                }
                stage_wait();
                __syncthreads();
#pragma unroll 1
                for (int cyc = 0; cyc < 3; ++cyc) {  // (P, X, Y) = (cyc, cyc + 1, cyc + 2)
                    const float* X = sA + ((cyc + 1) % 3) * fstr;
                    const float* Y = sA + ((cyc + 2) % 3) * fstr;
                    const float* pv = sPiv + cyc * 2 * TILE + (isD ? TILE : 0);
#pragma unroll 1
                    for (int t0 = 0; t0 < TILE; t0 += CON_FOLD) {
#pragma unroll
                        for (int i = 0; i < CB; ++i)
#pragma unroll
                            for (int j = 0; j < CB; ++j) acc[i][j] = make_float2(0.0f, 0.0f);
                        if (isS) {
#pragma unroll 2
                            for (int t = t0; t < t0 + CON_FOLD; ++t) {
                                const int l = (t + lane) & (TILE - 1);
                                const float w = pv[l];
                                float2 x[CB], y[CB];
#pragma unroll
                                for (int i = 0; i < CB; ++i) {
                                    x[i] = make_float2(w * X[o1[i] + l], w * X[o1[i] + TILE + l]);
                                    y[i] = make_float2(Y[o2[i] + l], Y[o2[i] + TILE + l]);
                                }
#pragma unroll
                                for (int j = 0; j < CB; ++j) {
                                    const float2 z = make_float2(y[j].y, -y[j].x);
#pragma unroll
                                    for (int i = 0; i < CB; ++i)
                                        acc[i][j] = __ffma2_rn(make_float2(x[i].x, x[i].x), y[j],
                                                               __ffma2_rn(make_float2(x[i].y, x[i].y), z, acc[i][j]));
                                }
                            }
                        } else if (isD) {
                            for (int t = t0; t < t0 + CON_FOLD; ++t) {
                                const int l = (t + lane) & (TILE - 1);
#pragma unroll
                                for (int i = 0; i < CB; ++i)
#pragma unroll
                                    for (int j = 0; j < CB; ++j)
                                        acc[i][j].x = fmaf(pv[l], X[o1[i] + l] * Y[o2[j] + l], acc[i][j].x);
                            }
                        }
#pragma unroll
                        for (int i = 0; i < CB; ++i)
#pragma unroll
                            for (int j = 0; j < CB; ++j) tot[i][j] = __fadd2_rn(tot[i][j], acc[i][j]);
                    }
                }
                ++run;
            }
            __syncthreads();
            if (run == CON_RUN || (s == nsub - 1 && run)) {
                run = 0;
                float* out = sA;
                if (isS || isD) {
#pragma unroll
                    for (int i = 0; i < CB; ++i)
#pragma unroll
                        for (int j = 0; j < CB; ++j) {
                            const int k1 = CB * b1 + i, k2 = CB * b2 + j;
                            if (k1 < K && k2 < K) {
                                if (isD) {
                                    out[2 * nm * KK + k1 * K + k2] = tot[i][j].x;
                                } else {
                                    out[2 * (ml * KK + k1 * K + k2)] = tot[i][j].x;
                                    out[2 * (ml * KK + k1 * K + k2) + 1] = tot[i][j].y;
                                }
                            }
                            tot[i][j] = make_float2(0.0f, 0.0f);
                        }
                }
                __syncthreads();
                for (int e = tid; e < 2 * nm * KK; e += BT) red_add_f32(slot + 2 * m0 * KK + e, out[e]);
                if (m0 == 0)
                    for (int e = tid; e < KK; e += BT) red_add_f32(slot + 2 * nS + e, out[2 * nm * KK + e]);
                __syncthreads();
            }
        }
    }
}

// ------------------------------------------------------------------------ blocks

// First bin of part s of S: parts of about equal area (E = sin^2(theta / 2) is linear in it).
__device__ __forceinline__ int part_bin(const double* E, int K, int s, int S) {
    if (s <= 0) return 0;
    if (s >= S) return K;
    const double want = E[0] + (E[K] - E[0]) * s / S;
    int k = 0;
    while (k < K && E[k] < want) ++k;
    if (k > 0 && want - E[k - 1] < E[k] - want) --k;
    return k;
}

// Block b of a call: one linear block, or T consecutive warp tiles.
template <int M, bool GROUPED>
struct Block {
    static constexpr int NP = walk_np(M), IM = GROUPED ? 1 : NP;
    bool lin;
    const int2* list;
    int T, nsub;  // warp tiles; subtiles
    __device__ __forceinline__ Block(const MapDev& g, const MapCall& c, long long b) {
        lin = b < c.nlin;
        list = lin ? c.lin_list + c.lin_lo + b : c.orb_list + c.orb_lo + (b - c.nlin) * c.tiles;
        T = lin ? 1 : (int)min((long long)c.tiles, c.norb - (b - c.nlin) * c.tiles);
        nsub = lin ? BW * NP : T * IM;
    }
    // pixel of pivot `l` of subtile s (one of the ring's)
    __device__ __forceinline__ long long pixel(const MapDev& g, int s, int l) const {
        const int2 tq = list[lin ? 0 : s / IM];
        return g.ring_first[tq.x] + (lin ? tq.y + s * TILE + l : tq.y + l + (s % IM) * (g.ring_n[tq.x] / IM));
    }
    // (w d, w) of pivot `l` of subtile s
    template <class L>
    __device__ __forceinline__ float2 value(const MapDev& g, const MapCall& c, const L& ld, int s, int l) const {
        const int2 tq = list[lin ? 0 : s / IM];
        const int n = g.ring_n[tq.x], group = GROUPED ? c.group : 1;
        int x = tq.y + (lin ? s * TILE : 0) + l;
        if (!lin && !GROUPED) x = x < n / IM ? x + (s % IM) * (n / IM) : n;
        return pivot_value(ld, c, g.ring_first[tq.x], n, group, (n + group - 1) / group, x);
    }
};

// Bit per subtile with a live pivot.  Called by every thread.
template <class F>
__device__ __forceinline__ unsigned block_live(int nsub, F&& on) {
    __shared__ unsigned s_live;
    if (threadIdx.x == 0) s_live = 0u;
    __syncthreads();
    for (int s = threadIdx.x >> 5; s < nsub; s += BW)
        if (__any_sync(0xffffffffu, on(s, threadIdx.x & 31)) && (threadIdx.x & 31) == 0) atomicOr(&s_live, 1u << s);
    __syncthreads();
    const unsigned live = s_live;
    __syncthreads();
    return live;
}

// Moments of bins [kb, ke) of a linear block's live subtiles into its workspace.  Called by every
// thread; complete after the caller's barrier.
template <int M, bool SELF, bool GROUPED, class L>
__device__ __forceinline__ void lin_block_moments(const MapDev& g, const MapCall& c, long long b, unsigned live, int kb,
                                               int ke, L ld, float* ws, size_t sub_floats, char* smem, int mr) {
    constexpr int NP = Block<M, GROUPED>::NP;
    const Block<M, GROUPED> B(g, c, b);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int group = GROUPED ? c.group : 1;
    const int2 tq = *B.list;
    const PivotRing PR = pivot_ring(g, tq.x);
    const int ng = (PR.n_i + group - 1) / group;
    auto pos = [&](int x) { return GROUPED ? group_middle(x, ng, group, PR.n_i) : min(x, PR.n_i - 1); };
    int q[NP];
    bool whole = !GROUPED;  // the lane's pivots are 32 pixels apart (not at a ring's ragged end)
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        q[j] = pos(tq.y + (warp * NP + j) * TILE + lane);
        whole = whole && q[j] == q[0] + 32 * j;
    }
    const bool on = ((live >> (warp * NP)) & ((1u << NP) - 1u)) != 0u;
    float* w = ws + (size_t)warp * NP * sub_floats;
    if (!GROUPED && __syncthreads_and(whole))
        lin_moments<M, NP, SELF, false>(g, PR, q, on, kb, ke, ld, w, sub_floats, smem, c.cells, c.flush, mr);
    else
        lin_moments<M, NP, SELF, true>(g, PR, q, on, kb, ke, ld, w, sub_floats, smem, c.cells, c.flush, mr);
}

// The same for the warp tiles of another block: its warps draw (tile, bin, slice) items; slice s has
// subtiles of its own, which block_fold adds up.
template <int M, bool SELF, bool GROUPED, class L>
__device__ __forceinline__ void orb_block_moments(const MapDev& g, const MapCall& c, long long b, unsigned live, int kb,
                                               int ke, L ld, float* ws, size_t sub_floats, char* smem, int mr) {
    constexpr int IM = Block<M, GROUPED>::IM;
    __shared__ int s_item;
    const Block<M, GROUPED> B(g, c, b);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int group = GROUPED ? c.group : 1;
    if (threadIdx.x == 0) s_item = 0;
    __syncthreads();
    const int S = c.slices, items = B.T * (ke - kb) * S;
    for (;;) {
        int it = 0;
        if (lane == 0) it = atomicAdd(&s_item, 1);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= items) break;
        const int sl = it % S, u = it / S;
        const int t = u % B.T, k = ke - 1 - u / B.T;  // outer (larger) bins first
        if (((live >> (t * IM)) & ((1u << IM) - 1u)) == 0u) continue;
        const int2 tq = B.list[t];
        const PivotRing PR = pivot_ring(g, tq.x);
        const int q = GROUPED ? group_middle(tq.y + lane, (PR.n_i + group - 1) / group, group, PR.n_i)
                              : min(tq.y + lane, PR.n_i / IM - 1);
        orbit_bin<M, IM, SELF>(g, PR, q, k, sl, S, ld, ws + (size_t)(sl * B.T + t) * IM * sub_floats, sub_floats,
                               smem + warp * 32 * ORB_STRIDE, c.flush, mr);
    }
}

template <int M, bool SELF, bool GROUPED, class L>
__device__ __forceinline__ void block_moments(const MapDev& g, const MapCall& c, long long b, unsigned live, int part,
                                              const L& ld, float* ws, size_t sub_floats, char* smem, int mr) {
    const int kb = part_bin(g.E, g.K, part, c.parts), ke = part_bin(g.E, g.K, part + 1, c.parts);
    if (b < c.nlin)
        lin_block_moments<M, SELF, GROUPED, L>(g, c, b, live, kb, ke, ld, ws, sub_floats, smem, mr);
    else
        orb_block_moments<M, SELF, GROUPED, L>(g, c, b, live, kb, ke, ld, ws, sub_floats, smem, mr);
}

template <int M, bool SELF, bool GROUPED, class L>
__device__ __forceinline__ void block_sums(const MapDev& g, const MapCall& c, long long b, unsigned live, L ld,
                                        const float* ws, size_t sub_floats, char* smem, double* slot, int mr) {
    const Block<M, GROUPED> B(g, c, b);
    block_contract<SELF>(g.K, mr, ws, sub_floats, B.nsub, live,
                         [&](int s, int l) { return B.value(g, c, ld, s, l); }, smem, slot, SELF && c.self_subtract,
                         c.norm);
}

// Adds the slices' subtiles of a block into the first slice's.  Called by every thread, between the
// barrier of block_complete and the contraction.
__device__ __forceinline__ void block_fold(const MapCall& c, long long b, int nsub, float* ws, size_t sub_floats) {
    if (c.slices == 1 || b < c.nlin) return;
    const int n = (int)(nsub * sub_floats / 4);  // (sub_floats is a multiple of 32)
    float4* w = reinterpret_cast<float4*>(ws);
    for (int e = threadIdx.x; e < n; e += BT) {
        float4 v = __ldcg(w + e);
        for (int s = 1; s < c.slices; ++s) {
            const float4 u = __ldcg(w + s * n + e);
            v = make_float4(v.x + u.x, v.y + u.y, v.z + u.z, v.w + u.w);
        }
        __stcg(w + e, v);
    }
    __syncthreads();
}

// True on the CTA that finishes the last part of block b.  Called by every thread.
__device__ __forceinline__ bool block_complete(const MapCall& c, long long b) {
    if (c.parts == 1) {
        __syncthreads();
        return true;
    }
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(c.done + b, 1) == c.parts - 1;
    __syncthreads();
    const bool last = s_last != 0;
    if (last) __threadfence();
    __syncthreads();
    return last;
}

// One work item of a forward: part `part` of block `b`; the block's last part contracts it into the
// slot.  Called by every thread of the CTA.
template <int M, bool SELF, bool GROUPED, class L>
__device__ __forceinline__ void fwd_block(const MapDev& g, const MapCall& c, long long b, int part, const L& ld,
                                          float* ws, double* slot, char* smem, int mr) {
    const Block<M, GROUPED> B(g, c, b);
    const size_t sub_floats = sub_floats_rt(g.K, mr, SELF);
    const unsigned live = block_live(B.nsub, [&](int s, int l) { return B.value(g, c, ld, s, l).y != 0.0f; });
    if (live == 0u) return;
    block_moments<M, SELF, GROUPED>(g, c, b, live, part, ld, ws, sub_floats, smem, mr);
    if (!block_complete(c, b)) return;
    block_fold(c, b, B.nsub, ws, sub_floats);
    block_sums<M, SELF, GROUPED, L>(g, c, b, live, ld, ws, sub_floats, smem, slot, mr);
    __syncthreads();
}

}  // namespace tpcf
