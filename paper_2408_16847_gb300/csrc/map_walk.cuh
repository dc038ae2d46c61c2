// Tile moments from shared position angles.
//
// A tile's 32 pivots are chosen so that they see the same position angles:
//   * "linear" tiles, on rings all of whose neighbour rings have the same pixel count
//     (the equatorial belt): 32 consecutive pivots.  Every pivot of the ring has the
//     same fractional offset to a neighbour ring, so a neighbour at pixel offset t has
//     the same angle for all of them, and the pixels at +t and -t are mirror images;
//   * "orbit" tiles, on the other rings: four orbits of eight pivots each under the
//     map's quarter turns and the reflection phi -> -phi (every HEALPix ring is
//     invariant under both).  The eight pivots of an orbit see images of the same
//     neighbours: the same angle, or minus it.
// The neighbours of a tile (per orbit) are listed bin by bin: a cell is (bin, ring), its
// entries are the ring's in-bin pixels (pixel pairs on linear tiles).  The cells of a
// group of bins are built by the whole CTA, their entry counts scanned, and the steps
// (one entry per orbit) split evenly over the warps, whatever rings or bins they
// fall in.  A warp takes 32 entries at a time: each lane evaluates the angle of one entry
// and puts it and the pixel indices into the warp's stage in shared memory; then the warp
// sweeps the staged entries.  Half a warp takes the even steps, half the odd ones, each lane
// carrying two pivots: it runs the harmonic recurrence once for the two.
#pragma once

namespace tpcf {

// Pivot t (0..31) of a tile of ring (n, s).  Linear: pixel start + t.  Orbits: u = start +
// (t & 3), turned by (t >> 2) & 3 quarters, reflected if t >= 16; the reflected image of a
// pivot on a symmetry meridian is one of its turns and is left out.  Pixels past the end
// are not valid and take the geometry of the last one.
struct TileSlot {
    int q;
    bool valid;
};

__host__ __device__ __forceinline__ int orbit_count(int n, int s) {
    const int quarter = n >> 2;
    return s ? (quarter + 1) >> 1 : (quarter >> 1) + 1;
}

__host__ __device__ __forceinline__ TileSlot tile_slot(bool lin, int n, int s, int start, int t) {
    TileSlot o;
    if (lin) {
        o.valid = start + t < n;
        o.q = o.valid ? start + t : n - 1;
        return o;
    }
    const int quarter = n >> 2, norb = orbit_count(n, s);
    int u = start + (t & 3);
    o.valid = u < norb;
    u = o.valid ? u : norb - 1;
    const int turn = ((t >> 2) & 3) * quarter;
    if (t < 16) {
        o.q = u + turn;
    } else {
        o.valid = o.valid && (2 * u + s) % quarter != 0;
        o.q = n - u - s + turn;
        if (o.q >= n) o.q -= n;
    }
    return o;
}

// Pixel in ring of the unturned, unreflected pivot of orbit slot o (0..3) of an orbit tile.
__host__ __device__ __forceinline__ int tile_orbit(int n, int s, int start, int o) {
    const int u = start + o, last = orbit_count(n, s) - 1;
    return u < last ? u : last;
}

// Position of bin edge e on a ring, in pixels relative to the pivot's cint: the first
// pixel p at or beyond the edge on the + side, the last n at or beyond it on the - side.
struct EdgePos {
    int kind;  // T_ZERO: every pixel at or beyond the edge; T_INF: none; else 0
    int p, n;
};

__device__ __forceinline__ EdgePos edge_pos(const LaneC& c, int2 T, double Ee, const ExactCtx& x, bool both) {
    EdgePos e;
    e.kind = T.x == T_ZERO ? T_ZERO : (T.x == T_INF ? T_INF : 0);
    e.p = e.n = 0;
    if (e.kind == 0) {
        e.p = pos_edge(c, T, Ee, x) - c.cint;
        if (both) e.n = neg_edge(c, T, Ee, x) - c.cint;
    }
    return e;
}

// Cell of a linear tile: pairs at offsets a .. a + n - 1 (offset 0 with no fraction is
// the single pixel on the pivot's meridian).
__device__ __forceinline__ void cell_lin(const EdgePos& lo, const EdgePos& hi, int crem, int& a, int& n) {
    const int none = crem == 0 ? 0 : 1;
    a = lo.kind == T_ZERO ? none : lo.p;
    n = max(0, (hi.kind == T_ZERO ? none : hi.p) - a);
}

// Cell of an orbit tile: n0 pixels from a0 upwards, then n1 pixels from a1 upwards.
__device__ __forceinline__ void cell_orbit(const EdgePos& lo, const EdgePos& hi, int nr, int& a0, int& n0, int& a1,
                                           int& n1) {
    a0 = a1 = n0 = n1 = 0;
    if (lo.kind == T_INF || hi.kind == T_ZERO) return;
    const int pe = hi.kind == T_INF ? nr / 2 : hi.p - 1;
    const int ns = hi.kind == T_INF ? 1 - nr / 2 : hi.n + 1;
    if (lo.kind == T_ZERO) {
        a0 = ns;
        n0 = max(0, pe - ns + 1);
    } else {
        a0 = lo.p;
        n0 = max(0, pe - a0 + 1);
        a1 = ns;
        n1 = max(0, lo.n - ns + 1);
    }
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

// Register sums of one bin for the lane's two pivots: index 0 holds (a_0, W).
template <int M, bool SELF>
struct WalkAcc {
    float2 a[M + 1], b[M + 1];
    float2 qa, qb;  // (sum (w d)^2, sum w^2), with SELF
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int m = 0; m <= M; ++m) a[m] = b[m] = make_float2(0.0f, 0.0f);
        qa = qb = make_float2(0.0f, 0.0f);
    }
};

// acc[m] += (v.x cos(m phi), v.y sin(m phi)), m = 1..M, for both pivots: the recurrence of
// harmonicsf with unit weights, run once for the two.
template <int M>
__device__ __forceinline__ void walk_fma(float4 f, float2 va, float2 vb, float2 (&a)[M + 1], float2 (&b)[M + 1],
                                         int mr) {
    if constexpr (M >= 1) {
        if (mr < 1) return;
        float2 X = make_float2(f.x, f.y), D = make_float2(0.5f * f.w, f.y);
        const float2 L2 = make_float2(f.w, f.w), S2 = make_float2(f.z, f.z);
        const float2 oa = __fmul2_rn(S2, va), ob = __fmul2_rn(S2, vb);  // odd multipoles take the fold's sign
        a[1] = __ffma2_rn(oa, X, a[1]);
        b[1] = __ffma2_rn(ob, X, b[1]);
#pragma unroll
        for (int m = 2; m <= M; ++m) {
            if (m > mr) break;
            D = __ffma2_rn(L2, X, D);
            X = __fadd2_rn(X, D);
            a[m] = __ffma2_rn((m & 1) ? oa : va, X, a[m]);
            b[m] = __ffma2_rn((m & 1) ? ob : vb, X, b[m]);
        }
    }
}

// Sweep of n staged steps (n rounded up to even: the entry after the last is staged too,
// pointing at the zero pixel g.npix) of a linear tile.
template <int M, bool SELF, bool WRAP, class L>
__device__ __forceinline__ void sweep_lin(const char* stage, int n, const L& ld, int npix, int nring, int qa, int qb,
                                          WalkAcc<M, SELF>& A, int mr) {
    constexpr int STR = WALK_STRIDE;
    const int h = (threadIdx.x >> 4) & 1;
    const char* row = stage + h * STR;
#pragma unroll 2
    for (int t = 0; t < n; t += 2, row += 2 * STR) {
        const int4 f = *reinterpret_cast<const int4*>(row);
        int pa, ma, pb, mb;
        if (WRAP) {  // f = (rel +, rel -, first, live bits)
            pa = wrap_idx(qa + f.x, nring) + f.z;
            ma = wrap_idx(qa + f.y, nring) + f.z;
            pb = wrap_idx(qb + f.x, nring) + f.z;
            mb = wrap_idx(qb + f.y, nring) + f.z;
            if (!(f.w & 1)) pa = pb = npix;
            if (!(f.w & 2)) ma = mb = npix;
        } else {  // f = (base +, base -, 0 or 1, 0 or 1): base + q, or the zero pixel
            pa = qa * f.z + f.x;
            ma = qa * f.w + f.y;
            pb = qb * f.z + f.x;
            mb = qb * f.w + f.y;
        }
        const float2 p0 = ld(pa), m0 = ld(ma), p1 = ld(pb), m1 = ld(mb);
        A.a[0] = __fadd2_rn(A.a[0], __fadd2_rn(p0, m0));
        A.b[0] = __fadd2_rn(A.b[0], __fadd2_rn(p1, m1));
        if (SELF) {
            A.qa = __ffma2_rn(p0, p0, __ffma2_rn(m0, m0, A.qa));
            A.qb = __ffma2_rn(p1, p1, __ffma2_rn(m1, m1, A.qb));
        }
        walk_fma<M>(*reinterpret_cast<const float4*>(row + 32), make_float2(p0.x + m0.x, p0.x - m0.x),
                    make_float2(p1.x + m1.x, p1.x - m1.x), A.a, A.b, mr);
    }
}

// The same on an orbit tile: the staged entry holds the pixel's eight images.
template <int M, bool SELF, class L>
__device__ __forceinline__ void sweep_orbit(const char* stage, int n, const L& ld, WalkAcc<M, SELF>& A, int mr) {
    constexpr int STR = WALK_STRIDE;
    const int lane = threadIdx.x & 31, h = lane >> 4, o = lane & 3, turn = (lane >> 2) & 3;
    const char* row = stage + (h * 4 + o) * STR;
#pragma unroll 2
    for (int t = 0; t < n; t += 2, row += 8 * STR) {
        const int2 f = *reinterpret_cast<const int2*>(row + 8 * turn);
        const float2 v0 = ld(f.x), v1 = ld(f.y);
        A.a[0] = __fadd2_rn(A.a[0], v0);
        A.b[0] = __fadd2_rn(A.b[0], v1);
        if (SELF) {
            A.qa = __ffma2_rn(v0, v0, A.qa);
            A.qb = __ffma2_rn(v1, v1, A.qb);
        }
        walk_fma<M>(*reinterpret_cast<const float4*>(row + 32), make_float2(v0.x, v0.x), make_float2(v1.x, v1.x), A.a,
                    A.b, mr);
    }
}

// Adds the register sums of bin k into the tile's moments.  Lane (h, l) holds partial
// sums of pivots l and l + 16; the halves exchange them, so that lane t ends with pivot t.
// sgn = -1 for the reflected pivots of an orbit tile, whose angles are the negatives.
template <int M, bool SELF, class Lay>
__device__ __forceinline__ void walk_flush(const Lay& lay, int k, WalkAcc<M, SELF>& A, float sgn, int mr) {
    const int lane = threadIdx.x & 31;
    const bool up = lane >= 16;
    auto join = [&](float a, float b) {
        return (up ? b : a) + __shfl_xor_sync(0xffffffffu, up ? a : b, 16);
    };
    atomicAdd(lay.a(k, 0, 0, lane), join(A.a[0].x, A.b[0].x));
    atomicAdd(lay.w(k, lane), join(A.a[0].y, A.b[0].y));
#pragma unroll
    for (int m = 1; m <= M; ++m) {
        if (m > mr) break;
        atomicAdd(lay.a(k, m, 0, lane), join(A.a[m].x, A.b[m].x));
        atomicAdd(lay.a(k, m, 1, lane), sgn * join(A.a[m].y, A.b[m].y));
    }
    if (SELF) {
        atomicAdd(lay.q(k, lane), join(A.qa.x, A.qb.x));
        atomicAdd(lay.qw(k, lane), join(A.qa.y, A.qb.y));
    }
    A.zero();
}

// All warps of the CTA: the moments of a tile into shared memory (zeroed by the caller,
// complete after the caller's barrier).  qa, qb: pixels in ring of pivots lane & 15 and
// (lane & 15) + 16; start: first orbit of the tile (orbit tiles).  scratch: walk_scratch_bytes(M, warps, cells), 16-byte aligned.
template <int M, bool SELF, class L, class Lay>
__device__ __forceinline__ void walk_tile(const MapDev& g, const PivotRing& P, bool lin, int qa, int qb, int start,
                                          const L& ld, const Lay& lay, char* scratch, int cells, int flush, int mr) {
    constexpr int STR = WALK_STRIDE;
    const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nthr >> 5;
    const int K = g.K;
    int* rlo = reinterpret_cast<int*>(scratch);  // [K] first ring of each bin
    int* cum = rlo + 32;                         // [K + 1] first cell of each bin
    int* ts = cum + 40;                          // [bins of the group + 1] first step of each bin
    int* ws = ts + 40;                           // [warps] scan
    int* pre = reinterpret_cast<int*>(scratch + WALK_HEAD);  // [cells + 1] entry counts, then their prefix sums
    short* c_a0 = reinterpret_cast<short*>(pre + cells + 4);
    short* c_a1 = c_a0 + cells;
    unsigned short* c_n0 = reinterpret_cast<unsigned short*>(c_a1 + cells);
    char* stage = reinterpret_cast<char*>(c_n0 + cells) + (size_t)warp * 32 * STR;
    const int npix = (int)g.npix;
    const int osh = lin ? 0 : 2, nc_max = cells >> osh;
    const int spc = 32 >> osh;  // steps per staged block
    flush <<= osh;
    // a linear tile none of whose rows wraps around the ring
    bool wrap = false;
    if (lin) {
        const int reach = g.ring_reach[P.i];
        wrap = !__all_sync(0xffffffffu, min(qa, qb) - reach >= 0 && max(qa, qb) + reach < P.n_i);
    }
    if (warp == 0) {
        int n = 0;
        if (lane < K) {
            const int2 br = g.bin_range[(long long)P.i * K + lane];
            rlo[lane] = br.x;
            n = br.y - br.x + 1;
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
    __syncthreads();
    const int X = cum[K];
    const float sgn = (!lin && lane >= 16) ? -1.0f : 1.0f;
    const int u = lin ? 0 : tile_orbit(P.n_i, P.s_i, start, lane & 3);
    WalkAcc<M, SELF> A;
    A.zero();
    for (int x0 = 0; x0 < X; x0 += nc_max) {
        const int nx = min(nc_max, X - x0);
        int ka = 0;
        while (cum[ka + 1] <= x0) ++ka;
        int kb = ka;
        while (cum[kb + 1] < x0 + nx) ++kb;
        const int nk = kb - ka + 1, nkc = (nk + 3) >> 2;
        // the cells: a thread takes four bins of one ring (and orbit), so that an edge
        // serves as the upper end of a bin and the lower end of the next
        {
            const int rb = rlo[kb];
            const int tasks = ((cum[kb + 1] - cum[kb]) * nkc) << osh;
            for (int t = tid; t < tasks; t += nthr) {
                const int o = t & ((1 << osh) - 1), rest = t >> osh;
                const int r = rb + rest / nkc, k0 = ka + 4 * (rest % nkc), k1 = min(k0 + 4, kb + 1);
                const int uo = lin ? 0 : tile_orbit(P.n_i, P.s_i, start, o);
                const ExactCtx x = exact_ctx(g, P, r);
                const LaneC c = lane_c(uo, P.s_i, P.n_i, g.ring_shift[r], x.n_r);
                const int2* T = g.pair_T + (P.pair0 + (r - P.rlo)) * (K + 1);
                EdgePos lo = edge_pos(c, T[k0], g.E[k0], x, !lin);
                for (int k = k0; k < k1; ++k) {
                    const EdgePos hi = edge_pos(c, T[k + 1], g.E[k + 1], x, !lin);
                    const int in = r - rlo[k], xi = cum[k] + in - x0;
                    if (in >= 0 && in < cum[k + 1] - cum[k] && xi >= 0 && xi < nx) {
                        const int ci = o * nx + xi;
                        int a0, n0, a1 = 0, n1 = 0;
                        if (lin)
                            cell_lin(lo, hi, c.crem, a0, n0);
                        else
                            cell_orbit(lo, hi, x.n_r, a0, n0, a1, n1);
                        pre[ci] = n0 + n1;
                        c_a0[ci] = (short)a0;
                        c_a1[ci] = (short)a1;
                        c_n0[ci] = (unsigned short)n0;
                    }
                    lo = hi;
                }
            }
        }
        __syncthreads();
        // exclusive scan of the entry counts
        {
            const int nc = nx << osh, per = (nc + nthr - 1) / nthr;
            const int b = min(nc, tid * per), e = min(nc, b + per);
            int s = 0;
            for (int i = b; i < e; ++i) s += pre[i];
            int inc = s;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, inc, d);
                if (lane >= d) inc += v;
            }
            if (lane == 31) ws[warp] = inc;
            __syncthreads();
            int base = inc - s;
            for (int w = 0; w < warp; ++w) base += ws[w];
            for (int i = b; i < e; ++i) {
                const int v = pre[i];
                pre[i] = base;
                base += v;
            }
            if (tid == nthr - 1) pre[nc] = base;
        }
        __syncthreads();
        if (warp == 0) {  // steps of each bin: the longest of the orbits' lists
            int n = 0;
            if (lane < nk) {
                const int xs = max(cum[ka + lane], x0) - x0, xe = min(cum[ka + lane + 1], x0 + nx) - x0;
                for (int o = 0; o < (1 << osh); ++o) n = max(n, pre[o * nx + xe] - pre[o * nx + xs]);
            }
            int s = n;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, s, d);
                if (lane >= d) s += v;
            }
            if (lane < nk) ts[lane + 1] = s;
            if (lane == 0) ts[0] = 0;
        }
        __syncthreads();
        const int total = ts[nk];
        int s = (int)((long long)total * warp / nw);
        const int send = (int)((long long)total * (warp + 1) / nw);
        int kk = 0;
        while (s < send) {
            while (ts[kk + 1] <= s) ++kk;
            const int k = ka + kk, e = min(send, ts[kk + 1]);
            const int xs = max(cum[k], x0) - x0, xe = min(cum[k + 1], x0 + nx) - x0;
            const int o = lane & ((1 << osh) - 1);
            const int row0 = o * nx;
            const int ent0 = pre[row0 + xs] - ts[kk], ent1 = pre[row0 + xe];
            const int rk = rlo[k] + x0 - cum[k];
            int blocks = 0, xlo = xs;
            for (; s < e; s += spc) {
                {
                    const int step = s + (lane >> osh);
                    int ent = ent0 + step;
                    const bool live = step < e && ent < ent1;
                    if (!live) ent = ent1 - 1;
                    int hi = xe - 1;
                    while (xlo < hi) {
                        const int mid = (xlo + hi + 1) >> 1;
                        if (pre[row0 + mid] <= ent) xlo = mid; else hi = mid - 1;
                    }
                    const int ci = row0 + xlo;
                    const int idx = max(0, ent - pre[ci]), n0 = c_n0[ci];
                    const int fi = idx < n0 ? c_a0[ci] + idx : c_a1[ci] + (idx - n0);
                    const int r = rk + xlo;
                    RingCtx R;
                    const WalkRing w = walk_ring(g, P, r, R);
                    int4* row = reinterpret_cast<int4*>(stage + lane * STR);
                    if (lin) {
                        const int d = P.s_i - w.shift, dq = d < 0 ? -1 : 0, half = d != 0 ? 1 : 0;
                        const bool single = half == 0 && fi == 0;
                        const int rp = dq + fi, rm = dq + half - fi;
                        const int on = live ? 1 : 0, on2 = live && !single ? 1 : 0;
                        if (wrap)
                            row[0] = make_int4(rp, rm, w.first, on | (on2 << 1));
                        else
                            row[0] = make_int4(on ? w.first + rp : npix, on2 ? w.first + rm : npix, on, on2);
                        *reinterpret_cast<float4*>(row + 2) = entry_angle(R, fi, half ? 0.5f : 0.0f);
                    } else {
                        const LaneC c = lane_c(u, P.s_i, P.n_i, w.shift, w.n);
                        const int p = wrap_idx(c.cint + fi, w.n), qn = w.n >> 2;
                        int m = -p - w.shift;
                        if (m < 0) m += w.n;
                        int im[8];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int x = p + j * qn, y = m + j * qn;
                            im[2 * j] = live ? w.first + (x >= w.n ? x - w.n : x) : npix;
                            im[2 * j + 1] = live ? w.first + (y >= w.n ? y - w.n : y) : npix;
                        }
                        row[0] = make_int4(im[0], im[1], im[2], im[3]);
                        row[1] = make_int4(im[4], im[5], im[6], im[7]);
                        *reinterpret_cast<float4*>(row + 2) = entry_angle(R, fi, c.cfrac);
                    }
                }
                __syncwarp();
                const int n = min(spc, e - s);
                if (!lin)
                    sweep_orbit<M, SELF>(stage, n, ld, A, mr);
                else if (wrap)
                    sweep_lin<M, SELF, true>(stage, n, ld, npix, P.n_i, qa, qb, A, mr);
                else
                    sweep_lin<M, SELF, false>(stage, n, ld, npix, P.n_i, qa, qb, A, mr);
                __syncwarp();
                if (++blocks == flush) {
                    blocks = 0;
                    walk_flush<M, SELF>(lay, k, A, sgn, mr);
                }
            }
            s = e;
            if (blocks) walk_flush<M, SELF>(lay, k, A, sgn, mr);
        }
        __syncthreads();
    }
}

}  // namespace tpcf
