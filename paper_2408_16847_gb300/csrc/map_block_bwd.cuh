// Adjoint of a block of pivots (map_block.cuh has the moments, phase 1).
//
// dL/d d_p for L(zeta), with C_m = (dL/dRe zeta + i dL/dIm zeta) / D and
// H_m(k,k') = conj(C_m(k,k')) + C_m(k',k) (prepared by adjoint_prep_kernel):
//   primary term      w_p * (1/2) sum_{k,m} Re[a_m^k(p) h_m^k(p)]
//   neighbour legs    w_p * sum_{i: p in nbr(i)} w_i d_i sum_m Re[e^{-i m phi_ip} h_m^{k(ip)}(i)]
//   with h_m^k(i) = sum_{k'} H_m(k,k') conj(a_m^{k'}(i)).
// Phase 2 turns the block's moments in the workspace into w_i d_i h, in place; phase 3 goes over
// the entries again.  Linear blocks: the rings in reach are taken a few rows at a time; each
// warp keeps the rows' sums for its own pivots in shared memory (a row is wider than the
// pivots by the reach on both sides; plain read-modify-write, the lanes of a step hit
// different words), the CTA stages the entries' harmonics bin by bin, and a warp holds h of the
// current bin in registers.  A finished row goes to the gradient with one reduction per
// pixel.  Other rings: per-lane angles as in phase 1, one reduction per image and entry.
//
// Forward + adjoint before (each lane's own angles, a reduction per pixel and pivot) and now: Nside 4096
// belt slice 126 -> 74 ms, masked Nside 1024 to 3 deg 1018 -> 557 ms.
#pragma once

namespace tpcf {

// Phase 2, four subtiles at a time: smem holds one multipole's moments of the four, H transposed,
// and the pivots' values and primary sums.
// value(s, lane): (w d, w) of the pivot; pixel(s, lane): its pixel; primary sums go to c.grad.
template <int M, bool SELF, class V, class X>
__device__ __forceinline__ void block_h(const MapCall& c, int K, int mr, float* ws, size_t sub_floats, int nsub,
                                        unsigned live, V&& value, X&& pixel, char* smem) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int Kp = (K + 3) & ~3, nA = 4 * K * 2 * TILE;
    // one or two buffers of (moments [4][K][2][32], H [k'][Kp]): with two, the next multipole is
    // staged while this one is used
    const size_t buf = (size_t)nA * sizeof(float) + (size_t)K * Kp * sizeof(float2);
    const bool two = 2 * buf + 3 * 4 * TILE * sizeof(float) <= adj_smem_bytes(M);
    float* sWd = reinterpret_cast<float*>(smem + (two ? 2 : 1) * buf);  // [4][32] w d
    float* sPrim = sWd + 4 * TILE;                                      // [4][32]
    float* sPw = sPrim + 4 * TILE;                                      // [4][32] w
    const float* cdiag = c.H + (size_t)(mr + 1) * K * K * 2;
    const int ksets = Kp >> 2;
    for (int s0 = 0; s0 < nsub; s0 += 4) {
        const unsigned on = (live >> s0) & 15u;
        if (on == 0u) continue;
        if (s0 + warp < nsub) {
            const float2 v = value(s0 + warp, lane);
            sWd[warp * TILE + lane] = v.x;
            sPw[warp * TILE + lane] = v.y;
        }
        sPrim[tid] = 0.0f;
        auto stage = [&](int m) {
            char* b = smem + (two ? (m & 1) * buf : 0);
            float* A = reinterpret_cast<float*>(b);
            float2* H = reinterpret_cast<float2*>(A + nA);
            for (int u = 0; u < 4; ++u)
                if ((on >> u) & 1u)
                    stage_copy(A + (size_t)u * K * 2 * TILE, ws + (s0 + u) * sub_floats + (size_t)m * K * 2 * TILE,
                               K * 2 * TILE);
            for (int e = tid; e < K * Kp; e += BT) {  // H(k, k') at [k'][k]; columns past K are zero
                const int kp = e / Kp, k = e - kp * Kp;
                H[e] = k < K ? __ldg(reinterpret_cast<const float2*>(c.H + (((size_t)m * K + k) * K + kp) * 2))
                             : make_float2(0.0f, 0.0f);
            }
        };
        if (two) stage(0);
        for (int m = 0; m <= mr; ++m) {
            if (!two) {
                __syncthreads();
                stage(m);
            }
            stage_wait();
            __syncthreads();
            if (two && m < mr) stage(m + 1);
            const float* sA = reinterpret_cast<const float*>(smem + (two ? (m & 1) * buf : 0));
            const float2* sH = reinterpret_cast<const float2*>(sA + nA);
            // a warp task: four bins of two subtiles, one pivot of each per lane
            for (int t = warp; t < 2 * ksets; t += BW) {
                const int pr = t & 1, k0 = (t >> 1) * 4;
                if (((on >> (2 * pr)) & 3u) == 0u) continue;
                const float* a0 = sA + (size_t)(2 * pr) * K * 2 * TILE + lane;
                const float* a1 = a0 + (size_t)K * 2 * TILE;
                float2 x[4], y[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) x[j] = y[j] = make_float2(0.0f, 0.0f);
                for (int kp = 0; kp < K; ++kp) {
                    // moments are a = re - i im, so h = H conj(a) = (Hr re - Hi im, Hr im + Hi re)
                    const float2 u = make_float2(a0[kp * 2 * TILE], a0[kp * 2 * TILE + TILE]);
                    const float2 v = make_float2(a1[kp * 2 * TILE], a1[kp * 2 * TILE + TILE]);
                    const float2 ur = make_float2(-u.y, u.x), vr = make_float2(-v.y, v.x);
                    const float4* h4 = reinterpret_cast<const float4*>(sH + (size_t)kp * Kp + k0);
                    const float4 ha = h4[0], hb = h4[1];
                    const float2 h[4] = {make_float2(ha.x, ha.y), make_float2(ha.z, ha.w), make_float2(hb.x, hb.y),
                                         make_float2(hb.z, hb.w)};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        x[j] = __ffma2_rn(make_float2(h[j].x, h[j].x), u, __ffma2_rn(make_float2(h[j].y, h[j].y), ur, x[j]));
                        y[j] = __ffma2_rn(make_float2(h[j].x, h[j].x), v, __ffma2_rn(make_float2(h[j].y, h[j].y), vr, y[j]));
                    }
                }
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int s = 2 * pr + u;
                    if (!((on >> s) & 1u)) continue;
                    const float* a = u ? a1 : a0;
                    const float wd = sWd[s * TILE + lane];
                    float* out = ws + (s0 + s) * sub_floats + ((size_t)m * K + k0) * 2 * TILE + lane;
                    float prim = 0.0f;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if (k0 + j >= K) break;
                        const float2 h = u ? y[j] : x[j];
                        prim = fmaf(a[(k0 + j) * 2 * TILE], h.x, fmaf(a[(k0 + j) * 2 * TILE + TILE], h.y, prim));
                        __stcg(out + j * 2 * TILE, wd * h.x);
                        __stcg(out + j * 2 * TILE + TILE, wd * h.y);
                    }
                    atomicAdd(sPrim + s * TILE + lane, prim);
                }
            }
        }
        __syncthreads();
        if ((on >> warp) & 1u) {
            const int s = s0 + warp;
            const float w = sPw[warp * TILE + lane];
            if (w != 0.0f) {
                float gp = 0.5f * w * sPrim[warp * TILE + lane];
                if (SELF) {  // the subtracted diagonal: -w_p Q^k(p) cdiag_k
                    const float* Q = ws + s * sub_floats + (size_t)(mr + 1) * K * 2 * TILE + K * TILE + lane;
                    float t = 0.0f;
                    for (int k = 0; k < K; ++k) t = fmaf(cdiag[k], __ldcg(Q + k * TILE), t);
                    gp = fmaf(-w, t, gp);
                }
                if (gp != 0.0f) atomicAdd(c.grad + pixel(s, lane), gp);
            }
        }
        __syncthreads();
    }
}

// w d h of bin k for the lane's NP pivots, from the workspace; zero for subtiles without a live pivot
// (bit j of `on` clear), which phase 2 skips.
template <int M, int NP>
__device__ __forceinline__ void load_h(float2 (&h)[NP][M + 1], const float* ws, size_t sub_floats, int K, int k,
                                       unsigned on, int mr) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < NP; ++j)
#pragma unroll
        for (int m = 0; m <= M; ++m) {
            const float* p = ws + j * sub_floats + ((size_t)m * K + k) * 2 * TILE + lane;
            h[j][m] = m <= mr && ((on >> j) & 1u) ? make_float2(__ldcg(p), __ldcg(p + TILE)) : make_float2(0.0f, 0.0f);
        }
}

// Where the legs of a linear block go: rows in shared memory, or straight to the gradient.
template <bool ROWS>
struct LegSink {
    float* row;       // ROWS: the warp's rows, at this lane's column for offset 0
    int width;        // ROWS: words per row
    const float2* wdw;
    float* grad;
    int n;
};

// Legs of staged entries [e0, e1).  Staged heads: HEAD_ROW (ROWS) or HEAD_WRAP.
template <int M, int P, bool SELF, bool ROWS>
__device__ __forceinline__ void lin_legs(const char* stage, int e0, int e1, const float2 (&h)[P][M + 1],
                                         const LegSink<ROWS>& S, const int (&q)[P], const float (&ck)[P], int mr) {
    constexpr int STR = lin_stride(M);
    const char* row = stage + (ptrdiff_t)e0 * STR;
#pragma unroll 2
    for (int e = e0; e < e1; ++e, row += STR) {
        const int4 f = *reinterpret_cast<const int4*>(row);
        const float hw = __int_as_float(f.z);
        float2 ev[P], od[P];  // (cosine part, sine part), two chains
#pragma unroll
        for (int j = 0; j < P; ++j) {
            ev[j] = make_float2(hw * h[j][0].x, 0.0f);
            od[j] = make_float2(0.0f, 0.0f);
        }
        const float4* co = reinterpret_cast<const float4*>(row) + 1;
#pragma unroll
        for (int i = 0; i < (M + 1) / 2; ++i) {
            const int m = 2 * i + 1;
            if (m > mr) break;
            const float4 v = co[i];
#pragma unroll
            for (int j = 0; j < P; ++j) od[j] = __ffma2_rn(make_float2(v.x, v.y), h[j][m], od[j]);
            if (m + 1 <= M) {
                if (m + 1 > mr) break;
#pragma unroll
                for (int j = 0; j < P; ++j) ev[j] = __ffma2_rn(make_float2(v.z, v.w), h[j][m + 1], ev[j]);
            }
        }
        float vp[P], vm[P];
#pragma unroll
        for (int j = 0; j < P; ++j) {
            const float2 t = __fadd2_rn(ev[j], od[j]);
            vp[j] = t.x + t.y;
            vm[j] = t.x - t.y;
        }
        if (ROWS) {
            // the + and the - pixels of a step may overlap: one after the other
            float* pp = S.row + f.w * S.width + f.x;
            float* pm = S.row + f.w * S.width + f.y;
            float t[P];
#pragma unroll
            for (int j = 0; j < P; ++j) t[j] = pp[32 * j];
#pragma unroll
            for (int j = 0; j < P; ++j) pp[32 * j] = t[j] + vp[j];
            __syncwarp();
#pragma unroll
            for (int j = 0; j < P; ++j) t[j] = pm[32 * j];
#pragma unroll
            for (int j = 0; j < P; ++j) pm[32 * j] = t[j] + vm[j];
            __syncwarp();
        } else {
#pragma unroll
            for (int j = 0; j < P; ++j) {
                const int ip = wrap_idx(q[j] + f.x, S.n) + f.w, im = wrap_idx(q[j] + f.y, S.n) + f.w;
                const float2 a = __ldg(S.wdw + ip), b = __ldg(S.wdw + im);
                if (SELF) {  // self-pair subtraction: -2 cdiag_k (w_p d_p) per neighbour p
                    vp[j] = fmaf(hw * ck[j], a.x, vp[j]);
                    vm[j] = fmaf(hw * ck[j], b.x, vm[j]);
                }
                atomicAdd(S.grad + ip, a.y * vp[j]);
                atomicAdd(S.grad + im, b.y * vm[j]);
            }
        }
    }
}

// Phase 3 of a linear block over part `part` of its rings.  Every thread calls it.
template <int M, int P, bool SELF>
__device__ __forceinline__ void lin_adjoint(const MapDev& g, const MapCall& c, const PivotRing& PR, int q0,
                                            const int (&q)[P], const float (&wd)[P], unsigned live, const float* ws,
                                            size_t sub_floats, char* smem, int part, int mr) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const LinTables t = lin_tables(smem, M, ADJ_CHUNK, ADJ_CELLS);
    float* rows = reinterpret_cast<float*>(smem + adj_head_bytes(M)) + warp * ADJ_ROW_FLOATS;
    const int K = g.K, reach = g.ring_reach[PR.i];
    const int width = P * TILE + 2 * reach;
    // rows that fit the warp's space; too wide (or self-pair subtraction, which needs the
    // neighbour's own value): straight to the gradient
    const bool use_rows = !SELF && width <= ADJ_ROW_FLOATS;
    const int nrow = use_rows ? min(ADJ_ROW_FLOATS / width, ADJ_CELLS / K) : ADJ_CELLS / K;
    const int2 all = g.ring_range[PR.i];
    const int nr = all.y - all.x + 1;
    const int ra0 = all.x + (int)((long long)nr * part / c.parts), ra1 = all.x + (int)((long long)nr * (part + 1) / c.parts);
    const float* cdiag = c.H + (size_t)(mr + 1) * K * K * 2;
    float2 h[P][M + 1];
    float ck[P];
#pragma unroll
    for (int j = 0; j < P; ++j) ck[j] = 0.0f;
    if (use_rows)
        for (int e = lane; e < nrow * width; e += 32) rows[e] = 0.0f;
    __syncwarp();
    for (int ra = ra0; ra < ra1; ra += nrow) {
        const int rb = min(ra + nrow, ra1) - 1;
        __syncthreads();
        if (warp == 0) bin_cells(g, PR.i, K, ra, rb, t.rlo, t.cum);
        __syncthreads();
        const int nx = t.cum[K];
        if (nx > 0) {
            lin_cells(g, PR, t, 0, K - 1, 0, nx);
            const int total = t.pre[nx];
            const int head = use_rows ? HEAD_ROW : HEAD_WRAP;
            lin_stage<M, ADJ_CHUNK>(g, PR, t, 0, K - 1, 0, nx, total, 0, head, ra, mr);
            __syncthreads();
            int pos = 0, k = 0, kh = -1;
            for (int ch = 0; ch * ADJ_CHUNK < total; ++ch) {
                lin_stage<M, ADJ_CHUNK>(g, PR, t, 0, K - 1, 0, nx, total, ch + 1, head, ra, mr);
                if (live) {
                    const int cend = min(total, (ch + 1) * ADJ_CHUNK);
                    const char* st = t.stage + (ptrdiff_t)((ch & 1) - ch) * ADJ_CHUNK * lin_stride(M);
                    while (pos < cend) {
                        while (t.pre[t.cum[k + 1]] <= pos) ++k;
                        const int e = min(t.pre[t.cum[k + 1]], cend);
                        if (k != kh) {
                            load_h<M, P>(h, ws, sub_floats, K, k, live, mr);
                            kh = k;
                            if (SELF)
#pragma unroll
                                for (int j = 0; j < P; ++j) ck[j] = -2.0f * cdiag[k] * wd[j];
                        }
                        if (use_rows)
                            lin_legs<M, P, SELF, true>(st, pos, e, h, LegSink<true>{rows + lane + reach, width, nullptr, nullptr, 0},
                                                       q, ck, mr);
                        else
                            lin_legs<M, P, SELF, false>(st, pos, e, h, LegSink<false>{nullptr, 0, c.wdw, c.grad, PR.n_i}, q,
                                                        ck, mr);
                        pos = e;
                    }
                }
                __syncthreads();
            }
        }
        if (use_rows && live) {  // the rows to the gradient
            for (int r = ra; r <= rb; ++r) {
                const int first = (int)g.ring_first[r];
                float* row = rows + (r - ra) * width;
                for (int e = lane; e < width; e += 32) {
                    const float v = row[e];
                    if (v != 0.0f) {
                        const int x = q0 - reach + e;  // within [-n, 2 n)
                        const int p = first + wrap_idx(x, PR.n_i);
                        atomicAdd(c.grad + p, v * __ldg(&c.wdw[p].y));
                        row[e] = 0.0f;
                    }
                }
            }
            __syncwarp();
        }
    }
}

// sum_m Re[e^{-i m phi} h_m] at offset fi for the lane's IM images.
template <int M, int IM, bool FAST>
__device__ __forceinline__ void orbit_leg(const RingCtx& R, float fi, float xneg, float uneg, const float2 (&h)[IM][M + 1],
                                          float (&u)[IM], int mr) {
    float cph, sph;
    pixel_dir<FAST>(fi, xneg, uneg, R, cph, sph);
    float2 ev[IM], od[IM];
    float sg = 1.0f;
#pragma unroll
    for (int j = 0; j < IM; ++j) {
        ev[j] = make_float2(h[j][0].x, 0.0f);
        od[j] = make_float2(0.0f, 0.0f);
    }
    if constexpr (M >= 1) {
        if (mr >= 1) {
            const Fold f = fold_angle(cph, sph);
            sg = f.sg;
            float2 X = make_float2(f.ac, f.ss), D = make_float2(0.5f * f.lam, f.ss);
            const float2 L2 = make_float2(f.lam, f.lam);
#pragma unroll
            for (int j = 0; j < IM; ++j) od[j] = __fmul2_rn(X, h[j][1]);
#pragma unroll
            for (int m = 2; m <= M; ++m) {
                if (m > mr) break;
                D = __ffma2_rn(L2, X, D);
                X = __fadd2_rn(X, D);
#pragma unroll
                for (int j = 0; j < IM; ++j) {
                    if (m & 1)
                        od[j] = __ffma2_rn(X, h[j][m], od[j]);
                    else
                        ev[j] = __ffma2_rn(X, h[j][m], ev[j]);
                }
            }
        }
    }
#pragma unroll
    for (int j = 0; j < IM; ++j) u[j] = fmaf(sg, od[j].x + od[j].y, ev[j].x + ev[j].y);
}

// Legs of the lane's two runs of one ring for its IM images.  Where nothing wraps, the part of a
// run that all lanes have goes without predicates, the pixels loaded one entry ahead.  (Summing
// a run in a patch in shared memory first, one reduction per pixel instead of one per entry,
// was slower: 39.5 against 32.1 ms for forward + adjoint of a polar slice; the reductions
// themselves cost about a tenth.)
template <int M, int IM, bool FAST, bool WRAP, bool SELF>
__device__ __forceinline__ void orbit_legs(const RingCtx& R, const WalkRing& w, const LaneC& c, BinRuns b,
                                           const float2 (&h)[IM][M + 1], const float (&ck)[IM],
                                           const float2* __restrict__ wdw, float* grad, int mr) {
    const float xneg = -c.cfrac * R.step, uneg = -c.cfrac * R.inv_n;
    auto put = [&](int x, float2 v, float u, float ckj) {
        if (SELF) u = fmaf(ckj, v.x, u);
        atomicAdd(grad + x, v.y * u);
    };
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
                v[j] = __ldg(wdw + x[j]);
                x0 = wrap_idx(x0 + w.n / IM, w.n);
            }
            float fi = (float)(a - c.cint);
#pragma unroll 2
            for (int t = 0; t < len; ++t, fi += 1.0f) {
                float2 vn[IM];  // (the one after the last is read and not used)
#pragma unroll
                for (int j = 0; j < IM; ++j) vn[j] = __ldg(wdw + x[j] + 1);
                float u[IM];
                orbit_leg<M, IM, FAST>(R, fi, xneg, uneg, h, u, mr);
#pragma unroll
                for (int j = 0; j < IM; ++j) {
                    put(x[j]++, v[j], u[j], ck[j]);
                    v[j] = vn[j];
                }
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
#pragma unroll 1
    for (int t = 0; t < maxt; ++t) {
        const bool on = t < cur.tot;
        float2 v[IM];
        int x[IM];
#pragma unroll
        for (int j = 0; j < IM; ++j) {
            x[j] = cur.pixel(t, j);
            v[j] = on ? __ldg(wdw + x[j]) : make_float2(0.0f, 0.0f);
        }
        float u[IM];
        orbit_leg<M, IM, FAST>(R, cur.offset(t), xneg, uneg, h, u, mr);
        if (on) {
#pragma unroll
            for (int j = 0; j < IM; ++j) put(x[j], v[j], u[j], ck[j]);
        }
    }
}

// Phase 3 of one (warp tile, bin) item.
template <int M, int IM, bool SELF>
__device__ __forceinline__ void orbit_adjoint(const MapDev& g, const MapCall& c, const PivotRing& P, int q, int k, int sl,
                                              const float (&wd)[IM], unsigned live, const float* ws, size_t sub_floats,
                                              char* stage, int mr) {
    float2 h[IM][M + 1];
    load_h<M, IM>(h, ws, sub_floats, g.K, k, live, mr);
    float ck[IM];
#pragma unroll
    for (int j = 0; j < IM; ++j) ck[j] = SELF ? -2.0f * c.H[(size_t)(mr + 1) * g.K * g.K * 2 + k] * wd[j] : 0.0f;
    orbit_rings<IM>(g, P, q, k, sl, c.slices, stage, [&](const RingCtx& R, const WalkRing& w, const LaneC& lc, const BinRuns& b, bool fast,
                                           bool flat) {
        if (!fast)
            orbit_legs<M, IM, false, true, SELF>(R, w, lc, b, h, ck, c.wdw, c.grad, mr);
        else if (flat)
            orbit_legs<M, IM, true, false, SELF>(R, w, lc, b, h, ck, c.wdw, c.grad, mr);
        else
            orbit_legs<M, IM, true, true, SELF>(R, w, lc, b, h, ck, c.wdw, c.grad, mr);
    });
}

// Phase 2 of a block.  Every thread calls it.
template <int M, bool SELF>
__device__ __forceinline__ void block_prim(const MapDev& g, const MapCall& c, long long b, unsigned live, float* ws,
                                        size_t sub_floats, char* smem, int mr) {
    const Block<M, false> B(g, c, b);
    const PackedLoad ld{c.wdw};
    block_h<M, SELF>(c, g.K, mr, ws, sub_floats, B.nsub, live, [&](int s, int l) { return B.value(g, c, ld, s, l); },
                  [&](int s, int l) { return B.pixel(g, s, l); }, smem);
}

// Phase 3 of part `part` of a linear block.  Every thread calls it.
template <int M, bool SELF>
__device__ __forceinline__ void lin_block_legs(const MapDev& g, const MapCall& c, long long b, unsigned live, int part,
                                            const float* ws, size_t sub_floats, char* smem, int mr) {
    constexpr int NP = Block<M, false>::NP;
    const Block<M, false> B(g, c, b);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int2 tq = *B.list;
    const PivotRing PR = pivot_ring(g, tq.x);
    int q[NP];
    float wd[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        q[j] = min(tq.y + (warp * NP + j) * TILE + lane, PR.n_i - 1);
        wd[j] = SELF ? B.value(g, c, PackedLoad{c.wdw}, warp * NP + j, lane).x : 0.0f;
    }
    lin_adjoint<M, NP, SELF>(g, c, PR, tq.y + warp * NP * TILE, q, wd, (live >> (warp * NP)) & ((1u << NP) - 1u),
                             ws + (size_t)warp * NP * sub_floats, sub_floats, smem, part, mr);
}

// Phase 3 of part `part` of another block: its warps draw (tile, bin) items.
template <int M, bool SELF>
__device__ __forceinline__ void orb_block_legs(const MapDev& g, const MapCall& c, long long b, unsigned live, int part,
                                            const float* ws, size_t sub_floats, char* smem, int mr) {
    constexpr int NP = Block<M, false>::NP;
    __shared__ int s_item;
    const Block<M, false> B(g, c, b);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_item = 0;
    __syncthreads();
    const int kb = part_bin(g.E, g.K, part, c.parts), ke = part_bin(g.E, g.K, part + 1, c.parts);
    const int S = c.slices, items = B.T * (ke - kb) * S;
    for (;;) {
        int it = 0;
        if (lane == 0) it = atomicAdd(&s_item, 1);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= items) break;
        const int sl = it % S, u = it / S;
        const int t = u % B.T, k = ke - 1 - u / B.T;
        const unsigned on = (live >> (t * NP)) & ((1u << NP) - 1u);
        if (on == 0u) continue;
        const int2 tq = B.list[t];
        const PivotRing PR = pivot_ring(g, tq.x);
        float wd[NP];
#pragma unroll
        for (int j = 0; j < NP; ++j) wd[j] = SELF ? B.value(g, c, PackedLoad{c.wdw}, t * NP + j, lane).x : 0.0f;
        orbit_adjoint<M, NP, SELF>(g, c, PR, min(tq.y + lane, PR.n_i / NP - 1), k, sl, wd, on, ws + (size_t)t * NP * sub_floats,
                                   sub_floats, smem + warp * 32 * ORB_STRIDE, mr);
    }
}

// One work item of an adjoint.  step 0: all phases of a block (parts = 1); 1: moments of a
// part, and phase 2 by the block's last part; 2: phase 3 of a part (blocks in the workspace from step 1).
template <int M, bool SELF>
__device__ __forceinline__ void bwd_block(const MapDev& g, const MapCall& c, long long b, int part, int step, float* ws,
                                          char* smem, int mr) {
    const Block<M, false> B(g, c, b);
    const size_t sub_floats = sub_floats_rt(g.K, mr, SELF);
    const PackedLoad ld{c.wdw};
    const unsigned live = block_live(B.nsub, [&](int s, int l) { return B.value(g, c, ld, s, l).y != 0.0f; });
    if (live == 0u) return;
    if (step != 2) {
        block_moments<M, SELF, false>(g, c, b, live, part, ld, ws, sub_floats, smem, mr);
        if (!block_complete(c, b)) return;
        block_fold(c, b, B.nsub, ws, sub_floats);
        block_prim<M, SELF>(g, c, b, live, ws, sub_floats, smem, mr);
    }
    if (step != 1) {
        if (b < c.nlin)
            lin_block_legs<M, SELF>(g, c, b, live, part, ws, sub_floats, smem, mr);
        else
            orb_block_legs<M, SELF>(g, c, b, live, part, ws, sub_floats, smem, mr);
    }
    __syncthreads();
}

}  // namespace tpcf
