// Tile kernels: a CTA of 8 warps takes 32 consecutive pivots of one ring at a time and keeps
// their moments in shared memory.  They serve the calls that have too few blocks for
// map_block.cuh (the rule and its figures: takes_blocks in api.cu): a tile's rings are split over
// eight warps and its pivots are not paired with images, so the chain of one warp is short where few
// warps have work.
//
//   * for every radial bin k the warps split the neighbour rings that can hold bin-k pixels;
//   * on a neighbour ring the bin-k pixels of a pivot form at most two contiguous runs, found
//     from the per-ring-pair edge offsets T_e of the plan; each lane walks its own runs, so
//     the (M+1) complex accumulators of the bin stay in registers across rings;
//   * in the equatorial belt a neighbour ring has as many pixels as the pivot ring: the
//     pixel at +phi and its mirror at -phi share one angle, which the warp's lanes share too;
//   * after all bins the CTA forms sum_i w_i d_i a^{k1} conj(a^{k2}) (eq. zetamEst2) and
//     sum_i w_i W^{k1} W^{k2} from shared memory, adding them in FP64 into a slot owned
//     by the CTA (FP32 pipe, or the tensor cores in map_tile_tc_kernel).
// Bound: latency (few warps).  Per call on a GB300, blocks against tiles, 8 multipoles: Nside 8, 2 bins
// to 60 deg 62 against 59 us; Nside 24, 1 bin 110 against 77 us; Nside 24, 8 bins 127 against 106 us.
#pragma once

namespace tpcf {

template <int M>
__device__ __forceinline__ void harmonics(float2 (&acc)[M + 1], float cph, float sph, float wc, float ws,
                                          int mr = M) {
    harmonicsf<M>(acc, fold_angle(cph, sph), wc, ws, mr);
}

// The same for two pixels a and b at once (two independent chains for
// instruction-level parallelism), from their folded angles.
template <int M>
__device__ __forceinline__ void harmonics2f(float2 (&acc)[M + 1], const Fold& fa, float wca, float wsa,
                                            const Fold& fb, float wcb, float wsb, int mr = M) {
    acc[0].x += wca + wcb;
    if constexpr (M >= 1) {
        if (mr < 1) return;
        float2 Xa = make_float2(wca * fa.ac, wsa * fa.ss), Da = make_float2(0.5f * fa.lam * wca, wsa * fa.ss);
        float2 Xb = make_float2(wcb * fb.ac, wsb * fb.ss), Db = make_float2(0.5f * fb.lam * wcb, wsb * fb.ss);
        const float2 Sa = make_float2(fa.sg, fa.sg), Sb = make_float2(fb.sg, fb.sg);
        const float2 La = make_float2(fa.lam, fa.lam), Lb = make_float2(fb.lam, fb.lam);
        acc[1] = __ffma2_rn(Sb, Xb, __ffma2_rn(Sa, Xa, acc[1]));
#pragma unroll
        for (int m = 2; m <= M; ++m) {
            if (m > mr) break;
            Da = __ffma2_rn(La, Xa, Da);
            Db = __ffma2_rn(Lb, Xb, Db);
            Xa = __fadd2_rn(Xa, Da);
            Xb = __fadd2_rn(Xb, Db);
            if (m & 1)
                acc[m] = __ffma2_rn(Sb, Xb, __ffma2_rn(Sa, Xa, acc[m]));
            else
                acc[m] = __fadd2_rn(acc[m], __fadd2_rn(Xa, Xb));
        }
    }
}

template <int M>
__device__ __forceinline__ void harmonics2(float2 (&acc)[M + 1], float ca, float sa, float wca, float wsa, float cb,
                                           float sb, float wcb, float wsb, int mr = M) {
    harmonics2f<M>(acc, fold_angle(ca, sa), wca, wsa, fold_angle(cb, sb), wcb, wsb, mr);
}

// A folded angle held by lane `src`, broadcast to the warp.
__device__ __forceinline__ Fold shfl_fold(const Fold& f, int src) {
    Fold g;
    g.ac = __shfl_sync(0xffffffffu, f.ac, src);
    g.ss = __shfl_sync(0xffffffffu, f.ss, src);
    g.sg = __shfl_sync(0xffffffffu, f.sg, src);
    g.lam = __shfl_sync(0xffffffffu, f.lam, src);
    return g;
}

// Walk pixels [a, a + len) of ring R (lane-private run), accumulating into the bin.
// Two pixels per iteration.  When no lane's run wraps around the ring, the first
// min-length iterations run without predicates or index wrapping; the rest (and
// wrapping runs) take the general loop.
template <int M, bool FAST, bool SELF, class L>
__device__ __forceinline__ void walk_run(const RingCtx& R, const L& ld, const LaneC& c, int a, int len,
                                         float2 (&acc)[M + 1], float& W, float& Q, float& QW, int mr = M) {
    const int maxlen = __reduce_max_sync(0xffffffffu, len);
    if (maxlen <= 0) return;
    const float i0 = (float)(a - c.cint);
    const float xneg = -c.cfrac * R.step, uneg = -c.cfrac * R.inv_n;
    int idx = wrap_idx(a, R.n);
    const auto row = ld.row(R.first);
    int t = 0;
    const int minlen = __reduce_min_sync(0xffffffffu, len);
    if (minlen >= 2 && __all_sync(0xffffffffu, idx + len <= R.n)) {
        float ft = i0;
        for (; t + 1 < minlen; t += 2, ft += 2.0f) {
            const float2 v0 = row(idx + t), v1 = row(idx + t + 1);
            float ca, sa, cb, sb;
            pixel_dir<FAST>(ft, xneg, uneg, R, ca, sa);
            pixel_dir<FAST>(ft + 1.0f, xneg, uneg, R, cb, sb);
            harmonics2<M>(acc, ca, sa, v0.x, v0.x, cb, sb, v1.x, v1.x, mr);
            W += v0.y + v1.y;
            if (SELF) {
                Q = fmaf(v0.x, v0.x, fmaf(v1.x, v1.x, Q));
                QW = fmaf(v0.y, v0.y, fmaf(v1.y, v1.y, QW));
            }
        }
        idx += t;
        if (idx >= R.n) idx -= R.n;
    }
    for (; t < maxlen; t += 2) {
        const bool on0 = t < len, on1 = t + 1 < len;
        const int idx1 = idx + 1 >= R.n ? idx + 1 - R.n : idx + 1;
        const float2 v0 = on0 ? row(idx) : make_float2(0.0f, 0.0f);
        const float2 v1 = on1 ? row(idx1) : make_float2(0.0f, 0.0f);
        const float oa = on0 ? i0 + (float)t : i0;
        const float ob = on1 ? i0 + (float)(t + 1) : i0;
        float ca, sa, cb, sb;
        pixel_dir<FAST>(oa, xneg, uneg, R, ca, sa);
        pixel_dir<FAST>(ob, xneg, uneg, R, cb, sb);
        harmonics2<M>(acc, ca, sa, v0.x, v0.x, cb, sb, v1.x, v1.x, mr);
        W += v0.y + v1.y;
        if (SELF) {
            Q = fmaf(v0.x, v0.x, fmaf(v1.x, v1.x, Q));
            QW = fmaf(v0.y, v0.y, fmaf(v1.y, v1.y, QW));
        }
        idx = idx1 + 1 >= R.n ? idx1 + 1 - R.n : idx1 + 1;
    }
}

// walk_run for a tile in the quadrant layout (tile_pivot): the four lanes l, l + 8,
// l + 16, l + 24 hold pivots a quarter turn apart, and since every ring has a multiple
// of four pixels they see ring r at the same fractional offset, with runs of the same
// length at the same offset from their own pivot, hence the same position angle at
// every step.  Each lane of a group computes the (folded) angle of one of every four
// steps and the group shares them by shuffles; every lane still sums its own pixels.
// The caller has checked runs_quad().
template <int M, bool FAST, bool SELF, class L>
__device__ __forceinline__ void walk_run_quad(const RingCtx& R, const L& ld, const LaneC& c, int a, int len,
                                              float2 (&acc)[M + 1], float& W, float& Q, float& QW, int mr = M) {
    const int maxlen = __reduce_max_sync(0xffffffffu, len);
    if (maxlen <= 0) return;
    const int lane = threadIdx.x & 31, j = lane >> 3, gb = lane & 7;
    const float i0 = (float)(a - c.cint);
    const float xneg = -c.cfrac * R.step, uneg = -c.cfrac * R.inv_n;
    const int last = max(len - 1, 0);
    int idx = wrap_idx(a, R.n);
    const auto row = ld.row(R.first);
    for (int t0 = 0; t0 < maxlen; t0 += 4) {
        Fold mine;
        {
            // steps past the run take its last offset, a valid direction (zero weight)
            const int tj = min(t0 + j, last);
            float cph, sph;
            pixel_dir<FAST>(i0 + (float)tj, xneg, uneg, R, cph, sph);
            mine = fold_angle(cph, sph);
        }
        // two steps at a time, so that only two shared angles are live
#pragma unroll
        for (int h = 0; h < 4; h += 2) {
            const Fold fa = shfl_fold(mine, gb + 8 * h), fb = shfl_fold(mine, gb + 8 * h + 8);
            const int i1 = idx + 1 >= R.n ? idx + 1 - R.n : idx + 1;
            // (the index test is a guard: a run's indices always lie within the ring)
            const bool ia = t0 + h < len && (unsigned)idx < (unsigned)R.n;
            const bool ib = t0 + h + 1 < len && (unsigned)i1 < (unsigned)R.n;
            const float2 va = ia ? row(idx) : make_float2(0.0f, 0.0f);
            const float2 vb = ib ? row(i1) : make_float2(0.0f, 0.0f);
            harmonics2f<M>(acc, fa, va.x, va.x, fb, vb.x, vb.x, mr);
            W += va.y + vb.y;
            if (SELF) {
                Q = fmaf(va.x, va.x, fmaf(vb.x, vb.x, Q));
                QW = fmaf(va.y, va.y, fmaf(vb.y, vb.y, QW));
            }
            idx = i1 + 1 >= R.n ? i1 + 1 - R.n : i1 + 1;
        }
    }
}

// True when each lane's run has the same offset from its pivot, the same length and
// the same fractional pivot position as the other three lanes of its quadrant group
// (an empty run matches any other empty run).  Every lane takes part in every shuffle.
__device__ __forceinline__ bool runs_quad(const LaneC& c, int a, int len) {
    const int gb = threadIdx.x & 7;
    const int rel = len > 0 ? a - c.cint : 0;
    const unsigned cf = __float_as_uint(c.cfrac);
    const int rel0 = __shfl_sync(0xffffffffu, rel, gb);
    const int len0 = __shfl_sync(0xffffffffu, len, gb);
    const unsigned cf0 = __shfl_sync(0xffffffffu, cf, gb);
    return __all_sync(0xffffffffu, rel == rel0 && len == len0 && cf == cf0);
}

// Walk the pixel pairs (p, mb - p), p in [a, a + len): mirror images about the
// pivot's meridian (belt rings with as many pixels as the pivot ring).  Two pairs
// (four pixels) per iteration; the same no-wrap fast loop as walk_run.
template <int M, bool FAST, bool SELF, class L>
__device__ __forceinline__ void walk_pairs(const RingCtx& R, const L& ld, const LaneC& c, int a, int len,
                                           int mb, float2 (&acc)[M + 1], float& W, float& Q,
                                           float& QW, int mr = M) {
    const int maxlen = __reduce_max_sync(0xffffffffu, len);
    if (maxlen <= 0) return;
    const float i0 = (float)(a - c.cint);
    const float xneg = -c.cfrac * R.step, uneg = -c.cfrac * R.inv_n;
    int ip = wrap_idx(a, R.n);
    int im_ = wrap_idx(mb - a, R.n);
    const auto row = ld.row(R.first);
    int t = 0;
    const int minlen = __reduce_min_sync(0xffffffffu, len);
    if (minlen >= 2 && __all_sync(0xffffffffu, ip + len <= R.n && im_ - len + 1 >= 0)) {
        float ft = i0;
        for (; t + 1 < minlen; t += 2, ft += 2.0f) {
            const float2 p0 = row(ip + t), m0 = row(im_ - t);
            const float2 p1 = row(ip + t + 1), m1 = row(im_ - t - 1);
            float ca, sa, cb, sb;
            pixel_dir<FAST>(ft, xneg, uneg, R, ca, sa);
            pixel_dir<FAST>(ft + 1.0f, xneg, uneg, R, cb, sb);
            harmonics2<M>(acc, ca, sa, p0.x + m0.x, p0.x - m0.x, cb, sb, p1.x + m1.x, p1.x - m1.x, mr);
            W += (p0.y + m0.y) + (p1.y + m1.y);
            if (SELF) {
                Q = fmaf(p0.x, p0.x, fmaf(m0.x, m0.x, fmaf(p1.x, p1.x, fmaf(m1.x, m1.x, Q))));
                QW = fmaf(p0.y, p0.y, fmaf(m0.y, m0.y, fmaf(p1.y, p1.y, fmaf(m1.y, m1.y, QW))));
            }
        }
        ip += t;
        if (ip >= R.n) ip -= R.n;
        im_ -= t;
        if (im_ < 0) im_ += R.n;
    }
    for (; t < maxlen; t += 2) {
        const bool on0 = t < len, on1 = t + 1 < len;
        const int ip1 = ip + 1 >= R.n ? ip + 1 - R.n : ip + 1;
        const int im1 = im_ - 1 < 0 ? im_ - 1 + R.n : im_ - 1;
        const float2 p0 = on0 ? row(ip) : make_float2(0.0f, 0.0f);
        const float2 m0 = on0 ? row(im_) : make_float2(0.0f, 0.0f);
        const float2 p1 = on1 ? row(ip1) : make_float2(0.0f, 0.0f);
        const float2 m1 = on1 ? row(im1) : make_float2(0.0f, 0.0f);
        const float oa = on0 ? i0 + (float)t : i0;
        const float ob = on1 ? i0 + (float)(t + 1) : i0;
        float ca, sa, cb, sb;
        pixel_dir<FAST>(oa, xneg, uneg, R, ca, sa);
        pixel_dir<FAST>(ob, xneg, uneg, R, cb, sb);
        harmonics2<M>(acc, ca, sa, p0.x + m0.x, p0.x - m0.x, cb, sb, p1.x + m1.x, p1.x - m1.x, mr);
        W += (p0.y + m0.y) + (p1.y + m1.y);
        if (SELF) {
            Q = fmaf(p0.x, p0.x, fmaf(m0.x, m0.x, fmaf(p1.x, p1.x, fmaf(m1.x, m1.x, Q))));
            QW = fmaf(p0.y, p0.y, fmaf(m0.y, m0.y, fmaf(p1.y, p1.y, fmaf(m1.y, m1.y, QW))));
        }
        ip = ip1 + 1 >= R.n ? ip1 + 1 - R.n : ip1 + 1;
        im_ = im1 - 1 < 0 ? im1 - 1 + R.n : im1 - 1;
    }
}

// walk_pairs for the case of a belt ring pair (the neighbour ring has as many pixels
// as the pivot ring): the 32 pivots of the tile then sit at the same fractional
// position relative to ring r, so every lane's run starts at the same offset from its
// own pivot and has the same length, and at step t all lanes see a neighbour at the
// same offset, hence the same position angle.  Each lane computes the (folded) angle of
// one step of a block of 32 and the warp shares them by shuffles, instead of every lane
// computing the same angle.  Lane l's pixels are those of lane 0 shifted by l, so the
// loads of a step stay coalesced.
template <int M, bool SELF, class L>
__device__ __forceinline__ void walk_pairs_shared(const RingCtx& R, const L& ld, const LaneC& c, int a, int len,
                                                  int mb, float2 (&acc)[M + 1], float& W, float& Q, float& QW,
                                                  int mr = M) {
    if (len <= 0) return;
    const int lane = threadIdx.x & 31;
    const float i0 = (float)(a - c.cint);
    const float xneg = -c.cfrac * R.step, uneg = -c.cfrac * R.inv_n;
    const auto row = ld.row(R.first);
    int ip = wrap_idx(a, R.n);
    int im_ = wrap_idx(mb - a, R.n);
    for (int t0 = 0; t0 < len; t0 += 32) {
        // this lane's step: t0 + lane
        Fold mine;
        {
            const float ft = i0 + (float)(t0 + lane);
            float cph, sph;
            if (fabsf(ft - c.cfrac) * R.step <= FAST_XMAX)
                pixel_dir<true>(ft, xneg, uneg, R, cph, sph);
            else
                pixel_dir<false>(ft, xneg, uneg, R, cph, sph);
            mine = fold_angle(cph, sph);
        }
        const int nstep = min(32, len - t0);
        int tt = 0;
        for (; tt + 1 < nstep; tt += 2) {
            const Fold fa = shfl_fold(mine, tt), fb = shfl_fold(mine, tt + 1);
            const int ip1 = ip + 1 >= R.n ? ip + 1 - R.n : ip + 1;
            const int im1 = im_ - 1 < 0 ? im_ - 1 + R.n : im_ - 1;
            const float2 p0 = row(ip), m0 = row(im_), p1 = row(ip1), m1 = row(im1);
            harmonics2f<M>(acc, fa, p0.x + m0.x, p0.x - m0.x, fb, p1.x + m1.x, p1.x - m1.x, mr);
            W += (p0.y + m0.y) + (p1.y + m1.y);
            if (SELF) {
                Q = fmaf(p0.x, p0.x, fmaf(m0.x, m0.x, fmaf(p1.x, p1.x, fmaf(m1.x, m1.x, Q))));
                QW = fmaf(p0.y, p0.y, fmaf(m0.y, m0.y, fmaf(p1.y, p1.y, fmaf(m1.y, m1.y, QW))));
            }
            ip = ip1 + 1 >= R.n ? ip1 + 1 - R.n : ip1 + 1;
            im_ = im1 - 1 < 0 ? im1 - 1 + R.n : im1 - 1;
        }
        if (tt < nstep) {
            const Fold fa = shfl_fold(mine, tt);
            const float2 p0 = row(ip), m0 = row(im_);
            harmonicsf<M>(acc, fa, p0.x + m0.x, p0.x - m0.x, mr);
            W += p0.y + m0.y;
            if (SELF) {
                Q = fmaf(p0.x, p0.x, fmaf(m0.x, m0.x, Q));
                QW = fmaf(p0.y, p0.y, fmaf(m0.y, m0.y, QW));
            }
            ip = ip + 1 >= R.n ? ip + 1 - R.n : ip + 1;
            im_ = im_ - 1 < 0 ? im_ - 1 + R.n : im_ - 1;
        }
    }
}

// True when every lane's run has lane 0's start offset and length (belt ring pairs).
__device__ __forceinline__ bool runs_shared(const LaneC& c, int a, int len) {
    const int rel = a - c.cint;
    const int rel0 = __shfl_sync(0xffffffffu, rel, 0), len0 = __shfl_sync(0xffffffffu, len, 0);
    const unsigned cf = __float_as_uint(c.cfrac), cf0 = __shfl_sync(0xffffffffu, cf, 0);
    return __all_sync(0xffffffffu, rel == rel0 && len == len0 && cf == cf0);
}

__device__ __forceinline__ RingCtx ring_ctx(const MapDev& g, const PivotRing& P, int r, long long pr) {
    RingCtx R;
    R.first = g.ring_first[r];
    R.n = g.ring_n[r];
    R.shift = g.ring_shift[r];
    R.s_r = g.ring_sf[r];
    R.s_lo = g.ring_sf_lo[r];
    const float2 Ap = g.pair_A[pr];
    R.A = Ap.x;
    R.A_lo = Ap.y;
    R.B = 2.0f * P.z_i * R.s_r;
    R.step = g.ring_step[r];
    R.step_lo = g.ring_step_lo[r];
    R.inv_n = g.ring_invn[r];
    R.invn_lo = g.ring_invn_lo[r];
    return R;
}

// Accumulate the bin-k moments of ring r into the lane's registers.
template <int M, bool SELF, class L>
__device__ __forceinline__ void fwd_ring_bin(const MapDev& g, const PivotRing& P, int r, int k, int q,
                                             const L& ld, float2 (&acc)[M + 1], float& W,
                                             float& Q, float& QW, int mr = M, bool quad = false) {
    const long long pr = P.pair0 + (r - P.rlo);
    const int2 Tk = g.pair_T[pr * (g.K + 1) + k];
    const int2 Tk1 = g.pair_T[pr * (g.K + 1) + k + 1];
    if (Tk.x == T_INF || Tk1.x == T_ZERO) return;  // no bin-k pixel on this ring
    const RingCtx R = ring_ctx(g, P, r, pr);
    const ExactCtx x = exact_ctx(g, P, r);
    const LaneC c = lane_c(q, P.s_i, P.n_i, R.shift, R.n);
    const bool sym = (R.n == P.n_i) && (Tk1.x != T_INF);
    const BinRuns b = bin_runs(c, Tk, Tk1, g.E[k], g.E[k + 1], x, R.n, sym);
    if (sym) {
        if (b.centre) {  // the pixel straight north or south of the pivot
            const float2 v = ld(R.first + wrap_idx(c.cint, R.n));
            float cph, sph;
            pixel_dir<false>(0.0f, 0.0f, -c.cfrac * R.inv_n, R, cph, sph);
            harmonics<M>(acc, cph, sph, v.x, v.x, mr);
            W += v.y;
            if (SELF) {
                Q = fmaf(v.x, v.x, Q);
                QW = fmaf(v.y, v.y, QW);
            }
        }
        if (runs_shared(c, b.a0, b.n0)) {
            walk_pairs_shared<M, SELF>(R, ld, c, b.a0, b.n0, b.mb, acc, W, Q, QW, mr);
            return;
        }
        const bool fast = __all_sync(0xffffffffu, run_omax(c, b.a0, b.n0) * R.step <= FAST_XMAX);
        if (fast)
            walk_pairs<M, true, SELF>(R, ld, c, b.a0, b.n0, b.mb, acc, W, Q, QW, mr);
        else
            walk_pairs<M, false, SELF>(R, ld, c, b.a0, b.n0, b.mb, acc, W, Q, QW, mr);
        return;
    }
    const float om = fmaxf(run_omax(c, b.a0, b.n0), run_omax(c, b.a1, b.n1));
    const bool fast = __all_sync(0xffffffffu, om * R.step <= FAST_XMAX);
    if (quad && runs_quad(c, b.a0, b.n0) && runs_quad(c, b.a1, b.n1)) {
        if (fast) {
            walk_run_quad<M, true, SELF>(R, ld, c, b.a0, b.n0, acc, W, Q, QW, mr);
            walk_run_quad<M, true, SELF>(R, ld, c, b.a1, b.n1, acc, W, Q, QW, mr);
        } else {
            walk_run_quad<M, false, SELF>(R, ld, c, b.a0, b.n0, acc, W, Q, QW, mr);
            walk_run_quad<M, false, SELF>(R, ld, c, b.a1, b.n1, acc, W, Q, QW, mr);
        }
        return;
    }
    if (fast) {
        walk_run<M, true, SELF>(R, ld, c, b.a0, b.n0, acc, W, Q, QW, mr);
        walk_run<M, true, SELF>(R, ld, c, b.a1, b.n1, acc, W, Q, QW, mr);
    } else {
        walk_run<M, false, SELF>(R, ld, c, b.a0, b.n0, acc, W, Q, QW, mr);
        walk_run<M, false, SELF>(R, ld, c, b.a1, b.n1, acc, W, Q, QW, mr);
    }

}

// Pivot of a lane in tile (ring i, start = 32 j).  Linear layout: q = start + lane.
// Quadrant layout (the forward kernels): q = 8 j + (lane & 7) + (lane >> 3) n_i / 4,
// four groups of eight consecutive pivots a quarter turn apart (walk_run_quad); a ring
// has ceil(n_i / 32) tiles either way.  `valid`: q is a pixel of the ring; lanes past
// the end take the geometry qg of the last pivot (of their quadrant), which keeps every
// unwrapped pixel index within [-n_r, 2 n_r).
struct TilePivot {
    int q, qg;
    bool valid;
};

__device__ __forceinline__ TilePivot tile_pivot(int start, int n_i, bool quad) {
    const int lane = threadIdx.x & 31;
    TilePivot t;
    if (quad) {
        const int quarter = n_i >> 2, qq = (start >> 2) + (lane & 7), off = (lane >> 3) * quarter;
        t.valid = qq < quarter;
        t.q = qq + off;
        t.qg = min(qq, quarter - 1) + off;
    } else {
        t.q = start + lane;
        t.valid = t.q < n_i;
        t.qg = min(t.q, n_i - 1);
    }
    return t;
}

// Where the tile's moments live in shared memory.  LayKM: A[k][m][re/im][32 pivots],
// W[k][32], Q[k][32], QW[k][32] (the FP32 contraction and the adjoint read this).
struct LayKM {
    float *sA, *sW, *sQ, *sQW;
    int M1;  // m_max + 1
    __device__ __forceinline__ float* a(int k, int m, int part, int lane) const {
        return sA + ((size_t)(k * M1 + m) * 2 + part) * TILE + lane;
    }
    __device__ __forceinline__ float* w(int k, int lane) const { return sW + k * TILE + lane; }
    __device__ __forceinline__ float* q(int k, int lane) const { return sQ + k * TILE + lane; }
    __device__ __forceinline__ float* qw(int k, int lane) const { return sQW + k * TILE + lane; }
};

// All warps of the CTA: accumulate the moments of the tile into shared memory.
// Smem must be zeroed beforehand; it is complete after the caller's __syncthreads().
template <int M, bool SELF, class L, class Lay>
__device__ __forceinline__ void tile_moments_l(const MapDev& g, const PivotRing& P, int q, const L& ld,
                                               const Lay& lay, int flush, int mr = M, bool quad = false) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = 0; k < g.K; ++k) {
        const int2 br = g.bin_range[(long long)P.i * g.K + k];
        if (br.x + warp > br.y) continue;
        float2 acc[M + 1];
#pragma unroll
        for (int m = 0; m <= M; ++m) acc[m] = make_float2(0.0f, 0.0f);
        float W = 0.0f, Q = 0.0f, QW = 0.0f;
        // Blocked summation: the registers sum `flush` rings, then the block is added into
        // shared memory, which keeps the running sums short.
        int nr = 0;
        for (int r = br.x + warp; r <= br.y; r += NWARPS) {
            fwd_ring_bin<M, SELF>(g, P, r, k, q, ld, acc, W, Q, QW, mr, quad);
            if (++nr == flush || r + NWARPS > br.y) {
                nr = 0;
#pragma unroll
                for (int m = 0; m <= M; ++m) {
                    if (m > mr) break;
                    atomicAdd(lay.a(k, m, 0, lane), acc[m].x);
                    atomicAdd(lay.a(k, m, 1, lane), acc[m].y);
                    acc[m] = make_float2(0.0f, 0.0f);
                }
                atomicAdd(lay.w(k, lane), W);
                W = 0.0f;
                if (SELF) {
                    atomicAdd(lay.q(k, lane), Q);
                    atomicAdd(lay.qw(k, lane), QW);
                    Q = 0.0f;
                    QW = 0.0f;
                }
            }
        }
    }
}

template <int M, bool SELF, class L>
__device__ __forceinline__ void tile_moments(const MapDev& g, const PivotRing& P, int q, const L& ld, float* sA,
                                             float* sW, float* sQ, float* sQW, int flush, int mr = M,
                                             bool quad = false) {
    tile_moments_l<M, SELF>(g, P, q, ld, LayKM{sA, sW, sQ, sQW, mr + 1}, flush, mr, quad);
}

// Per-pivot normalisation of the tile's moments (Sec. 3.1): each lane's a_m^k is
// divided by its bin weight W^k (NORM_BIN_MEAN) or by its total sum_k W^k
// (NORM_PIVOT_TOTAL), 0 where that weight is 0; W^k is then set to 1, so that the
// contraction's D entries become the tile's sum of pivot weights.  Layout of
// tile_moments (m-major within each bin, TILE lanes innermost).  Called by every
// thread of the CTA after the moments are complete (contains barriers).
template <int M>
__device__ __forceinline__ void tile_normalize(int K, float* sA, float* sW, int norm, int mr = M) {
    constexpr int PER = (TPCF_MAX_BINS * TILE + NTHREADS - 1) / NTHREADS;
    float inv[PER];
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int e = threadIdx.x + u * NTHREADS;
        float W = 0.0f;
        if (e < K * TILE) {
            if (norm == NORM_BIN_MEAN) {
                W = sW[e];
            } else {
                const int l = e & (TILE - 1);
                for (int k = 0; k < K; ++k) W += sW[k * TILE + l];
            }
        }
        inv[u] = W > 0.0f ? 1.0f / W : 0.0f;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int e = threadIdx.x + u * NTHREADS;
        if (e < K * TILE) {
            const int k = e / TILE, l = e & (TILE - 1);
            float* a = sA + (size_t)k * (mr + 1) * 2 * TILE + l;
            for (int j = 0; j < 2 * (mr + 1); ++j) a[j * TILE] *= inv[u];
            sW[e] = 1.0f;
        }
    }
    __syncthreads();
}

// Per-tile partial sums into the CTA's FP64 slot (eq. zetamEst2 summed over the
// tile's pivots).  Slot layout: for m, for pair (k1 <= k2): (Re S, Im S); then D for
// pairs; then sum_i w_i d_i Q^k(i) and sum_i w_i QW^k(i) for k.
template <int M>
__device__ __forceinline__ void tile_contract(int K, const float* sA, const float* sW, const float* sQ,
                                              const float* sQW, const float* sPiv, double* slot,
                                              bool self, int mr = M) {
    const int P = n_pairs_tri(K);
    const int nS = (mr + 1) * P;
    const float* wd = sPiv;
    const float* wt = sPiv + TILE;
    for (int e = threadIdx.x; e < nS + P + (self ? K : 0); e += NTHREADS) {
        if (e < nS) {
            const int m = e / P;
            const int pidx = e - m * P;
            int k2 = (int)((sqrtf(8.0f * pidx + 1.0f) - 1.0f) * 0.5f);
            while (k2 * (k2 + 1) / 2 > pidx) --k2;
            while ((k2 + 1) * (k2 + 2) / 2 <= pidx) ++k2;
            const int k1 = pidx - k2 * (k2 + 1) / 2;
            const float* r1 = sA + ((size_t)k1 * (mr + 1) + m) * 2 * TILE;
            const float* i1 = r1 + TILE;
            const float* r2 = sA + ((size_t)k2 * (mr + 1) + m) * 2 * TILE;
            const float* i2 = r2 + TILE;
            float sr = 0.0f, si = 0.0f;
            // start each thread at its own lane so a warp's 32 rows hit 32 banks
#pragma unroll 8
            for (int j = 0; j < TILE; ++j) {
                const int l = (j + threadIdx.x) & (TILE - 1);
                const float a = r1[l], b = i1[l], cc = r2[l], d = i2[l];
                sr = fmaf(wd[l], fmaf(a, cc, b * d), sr);
                si = fmaf(wd[l], fmaf(a, d, -b * cc), si);
            }
            red_add_f32(slot + 2 * e, sr);
            red_add_f32(slot + 2 * e + 1, si);
        } else if (e < nS + P) {
            const int pidx = e - nS;
            int k2 = (int)((sqrtf(8.0f * pidx + 1.0f) - 1.0f) * 0.5f);
            while (k2 * (k2 + 1) / 2 > pidx) --k2;
            while ((k2 + 1) * (k2 + 2) / 2 <= pidx) ++k2;
            const int k1 = pidx - k2 * (k2 + 1) / 2;
            float s = 0.0f;
#pragma unroll 8
            for (int j = 0; j < TILE; ++j) {
                const int l = (j + threadIdx.x) & (TILE - 1);
                s = fmaf(wt[l], sW[k1 * TILE + l] * sW[k2 * TILE + l], s);
            }
            red_add_f32(slot + nS + e, s);
        } else {
            const int k = e - nS - P;
            float s1 = 0.0f, s2 = 0.0f;
            for (int j = 0; j < TILE; ++j) {
                const int l = (j + threadIdx.x) & (TILE - 1);
                s1 = fmaf(wd[l], sQ[k * TILE + l], s1);
                s2 = fmaf(wt[l], sQW[k * TILE + l], s2);
            }
            red_add_f32(slot + 2 * nS + P + k, s1);
            red_add_f32(slot + 2 * nS + P + K + k, s2);
        }
    }
}


struct LayTC {
    float* sX;
    float *sQ, *sQW;
    int Rm, D0;
    __device__ __forceinline__ float* a(int k, int m, int part, int lane) const {
        return sX + kmaj(m * Rm + 2 * k + part, lane);
    }
    __device__ __forceinline__ float* w(int k, int lane) const { return sX + kmaj(D0 + k, lane); }
    __device__ __forceinline__ float* q(int k, int lane) const { return sQ + k * TILE + lane; }
    __device__ __forceinline__ float* qw(int k, int lane) const { return sQW + k * TILE + lane; }
};

// One forward tile: the moments of its 32 pivots, then their partial sums added to
// the CTA's slot.  Called by every thread of the CTA (contains barriers).
template <int M, bool SELF, bool DIRECT, bool GROUPED = false>
__device__ __forceinline__ void fwd_tile(const MapDev& g, const MapCall& c, int tile, double* slot, float* smem,
                                         int mr = M) {
    const int K = g.K;
    float* sA = smem;
    float* sW = sA + (size_t)K * (mr + 1) * 2 * TILE;
    float* sQ = sW + K * TILE;
    float* sQW = sQ + K * TILE;
    float* sPiv = sQW + K * TILE;
    const int lane = threadIdx.x & 31;
    const size_t nfl = tile_floats_rt(K, mr) - 2 * TILE;
    constexpr bool grouped = GROUPED;  // shared neighbour lists (c.group > 1): own instantiation
    const int2 tq = grouped ? c.gtiles[tile] : g.tiles[tile];
    if (tq.x < 0 || tq.x >= g.nrings) {
        if (threadIdx.x == 0) atomicOr(c.status, ST_BAD_TILE);
        __syncthreads();
        return;
    }
    const PivotRing P = pivot_ring(g, tq.x);
    float2 pv = make_float2(0.0f, 0.0f);
    int qg;  // the lane's geometry; lanes past the ring's end: zero weight, valid geometry
    if (grouped) {
        // shared neighbour lists: the lane stands for the run of c.group consecutive ring
        // pixels gi, sits at the run's middle pixel and carries the run's summed weights
        const int ng = (P.n_i + c.group - 1) / c.group;
        const int gi = tq.y + lane;
        const int s0 = min(gi, ng - 1) * c.group, ln = min(c.group, P.n_i - s0);
        qg = s0 + (ln - 1) / 2;
        if (gi < ng) {
            const long long f = g.ring_first[P.i] + s0;
            for (int u = 0; u < ln; ++u) {
                const long long pix = f + u;
                if (pix >= c.piv_lo && pix < c.piv_hi) {
                    const float2 v = DIRECT ? DirectLoad{c.delta, c.w}(pix) : c.wdw[pix];
                    pv.x += v.x;
                    pv.y += v.y;
                }
            }
        }
    } else {
        const TilePivot tp = tile_pivot(tq.y, P.n_i, c.quad != 0);
        const long long pix = g.ring_first[P.i] + tp.q;
        if (tp.valid && pix >= c.piv_lo && pix < c.piv_hi)
            pv = DIRECT ? DirectLoad{c.delta, c.w}(pix) : c.wdw[pix];
        qg = tp.qg;
    }
    if (!__syncthreads_or(pv.y != 0.0f)) return;
    for (size_t e = threadIdx.x; e < nfl; e += NTHREADS) sA[e] = 0.0f;
    if (threadIdx.x < TILE) {
        sPiv[lane] = pv.x;
        sPiv[TILE + lane] = pv.y;
    }
    __syncthreads();
    if (DIRECT)
        tile_moments<M, SELF>(g, P, qg, DirectLoad{c.delta, c.w}, sA, sW, sQ, sQW, c.flush, mr,
                              !grouped && c.quad);
    else
        tile_moments<M, SELF>(g, P, qg, PackedLoad{c.wdw}, sA, sW, sQ, sQW, c.flush, mr, !grouped && c.quad);
    __syncthreads();
    if (c.norm != NORM_NONE) tile_normalize<M>(K, sA, sW, c.norm, mr);
    tile_contract<M>(K, sA, sW, sQ, sQW, sPiv, slot, SELF && c.self_subtract, mr);
    __syncthreads();
}

// One forward tile with the tensor-core contraction: the moments accumulate in the
// tensor-core layout of tc_layout(), then tile_contract_tc.
template <int M, bool SELF>
__device__ __forceinline__ void fwd_tile_tc(const MapDev& g, const MapCall& c, int tile, double* slot, float* base,
                                            TcState& tc) {
    const int K = g.K;
    const int lane = threadIdx.x & 31;
    const int2 tq = g.tiles[tile];
    if (tq.x < 0 || tq.x >= g.nrings) {
        if (threadIdx.x == 0) atomicOr(c.status, ST_BAD_TILE);
        __syncthreads();
        return;
    }
    const PivotRing P = pivot_ring(g, tq.x);
    const TilePivot tp = tile_pivot(tq.y, P.n_i, c.quad != 0);
    const long long pix = g.ring_first[P.i] + tp.q;
    const bool in = tp.valid && pix >= c.piv_lo && pix < c.piv_hi;
    float2 pv = make_float2(0.0f, 0.0f);
    if (in) pv = c.wdw[pix];
    const int qg = tp.qg;
    if (!__syncthreads_or(pv.y != 0.0f)) return;
    {
        const TcLayout L = tc_layout(K, M, SELF);
        const int nx = (L.D0 + L.RD) * TILE;
        for (int e = threadIdx.x; e < nx; e += NTHREADS) base[e] = 0.0f;
        if (SELF)
            for (int e = threadIdx.x; e < 2 * K * TILE; e += NTHREADS) base[L.offQ + e] = 0.0f;
        if (threadIdx.x < TILE) {
            base[L.offPiv + lane] = pv.x;
            base[L.offPiv + TILE + lane] = pv.y;
        }
    }
    __syncthreads();
    {
        const int Rm = (2 * K + 7) & ~7, D0 = (M + 1) * Rm;
        const TcLayout L = tc_layout(K, M, SELF);
        tile_moments_l<M, SELF>(g, P, qg, PackedLoad{c.wdw}, LayTC{base, base + L.offQ, base + L.offQW, Rm, D0},
                                c.flush, M, c.quad != 0);
    }
    __syncthreads();
    tile_contract_tc<M, SELF, NTHREADS>(K, base, slot, tc, c.status);
    __syncthreads();
}

// OCC: CTAs per SM the register allocation is sized for (3: 80 registers, 2: 128);
// the autotuner picks the variant and the grid.
template <int M, bool SELF, bool DIRECT, int OCC = 3, bool GROUPED = false>
__global__ void __launch_bounds__(NTHREADS, OCC) map_tile_fwd_kernel(MapDev g, MapCall c) {
    extern __shared__ __align__(16) float smem[];
    __shared__ int s_tile;
    double* slot = c.slots + (size_t)blockIdx.x * n_entries(g.K, M);
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(c.counter, 1);
        __syncthreads();
        const long long tile = c.tile_lo + s_tile;
        if (tile >= c.tile_hi) break;
        fwd_tile<M, SELF, DIRECT, GROUPED>(g, c, (int)tile, slot, smem);
    }
}

// The forward with the tensor-core contraction (3 CTAs per SM where the shared
// memory allows it; 128 accumulator columns each, so at most 4 fit an SM's TMEM).
template <int M, bool SELF>
__global__ void __launch_bounds__(NTHREADS, 3) map_tile_tc_kernel(MapDev g, MapCall c) {
    extern __shared__ __align__(16) float smem_tc[];
    __shared__ int s_tile;
    __shared__ uint32_t s_tmem;
    __shared__ __align__(8) uint64_t s_mbar;
    __shared__ int s_fail;
    if (threadIdx.x == 0) s_fail = 0;
    tc_setup(&s_tmem, &s_mbar);
    TcState tc{s_tmem, smem_u32(&s_mbar), 0u, &s_fail};
    // the no-swizzle operand layout needs 16-byte alignment only
    float* base = smem_tc;
    double* slot = c.slots + (size_t)blockIdx.x * n_entries(g.K, M);
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(c.counter, 1);
        __syncthreads();
        const long long tile = c.tile_lo + s_tile;
        if (tile >= c.tile_hi || s_fail) break;
        fwd_tile_tc<M, SELF>(g, c, (int)tile, slot, base, tc);
    }
    tc_teardown(s_tmem);
}

// batch_fwd_kernel by tiles: the same queue over the members' tiles; a tile runs with its plan's
// shared-memory layout.
template <int M>
__global__ void __launch_bounds__(NTHREADS, 2) batch_tile_fwd_kernel(const BatchItem* __restrict__ items, int n,
                                                               long long total, unsigned long long* counter) {
    extern __shared__ __align__(16) float smem[];
    __shared__ long long s_t;
    __shared__ long long s_first[TPCF_MAX_BATCH + 1];
    for (int i = threadIdx.x; i <= n; i += NTHREADS) s_first[i] = i < n ? items[i].tile0 : total;
    __syncthreads();
    for (;;) {
        if (threadIdx.x == 0) s_t = (long long)atomicAdd(counter, 1ull);
        __syncthreads();
        const long long t = s_t;
        if (t >= total) break;
        int lo = 0, hi = n - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) / 2;
            if (s_first[mid] <= t) lo = mid; else hi = mid - 1;
        }
        const BatchItem& it = items[lo];
        double* slot = it.c.slots + (size_t)blockIdx.x * n_entries(it.g.K, it.g.M);
        fwd_tile<M, true, false>(it.g, it.c, (int)(t - s_first[lo]), slot, smem, it.g.M);
    }
}

// ------------------------------------------------------------ multi-field
// Three fields A, B, C on the same pixels (end of Sec. 2, after eq. ubEstimator): a
// tile accumulates the moments a^k(i; F), W^k(i; F) of every field F in its own block
// of shared memory (three passes of the single-field walk), then adds, over the
// cyclic permutations (P, X, Y) of (A, B, C),
//     S_m(k1,k2) += sum_i w^P_i P_i a_m^{k1}(i; X) conj(a_m^{k2}(i; Y)),
//     D(k1,k2)   += sum_i w^P_i W^{k1}(i; X) W^{k2}(i; Y),
// into the CTA's FP64 slot.  These sums are not Hermitian: the slot holds the full
// K x K matrices, for m, for (k1, k2): (Re S, Im S); then D for (k1, k2).
__host__ __device__ inline size_t multi_field_floats(int K, int M) { return (size_t)K * (M + 1) * 2 * TILE + (size_t)K * TILE; }
__host__ __device__ inline size_t multi_tile_floats(int K, int M) { return 3 * multi_field_floats(K, M) + 6 * TILE; }

template <int M>
__device__ __forceinline__ void tile_contract_multi(int K, const float* sF, const float* sPiv, double* slot) {
    const size_t fsz = multi_field_floats(K, M);
    const int KK = K * K;
    const int nS = (M + 1) * KK;
    const int cyc[3][3] = {{0, 1, 2}, {1, 2, 0}, {2, 0, 1}};
    for (int e = threadIdx.x; e < nS + KK; e += NTHREADS) {
        if (e < nS) {
            const int m = e / KK, r = e - m * KK, k1 = r / K, k2 = r - k1 * K;
            float sr = 0.0f, si = 0.0f;
#pragma unroll
            for (int t = 0; t < 3; ++t) {
                const float* wd = sPiv + cyc[t][0] * 2 * TILE;
                const float* r1 = sF + cyc[t][1] * fsz + ((size_t)k1 * (M + 1) + m) * 2 * TILE;
                const float* i1 = r1 + TILE;
                const float* r2 = sF + cyc[t][2] * fsz + ((size_t)k2 * (M + 1) + m) * 2 * TILE;
                const float* i2 = r2 + TILE;
#pragma unroll 8
                for (int j = 0; j < TILE; ++j) {
                    const int l = (j + threadIdx.x) & (TILE - 1);
                    const float a = r1[l], b = i1[l], cc = r2[l], d = i2[l];
                    sr = fmaf(wd[l], fmaf(a, cc, b * d), sr);
                    si = fmaf(wd[l], fmaf(a, d, -b * cc), si);
                }
            }
            red_add_f32(slot + 2 * e, sr);
            red_add_f32(slot + 2 * e + 1, si);
        } else {
            const int idx = e - nS, k1 = idx / K, k2 = idx - k1 * K;
            float sd = 0.0f;
#pragma unroll
            for (int t = 0; t < 3; ++t) {
                const float* wt = sPiv + cyc[t][0] * 2 * TILE + TILE;
                const float* W1 = sF + cyc[t][1] * fsz + (size_t)K * (M + 1) * 2 * TILE + k1 * TILE;
                const float* W2 = sF + cyc[t][2] * fsz + (size_t)K * (M + 1) * 2 * TILE + k2 * TILE;
                for (int j = 0; j < TILE; ++j) {
                    const int l = (j + threadIdx.x) & (TILE - 1);
                    sd = fmaf(wt[l], W1[l] * W2[l], sd);
                }
            }
            red_add_f32(slot + 2 * nS + idx, sd);
        }
    }
}

// The multi-field forward: c.wdw holds (w d, w) of field A, wdwB and wdwC those of
// B and C.
template <int M>
__global__ void __launch_bounds__(NTHREADS, 2) map_tile_multi_kernel(MapDev g, MapCall c,
                                                                     const float2* __restrict__ wdwB,
                                                                    const float2* __restrict__ wdwC) {
    extern __shared__ __align__(16) float smem[];
    __shared__ int s_tile;
    const int K = g.K;
    const size_t fsz = multi_field_floats(K, M);
    float* sF = smem;
    float* sPiv = smem + 3 * fsz;  // [field][w d, w][32]
    double* slot = c.slots + (size_t)blockIdx.x * n_entries_multi(K, M);
    const int lane = threadIdx.x & 31;
    const float2* arr[3] = {c.wdw, wdwB, wdwC};
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(c.counter, 1);
        __syncthreads();
        const long long tile = c.tile_lo + s_tile;
        if (tile >= c.tile_hi) break;
        const int2 tq = g.tiles[tile];
        if (tq.x < 0 || tq.x >= g.nrings) {
            if (threadIdx.x == 0) atomicOr(c.status, ST_BAD_TILE);
            __syncthreads();
            continue;
        }
        const PivotRing P = pivot_ring(g, tq.x);
        const TilePivot tp = tile_pivot(tq.y, P.n_i, true);
        const long long pix = g.ring_first[P.i] + tp.q;
        const bool in = tp.valid && pix >= c.piv_lo && pix < c.piv_hi;
        float2 pv[3];
        bool live = false;
#pragma unroll
        for (int f = 0; f < 3; ++f) {
            pv[f] = in ? arr[f][pix] : make_float2(0.0f, 0.0f);
            live = live || pv[f].y != 0.0f;
        }
        const int qg = tp.qg;
        if (!__syncthreads_or(live)) continue;
        for (size_t e = threadIdx.x; e < 3 * fsz; e += NTHREADS) sF[e] = 0.0f;
        if (threadIdx.x < TILE) {
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                sPiv[f * 2 * TILE + lane] = pv[f].x;
                sPiv[f * 2 * TILE + TILE + lane] = pv[f].y;
            }
        }
        __syncthreads();
        for (int f = 0; f < 3; ++f) {
            float* sA = sF + f * fsz;
            tile_moments<M, false>(g, P, qg, PackedLoad{arr[f]}, sA, sA + (size_t)K * (M + 1) * 2 * TILE, nullptr,
                                   nullptr, c.flush, M, true);
        }
        __syncthreads();
        tile_contract_multi<M>(K, sF, sPiv, slot);
        __syncthreads();
    }
}

// ------------------------------------------------------------------ adjoint
//
// dL/d d_p for L(zeta), with C_m = (dL/dRe zeta + i dL/dIm zeta) / D and
// H_m(k,k') = conj(C_m(k,k')) + C_m(k',k) (prepared by the host side):
//   primary term      w_p * (1/2) sum_{k,m} Re[a_m^k(p) h_m^k(p)]
//   neighbour legs    w_p * sum_{i: p in nbr(i)} w_i d_i sum_m Re[e^{-i m phi_ip} h_m^{k(ip)}(i)]
//   with h_m^k(i) = sum_{k'} H_m(k,k') conj(a_m^{k'}(i)).
// A tile recomputes its a (as the forward), turns it into h in place, then sweeps its
// neighbour rings again; each warp gathers its ring's contributions in a shared-memory
// row buffer and flushes the row to the gradient with one atomic add per pixel.


// val = sum_m (cos(m phi) hr_m + sin(m phi) hi_m): X the cosine part, Y the sine part.
// h[m] = (hr_m, hi_m); the (cos, sin) chains run packed, in the folded frame psi, by
// the recurrence of harmonics(); even and odd multipoles are summed apart and the odd
template <int M>
__device__ __forceinline__ void adj_harmonics(const float2 (&h)[M + 1], float cph, float sph, float& X, float& Y,
                                              int mr = M) {
    adj_harmonicsf<M>(h, fold_angle(cph, sph), X, Y, mr);
}

// Where the contribution to pixel p (unwrapped index on ring R) goes.
struct RowSink {
    float* buf;     // warp row buffer, or NULL for direct global adds
    int lo;         // buffer index = p - lo (window mode) ...
    bool whole;     // ... or = wrap(p) (whole-ring mode)
    float* grad;    // gradient row base (grad + first of ring)
    int n;
};

__device__ __forceinline__ void sink_add(const RowSink& s, int p_unwrapped, int p_wrapped, float v) {
    if (s.buf) {
        atomicAdd(s.buf + (s.whole ? p_wrapped : p_unwrapped - s.lo), v);
    } else {
        atomicAdd(s.grad + p_wrapped, v);
    }
}

template <int M>
__device__ __forceinline__ void adj_harmonics2f(const float2 (&h)[M + 1], const Fold& fa, const Fold& fb, float& Xa,
                                                float& Ya, float& Xb, float& Yb, int mr = M) {
    float2 eva = make_float2(h[0].x, 0.0f), evb = eva;
    float2 oda = make_float2(0.0f, 0.0f), odb = oda;
    float sga = 1.0f, sgb = 1.0f;
    if constexpr (M >= 1) {
        if (mr < 1) {
            Xa = Xb = eva.x;
            Ya = Yb = eva.y;
            return;
        }
        sga = fa.sg;
        sgb = fb.sg;
        float2 Ta = make_float2(fa.ac, fa.ss), Da = make_float2(0.5f * fa.lam, fa.ss);
        float2 Tb = make_float2(fb.ac, fb.ss), Db = make_float2(0.5f * fb.lam, fb.ss);
        const float2 La = make_float2(fa.lam, fa.lam), Lb = make_float2(fb.lam, fb.lam);
        oda = __ffma2_rn(Ta, h[1], oda);
        odb = __ffma2_rn(Tb, h[1], odb);
#pragma unroll
        for (int m = 2; m <= M; ++m) {
            if (m > mr) break;
            Da = __ffma2_rn(La, Ta, Da);
            Db = __ffma2_rn(Lb, Tb, Db);
            Ta = __fadd2_rn(Ta, Da);
            Tb = __fadd2_rn(Tb, Db);
            if (m & 1) {
                oda = __ffma2_rn(Ta, h[m], oda);
                odb = __ffma2_rn(Tb, h[m], odb);
            } else {
                eva = __ffma2_rn(Ta, h[m], eva);
                evb = __ffma2_rn(Tb, h[m], evb);
            }
        }
    }
    Xa = fmaf(sga, oda.x, eva.x);
    Ya = fmaf(sga, oda.y, eva.y);
    Xb = fmaf(sgb, odb.x, evb.x);
    Yb = fmaf(sgb, odb.y, evb.y);
}

template <int M>
__device__ __forceinline__ void adj_harmonics2(const float2 (&h)[M + 1], float ca, float sa, float cb, float sb,
                                               float& Xa, float& Ya, float& Xb, float& Yb, int mr = M) {
    adj_harmonics2f<M>(h, fold_angle(ca, sa), fold_angle(cb, sb), Xa, Ya, Xb, Yb, mr);
}

template <int M, bool FAST, bool SELF = false>
__device__ __forceinline__ void adj_run(const RingCtx& R, const float2* __restrict__ wdw, const LaneC& c,
                                        int a, int len, const float2 (&h)[M + 1], float wdi, const RowSink& s,
                                        float ck = 0.0f, int mr = M) {
    const int maxlen = __reduce_max_sync(0xffffffffu, len);
    const float i0 = (float)(a - c.cint);
    const float xneg = -c.cfrac * R.step, uneg = -c.cfrac * R.inv_n;
    int idx = wrap_idx(a, R.n);
    const float2* row = wdw + R.first;
    for (int t = 0; t < maxlen; t += 2) {
        const bool on0 = t < len, on1 = t + 1 < len;
        const int idx1 = idx + 1 >= R.n ? idx + 1 - R.n : idx + 1;
        const float2 v0 = on0 ? __ldg(row + idx) : make_float2(0.0f, 0.0f);
        const float2 v1 = on1 ? __ldg(row + idx1) : make_float2(0.0f, 0.0f);
        const float oa = on0 ? i0 + (float)t : i0;
        const float ob = on1 ? i0 + (float)(t + 1) : i0;
        float ca, sa, cb, sb, Xa, Ya, Xb, Yb;
        pixel_dir<FAST>(oa, xneg, uneg, R, ca, sa);
        pixel_dir<FAST>(ob, xneg, uneg, R, cb, sb);
        adj_harmonics2<M>(h, ca, sa, cb, sb, Xa, Ya, Xb, Yb, mr);
        if (SELF) {  // self-pair subtraction: -2 cdiag_k (w_p d_p) per neighbour p
            Xa = fmaf(ck, v0.x, Xa);
            Xb = fmaf(ck, v1.x, Xb);
        }
        if (on0) sink_add(s, a + t, idx, wdi * v0.y * (Xa + Ya));
        if (on1) sink_add(s, a + t + 1, idx1, wdi * v1.y * (Xb + Yb));
        idx = idx1 + 1 >= R.n ? idx1 + 1 - R.n : idx1 + 1;
    }
}

template <int M, bool FAST, bool SELF = false>
__device__ __forceinline__ void adj_pairs(const RingCtx& R, const float2* __restrict__ wdw, const LaneC& c,
                                          int a, int len, int mb, const float2 (&h)[M + 1], float wdi,
                                          const RowSink& s, float ck = 0.0f, int mr = M) {
    const int maxlen = __reduce_max_sync(0xffffffffu, len);
    const float i0 = (float)(a - c.cint);
    const float xneg = -c.cfrac * R.step, uneg = -c.cfrac * R.inv_n;
    int ip = wrap_idx(a, R.n);
    int im_ = wrap_idx(mb - a, R.n);
    const float2* row = wdw + R.first;
    for (int t = 0; t < maxlen; t += 2) {
        const bool on0 = t < len, on1 = t + 1 < len;
        const int ip1 = ip + 1 >= R.n ? ip + 1 - R.n : ip + 1;
        const int im1 = im_ - 1 < 0 ? im_ - 1 + R.n : im_ - 1;
        const float2 p0 = on0 ? __ldg(row + ip) : make_float2(0.0f, 0.0f);
        const float2 m0 = on0 ? __ldg(row + im_) : make_float2(0.0f, 0.0f);
        const float2 p1 = on1 ? __ldg(row + ip1) : make_float2(0.0f, 0.0f);
        const float2 m1 = on1 ? __ldg(row + im1) : make_float2(0.0f, 0.0f);
        const float oa = on0 ? i0 + (float)t : i0;
        const float ob = on1 ? i0 + (float)(t + 1) : i0;
        float ca, sa, cb, sb, Xa, Ya, Xb, Yb;
        pixel_dir<FAST>(oa, xneg, uneg, R, ca, sa);
        pixel_dir<FAST>(ob, xneg, uneg, R, cb, sb);
        adj_harmonics2<M>(h, ca, sa, cb, sb, Xa, Ya, Xb, Yb, mr);
        if (on0) {
            sink_add(s, a + t, ip, wdi * p0.y * (Xa + Ya + (SELF ? ck * p0.x : 0.0f)));
            sink_add(s, mb - a - t, im_, wdi * m0.y * (Xa - Ya + (SELF ? ck * m0.x : 0.0f)));
        }
        if (on1) {
            sink_add(s, a + t + 1, ip1, wdi * p1.y * (Xb + Yb + (SELF ? ck * p1.x : 0.0f)));
            sink_add(s, mb - a - t - 1, im1, wdi * m1.y * (Xb - Yb + (SELF ? ck * m1.x : 0.0f)));
        }
        ip = ip1 + 1 >= R.n ? ip1 + 1 - R.n : ip1 + 1;
        im_ = im1 - 1 < 0 ? im1 - 1 + R.n : im1 - 1;
    }
}

// adj_pairs for a belt ring pair, with the position angles shared across the warp
// (see walk_pairs_shared).
template <int M, bool SELF = false>
__device__ __forceinline__ void adj_pairs_shared(const RingCtx& R, const float2* __restrict__ wdw, const LaneC& c,
                                                 int a, int len, int mb, const float2 (&h)[M + 1], float wdi,
                                                 const RowSink& s, float ck = 0.0f, int mr = M) {
    if (len <= 0) return;
    const int lane = threadIdx.x & 31;
    const float i0 = (float)(a - c.cint);
    const float xneg = -c.cfrac * R.step, uneg = -c.cfrac * R.inv_n;
    int ip = wrap_idx(a, R.n);
    int im_ = wrap_idx(mb - a, R.n);
    const float2* row = wdw + R.first;
    for (int t0 = 0; t0 < len; t0 += 32) {
        Fold mine;
        {
            const float ft = i0 + (float)(t0 + lane);
            float cph, sph;
            if (fabsf(ft - c.cfrac) * R.step <= FAST_XMAX)
                pixel_dir<true>(ft, xneg, uneg, R, cph, sph);
            else
                pixel_dir<false>(ft, xneg, uneg, R, cph, sph);
            mine = fold_angle(cph, sph);
        }
        const int nstep = min(32, len - t0);
        for (int tt = 0; tt < nstep; tt += 2) {
            const int t = t0 + tt;
            const bool two = tt + 1 < nstep;
            const Fold fa = shfl_fold(mine, tt), fb = shfl_fold(mine, two ? tt + 1 : tt);
            const int ip1 = ip + 1 >= R.n ? ip + 1 - R.n : ip + 1;
            const int im1 = im_ - 1 < 0 ? im_ - 1 + R.n : im_ - 1;
            const float2 p0 = __ldg(row + ip), m0 = __ldg(row + im_);
            const float2 p1 = two ? __ldg(row + ip1) : make_float2(0.0f, 0.0f);
            const float2 m1 = two ? __ldg(row + im1) : make_float2(0.0f, 0.0f);
            float Xa, Ya, Xb, Yb;
            adj_harmonics2f<M>(h, fa, fb, Xa, Ya, Xb, Yb, mr);
            sink_add(s, a + t, ip, wdi * p0.y * (Xa + Ya + (SELF ? ck * p0.x : 0.0f)));
            sink_add(s, mb - a - t, im_, wdi * m0.y * (Xa - Ya + (SELF ? ck * m0.x : 0.0f)));
            if (two) {
                sink_add(s, a + t + 1, ip1, wdi * p1.y * (Xb + Yb + (SELF ? ck * p1.x : 0.0f)));
                sink_add(s, mb - a - t - 1, im1, wdi * m1.y * (Xb - Yb + (SELF ? ck * m1.x : 0.0f)));
            }
            ip = ip1 + 1 >= R.n ? ip1 + 1 - R.n : ip1 + 1;
            im_ = im1 - 1 < 0 ? im1 - 1 + R.n : im1 - 1;
        }
    }
}

// Neighbour legs of one ring r for the warp's lanes (all bins of r).
template <int M, bool SELF = false>
__device__ __forceinline__ void adj_ring(const MapDev& g, const PivotRing& P, int r, int q, float wdi,
                                         const float2* __restrict__ wdw, const float* sH, float* rowbuf,
                                         float* grad, int* status,
                                         const float* cdiag = nullptr, int mr = M) {
    const int lane = threadIdx.x & 31;
    const long long pr = P.pair0 + (r - P.rlo);
    const int2 TK = g.pair_T[pr * (g.K + 1) + g.K];
    if (TK.x == T_ZERO) return;
    const RingCtx R = ring_ctx(g, P, r, pr);
    const ExactCtx x = exact_ctx(g, P, r);
    const LaneC c = lane_c(q, P.s_i, P.n_i, R.shift, R.n);
    // row window: every pixel of r within the outer edge of some lane's pivot
    RowSink s;
    s.grad = grad + R.first;
    s.n = R.n;
    s.whole = false;
    s.lo = 0;
    s.buf = rowbuf;
    int width;
    {
        const int clo = __shfl_sync(0xffffffffu, c.cint, 0);
        const int chi = __shfl_sync(0xffffffffu, c.cint, 31);
        if (TK.x != T_INF) {
            s.lo = clo - TK.x - 2;
            width = chi + TK.x + 3 - s.lo + 1;
        } else {
            width = ROW + 1;
        }
        if (width > ROW || width >= R.n) {
            if (R.n <= ROW) {
                s.whole = true;
                width = R.n;
            } else {
                s.buf = nullptr;
                width = 0;
                if (lane == 0) atomicOr(status, ST_ROW_OVERFLOW);
            }
        }
    }
    for (int e = lane; e < width; e += 32) rowbuf[e] = 0.0f;
    __syncwarp();
    for (int k = 0; k < g.K; ++k) {
        const int2 br = g.bin_range[(long long)P.i * g.K + k];
        if (r < br.x || r > br.y) continue;
        const int2 Tk = g.pair_T[pr * (g.K + 1) + k];
        const int2 Tk1 = g.pair_T[pr * (g.K + 1) + k + 1];
        if (Tk.x == T_INF || Tk1.x == T_ZERO) continue;
        float2 h[M + 1];
        const float* hk = sH + (size_t)k * (mr + 1) * 2 * TILE;
#pragma unroll
        for (int m = 0; m <= M; ++m) {
            h[m] = m <= mr ? make_float2(hk[(2 * m) * TILE + lane], hk[(2 * m + 1) * TILE + lane])
                           : make_float2(0.0f, 0.0f);
        }
        const bool sym = (R.n == P.n_i) && (Tk1.x != T_INF);
        const BinRuns b = bin_runs(c, Tk, Tk1, g.E[k], g.E[k + 1], x, R.n, sym);
        const float ck = SELF ? -2.0f * cdiag[k] : 0.0f;
        if (sym) {
            if (b.centre) {
                const int p = c.cint;
                const int pw = wrap_idx(p, R.n);
                const float2 v = __ldg(wdw + R.first + pw);
                float cph, sph, X, Y;
                pixel_dir<false>(0.0f, 0.0f, -c.cfrac * R.inv_n, R, cph, sph);
                adj_harmonics<M>(h, cph, sph, X, Y, mr);
                if (SELF) X = fmaf(ck, v.x, X);
                sink_add(s, p, pw, wdi * v.y * (X + Y));
            }
            if (runs_shared(c, b.a0, b.n0)) {
                adj_pairs_shared<M, SELF>(R, wdw, c, b.a0, b.n0, b.mb, h, wdi, s, ck, mr);
            } else {
                const bool fast = __all_sync(0xffffffffu, run_omax(c, b.a0, b.n0) * R.step <= FAST_XMAX);
                if (fast)
                    adj_pairs<M, true, SELF>(R, wdw, c, b.a0, b.n0, b.mb, h, wdi, s, ck, mr);
                else
                    adj_pairs<M, false, SELF>(R, wdw, c, b.a0, b.n0, b.mb, h, wdi, s, ck, mr);
            }
        } else {
            const float om = fmaxf(run_omax(c, b.a0, b.n0), run_omax(c, b.a1, b.n1));
            const bool fast = __all_sync(0xffffffffu, om * R.step <= FAST_XMAX);
            if (fast) {
                adj_run<M, true, SELF>(R, wdw, c, b.a0, b.n0, h, wdi, s, ck, mr);
                adj_run<M, true, SELF>(R, wdw, c, b.a1, b.n1, h, wdi, s, ck, mr);
            } else {
                adj_run<M, false, SELF>(R, wdw, c, b.a0, b.n0, h, wdi, s, ck, mr);
                adj_run<M, false, SELF>(R, wdw, c, b.a1, b.n1, h, wdi, s, ck, mr);
            }
        }
    }
    __syncwarp();
    if (s.buf) {
        for (int e = lane; e < width; e += 32) {
            const float v = rowbuf[e];
            if (v != 0.0f) {
                const int pw = s.whole ? e : wrap_idx(s.lo + e, R.n);
                atomicAdd(s.grad + pw, v);
            }
        }
        __syncwarp();
    }
}

// One adjoint tile (all three phases).  Called by every thread of the CTA.  With
// SELF (self-pair subtraction) the subtracted diagonal adds, per bin k with
// cdiag_k = sum_m Re C_m(k,k), -w_p Q^k(p) cdiag_k to a pivot and
// -2 w_p^2 d_p w_i d_i cdiag_k to each neighbour p of pivot i.
template <int M, bool SELF = false>
__device__ __forceinline__ void bwd_tile(const MapDev& g, const MapCall& c, int tile, float* smem, int mr = M) {
    const int K = g.K;
    float* sA = smem;
    float* sW = sA + (size_t)K * (mr + 1) * 2 * TILE;
    float* sQ = sW + K * TILE;
    float* sQW = sQ + K * TILE;
    float* sPiv = sQW + K * TILE;
    float* sPrim = sPiv + 2 * TILE;
    float* sHm = sPrim + TILE;                  // [K][K][2] one m at a time
    float* sRow = sW;                           // [NWARPS][ROW], phase 3 only
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t nfl = (size_t)K * (mr + 1) * 2 * TILE + 3 * (size_t)K * TILE;

    const int2 tq = g.tiles[tile];
    if (tq.x < 0 || tq.x >= g.nrings) {
        if (threadIdx.x == 0) atomicOr(c.status, ST_BAD_TILE);
        __syncthreads();
        return;
    }
    const PivotRing P = pivot_ring(g, tq.x);
    const int q = tq.y + lane;
    const long long pix = g.ring_first[P.i] + q;
    const bool in = (q < P.n_i) && pix >= c.piv_lo && pix < c.piv_hi;
    const float2 pv = in ? c.wdw[pix] : make_float2(0.0f, 0.0f);
    const int qg = min(q, P.n_i - 1);  // (tile_pivot)
    if (!__syncthreads_or(pv.y != 0.0f)) return;  // no pivot with w != 0: no term
    for (size_t e = threadIdx.x; e < nfl; e += NTHREADS) sA[e] = 0.0f;
    if (threadIdx.x < TILE) {
        sPiv[lane] = pv.x;
        sPiv[TILE + lane] = pv.y;
        sPrim[lane] = 0.0f;
    }
    __syncthreads();
    // phase 1: the tile's moments, exactly as in the forward
    tile_moments<M, SELF>(g, P, qg, PackedLoad{c.wdw}, sA, sW, sQ, sQW, c.flush, mr);
    __syncthreads();
    // phase 2: h = H conj(a) per m, in place; primary term (1/2) sum Re[a h]
    for (int m = 0; m <= mr; ++m) {
        for (int e = threadIdx.x; e < K * K * 2; e += NTHREADS)
            sHm[e] = c.H[(size_t)m * K * K * 2 + e];
        __syncthreads();
        float hrv[(TPCF_MAX_BINS * TILE + NTHREADS - 1) / NTHREADS];
        float hiv[(TPCF_MAX_BINS * TILE + NTHREADS - 1) / NTHREADS];
        int nmine = 0;
        for (int e = threadIdx.x; e < K * TILE; e += NTHREADS, ++nmine) {
            const int k = e / TILE, l = e - k * TILE;
            float hr = 0.0f, hi = 0.0f;
            for (int kp = 0; kp < K; ++kp) {
                const float Hr = sHm[(k * K + kp) * 2], Hi = sHm[(k * K + kp) * 2 + 1];
                const float* ap = sA + ((size_t)kp * (mr + 1) + m) * 2 * TILE;
                const float tr = ap[l], ti = ap[TILE + l];
                hr = fmaf(Hr, tr, fmaf(-Hi, ti, hr));
                hi = fmaf(Hr, ti, fmaf(Hi, tr, hi));
            }
            const float* ak = sA + ((size_t)k * (mr + 1) + m) * 2 * TILE;
            atomicAdd(sPrim + l, fmaf(ak[l], hr, ak[TILE + l] * hi));
            hrv[nmine] = hr;
            hiv[nmine] = hi;
        }
        __syncthreads();
        nmine = 0;
        for (int e = threadIdx.x; e < K * TILE; e += NTHREADS, ++nmine) {
            const int k = e / TILE, l = e - k * TILE;
            float* ak = sA + ((size_t)k * (mr + 1) + m) * 2 * TILE;
            ak[l] = hrv[nmine];
            ak[TILE + l] = hiv[nmine];
        }
        __syncthreads();
    }
    const float* cdiag = SELF ? c.H + (size_t)(mr + 1) * K * K * 2 : nullptr;
    if (threadIdx.x < TILE && in) {
        float gp = 0.5f * pv.y * sPrim[lane];
        if (SELF) {
            float t = 0.0f;
            for (int k = 0; k < K; ++k) t = fmaf(cdiag[k], sQ[k * TILE + lane], t);
            gp = fmaf(-pv.y, t, gp);
        }
        if (gp != 0.0f) atomicAdd(c.grad + pix, gp);
    }
    __syncthreads();  // the row buffers of phase 3 overlay sPrim and the rest
    // phase 3: neighbour legs, warps split the neighbour rings
    const int2 rr = g.ring_range[P.i];
    for (int r = rr.x + warp; r <= rr.y; r += NWARPS)
        adj_ring<M, SELF>(g, P, r, qg, pv.x, c.wdw, sA, sRow + (size_t)warp * ROW, c.grad, c.status, cdiag, mr);
    __syncthreads();
}

template <int M, bool SELF, int OCC = 3>
__global__ void __launch_bounds__(NTHREADS, OCC) map_tile_bwd_kernel(MapDev g, MapCall c) {
    extern __shared__ __align__(16) float smem[];
    __shared__ int s_tile;
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(c.counter, 1);
        __syncthreads();
        const long long tile = c.tile_lo + s_tile;
        if (tile >= c.tile_hi) break;
        bwd_tile<M, SELF>(g, c, (int)tile, smem);
    }
}

template <int M>
__global__ void __launch_bounds__(NTHREADS, 2) batch_tile_bwd_kernel(const BatchItem* __restrict__ items, int n,
                                                               long long total, unsigned long long* counter) {
    extern __shared__ __align__(16) float smem[];
    __shared__ long long s_t;
    __shared__ long long s_first[TPCF_MAX_BATCH + 1];
    for (int i = threadIdx.x; i <= n; i += NTHREADS) s_first[i] = i < n ? items[i].tile0 : total;
    __syncthreads();
    for (;;) {
        if (threadIdx.x == 0) s_t = (long long)atomicAdd(counter, 1ull);
        __syncthreads();
        const long long t = s_t;
        if (t >= total) break;
        int lo = 0, hi = n - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) / 2;
            if (s_first[mid] <= t) lo = mid; else hi = mid - 1;
        }
        bwd_tile<M>(items[lo].g, items[lo].c, (int)(t - s_first[lo]), smem, items[lo].g.M);
    }
}

}  // namespace tpcf
