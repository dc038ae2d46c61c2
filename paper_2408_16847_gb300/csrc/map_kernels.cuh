// Map-path kernels of the binned harmonic 3PCF estimator (arXiv:2408.16847,
// section 3.1), templated on the largest multipole M.  Included by map_inst.cu,
// which is compiled once per M.
//
// What all map kernels share: positions of pivots and bin edges on a ring, the runs of a bin, the
// position angle of a neighbour and its harmonics, data access, and the tensor-core contraction; then the
// block kernels' entry points (map_block.cuh, map_block_bwd.cuh: large calls), the pair count, and the tile
// kernels (map_tile.cuh: small calls).
//   * on a neighbour ring the bin-k pixels of a pivot form at most two contiguous runs, found from
//     the per-ring-pair edge offsets T_e built by the plan (an exact ring-range disc query);
//   * within a run e^{-i m phi} comes from a trig-free recurrence in m (the harmonic step the paper
//     describes in Sec. 3.1 and 3.2, a few operations per m): Reinsch's stable form of the
//     three-term relation on the angle folded into |psi| <= pi/2, the cos and sin chains
//     packed into f32x2 FMAs (fold_angle, harmonicsf);
//   * a pivot's moments are contracted to sum_i w_i d_i a^{k1} conj(a^{k2}) (eq. zetamEst2) and
//     sum_i w_i W^{k1} W^{k2}, added in FP64 into a slot owned by the CTA.
#pragma once

#include <math.h>

#include "tpcf_internal.cuh"

namespace tpcf {

constexpr float AMBIGUITY = 1.0e-6f;  // > worst fp32 error of the edge position (~1.5e-7 px)
constexpr float FAST_XMAX = 0.25f;    // |half longitude offset| covered by the polynomial

// Fire-and-forget FP64 reduction of an fp32 partial sum into a CTA slot.  The float
// is widened by moving its IEEE 754 fields (exponent re-biased by 1023 - 127 = 896,
// mantissa shifted up by 52 - 23 = 29 bits), an exact conversion on the integer pipe:
// the FP64 pipe of this part runs at a few percent of the FP32 rate, and one
// conversion per slot entry and tile kept it half busy on small tiles.  Zeros add
// nothing and are skipped; subnormal, infinite and NaN values take the ordinary
// conversion.
__device__ __forceinline__ void red_add_f32(double* p, float x) {
    const unsigned u = __float_as_uint(x);
    if ((u & 0x7fffffffu) == 0u) return;
    const unsigned e = (u >> 23) & 0xffu;
    double d;
    if (e == 0u || e == 0xffu) {
        d = (double)x;
    } else {
        d = __longlong_as_double((long long)(((unsigned long long)(u >> 31) << 63) |
                                             ((unsigned long long)(e + 896u) << 52) |
                                             ((unsigned long long)(u & 0x7fffffu) << 29)));
    }
    atomicAdd(p, d);  // result unused: a reduction, no wait
}

// Position of the lane's pivot in units of ring-r pixels: c = cint + crem / den,
// so that pixel p of ring r is at longitude offset o = p - c pixels from the pivot.
struct LaneC {
    int cint, crem, den;
    float cfrac;
};

// floor(num / den) from an fp32 estimate corrected in exact integer arithmetic (the
// estimate is within one of the true quotient for the sizes used here).
__device__ __forceinline__ LaneC lane_c(int q, int s_i, int n_i, int s_r, int n_r) {
    if (n_r == n_i) {  // same pixel count: c = q + (s_i - s_r) / 2, no division
        LaneC c;
        const int d = s_i - s_r;  // -1, 0 or 1
        c.cint = q + (d < 0 ? -1 : 0);
        c.crem = d != 0 ? n_i : 0;
        c.den = 2 * n_i;
        c.cfrac = d != 0 ? 0.5f : 0.0f;
        return c;
    }
    const long long num = (long long)n_r * (2LL * q + s_i) - (long long)s_r * n_i;
    const int den = 2 * n_i;
    int ci = (int)floorf(__fdividef((float)num, (float)den));
    long long rem = num - (long long)ci * den;
    if (rem < 0) {
        --ci;
        rem += den;
    } else if (rem >= den) {
        ++ci;
        rem -= den;
    }
    LaneC c;
    c.cint = ci;
    c.crem = (int)rem;
    c.den = den;
    c.cfrac = __fdiv_rn((float)c.crem, (float)den);
    return c;
}

// The same in 32 bits, for pivots in the first half of their ring: n_r (2 q + 1) <= 16 nside^2 < 2^31.
__device__ __forceinline__ LaneC lane_c32(int q, int s_i, int n_i, int s_r, int n_r) {
    const int num = n_r * (2 * q + s_i) - s_r * n_i, den = 2 * n_i;
    int ci = (int)floorf(__fdividef((float)num, (float)den));
    int rem = num - ci * den;
    if (rem < 0) {
        --ci;
        rem += den;
    } else if (rem >= den) {
        ++ci;
        rem -= den;
    }
    LaneC c;
    c.cint = ci;
    c.crem = rem;
    c.den = den;
    c.cfrac = __fdiv_rn((float)rem, (float)den);
    return c;
}

// Exact (FP64) quarter squared chord of pixel p of ring r about the pivot:
// f = sin^2((theta_r - theta_i)/2) + s_i s_r sin^2(pi o / n_r).  Only evaluated for
// the rare edge pixels whose fp32 position is ambiguous, so the context holds the
// raw ring values and the FP64 trigonometry runs inside the rare branch.
struct ExactCtx {
    double th_i, th_r, s_i, s_r;
    int n_r;
};

static __device__ __noinline__ double exact_f(double th_i, double th_r, double s_i, double s_r, int n_r,
                                              int cint, int crem, int den, int p) {
    const double h = sin(0.5 * (th_r - th_i));
    const double o = (double)(p - cint) - (double)crem / (double)den;
    const double sp = sinpi(o / (double)n_r);
    return h * h + (s_i * s_r) * sp * sp;
}

// First pixel p (unwrapped index) with p - c >= T (T finite, positive).
__device__ __forceinline__ int pos_edge(const LaneC& c, int2 T, double Ee, const ExactCtx& x) {
    const float y = c.cfrac + __int_as_float(T.y);
    const float ry = rintf(y);
    const int base = c.cint + T.x;
    if (fabsf(y - ry) > AMBIGUITY) return base + (int)ceilf(y);
    const int ps = base + (int)ry;
    return (exact_f(x.th_i, x.th_r, x.s_i, x.s_r, x.n_r, c.cint, c.crem, c.den, ps) >= Ee) ? ps : ps + 1;
}

// Last pixel p with p - c <= -T.
__device__ __forceinline__ int neg_edge(const LaneC& c, int2 T, double Ee, const ExactCtx& x) {
    const float y = c.cfrac - __int_as_float(T.y);
    const float ry = rintf(y);
    const int base = c.cint - T.x;
    if (fabsf(y - ry) > AMBIGUITY) return base + (int)floorf(y);
    const int ps = base + (int)ry;
    return (exact_f(x.th_i, x.th_r, x.s_i, x.s_r, x.n_r, c.cint, c.crem, c.den, ps) >= Ee) ? ps : ps - 1;
}

// The same with the FP64 values of the rare ambiguous edges read only when needed: whether the
// pixel p lies at or beyond edge k + e of rings (i, r).
struct LazyEdge {
    const MapDev& g;
    int i, r, k;
    __device__ __forceinline__ bool beyond(const LaneC& c, int p, int e) const {
        return exact_f(g.ring_th[i], g.ring_th[r], g.ring_s[i], g.ring_s[r], g.ring_n[r], c.cint, c.crem, c.den, p) >=
               g.E[k + e];
    }
};

__device__ __forceinline__ int pos_edge(const LaneC& c, int2 T, const LazyEdge& x, int e) {
    const float y = c.cfrac + __int_as_float(T.y);
    const float ry = rintf(y);
    const int base = c.cint + T.x;
    if (fabsf(y - ry) > AMBIGUITY) return base + (int)ceilf(y);
    const int ps = base + (int)ry;
    return x.beyond(c, ps, e) ? ps : ps + 1;
}

__device__ __forceinline__ int neg_edge(const LaneC& c, int2 T, const LazyEdge& x, int e) {
    const float y = c.cfrac - __int_as_float(T.y);
    const float ry = rintf(y);
    const int base = c.cint - T.x;
    if (fabsf(y - ry) > AMBIGUITY) return base + (int)floorf(y);
    const int ps = base + (int)ry;
    return x.beyond(c, ps, e) ? ps : ps - 1;
}

// Warp-uniform description of neighbour ring r for pivot ring i.
struct RingCtx {
    long long first;
    int n, shift;
    float s_r, s_lo;      // sin(colatitude of r) as an unevaluated fp32 sum s_r + s_lo
    float A, A_lo;        // sin(theta_i - theta_r), likewise
    float B;              // 2 cos(theta_i) sin(theta_r)
    float step, step_lo;  // pi / n (half longitude step) as fp32 hi + lo
    float inv_n, invn_lo; // 1 / n likewise
};

// sin x and cos x for |x| <= FAST_XMAX from their Taylor series (truncation error
// below 2e-11 relative at the end of the range).
__device__ __forceinline__ void sin_cos_series(float x, float& s, float& c) {
    const float x2 = x * x;
    s = x * fmaf(x2, fmaf(x2, fmaf(x2, -1.98412698e-4f, 8.33333333e-3f), -1.66666667e-1f), 1.0f);
    c = fmaf(x2, fmaf(x2, fmaf(x2, fmaf(x2, 2.48015873e-5f, -1.38888889e-3f), 4.16666667e-2f), -0.5f),
             1.0f);
}

// Direction (cos phi, sin phi) of a neighbour at longitude offset o (ring-r pixels):
// with x = pi o / n (half the longitude difference),
//   east  component  E = s_r sin(2x)
//   north component  N = sin(theta_i - theta_r) + 2 cos(theta_i) s_r sin^2 x,
// the cancellation-free form of n_j . e_N(i); phi is measured from north to east.
// The per-ring constants carry a second fp32 word: their single-fp32 rounding is the
// same for every pixel of a ring and would shift phi coherently ring by ring.  The
// offset o = fi - cfrac is passed as its integer part fi (exact in fp32) and the run
// constants xneg = -cfrac pi/n, uneg = -cfrac/n, so x = pi o / n has one rounding.
template <bool FAST>
__device__ __forceinline__ void pixel_dir(float fi, float xneg, float uneg, const RingCtx& R, float& cph,
                                          float& sph) {
    float sx, cx;
    if (FAST) {
        sin_cos_series(fmaf(fi, R.step, fmaf(fi, R.step_lo, xneg)), sx, cx);
    } else {
        sincospif(fmaf(fi, R.inv_n, fmaf(fi, R.invn_lo, uneg)), &sx, &cx);
    }
    const float s2x = 2.0f * sx * cx;
    const float E = fmaf(R.s_r, s2x, R.s_lo * s2x);
    const float N = fmaf(R.B, sx * sx, R.A_lo) + R.A;
    // the floor only matters for the masked-out iterations of a run (zero weight),
    // which may sit on the pivot itself; real neighbours have N^2 + E^2 = sin^2 theta.
    const float rinv = rsqrtf(fmaxf(fmaf(N, N, E * E), 1e-30f));
    cph = N * rinv;
    sph = E * rinv;
}

// e^{-i m phi} for m = 0..M by Reinsch's modification of the three-term recurrence
// (as in Stoer & Bulirsch, Introduction to Numerical Analysis, chapter 1).  The plain
// Chebyshev recurrence cos((m+1)p) = 2 cos(p) cos(mp) - cos((m-1)p) only sees cos(p),
// which in fp32 loses the angle near p = 0 and pi (an error of roughly m eps/|sin p|)
// and amplifies its rounding like m^2 there.  Here the angle is first folded to
// psi = phi (cos phi >= 0) or phi - pi (cos phi < 0), so that cos psi = |cos phi|,
// sin psi = sigma sin phi with sigma = sign(cos phi), and e^{i m phi} = sigma^m e^{i m psi}.
// With lambda = 2 (cos psi - 1) = -2 sin^2 psi / (1 + cos psi) (no cancellation) and
// the differences D_m = X_m - X_{m-1}, the recurrence
//     D_{m+1} = D_m + lambda X_m,     X_{m+1} = X_m + D_{m+1}
// is the same three-term relation, but its rounding errors grow only about linearly
// in m for every |psi| <= pi/2.  The cosine and sine chains share lambda, so each step
// is one packed f32x2 FMA and one packed add on (cos part, sin part); the neighbour
// weights are folded into the start values, and the sigma^m sign is applied when the
// odd multipoles are accumulated (a packed FMA in place of the packed add).
struct Fold {
    float ac;   // |cos phi| = cos psi
    float ss;   // sigma sin phi = sin psi
    float sg;   // sigma
    float lam;  // 2 (cos psi - 1)
};

__device__ __forceinline__ Fold fold_angle(float cph, float sph) {
    Fold f;
    f.ac = fabsf(cph);
    f.sg = cph < 0.0f ? -1.0f : 1.0f;
    f.ss = f.sg * sph;
    f.lam = -2.0f * __fdividef(sph * sph, 1.0f + f.ac);
    return f;
}

// acc[m] += (wc cos(m phi), ws sin(m phi)), m = 0..M, from the folded angle.
// mr <= M: the multipoles computed (a runtime m_max below the compiled one).
template <int M>
__device__ __forceinline__ void harmonicsf(float2 (&acc)[M + 1], const Fold& f, float wc, float ws, int mr = M) {
    acc[0].x += wc;
    if constexpr (M >= 1) {
        if (mr < 1) return;
        float2 X = make_float2(wc * f.ac, ws * f.ss);           // X_1 (psi frame)
        float2 D = make_float2(0.5f * f.lam * wc, ws * f.ss);   // X_1 - X_0
        const float2 S2 = make_float2(f.sg, f.sg);
        const float2 L2 = make_float2(f.lam, f.lam);
        acc[1] = __ffma2_rn(S2, X, acc[1]);
#pragma unroll
        for (int m = 2; m <= M; ++m) {
            if (m > mr) break;
            D = __ffma2_rn(L2, X, D);
            X = __fadd2_rn(X, D);
            acc[m] = (m & 1) ? __ffma2_rn(S2, X, acc[m]) : __fadd2_rn(acc[m], X);
        }
    }
}

// p mod n for -n <= p < 2n (every unwrapped index of a run lies in that range).
__device__ __forceinline__ int wrap_idx(int p, int n) {
    return p < 0 ? p + n : (p >= n ? p - n : p);
}

// Neighbour data access: the packed (w d, w) array the library prepares, or the
// caller's delta and w read directly (used where no packing buffer may be allocated).
struct PackedLoad {
    const float2* __restrict__ p;
    __device__ __forceinline__ float2 operator()(long long i) const { return __ldg(p + i); }
    // accessor of one ring's pixels (index relative to the ring's first pixel)
    struct Row {
        const float2* __restrict__ p;
        __device__ __forceinline__ float2 operator()(int i) const { return __ldg(p + i); }
    };
    __device__ __forceinline__ Row row(long long first) const { return Row{p + first}; }
};
struct DirectLoad {
    const float* __restrict__ d;
    const float* __restrict__ w;
    __device__ __forceinline__ float2 operator()(long long i) const {
        const float wi = __ldg(w + i);
        return make_float2(wi * __ldg(d + i), wi);
    }
    struct Row {
        const float* __restrict__ d;
        const float* __restrict__ w;
        __device__ __forceinline__ float2 operator()(int i) const {
            const float wi = __ldg(w + i);
            return make_float2(wi * __ldg(d + i), wi);
        }
    };
    __device__ __forceinline__ Row row(long long first) const { return Row{d + first, w + first}; }
};

// Runs of bin k on ring r for the lane's pivot.  Fills up to two runs (a, len) and,
// in mirror mode, one pair run plus an optional centre pixel.
struct BinRuns {
    int a0, n0, a1, n1;  // plain runs
    bool sym;            // pair mode: pairs (p, mb - p), p in [a0, a0 + n0)
    int mb;              // mirror base
    bool centre;         // pixel cint (offset 0) also belongs to the bin (pair mode)
};

__device__ __forceinline__ BinRuns bin_runs(const LaneC& c, int2 Tk, int2 Tk1, double Ek, double Ek1,
                                            const ExactCtx& x, int n_r, bool sym) {
    BinRuns b;
    b.sym = sym;
    b.centre = false;
    b.mb = 0;
    b.a1 = 0;
    b.n1 = 0;
    // upper end of the + side, lower end of the - side
    int pe, ns;
    if (Tk1.x == T_INF) {
        pe = c.cint + n_r / 2;
        ns = c.cint - n_r / 2 + 1;
    } else {
        pe = pos_edge(c, Tk1, Ek1, x) - 1;
        ns = neg_edge(c, Tk1, Ek1, x) + 1;
    }
    if (sym) {
        int a;
        if (Tk.x == T_ZERO) {
            a = c.cint + 1;
            b.centre = (c.crem == 0);
        } else {
            a = pos_edge(c, Tk, Ek, x);
        }
        b.a0 = a;
        b.n0 = max(0, pe - a + 1);
        b.mb = 2 * c.cint + (c.crem != 0 ? 1 : 0);
        return b;
    }
    if (Tk.x == T_ZERO) {
        b.a0 = ns;
        b.n0 = max(0, pe - ns + 1);
    } else {
        const int pa = pos_edge(c, Tk, Ek, x);
        const int nb = neg_edge(c, Tk, Ek, x);
        b.a0 = pa;
        b.n0 = max(0, pe - pa + 1);
        b.a1 = ns;
        b.n1 = max(0, nb - ns + 1);
    }
    return b;
}

// The plain runs (two at most) of bin k, edges decided with LazyEdge.
__device__ __forceinline__ BinRuns bin_runs(const LaneC& c, int2 Tk, int2 Tk1, const LazyEdge& x, int n_r) {
    BinRuns b;
    b.sym = b.centre = false;
    b.mb = b.a1 = b.n1 = 0;
    const int pe = Tk1.x == T_INF ? c.cint + n_r / 2 : pos_edge(c, Tk1, x, 1) - 1;
    const int ns = Tk1.x == T_INF ? c.cint - n_r / 2 + 1 : neg_edge(c, Tk1, x, 1) + 1;
    if (Tk.x == T_ZERO) {
        b.a0 = ns;
        b.n0 = max(0, pe - ns + 1);
    } else {
        b.a0 = pos_edge(c, Tk, x, 0);
        b.n0 = max(0, pe - b.a0 + 1);
        b.a1 = ns;
        b.n1 = max(0, neg_edge(c, Tk, x, 0) - ns + 1);
    }
    return b;
}

// Largest |o| a run reaches, for the FAST test.
__device__ __forceinline__ float run_omax(const LaneC& c, int a, int len) {
    if (len <= 0) return 0.0f;
    const float o0 = (float)(a - c.cint) - c.cfrac;
    return fmaxf(fabsf(o0), fabsf(o0 + (float)(len - 1)));
}

// Everything a warp needs about pivot ring i.
struct PivotRing {
    int i, n_i, s_i;
    float z_i;
    double th_i, s_i_d;
    int rlo;
    long long pair0;
};

__device__ __forceinline__ ExactCtx exact_ctx(const MapDev& g, const PivotRing& P, int r) {
    ExactCtx x;
    x.th_i = P.th_i;
    x.th_r = g.ring_th[r];
    x.s_i = P.s_i_d;
    x.s_r = g.ring_s[r];
    x.n_r = g.ring_n[r];
    return x;
}

// Load the tile's pivot description; returns false if no lane has w != 0.
__device__ __forceinline__ PivotRing pivot_ring(const MapDev& g, int i) {
    PivotRing P;
    P.i = i;
    P.n_i = g.ring_n[i];
    P.s_i = g.ring_shift[i];
    P.z_i = g.ring_zf[i];
    P.th_i = g.ring_th[i];
    P.s_i_d = g.ring_s[i];
    P.rlo = g.ring_range[i].x;
    P.pair0 = g.pair_off[i];
    return P;
}

// Block (b1 <= b2) number i of the CB x CB blocks of a triangle, columns first.
__device__ __forceinline__ void tri_block(int i, int& b1, int& b2) {
    b2 = (int)((sqrtf(8.0f * i + 1.0f) - 1.0f) * 0.5f);
    while (b2 * (b2 + 1) / 2 > i) --b2;
    while ((b2 + 1) * (b2 + 2) / 2 <= i) ++b2;
    b1 = i - b2 * (b2 + 1) / 2;
}

constexpr int CB = 4;  // bins on a side of a block of the contraction

// ------------------------------------------------- tensor-core contraction (TF32x3)
// The contraction of eq. zetamEst2 over a tile's 32 pivots is, for each m, the Gram
// matrix G = X diag(w d) X^T of X = [Re a ; Im a] (rows r = 2k + part, 32 pivot
// columns): S_m(k1,k2) = G[2k1][2k2] + G[2k1+1][2k2+1] + i (G[2k1][2k2+1] - G[2k1+1][2k2])
// in the convention a = re - i im; D is the Gram matrix of the W^k rows with the
// weights w.  On the 5th-generation tensor cores (kind::tf32, FP32 accumulation in
// tensor memory), per block of rows (each m, then the W block):
//   * the moments are staged from the workspace in the layout the MMA reads (K-major,
//     no swizzle: 8-row x 16-byte core matrices, pivot-adjacent ones 128 B apart,
//     8-row groups 1024 B apart, blocks starting on a row group);
//   * with Y = X diag(sqrt|w d|) and s = sign(w d), G = Y diag(s) Y^T.  Y is split into
//     a tf32 part hi (its low 13 mantissa bits cleared, written back in place) and
//     the fp32 remainder lo, and G = hi s hi^T + C + C^T with C = hi s lo^T (the
//     dropped lo s lo^T term is below 2^-22 relative): two MMAs per 8-pivot step,
//     A = hi in place, B = s hi and s lo in a small staging buffer;
//   * the MMA is 128 x N; rows of A beyond the block come from the following shared
//     memory and only reach accumulator rows that are never read;
//   * one thread issues, an mbarrier tracks completion (bounded wait), warps 0-1 read
//     the two accumulators back, C^T goes through shared memory, and S (or D) is added
//     into the CTA's FP64 slot.
constexpr int TC_TMEM_COLS = 128;  // two accumulators of up to 64 columns
constexpr int ST_TC_TIMEOUT = ST_TC_TIMEOUT_BIT;

// Shared-memory plan of the tensor-core forward tile (in floats from the dynamic
// shared memory base; blocks start on 8-row groups).
struct TcLayout {
    int Rm, RD, NBm, NBd;  // rows per m block and of the W block; MMA N of each
    int x0, D0;            // first row of the moments; first row of the W block
    int offB, offPiv, offSc, offQ, offQW;
    int total;             // floats
};

__host__ __device__ inline TcLayout tc_layout(int K, int M, bool self) {
    TcLayout L;
    L.Rm = (2 * K + 7) & ~7;
    L.RD = (K + 7) & ~7;
    L.NBm = (2 * K + 15) & ~15;
    L.NBd = (K + 15) & ~15;
    L.x0 = 0;
    L.D0 = (M + 1) * L.Rm;
    int off = (L.D0 + L.RD) * TILE;
    L.offPiv = off;  // (w d, w) of the pivots
    off += 2 * TILE;
    L.offSc = off;  // sqrt|w d|, sign(w d), sqrt w
    off += 3 * TILE;
    L.offQ = off;
    L.offQW = off + (self ? K * TILE : 0);
    if (self) off += 2 * K * TILE;
    L.offB = off;  // B hi rows, then B lo rows (NBm each); reused for the C^T staging
    off += 2 * L.NBm * TILE;
    // the MMA of the last block reads 128 rows from its start
    const int need = (L.D0 + 128) * TILE;
    L.total = off > need ? off : need;
    return L;
}

// bytes of dynamic shared memory of the tile and of the block kernel
__host__ __device__ inline size_t tc_tile_bytes(int K, int M, bool self) {
    return (size_t)tc_layout(K, M, self).total * sizeof(float);
}
__host__ __device__ inline size_t tc_smem_bytes(int K, int M, bool self) {
    const size_t a = tc_tile_bytes(K, M, self), b = block_smem_bytes(M);
    return a > b ? a : b;
}

// Position of (row r, pivot p) in the K-major canonical layout without swizzle: core
// matrices of 8 rows x 4 pivots (128 contiguous bytes, rows 16 B apart), the 8
// pivot-adjacent core matrices of a row group 128 B apart, row groups 1024 B apart.
__device__ __forceinline__ int kmaj(int r, int p) { return ((r >> 3) << 8) + ((p >> 2) << 5) + ((r & 7) << 2) + (p & 3); }

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// UMMA shared-memory descriptor, K-major without swizzle: start address, leading
// (pivot-direction) core-matrix offset 128 B, row-group stride 1024 B, descriptor
// version 1.
__device__ __forceinline__ uint64_t tc_sdesc(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(128u >> 4) << 16) | ((uint64_t)(1024u >> 4) << 32) |
           (1ull << 46);
}

// Instruction descriptor: D f32, A and B tf32, both K-major, N, M = 128.
__device__ __forceinline__ uint32_t tc_idesc(int N) {
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, int acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc));
}

// Waits for the mbarrier phase; false after about one second (error path).
__device__ __forceinline__ bool tc_wait(uint32_t mbar, uint32_t phase) {
    uint64_t t0;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    for (;;) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done)
            : "r"(mbar), "r"(phase)
            : "memory");
        if (done) return true;
        uint64_t t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t - t0 > 1000000000ull) return false;
    }
}

__device__ __forceinline__ void tc_ld8(uint32_t taddr, float (&v)[8]) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// Per-CTA tensor-core state: TMEM accumulator base, mbarrier and its phase.
struct TcState {
    uint32_t tmem;
    uint32_t mbar;    // shared address of the mbarrier
    uint32_t phase;
    int* fail;        // shared flag: a wait gave up
};

// Warp 0 allocates the accumulator columns; thread 0 initialises the mbarrier.
__device__ __forceinline__ void tc_setup(uint32_t* s_tmem, uint64_t* s_mbar) {
    if ((threadIdx.x >> 5) == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)),
                     "r"(TC_TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(s_mbar)));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tc_teardown(uint32_t tmem) {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if ((threadIdx.x >> 5) == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC_TMEM_COLS));
}

// The tile's S and D partial sums on the tensor cores (see above); the self-pair
// diagonals stay on the FP32 pipe.  Called by every thread; the moments in sX are
// consumed (truncated in place).
template <int M, bool SELF, int NT>
__device__ void tile_contract_tc(int K, float* base, double* slot, TcState& tc, int* status) {
    const TcLayout L = tc_layout(K, M, SELF);
    const int P = n_pairs_tri(K);
    const int nS = (M + 1) * P;
    float* sX = base;
    float* Bhi = base + L.offB;
    const float* sPiv = base + L.offPiv;
    float* sc = base + L.offSc;  // [0] sqrt|w d|, [1] sign(w d), [2] sqrt w
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x < TILE) {
        const float wd = sPiv[lane], w = sPiv[TILE + lane];
        sc[lane] = sqrtf(fabsf(wd));
        sc[TILE + lane] = wd < 0.0f ? -1.0f : 1.0f;
        sc[2 * TILE + lane] = sqrtf(w);
    }
    __syncthreads();
    for (int b = 0; b <= M + 1; ++b) {
        const bool isD = b == M + 1;
        const int rows = isD ? K : 2 * K;
        const int N = isD ? L.NBd : L.NBm;
        const int r0 = isD ? L.D0 : b * L.Rm;
        float* Blo = Bhi + N * TILE;
        // split the block: hi in place, (s hi, s lo) into the staging rows; rows of B
        // beyond the block are zero.  e runs over the layout in memory order (row group,
        // pivot chunk, row in group, pivot in chunk); r0 is a multiple of 8, so the
        // block's element e sits at sX[r0 * 32 + e] and B's at B[e].
        for (int e = threadIdx.x; e < N * TILE; e += NT) {
            const int i = ((e >> 8) << 3) + ((e >> 2) & 7);
            const int p = (((e >> 5) & 7) << 2) + (e & 3);
            float bh = 0.0f, bl = 0.0f;
            if (i < rows) {
                const float x = sX[r0 * TILE + e] * (isD ? sc[2 * TILE + p] : sc[p]);
                const float hi = __uint_as_float(__float_as_uint(x) & 0xFFFFE000u);
                const float sg = isD ? 1.0f : sc[TILE + p];
                sX[r0 * TILE + e] = hi;
                bh = sg * hi;
                bl = sg * (x - hi);
            }
            Bhi[e] = bh;
            Blo[e] = bl;
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (threadIdx.x == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t idesc = tc_idesc(N);
            const uint32_t a0 = smem_u32(sX + r0 * TILE), bh = smem_u32(Bhi), bl = smem_u32(Blo);
#pragma unroll
            for (int k8 = 0; k8 < TILE / 8; ++k8) {
                const uint32_t o = (uint32_t)k8 * 256u;  // 8 tf32 pivots = two core matrices per MMA
                tc_mma(tc.tmem, tc_sdesc(a0 + o), tc_sdesc(bh + o), idesc, k8 > 0);
                tc_mma(tc.tmem + (uint32_t)L.NBm, tc_sdesc(a0 + o), tc_sdesc(bl + o), idesc, k8 > 0);
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             tc.mbar)
                         : "memory");
            if (!tc_wait(tc.mbar, tc.phase)) {
                *tc.fail = 1;
                atomicOr(status, ST_TC_TIMEOUT);
            }
        }
        tc.phase ^= 1u;
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (*tc.fail) return;
        // C rows into the staging area (the B rows are no longer read): Cst[r][c]
        float* Cst = Bhi;
        const int r = warp * 32 + lane;
        if (warp * 32 < rows) {
            for (int c0 = 0; c0 < N; c0 += 8) {
                float v[8];
                tc_ld8(tc.tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(L.NBm + c0), v);
                if (r < rows) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) Cst[r * N + c0 + j] = v[j];
                }
            }
        }
        __syncthreads();
        if (warp * 32 < rows) {
            for (int c0 = 0; c0 < N; c0 += 8) {
                float gv[8];
                tc_ld8(tc.tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, gv);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int s2 = c0 + j;
                    if (r < rows && s2 < rows) gv[j] += Cst[r * N + s2] + Cst[s2 * N + r];
                }
                if (isD) {
                    if (r < K) {
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const int k2 = c0 + j;
                            if (k2 >= r && k2 < K) red_add_f32(slot + 2 * nS + k2 * (k2 + 1) / 2 + r, gv[j]);
                        }
                    }
                } else {
                    float u[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) u[j] = __shfl_down_sync(0xffffffffu, gv[j], 1);
                    if ((r & 1) == 0 && r < rows) {
                        const int k1 = r >> 1;
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int k2 = (c0 >> 1) + j;
                            if (k2 >= k1 && k2 < K) {
                                const int e = b * P + k2 * (k2 + 1) / 2 + k1;
                                red_add_f32(slot + 2 * e, (gv[2 * j] + u[2 * j + 1]));
                                red_add_f32(slot + 2 * e + 1, (gv[2 * j + 1] - u[2 * j]));
                            }
                        }
                    }
                }
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
    }
    if (SELF) {
        const float* wd = sPiv;
        const float* wt = sPiv + TILE;
        const float* sQ = base + L.offQ;
        const float* sQW = base + L.offQW;
        for (int k = threadIdx.x; k < K; k += NT) {
            float s1 = 0.0f, s2 = 0.0f;
            for (int j = 0; j < TILE; ++j) {
                s1 = fmaf(wd[j], sQ[k * TILE + j], s1);
                s2 = fmaf(wt[j], sQW[k * TILE + j], s2);
            }
            red_add_f32(slot + 2 * nS + P + k, s1);
            red_add_f32(slot + 2 * nS + P + K + k, s2);
        }
    }
}

}  // namespace tpcf

#include "map_block.cuh"
#include "map_block_bwd.cuh"

namespace tpcf {

// One work item of the forward with the tensor-core contraction: the block's moments as in
// fwd_block, then each live subtile is brought into the layout of tc_layout() and
// contracted by tile_contract_tc.
template <int M, bool SELF>
__device__ __forceinline__ void fwd_block_tc(const MapDev& g, const MapCall& c, long long b, int part, float* ws,
                                             double* slot, float* base, TcState& tc) {
    const int K = g.K, lane = threadIdx.x & 31;
    const Block<M, false> B(g, c, b);
    const size_t sub_floats = sub_floats_rt(K, M, SELF);
    const PackedLoad ld{c.wdw};
    auto value = [&](int s, int l) { return B.value(g, c, ld, s, l); };
    const unsigned live = block_live(B.nsub, [&](int s, int l) { return value(s, l).y != 0.0f; });
    if (live == 0u) return;
    block_moments<M, SELF, false>(g, c, b, live, part, ld, ws, sub_floats, reinterpret_cast<char*>(base), M);
    if (!block_complete(c, b)) return;
    block_fold(c, b, B.nsub, ws, sub_floats);
    const TcLayout L = tc_layout(K, M, SELF);
    for (int s = 0; s < B.nsub; ++s) {
        if (!((live >> s) & 1u)) continue;
        const float* sub = ws + (size_t)s * sub_floats;
        const float* W = sub + (size_t)(M + 1) * K * 2 * TILE;
        // every row of the layout: rows beyond a block's 2 K (or K) are zero
        for (int r = threadIdx.x >> 5; r < L.D0 + L.RD; r += BW) {
            float v = 0.0f;
            if (r < L.D0) {
                const int m = r / L.Rm, i = r - m * L.Rm;
                if (i < 2 * K) v = __ldcg(sub + ((size_t)m * 2 * K + i) * TILE + lane);
            } else if (r - L.D0 < K) {
                v = __ldcg(W + (r - L.D0) * TILE + lane);
            }
            base[kmaj(r, lane)] = v;
        }
        if (SELF)
            for (int e = threadIdx.x; e < 2 * K * TILE; e += BT) base[L.offQ + e] = __ldcg(W + K * TILE + e);
        if (threadIdx.x < TILE) {
            const float2 v = value(s, lane);
            base[L.offPiv + lane] = v.x;
            base[L.offPiv + TILE + lane] = v.y;
        }
        __syncthreads();
        tile_contract_tc<M, SELF, BT>(K, base, slot, tc, c.status);
        __syncthreads();
        if (*tc.fail) return;
    }
}

// Persistent CTAs draw work items (block, part) from a counter.
template <int M, bool SELF, bool GROUPED = false>
__global__ void __launch_bounds__(BT, 4) map_fwd_kernel(MapDev g, MapCall c) {
    extern __shared__ __align__(16) float smem[];
    __shared__ int s_tile;
    double* slot = c.slots + (size_t)blockIdx.x * n_entries(g.K, M);
    const long long nblk = c.nlin + (c.norb + c.tiles - 1) / c.tiles;
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(c.counter, 1);
        __syncthreads();
        const long long item = s_tile;
        if (item >= nblk * c.parts) break;
        const long long b = item / c.parts;
        float* ws = c.ws + (c.parts > 1 ? (size_t)b : (size_t)blockIdx.x) * c.ws_floats;
        const int part = (int)(item - b * c.parts);
        fwd_block<M, SELF, GROUPED>(g, c, b, part, PackedLoad{c.wdw}, ws, slot, reinterpret_cast<char*>(smem), M);
    }
}

// The forward with the tensor-core contraction (128 accumulator columns per CTA).
template <int M, bool SELF>
__global__ void __launch_bounds__(BT, 4) map_fwd_tc_kernel(MapDev g, MapCall c) {
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
    const long long nblk = c.nlin + (c.norb + c.tiles - 1) / c.tiles;
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(c.counter, 1);
        __syncthreads();
        const long long item = s_tile;
        if (item >= nblk * c.parts || s_fail) break;
        const long long b = item / c.parts;
        float* ws = c.ws + (c.parts > 1 ? (size_t)b : (size_t)blockIdx.x) * c.ws_floats;
        fwd_block_tc<M, SELF>(g, c, b, (int)(item - b * c.parts), ws, slot, base, tc);
    }
    tc_teardown(s_tmem);
}

// Batched forward over all the plans of a batch, one launch: one work queue over the
// concatenated blocks of all its plans (plan-major); each CTA adds into that plan's
// slot number blockIdx.x.  Compiled for the largest m_max of the batch (M); each
// plan's blocks run with its own m_max (the multipole loops stop there) and its own self-pair mode.
template <int M>
__global__ void __launch_bounds__(BT, 4) batch_fwd_kernel(const BatchItem* __restrict__ items, int n,
                                                               long long total, unsigned long long* counter) {
    extern __shared__ __align__(16) float smem[];
    __shared__ long long s_t;
    __shared__ long long s_first[TPCF_MAX_BATCH + 1];
    for (int i = threadIdx.x; i <= n; i += BT) s_first[i] = i < n ? items[i].tile0 : total;
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
        const MapDev& g = items[lo].g;
        const MapCall& c = items[lo].c;
        double* slot = c.slots + (size_t)blockIdx.x * n_entries(g.K, g.M);
        fwd_block<M, true, false>(g, c, t - s_first[lo], 0, PackedLoad{c.wdw}, c.ws + (size_t)blockIdx.x * c.ws_floats,
                                  slot, reinterpret_cast<char*>(smem), g.M);
    }
}

// ------------------------------------------------------------ multi-field
// Three fields A, B, C on the same pixels (end of Sec. 2, after eq. ubEstimator): the moments
// a^k(i; F), W^k(i; F) of every field F (three walks of the single-field kind), then, over the
// cyclic permutations (P, X, Y) of (A, B, C),
//     S_m(k1,k2) += sum_i w^P_i P_i a_m^{k1}(i; X) conj(a_m^{k2}(i; Y)),
//     D(k1,k2)   += sum_i w^P_i W^{k1}(i; X) W^{k2}(i; Y),
// into the CTA's FP64 slot.  These sums are not Hermitian: the slot holds the full
// K x K matrices, for m, for (k1, k2): (Re S, Im S); then D for (k1, k2).
// The multi-field forward: c.wdw holds (w d, w) of field A, wdwB and wdwC those of
// B and C; the block's workspace holds the three fields' in turn.
template <int M>
__global__ void __launch_bounds__(BT, 4) map_fwd_multi_kernel(MapDev g, MapCall c,
                                                                    const float2* __restrict__ wdwB,
                                                                    const float2* __restrict__ wdwC) {
    extern __shared__ __align__(16) float smem[];
    __shared__ int s_tile;
    const int K = g.K;
    const size_t sub_floats = sub_floats_rt(K, M, false), field_ws = c.ws_floats / 3;
    double* slot = c.slots + (size_t)blockIdx.x * n_entries_multi(K, M);
    const long long nblk = c.nlin + (c.norb + c.tiles - 1) / c.tiles;
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(c.counter, 1);
        __syncthreads();
        const long long item = s_tile;
        if (item >= nblk * c.parts) break;
        const long long b = item / c.parts;
        const int part = (int)(item - b * c.parts);
        float* ws = c.ws + (c.parts > 1 ? (size_t)b : (size_t)blockIdx.x) * c.ws_floats;
        const Block<M, false> B(g, c, b);
        auto value = [&](int f, int s, int l) {
            return B.value(g, c, PackedLoad{f == 0 ? c.wdw : (f == 1 ? wdwB : wdwC)}, s, l);
        };
        const unsigned live = block_live(B.nsub, [&](int s, int l) {
            return value(0, s, l).y != 0.0f || value(1, s, l).y != 0.0f || value(2, s, l).y != 0.0f;
        });
        if (live == 0u) continue;
#pragma unroll 1
        for (int f = 0; f < 3; ++f) {
            block_moments<M, false, false>(g, c, b, live, part, PackedLoad{f == 0 ? c.wdw : (f == 1 ? wdwB : wdwC)},
                                           ws + f * field_ws, sub_floats, reinterpret_cast<char*>(smem), M);
            __syncthreads();
        }
        if (!block_complete(c, b)) continue;
        for (int f = 0; f < 3; ++f) block_fold(c, b, B.nsub, ws + f * field_ws, sub_floats);
        block_contract_multi(K, M, ws, field_ws, sub_floats, B.nsub, live, value, reinterpret_cast<char*>(smem), slot);
        __syncthreads();
    }
}

// ------------------------------------------------------------- pair count
#if defined(TPCF_M) && TPCF_M == 0  // one definition, in the M = 0 object
// counts[0] += in-bin ordered pairs (i, j) of the pivots with w_i != 0 (any w_j); counts[1] += those
// on rings with the pivot ring's pixel count, where pixels are mirror images about the pivot's
// meridian, counts[2] += the others and the pixels on the meridian.  The runs of the tile
// kernels, without touching pixel data; the blocks' edges are the same positions (pos_edge).
__global__ void __launch_bounds__(NTHREADS) map_count_kernel(MapDev g, const float2* __restrict__ wdw,
                                                             long long piv_lo, long long piv_hi,
                                                             long long tile_lo, long long tile_hi,
                                                             unsigned long long* counts) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (long long tile = tile_lo + blockIdx.x; tile < tile_hi; tile += gridDim.x) {
        const int2 tq = g.tiles[tile];
        const PivotRing P = pivot_ring(g, tq.x);
        const int q = tq.y + lane;
        const long long pix = g.ring_first[P.i] + q;
        const bool in = (q < P.n_i) && pix >= piv_lo && pix < piv_hi;
        const bool live = in && wdw[pix].y != 0.0f;
        if (!__syncthreads_or(live)) continue;
        const int qg = min(q, P.n_i - 1);
        unsigned long long n_sym = 0, n_plain = 0;
        for (int k = 0; k < g.K; ++k) {
            const int2 br = g.bin_range[(long long)P.i * g.K + k];
            for (int r = br.x + warp; r <= br.y; r += NWARPS) {
                const long long pr = P.pair0 + (r - P.rlo);
                const int2 Tk = g.pair_T[pr * (g.K + 1) + k];
                const int2 Tk1 = g.pair_T[pr * (g.K + 1) + k + 1];
                if (Tk.x == T_INF || Tk1.x == T_ZERO) continue;
                const int n_r = g.ring_n[r];
                const ExactCtx x = exact_ctx(g, P, r);
                const LaneC c = lane_c(qg, P.s_i, P.n_i, g.ring_shift[r], n_r);
                const bool sym = (n_r == P.n_i) && (Tk1.x != T_INF);
                const BinRuns b = bin_runs(c, Tk, Tk1, g.E[k], g.E[k + 1], x, n_r, sym);
                if (sym) {
                    n_sym += 2ull * (unsigned long long)b.n0;
                    n_plain += b.centre ? 1ull : 0ull;
                } else {
                    n_plain += (unsigned long long)(b.n0 + b.n1);
                }
            }
        }
        if (live) {
            atomicAdd(counts, n_sym + n_plain);
            atomicAdd(counts + 1, n_sym);
            atomicAdd(counts + 2, n_plain);
        }
    }
}
#endif

// val = sum_m (cos(m phi) hr_m + sin(m phi) hi_m): X the cosine part, Y the sine part.
// h[m] = (hr_m, hi_m); the (cos, sin) chains run packed, in the folded frame psi, by
// the recurrence of harmonicsf(); even and odd multipoles are summed apart and the odd
// sum takes the sign sigma at the end.
template <int M>
__device__ __forceinline__ void adj_harmonicsf(const float2 (&h)[M + 1], const Fold& f, float& X, float& Y,
                                               int mr = M) {
    float2 ev = make_float2(h[0].x, 0.0f);
    float2 od = make_float2(0.0f, 0.0f);
    float sg = 1.0f;
    if constexpr (M >= 1) {
        if (mr < 1) {
            X = ev.x;
            Y = ev.y;
            return;
        }
        sg = f.sg;
        float2 T = make_float2(f.ac, f.ss);
        float2 D = make_float2(0.5f * f.lam, f.ss);
        const float2 L2 = make_float2(f.lam, f.lam);
        od = __ffma2_rn(T, h[1], od);
#pragma unroll
        for (int m = 2; m <= M; ++m) {
            if (m > mr) break;
            D = __ffma2_rn(L2, T, D);
            T = __fadd2_rn(T, D);
            if (m & 1)
                od = __ffma2_rn(T, h[m], od);
            else
                ev = __ffma2_rn(T, h[m], ev);
        }
    }
    X = fmaf(sg, od.x, ev.x);
    Y = fmaf(sg, od.y, ev.y);
}

// Adjoint: persistent CTAs draw work items (block, part); c.step: see bwd_block.
template <int M, bool SELF>
__global__ void __launch_bounds__(BT, 4) map_bwd_kernel(MapDev g, MapCall c) {
    extern __shared__ __align__(16) float smem[];
    __shared__ int s_tile;
    const long long nblk = c.nlin + (c.norb + c.tiles - 1) / c.tiles;
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(c.counter, 1);
        __syncthreads();
        const long long item = s_tile;
        if (item >= nblk * c.parts) break;
        const long long b = item / c.parts;
        float* ws = c.ws + (c.step != 0 ? (size_t)b : (size_t)blockIdx.x) * c.ws_floats;
        bwd_block<M, SELF>(g, c, b, (int)(item - b * c.parts), c.step, ws, reinterpret_cast<char*>(smem), M);
    }
}

// The adjoint of all the plans of a batch, one launch (the work queue of batch_fwd_kernel).
template <int M>
__global__ void __launch_bounds__(BT, 4) batch_bwd_kernel(const BatchItem* __restrict__ items, int n,
                                                               long long total, unsigned long long* counter) {
    extern __shared__ __align__(16) float smem[];
    __shared__ long long s_t;
    __shared__ long long s_first[TPCF_MAX_BATCH + 1];
    for (int i = threadIdx.x; i <= n; i += BT) s_first[i] = i < n ? items[i].tile0 : total;
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
        const MapDev& g = items[lo].g;
        const MapCall& c = items[lo].c;
        bwd_block<M, false>(g, c, t - s_first[lo], 0, 0, c.ws + (size_t)blockIdx.x * c.ws_floats,
                            reinterpret_cast<char*>(smem), g.M);
    }
}

}  // namespace tpcf

#include "map_tile.cuh"
