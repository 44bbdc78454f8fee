// Pieces of the leave-one-out grid kernel shared by the single-dataset launch
// (loo_grid.cu), the persistent batched launch (batch.cu) and the
// allocation-free launch (noalloc.cu): the argument block, coefficient access,
// the exact joint-shift fallback and the FP64 per-unit epilogue.  The tile
// body (tensor-core outer product) is in loo_mma.cuh; loo_grid.cu describes
// the method.
#pragma once

#include <climits>
#include <cstdint>

#include "cde_internal.h"

namespace cde {

struct LooArgs {
    const float* xs;        // [d][Np] structure-of-arrays x (standardised if asked)
    const float* y;         // [Np]
    const float* mx;        // [N] nearest squared x distance per row
    const float* my;        // [N] nearest squared y distance per row
    const float* qx;        // [N] dx^2 of each row's y-nearest point (fallback bounds)
    const float* qy;        // [N] dy^2 of each row's x-nearest point
    const int64_t* rows;    // optional list of rows (null: rows 0..n_rows-1)
    double* part;           // [n_tiles][2][T1*T2] FP64 tile partials (L_cond, sum ln A)
    double* fb;             // d >= 16 kernel: [grid][16384] per-CTA recomputed log2 At
    double* ell_rows;       // optional per-row ell output
    int64_t ell_ld_row;     // row stride of ell_rows (doubles)
    int ell_ld_k;           // k stride of ell_rows
    int G1r, G2r;           // real (unpadded) sizes of this grid block
    int64_t N, Np, n_rows;
    int d;
    int n_units, units_per_tile, n_tiles;
    // tile partition (LooTiles): big_levels levels of big_g tiles each, the tiles of
    // level l holding big_s0 >> l units; the rest hold units_per_tile consecutive
    // units.  big_levels = 0: all tiles are small.
    int big_g, big_levels, big_s0;
    int win0, win1;         // units m of each tile processed by this launch: [win0, win1)
    int tile_base;          // batched launch: first global tile of this item
    int* work;              // batched launch: queue counter
    int kern;               // CDE_KERNEL_GAUSS or CDE_KERNEL_EPAN
    float thresh;           // cells with shifted numerator below this are recomputed
    double logn1;           // ln(N - 1)
    // per-bandwidth coefficients, padded by repeating the last bandwidth:
    //   Gaussian:     a = log2(e)/(2 h^2), lam1 = d ln(sqrt(2 pi) h1), kap2 = ln(sqrt(2 pi) h2)
    //   Epanechnikov: a = 1/h^2,           lam1 = d ln h1 - ln c_d,     kap2 = ln h2 - ln c_1
    float a1[32], a2[32];
    double lam1[32];
    double kap2[32];
};

__device__ __forceinline__ float ex2_approx(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// a * b + c clamped to [0, 1] in the same instruction (NaN -> 0)
__device__ __forceinline__ float fma_sat(float a, float b, float c) {
    float r;
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Kernel factors of two values that share nothing but the family.
//   Gaussian (KERN 0):     t = shifted negative squared distance, factor 2^{c t}
//   Epanechnikov (KERN 1): t = squared distance, factor (1 - c t)_+ (c = 1/h^2;
//                          t = +inf gives exactly 0)
template <int KERN>
__device__ __forceinline__ float2 kernel_factor2(float2 c, float2 t) {
    if constexpr (KERN == 0) {
        const float2 a = __fmul2_rn(c, t);
        return make_float2(ex2_approx(a.x), ex2_approx(a.y));
    } else {
        return make_float2(fma_sat(-c.x, t.x, 1.f), fma_sat(-c.y, t.y, 1.f));
    }
}

// log2 of a positive normal float, returned in FP64: exact exponent plus the
// FP32 log2 of the mantissa in [1, 2) (absolute error below 1e-7).
__device__ __forceinline__ double log2_wide(float v) {
    int e;
    const float m = frexpf(v, &e);
    return (double)(e - 1) + (double)log2f(2.0f * m);
}

// Fixed-order reduction of four adjacent grid cells over the tile partials (a CTA
// of 256 threads): thread (cell q = tid % 4, t = tid / 4) sums tiles t, t + 64, ... in
// order, then a fixed tree over t.  The four cells are one 32-byte sector of every
// slot.  Returns with the sums in the threads tid < 4.  (One warp per cell, reading a
// sector per slot and cell: 28 us for the 3,001 slots of a 4 x 4 grid, 11 us for the
// 250 of an 8 x 8 grid.)
constexpr int kFinalThreads = 256, kFinalCells = 4;

__device__ __forceinline__ void loo_final_cells(const double* __restrict__ part, int n_tiles, int GG, int cell0,
                                                double& sc, double& se) {
    __shared__ double rc[kFinalThreads / 32][kFinalCells], re[kFinalThreads / 32][kFinalCells];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double* p = part + cell0 + (tid & 3);
    sc = 0.0;
    se = 0.0;
#pragma unroll 8
    for (int t = tid >> 2; t < n_tiles; t += kFinalThreads / kFinalCells) {
        sc += p[(int64_t)t * 2 * GG];
        se += p[(int64_t)t * 2 * GG + GG];
    }
#pragma unroll
    for (int o = 16; o >= kFinalCells; o >>= 1) {
        sc += __shfl_xor_sync(0xffffffffu, sc, o);
        se += __shfl_xor_sync(0xffffffffu, se, o);
    }
    if (lane < kFinalCells) {
        rc[warp][lane] = sc;
        re[warp][lane] = se;
    }
    __syncthreads();
    if (tid < kFinalCells)
#pragma unroll
        for (int w = 1; w < kFinalThreads / 32; ++w) {
            sc += rc[w][tid];
            se += re[w][tid];
        }
}

// Tile partition of a launch's units.  One partial slot per tile; a tile's units
// are added to its slot in order, and the slots are reduced in a fixed order, so
// the result depends on the partition only, not on which CTA runs which tile or
// in which launch.  With enough work the tiles shrink as the launch proceeds
// (guided self-scheduling): level l holds G tiles (one per resident CTA) of
// s0 >> l units, s0 = n_units / 2G, interleaved with stride G inside the level's
// range so that every tile samples the whole dataset; levels stop before the
// size falls under 2 units_per_tile, and small tiles of units_per_tile
// consecutive units take the rest.  The atomic queue hands tiles out in index
// order, so the launch ends on small tiles as with uniform ones, with
// G log2(n_units / G) + 2G slots instead of one per small tile.
struct LooTiles {
    int big_g, big_levels, big_s0, n_tiles;
};

__host__ __device__ inline LooTiles loo_tiles(int n_units, int upt, int G) {
    LooTiles p{0, 0, 0, 0};
    if (G > 0 && (int64_t)n_units >= 8LL * G * upt) {
        p.big_g = G;
        p.big_s0 = n_units / (2 * G);
        while (p.big_levels < 16 && (p.big_s0 >> p.big_levels) >= 2 * upt) ++p.big_levels;
        int64_t covered = 0;
        for (int l = 0; l < p.big_levels; ++l) covered += p.big_s0 >> l;
        const int rest = n_units - (int)(covered * G);
        p.n_tiles = p.big_levels * G + (rest + upt - 1) / upt;
    } else {
        p.n_tiles = (n_units + upt - 1) / upt;
    }
    return p;
}

// first unit of level l (the units of levels 0 .. l-1 come before it)
__host__ __device__ __forceinline__ int loo_level_base(const LooArgs& a, int l) {
    int s = 0;
    for (int i = 0; i < l; ++i) s += a.big_s0 >> i;
    return s * a.big_g;
}

// tile t's units: u0 + m stride for m < len
__host__ __device__ __forceinline__ void loo_tile_span(const LooArgs& a, int t, int& u0, int& stride, int& len) {
    const int nb = a.big_levels * a.big_g;
    if (t < nb) {
        const int l = t / a.big_g;
        u0 = loo_level_base(a, l) + (t - l * a.big_g);
        stride = a.big_g;
        len = a.big_s0 >> l;
    } else {
        u0 = loo_level_base(a, a.big_levels) + (t - nb) * a.units_per_tile;
        stride = 1;
        len = a.units_per_tile < a.n_units - u0 ? a.units_per_tile : a.n_units - u0;
    }
}

// Coefficient access from shared memory (batched launch: one item at a time).
struct CoefSmem {
    const float* a1s;
    const float* a2s;
    __device__ __forceinline__ float a1(int k) const { return a1s[k]; }
    __device__ __forceinline__ float a2(int l) const { return a2s[l]; }
};

// Coefficient access straight from the kernel's parameter block.
struct CoefParam {
    const LooArgs& a;
    __device__ __forceinline__ float a1(int k) const { return a.a1[k]; }
    __device__ __forceinline__ float a2(int l) const { return a.a2[l]; }
};

// log2(1 + 5.12e-8): ex2.approx.ftz.f32 is low by 5.12e-8 relative on average
// (measured on sm_103a); the fallback's terms carry it in their exponent, as
// the tile body's factors do
constexpr float kFbEx2Fix = 7.39e-8f;

// An anchor of the one-pass recomputation moves once a term would exceed 2^kFbMove of its
// scale: the terms within 20 of the minimum see a handful of moves.  (Anchors that follow
// every lower point were off by 7.0e-5 where N = 100,000 rows lie in descending order of e.)
constexpr float kFbMove = 4.f;

// 2^e (e <= 0, or the rounding of a 0) as (1 + p) m, applied to about an ulp (ex2.approx alone is off by two, the
// same way at every move): m = 2^n, n = round(e), p the Taylor series of exp((e - n) ln 2) - 1
struct Exp2Scale {
    float p, m;
    __device__ __forceinline__ explicit Exp2Scale(float e) {
        const float n = rintf(fmaxf(e, -126.f));
        const float z = fmaxf(e - n, -0.5f) * 0.693147181f;
        p = fmaf(z, 1.f / 5040.f, 1.f / 720.f);
        p = fmaf(z, p, 1.f / 120.f);
        p = fmaf(z, p, 1.f / 24.f);
        p = fmaf(z, p, 1.f / 6.f);
        p = fmaf(z, p, 0.5f);
        p = fmaf(z * z, p, z);
        m = __int_as_float(((int)n + 127) << 23);
    }
    __device__ __forceinline__ float operator()(float v) const { return fmaf(v, p, v) * m; }
};

// s + v into the unevaluated sum s + c (Knuth's two-sum)
__device__ __forceinline__ void add_two(float& s, float& c, float v) {
    const float t = __fadd_rn(s, v), b = __fsub_rn(t, s);
    c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(v, b)));
    s = t;
}

// Exact joint-shift recomputation of the flagged cells of one unit (whole
// CTA).  For a cell (row j, k, l) let e_i = a1_k (dx2_i - m_x,j) + a2_l (dy2_i - m_y,j).
// Then At = sum_i 2^{-e_i} = 2^{-e_a} S with S = sum_i 2^{-(e_i - e_a)} for any anchor
// point a, where e_i - e_a = a1_k (dx2_i - dx2_a) + a2_l (dy2_i - dy2_a) is formed from
// differences of distances (no cancellation at large e), and log2 At = -e_a + log2 S
// with e_a in FP64.  One pass over the points: every warp takes chunks of 64
// consecutive points (two per lane, packed FP32x2 distances, the tile body's formula)
// and keeps, per flagged cell, its own anchor -- a point within 2^kFbMove of the smallest e
// it has met -- and the sum relative to it; a point further below rescales the sum and
// becomes the anchor.  All anchors start at the better of the x-nearest and the y-nearest
// point (their distances are stored with the dataset), so the warps' sums never overflow
// (terms are at most 2^kFbMove), and the warps are merged in fixed order at the lowest anchor.
//
// Precision.  A chunk's terms are summed in four floats (at most 16 terms each), which are
// added to the cell's sum with a compensated add: the error of 18 FP32 additions, whatever N
// is (the two-pass form: of 32; one running float: 3.1e-5 on 20,000 tied points).  The
// compensation and the low parts' 4 bytes per cell and warp cost 3.71 -> 3.74 ms of a new
// dataset with a 4 x 4 grid at N = 24,007, d = 12.
//
// Candidates.  A term with e_i > e_a + T, T = 32 + ceil(log2 N), adds less than 2^-T of
// the cell's sum (all of them together less than 2^-32), so only points with
// X <= max_f (e_af + T)/a1_f and Y <= max_f (e_af + T)/a2_f over the row's cells are
// looked at; the box follows the warp's anchors down.  A row's candidates of a chunk
// are compacted into the warp's list (lane = point), then lane = cell: each lane runs
// its cells over the list.  Every warp's work is a fixed function of the row and the
// points, so the result does not depend on scheduling.
//
// Bound by the distance pass (issue).  Tile kernel with this pass against the two-pass
// form below, Gaussian, standardised six-component mixture: N = 12,000, d = 12: 4 x 4 0.88
// against 1.75 ms, 16 x 8 1.72 / 2.61, 16 x 16 2.03 / 2.95, 32 x 16 2.95 / 4.05; N = 20,000,
// d = 5: 4 x 4 1.20 / 1.42, 16 x 16 3.92 / 4.06, 32 x 16 6.20 / 6.24.
template <class C, class Coef>
__device__ __forceinline__ void loo_fallback(const LooArgs& a, const Coef& cf, float* sm, int nfl) {
    constexpr int GG = C::GG, G2 = C::G2v, JW = C::JW, NT = C::kThreads, NW = C::kWarps;
    constexpr int LG2 = G2 == 4 ? 2 : G2 == 8 ? 3 : (G2 == 16 ? 4 : 5);
    constexpr int JG = JW * GG, CAP = C::FBCAP;
    static_assert(JW <= 8, "per-row bounds hold 8 rows");
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int d = a.d;
    const int64_t N = a.N, Np = a.Np;
    const float* xj_s = sm + C::off_xj(d);
    const float* yj_s = sm + C::off_yj(d);
    const float* mx_s = sm + C::off_mx(d);
    const float* my_s = sm + C::off_my(d);
    const long long* ji_s = reinterpret_cast<const long long*>(sm + C::off_ji(d));
    const int* flag_s = reinterpret_cast<const int*>(sm + C::off_flag(d));
    double* la2 = reinterpret_cast<double*>(sm);
    float* As = sm + 2 * JG;                       // the round's cells: coefficients
    float* Bs = sm + 3 * JG;
    float* Ss = sm + C::off_fbS(d);                // [warp][CAP] sums and their low parts; the anchors' dx2, dy2
    float* Cs = sm + C::off_fbC(d);
    float* Xs = sm + C::off_fbX(d);
    float* Ys = Xs + NW * CAP;
    // per warp: a chunk's candidates of one row, and the rows' boxes; then the row ranges
    float* fbw = sm + C::off_fbw(d);
    float* lx = fbw + warp * 144;
    float* ly = lx + 64;
    float* bx = ly + 64;
    float* by = bx + 8;
    int* rs = reinterpret_cast<int*>(fbw + NW * 144);   // cells [rs, re) of the row in the round
    int* re = rs + 8;
    float* Sw = Ss + warp * CAP;
    float* Cw = Cs + warp * CAP;
    float* Xw = Xs + warp * CAP;
    float* Yw = Ys + warp * CAP;

    int lg = 0;
    while (((int64_t)1 << lg) < N) ++lg;
    const float T = (float)(32 + lg);

    // the warp's box of a row from its cells' anchors (all lanes return with it stored)
    const auto box = [&](int r, int f0, int f1) {
        const float mxr = mx_s[r], myr = my_s[r];
        float x = 0.f, y = 0.f;
        for (int f = f0 + lane; f < f1; f += 32) {
            const float A = As[f], B = Bs[f];
            // (the factor covers the rounding of e where it is large next to T)
            const float e = fmaf(fmaf(A, Xw[f] - mxr, B * (Yw[f] - myr)), 1.f + 0x1p-20f, T);
            x = fmaxf(x, __fdividef(e, A));
            y = fmaxf(y, __fdividef(e, B));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
            y = fmaxf(y, __shfl_xor_sync(0xffffffffu, y, o));
        }
        __syncwarp();
        if (lane == 0) {
            bx[r] = mxr + x;
            by[r] = myr + y;
        }
        __syncwarp();
    };

    for (int base = 0; base < nfl; base += CAP) {
        const int n = min(CAP, nfl - base);
        if (tid < JW) rs[tid] = re[tid] = 0;
        __syncthreads();
        for (int f = tid; f < n; f += NT) {
            const int c = flag_s[base + f], r = c / GG, kl = c - r * GG, k = kl >> LG2, l = kl & (G2 - 1);
            const float A = cf.a1(k), B = cf.a2(l);
            As[f] = A;
            Bs[f] = B;
            if (f == 0 || flag_s[base + f - 1] / GG != r) rs[r] = f;
            if (f == n - 1 || flag_s[base + f + 1] / GG != r) re[r] = f + 1;
            // the x-nearest point is (m_x, q_y), the y-nearest (q_x, m_y)
            const long long j = ji_s[r];
            const float qx = a.qx[j], qy = a.qy[j];
            const bool xn = B * (qy - my_s[r]) <= A * (qx - mx_s[r]);
            const float X0 = xn ? mx_s[r] : qx, Y0 = xn ? qy : my_s[r];
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                Ss[w * CAP + f] = Cs[w * CAP + f] = 0.f;
                Xs[w * CAP + f] = X0;
                Ys[w * CAP + f] = Y0;
            }
        }
        __syncthreads();
        const auto boxes = [&]() {
#pragma unroll 1
            for (int r = 0; r < JW; ++r)
                if (rs[r] < re[r]) box(r, rs[r], re[r]);
        };
        // One chunk: the candidates of every row with cells
        const auto chunk = [&](int64_t i0) {
            const int64_t i = i0 + 2 * lane;   // this lane's points i, i + 1 (inside the padded length)
            float2 xi[8];
#pragma unroll
            for (int c = 0; c < 8; ++c)
                if (c < d) {
                    const float2 v = *reinterpret_cast<const float2*>(a.xs + (int64_t)c * Np + CDE_CK(i, Np - 1, 108));
                    xi[c] = make_float2(-v.x, -v.y);
                }
            const float2 yi = *reinterpret_cast<const float2*>(a.y + i);
#pragma unroll 1
            for (int r = 0; r < JW; ++r) {
                const int f0 = rs[r], f1 = re[r];
                if (f0 == f1) continue;
                const float* xjr = xj_s + r * d;
                float2 dx2 = make_float2(0.f, 0.f);
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    if (c < d) {
                        const float2 t = __fadd2_rn(make_float2(xjr[c], xjr[c]), xi[c]);
                        dx2 = __ffma2_rn(t, t, dx2);
                    }
#pragma unroll 4
                for (int c = 8; c < d; ++c) {
                    const float2 v = *reinterpret_cast<const float2*>(a.xs + (int64_t)c * Np + i);
                    const float2 t = __fadd2_rn(make_float2(xjr[c], xjr[c]), make_float2(-v.x, -v.y));
                    dx2 = __ffma2_rn(t, t, dx2);
                }
                const float yr = yj_s[r];
                const float2 dy = __fadd2_rn(make_float2(yr, yr), make_float2(-yi.x, -yi.y));
                const float2 dy2 = __fmul2_rn(dy, dy);
                const int64_t j = ji_s[r];
                const float RX = bx[r], RY = by[r];
                const bool in0 = i < N && i != j && dx2.x <= RX && dy2.x <= RY;
                const bool in1 = i + 1 < N && i + 1 != j && dx2.y <= RX && dy2.y <= RY;
                const unsigned m0 = __ballot_sync(0xffffffffu, in0), m1 = __ballot_sync(0xffffffffu, in1);
                if ((m0 | m1) == 0u) continue;
                const unsigned lt = (1u << lane) - 1u;
                const int p = __popc(m0 & lt) + __popc(m1 & lt);
                if (in0) {
                    lx[p] = dx2.x;
                    ly[p] = dy2.x;
                }
                if (in1) {
                    lx[p + in0] = dx2.y;
                    ly[p + in0] = dy2.y;
                }
                const int nc = __popc(m0) + __popc(m1);
                if (lane < (-nc & 3)) lx[nc + lane] = ly[nc + lane] = INFINITY;   // up to a multiple of four
                __syncwarp();
                bool moved = false;
                for (int f = f0 + lane; f < f1; f += 32) {
                    const float A = As[f], B = Bs[f];
                    float X = Xw[f], Y = Yw[f], S = Sw[f], Sc = Cw[f];
                    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll 1
                    for (int q = 0; q < nc; q += 4) {
                        const float4 qx = *reinterpret_cast<const float4*>(lx + q);
                        const float4 qy = *reinterpret_cast<const float4*>(ly + q);
                        const auto ex = [&](float x, float y) { return fmaf(A, x - X, B * (y - Y)); };
                        float e0 = ex(qx.x, qy.x), e1 = ex(qx.y, qy.y), e2 = ex(qx.z, qy.z), e3 = ex(qx.w, qy.w);
                        const float lo = fminf(fminf(e0, e1), fminf(e2, e3));
                        if (lo < -kFbMove) {   // a lower point: the new anchor
                            const Exp2Scale by(lo);
                            S = by(S);
                            Sc = by(Sc);
                            s0 = by(s0);
                            s1 = by(s1);
                            s2 = by(s2);
                            s3 = by(s3);
                            X = lo == e0 ? qx.x : lo == e1 ? qx.y : lo == e2 ? qx.z : qx.w;
                            Y = lo == e0 ? qy.x : lo == e1 ? qy.y : lo == e2 ? qy.z : qy.w;
                            e0 = ex(qx.x, qy.x);
                            e1 = ex(qx.y, qy.y);
                            e2 = ex(qx.z, qy.z);
                            e3 = ex(qx.w, qy.w);
                            moved = true;
                        }
                        s0 += ex2_approx(kFbEx2Fix - e0);
                        s1 += ex2_approx(kFbEx2Fix - e1);
                        s2 += ex2_approx(kFbEx2Fix - e2);
                        s3 += ex2_approx(kFbEx2Fix - e3);
                    }
                    add_two(S, Sc, (s0 + s1) + (s2 + s3));
                    Xw[f] = X;
                    Yw[f] = Y;
                    Sw[f] = S;
                    Cw[f] = Sc;
                }
                __syncwarp();
                if (__any_sync(0xffffffffu, moved)) box(r, f0, f1);
            }
        };
        boxes();
#pragma unroll 1
        for (int64_t i0 = (int64_t)warp * 64; i0 < N; i0 += NW * 64) chunk(i0);
        __syncthreads();
        // merge the warps at the lowest anchor, in warp order
        for (int f = tid; f < n; f += NT) {
            const int c = flag_s[base + f], r = c / GG;
            const float A = As[f], B = Bs[f];
            float X = Xs[f], Y = Ys[f];
#pragma unroll
            for (int w = 1; w < NW; ++w) {
                const float Xo = Xs[w * CAP + f], Yo = Ys[w * CAP + f];
                if (fmaf(A, Xo - X, B * (Yo - Y)) < 0.f) {
                    X = Xo;
                    Y = Yo;
                }
            }
            float tot = 0.f, low = 0.f;
#pragma unroll
            for (int w = 0; w < NW; ++w)
                add_two(tot, low, Exp2Scale(-fmaf(A, Xs[w * CAP + f] - X, B * (Ys[w * CAP + f] - Y)))(
                                      Ss[w * CAP + f] + Cs[w * CAP + f]));
            tot += low;
            const double e = (double)A * ((double)X - (double)mx_s[r]) + (double)B * ((double)Y - (double)my_s[r]);
            la2[c] = -e + log2_wide(tot);
        }
        __syncthreads();
    }
}

// The same recomputation in two passes, for the 32 x 32 shape: there the code of the
// one-pass form costs the tile body's main loop more than the pass saves (the compiler
// schedules that loop at its register limit: N = 20,000, d = 5 11.4 against 10.1 ms,
// d = 2 4.2 / 3.7; only at d = 12, N = 12,000 it would gain, 5.0 / 5.6), as a call or inline.
// For a cell (row j, k, l) let X_i = dx2_i - m_x,j, Y_i = dy2_i - m_y,j and
// e_i = a1_k X_i + a2_l Y_i.  Then At = sum_i 2^{-e_i} = 2^{-e_*} S with
// S = sum_i 2^{-(a1_k (dx2_i - dx2_*) + a2_l (dy2_i - dy2_*))} for the minimiser
// i* (its term is exactly 1), and log2 At = -e_* + log2 S.  All flagged cells
// of the unit are processed together in two passes over the points:
//  1. the minimiser of every cell.  It is no worse than the x-nearest point
//     (X = 0, Y = Yh) and the y-nearest point (X = Xh, Y = 0), so
//     e_* <= min(a2 Yh, a1 Xh): only points with dx2 <= qx and dy2 <= qy
//     (qx, qy: the dataset's stored other-coordinate distances of the two
//     neighbours), and inside the union over the row's cells of those
//     triangles, are candidates.  A cell keeps the smallest key (e bits, i):
//     the smallest e, ties to the smallest index, whatever the order of visits.
//  2. the sums.  A point with e_i > e_* + T adds less than 2^-T; with
//     T = 32 + ceil(log2 N) all of them together add less than 2^-32 of S.
//     So only points with X <= max_f (e_*f + T)/a1_f and Y <= max_f (e_*f + T)/a2_f
//     (the row's box) are candidates.
// Each warp takes chunks of 32 consecutive points (lane = point: distances to
// every flagged row, candidate tests) and compacts a row's candidates into a
// shared list; then lane = cell: each lane runs its cells over the list.
// Pass 1 folds the list into the lane's (e, i) minimum and merges it with a
// 64-bit shared atomicMin; pass 2 sums the list's terms in FP32 (list order)
// and adds the chunk sum as an integer in units of 2^-(62 - ceil(log2 N))
// (64-bit shared atomicAdd: exact, so the cell's sum is the same whatever the
// order in which warps finish, and it cannot overflow).  Both passes compute
// dx2 and dy2 with the tile body's FP32 formula.
template <class C, class Coef>
__device__ __forceinline__ void loo_fallback_two_pass(const LooArgs& a, const Coef& cf, float* sm, int nfl) {
    constexpr int GG = C::GG, G2 = C::G2v, JW = C::JW, NT = C::kThreads, NW = C::kWarps;
    constexpr int LG2 = G2 == 4 ? 2 : G2 == 8 ? 3 : (G2 == 16 ? 4 : 5);
    constexpr int JG = JW * GG;
    static_assert(8 * JG <= C::COMB, "fallback scratch must fit in the combine buffer");
    static_assert(JW <= 8, "per-row fallback parameters hold 8 rows");
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int d = a.d;
    const int64_t N = a.N, Np = a.Np;
    const float* xj_s = sm + C::off_xj(d);
    const float* yj_s = sm + C::off_yj(d);
    const float* mx_s = sm + C::off_mx(d);
    const float* my_s = sm + C::off_my(d);
    const long long* ji_s = reinterpret_cast<const long long*>(sm + C::off_ji(d));
    int* flag_s = reinterpret_cast<int*>(sm + C::off_flag(d));
    double* la2 = reinterpret_cast<double*>(sm);
    // per flagged cell f (after la2): the pass-1 key, reused for the pass-2 sum;
    // the minimiser's distances; the cell's coefficients
    unsigned long long* best = reinterpret_cast<unsigned long long*>(sm + 2 * JG);
    unsigned long long* acc = best;
    float* dxs = sm + 4 * JG;
    float* dys = sm + 5 * JG;
    float* As = sm + 6 * JG;
    float* Bs = sm + 7 * JG;
    // per warp: the candidate list of one (chunk, row); per row: bounds and cell range
    float* fbw = sm + C::off_fbw(d);
    float* lx = fbw + warp * 96;
    float* ly = lx + 32;
    int* li = reinterpret_cast<int*>(ly + 32);
    float* rqx = fbw + NW * 96;
    float* rqy = rqx + 8;
    int* rlo_b = reinterpret_cast<int*>(rqy + 8);   // float bits of positive values (0: none)
    int* rhi_b = rlo_b + 8;
    int* rx_b = rhi_b + 8;
    int* ry_b = rx_b + 8;
    int* rs = ry_b + 8;                              // cells [rs, re) of the row in flag_s
    int* re = rs + 8;

    // sort the (distinct) flagged cell ids in place: each thread ranks its entries
    int mine[4], rank[4];
    int nm = 0;
    for (int q = tid; q < nfl; q += NT) {
        const int v = flag_s[q];
        int r = 0;
        for (int t = 0; t < nfl; ++t) r += flag_s[t] < v;
        mine[nm] = v;
        rank[nm] = r;
        ++nm;
    }
    if (tid < JW) {
        rs[tid] = re[tid] = 0;
        rlo_b[tid] = 0;
        rhi_b[tid] = __float_as_int(INFINITY);
        rx_b[tid] = ry_b[tid] = 0;
        const long long j = ji_s[tid];
        rqx[tid] = a.qx[j];
        rqy[tid] = a.qy[j];
    }
    __syncthreads();
    for (int m = 0; m < nm; ++m) flag_s[rank[m]] = mine[m];
    __syncthreads();

    int lg = 0;
    while (((int64_t)1 << lg) < N) ++lg;
    const float T = (float)(32 + lg);
    const int SC = 62 - lg;            // fixed-point scale of the sums
    const float scale = ldexpf(1.f, SC), inv_scale_f = ldexpf(1.f, -SC);

    // cells: coefficients, row ranges, and the triangles of the argmin region --
    // cells with rho = a2/a1 <= Xh/Yh are bounded by the x-nearest point
    // (X + rho Y <= rho Yh; the largest rho covers the others), the rest by the
    // y-nearest point (X + rho Y <= Xh; the smallest rho)
    for (int f = tid; f < nfl; f += NT) {
        const int c = flag_s[f], r = c / GG, kl = c - r * GG, k = kl >> LG2, l = kl & (G2 - 1);
        const float A = cf.a1(k), B = cf.a2(l);
        As[f] = A;
        Bs[f] = B;
        best[f] = ~0ull;
        if (f == 0 || flag_s[f - 1] / GG != r) rs[r] = f;
        if (f == nfl - 1 || flag_s[f + 1] / GG != r) re[r] = f + 1;
        const float Xh = rqx[r] - mx_s[r], Yh = rqy[r] - my_s[r];
        const float rho = B / A;
        if (rho * Yh <= Xh) atomicMax(rlo_b + r, __float_as_int(rho));
        else atomicMin(rhi_b + r, __float_as_int(rho));
    }
    __syncthreads();

    // squared distances of a chunk's point (lane) to row r, the tile body's formula
    const auto dist = [&](int r, const float (&xi)[8], int64_t i, float yi, float& dx2, float& dy2) {
        const float* xjr = xj_s + r * d;
        float s = 0.f;
#pragma unroll
        for (int cc = 0; cc < 8; ++cc)
            if (cc < d) {
                const float t = xjr[cc] - xi[cc];
                s = fmaf(t, t, s);
            }
        for (int cc = 8; cc < d; ++cc) {
            const float t = xjr[cc] - a.xs[(int64_t)cc * Np + i];
            s = fmaf(t, t, s);
        }
        dx2 = s;
        const float dy = yj_s[r] - yi;
        dy2 = dy * dy;
    };

    // ---- pass 1: the minimiser of every flagged cell ----
    for (int64_t base = (int64_t)warp * 32; base < N; base += NW * 32) {
        const int64_t i = base + lane;
        const bool v = i < N;
        const int64_t ic = v ? i : base;
        float xi[8];
#pragma unroll
        for (int cc = 0; cc < 8; ++cc) xi[cc] = cc < d ? a.xs[(int64_t)cc * Np + CDE_CK(ic, N, 108)] : 0.f;
        const float yi = a.y[ic];
        for (int r = 0; r < JW; ++r) {
            const int f0 = rs[r], f1 = re[r];
            if (f0 == f1) continue;
            float dx2, dy2;
            dist(r, xi, ic, yi, dx2, dy2);
            const float mxr = mx_s[r], myr = my_s[r];
            const float X = dx2 - mxr, Y = dy2 - myr;
            const float Xh = rqx[r] - mxr, Yh = rqy[r] - myr;
            const float rlo = __int_as_float(rlo_b[r]), rhi = __int_as_float(rhi_b[r]);
            const bool in = v && i != ji_s[r] && dx2 <= rqx[r] && dy2 <= rqy[r] &&
                            ((rlo > 0.f && fmaf(rlo, Y, X) <= rlo * Yh) || (rhi < INFINITY && fmaf(rhi, Y, X) <= Xh));
            const unsigned m = __ballot_sync(0xffffffffu, in);
            if (m == 0u) continue;
            if (in) {
                const int p = __popc(m & ((1u << lane) - 1u));
                lx[p] = X;
                ly[p] = Y;
                li[p] = (int)i;
            }
            __syncwarp();
            const int nc = __popc(m);
            for (int f = f0 + lane; f < f1; f += 32) {
                const float A = As[f], B = Bs[f];
                float emin = INFINITY;
                int imin = 0;
                for (int q = 0; q < nc; ++q) {
                    const float e = fmaxf(fmaf(A, lx[q], B * ly[q]), 0.f);
                    if (e < emin) {
                        emin = e;
                        imin = li[q];
                    }
                }
                const unsigned long long key = ((unsigned long long)__float_as_uint(emin) << 32) | (unsigned int)imin;
                if (key < best[f]) atomicMin(best + f, key);
            }
            __syncwarp();
        }
    }
    __syncthreads();

    // ---- the minimisers' distances; the rows' boxes of pass 2 ----
    for (int f = tid; f < nfl; f += NT) {
        const int r = flag_s[f] / GG;
        const long long j = ji_s[r];
        const unsigned long long b = best[f];
        // no point in the region (cannot happen: the two neighbours are in it):
        // anchor at the x-nearest bound
        const bool none = b == ~0ull;
        const int64_t is = none ? (j == 0 ? 1 : 0) : (int64_t)(unsigned int)b;
        const float* xjr = xj_s + r * d;
        float t2 = 0.f;
        for (int cc = 0; cc < d; ++cc) {
            const float t = xjr[cc] - a.xs[(int64_t)cc * Np + CDE_CK(is, N, 108)];
            t2 = fmaf(t, t, t2);
        }
        const float t = yj_s[r] - a.y[is];
        dxs[f] = t2;
        dys[f] = t * t;
        const float A = As[f], B = Bs[f];
        const float es = fmaxf(fmaf(A, t2 - mx_s[r], B * (t * t - my_s[r])), 0.f);
        atomicMax(rx_b + r, __float_as_int((es + T) / A));
        atomicMax(ry_b + r, __float_as_int((es + T) / B));
        acc[f] = 0ull;   // the key of this cell has been read
    }
    __syncthreads();

    // ---- pass 2: the shifted sums over the points that can matter ----
    for (int64_t base = (int64_t)warp * 32; base < N; base += NW * 32) {
        const int64_t i = base + lane;
        const bool v = i < N;
        const int64_t ic = v ? i : base;
        float xi[8];
#pragma unroll
        for (int cc = 0; cc < 8; ++cc) xi[cc] = cc < d ? a.xs[(int64_t)cc * Np + CDE_CK(ic, N, 108)] : 0.f;
        const float yi = a.y[ic];
        for (int r = 0; r < JW; ++r) {
            const int f0 = rs[r], f1 = re[r];
            if (f0 == f1) continue;
            float dx2, dy2;
            dist(r, xi, ic, yi, dx2, dy2);
            const float RXd = mx_s[r] + __int_as_float(rx_b[r]), RYd = my_s[r] + __int_as_float(ry_b[r]);
            const bool in = v && i != ji_s[r] && dx2 <= RXd && dy2 <= RYd;
            const unsigned m = __ballot_sync(0xffffffffu, in);
            if (m == 0u) continue;
            if (in) {
                const int p = __popc(m & ((1u << lane) - 1u));
                lx[p] = dx2;
                ly[p] = dy2;
            }
            __syncwarp();
            const int nc = __popc(m);
            for (int f = f0 + lane; f < f1; f += 32) {
                const float A = As[f], B = Bs[f], dxf = dxs[f], dyf = dys[f];
                float s = 0.f;
                for (int q = 0; q < nc; ++q)
                    s += ex2_approx(kFbEx2Fix - (A * (lx[q] - dxf) + B * (ly[q] - dyf)));
                const unsigned long long qv = __float2ull_rn(s * scale);
                if (qv) atomicAdd(acc + f, qv);
            }
            __syncwarp();
        }
    }
    __syncthreads();
    for (int f = tid; f < nfl; f += NT) {
        const int c = flag_s[f], r = c / GG;
        const float tot = (float)((double)acc[f] * (double)inv_scale_f);
        const double es = (double)As[f] * ((double)dxs[f] - (double)mx_s[r]) +
                          (double)Bs[f] * ((double)dys[f] - (double)my_s[r]);
        la2[c] = -es + log2_wide(tot);
    }
    __syncthreads();
}

// Per-unit epilogue shared by the tile bodies.  On entry At[m] holds the
// warp-combined shifted numerator of cell tid + 256 m and btl_s the FP64 log2
// of the shifted denominators; `big` (the first BIG floats of shared memory)
// is free.  Flags cells below the threshold, recomputes them exactly, and adds
// the FP64 log-ratios of the unit's rows into the tile partial (thread-owned
// cells, rows in order; `first`: the tile's first unit, which stores instead).
template <class C, int KERN, class Coef>
__device__ __forceinline__ void loo_unit_epilogue(const LooArgs& a, const Coef& cf, float* sm, int u,
                                                  bool first, int tile,
                                                  const float (&At)[(C::JW * C::GG + 255) / 256]) {
    constexpr int JW = C::JW, GG = C::GG, G1 = C::G1v, G2 = C::G2v, CELLS = JW * GG;
    constexpr double LN2 = 0.69314718055994530942;
    const int tid = threadIdx.x;
    const int d = a.d;
    float* big = sm;
    float* mx_s = sm + C::off_mx(d);
    float* my_s = sm + C::off_my(d);
    int* vr_s = reinterpret_cast<int*>(sm + C::off_vr(d));
    double* btl_s = reinterpret_cast<double*>(sm + C::off_btl(d));
    int* flag_s = reinterpret_cast<int*>(sm + C::off_flag(d));
    int* nflag_s = reinterpret_cast<int*>(sm + C::off_nflag(d));
        // ---- shifted log numerators; flag cells that lost range ----
        double* la2 = reinterpret_cast<double*>(big);
        constexpr int NC = (CELLS + 255) / 256;
        // cell c of this thread: its log numerator, unless it is to be recomputed.  Cells of
        // the padded grid (the last bandwidth repeated) are never output: they are not
        // recomputed either.
        const auto flagged = [&](int m, int c) {
            const int jl = c / GG;
            if (!vr_s[jl]) return false;
            const float v = At[m];
            const int kl = c - jl * GG;
            const bool padded = kl / G2 >= a.G1r || kl % G2 >= a.G2r;
            if (v >= a.thresh || padded) {
                la2[c] = log2_wide(v);
                return false;
            }
            return true;
        };
        if constexpr (KERN == 0 && C::kOnePass) {
            // list the flagged cells in cell order: offsets from the (m, warp) counts
            const int warp = tid >> 5, lane = tid & 31;
            unsigned fm[NC];
#pragma unroll
            for (int m = 0; m < NC; ++m) {
                const int c = tid + 256 * m;
                const bool f = (CELLS % 256 == 0 || c < CELLS) && flagged(m, c);
                fm[m] = __ballot_sync(0xffffffffu, f);
                if (lane == 0) nflag_s[8 * m + warp] = __popc(fm[m]);
            }
            __syncthreads();
            const int cnt = lane < 8 * NC ? nflag_s[lane] : 0;
            int incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            const int nfl = __shfl_sync(0xffffffffu, incl, 31);
            if (nfl > 0) {
#pragma unroll
                for (int m = 0; m < NC; ++m) {
                    const int b0 = __shfl_sync(0xffffffffu, incl - cnt, 8 * m + warp);
                    if ((fm[m] >> lane) & 1u) flag_s[b0 + __popc(fm[m] & ((1u << lane) - 1u))] = tid + 256 * m;
                }
                __syncthreads();
                loo_fallback<C>(a, cf, sm, nfl);
            }
        } else if constexpr (KERN == 1 && C::kOnePass) {
            // Epanechnikov sums need no shift and no recomputation (at 32 x 32 the branch below,
            // which then flags nothing, leaves the compiler a 1% to 3% faster main loop)
#pragma unroll
            for (int m = 0; m < NC; ++m) {
                const int c = tid + 256 * m;
                if (CELLS % 256 == 0 || c < CELLS) la2[c] = log2_wide(At[m]);
            }
        } else {
#pragma unroll
            for (int m = 0; m < NC; ++m) {
                const int c = tid + 256 * m;
                if (CELLS % 256 != 0 && c >= CELLS) continue;
                if (flagged(m, c)) {
                    const int q = atomicAdd(nflag_s, 1);
                    flag_s[q] = c;
                }
            }
            __syncthreads();
            if constexpr (KERN == 0) {
                // (Epanechnikov sums need no shift: their threshold is 0, nothing is flagged)
                const int nfl = *nflag_s;
                if (nfl > 0) loo_fallback_two_pass<C>(a, cf, sm, nfl);
            }
        }
        __syncthreads();

        // ---- FP64 log-ratio: a row's terms of cell (k, l) ----
        const auto terms = [&](int jl, int k, int l, double a1k, double a2l, double lam, double kap, double& ell,
                               double& lnA) {
            const double shy = a2l * (double)my_s[jl];
            const double lA = la2[jl * GG + k * G2 + l];
            // a zero numerator (Epanechnikov: empty support, also when
            // the denominator is zero) is ell = -inf, never NaN
            ell = lA == -INFINITY ? -INFINITY : LN2 * (lA - btl_s[jl * G1 + k] - shy) - kap;
            lnA = LN2 * (lA - a1k * (double)mx_s[jl] - shy) - lam - kap;
            if (a.ell_rows && k < a.G1r && l < a.G2r) {
                const int64_t r = CDE_CK((int64_t)u * JW + jl, a.n_rows, 107);
                a.ell_rows[r * a.ell_ld_row + (int64_t)k * a.ell_ld_k + l] = ell;
            }
        };
        // each thread adds whole grid cells (the unit's rows in row order) to the tile partial
        double* part = a.part + CDE_CK(tile, a.n_tiles, 106) * 2 * GG;
        const auto add_cell = [&](int kl, double sc, double se) {
            if (first) {
                part[kl] = sc;
                part[GG + kl] = se;
            } else {
                part[kl] += sc;
                part[GG + kl] += se;
            }
        };
        if constexpr (GG < 256) {
            // fewer cells than threads: every thread forms terms (else GG of the 256 threads
            // would form all JW rows' in turn), then the cells' owners add them in row order
            double* ells = la2 + CELLS;
            double* lnAs = ells + CELLS;
#pragma unroll
            for (int m = 0; m < (CELLS + 255) / 256; ++m) {
                const int c = tid + 256 * m;
                if (CELLS % 256 != 0 && c >= CELLS) continue;
                const int jl = c / GG, kl = c - jl * GG, k = kl / G2, l = kl - k * G2;
                double ell = 0.0, lnA = 0.0;
                if (vr_s[jl]) terms(jl, k, l, (double)cf.a1(k), (double)cf.a2(l), a.lam1[k], a.kap2[l], ell, lnA);
                ells[c] = ell;
                lnAs[c] = lnA;
            }
            __syncthreads();
            if (tid < GG) {
                double sc = 0.0, se = 0.0;
#pragma unroll
                for (int jl = 0; jl < JW; ++jl) {   // rows past the last add an exact 0
                    sc += ells[jl * GG + tid];
                    se += lnAs[jl * GG + tid];
                }
                add_cell(tid, sc, se);
            }
        } else {
#pragma unroll
            for (int s = 0; s < GG / 256; ++s) {
                const int kl = tid + 256 * s;
                const int k = kl / G2, l = kl - k * G2;
                const double a1k = (double)cf.a1(k), a2l = (double)cf.a2(l);
                const double lam = a.lam1[k], kap = a.kap2[l];
                double sc = 0.0, se = 0.0;
                for (int jl = 0; jl < JW; ++jl) {
                    if (!vr_s[jl]) continue;
                    double ell, lnA;
                    terms(jl, k, l, a1k, a2l, lam, kap, ell, lnA);
                    sc += ell;
                    se += lnA;
                }
                add_cell(kl, sc, se);
            }
        }
}

// Grid shapes of the tile kernels: k (h1) padded to an M-tile multiple of 16,
// l (h2) to 8, 16 or 32.  The autotuner's classes are these shapes.
inline int loo_pad1(int g) { return g <= 16 ? 16 : 32; }
inline int loo_pad2(int g) { return g <= 8 ? 8 : (g <= 16 ? 16 : 32); }
// Grids of at most 8 x 8 on the direct kernel (d_x < 16, or `direct`) take the packed
// body (loo_pack.cuh) with 4 or 8 bandwidths per axis, in the 16 x 8 body's place (and
// in its tuning class: the units have the same 8 rows).  The d >= 16 kernel takes the shape
// whose units fill the GPU best.  A row's terms do not depend on the shape.
void loo_shape(int sm_count, const Dataset& D, int g1, int g2, bool direct, int& T1, int& T2);
// rows per unit of a (direct) shape
inline int loo_unit_rows(int T1, int T2) { return T1 < 16 ? 8 : 1024 / (T1 * T2); }

int launch_loo_tile_kernel(int T1, int T2, const LooArgs& a, int grid, cudaStream_t st);
// the tile partials of one grid block summed into Lc, Le (row stride ld; either may be null)
int loo_final_enqueue(const double* part, int n_tiles, int T1, int T2, int g1, int g2, int ld, int64_t N, double* Lc,
                      double* Le, cudaStream_t st);
// d_x >= 16: the kernel with the x cross-term on the tensor cores (loo_gram.cu)
constexpr int kGramMinD = 16;
int launch_loo_gram(int T1, int T2, const LooArgs& a, int grid, cudaStream_t st);
int loo_gram_rows_per_unit(int T1, int T2);
size_t loo_gram_fb_bytes_per_cta();
size_t loo_gram_smem_bytes(int T1, int T2, int d);
// whether a grid block of this shape over this dataset runs on the d >= 16 kernel
bool loo_use_gram(const Dataset& D, int T1, int T2);
void fill_loo_args(LooArgs& a, const Dataset& D, const double* h1, int g1, const double* h2,
                   int g2, int T1, int T2);
// units per tile of a grid block shape over n_rows rows (the tuned value when set; n_rows = 0:
// the per-shape default without the small-grid reduction)
int loo_units_per_tile(cde_ctx* ctx, int T1, int T2, int64_t n_rows);
// the autotuner's candidate for a shape class, used by this thread's launches only
void tuning_candidate(int T1, int T2, int units_per_tile, int ctas_per_sm);
void tuning_candidate_clear();

// (the launch plan behind the opaque LooChunked of cde_internal.h)
struct LooChunked {
    LooArgs a;
    int T1, T2, G1, G2;
    bool gram;
    int n_tiles, cmax;
    size_t part_bytes, fb_bytes, bytes;
    int64_t N;
    int next_l;     // levels < next_l are done
    int next_m;     // level next_l: units m < next_m of its tiles are done
    int next_t;     // small tiles: tiles < next_t are done
};
int loo_grid_ctas(cde_ctx* ctx, int T1, int T2);

}  // namespace cde
