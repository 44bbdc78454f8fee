// Tile body of the leave-one-out grid kernel for grids of at most 8 x 8
// bandwidths: several rows share one MMA tile.
//
// The sums are those of loo_mma.cuh (At_j(k,l) = sum_i u_i(k) w_i(l), with the
// same factors, splits, 64-point chunks and warp order, so every row's result
// is bitwise the one of the 16 x 8 body).  That body gives a row a whole
// m16n8 tile; of a 4 x 4 grid it uses 16 of the 128 accumulators and makes 24
// factors per pair where 8 are needed.  Here an M tile holds RM = 16 / K1 rows
// (K1 = G1 padded to 4 or 8) and an N tile RN = 8 / K2 rows (K2 likewise), and
// an N tile is multiplied with the one M tile that holds its rows.  The
// accumulators whose two rows differ are the price (they are ignored): what is
// saved is factors, splits and MMAs.  Per 8 rows and 8 points:
//
//               16 x 8 body   8 x 8   8 x 4   4 x 8   4 x 4
//   ex2             48          32      24      24      16
//   MMAs            16          16       8      16       8
//
// The distance pass takes the 8 rows of a unit together (rows in packed FP32x2
// pairs, two points per lane), so a point's coordinates are loaded once per
// chunk and not once per row: at d_x > 8 those reloads were most of the 16 x 8
// body's time.  The valid accumulators of an N tile are two per lane, so the
// FP32 running totals stay in registers.
//
// Bound by instruction issue (61% active, the tensor pipe 9%).  Measured against the
// 16 x 8 body, tile kernel alone: N = 24,007, d = 12, 4 x 4: 8.3 -> 5.2 ms, of which
// the exact recomputation of underflowing cells was 3.7 ms on both sides (4.6 -> 1.5 ms
// without it; with the one-pass recomputation of loo_common.cuh 2.5 ms in all);
// N = 2,000, d = 1, 8 x 8: 63 -> 51 us (then 38).  Grids with more than 8
// bandwidths on an axis keep the one-row tiles: at K1 = 16 nothing is shared.
#pragma once

#include "loo_mma.cuh"

namespace cde {

template <int K1, int K2>
struct PackCfg {
    static_assert((K1 == 4 || K1 == 8) && (K2 == 4 || K2 == 8), "rows per tile");
    static constexpr int kThreads = 256, kWarps = 8;
    static constexpr int G1v = K1, G2v = K2, GG = K1 * K2;
    static constexpr int JW = 8;                    // rows per unit
    static constexpr int RM = 16 / K1, RN = 8 / K2; // rows per M tile, per N tile
    static constexpr int MT = JW / RM, NT = JW / RN;
    static constexpr int IC = 64;
    // per warp: t1 of each row pair (a, b) interleaved by point, t2 of each row; the
    // strides put the two row groups that lanes of one load read on different banks
    static constexpr int T1S = 2 * IC + 16, T2S = IC + 8;
    static constexpr int WST = (JW / 2) * T1S + JW * T2S;
    static constexpr int COMB = kWarps * JW * GG + kWarps * JW * K1;
    __host__ __device__ static int big(int) {
        const int s = kWarps * WST, f = 36 * JW * GG;   // f: the exact recomputation
        const int m = s > COMB ? s : COMB;
        return m > f ? m : f;
    }
    __host__ __device__ static int dpad(int d) { return JW * d; }
    __host__ __device__ static int off_xj(int d) { return big(d); }                   // [JW][d]
    __host__ __device__ static int off_xp(int d) { return off_xj(d) + dpad(d); }      // [d][JW], row pairs adjacent
    __host__ __device__ static int off_yj(int d) { return off_xp(d) + dpad(d); }
    __host__ __device__ static int off_mx(int d) { return off_yj(d) + 16; }
    __host__ __device__ static int off_my(int d) { return off_yj(d) + 32; }
    __host__ __device__ static int off_ji(int d) { return off_yj(d) + 48; }
    __host__ __device__ static int off_vr(int d) { return off_yj(d) + 64; }
    __host__ __device__ static int off_rp(int d) { return off_yj(d) + 80; }           // pair order: y, mx, my, j
    __host__ __device__ static int off_btl(int d) { return off_rp(d) + 4 * JW; }
    __host__ __device__ static int off_flag(int d) { return off_btl(d) + 2 * JW * K1; }
    __host__ __device__ static int off_nflag(int d) { return off_flag(d) + JW * GG; }
    // exact recomputation (see MmaCfg): one round holds every cell
    static constexpr bool kOnePass = true;
    static constexpr int FBCAP = JW * GG;
    static constexpr int FBW = kWarps * 144 + 2 * 8;
    __host__ __device__ static int off_fbw(int d) { return off_nflag(d) + 32; }
    __host__ __device__ static int off_fbS(int) { return 4 * JW * GG; }
    __host__ __device__ static int off_fbX(int) { return (4 + kWarps) * JW * GG; }
    __host__ __device__ static int off_fbC(int) { return (4 + 3 * kWarps) * JW * GG; }
    static size_t smem_bytes(int d) { return (size_t)(off_fbw(d) + FBW) * sizeof(float); }
    // position of row r in the pair order: its pair (one row of each half of the M
    // tile), then its half
    __host__ __device__ static constexpr int pair_pos(int r) {
        const int mt = r / RM, w = r % RM;
        return 2 * (mt * (RM / 2) + w % (RM / 2)) + w / (RM / 2);
    }
};

// hi = TF32 truncation, lo the remainder (u: exact; w: w' r - hi, see loo_mma.cuh)
__device__ __forceinline__ float2 tf32_trunc2(float2 v) {
    return make_float2(__uint_as_float(__float_as_uint(v.x) & 0xffffe000u),
                       __uint_as_float(__float_as_uint(v.y) & 0xffffe000u));
}

template <int K1, int K2, int KERN, class Coef>
__device__ __forceinline__ void loo_tile_pack(const LooArgs& a, const Coef& cf, int tile, float* sm) {
    using C = PackCfg<K1, K2>;
    constexpr int JW = C::JW, RM = C::RM, RN = C::RN, MT = C::MT, NT = C::NT, GG = C::GG, IC = C::IC;
    constexpr int NP = JW / 2, CELLS = JW * GG;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, t = lane & 3;
    const int d = a.d;
    float* xj_s = sm + C::off_xj(d);
    float* xp_s = sm + C::off_xp(d);
    float* rp_s = sm + C::off_rp(d);
    long long* ji_s = reinterpret_cast<long long*>(sm + C::off_ji(d));
    int* vr_s = reinterpret_cast<int*>(sm + C::off_vr(d));
    double* btl_s = reinterpret_cast<double*>(sm + C::off_btl(d));
    float* t1s = sm + warp * C::WST;
    float* t2s = t1s + NP * C::T1S;
    // this lane's fragment rows and columns: A row g (and g + 8) is bandwidth g % K1 of
    // row h of the tile's first (second) half; B column g is bandwidth g % K2 of row g / K2
    const int h = g / K1, rn = g / K2;
    const float ca = cf.a1(g % K1), cb = cf.a2(g % K2);
    const float2 ca2 = make_float2(ca, ca), cb2 = make_float2(cb, cb);

    __shared__ int ls_u, ls_end, ls_stride, ls_first;   // the unit loop's state (loo_mma.cuh)
    if (tid == 0) {
        int u_first, u_stride, u_len;
        loo_tile_span(a, tile, u_first, u_stride, u_len);
        ls_u = u_first + max(a.win0, 0) * u_stride;
        ls_end = u_first + min(u_len, a.win1) * u_stride;
        ls_stride = u_stride;
        ls_first = u_first;
    }
    const int64_t N = a.N, Np = a.Np;
    const int64_t n_chunks = (N + IC - 1) / IC;
    const int N32 = (int)N;  // N < 2^31

    for (;;) {
        __syncthreads();
        const int u = ls_u;
        if (u >= ls_end) break;
        const bool first_u = u == ls_first;
        if (tid < JW) {
            const int64_t r = (int64_t)u * JW + tid;
            const bool v = r < a.n_rows;
            const int64_t r0 = v ? r : 0;
            const int64_t j = CDE_CK(a.rows ? a.rows[CDE_CK(r0, a.n_rows, 131)] : r0, a.N, 132);
            const int p = C::pair_pos(tid);
            const float yj = a.y[j], mx = a.mx[j], my = a.my[j];
            ji_s[tid] = j;
            vr_s[tid] = v;
            (sm + C::off_yj(d))[tid] = yj;
            (sm + C::off_mx(d))[tid] = mx;
            (sm + C::off_my(d))[tid] = my;
            rp_s[p] = yj;
            rp_s[JW + p] = mx;
            rp_s[2 * JW + p] = my;
            reinterpret_cast<int*>(rp_s)[3 * JW + p] = (int)j;
        }
        __syncthreads();
        for (int e = tid; e < JW * d; e += C::kThreads) {
            const int r = e & (JW - 1), c = e / JW;
            const float v = a.xs[(int64_t)c * Np + ji_s[r]];
            xj_s[r * d + c] = v;
            xp_s[c * JW + C::pair_pos(r)] = v;
        }
        __syncthreads();

        float2 tot[NT];   // running totals: the valid accumulators of each N tile
        float2 bt[MT];    // denominator partials of the M tile's rows h and RM / 2 + h
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) tot[nt] = make_float2(0.f, 0.f);
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) bt[mt] = make_float2(0.f, 0.f);

        // points 2 lane, 2 lane + 1 of the chunk: y and the first 8 coordinates, one chunk ahead
        float2 xin[8], yin;
        int64_t ch = warp;
        if (ch < n_chunks) {
            const int64_t i = CDE_CK(ch * IC + 2 * lane, Np - 1, 133);
#pragma unroll
            for (int c = 0; c < 8; ++c)
                xin[c] = c < d ? *reinterpret_cast<const float2*>(a.xs + (int64_t)c * Np + i) : make_float2(0.f, 0.f);
            yin = *reinterpret_cast<const float2*>(a.y + i);
        }
        for (; ch < n_chunks; ch += C::kWarps) {
            // ---- distance pass: all rows of the unit, rows in packed pairs ----
            __syncwarp();
            {
                const int64_t i0 = ch * IC + 2 * lane;
                float2 dx2[NP][2];
#pragma unroll
                for (int p = 0; p < NP; ++p) dx2[p][0] = dx2[p][1] = make_float2(0.f, 0.f);
                const auto add_dim = [&](int c, float2 x) {
                    const float4* xr = reinterpret_cast<const float4*>(xp_s + c * JW);
#pragma unroll
                    for (int q = 0; q < JW / 4; ++q) {
                        const float4 v = xr[q];
                        const float2 rr[2] = {make_float2(v.x, v.y), make_float2(v.z, v.w)};
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const float2 q0 = __fadd2_rn(rr[e], make_float2(-x.x, -x.x));
                            const float2 q1 = __fadd2_rn(rr[e], make_float2(-x.y, -x.y));
                            dx2[2 * q + e][0] = __ffma2_rn(q0, q0, dx2[2 * q + e][0]);
                            dx2[2 * q + e][1] = __ffma2_rn(q1, q1, dx2[2 * q + e][1]);
                        }
                    }
                };
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    if (c < d) add_dim(c, xin[c]);
                for (int c = 8; c < d; c += 4) {
                    float2 xv[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        xv[e] = c + e < d ? *reinterpret_cast<const float2*>(a.xs + (int64_t)(c + e) * Np +
                                                                             CDE_CK(i0, Np - 1, 134))
                                          : make_float2(0.f, 0.f);
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (c + e < d) add_dim(c + e, xv[e]);
                }
                const bool v0 = (int)i0 < N32, v1 = (int)i0 + 1 < N32;
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    const float2 yr = *reinterpret_cast<const float2*>(rp_s + 2 * p);
                    const int2 jr = *reinterpret_cast<const int2*>(rp_s + 3 * JW + 2 * p);
                    const float2 dy0 = __fadd2_rn(yr, make_float2(-yin.x, -yin.x));
                    const float2 dy1 = __fadd2_rn(yr, make_float2(-yin.y, -yin.y));
                    const float2 e0 = __fmul2_rn(dy0, dy0), e1 = __fmul2_rn(dy1, dy1);
                    const bool oka0 = v0 && (int)i0 != jr.x, okb0 = v0 && (int)i0 != jr.y;
                    const bool oka1 = v1 && (int)i0 + 1 != jr.x, okb1 = v1 && (int)i0 + 1 != jr.y;
                    float2 s0, s1, w0, w1;
                    if constexpr (KERN == 0) {
                        // shifted exponents; masked pairs -inf in both (loo_mma.cuh)
                        const float2 mx = *reinterpret_cast<const float2*>(rp_s + JW + 2 * p);
                        const float2 my = *reinterpret_cast<const float2*>(rp_s + 2 * JW + 2 * p);
                        s0 = __fadd2_rn(mx, make_float2(-dx2[p][0].x, -dx2[p][0].y));
                        s1 = __fadd2_rn(mx, make_float2(-dx2[p][1].x, -dx2[p][1].y));
                        w0 = __fadd2_rn(my, make_float2(-e0.x, -e0.y));
                        w1 = __fadd2_rn(my, make_float2(-e1.x, -e1.y));
                        s0 = make_float2(oka0 ? s0.x : -INFINITY, okb0 ? s0.y : -INFINITY);
                        s1 = make_float2(oka1 ? s1.x : -INFINITY, okb1 ? s1.y : -INFINITY);
                        w0 = make_float2(oka0 ? w0.x : -INFINITY, okb0 ? w0.y : -INFINITY);
                        w1 = make_float2(oka1 ? w1.x : -INFINITY, okb1 ? w1.y : -INFINITY);
                    } else {
                        // squared distances; masked pairs +inf
                        s0 = make_float2(oka0 ? dx2[p][0].x : INFINITY, okb0 ? dx2[p][0].y : INFINITY);
                        s1 = make_float2(oka1 ? dx2[p][1].x : INFINITY, okb1 ? dx2[p][1].y : INFINITY);
                        w0 = e0;
                        w1 = e1;
                    }
                    const int ra = (p / (RM / 2)) * RM + p % (RM / 2), rb = ra + RM / 2;   // the pair's rows
                    *reinterpret_cast<float4*>(t1s + p * C::T1S + 4 * lane) = make_float4(s0.x, s0.y, s1.x, s1.y);
                    *reinterpret_cast<float2*>(t2s + ra * C::T2S + 2 * lane) = make_float2(w0.x, w1.x);
                    *reinterpret_cast<float2*>(t2s + rb * C::T2S + 2 * lane) = make_float2(w0.y, w1.y);
                }
            }
            if (ch + C::kWarps < n_chunks) {
                const int64_t i = CDE_CK((ch + C::kWarps) * IC + 2 * lane, Np - 1, 135);
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    xin[c] = c < d ? *reinterpret_cast<const float2*>(a.xs + (int64_t)c * Np + i) : make_float2(0.f, 0.f);
                yin = *reinterpret_cast<const float2*>(a.y + i);
            }
            __syncwarp();
            // ---- MMA pass: IC / 8 k-steps of 8 points ----
            float D[NT][4];
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int q = 0; q < 4; ++q) D[nt][q] = 0.f;
#pragma unroll 4
            for (int s = 0; s < IC / 8; ++s) {
                const int pt = 8 * s + 2 * t;   // this lane's points pt, pt + 1
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    // A: (row h, pt), (row RM/2 + h, pt), then the same at pt + 1
                    const float4 q1 = *reinterpret_cast<const float4*>(t1s + (mt * (RM / 2) + h) * C::T1S + 2 * pt);
                    const float2 p0 = make_float2(q1.x, q1.y), p1 = make_float2(q1.z, q1.w);
                    const float2 u0 = KERN == 0 ? gauss_factor2(ca2, p0, kEx2Fix) : kernel_factor2<KERN>(ca2, p0);
                    const float2 u1 = KERN == 0 ? gauss_factor2(ca2, p1, kEx2Fix) : kernel_factor2<KERN>(ca2, p1);
                    bt[mt] = __fadd2_rn(bt[mt], __fadd2_rn(u0, u1));
                    const float2 h0 = tf32_trunc2(u0), h1 = tf32_trunc2(u1);
                    const float2 l0 = __ffma2_rn(h0, make_float2(-1.f, -1.f), u0);
                    const float2 l1 = __ffma2_rn(h1, make_float2(-1.f, -1.f), u1);
                    const uint32_t ah[4] = {__float_as_uint(h0.x), __float_as_uint(h0.y), __float_as_uint(h1.x),
                                            __float_as_uint(h1.y)};
                    const uint32_t ax[4] = {pack_bf16x2(h0.x, h1.x), pack_bf16x2(h0.y, h1.y),
                                            pack_bf16x2(l0.x, l1.x), pack_bf16x2(l0.y, l1.y)};
                    // the N tiles of this M tile's rows
#pragma unroll
                    for (int n = 0; n < RM / RN; ++n) {
                        const int nt = mt * (RM / RN) + n;
                        const float2 t2p = *reinterpret_cast<const float2*>(t2s + (nt * RN + rn) * C::T2S + pt);
                        const float2 w = KERN == 0 ? gauss_factor2(cb2, t2p, kWc) : kernel_factor2<KERN>(cb2, t2p);
                        const float2 hw = tf32_trunc2(w);
                        const float2 lw = KERN == 0 ? __ffma2_rn(w, make_float2(kWr, kWr), make_float2(-hw.x, -hw.y))
                                                    : __ffma2_rn(hw, make_float2(-1.f, -1.f), w);
                        mma_tf32(D[nt], ah, __float_as_uint(hw.x), __float_as_uint(hw.y));
                        mma_bf16(D[nt], ax, pack_bf16x2(lw.x, lw.y), pack_bf16x2(hw.x, hw.y));
                    }
                }
            }
            // of an N tile's accumulators the ones with the same row in both tiles count:
            // the first or the second half (the tile's rows are in one half), or, where
            // the N tile holds both rows of the M tile, the half of the column's row
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                const bool second = RM == 2 && RN == 2 ? t >= 2 : ((nt * RN) % RM) >= RM / 2;
                const float2 v = second ? make_float2(D[nt][2], D[nt][3]) : make_float2(D[nt][0], D[nt][1]);
                tot[nt] = __fadd2_rn(tot[nt], v);
            }
        }

        // ---- combine the 8 warps in fixed order ----
        __syncthreads();
        float* accS = sm;
        float* btS = sm + C::kWarps * CELLS;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const int rc = (2 * t) / K2, r = nt * RN + rc;   // the column's row
            if (r % (RM / 2) == h) {
                const int l = (2 * t) % K2;
                *reinterpret_cast<float2*>(accS + warp * CELLS + r * GG + (g % K1) * K2 + l) = tot[nt];
            }
        }
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                float v = q ? bt[mt].y : bt[mt].x;
                v += __shfl_xor_sync(0xffffffffu, v, 1);
                v += __shfl_xor_sync(0xffffffffu, v, 2);
                if (t == 0) btS[(warp * JW + mt * RM + q * (RM / 2) + h) * K1 + g % K1] = v;
            }
        __syncthreads();
        constexpr int NC = (CELLS + 255) / 256;
        float At[NC];
#pragma unroll
        for (int m = 0; m < NC; ++m) {
            const int c = tid + 256 * m;
            float s = 0.f;
            if (c < CELLS)
#pragma unroll
                for (int w = 0; w < C::kWarps; ++w) s += accS[w * CELLS + c];
            At[m] = s;
        }
        for (int e = tid; e < JW * K1; e += C::kThreads) {
            float s = 0.f;
            for (int w = 0; w < C::kWarps; ++w) s += btS[w * JW * K1 + e];
            btl_s[e] = log2_wide(s);
        }
        __syncthreads();
        loo_unit_epilogue<C, KERN>(a, cf, sm, u, first_u, tile, At);
        if (tid == 0) ls_u += ls_stride;
    }
}

// The tile body and layout of a grid shape
template <int G1, int G2, bool Packed = (G1 < 16)>
struct LooBody {
    using Cfg = MmaCfg<G1, G2>;
    template <int KERN, class Coef>
    static __device__ __forceinline__ void tile(const LooArgs& a, const Coef& cf, int t, float* sm) {
        loo_tile_mma<G1, G2, KERN>(a, cf, t, sm);
    }
};
template <int G1, int G2>
struct LooBody<G1, G2, true> {
    using Cfg = PackCfg<G1, G2>;
    template <int KERN, class Coef>
    static __device__ __forceinline__ void tile(const LooArgs& a, const Coef& cf, int t, float* sm) {
        loo_tile_pack<G1, G2, KERN>(a, cf, t, sm);
    }
};

template <int G1, int G2, int KERN>
__global__ void __launch_bounds__(256, 2) k_loo_mma(const LooArgs a) {
    extern __shared__ float4 sm4[];
    __shared__ int next_tile;
    const CoefParam cf{a};
    for (int t0 = blockIdx.x;; t0 += gridDim.x) {
        if (threadIdx.x == 0) next_tile = a.work ? atomicAdd(a.work, 1) : t0;
        __syncthreads();
        const int t = next_tile;
        if (t >= a.n_tiles) break;
        LooBody<G1, G2>::template tile<KERN>(a, cf, t, reinterpret_cast<float*>(sm4));
    }
}

}  // namespace cde
