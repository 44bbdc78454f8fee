// Products of the conditional density estimate at query points, as the
// paper's evaluation uses them (Sec. 4, Sec. 4.2):
//
//   E[y | x_q]      = sum_i u_qi y_i / sum_i u_qi   (the y kernel is symmetric)
//   fhat(y_q | x_q) = sum_i u_qi K_h2(y_q - y_i) / sum_i u_qi   (Eq. 1 at one point)
//   prediction interval: the narrowest window holding a fraction 1 - alpha of
//   S draws from fhat(. | x_q) (Sec. 4).
//
// u_qi are the x weights of Eq. 1 (Gaussian: 2^{a1 (m_q - |x_q - x_i|^2)} with
// the query's nearest squared distance m_q; Epanechnikov: (1 - |x_q - x_i|^2/h1^2)_+).
//
// k_cond_stats: the three sums per query, queries in registers (four per
// thread up to d = 8, two up to 16, else one), data points staged through
// shared memory point-major, the data range split
// over gridDim.y; split partials are summed in FP64 in split order.
//
// k_chunk_weights and k_cond_sample: a draw from fhat(.|x_q) is a mixture
// draw: an index i with probability u_qi / sum u (inverse CDF over the
// cumulative weights), then y_i + h2 e with e from the y kernel (inverse CDF:
// Phi^{-1} for the Gaussian, 2 sin(asin(2V - 1)/3) for the Epanechnikov kernel,
// whose CDF is (2 + 3t - t^3)/4).  The cumulative weights are summed in a fixed
// order: inside a chunk of 256 points by a scan (32-point segments pairwise, then
// the segments in turn), over the chunks in turn.  k_chunk_weights forms the
// chunk totals with one query per lane (the points are broadcast, a segment's
// pairwise sum is a tree in registers: no shuffles and one barrier per chunk);
// k_cond_sample, one CTA per query, sums them, sorts the S index targets, finds each
// target's chunk and 32-point segment in the running totals, and scans only that
// segment (a warp per target, four at a time).  Where a target lies within rounding of
// a prefix (2^-19 relative: the float prefixes of neighbouring points need not be
// ordered there) the whole chunk is scanned and searched, so that every draw is the
// one the search over the chunk's 256 prefixes finds.  The S values are then sorted
// and the narrowest window of ceil((1 - alpha) S) consecutive values is taken.  Random numbers: value k of the SplitMix64 stream of the seed,
// k = 2 (q S + s) for the index draw of sample s of query q and k + 1 for its
// kernel offset; 24 random bits give u = (bits + 1/2) 2^-24 in (0, 1).
#include <algorithm>
#include <cmath>

#include "cde_internal.h"

namespace cde {

__global__ void k_query_pack(const float* __restrict__ xq, int64_t Q, int64_t Qp, int d,
                             const double* __restrict__ stats, float* __restrict__ out);

__device__ __forceinline__ float ex2p(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float fma_sat_p(float a, float b, float c) {
    float r;
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// x weight from the squared distance (Gaussian: shifted by the query's m_q)
template <int KERN>
__device__ __forceinline__ float xweight(float dx2, float a1, float mq) {
    if constexpr (KERN == 0) return ex2p(a1 * (mq - dx2));
    else return fma_sat_p(-a1, dx2, 1.f);
}

// y kernel profile at squared distance t2 (constant applied in the epilogue)
template <int KERN>
__device__ __forceinline__ float yprofile(float t2, float a2) {
    if constexpr (KERN == 0) return ex2p(-a2 * t2);
    else return fma_sat_p(-a2, t2, 1.f);
}

__device__ __forceinline__ uint64_t splitmix64_dev(uint64_t seed, uint64_t k) {
    uint64_t z = seed + (k + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__device__ __forceinline__ float uniform24(uint64_t seed, uint64_t k) {
    return ((float)(splitmix64_dev(seed, k) >> 40) + 0.5f) * 0x1p-24f;
}

// --------------------------------------------------------------------------
// Per-query sums
// --------------------------------------------------------------------------
constexpr int kCSThreads = 128;

struct StatArgs {
    const float* xs;   // [d][Np]
    const float* y;    // [Np]
    const float* xq;   // [d][Qp] standardised like the data
    const float* yq;   // [Q] or null
    const float* mq;   // [Q] (Gaussian)
    int64_t N, Np, Q, Qp;
    int d;
    float a1, a2;
    int64_t i_per_split;
    float* part;       // [splits][Q][3]: sum u, sum u y, sum u w
};

template <int KERN, int DREG, int kCSJB>
__global__ void __launch_bounds__(kCSThreads) k_cond_stats(const StatArgs a) {
    __shared__ __align__(16) float xt[kCSThreads][DREG];  // point-major: 128-bit broadcast loads
    __shared__ float yt[kCSThreads];
    const int tid = threadIdx.x;
    const int64_t qbase = (int64_t)blockIdx.x * kCSThreads * kCSJB + tid;
    const int64_t i0 = (int64_t)blockIdx.y * a.i_per_split;
    const int64_t i1 = min(a.N, i0 + a.i_per_split);
    const int d = a.d;
    const bool has_yq = a.yq != nullptr;
    float xq[kCSJB][DREG], yq[kCSJB], mq[kCSJB], amq[kCSJB], S0[kCSJB], S1[kCSJB], S2[kCSJB];
#pragma unroll
    for (int b = 0; b < kCSJB; ++b) {
        const int64_t q = qbase + (int64_t)b * kCSThreads;
        const int64_t qc = q < a.Q ? q : 0;
#pragma unroll
        for (int c = 0; c < DREG; ++c) xq[b][c] = c < d ? a.xq[(int64_t)c * a.Qp + qc] : 0.f;
        yq[b] = has_yq ? a.yq[qc] : 0.f;
        mq[b] = KERN == 0 ? a.mq[qc] : 0.f;
        amq[b] = a.a1 * mq[b];
        S0[b] = S1[b] = S2[b] = 0.f;
    }
    for (int64_t t0 = i0; t0 < i1; t0 += kCSThreads) {
        __syncthreads();
        const int64_t it = CDE_CK(t0 + tid, a.Np, 301);  // < Np: splits and Np are multiples of 128
#pragma unroll
        for (int c = 0; c < DREG; ++c) xt[tid][c] = c < d ? a.xs[(int64_t)c * a.Np + it] : 0.f;
        yt[tid] = a.y[it];
        __syncthreads();
        const int n = (int)min((int64_t)kCSThreads, i1 - t0);
        for (int t = 0; t < n; ++t) {
            const float yi = yt[t];
            float xi[DREG];
#pragma unroll
            for (int c = 0; c < DREG; c += 4) {
                const float4 v4 = *reinterpret_cast<const float4*>(&xt[t][c]);
                xi[c] = v4.x;
                xi[c + 1] = v4.y;
                xi[c + 2] = v4.z;
                xi[c + 3] = v4.w;
            }
            if constexpr (kCSJB % 2 == 0) {
                // two queries per packed FP32x2 instruction (xq - x_i as fma(x_i, -1, xq),
                // the scalar subtraction's rounding; the x argument a1 m_q - a1 dx2 as one FMA)
                const float2 m1 = make_float2(-1.f, -1.f), yi2 = make_float2(yi, yi);
#pragma unroll
                for (int b = 0; b < kCSJB; b += 2) {
                    float2 dx2 = make_float2(0.f, 0.f);
#pragma unroll
                    for (int c = 0; c < DREG; ++c) {
                        const float2 v = __ffma2_rn(make_float2(xi[c], xi[c]), m1, make_float2(xq[b][c], xq[b + 1][c]));
                        dx2 = __ffma2_rn(v, v, dx2);
                    }
                    float2 u;
                    if constexpr (KERN == 0) {
                        const float2 arg = __ffma2_rn(dx2, make_float2(-a.a1, -a.a1), make_float2(amq[b], amq[b + 1]));
                        u = make_float2(ex2p(arg.x), ex2p(arg.y));
                    } else {
                        u = make_float2(fma_sat_p(-a.a1, dx2.x, 1.f), fma_sat_p(-a.a1, dx2.y, 1.f));
                    }
                    const float2 s0 = __fadd2_rn(make_float2(S0[b], S0[b + 1]), u);
                    const float2 s1 = __ffma2_rn(u, yi2, make_float2(S1[b], S1[b + 1]));
                    S0[b] = s0.x;
                    S0[b + 1] = s0.y;
                    S1[b] = s1.x;
                    S1[b + 1] = s1.y;
                    if (has_yq) {
                        const float2 dy = __ffma2_rn(yi2, m1, make_float2(yq[b], yq[b + 1]));
                        const float2 t2 = __fmul2_rn(dy, dy);
                        float2 w;
                        if constexpr (KERN == 0) {
                            const float2 arg = __fmul2_rn(make_float2(-a.a2, -a.a2), t2);
                            w = make_float2(ex2p(arg.x), ex2p(arg.y));
                        } else {
                            w = make_float2(fma_sat_p(-a.a2, t2.x, 1.f), fma_sat_p(-a.a2, t2.y, 1.f));
                        }
                        const float2 s2 = __ffma2_rn(u, w, make_float2(S2[b], S2[b + 1]));
                        S2[b] = s2.x;
                        S2[b + 1] = s2.y;
                    }
                }
            } else {
#pragma unroll
                for (int b = 0; b < kCSJB; ++b) {
                    float dx2 = 0.f;
#pragma unroll
                    for (int c = 0; c < DREG; ++c) {
                        const float v = xq[b][c] - xi[c];
                        dx2 = fmaf(v, v, dx2);
                    }
                    const float u = xweight<KERN>(dx2, a.a1, mq[b]);
                    S0[b] += u;
                    S1[b] = fmaf(u, yi, S1[b]);
                    if (has_yq) {
                        const float dy = yq[b] - yi;
                        S2[b] = fmaf(u, yprofile<KERN>(dy * dy, a.a2), S2[b]);
                    }
                }
            }
        }
    }
#pragma unroll
    for (int b = 0; b < kCSJB; ++b) {
        const int64_t q = qbase + (int64_t)b * kCSThreads;
        if (q >= a.Q) continue;
        float* p = a.part + ((int64_t)blockIdx.y * a.Q + q) * 3;
        p[0] = S0[b];
        p[1] = S1[b];
        p[2] = S2[b];
    }
}

// mean = sum u y / sum u (NaN when sum u = 0), fat = norm * sum u w / sum u (0 then).
// A CTA sums 16 queries' split partials in FP64, sixteen threads per query over the splits
// (one thread per query waited for one strided load after the other: 173 us for 1,000
// queries x 391 splits).
__global__ void __launch_bounds__(256) k_cond_stats_final(const float* __restrict__ part, int n_split, int64_t Q,
                                                          double norm, double* __restrict__ mean,
                                                          double* __restrict__ fat) {
    constexpr int NG = 16;
    __shared__ double red[NG][16][3];
    const int lane = threadIdx.x & 15, g = threadIdx.x >> 4;
    const int64_t q = (int64_t)blockIdx.x * 16 + lane;
    double s0 = 0, s1 = 0, s2 = 0;
    if (q < Q) {
#pragma unroll 8
        for (int s = g; s < n_split; s += NG) {
            const float* p = part + ((int64_t)s * Q + q) * 3;
            s0 += p[0];
            s1 += p[1];
            s2 += p[2];
        }
    }
    red[g][lane][0] = s0;
    red[g][lane][1] = s1;
    red[g][lane][2] = s2;
    __syncthreads();
    if (g != 0 || q >= Q) return;
#pragma unroll
    for (int w = 1; w < NG; ++w) {
        s0 += red[w][lane][0];
        s1 += red[w][lane][1];
        s2 += red[w][lane][2];
    }
    if (mean) mean[q] = s1 / s0;
    if (fat) fat[q] = s0 > 0.0 ? norm * s2 / s0 : 0.0;
}

// --------------------------------------------------------------------------
// Sampling and the narrowest interval
// --------------------------------------------------------------------------
constexpr int kSmpThreads = 256, kSmpWarps = kSmpThreads / 32, kSmpMax = 4096;
constexpr int kChunk = 256;           // points per chunk of the cumulative weights
constexpr int kSegs = kChunk / 32;    // its 32-point segments
constexpr int kEndsMax = 2048;        // chunk ends kept in shared memory

struct SampleArgs {
    const float* xs;
    const float* y;
    const float* xq;   // [d][Qp]
    const float* mq;   // [Q] (Gaussian)
    int64_t N, Np, Q, Qp;
    int64_t q0, nq;    // this launch's queries q0 .. q0 + nq - 1
    int64_t n_chunks;
    int d, S, SP, m_keep;   // samples, padded power of two, window size ceil((1-alpha) S)
    float a1, h2;
    uint64_t seed;
    float* ct;         // [n_chunks][8][nq] running sums of a chunk after each of its 32-point segments
    float* ends;       // [n_chunks][nq] running totals after each chunk (more than kEndsMax chunks)
    float* lo;         // [Q]
    float* hi;         // [Q]
    float* samples;    // [Q][S] sorted, or null
};

// pairwise sum of n consecutive terms: f(p) the p-th
template <int n, class F>
__device__ __forceinline__ float2 tree_sum2(const F& f, int p) {
    if constexpr (n == 1) return f(p);
    else return __fadd2_rn(tree_sum2<n / 2>(f, p), tree_sum2<n / 2>(f, p + n / 2));
}

// Chunk totals: two queries per thread (packed FP32x2), points point-major in shared
// memory.  Points past N are infinitely far (weight exactly 0).
constexpr int kCwThreads = 64, kCwQ = 2 * kCwThreads;

template <int KERN, int DREG>
__global__ void __launch_bounds__(kCwThreads) k_chunk_weights(const SampleArgs a, int64_t chunks_per_cta) {
    constexpr int TP = DREG > 32 ? kChunk / 2 : kChunk;   // points staged at a time (at most 32 KB)
    __shared__ __align__(16) float xt[TP][DREG];
    const int tid = threadIdx.x;
    const int64_t qa = a.q0 + (int64_t)blockIdx.x * kCwQ + tid, qb = qa + kCwThreads, qe = a.q0 + a.nq;
    const int64_t qac = qa < qe ? qa : a.q0, qbc = qb < qe ? qb : a.q0;
    const int d = a.d;
    float2 xq[DREG];
#pragma unroll
    for (int c = 0; c < DREG; ++c)
        xq[c] = c < d ? make_float2(a.xq[(int64_t)c * a.Qp + qac], a.xq[(int64_t)c * a.Qp + qbc])
                      : make_float2(0.f, 0.f);
    const float2 mq = KERN == 0 ? make_float2(a.mq[qac], a.mq[qbc]) : make_float2(0.f, 0.f);
    const float a1 = a.a1;
    const int64_t k1 = min(a.n_chunks, ((int64_t)blockIdx.y + 1) * chunks_per_cta);
    for (int64_t k = (int64_t)blockIdx.y * chunks_per_cta; k < k1; ++k) {
        const auto weight = [&](int p) {
            float2 dx2 = make_float2(0.f, 0.f);
#pragma unroll
            for (int c = 0; c < DREG; c += 4) {
                const float4 v = *reinterpret_cast<const float4*>(&xt[p][c]);
                const float x[4] = {-v.x, -v.y, -v.z, -v.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 t = __fadd2_rn(xq[c + e], make_float2(x[e], x[e]));
                    dx2 = __ffma2_rn(t, t, dx2);
                }
            }
            if constexpr (KERN == 0) {
                const float2 arg = __fmul2_rn(make_float2(a1, a1), __fadd2_rn(mq, make_float2(-dx2.x, -dx2.y)));
                return make_float2(ex2p(arg.x), ex2p(arg.y));
            } else {
                return make_float2(fma_sat_p(-a1, dx2.x, 1.f), fma_sat_p(-a1, dx2.y, 1.f));
            }
        };
        float2 tot = make_float2(0.f, 0.f);
#pragma unroll 1
        for (int p0 = 0; p0 < kChunk; p0 += TP) {
            __syncthreads();
            for (int p = tid; p < TP; p += kCwThreads) {
                const int64_t i = k * kChunk + p0 + p;
#pragma unroll
                for (int c = 0; c < DREG; ++c)
                    xt[p][c] = c < d ? (i < a.N ? a.xs[(int64_t)c * a.Np + CDE_CK(i, a.Np, 303)] : INFINITY) : 0.f;
            }
            __syncthreads();
            // (the first segment's sum plus an exact 0)
#pragma unroll 1
            for (int s = 0; s < TP; s += 32) {
                tot = __fadd2_rn(tree_sum2<32>(weight, s), tot);
                float* ct = a.ct + (k * kSegs + (p0 + s) / 32) * a.nq;
                if (qa < qe) ct[qa - a.q0] = tot.x;
                if (qb < qe) ct[qb - a.q0] = tot.y;
            }
        }
    }
}

struct SampleSmem {
    float val[kSmpMax];   // targets, then sample values
    int idx[kSmpMax];     // resolved data index per target
    float ends[kEndsMax]; // running totals after each chunk (a tile of them at a time)
    float P[kSmpWarps][kChunk]; // inclusive scan of a warp's chunk
    float xq[kMaxD];
    float total;
    int last;             // the last chunk with weight
    float best_w[kSmpWarps];
    int best_k[kSmpWarps];
};

__device__ __forceinline__ void bitonic_sort(float* v, int n) {
    for (int k = 2; k <= n; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < n; i += blockDim.x) {
                const int ixj = i ^ j;
                if (ixj > i) {
                    const bool up = (i & k) == 0;
                    const float x = v[i], z = v[ixj];
                    if ((x > z) == up) {
                        v[i] = z;
                        v[ixj] = x;
                    }
                }
            }
            __syncthreads();
        }
}

// inclusive scan over the warp in the fixed (shuffle) order of the cumulative weights
__device__ __forceinline__ float warp_scan(float v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float n = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += n;
    }
    return v;
}

// One chunk's weights (point 32 s + lane of the chunk in u[s])
template <int KERN>
__device__ __forceinline__ void chunk_weights(const SampleArgs& a, const SampleSmem& S, int64_t k, float mq,
                                              float (&u)[kChunk / 32]) {
    constexpr int NS = kChunk / 32;
    const int lane = threadIdx.x & 31;
    const float* x = a.xs + CDE_CK(k * kChunk, a.Np - kChunk + 1, 304) + lane;   // Np is a multiple of 256
    float dx2[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) dx2[s] = 0.f;
    for (int c = 0; c < a.d; ++c) {
        const float xqc = S.xq[c];
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const float v = xqc - x[(int64_t)c * a.Np + 32 * s];
            dx2[s] = fmaf(v, v, dx2[s]);
        }
    }
#pragma unroll
    for (int s = 0; s < NS; ++s)
        u[s] = k * kChunk + 32 * s + lane < a.N ? xweight<KERN>(dx2[s], a.a1, mq) : 0.f;
}

template <int KERN>
__global__ void __launch_bounds__(kSmpThreads) k_cond_sample(const SampleArgs a) {
    extern __shared__ float4 smp4[];
    SampleSmem& S = *reinterpret_cast<SampleSmem*>(smp4);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t q = a.q0 + blockIdx.x;
    const int64_t nch = a.n_chunks;
    const float* ct = a.ct + blockIdx.x;   // stride nq
    float* ge = a.ends + blockIdx.x;
    for (int c = tid; c < a.d; c += kSmpThreads) S.xq[c] = a.xq[(int64_t)c * a.Qp + q];
    const float mq = KERN == 0 ? a.mq[q] : 0.f;
    if (tid == 0) {
        S.total = 0.f;
        S.last = -1;
    }
    // running totals over the chunks, in turn (more than kEndsMax chunks: also to global)
    const bool local = nch <= kEndsMax;
    for (int64_t k0 = 0; k0 < nch; k0 += kEndsMax) {
        const int n = (int)min((int64_t)kEndsMax, nch - k0);
        __syncthreads();
        int last = -1;
        for (int k = tid; k < n; k += kSmpThreads) {
            const float v = ct[((k0 + k) * kSegs + kSegs - 1) * a.nq];
            S.ends[k] = v;
            if (v > 0.f) last = (int)(k0 + k);
        }
        if (last >= 0) atomicMax(&S.last, last);
        __syncthreads();
        if (tid == 0) {
            float t = S.total;
#pragma unroll 8
            for (int k = 0; k < n; ++k) {
                t = t + S.ends[k];
                S.ends[k] = t;
            }
            S.total = t;
        }
        __syncthreads();
        if (!local)
            for (int k = tid; k < n; k += kSmpThreads) ge[(k0 + k) * a.nq] = S.ends[k];
    }
    const auto end_of = [&](int64_t k) { return k < 0 ? 0.f : local ? S.ends[k] : ge[k * a.nq]; };
    const float total = S.total;
    const int last = S.last;
    if (last < 0 || !(total > 0.f)) {  // no weight (Epanechnikov: no x-neighbour)
        if (tid == 0) {
            a.lo[q] = NAN;
            a.hi[q] = NAN;
        }
        if (a.samples)
            for (int s = tid; s < a.S; s += kSmpThreads) a.samples[q * a.S + s] = NAN;
        return;
    }
    // sorted index targets
    for (int s = tid; s < a.SP; s += kSmpThreads)
        S.val[s] = s < a.S ? uniform24(a.seed, 2 * ((uint64_t)q * a.S + s)) * total : INFINITY;
    __syncthreads();
    bitonic_sort(S.val, a.SP);
    // The index of one target by the whole chunk: its prefixes to shared memory, the first
    // above t by binary search (the same in every lane)
    const auto by_chunk = [&](int64_t k, float t) {
        float u[kSegs];
        chunk_weights<KERN>(a, S, k, mq, u);
        int chunk_last = -1;
        float before = 0.f;   // the segments before this one
#pragma unroll
        for (int g = 0; g < kSegs; ++g) {
            const unsigned pos = __ballot_sync(0xffffffffu, u[g] > 0.f);
            if (pos) chunk_last = 32 * g + 31 - __clz(pos);
            const float v = warp_scan(u[g]);
            const float seg = __shfl_sync(0xffffffffu, v, 31);
            S.P[warp][32 * g + lane] = g > 0 ? v + before : v;
            before = g > 0 ? seg + before : seg;
        }
        __syncwarp();
        int lo = 0, hi = kChunk;  // first prefix above t
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (S.P[warp][mid] <= t) lo = mid + 1;
            else hi = mid;
        }
        __syncwarp();
        if (lo > chunk_last) lo = chunk_last;  // rounding at the chunk's end
        return (int)(k * kChunk + lo);
    };
    // Resolve the targets, 32 at a time per warp.  Lane = target: the first chunk whose end
    // lies above it, then the first of its segments whose running sum does; then four targets
    // at a time, lane = point of the target's segment.
    constexpr float kNear = 0x1p-19f;   // prefixes closer to a target than this (relative) decide nothing
    for (int b0 = 32 * warp; b0 < a.S; b0 += kSmpThreads) {
        const int s = b0 + lane;
        int64_t k = -1;
        int g = 0;
        float t = 0.f, before = 0.f;
        bool whole = false;
        if (s < a.S && S.val[s] < total) {
            const float v = S.val[s];
            int64_t lo = 0, hi = nch - 1;   // first chunk with its end above v (the last one's is `total`)
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                if (end_of(mid) > v) hi = mid;
                else lo = mid + 1;
            }
            k = lo;
            t = v - end_of(k - 1);
            const float* seg = ct + k * kSegs * a.nq;
            float c[kSegs];
#pragma unroll
            for (int e = 0; e < kSegs; ++e) c[e] = seg[e * a.nq];
#pragma unroll
            for (int e = 0; e < kSegs; ++e)
                if (c[e] <= t) {
                    g = e + 1;
                    before = c[e];
                }
            whole = g == kSegs || (g > 0 && t - before <= kNear * t);
        }
        const unsigned live = __ballot_sync(0xffffffffu, k >= 0);
        const unsigned full = __ballot_sync(0xffffffffu, whole);
        for (int j0 = 0; j0 < 32; j0 += 4) {
            if (((live >> j0) & 15u) == 0u) continue;
            float u[4], tt[4], bf[4];
            int64_t kk[4];
            int gg[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                kk[e] = __shfl_sync(0xffffffffu, k, j0 + e);
                gg[e] = __shfl_sync(0xffffffffu, g, j0 + e) & (kSegs - 1);
                tt[e] = __shfl_sync(0xffffffffu, t, j0 + e);
                bf[e] = __shfl_sync(0xffffffffu, before, j0 + e);
            }
            float dx2[4] = {0.f, 0.f, 0.f, 0.f};
            const float* x[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)   // (dead targets: the first segment)
                x[e] = a.xs + CDE_CK(max(kk[e], (int64_t)0) * kChunk + 32 * gg[e], a.Np - 31, 306) + lane;
#pragma unroll 4
            for (int c = 0; c < a.d; ++c) {
                const float xqc = S.xq[c];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float v = xqc - x[e][(int64_t)c * a.Np];
                    dx2[e] = fmaf(v, v, dx2[e]);
                }
            }
#pragma unroll
            for (int e = 0; e < 4; ++e)
                u[e] = max(kk[e], (int64_t)0) * kChunk + 32 * gg[e] + lane < a.N ? xweight<KERN>(dx2[e], a.a1, mq) : 0.f;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const unsigned bit = 1u << (j0 + e);
                if (!(live & bit)) continue;
                const float v = warp_scan(u[e]);
                const float P = gg[e] > 0 ? v + bf[e] : v;
                const unsigned below = __ballot_sync(0xffffffffu, P <= tt[e]);
                const bool near = __any_sync(0xffffffffu, fabsf(P - tt[e]) <= kNear * tt[e]);
                int at;
                if (near || (full & bit) || below == 0xffffffffu) at = by_chunk(kk[e], tt[e]);
                else at = (int)(kk[e] * kChunk + 32 * gg[e] + __popc(below));
                if (lane == 0) S.idx[CDE_CK(b0 + j0 + e, kSmpMax, 305)] = at;
            }
        }
    }
    int top = 0;   // first target >= total: from there on the last point with weight
    for (int hi = a.S; top < hi;) {
        const int mid = (top + hi) >> 1;
        if (S.val[mid] < total) top = mid + 1;
        else hi = mid;
    }
    if (top < a.S && warp == 0) {
        float u[kChunk / 32];
        chunk_weights<KERN>(a, S, last, mq, u);
        int at = 0;
#pragma unroll
        for (int g = 0; g < kChunk / 32; ++g) {
            const unsigned pos = __ballot_sync(0xffffffffu, u[g] > 0.f);
            if (pos) at = 32 * g + 31 - __clz(pos);
        }
        for (int s = top + lane; s < a.S; s += 32) S.idx[s] = (int)((int64_t)last * kChunk + at);
    }
    __syncthreads();
    // sample values, sorted
    for (int s = tid; s < a.SP; s += kSmpThreads) {
        float v = INFINITY;
        if (s < a.S) {
            const float V = uniform24(a.seed, 2 * ((uint64_t)q * a.S + s) + 1);
            const float e = KERN == 0 ? normcdfinvf(V) : 2.f * sinf(asinf(2.f * V - 1.f) * (1.f / 3.f));
            v = a.y[CDE_CK(S.idx[s], a.N, 302)] + a.h2 * e;
        }
        S.val[s] = v;
    }
    __syncthreads();
    bitonic_sort(S.val, a.SP);
    // narrowest window of m_keep consecutive values (first minimum)
    const int m = a.m_keep;
    float bw = INFINITY;
    int bk = 0x7fffffff;
    for (int k = tid; k + m - 1 < a.S; k += kSmpThreads) {
        const float w = S.val[k + m - 1] - S.val[k];
        if (w < bw) {
            bw = w;
            bk = k;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ow = __shfl_xor_sync(0xffffffffu, bw, o);
        const int ok = __shfl_xor_sync(0xffffffffu, bk, o);
        if (ow < bw || (ow == bw && ok < bk)) {
            bw = ow;
            bk = ok;
        }
    }
    if ((tid & 31) == 0) {
        S.best_w[tid >> 5] = bw;
        S.best_k[tid >> 5] = bk;
    }
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < kSmpThreads / 32; ++w)
            if (S.best_w[w] < bw || (S.best_w[w] == bw && S.best_k[w] < bk)) {
                bw = S.best_w[w];
                bk = S.best_k[w];
            }
        a.lo[q] = S.val[bk];
        a.hi[q] = S.val[bk + m - 1];
    }
    if (a.samples)
        for (int s = tid; s < a.S; s += kSmpThreads) a.samples[q * a.S + s] = S.val[s];
}

// --------------------------------------------------------------------------
// Host side
// --------------------------------------------------------------------------
// Standardised SoA queries (and the Gaussian shifts) on the stream; caller frees.
static int prep_queries(cde_ctx* ctx, const Dataset& D, const float* d_xq, int64_t Q, int64_t Qp,
                        float** xq_out, float** mq_out, cudaStream_t st) {
    float *xq = nullptr, *mq = nullptr;
    CDE_CUDA(pool_alloc(ctx, (void**)&xq, (size_t)Qp * D.d * sizeof(float), st));
    CDE_CUDA(pool_alloc(ctx, (void**)&mq, (size_t)Q * sizeof(float), st));
    k_query_pack<<<(unsigned)((Qp + 255) / 256), 256, 0, st>>>(d_xq, Q, Qp, D.d, D.stats, xq);
    CDE_CUDA(cudaGetLastError());
    if (D.kernel == CDE_KERNEL_GAUSS) {
        const int rc = query_shift_enqueue(ctx->sm_count, D, xq, Q, Qp, mq, st);
        if (rc != CDE_OK) return rc;
    }
    *xq_out = xq;
    *mq_out = mq;
    return CDE_OK;
}

// queries per thread: more while the coordinates fit in registers
static int stats_jb(int d) { return d <= 8 ? 4 : d <= 16 ? 2 : 1; }

template <int KERN>
static void launch_stats_d(const StatArgs& a, dim3 grid, cudaStream_t st) {
    if (a.d <= 4) k_cond_stats<KERN, 4, 4><<<grid, kCSThreads, 0, st>>>(a);
    else if (a.d <= 8) k_cond_stats<KERN, 8, 4><<<grid, kCSThreads, 0, st>>>(a);
    else if (a.d <= 16) k_cond_stats<KERN, 16, 2><<<grid, kCSThreads, 0, st>>>(a);
    else k_cond_stats<KERN, 64, 1><<<grid, kCSThreads, 0, st>>>(a);
}

template <int KERN>
static void launch_chunk_weights(const SampleArgs& a, dim3 grid, int64_t cpc, cudaStream_t st) {
    if (a.d <= 4) k_chunk_weights<KERN, 4><<<grid, kCwThreads, 0, st>>>(a, cpc);
    else if (a.d <= 8) k_chunk_weights<KERN, 8><<<grid, kCwThreads, 0, st>>>(a, cpc);
    else if (a.d <= 16) k_chunk_weights<KERN, 16><<<grid, kCwThreads, 0, st>>>(a, cpc);
    else if (a.d <= 32) k_chunk_weights<KERN, 32><<<grid, kCwThreads, 0, st>>>(a, cpc);
    else k_chunk_weights<KERN, kMaxD><<<grid, kCwThreads, 0, st>>>(a, cpc);
}

static int cond_stats_enqueue(cde_ctx* ctx, const Dataset& D, double h1, double h2, const float* d_xq,
                              const float* d_yq, int64_t Q, double* d_mean, double* d_fat, cudaStream_t st) {
    timing_reset(ctx);
    const int64_t Qp = (Q + 255) / 256 * 256;
    float *xq = nullptr, *mq = nullptr, *part = nullptr;
    int rc = prep_queries(ctx, D, d_xq, Q, Qp, &xq, &mq, st);
    if (rc != CDE_OK) return rc;
    const bool epan = D.kernel == CDE_KERNEL_EPAN;
    StatArgs a{};
    a.xs = D.xs;
    a.y = D.y;
    a.xq = xq;
    a.yq = d_yq;
    a.mq = mq;
    a.N = D.N;
    a.Np = D.Np;
    a.Q = Q;
    a.Qp = Qp;
    a.d = D.d;
    const double L2E = 1.4426950408889634074;
    a.a1 = (float)(epan ? 1.0 / (h1 * h1) : L2E / (2 * h1 * h1));
    a.a2 = (float)(epan ? 1.0 / (h2 * h2) : L2E / (2 * h2 * h2));
    const int64_t per_cta = (int64_t)kCSThreads * stats_jb(D.d);
    const int64_t gx = (Q + per_cta - 1) / per_cta;
    const int64_t tiles = (D.N + kCSThreads - 1) / kCSThreads;
    int64_t ns = (8LL * ctx->sm_count + gx - 1) / gx;
    if (ns > tiles) ns = tiles;
    if (ns < 1) ns = 1;
    const int64_t tps = (tiles + ns - 1) / ns;
    ns = (tiles + tps - 1) / tps;
    a.i_per_split = tps * kCSThreads;
    CDE_CUDA(pool_alloc(ctx, (void**)&part, (size_t)ns * Q * 3 * sizeof(float), st));
    a.part = part;
    const dim3 grid((unsigned)gx, (unsigned)ns);
    timing_begin(ctx, st);
    if (epan) launch_stats_d<1>(a, grid, st);
    else launch_stats_d<0>(a, grid, st);
    timing_end(ctx, st);
    CDE_CUDA(cudaGetLastError());
    const double norm = epan ? std::exp(epan_log_norm(1)) / h2 : 1.0 / (2.5066282746310002 * h2);
    k_cond_stats_final<<<(unsigned)((Q + 15) / 16), 256, 0, st>>>(part, (int)ns, Q, norm, d_mean,
                                                                   d_yq ? d_fat : nullptr);
    CDE_CUDA(cudaGetLastError());
    cudaFreeAsync(part, st);
    cudaFreeAsync(xq, st);
    cudaFreeAsync(mq, st);
    return CDE_OK;
}

static int cond_interval_enqueue(cde_ctx* ctx, const Dataset& D, double h1, double h2, const float* d_xq,
                                 int64_t Q, int S, double alpha, uint64_t seed, float* d_lo, float* d_hi,
                                 float* d_samples, cudaStream_t st) {
    const int64_t Qp = (Q + 255) / 256 * 256;
    float *xq = nullptr, *mq = nullptr;
    int rc = prep_queries(ctx, D, d_xq, Q, Qp, &xq, &mq, st);
    if (rc != CDE_OK) return rc;
    const bool epan = D.kernel == CDE_KERNEL_EPAN;
    SampleArgs a{};
    a.xs = D.xs;
    a.y = D.y;
    a.xq = xq;
    a.mq = mq;
    a.N = D.N;
    a.Np = D.Np;
    a.Q = Q;
    a.Qp = Qp;
    a.d = D.d;
    a.S = S;
    int sp = 1;
    while (sp < S) sp <<= 1;
    a.SP = sp;
    a.m_keep = (int)std::ceil((1.0 - alpha) * S - 1e-9);
    if (a.m_keep < 1) a.m_keep = 1;
    if (a.m_keep > S) a.m_keep = S;
    const double L2E = 1.4426950408889634074;
    a.a1 = (float)(epan ? 1.0 / (h1 * h1) : L2E / (2 * h1 * h1));
    a.h2 = (float)h2;
    a.seed = seed;
    a.lo = d_lo;
    a.hi = d_hi;
    a.samples = d_samples;
    static std::atomic<uint64_t> attr0{0}, attr1{0};
    CDE_CUDA(smem_attr_once(attr0, k_cond_sample<0>, (int)sizeof(SampleSmem)));
    CDE_CUDA(smem_attr_once(attr1, k_cond_sample<1>, (int)sizeof(SampleSmem)));
    a.n_chunks = (D.N + kChunk - 1) / kChunk;
    // queries in batches whose running sums fit 128 MB (at least 128)
    const int64_t qmax = std::max<int64_t>(kCwQ, ((int64_t)32 << 20) / (a.n_chunks * kSegs) / kCwQ * kCwQ);
    const int64_t qbatch = std::min(Q, qmax);
    const bool more = a.n_chunks > kEndsMax;
    CDE_CUDA(pool_alloc(ctx, (void**)&a.ct, (size_t)(a.n_chunks * (kSegs + (more ? 1 : 0)) * qbatch) * sizeof(float), st));
    a.ends = a.ct + a.n_chunks * kSegs * qbatch;
    for (int64_t q0 = 0; q0 < Q; q0 += qbatch) {
        a.q0 = q0;
        a.nq = std::min(qbatch, Q - q0);
        const int64_t gx = (a.nq + kCwQ - 1) / kCwQ;
        // about 16 CTAs of 64 threads per SM, each a run of chunks
        const int64_t gy = std::min(a.n_chunks, std::min<int64_t>(65535, std::max<int64_t>(1, 16LL * ctx->sm_count / gx)));
        const int64_t cpc = (a.n_chunks + gy - 1) / gy;
        const dim3 cg((unsigned)gx, (unsigned)((a.n_chunks + cpc - 1) / cpc));
        if (epan) launch_chunk_weights<1>(a, cg, cpc, st);
        else launch_chunk_weights<0>(a, cg, cpc, st);
        CDE_CUDA(cudaGetLastError());
        // one CTA per query
        if (epan) k_cond_sample<1><<<(unsigned)a.nq, kSmpThreads, sizeof(SampleSmem), st>>>(a);
        else k_cond_sample<0><<<(unsigned)a.nq, kSmpThreads, sizeof(SampleSmem), st>>>(a);
        CDE_CUDA(cudaGetLastError());
    }
    cudaFreeAsync(a.ct, st);
    cudaFreeAsync(xq, st);
    cudaFreeAsync(mq, st);
    return CDE_OK;
}

#ifdef CDE_CHECKS
CDE_CHECK_READER(check_status_products)
#endif

}  // namespace cde

using namespace cde;

static int check_bw(double h1, double h2, const char* who) {
    if (!std::isfinite(h1) || !std::isfinite(h2) || h1 < 1e-12 || h2 < 1e-12 || h1 > 1e12 || h2 > 1e12)
        return set_error(CDE_EINVAL, std::string(who) + ": bandwidth must be finite in [1e-12, 1e12]");
    return CDE_OK;
}

extern "C" int cde_cond_stats(cde_ctx* ctx, cde_dataset ds, double h1, double h2, const float* xq,
                              const float* yq, int64_t Q, double* mean_out, double* fat_out, int flags,
                              void* stream) {
    CDE_NVTX("cde_cond_stats");
    if (!ctx) return set_error(CDE_EINVAL, "cde_cond_stats: null context");
    int rc = check_bw(h1, h2, "cde_cond_stats");
    if (rc != CDE_OK) return rc;
    if (Q < 0 || (Q > 0 && (!xq || (!mean_out && !fat_out) || (fat_out && !yq))))
        return set_error(CDE_EINVAL, "cde_cond_stats: bad sizes or null pointers");
    auto D = find_dataset(ctx, ds);
    if (!D) return set_error(CDE_ENOTFOUND, "cde_cond_stats: unknown dataset");
    if (Q == 0) return CDE_OK;
    std::lock_guard<std::recursive_mutex> lk(ctx->mu);
    CDE_CUDA(cudaSetDevice(ctx->device));
    cudaStream_t st = pick_stream(ctx, stream);
    const bool in_dev = flags & CDE_IN_DEVICE, out_dev = flags & CDE_OUT_DEVICE;
    const float* dq = xq;
    const float* dy = yq;
    float *dxq = nullptr, *dyq = nullptr;
    double *dmean = out_dev ? mean_out : nullptr, *dfat = out_dev ? fat_out : nullptr;
    if (!in_dev) {
        for (int64_t e = 0; e < Q * D->d; ++e)
            if (!std::isfinite(xq[e])) return set_error(CDE_EINVAL, "cde_cond_stats: non-finite query");
        CDE_CUDA(pool_alloc(ctx, (void**)&dxq, (size_t)Q * D->d * sizeof(float), st));
        CDE_CUDA(cudaMemcpyAsync(dxq, xq, (size_t)Q * D->d * sizeof(float), cudaMemcpyHostToDevice, st));
        dq = dxq;
        if (yq) {
            CDE_CUDA(pool_alloc(ctx, (void**)&dyq, (size_t)Q * sizeof(float), st));
            CDE_CUDA(cudaMemcpyAsync(dyq, yq, (size_t)Q * sizeof(float), cudaMemcpyHostToDevice, st));
            dy = dyq;
        }
    }
    if (!out_dev) {
        if (mean_out) CDE_CUDA(pool_alloc(ctx, (void**)&dmean, (size_t)Q * sizeof(double), st));
        if (fat_out) CDE_CUDA(pool_alloc(ctx, (void**)&dfat, (size_t)Q * sizeof(double), st));
    }
    HostCopies out(ctx);
    rc = cond_stats_enqueue(ctx, *D, h1, h2, dq, fat_out ? dy : nullptr, Q, dmean, dfat, st);
    cudaError_t e = cudaSuccess;
    if (rc == CDE_OK && !out_dev) {
        if (mean_out) e = out.add(mean_out, dmean, (size_t)Q * sizeof(double), st);
        if (e == cudaSuccess && fat_out) e = out.add(fat_out, dfat, (size_t)Q * sizeof(double), st);
    }
    if (dxq) cudaFreeAsync(dxq, st);
    if (dyq) cudaFreeAsync(dyq, st);
    if (!out_dev) {
        if (dmean) cudaFreeAsync(dmean, st);
        if (dfat) cudaFreeAsync(dfat, st);
        cudaError_t e2 = cudaStreamSynchronize(st);
        if (rc == CDE_OK && e == cudaSuccess && e2 != cudaSuccess) e = e2;
    }
    if (rc != CDE_OK) return rc;
    if (e != cudaSuccess) return cuda_error(e, "cde_cond_stats");
    out.finish();
    return CDE_OK;
}

extern "C" int cde_cond_interval(cde_ctx* ctx, cde_dataset ds, double h1, double h2, const float* xq,
                                 int64_t Q, int S, double alpha, uint64_t seed, float* lo_out, float* hi_out,
                                 float* samples_out, int flags, void* stream) {
    CDE_NVTX("cde_cond_interval");
    if (!ctx) return set_error(CDE_EINVAL, "cde_cond_interval: null context");
    int rc = check_bw(h1, h2, "cde_cond_interval");
    if (rc != CDE_OK) return rc;
    if (Q < 0 || S < 1 || S > kSmpMax || !(alpha > 0.0 && alpha < 1.0) ||
        (Q > 0 && (!xq || !lo_out || !hi_out)))
        return set_error(CDE_EINVAL, "cde_cond_interval: need 1 <= S <= 4096, 0 < alpha < 1, non-null pointers");
    auto D = find_dataset(ctx, ds);
    if (!D) return set_error(CDE_ENOTFOUND, "cde_cond_interval: unknown dataset");
    if (Q == 0) return CDE_OK;
    std::lock_guard<std::recursive_mutex> lk(ctx->mu);
    CDE_CUDA(cudaSetDevice(ctx->device));
    cudaStream_t st = pick_stream(ctx, stream);
    const bool in_dev = flags & CDE_IN_DEVICE, out_dev = flags & CDE_OUT_DEVICE;
    const float* dq = xq;
    float* dxq = nullptr;
    float *dlo = out_dev ? lo_out : nullptr, *dhi = out_dev ? hi_out : nullptr;
    float* dsm = out_dev ? samples_out : nullptr;
    if (!in_dev) {
        for (int64_t e = 0; e < Q * D->d; ++e)
            if (!std::isfinite(xq[e])) return set_error(CDE_EINVAL, "cde_cond_interval: non-finite query");
        CDE_CUDA(pool_alloc(ctx, (void**)&dxq, (size_t)Q * D->d * sizeof(float), st));
        CDE_CUDA(cudaMemcpyAsync(dxq, xq, (size_t)Q * D->d * sizeof(float), cudaMemcpyHostToDevice, st));
        dq = dxq;
    }
    if (!out_dev) {
        CDE_CUDA(pool_alloc(ctx, (void**)&dlo, (size_t)Q * sizeof(float), st));
        CDE_CUDA(pool_alloc(ctx, (void**)&dhi, (size_t)Q * sizeof(float), st));
        if (samples_out) CDE_CUDA(pool_alloc(ctx, (void**)&dsm, (size_t)Q * S * sizeof(float), st));
    }
    HostCopies out(ctx);
    rc = cond_interval_enqueue(ctx, *D, h1, h2, dq, Q, S, alpha, seed, dlo, dhi, dsm, st);
    cudaError_t e = cudaSuccess;
    if (rc == CDE_OK && !out_dev) {
        e = out.add(lo_out, dlo, (size_t)Q * sizeof(float), st);
        if (e == cudaSuccess) e = out.add(hi_out, dhi, (size_t)Q * sizeof(float), st);
        if (e == cudaSuccess && samples_out) e = out.add(samples_out, dsm, (size_t)Q * S * sizeof(float), st);
    }
    if (dxq) cudaFreeAsync(dxq, st);
    if (!out_dev) {
        cudaFreeAsync(dlo, st);
        cudaFreeAsync(dhi, st);
        if (dsm) cudaFreeAsync(dsm, st);
        cudaError_t e2 = cudaStreamSynchronize(st);
        if (rc == CDE_OK && e == cudaSuccess && e2 != cudaSuccess) e = e2;
    }
    if (rc != CDE_OK) return rc;
    if (e != cudaSuccess) return cuda_error(e, "cde_cond_interval");
    out.finish();
    return CDE_OK;
}
