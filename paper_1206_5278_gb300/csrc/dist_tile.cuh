// Register-tiled squared distances between 128 rows and tiles of 64 points, for
// the nearest-distance kernels (dataset shifts, loo_grid.cu; query shifts,
// density.cu) at d_x > 8.
//
// A CTA of 256 threads holds its rows' coordinates in shared memory for the
// whole kernel and streams the points in two cp.async buffers; a thread forms 8
// rows x 4 points (rows in packed FP32x2 pairs): per dimension three 128-bit
// shared loads feed 32 packed instructions, so the FMA pipe is the limit (2 d
// lane operations per pair) and not the coordinate loads.  Each distance is
// accumulated dimension 0 first, one fused multiply-add per dimension on the
// rounded difference: bitwise every other pair kernel's value.
//
// Measured, dataset shifts: N = 24,007, d = 12: 5.5 -> 0.71 ms; N = 100,003, d = 32:
// 129 -> 23 ms (before: one row per thread, coordinates past the eighth re-read from
// global memory for every pair, one CTA per 256 rows).  At N = 50,000 a dimension costs
// 0.0167 clocks per pair and SM (0.0156: the FMA pipe), the two running keys 0.18 (the
// ALU pipe).  At d <= 8 the split kernel with its rows in registers is as fast or faster
// (dataset creation at N = 50,000: d = 4 1.86 against 2.29 ms, d = 8 2.33 against 2.87;
// query shifts within 3%), so it stays there.
#pragma once

#include <cstdint>

#include "cde_internal.h"
#include "tc_util.cuh"

namespace cde {

constexpr int kDtRows = 128, kDtPts = 64, kDtThreads = 256;

// shared memory in floats: rows [d][128], then two point buffers [d + with_y][64]
__host__ __device__ inline int dt_smem_floats(int d, bool with_y) {
    return d * kDtRows + 2 * (d + (with_y ? 1 : 0)) * kDtPts;
}

// start copying point tile i0 .. i0 + 63 (i0 a multiple of 64, inside the padded length)
__device__ __forceinline__ void dt_fetch(const float* __restrict__ xs, const float* __restrict__ y, int64_t Np, int d,
                                         int64_t i0, float* buf) {
    const int n = (d + (y ? 1 : 0)) * (kDtPts / 4);
    for (int e = threadIdx.x; e < n; e += kDtThreads) {
        const int c = e / (kDtPts / 4), p = 4 * (e % (kDtPts / 4));
        const float* src = (c < d ? xs + (int64_t)c * Np : y) + CDE_CK(i0 + p, Np - 3, 141);
        cp_async16(smem_u32(buf + c * kDtPts + p), src);
    }
    cp_async_commit();
}

// acc[q][e]: squared distances of the thread's row pair q (rows 8 rg + 2q, + 1) to its
// point e (4 pg + e)
__device__ __forceinline__ void dt_distances(const float* rows, const float* pts, int d, int rg, int pg,
                                             float2 (&acc)[4][4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[q][e] = make_float2(0.f, 0.f);
    const float* rp = rows + 8 * rg;
    const float* pp = pts + 4 * pg;
#pragma unroll 2
    for (int c = 0; c < d; ++c) {
        const float4 ra = *reinterpret_cast<const float4*>(rp + c * kDtRows);
        const float4 rb = *reinterpret_cast<const float4*>(rp + c * kDtRows + 4);
        const float4 p4 = *reinterpret_cast<const float4*>(pp + c * kDtPts);
        const float2 r[4] = {make_float2(ra.x, ra.y), make_float2(ra.z, ra.w), make_float2(rb.x, rb.y),
                             make_float2(rb.z, rb.w)};
        const float p[4] = {-p4.x, -p4.y, -p4.z, -p4.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 t = __fadd2_rn(r[q], make_float2(p[e], p[e]));
                acc[q][e] = __ffma2_rn(t, t, acc[q][e]);
            }
    }
}

// point splits of a kernel with row blocks of 128: about four waves of two CTAs per SM,
// at least four tiles each; returns points per split (a multiple of 64)
inline int64_t dt_points_per_split(int64_t row_blocks, int64_t N, int sm_count, int64_t* splits) {
    const int64_t tiles = (N + kDtPts - 1) / kDtPts;
    int64_t ns = (8LL * sm_count + row_blocks - 1) / row_blocks;
    if (ns > (tiles + 3) / 4) ns = (tiles + 3) / 4;
    if (ns < 1) ns = 1;
    const int64_t tps = (tiles + ns - 1) / ns;
    *splits = (tiles + tps - 1) / tps;
    return tps * kDtPts;
}

}  // namespace cde
