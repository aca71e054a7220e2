// dar_prep.cuh -- the query-side set-up of a decode call, as blocks of a kernel of
// its own or of the step's first kernel.
#pragma once

#include "dar_common.cuh"
#include "dar_launch.h"

namespace dar {

// q~ = q Uk^T for every (b, h) row, one row per warp (fp32, four partial sums
// over t mod 4), and zeroed group counters.  In the direct variant of Sec. 5
// (a.qd set) q~ is the row's own d_down query times scale_down / scale, so the
// stream kernel's global scores scale * q~ . k^D are scale_down * q^D . k^D.
// Reads q and Uk only.  `block` of `blocks` blocks of THREADS threads.
template <typename T, int DD, int THREADS>
__device__ __forceinline__ void prep_rows(const DecodeArgs &a, int block, int blocks)
{
    constexpr int QR = DD > 32 ? 2 : 1;  // q~ entries per lane
    constexpr int warps = THREADS / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rows = a.B * a.Hq;
    for (int row = warp * blocks + block; row < rows; row += blocks * warps) {  // few rows: spread over the blocks
        if (a.qd) {  // direct variant: the row's own d_down query, rescaled to the local scale
            for (int c = lane; c < DD; c += 32)
                a.qt[(size_t)row * DD + c] = to_f32(static_cast<const T *>(a.qd)[(size_t)row * DD + c]) * a.qd_ratio;
            continue;
        }
        const T *qrow = static_cast<const T *>(a.q) + (size_t)row * kHeadDim;
        const float q0 = to_f32(qrow[lane]), q1 = to_f32(qrow[lane + 32]);
        const int g = (row % a.Hq) / a.G;
#pragma unroll
        for (int rr = 0; rr < QR; ++rr) {
            const int c = lane + 32 * rr;
            const float4 *u4 = reinterpret_cast<const float4 *>(a.Uk + ((size_t)g * DD + (c < DD ? c : 0)) * kHeadDim);
            float4 uk[kHeadDim / 4];
#pragma unroll
            for (int t4 = 0; t4 < kHeadDim / 4; ++t4)
                uk[t4] = c < DD ? __ldg(u4 + t4) : make_float4(0.f, 0.f, 0.f, 0.f);
            float p[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int t4 = 0; t4 < kHeadDim / 4; ++t4) {
                const float uu[4] = {uk[t4].x, uk[t4].y, uk[t4].z, uk[t4].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int t = 4 * t4 + e;
                    const float qv = __shfl_sync(0xffffffffu, t < 32 ? q0 : q1, t & 31);
                    p[e] = fmaf(qv, uu[e], p[e]);
                }
            }
            if (c < DD)
                a.qt[(size_t)row * DD + c] = (p[0] + p[1]) + (p[2] + p[3]);
        }
    }
    const int ngroups = a.B * a.Hkv * a.HS;  // group counters, then the pool's claim counter
    for (int i = block * THREADS + (int)threadIdx.x; i <= ngroups; i += blocks * THREADS)
        a.counters[i] = 0;
}

}  // namespace dar
