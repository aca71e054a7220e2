// dar_project.cuh -- rows of 64 values times a 64 x DD fp32 matrix on the CUDA
// cores, each output ONE fp32 fused-multiply-add chain over t = 0..63 starting
// from +0.0f (Eq. 1).
#pragma once

#include "dar_common.cuh"
#include "dar_sm100.cuh"

namespace dar {

// A CTA stages kStageBytesBulk of rows in shared memory, 16-byte chunk c of row
// r at chunk c ^ (r & 7), so that a warp reading one chunk of 32 different rows
// touches every bank group once.  A thread holds 16 to 64 sums: one 16-byte read of
// W[t][c..c+3] (the same address in the whole warp) feeds a product for each of its
// rows, and fewer sums per thread put more warps on an SM while tiles arrive.
// Measured, columns x rows per thread, 32 prompts of 1000 to 4096 tokens, 12 heads,
// appended, us: d_down 8 8x4 97, 8x2 81, 8x1 86; 16 16x4 141, 16x2 117, 8x4 118,
// 8x2 127; 32 32x2 201, 16x4 215, 16x2 208; 64 16x4 494, 16x2 488 (but 230 instead
// of 195 for the bulk projection of 1 M rows), 32x2 503.
constexpr int kStageBytesBulk = 32 << 10;

template <typename T>
__host__ __device__ constexpr int rows_bulk()
{
    return kStageBytesBulk / (kHeadDim * (int)sizeof(T));
}
template <int DD>
__host__ __device__ constexpr int cols_per_thread()
{
    return DD < 16 || DD == 32 ? DD : 16;
}
template <int DD>
__host__ __device__ constexpr int rows_per_thread()
{
    return DD == 64 ? 4 : 2;
}
// Threads that share out the columns of a row.
template <int DD>
__host__ __device__ constexpr int slices()
{
    return DD / cols_per_thread<DD>();
}

// Start the copies of rows [0, nr) (contiguous in memory) into the tile.
template <typename T>
__device__ __forceinline__ void stage_tile(unsigned char *rows, const T *x, int nr, int tid, int threads)
{
    constexpr int CPR = kHeadDim * (int)sizeof(T) / 16;
    const uint32_t s = sm100::smem_u32(rows);
    const uint4 *src = reinterpret_cast<const uint4 *>(x);
    for (int i = tid; i < nr * CPR; i += threads) {
        const int r = i / CPR, c = i % CPR;
        sm100::cp_async16(s + (r * CPR + (c ^ (r & 7))) * 16, src + i);
    }
}

// The chains of rows r0 + k * rstep (k < RPT) over the CW columns at Ws (row
// stride DD floats).
template <typename T, int DD, int CW, int RPT>
__device__ __forceinline__ void project_rows(const unsigned char *rows, const float *Ws, int r0, int rstep,
                                             float (&acc)[RPT][CW])
{
    constexpr int E = Granule<T>::kElems;
    constexpr int CPR = kHeadDim / E;  // 16-byte chunks per row (8 for bf16, 16 for fp32)
#pragma unroll
    for (int k = 0; k < RPT; ++k)
#pragma unroll
        for (int c = 0; c < CW; ++c)
            acc[k][c] = 0.0f;
#pragma unroll 1
    for (int q = 0; q < CPR; ++q) {
        float xf[RPT][E];
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
            const int r = r0 + k * rstep;
            unpack(reinterpret_cast<const uint4 *>(rows)[r * CPR + (q ^ (r & 7))], xf[k], T());
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int t = q * E + e;
#pragma unroll
            for (int c = 0; c < CW; c += 4) {
                const float4 w4 = *reinterpret_cast<const float4 *>(Ws + t * DD + c);
#pragma unroll
                for (int k = 0; k < RPT; ++k) {
                    sm100::ffma2(acc[k][c], acc[k][c + 1], xf[k][e], xf[k][e], w4.x, w4.y, acc[k][c], acc[k][c + 1]);
                    sm100::ffma2(acc[k][c + 2], acc[k][c + 3], xf[k][e], xf[k][e], w4.z, w4.w, acc[k][c + 2],
                                 acc[k][c + 3]);
                }
            }
        }
    }
}

// CW fp32 values rounded once to T and stored as 16-byte words (o is 16-byte aligned).
template <typename T, int CW>
__device__ __forceinline__ void store_row(T *o, const float (&x)[CW])
{
    constexpr int OE = 16 / sizeof(T);
    static_assert(CW % OE == 0, "whole 16-byte words");
#pragma unroll
    for (int c = 0; c < CW; c += OE) {
        uint32_t u[4];
        if constexpr (sizeof(T) == 2) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                u[i] = sm100::cvt_bf16x2(x[c + 2 * i], x[c + 2 * i + 1]);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                u[i] = __float_as_uint(x[c + i]);
        }
        *reinterpret_cast<uint4 *>(o + c) = make_uint4(u[0], u[1], u[2], u[3]);
    }
}

}  // namespace dar
