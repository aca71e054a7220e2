// dar_project_tc.cuh -- rows of 64 bf16 values times a 64 x C fp32 matrix on the
// tensor cores (mma.sync m16n8k16), for results that need fp32 accuracy but not
// the one chain of Eq. 1's vectors: the backward's q~ and dO~.
//
// The matrix enters as the sum of three bf16 terms: its top 8 significant bits,
// the next 8 and the last 8, so the split is exact and a product x w is off by no
// more than its fp32 rounding.  A warp holds the terms of 32 columns at most in
// registers as B fragments and streams 16 rows at a time straight from memory:
// the contraction index may run in any order, so a lane's k indices are chosen
// such that two 16-byte loads per row bring its A fragments, and the columns such
// that its results are consecutive.  Memory bounds it (figures at bwd_rows_tc_kernel).
#pragma once

#include "dar_common.cuh"
#include "dar_launch.h"
#include "dar_project.cuh"
#include "dar_sm100.cuh"

namespace dar {

// w as three bf16 terms (high halves of the words); infinities and NaN stay in the first.
__device__ __forceinline__ void split3(float w, uint32_t (&t)[3])
{
    const bool fin = fabsf(w) < INFINITY;
    t[0] = __float_as_uint(fin ? w : w != w ? __uint_as_float(0x7fc00000u) : w) & 0xffff0000u;
    const float r1 = fin ? w - __uint_as_float(t[0]) : 0.f;
    t[1] = __float_as_uint(r1) & 0xffff0000u;
    t[2] = __float_as_uint(r1 - __uint_as_float(t[1]));
}

// NT n-tiles of 8 columns: column slot j of n-tile n is column (j / 2) 2 NT + 2 n + j % 2.
template <int NT>
struct ProjectTc {
    static constexpr int COLS = 8 * NT;
    uint32_t b[3][4][NT][2];

    // w(t, c): the matrix, c relative to this warp's first column
    template <typename F>
    __device__ __forceinline__ void load(int lane, F &&w)
    {
        const int grp = lane >> 2, tig = lane & 3;
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int t = 8 * (tig + 4 * (s >> 1)) + 4 * (s & 1) + 2 * e;
                    const int c = grp / 2 * (2 * NT) + 2 * n + (grp & 1);
                    uint32_t lo[3], hi[3];
                    split3(w(t, c), lo);
                    split3(w(t + 1, c), hi);
#pragma unroll
                    for (int k = 0; k < 3; ++k)
                        b[k][s][n][e] = lo[k] >> 16 | (hi[k] & 0xffff0000u);
                }
    }

    // y[hr][2 n + j] = columns tig 2 NT + 2 n + j of row grp + 8 hr, x[hr][i] = chunk tig + 4 i of that row
    __device__ __forceinline__ void products(const uint4 (&x)[2][2], float (&y)[2][2 * NT]) const
    {
        float acc[NT][4];
#pragma unroll
        for (int n = 0; n < NT; ++n)
            acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
#pragma unroll
        for (int k = 2; k >= 0; --k)  // small terms first
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const uint4 &u = x[0][s >> 1], &v = x[1][s >> 1];
                const uint32_t a[4] = {s & 1 ? u.z : u.x, s & 1 ? v.z : v.x, s & 1 ? u.w : u.y, s & 1 ? v.w : v.y};
#pragma unroll
                for (int n = 0; n < NT; ++n)
                    sm100::mma_bf16_acc(acc[n], a, b[k][s][n][0], b[k][s][n][1]);
            }
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                y[e >> 1][2 * n + (e & 1)] = acc[n][e];
    }
};

// Whether some bf16 of these words is an infinity or NaN (exponent bits all ones).
__device__ __forceinline__ uint32_t nonfinite(const uint4 &v)
{
    auto one = [](uint32_t u) { return (u & 0x7f807f80u) + 0x00800080u; };
    return (one(v.x) | one(v.y) | one(v.z) | one(v.w)) & 0x80008000u;
}

// W consecutive bf16 (W even; o aligned to min(2 W, 16) bytes).
template <int W>
__device__ __forceinline__ void store_cols(bf16 *o, const float (&y)[W])
{
    uint32_t u[W / 2];
#pragma unroll
    for (int i = 0; i < W / 2; ++i)
        u[i] = sm100::cvt_bf16x2(y[2 * i], y[2 * i + 1]);
    if constexpr (W == 2)
        *reinterpret_cast<uint32_t *>(o) = u[0];
    else if constexpr (W == 4)
        *reinterpret_cast<uint2 *>(o) = make_uint2(u[0], u[1]);
    else
        *reinterpret_cast<uint4 *>(o) = make_uint4(u[0], u[1], u[2], u[3]);
}

constexpr int kTcWarps = 4;

// Rows [r0, r1) of x (a warp's share) times the columns of `p`, into out (row
// stride ostride): 16 rows at a time, the next ones loaded meanwhile.  Rows with
// an infinity or NaN would meet it in every term of the split (infinity times a
// zero or negative rest), so 16 rows that hold one take fp32 chains over w(t, c).
// each(x, r): what else the caller does with 16 rows (x as in products(), rows r + grp, + 8).
template <int NT, typename F, typename G>
__device__ __forceinline__ void project_rows_tc(const bf16 *x, bf16 *out, int ostride, int r0, int r1,
                                                const ProjectTc<NT> &p, int lane, F &&w, G &&each)
{
    const int grp = lane >> 2, tig = lane & 3;
    auto fetch = [&](uint4(&v)[2][2], int r) {
#pragma unroll
        for (int hr = 0; hr < 2; ++hr)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int row = r + grp + 8 * hr;
                v[hr][i] = row < r1 ? __ldg(reinterpret_cast<const uint4 *>(x + (size_t)row * kHeadDim) + tig + 4 * i)
                                    : make_uint4(0u, 0u, 0u, 0u);
            }
    };
    uint4 next[2][2];
    fetch(next, r0);
    for (int r = r0; r < r1; r += 16) {
        uint4 v[2][2];
#pragma unroll
        for (int hr = 0; hr < 2; ++hr)
#pragma unroll
            for (int i = 0; i < 2; ++i)
                v[hr][i] = next[hr][i];
        if (r + 16 < r1)
            fetch(next, r + 16);
        each(v, r);
        const uint32_t bad = nonfinite(v[0][0]) | nonfinite(v[0][1]) | nonfinite(v[1][0]) | nonfinite(v[1][1]);
        if (__builtin_expect(__any_sync(0xffffffffu, bad != 0u), 0)) {
            const int n = min(16, r1 - r) * ProjectTc<NT>::COLS;
            for (int o = lane; o < n; o += 32) {
                const int row = r + o / ProjectTc<NT>::COLS, c = o % ProjectTc<NT>::COLS;
                float acc = 0.f;
                for (int t = 0; t < kHeadDim; ++t)
                    acc = fmaf(__bfloat162float(x[(size_t)row * kHeadDim + t]), w(t, c), acc);
                out[(size_t)row * ostride + c] = __float2bfloat16_rn(acc);
            }
            continue;
        }
        float y[2][2 * NT];
        p.products(v, y);
#pragma unroll
        for (int hr = 0; hr < 2; ++hr)
            if (r + grp + 8 * hr < r1)
                store_cols<2 * NT>(out + (size_t)(r + grp + 8 * hr) * ostride + tig * 2 * NT, y[hr]);
    }
}

// Rows per CTA: enough that the split of the matrix is paid once for many rows, as
// long as the chip is filled a few times over.
__host__ inline int project_tc_rows(long long rows_per_head, long long heads)
{
    int r = 16 * kTcWarps * 16;
    while (r > 16 * kTcWarps && (rows_per_head + r - 1) / r * heads < kSms * 8)
        r /= 2;
    return r;
}

}  // namespace dar
