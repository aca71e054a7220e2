// dar_backward_tc.cu -- the backward pass for bf16 storage on the tensor
// cores (mma.sync m16n8k16: bf16 operands, fp32 accumulators).
//
// The gradients of dar_backward.cuh as FlashAttention-style recomputation with
// the local (full-width) and the global (d_down-wide) pairs in kernels of
// their own, so that each holds only its own accumulators and operands:
//  - rows: q~ = q Uk^T, dO~ = dO Uv^T (bf16) and -D = -dO . o.
//  - dq, per tile of query rows, ONE pass over the keys.  D does not depend on
//    the softmax, so every sum is linear in the weights and can be taken with
//    the running maximum m of an online softmax instead of the log-sum-exp:
//      dS' = 2^(s c2 - m) (dP - D),  dq' += dS' K,  l += 2^(s c2 - m),
//    and the row is divided by l at its end.  The global kernel leaves its
//    unnormalised dq~ and O^D with (m, l); the local kernel, run after it,
//    merges both parts into the row's log-sum-exp, lifts dq~ and writes dq and
//    the factor that normalises the global part's sums.
//  - dk/dv, per tile of keys over the query heads of the group and the query
//    rows that see them, from the log-sum-exp:
//      dv += P dO, dk += dS Q (local) | dv^D += P dO~, dk^D += dS q~ (global);
//    the local kernel, run after the global one, lifts dk^D and dv^D into its
//    own dk and dv.
// Both kinds of kernel hold the scores of a 16-key (16-query) step in registers
// and turn them into A operands of the next products.  -D enters as the
// accumulator input of dP, so dP - D costs no instruction; scores, weights and
// sums advance two per instruction (f32x2).  A warp takes 32 rows where the
// accumulators allow it, so an operand read from shared memory feeds two
// products: with 16 rows the reads alone would take longer than the products.
// Tiles arrive by 16-byte cp.async copies in padded rows (stride a multiple of
// 16 bytes plus 16: the eight rows of an ldmatrix fall in distinct banks),
// three stages deep.
#include "dar_backward.cuh"
#include "dar_project_tc.cuh"
#include "dar_sm100.cuh"

namespace dar {
namespace bwd {

using sm100::add2;
using sm100::cp_async_commit;
using sm100::cp_async_wait;
using sm100::cvt_bf16x2;
using sm100::ex2_approx;
using sm100::ffma2;
using sm100::ldsm_x4;
using sm100::ldsm_x4_t;
using sm100::mma_bf16_acc;
using sm100::mma_bf16_c;
using sm100::mul2;
using sm100::smem_u32;

constexpr int kTc = 128;  // threads: four warps
constexpr float kRaise = 8.0f;  // log2 units: a weight stays below 2^8 between raises of a running maximum

// 16-byte copy, or 16 zero bytes when !valid (src must still be an address in the tensor).
__device__ __forceinline__ void cp16z(uint32_t dst, const void *src, bool valid)
{
    const int n = valid ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}

// Bytes per padded row of a W-wide bf16 tile.
template <int W>
__host__ __device__ constexpr int ld_of()
{
    return W * 2 + 16;
}

// Rows [0, n) of a row-major [*][W] bf16 matrix into a padded tile of ROWS rows; the others are zero.
template <int W, int ROWS>
__device__ __forceinline__ void stage_rows(uint32_t dst, const bf16 *src, int n, int tid)
{
    constexpr int CH = W / 8;
    static_assert(ROWS * CH % kTc == 0, "every thread copies the same number of chunks");
#pragma unroll
    for (int e = 0; e < ROWS * CH / kTc; ++e) {
        const int i = tid + e * kTc, r = i / CH, c = i % CH;
        const bool ok = r < n;
        cp16z(dst + r * ld_of<W>() + c * 16, src + (ok ? (size_t)r * W + c * 8 : 0), ok);
    }
}

// A fragment of a 16 x 16 k-step from two 16 x 8 accumulator fragments.
__device__ __forceinline__ void frag_a(uint32_t (&a)[4], const float (&c0)[4], const float (&c1)[4])
{
    a[0] = cvt_bf16x2(c0[0], c0[1]);
    a[1] = cvt_bf16x2(c0[2], c0[3]);
    a[2] = cvt_bf16x2(c1[0], c1[1]);
    a[3] = cvt_bf16x2(c1[2], c1[3]);
}

// Lane offset for ldmatrix (non-transposed, B operand of two n-tiles): 16 rows
// of a tile with row stride LD, first 16 columns.
template <int LD>
__device__ __forceinline__ uint32_t b_lane(int lane)
{
    return ((lane & 7) + ((lane >> 4) << 3)) * LD + ((lane >> 3) & 1) * 16;
}
// Lane offset for ldmatrix.trans (B operand [k][n] of two n-tiles): 16 rows k, first 16 columns n.
template <int LD>
__device__ __forceinline__ uint32_t bt_lane(int lane)
{
    return ((lane & 7) + (((lane >> 3) & 1) << 3)) * LD + (lane >> 4) * 16;
}

// Lane offset for ldmatrix of an A operand: 16 rows, first 16 columns.
template <int LD>
__device__ __forceinline__ uint32_t a_lane(int lane)
{
    return (lane & 15) * LD + (lane >> 4) * 16;
}
// A fragments of 16 rows of a padded W-wide tile.
template <int W>
__device__ __forceinline__ void load_a(uint32_t (&f)[W / 16][4], uint32_t rows, int lane)
{
#pragma unroll
    for (int kk = 0; kk < W / 16; ++kk)
        ldsm_x4(rows + a_lane<ld_of<W>()>(lane) + kk * 32, f[kk]);
}

// C (+)= A B^T over W columns: A fragments of MT row tiles, B the 16 rows whose
// ldmatrix lane address is `b`; c0 holds the accumulator input of each tile.
template <int W, int MT>
__device__ __forceinline__ void scores(float (&s)[MT][2][4], const uint32_t (&a)[MT][W / 16][4], uint32_t b,
                                       const float (&c0)[MT][2][4])
{
#pragma unroll
    for (int kk = 0; kk < W / 16; ++kk) {
        uint32_t f[4];
        ldsm_x4(b + kk * 32, f);
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            if (kk == 0) {
                mma_bf16_c(s[mt][0], a[mt][kk], f[0], f[1], c0[mt][0]);
                mma_bf16_c(s[mt][1], a[mt][kk], f[2], f[3], c0[mt][1]);
            } else {
                mma_bf16_acc(s[mt][0], a[mt][kk], f[0], f[1]);
                mma_bf16_acc(s[mt][1], a[mt][kk], f[2], f[3]);
            }
        }
    }
}

// acc += A B over 16 rows: B [16 rows][W] read transposed at lane address `b`.
template <int W, int MT>
__device__ __forceinline__ void accumulate(float (&acc)[MT][W / 8][4], const uint32_t (&a)[MT][4], uint32_t b)
{
#pragma unroll
    for (int n = 0; n < W / 8; n += 2) {
        uint32_t f[4];
        ldsm_x4_t(b + n * 16, f);
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            mma_bf16_acc(acc[mt][n], a[mt], f[0], f[1]);
            mma_bf16_acc(acc[mt][n + 1], a[mt], f[2], f[3]);
        }
    }
}

// o[r][n] (columns 8n + 2 tig, + 1 of two rows) += sum_c x_r[c] M[c][t], fp32:
// M in shared memory with row stride LS floats.
template <int DD, int LS>
__device__ __forceinline__ void lift_rows(float (&o)[2][8][2], const float *x0, const float *x1, const float *M, int tig)
{
#pragma unroll 2
    for (int c = 0; c < DD; ++c) {
        const float a0 = x0[c], a1 = x1[c];
#pragma unroll
        for (int n = 0; n < 8; ++n) {
            const float2 m = *reinterpret_cast<const float2 *>(M + c * LS + 8 * n + 2 * tig);
            ffma2(o[0][n][0], o[0][n][1], a0, a0, m.x, m.y, o[0][n][0], o[0][n][1]);
            ffma2(o[1][n][0], o[1][n][1], a1, a1, m.x, m.y, o[1][n][0], o[1][n][1]);
        }
    }
}
constexpr int kLiftLd = 66;  // row stride of a transposed W_down: its column-wise stores fall in distinct banks

template <int V>
struct Int {
    static constexpr int value = V;
};

// Row tiles per warp and rows of the streamed tile per stage.
template <int W, bool LOCAL>
struct Shape {
    static constexpr int MT = !LOCAL && W <= 32 ? 2 : 1;
    static constexpr int ROWS = 64 * MT;                   // rows of a CTA's tile
    static constexpr int BK = !LOCAL && W <= 32 ? 128 : 64;  // streamed rows per stage
    static constexpr int NS = 3;
    static constexpr int MINB = LOCAL ? 3 : 2;
    // 16-key blocks a dq step takes, 16-query steps in flight of dk/dv.  The
    // 16-wide global kernels do best with few warps and long independent runs
    // (B8 H16 N8192 w512, us, dq / dk, dv: 1431 / 1345 at 4, 8 and two CTAs per
    // SM; 1461 / 1349 at 2, 2 and four; 1536 / 1378 at 1, 1 and four; at B8 H8
    // N2047 w128 59 / 51, 69 / 57 and 65 / 58).  Wider ones gain little from more
    // (forward and backward of the larger shape, ms, d_down 32 and 64: 9.12 and 16.5
    // at 1, 1; 8.85 and 15.9 at 2, 2; 8.82 and 15.8 at 2, 8; 8.78 and 15.6 at 4, 4)
    static constexpr int KSQ = W == 16 ? 4 : 2, UNKV = W == 16 ? 8 : 2;
    // a stage also takes the CTA's own rows, whose A fragments are read before it is needed
    static_assert(ROWS <= BK, "the CTA's tile fits in a stage");
};

// ---------------------------------------------------------------- dq

template <int W, bool LOCAL, int DD>
struct DqSmem {
    using Sh = Shape<W, LOCAL>;
    static constexpr uint32_t V = Sh::BK * ld_of<W>(), STAGE = 2 * V;
    static constexpr uint32_t TOTAL = Sh::NS * STAGE;
    // the epilogue's lift: [64][DD + 1] dq~ rows and Uk
    static_assert(!LOCAL || 64 * (DD + 1) * 4 + DD * 64 * 4 <= TOTAL, "the lift fits in the stage area");
};

template <int W, bool LOCAL, int DD>
__global__ void __launch_bounds__(kTc, Shape<W, LOCAL>::MINB) bwd_dq_tc_kernel(Args a)
{
    using Sh = Shape<W, LOCAL>;
    using Sm = DqSmem<W, LOCAL, DD>;
    constexpr int MT = Sh::MT, ROWS = Sh::ROWS, BK = Sh::BK, NS = Sh::NS, LD = ld_of<W>(), NT = W / 8;
    extern __shared__ __align__(128) unsigned char tsm[];
    const uint32_t sb = smem_u32(tsm);
    const int N = a.N, w = min(a.w, N);  // (a window past the sequence's length makes every pair local too)
    const int heads = a.B * a.Hq, bh = blockIdx.x % heads, b = bh / a.Hq, h = bh % a.Hq, g = h / a.G;
    const int i0 = ((int)(gridDim.x / heads) - 1 - (int)(blockIdx.x / heads)) * ROWS;  // longest rows first
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, grp = lane >> 2, tig = lane & 3;
    const size_t headrow = (size_t)bh * N;
    const size_t kvbase = ((size_t)b * a.Hkv + g) * N;
    const bf16 *kp = static_cast<const bf16 *>(LOCAL ? a.k : a.kd) + kvbase * W;
    const bf16 *vp = static_cast<const bf16 *>(LOCAL ? a.v : a.vd) + kvbase * W;
    const int i_last = min(N, i0 + ROWS) - 1;
    // keys [jlo, jhi): local i - w < j <= i, global j <= i - w
    const int jlo = LOCAL ? max(0, i0 - w + 1) / 16 * 16 : 0;
    const int jhi = LOCAL ? (w > 0 ? i_last + 1 : jlo) : max(0, i_last - w + 1);
    const int ntiles = (jhi - jlo + BK - 1) / BK;
    auto stage = [&](int t) {
        if (t < ntiles) {
            const int j = jlo + t * BK;
            const uint32_t dst = sb + (t % NS) * Sm::STAGE;
            stage_rows<W, BK>(dst, kp + (size_t)j * W, N - j, tid);
            stage_rows<W, BK>(dst + Sm::V, vp + (size_t)j * W, N - j, tid);
        }
        cp_async_commit();
    };
    // this CTA's rows into the last stage, then the first tiles
    stage_rows<W, ROWS>(sb + (NS - 1) * Sm::STAGE,
                        (LOCAL ? static_cast<const bf16 *>(a.q) : a.qtb) + (headrow + i0) * W, N - i0, tid);
    stage_rows<W, ROWS>(sb + (NS - 1) * Sm::STAGE + Sm::V,
                        (LOCAL ? static_cast<const bf16 *>(a.dout) : a.dotb) + (headrow + i0) * W, N - i0, tid);
    cp_async_commit();
    for (int t = 0; t < NS - 1; ++t)
        stage(t);

    const int r0 = i0 + 16 * MT * warp;  // this warp's rows r0 .. r0 + 16 MT - 1
    uint32_t qa[MT][W / 16][4], da[MT][W / 16][4];
    float nD[MT][2][4], zero[MT][2][4];
    float m[MT][2], l[MT][2][2], drow[MT][2];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int hr = 0; hr < 2; ++hr) {
            const int i = r0 + 16 * mt + grp + 8 * hr;
            drow[mt][hr] = i < N ? a.drow[headrow + i] : 0.f;
        }
    cp_async_wait<NS - 1>();
    __syncthreads();
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
        const uint32_t own = sb + (NS - 1) * Sm::STAGE + 16 * (MT * warp + mt) * LD;
        load_a<W>(qa[mt], own, lane);
        load_a<W>(da[mt], own + Sm::V, lane);
#pragma unroll
        for (int hr = 0; hr < 2; ++hr) {
            const float d = drow[mt][hr];
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
                nD[mt][nt][2 * hr] = nD[mt][nt][2 * hr + 1] = d;
                zero[mt][nt][2 * hr] = zero[mt][nt][2 * hr + 1] = 0.f;
            }
            m[mt][hr] = -INFINITY;
            l[mt][hr][0] = l[mt][hr][1] = 0.f;
        }
    }
    // dq~ and O^D (global), dq (local)
    float dq[MT][NT][4], od[LOCAL ? 1 : MT][LOCAL ? 1 : NT][4];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                dq[mt][n][e] = 0.f;
                if constexpr (!LOCAL)
                    od[mt][n][e] = 0.f;
            }
    const float c2 = a.c2;
    bool fresh = true;  // some row of the warp may still have m = -infinity

    // raise the running maxima to those of these scores
    auto raise = [&](const float (&s)[MT][2][4]) {
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int hr = 0; hr < 2; ++hr) {
                float x = fmaxf(fmaxf(s[mt][0][2 * hr], s[mt][0][2 * hr + 1]), fmaxf(s[mt][1][2 * hr], s[mt][1][2 * hr + 1]));
                x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 1));
                x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 2));
                const float mn = fmaxf(m[mt][hr], x * c2);
                const float f = m[mt][hr] == -INFINITY ? 0.f : ex2_approx(m[mt][hr] - mn);
                m[mt][hr] = mn;
                l[mt][hr][0] *= f;
                l[mt][hr][1] *= f;
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    dq[mt][n][2 * hr] *= f;
                    dq[mt][n][2 * hr + 1] *= f;
                    if constexpr (!LOCAL) {
                        od[mt][n][2 * hr] *= f;
                        od[mt][n][2 * hr + 1] *= f;
                    }
                }
            }
    };
    auto exponents = [&](float (&s)[MT][2][4]) {
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int hr = 0; hr < 2; ++hr) {
                const float nm = m[mt][hr] == -INFINITY ? 0.f : -m[mt][hr];
#pragma unroll
                for (int nt = 0; nt < 2; ++nt)
                    ffma2(s[mt][nt][2 * hr], s[mt][nt][2 * hr + 1], s[mt][nt][2 * hr], s[mt][nt][2 * hr + 1], c2, c2,
                          nm, nm);
            }
    };

    // KS 16-key blocks at once, the first at shared-memory row address kst and
    // position j; ALL: every pair is of this kernel's kind, else the others are
    // masked: their weight is 0, and their dP - D is set to 0 too, so that no
    // 0 * infinity arises from a key the row does not see.
    auto step = [&](auto all_c, auto ks_c, uint32_t kst, int j) {
        constexpr bool ALL = decltype(all_c)::value != 0;
        constexpr int KS = decltype(ks_c)::value;
        float s[KS][MT][2][4];
        auto in_kind = [&](int k, int mt, int nt, int e) {
            const int i = r0 + 16 * mt + grp + 8 * (e >> 1), jj = j + 16 * k + 8 * nt + 2 * tig + (e & 1);
            return LOCAL ? jj <= i && jj > i - w : jj <= i - w;
        };
        auto masked_scores = [&]() {
#pragma unroll
            for (int k = 0; k < KS; ++k) {
                scores<W, MT>(s[k], qa, kst + 16 * k * LD + b_lane<LD>(lane), zero);
                if constexpr (!ALL) {
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                s[k][mt][nt][e] = in_kind(k, mt, nt, e) ? s[k][mt][nt][e] : -INFINITY;
                }
            }
        };
        masked_scores();
        float top = -INFINITY;
#pragma unroll
        for (int k = 0; k < KS; ++k) {
            exponents(s[k]);
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int nt = 0; nt < 2; ++nt) {
                    top = sm100::max3(top, s[k][mt][nt][0], s[k][mt][nt][1]);
                    top = sm100::max3(top, s[k][mt][nt][2], s[k][mt][nt][3]);
                }
        }
        if (__builtin_expect(__any_sync(0xffffffffu, top > kRaise) || fresh, 0)) {
            // rare: the scores again (they were overwritten), then larger maxima
            masked_scores();
#pragma unroll
            for (int k = 0; k < KS; ++k)
                raise(s[k]);
#pragma unroll
            for (int k = 0; k < KS; ++k)
                exponents(s[k]);
            bool none = false;  // once no maximum is -infinity, every row has seen a key
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
                none = none || m[mt][0] == -INFINITY || m[mt][1] == -INFINITY;
            fresh = __any_sync(0xffffffffu, none);
        }
#pragma unroll
        for (int k = 0; k < KS; ++k) {
            const uint32_t kr = kst + 16 * k * LD, vr = kr + Sm::V;
            float dp[MT][2][4];
            scores<W, MT>(dp, da, vr + b_lane<LD>(lane), nD);
            if constexpr (!ALL) {
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            dp[mt][nt][e] = in_kind(k, mt, nt, e) ? dp[mt][nt][e] : 0.f;
            }
            uint32_t ds[MT][4], pa[MT][4];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
#pragma unroll
                for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                    for (int hr = 0; hr < 2; ++hr) {
                        float &p0 = s[k][mt][nt][2 * hr], &p1 = s[k][mt][nt][2 * hr + 1];
                        p0 = ex2_approx(p0);
                        p1 = ex2_approx(p1);
                        add2(l[mt][hr][0], l[mt][hr][1], p0, p1, l[mt][hr][0], l[mt][hr][1]);
                        mul2(dp[mt][nt][2 * hr], dp[mt][nt][2 * hr + 1], p0, p1, dp[mt][nt][2 * hr],
                             dp[mt][nt][2 * hr + 1]);
                    }
                frag_a(ds[mt], dp[mt][0], dp[mt][1]);
                if constexpr (!LOCAL)
                    frag_a(pa[mt], s[k][mt][0], s[k][mt][1]);
            }
            accumulate<W, MT>(dq, ds, kr + bt_lane<LD>(lane));
            if constexpr (!LOCAL)
                accumulate<W, MT>(od, pa, vr + bt_lane<LD>(lane));
        }
    };

    for (int t = 0; t < ntiles; ++t) {
        cp_async_wait<NS - 2>();
        __syncthreads();  // tile t is in; every warp is done with tile t - 1
        stage(t + NS - 1);
        const uint32_t ks = sb + (t % NS) * Sm::STAGE;
        const int jt = jlo + t * BK;
        // Eq. 3 over the warp's rows: a tile, or a 16-key block, all of whose pairs are of this kind
        auto whole = [&](int j, int n) {
            return LOCAL ? j + n - 1 <= r0 && j > r0 + 16 * MT - 1 - w : j + n - 1 <= r0 - w;
        };
        if (whole(jt, BK)) {
#pragma unroll 1
            for (int kc = 0; kc < BK / 16; kc += Sh::KSQ)
                step(Int<1>(), Int<Sh::KSQ>(), ks + 16 * kc * LD, 0);
            continue;
        }
#pragma unroll 1
        for (int kc = 0; kc < BK / 16; ++kc) {
            const int j = jt + 16 * kc;
            if (LOCAL ? j > r0 + 16 * MT - 1 : j > r0 + 16 * MT - 1 - w)
                break;  // no pair of this block or a later one
            if (LOCAL && j + 15 <= r0 - w)
                continue;
            if (whole(j, 16))
                step(Int<1>(), Int<1>(), ks + 16 * kc * LD, 0);
            else
                step(Int<0>(), Int<1>(), ks + 16 * kc * LD, j);
        }
    }

    float lsum[MT][2];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int hr = 0; hr < 2; ++hr) {
            float x = l[mt][hr][0] + l[mt][hr][1];
            x += __shfl_xor_sync(0xffffffffu, x, 1);
            x += __shfl_xor_sync(0xffffffffu, x, 2);
            lsum[mt][hr] = x;
        }
    if constexpr (!LOCAL) {
        // the global part's sums relative to 2^m: dq~ (times scale), O^D, m, l
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int hr = 0; hr < 2; ++hr) {
                const int i = r0 + 16 * mt + grp + 8 * hr;
                if (i >= N)
                    continue;
                const size_t row = headrow + i;
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    const int c = 8 * n + 2 * tig;
                    *reinterpret_cast<float2 *>(a.dqt + row * W + c) =
                        make_float2(dq[mt][n][2 * hr] * a.scale, dq[mt][n][2 * hr + 1] * a.scale);
                    *reinterpret_cast<float2 *>(a.od + row * W + c) = make_float2(od[mt][n][2 * hr], od[mt][n][2 * hr + 1]);
                }
                if (tig == 0) {
                    a.gm[row] = m[mt][hr];
                    a.gl[row] = lsum[mt][hr];
                }
            }
    } else {
        static_assert(!LOCAL || MT == 1, "the lift stages 64 rows");
        // merge with the global part; dq = scale dq_loc / l + (dq~ / l) Uk
        cp_async_wait<0>();
        __syncthreads();  // the stage area is idle
        float *lift = reinterpret_cast<float *>(tsm);  // [64][DD + 1]
        float *uk = lift + 64 * (DD + 1);              // [DD][64]; 16-byte words: 64 * (DD + 1) floats come before
        for (int e = tid; e < DD * 16; e += kTc)
            reinterpret_cast<float4 *>(uk)[e] = __ldg(reinterpret_cast<const float4 *>(a.Uk + (size_t)g * DD * 64) + e);
        const int nv = min(ROWS, N - i0);
        for (int e = tid; e < nv * DD; e += kTc)
            lift[(e / DD) * (DD + 1) + e % DD] = a.dqt[(headrow + i0) * DD + e];
        __syncthreads();
        float o[2][8][2];
#pragma unroll
        for (int n = 0; n < 8; ++n)
            o[0][n][0] = o[0][n][1] = o[1][n][0] = o[1][n][1] = 0.f;
        const float *x = lift + (16 * warp + grp) * (DD + 1);  // (rows past the end lift stale bytes and are not stored)
        lift_rows<DD, 64>(o, x, x + 8 * (DD + 1), uk, tig);
#pragma unroll
        for (int hr = 0; hr < 2; ++hr) {
            const int i = r0 + grp + 8 * hr;
            if (i >= N)
                continue;
            const size_t row = headrow + i;
            const float mg = a.gm[row], lg = a.gl[row], ml = m[0][hr], M = fmaxf(mg, ml);
            const float L = (mg == -INFINITY ? 0.f : lg * ex2_approx(mg - M)) +
                            (ml == -INFINITY ? 0.f : lsum[0][hr] * ex2_approx(ml - M));
            const float lse = M + log2f(L);
            const float fl = ml == -INFINITY ? 0.f : exp2f(ml - lse) * a.scale;
            const float fg = mg == -INFINITY ? 0.f : exp2f(mg - lse);
            if (tig == 0) {
                a.lse[row] = -lse;
                a.fac[row] = fg;
            }
            bf16 *dst = static_cast<bf16 *>(a.dq) + row * 64;
#pragma unroll
            for (int n = 0; n < 8; ++n)
                *reinterpret_cast<uint32_t *>(dst + 8 * n + 2 * tig) = cvt_bf16x2(
                    fmaf(dq[0][n][2 * hr], fl, o[hr][n][0] * fg), fmaf(dq[0][n][2 * hr + 1], fl, o[hr][n][1] * fg));
        }
    }
}

// ---------------------------------------------------------------- dk, dv

template <int W, bool LOCAL, int DD>
struct DkvSmem {
    using Sh = Shape<W, LOCAL>;
    static constexpr uint32_t DO = Sh::BK * ld_of<W>();
    static constexpr uint32_t LSE = 2 * DO, DR = LSE + Sh::BK * 4, STAGE = DR + Sh::BK * 4;
    static constexpr uint32_t TOTAL = Sh::NS * STAGE;
    // the epilogue's lift: [64][DD + 1] rows and W_down^T
    static_assert(!LOCAL || 64 * (DD + 1) * 4 + DD * kLiftLd * 4 <= TOTAL, "the lift fits in the stage area");
};

template <int W, bool LOCAL, int DD>
__global__ void __launch_bounds__(kTc, Shape<W, LOCAL>::MINB) bwd_dkv_tc_kernel(Args a)
{
    using Sh = Shape<W, LOCAL>;
    using Sm = DkvSmem<W, LOCAL, DD>;
    constexpr int MT = Sh::MT, ROWS = Sh::ROWS, BK = Sh::BK, NS = Sh::NS, LD = ld_of<W>(), NT = W / 8;
    extern __shared__ __align__(128) unsigned char tsm[];
    const uint32_t sb = smem_u32(tsm);
    const int N = a.N, w = min(a.w, N);
    const int heads = a.B * a.Hkv, bg = blockIdx.x % heads, b = bg / a.Hkv, g = bg % a.Hkv;
    const int j0 = blockIdx.x / heads * ROWS;  // keys with the most queries first
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, grp = lane >> 2, tig = lane & 3;
    const size_t kvbase = (size_t)bg * N;
    // queries [ilo, ihi): local j <= i < j + w, global i >= j + w
    const int j_last = min(N, j0 + ROWS) - 1;
    const int ilo = LOCAL ? j0 : (w < N - j0 ? j0 + w : N);
    const int ihi = LOCAL ? (w > 0 ? (w < N - j_last ? j_last + w : N) : j0) : N;
    const int per_head = (ihi - ilo + BK - 1) / BK, ntiles = a.G * per_head;
    auto stage = [&](int t) {
        if (t < ntiles) {
            const int i = ilo + (t % per_head) * BK, n = N - i;
            const size_t row = ((size_t)b * a.Hq + g * a.G + t / per_head) * N + i;
            const uint32_t dst = sb + (t % NS) * Sm::STAGE;
            stage_rows<W, BK>(dst, (LOCAL ? static_cast<const bf16 *>(a.q) : a.qtb) + row * W, n, tid);
            stage_rows<W, BK>(dst + Sm::DO, (LOCAL ? static_cast<const bf16 *>(a.dout) : a.dotb) + row * W, n, tid);
            if (tid < BK) {
                if (tid < n) {
                    sm100::cp_async4(dst + Sm::LSE + tid * 4, a.lse + row + tid);
                    sm100::cp_async4(dst + Sm::DR + tid * 4, a.drow + row + tid);
                } else {  // past the end: weights 2^(-infinity) = 0
                    float *f = reinterpret_cast<float *>(tsm + (t % NS) * Sm::STAGE);
                    f[Sm::LSE / 4 + tid] = -INFINITY;
                    f[Sm::DR / 4 + tid] = 0.f;
                }
            }
        }
        cp_async_commit();
    };
    // this CTA's keys and values into the last stage, then the first tiles
    stage_rows<W, ROWS>(sb + (NS - 1) * Sm::STAGE, static_cast<const bf16 *>(LOCAL ? a.k : a.kd) + (kvbase + j0) * W,
                        N - j0, tid);
    stage_rows<W, ROWS>(sb + (NS - 1) * Sm::STAGE + Sm::DO,
                        static_cast<const bf16 *>(LOCAL ? a.v : a.vd) + (kvbase + j0) * W, N - j0, tid);
    cp_async_commit();
    for (int t = 0; t < NS - 1; ++t)
        stage(t);
    cp_async_wait<NS - 1>();
    __syncthreads();

    const int r0 = j0 + 16 * MT * warp;  // this warp's keys r0 .. r0 + 16 MT - 1
    uint32_t ka[MT][W / 16][4], va[MT][W / 16][4];
    float dk[MT][NT][4], dv[MT][NT][4], zero[MT][2][4];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
        const uint32_t own = sb + (NS - 1) * Sm::STAGE + 16 * (MT * warp + mt) * LD;
        load_a<W>(ka[mt], own, lane);
        load_a<W>(va[mt], own + Sm::DO, lane);
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                dk[mt][n][e] = dv[mt][n][e] = 0.f;
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                zero[mt][nt][e] = 0.f;
    }
    const float c2 = a.c2;

    // the 16 queries at shared-memory row address qst (log-sum-exp and D at
    // `rows`) and position i; ALL as in the dq kernel
    auto step = [&](auto all_c, uint32_t qst, const float *rows, int i) {
        constexpr bool ALL = decltype(all_c)::value != 0;
        const uint32_t dst = qst + Sm::DO;
        float s[MT][2][4], dp[MT][2][4], nD[MT][2][4];
        float2 nl[2];
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
            const float2 d = *reinterpret_cast<const float2 *>(rows + (Sm::DR - Sm::LSE) / 4 + 8 * nt + 2 * tig);
            nl[nt] = *reinterpret_cast<const float2 *>(rows + 8 * nt + 2 * tig);
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                nD[mt][nt][0] = nD[mt][nt][2] = d.x;
                nD[mt][nt][1] = nD[mt][nt][3] = d.y;
            }
        }
        scores<W, MT>(s, ka, qst + b_lane<LD>(lane), zero);
        scores<W, MT>(dp, va, dst + b_lane<LD>(lane), nD);
        if constexpr (!ALL) {
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int jj = r0 + 16 * mt + grp + 8 * (e >> 1), ii = i + 8 * nt + 2 * tig + (e & 1);
                        const bool in = LOCAL ? jj <= ii && jj > ii - w : jj <= ii - w;
                        s[mt][nt][e] = in ? s[mt][nt][e] : -INFINITY;
                        dp[mt][nt][e] = in ? dp[mt][nt][e] : 0.f;
                    }
        }
        uint32_t pa[MT][4], ds[MT][4];
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int hr = 0; hr < 2; ++hr) {
                    float &p0 = s[mt][nt][2 * hr], &p1 = s[mt][nt][2 * hr + 1];
                    ffma2(p0, p1, p0, p1, c2, c2, nl[nt].x, nl[nt].y);
                    p0 = ex2_approx(p0);
                    p1 = ex2_approx(p1);
                    mul2(dp[mt][nt][2 * hr], dp[mt][nt][2 * hr + 1], p0, p1, dp[mt][nt][2 * hr],
                         dp[mt][nt][2 * hr + 1]);
                }
            frag_a(pa[mt], s[mt][0], s[mt][1]);
            frag_a(ds[mt], dp[mt][0], dp[mt][1]);
        }
        accumulate<W, MT>(dv, pa, dst + bt_lane<LD>(lane));
        accumulate<W, MT>(dk, ds, qst + bt_lane<LD>(lane));
    };

    for (int t = 0; t < ntiles; ++t) {
        cp_async_wait<NS - 2>();
        __syncthreads();
        stage(t + NS - 1);
        const uint32_t qs = sb + (t % NS) * Sm::STAGE;
        const float *rows = reinterpret_cast<const float *>(tsm + (t % NS) * Sm::STAGE + Sm::LSE);
        const int it = ilo + (t % per_head) * BK;
        auto whole = [&](int i, int n) {  // (rows past the sequence's end have weight 0)
            return LOCAL ? i >= r0 + 16 * MT - 1 && i + n - 1 < r0 + w : i >= r0 + 16 * MT - 1 + w;
        };
        if (whole(it, BK)) {
#pragma unroll Sh::UNKV
            for (int qc = 0; qc < BK / 16; ++qc)
                step(Int<1>(), qs + 16 * qc * LD, rows + 16 * qc, 0);
            continue;
        }
#pragma unroll 1
        for (int qc = 0; qc < BK / 16; ++qc) {
            const int i = it + 16 * qc;
            if (i >= N || (LOCAL && i >= r0 + 16 * MT - 1 + w))
                break;
            if (LOCAL ? i + 15 < r0 : i + 15 < r0 + w)
                continue;
            if (whole(i, 16))
                step(Int<1>(), qs + 16 * qc * LD, rows + 16 * qc, 0);
            else
                step(Int<0>(), qs + 16 * qc * LD, rows + 16 * qc, i);
        }
    }

    if constexpr (!LOCAL) {
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int hr = 0; hr < 2; ++hr) {
                const int j = r0 + 16 * mt + grp + 8 * hr;
                if (j >= N)
                    continue;
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    const size_t at = (kvbase + j) * W + 8 * n + 2 * tig;
                    *reinterpret_cast<float2 *>(a.dkd + at) =
                        make_float2(dk[mt][n][2 * hr] * a.scale, dk[mt][n][2 * hr + 1] * a.scale);
                    *reinterpret_cast<float2 *>(a.dvd + at) = make_float2(dv[mt][n][2 * hr], dv[mt][n][2 * hr + 1]);
                }
            }
    } else {
        static_assert(!LOCAL || MT == 1, "the lift stages 64 rows");
        // dk = scale dk_loc + dk^D Dk^T, dv = dv_loc + dv^D Dv^T, one after the other
        float *lift = reinterpret_cast<float *>(tsm);  // [64][DD + 1]
        float *wt = lift + 64 * (DD + 1);              // [DD][kLiftLd] W_down^T
        const int nv = min(ROWS, N - j0);
#pragma unroll
        for (int kv = 0; kv < 2; ++kv) {
            cp_async_wait<0>();
            __syncthreads();  // the stage area (or the other lift) is idle
            const float *Wd = (kv ? a.Dv : a.Dk) + (size_t)g * 64 * DD;
            const float *x = (kv ? a.dvd : a.dkd) + (kvbase + j0) * DD;
            for (int e = tid; e < 64 * DD; e += kTc)
                wt[(e % DD) * kLiftLd + e / DD] = __ldg(Wd + e);
            for (int e = tid; e < nv * DD; e += kTc)
                lift[(e / DD) * (DD + 1) + e % DD] = x[e];
            __syncthreads();
            float o[2][8][2];
#pragma unroll
            for (int hr = 0; hr < 2; ++hr)
#pragma unroll
                for (int n = 0; n < 8; ++n) {
                    o[hr][n][0] = kv ? dv[0][n][2 * hr] : dk[0][n][2 * hr] * a.scale;
                    o[hr][n][1] = kv ? dv[0][n][2 * hr + 1] : dk[0][n][2 * hr + 1] * a.scale;
                }
            const float *xr = lift + (16 * warp + grp) * (DD + 1);
            lift_rows<DD, kLiftLd>(o, xr, xr + 8 * (DD + 1), wt, tig);
#pragma unroll
            for (int hr = 0; hr < 2; ++hr) {
                const int j = r0 + grp + 8 * hr;
                if (j >= N)
                    continue;
                bf16 *dst = static_cast<bf16 *>(kv ? a.dv : a.dk) + (kvbase + j) * 64;
#pragma unroll
                for (int n = 0; n < 8; ++n)
                    *reinterpret_cast<uint32_t *>(dst + 8 * n + 2 * tig) = cvt_bf16x2(o[hr][n][0], o[hr][n][1]);
            }
        }
    }
}

// ---------------------------------------------------------------- rows

// Per query row: blockIdx.z % 2 = 0: q~ = q Uk^T; 1: dO~ = dO Uv^T and -D = -dO . o;
// blockIdx.z / 2: block of 32 columns.  A CTA takes `rows` rows.  On the CUDA cores
// this took 143 us at B8 H16 N8192, d_down 16 (469 MB, 69 us at the copy rate), so 99.
template <int DD>
__global__ void __launch_bounds__(32 * kTcWarps) bwd_rows_tc_kernel(Args a, int rows)
{
    constexpr int COLS = DD < 32 ? DD : 32, NT = COLS / 8;
    const bool z = blockIdx.z & 1;
    const int c0 = (blockIdx.z >> 1) * COLS, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tig = lane & 3;
    const int bh = blockIdx.y, g = bh % a.Hq / a.G;
    const size_t row0 = (size_t)bh * a.N;
    const bf16 *x = static_cast<const bf16 *>(z ? a.dout : a.q) + row0 * 64;
    const float *U = (z ? a.Uv : a.Uk) + ((size_t)g * DD + c0) * 64;
    const auto w = [&](int t, int c) { return __ldg(U + c * 64 + t); };
    const int share = rows / kTcWarps, r0 = blockIdx.x * rows + warp * share, r1 = min(a.N, r0 + share);
    if (r0 >= r1)
        return;
    ProjectTc<NT> p;
    p.load(lane, w);
    const bf16 *o = static_cast<const bf16 *>(a.out) + row0 * 64;
    auto each = [&](const uint4(&v)[2][2], int r) {
        if (!z || c0 > 0)
            return;
#pragma unroll
        for (int hr = 0; hr < 2; ++hr) {
            const int row = r + (lane >> 2) + 8 * hr;
            float s[2] = {0.f, 0.f};  // a chain per 16-byte chunk, the eight added pairwise
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                float d[8], y[8];
                unpack(v[hr][i], d, bf16());
                unpack(row < r1 ? __ldg(reinterpret_cast<const uint4 *>(o + (size_t)row * 64) + tig + 4 * i)
                                : make_uint4(0u, 0u, 0u, 0u),
                       y, bf16());
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    s[i] = fmaf(d[k], y[k], s[i]);
                s[i] += __shfl_xor_sync(0xffffffffu, s[i], 1);
                s[i] += __shfl_xor_sync(0xffffffffu, s[i], 2);
            }
            if (tig == 0 && row < r1)
                a.drow[row0 + row] = -(s[0] + s[1]);
        }
    };
    project_rows_tc<NT>(x, (z ? a.dotb : a.qtb) + row0 * DD + c0, DD, r0, r1, p, lane, w, each);
}

// ---------------------------------------------------------------- projection gradients

// bwd_wpart on the tensor cores: X is bf16, and Y (fp32) enters as the sum of
// three bf16 terms, hi + mid + lo, each the rounded rest of the one before
// (24 bits together, so a product is off by no more than an fp32 one's
// rounding), accumulated in fp32.  X^T is the A operand (ldmatrix.trans from
// rows of 64), Y the B operand, split in registers.  Eight warps share out the
// columns (32 at most each) and the 16-row steps of a stage of 128 rows and are
// added up in warp order.  The CUDA-core kernel spent 344 us on B8 H16 N8192,
// d_down 16, on instructions: 19 per 16 products.
constexpr int kWtRows = 128;

template <int DD>
struct WpartTc {
    static constexpr int NC = DD < 32 ? DD : 32;       // columns per warp
    static constexpr int CG = DD / NC, RW = 8 / CG;    // column groups, warps that share out the rows
    static constexpr int XLD = 64 * 2 + 16, YLD = DD + 4;  // bytes / floats per padded row
    static constexpr uint32_t Y = kWtRows * XLD, FAC = Y + kWtRows * YLD * 4, STAGE = FAC + kWtRows * 4;
    static constexpr uint32_t TOTAL = 2 * STAGE;
    static_assert(RW * 64 * DD * 4 <= (int)TOTAL, "the warps' sums fit in the stage area");
};

// The same sums as fp32 chains on the CUDA cores, for a chunk whose tensor-core sums
// are not all finite: an infinity times the split's rests (of either sign, or 0) is
// NaN there also where the product itself is an infinity.  Row r of the sum is token
// r % N of one of `heads` heads from head0 (of all_heads) of sequence r / (N heads).
template <int DD>
__device__ __noinline__ void wpart_chains(const bf16 *X, const float *Y, const float *fac, long r0, long r1, int N,
                                          int heads, int head0, int all_heads, float *dst)
{
    for (int o = threadIdx.x; o < 64 * DD; o += 256) {
        float s = 0.f;
        for (long r = r0; r < r1; ++r) {
            const long u = r / N, at = (u / heads * all_heads + head0 + u % heads) * N + r % N;
            const float y = Y[at * DD + o % DD];
            s = fmaf(__bfloat162float(X[at * 64 + o / DD]), fac ? y * fac[at] : y, s);
        }
        dst[o] = s;
    }
}

template <int DD>
__global__ void __launch_bounds__(256) bwd_wpart_tc_kernel(Args a)
{
    using L = WpartTc<DD>;
    constexpr int NC = L::NC, RW = L::RW;
    extern __shared__ __align__(128) unsigned char tsm[];
    const uint32_t sb = smem_u32(tsm);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, grp = lane >> 2, tig = lane & 3;
    const int chunk = blockIdx.x, g = blockIdx.y, which = blockIdx.z;
    const bool per_kv = which == 0 || which == 2;
    const int heads = per_kv ? 1 : a.G;
    const long nrows = (long)a.B * heads * a.N;
    const long r0 = nrows * chunk / kChunks, r1 = nrows * (chunk + 1) / kChunks;
    const bf16 *X = static_cast<const bf16 *>(which == 0 ? a.k : which == 1 ? a.q : which == 2 ? a.v : a.dout);
    const float *Yp = which == 0 ? a.dkd : which == 1 ? a.dqt : which == 2 ? a.dvd : a.od;
    const int ntiles = (int)((r1 - r0 + kWtRows - 1) / kWtRows);
    // the next tile to stage starts at row i of sequence-and-head u
    long u = r0 / a.N;
    int i = (int)(r0 % a.N);
    auto base_of = [&](long v) -> long {
        return (per_kv ? v * a.Hkv + g : v / a.G * a.Hq + g * a.G + v % a.G) * a.N;
    };
    long base = base_of(u);
    auto stage = [&](int t) {
        const uint32_t d = sb + (t & 1) * L::STAGE;
        const int n = (int)min((long)kWtRows, r1 - r0 - (long)t * kWtRows);
        auto row_of = [&](int r) -> long {
            int k = i + r;
            if (k < a.N)
                return base + k;
            long v = u;
            for (; k >= a.N; k -= a.N)
                ++v;
            return base_of(v) + k;
        };
#pragma unroll
        for (int e = 0; e < kWtRows * 8 / 256; ++e) {
            const int r = tid / 8 + 32 * e, c = tid % 8;
            const bool ok = r < n;
            cp16z(d + r * L::XLD + c * 16, X + (ok ? row_of(r) * 64 + c * 8 : 0), ok);
        }
#pragma unroll
        for (int e = 0; e < kWtRows * (DD / 4) / 256; ++e) {
            const int r = tid / (DD / 4) + 256 / (DD / 4) * e, c = tid % (DD / 4);
            const bool ok = r < n;
            cp16z(d + L::Y + r * (L::YLD * 4) + c * 16, Yp + (ok ? row_of(r) * DD + c * 4 : 0), ok);
        }
        if (!per_kv && tid < kWtRows) {
            if (tid < n)
                sm100::cp_async4(d + L::FAC + tid * 4, a.fac + row_of(tid));
            else
                reinterpret_cast<float *>(tsm + (t & 1) * L::STAGE + L::FAC)[tid] = 0.f;
        }
        cp_async_commit();
        for (i += kWtRows; i >= a.N; i -= a.N)
            base = base_of(++u);
    };
    float acc[4][NC / 8][4];
#pragma unroll
    for (int mt = 0; mt < 4; ++mt)
#pragma unroll
        for (int n = 0; n < NC / 8; ++n)
            acc[mt][n][0] = acc[mt][n][1] = acc[mt][n][2] = acc[mt][n][3] = 0.f;
    const int c0 = warp / RW * NC, k0 = warp % RW;
    if (ntiles > 0)
        stage(0);
    for (int t = 0; t < ntiles; ++t) {
        cp_async_wait<0>();
        __syncthreads();  // tile t is in; every warp is done with tile t - 1
        if (t + 1 < ntiles)
            stage(t + 1);
        const uint32_t xs = sb + (t & 1) * L::STAGE;
        const float *ys = reinterpret_cast<const float *>(tsm + (t & 1) * L::STAGE + L::Y);
        const float *fs = reinterpret_cast<const float *>(tsm + (t & 1) * L::STAGE + L::FAC);
#pragma unroll
        for (int ks = 0; ks < kWtRows / 16 / RW; ++ks) {
            const int row = 16 * (k0 + RW * ks);
            uint32_t xa[4][4];
#pragma unroll
            for (int mt = 0; mt < 4; ++mt)
                ldsm_x4_t(xs + (row + (lane & 7) + ((lane >> 4) << 3)) * L::XLD + (16 * mt + ((lane >> 3) & 1) * 8) * 2,
                          xa[mt]);
            float f[4] = {1.f, 1.f, 1.f, 1.f};
            if (!per_kv)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    f[e] = fs[row + 2 * tig + (e & 1) + 8 * (e >> 1)];
#pragma unroll
            for (int n = 0; n < NC / 8; ++n) {
                uint32_t b[3][2];  // hi, mid, lo of rows 2 tig, + 1 (and + 8) of column grp
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float *y = ys + (row + 2 * tig + 8 * e) * L::YLD + c0 + 8 * n + grp;
                    float y0 = y[0], y1 = y[L::YLD];
                    if (!per_kv) {
                        y0 *= f[2 * e];
                        y1 *= f[2 * e + 1];
                    }
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        b[k][e] = cvt_bf16x2(y0, y1);
                        // (an infinity gives NaN here; see wpart_chains)
                        y0 -= bf16lo(b[k][e]);
                        y1 -= bf16hi(b[k][e]);
                    }
                }
#pragma unroll
                for (int mt = 0; mt < 4; ++mt)
#pragma unroll
                    for (int k = 0; k < 3; ++k)
                        mma_bf16_acc(acc[mt][n], xa[mt], b[k][0], b[k][1]);
            }
        }
    }
    __syncthreads();
    float *red = reinterpret_cast<float *>(tsm);  // [RW][64][DD]
#pragma unroll
    for (int mt = 0; mt < 4; ++mt)
#pragma unroll
        for (int n = 0; n < NC / 8; ++n)
#pragma unroll
            for (int hr = 0; hr < 2; ++hr)
                *reinterpret_cast<float2 *>(red + (size_t)k0 * 64 * DD + (16 * mt + grp + 8 * hr) * DD + c0 + 8 * n + 2 * tig) =
                    make_float2(acc[mt][n][2 * hr], acc[mt][n][2 * hr + 1]);
    __syncthreads();
    float *dst = a.part + (((size_t)chunk * 4 + which) * a.Hkv + g) * 64 * DD;
    bool bad = false;
    for (int o = tid; o < 64 * DD; o += 256) {
        float s = red[o];
#pragma unroll
        for (int k = 1; k < RW; ++k)
            s += red[k * 64 * DD + o];
        bad |= !(fabsf(s) < INFINITY);
        dst[o] = s;
    }
    if (__syncthreads_or(bad))
        wpart_chains<DD>(X, Yp, per_kv ? nullptr : a.fac, r0, r1, a.N, heads, g * heads, per_kv ? a.Hkv : a.Hq, dst);
}

// ---------------------------------------------------------------- host side

template <typename K>
static cudaError_t opt_in(K kern, size_t smem)
{
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess)  // several CTAs per SM need the largest shared-memory carve-out
        e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
    return e;
}

template <int DD>
static cudaError_t run_tc(const Args &a, cudaStream_t s)
{
    auto dq_g = bwd_dq_tc_kernel<DD, false, DD>;
    auto dq_l = bwd_dq_tc_kernel<64, true, DD>;
    auto dkv_g = bwd_dkv_tc_kernel<DD, false, DD>;
    auto dkv_l = bwd_dkv_tc_kernel<64, true, DD>;
    constexpr size_t sq_g = DqSmem<DD, false, DD>::TOTAL, sq_l = DqSmem<64, true, DD>::TOTAL;
    constexpr size_t sk_g = DkvSmem<DD, false, DD>::TOTAL, sk_l = DkvSmem<64, true, DD>::TOTAL;
    static PerDeviceOnce once;
    cudaError_t e = per_device_once(once, [&](int) {
        cudaError_t e2 = opt_in(dq_g, sq_g);
        if (e2 == cudaSuccess)
            e2 = opt_in(dq_l, sq_l);
        if (e2 == cudaSuccess)
            e2 = opt_in(dkv_g, sk_g);
        if (e2 == cudaSuccess)
            e2 = opt_in(dkv_l, sk_l);
        if (e2 == cudaSuccess)
            e2 = opt_in(bwd_wpart_tc_kernel<DD>, WpartTc<DD>::TOTAL);
        return e2;
    });
    if (e != cudaSuccess)
        return e;
    constexpr int blocks = 2 * (DD < 32 ? 1 : DD / 32);
    const int rows = project_tc_rows(a.N, (long long)a.B * a.Hq * blocks);
    bwd_rows_tc_kernel<DD><<<dim3((a.N + rows - 1) / rows, a.B * a.Hq, blocks), 32 * kTcWarps, 0, s>>>(a, rows);
    constexpr int RG = Shape<DD, false>::ROWS, RL = Shape<64, true>::ROWS;
    const unsigned tg = (a.N + RG - 1) / RG, tl = (a.N + RL - 1) / RL;
    dq_g<<<a.B * a.Hq * tg, kTc, sq_g, s>>>(a);
    dq_l<<<a.B * a.Hq * tl, kTc, sq_l, s>>>(a);
    dkv_g<<<a.B * a.Hkv * tg, kTc, sk_g, s>>>(a);
    dkv_l<<<a.B * a.Hkv * tl, kTc, sk_l, s>>>(a);
    bwd_wpart_tc_kernel<DD><<<dim3(kChunks, a.Hkv, 4), 256, WpartTc<DD>::TOTAL, s>>>(a);
    bwd_wsum_kernel<DD><<<(4 * a.Hkv * 64 * DD + kThreads - 1) / kThreads, kThreads, 0, s>>>(a);
    return cudaGetLastError();
}

// bf16 storage: the tensor-core kernels for d_down >= 16 (whole 16-wide
// k-steps); d_down = 8 keeps the CUDA-core kernels.
cudaError_t run_bf16(int dd, const Args &a, cudaStream_t s)
{
    switch (dd) {
    case 8: return run<bf16, 8>(a, s);
    case 16: return run_tc<16>(a, s);
    case 32: return run_tc<32>(a, s);
    case 64: return run_tc<64>(a, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace bwd
}  // namespace dar
