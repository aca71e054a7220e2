// dar_prefill_simt.cu -- causal DAR attention forward on the CUDA cores (fp32
// FFMA).  Used for fp32 storage, where the 1e-5 accuracy target rules out
// TF32 tensor cores.
//
// One warp = 4 query rows of one head, NW warps per CTA share key tiles of 64.
// For a warp, a key tile is all-global (every pair has i - j >= w), all-local
// (every pair i - j < w) or a band tile that holds both kinds; the element rule
// is Eq. 3 (local iff i - j < w).  Local pairs score q . k (d = 64); global
// pairs score q~ . k^D with q~ = q Uk^T (d_down; in the direct variant of
// Sec. 5, q~ is the row's own d_down query times scale_down / scale).  One
// online softmax covers both kinds, values accumulate in d (local) and d_down
// (global) and the global part is lifted once with Uv in the epilogue:
// o = (o_loc + o_glob Uv) / l.
//
// fp32 calls are small (gradient checks, reference runs), so what bounds them
// is the chain of steps of one row tile: short tiles put a call of 4 heads and
// 256 rows on 64 CTAs, tiles arrive by cp.async while the one before is worked
// on, and a thread takes 2 rows x 4 keys of the scores and 2 rows x 4 columns of
// the values, so that 6 16-byte shared-memory reads feed 32 products.  Measured
// against 64-row CTAs with one row x 16 keys per thread and no copies ahead
// (with the Eq. 1 kernel): B 1, 4 heads, N 256, w 32, d_down 16 73 -> 16 us;
// B 2, 16 heads, N 700, w 64 228 -> 115 us; B 1, 16 heads, N 700, w 500,
// d_down 8 335 -> 75 us.
#include "dar_common.cuh"
#include "dar_launch.h"
#include "dar_sm100.cuh"

namespace dar {

constexpr int kSimtKeys = 64, kSimtLd = kHeadDim + 4;  // padded rows: 8 consecutive ones fall in distinct banks

template <int DD, int NW>
struct SimtLayout {
    static constexpr int ROWS = 4 * NW, LDD = DD + 4;
    // floats of one stage: K, V, K^D, V^D of 64 keys
    static constexpr int V = kSimtKeys * kSimtLd, KD = V + kSimtKeys * kHeadDim, VD = KD + kSimtKeys * LDD;
    static constexpr int STAGE = VD + kSimtKeys * LDD;
    // after the two stages: q, weights of local and of global pairs, q~ (then the global values)
    static constexpr int Q = 2 * STAGE, PL = Q + ROWS * kSimtLd, PG = PL + ROWS * kSimtLd, QT = PG + ROWS * kSimtLd;
    static constexpr int BYTES = (QT + ROWS * LDD) * 4;
};

// s[r][i] = row r of x . row kg + 16 i of y over W columns (even and odd columns in sums of their own).
template <int W, int LDX, int LDY>
__device__ __forceinline__ void score_tile(const float *x, const float *y, int kg, float (&s)[2][4])
{
    float lo[2][4], hi[2][4];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int i = 0; i < 4; ++i)
            lo[r][i] = hi[r][i] = 0.f;
#pragma unroll 4
    for (int t = 0; t < W; t += 4) {
        float4 a[2];
#pragma unroll
        for (int r = 0; r < 2; ++r)
            a[r] = *reinterpret_cast<const float4 *>(x + r * LDX + t);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 b = *reinterpret_cast<const float4 *>(y + (kg + 16 * i) * LDY + t);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                sm100::ffma2(lo[r][i], hi[r][i], a[r].x, a[r].y, b.x, b.y, lo[r][i], hi[r][i]);
                sm100::ffma2(lo[r][i], hi[r][i], a[r].z, a[r].w, b.z, b.w, lo[r][i], hi[r][i]);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int i = 0; i < 4; ++i)
            s[r][i] = lo[r][i] + hi[r][i];
}

template <int DD, int NW>
__global__ void __launch_bounds__(32 * NW) prefill_simt_kernel(PrefillArgs a)
{
    using Lay = SimtLayout<DD, NW>;
    constexpr int ROWS = Lay::ROWS, LDD = Lay::LDD, NT = 32 * NW;
    extern __shared__ __align__(16) float sm[];
    const int N = a.N, w = a.w;
    const int bh = blockIdx.y, b = bh / a.Hq, h = bh % a.Hq, g = h / (a.Hq / a.Hkv);
    const int i0 = (gridDim.x - 1 - blockIdx.x) * ROWS;  // the longest rows first
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float *q = static_cast<const float *>(a.q) + ((size_t)b * a.Hq + h) * N * kHeadDim;
    const size_t bg = (size_t)b * a.Hkv + g;
    const float *k = static_cast<const float *>(a.k) + bg * N * kHeadDim;
    const float *v = static_cast<const float *>(a.v) + bg * N * kHeadDim;
    const float *kd = static_cast<const float *>(a.kd) + bg * N * DD;
    const float *vd = static_cast<const float *>(a.vd) + bg * N * DD;
    const float *Uk = a.Uk + (size_t)g * DD * kHeadDim;
    const float *Uv = a.Uv + (size_t)g * DD * kHeadDim;

    // start the copies of rows [j0, j0 + 64) of a W-wide tensor (rows past N: zeros)
    auto copy_rows = [&](float *dst, int ld, const float *src, int W, int j0) {
        const int ch = W / 4;
        for (int c = tid; c < kSimtKeys * ch; c += NT) {
            const int r = c / ch, e = c % ch * 4;
            float *d = dst + r * ld + e;
            if (j0 + r < N)
                sm100::cp_async16(sm100::smem_u32(d), src + (size_t)(j0 + r) * W + e);
            else
                *reinterpret_cast<float4 *>(d) = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    const int imax = min(N, i0 + ROWS) - 1, tiles = imax / kSimtKeys + 1;
    auto load_full = [&](int t) {  // what the local pairs of tile t read
        const int j0 = t * kSimtKeys;
        if (t < tiles && i0 - (j0 + kSimtKeys - 1) < w) {
            float *st = sm + (t & 1) * Lay::STAGE;
            copy_rows(st, kSimtLd, k, kHeadDim, j0);
            copy_rows(st + Lay::V, kHeadDim, v, kHeadDim, j0);
        }
    };
    auto load_down = [&](int t) {  // and the global ones
        const int j0 = t * kSimtKeys;
        if (t < tiles && i0 + ROWS - 1 - j0 >= w) {
            float *st = sm + (t & 1) * Lay::STAGE;
            copy_rows(st + Lay::KD, LDD, kd, DD, j0);
            copy_rows(st + Lay::VD, LDD, vd, DD, j0);
        }
    };
    load_full(0);

    // this warp's rows, scaled, and their q~ (a lane's rows: ra, ra + 1)
    const int wr = 4 * warp, ra = wr + (lane >> 4) * 2, kg = lane & 15;
    float *Qs = sm + Lay::Q, *Qt = sm + Lay::QT;
#pragma unroll
    for (int c = lane; c < 4 * kHeadDim / 4; c += 32) {
        const int r = wr + c / 16, e = c % 16 * 4;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i0 + r < N)
            x = __ldg(reinterpret_cast<const float4 *>(q + (size_t)(i0 + r) * kHeadDim + e));
        *reinterpret_cast<float4 *>(Qs + r * kSimtLd + e) =
            make_float4(x.x * a.qscale, x.y * a.qscale, x.z * a.qscale, x.w * a.qscale);
    }
    __syncwarp();
    for (int o = lane; o < 4 * DD; o += 32) {
        const int r = wr + o / DD, c = o % DD;
        float acc = 0.f;
        if (a.qd) {  // direct variant (Sec. 5): the row's own d_down query, at the global scale
            if (i0 + r < N)
                acc = static_cast<const float *>(a.qd)[(((size_t)b * a.Hq + h) * N + i0 + r) * DD + c] * a.qd_ratio *
                      a.qscale;
        } else {
#pragma unroll
            for (int t = 0; t < kHeadDim; t += 4) {
                const float4 u = __ldg(reinterpret_cast<const float4 *>(Uk + c * kHeadDim + t));
                const float4 x = *reinterpret_cast<const float4 *>(Qs + r * kSimtLd + t);
                acc = fmaf(x.x, u.x, acc);
                acc = fmaf(x.y, u.y, acc);
                acc = fmaf(x.z, u.z, acc);
                acc = fmaf(x.w, u.w, acc);
            }
        }
        Qt[r * LDD + c] = acc;
    }
    sm100::grid_dep_wait();  // k^D and v^D come from the kernel before
    load_down(0);

    // local values: rows ra, ra + 1, columns 4 kg ..; global values: row
    // ra + (lane / 8 & 1), the keys 8 x + lane % 8 of each tile, all columns
    float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f}, ol[2][4], og[DD];
#pragma unroll
    for (int e = 0; e < 4; ++e)
        ol[0][e] = ol[1][e] = 0.f;
#pragma unroll
    for (int c = 0; c < DD; ++c)
        og[c] = 0.f;
    const int gr = lane >> 3 & 1, gs = lane & 7;
    float *Pl = sm + Lay::PL, *Pg = sm + Lay::PG;
    const int wi = i0 + wr;  // the warp's first row

    for (int t = 0; t < tiles; ++t) {
        const int j0 = t * kSimtKeys;
        sm100::cp_async_wait_all();
        __syncthreads();  // tile t has landed and everyone is done with the stage that is filled next
        load_full(t + 1);
        load_down(t + 1);
        if (wi >= N || j0 > wi + 3)
            continue;  // (whole warp) nothing to see in this tile
        const float *st = sm + (t & 1) * Lay::STAGE;
        const bool any_local = wi - (j0 + kSimtKeys - 1) < w, any_global = wi + 3 - j0 >= w;
        float s[2][4];
        if (any_global)
            score_tile<DD, LDD, LDD>(Qt + ra * LDD, st + Lay::KD, kg, s);
        if (any_local) {
            float sl[2][4];
            score_tile<kHeadDim, kSimtLd, kSimtLd>(Qs + ra * kSimtLd, st, kg, sl);
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (i0 + ra + r - (j0 + kg + 16 * i) < w)
                        s[r][i] = sl[r][i];
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int row = i0 + ra + r;
            float mx = -INFINITY;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (row >= N || j0 + kg + 16 * i > row)
                    s[r][i] = -INFINITY;
                mx = fmaxf(mx, s[r][i]);
            }
#pragma unroll
            for (int x = 8; x; x >>= 1)
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, x));
            const float mnew = fmaxf(m[r], mx);
            const float alpha = m[r] == -INFINITY ? 0.f : exp2f(m[r] - mnew);
            m[r] = mnew;
            l[r] *= alpha;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int j = j0 + kg + 16 * i;
                const float p = s[r][i] == -INFINITY ? 0.f : exp2f(s[r][i] - mnew);
                const bool loc = row - j < w;
                l[r] += p;
                if (any_local)
                    Pl[(ra + r) * kSimtLd + kg + 16 * i] = loc ? p : 0.f;
                if (any_global)
                    Pg[(ra + r) * kSimtLd + kg + 16 * i] = loc ? 0.f : p;
            }
#pragma unroll
            for (int e = 0; e < 4; ++e)
                ol[r][e] *= alpha;
            if (gr == r) {
#pragma unroll
                for (int c = 0; c < DD; ++c)
                    og[c] *= alpha;
            }
        }
        __syncwarp();
        if (any_local) {
            const float *V = st + Lay::V + 4 * kg, *p = Pl + ra * kSimtLd;
#pragma unroll 4
            for (int j = 0; j < kSimtKeys; j += 4) {
                const float4 p0 = *reinterpret_cast<const float4 *>(p + j);
                const float4 p1 = *reinterpret_cast<const float4 *>(p + kSimtLd + j);
                const float pa[4] = {p0.x, p0.y, p0.z, p0.w}, pb[4] = {p1.x, p1.y, p1.z, p1.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 x = *reinterpret_cast<const float4 *>(V + (j + i) * kHeadDim);
                    sm100::ffma2(ol[0][0], ol[0][1], pa[i], pa[i], x.x, x.y, ol[0][0], ol[0][1]);
                    sm100::ffma2(ol[0][2], ol[0][3], pa[i], pa[i], x.z, x.w, ol[0][2], ol[0][3]);
                    sm100::ffma2(ol[1][0], ol[1][1], pb[i], pb[i], x.x, x.y, ol[1][0], ol[1][1]);
                    sm100::ffma2(ol[1][2], ol[1][3], pb[i], pb[i], x.z, x.w, ol[1][2], ol[1][3]);
                }
            }
        }
        if (any_global) {
#pragma unroll 4
            for (int j = gs; j < kSimtKeys; j += 8) {
                const float p = Pg[(ra + gr) * kSimtLd + j];
#pragma unroll
                for (int c = 0; c < DD; c += 4) {
                    const float4 x = *reinterpret_cast<const float4 *>(st + Lay::VD + j * LDD + c);
                    sm100::ffma2(og[c], og[c + 1], p, p, x.x, x.y, og[c], og[c + 1]);
                    sm100::ffma2(og[c + 2], og[c + 3], p, p, x.z, x.w, og[c + 2], og[c + 3]);
                }
            }
        }
        __syncwarp();  // the next tile's weights overwrite these
    }

    // epilogue: o = (o_loc + o_glob Uv) / l
#pragma unroll
    for (int c = 0; c < DD; ++c)
#pragma unroll
        for (int x = 4; x; x >>= 1)
            og[c] += __shfl_xor_sync(0xffffffffu, og[c], x);
    if (gs == 0) {
#pragma unroll
        for (int c = 0; c < DD; c += 4)
            *reinterpret_cast<float4 *>(Qt + (ra + gr) * LDD + c) = make_float4(og[c], og[c + 1], og[c + 2], og[c + 3]);
    }
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int x = 8; x; x >>= 1)
            l[r] += __shfl_xor_sync(0xffffffffu, l[r], x);
    __syncwarp();
#pragma unroll 8
    for (int c = 0; c < DD; ++c) {
        const float4 u = __ldg(reinterpret_cast<const float4 *>(Uv + c * kHeadDim + 4 * kg));
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const float x = Qt[(ra + r) * LDD + c];
            ol[r][0] = fmaf(x, u.x, ol[r][0]);
            ol[r][1] = fmaf(x, u.y, ol[r][1]);
            ol[r][2] = fmaf(x, u.z, ol[r][2]);
            ol[r][3] = fmaf(x, u.w, ol[r][3]);
        }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int i = i0 + ra + r;
        if (i < N) {
            const float inv = 1.f / l[r];
            *reinterpret_cast<float4 *>(static_cast<float *>(a.out) + (((size_t)b * a.Hq + h) * N + i) * kHeadDim +
                                        4 * kg) =
                make_float4(ol[r][0] * inv, ol[r][1] * inv, ol[r][2] * inv, ol[r][3] * inv);
        }
    }
}

template <int DD, int NW>
static cudaError_t simt_launch(const PrefillArgs &a, cudaStream_t s)
{
    auto kern = prefill_simt_kernel<DD, NW>;
    constexpr int smem = SimtLayout<DD, NW>::BYTES;
    static PerDeviceOnce once;  // attribute set-up per instantiation and device
    const cudaError_t e = per_device_once(once, [&](int) {
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    });
    if (e != cudaSuccess)
        return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((a.N + 4 * NW - 1) / (4 * NW), a.B * a.Hq);
    cfg.blockDim = dim3(32 * NW);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

// Rows per CTA: 8 as long as every tile has an SM, 32 where that makes a single
// wave (operands are read once for more rows), otherwise 16.  Measured, us, 8 /
// 16 / 32 rows: 4 heads x N 256 16.0 / 17.3 / 23.2; 8 heads x N 500, d_down 32
// 49 / 57 / 46; 32 heads x N 350 68 / 53 / 58; 32 heads x N 700 162 / 115 / 125.
template <int DD>
static cudaError_t simt_dd(const PrefillArgs &a, cudaStream_t s)
{
    const auto ctas = [&](int rows) { return ((long long)a.N + rows - 1) / rows * a.B * a.Hq; };
    if (ctas(8) <= kSms)
        return simt_launch<DD, 2>(a, s);
    return ctas(32) > kSms ? simt_launch<DD, 4>(a, s) : simt_launch<DD, 8>(a, s);
}

cudaError_t launch_prefill_simt(int dd, const PrefillArgs &a, cudaStream_t s)
{
    if (a.B == 0 || a.N == 0)
        return cudaSuccess;
    switch (dd) {
    case 8: return simt_dd<8>(a, s);
    case 16: return simt_dd<16>(a, s);
    case 32: return simt_dd<32>(a, s);
    case 64: return simt_dd<64>(a, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace dar
