// dar_append.cu -- Eq. 1 (bottleneck down-projection) as a bulk kernel and as
// the window-exit migration of the mixed-dimension cache.
//
// Every bottleneck element is ONE fp32 fused-multiply-add chain over
// t = 0..63 starting from +0.0f, rounded once to the storage type, so a
// token's cached vector is bit-identical whichever kernel produced it.
#include "dar_common.cuh"
#include "dar_launch.h"
#include "dar_prep.cuh"
#include "dar_project.cuh"
#include "dar_sm100.cuh"

namespace dar {

// ---------------------------------------------------------------- bulk Eq. 1
//
// A block takes a tile of contiguous token rows (dar_project.cuh); two chains
// advance per instruction (fma.rn.f32x2: outputs c and c + 1 share x_t) and
// each element is still the exact fp32 chain acc = fma(x_t, W[t][c], acc).
// Threads take RPT rows each, NR apart.
// blockIdx.z selects the tensor: 0 = (x0, W0, out0), 1 = (x1, W1, out1).
struct BulkArgs {
    const void *x[2];
    const float *W[2];
    void *out[2];
    int Hkv, n;
    int ostride[2];   // output row stride of each tensor (columns dd.. are padding)
    int ones_col[2];  // first of 16 padding columns set to 1 (-1: all padding is 0)
};

template <typename T, int DD, int RPT, int NR>
__global__ void __launch_bounds__(NR *slices<DD>()) down_project_kernel(BulkArgs a)
{
    constexpr int R = RPT * NR, NT = NR * slices<DD>();
    constexpr int CW = cols_per_thread<DD>();
    __shared__ __align__(16) unsigned char rows[R * kHeadDim * sizeof(T)];
    __shared__ __align__(16) float Ws[kHeadDim * DD];
    const bool z = blockIdx.z != 0;  // (selects, not indexes: the arguments stay in parameter space)
    const T *x = static_cast<const T *>(z ? a.x[1] : a.x[0]);
    const int bg = blockIdx.y, g = bg % a.Hkv;
    const int j0 = blockIdx.x * R;
    const int nr = min(R, a.n - j0);
    stage_tile(rows, x + ((size_t)bg * a.n + j0) * kHeadDim, nr, threadIdx.x, NT);
    const float *W = (z ? a.W[1] : a.W[0]) + (size_t)g * kHeadDim * DD;
    for (int i = threadIdx.x; i < kHeadDim * DD / 4; i += NT)
        reinterpret_cast<float4 *>(Ws)[i] = __ldg(reinterpret_cast<const float4 *>(W) + i);
    sm100::cp_async_wait_all();
    __syncthreads();
    // this thread's rows: r0 + k * NR, columns c0 .. c0 + CW - 1 (rows past nr
    // compute on stale staging bytes and are not stored)
    const int r0 = threadIdx.x % NR, c0 = slices<DD>() > 1 ? (int)threadIdx.x / NR * CW : 0;
    float acc[RPT][CW];
    project_rows<T, DD, CW, RPT>(rows, Ws + c0, r0, NR, acc);
    const int ostride = z ? a.ostride[1] : a.ostride[0];
    const int ones_col = z ? a.ones_col[1] : a.ones_col[0];
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
        const int r = r0 + k * NR;
        if (r >= nr)
            continue;
        T *o = static_cast<T *>(z ? a.out[1] : a.out[0]) + ((size_t)bg * a.n + j0 + r) * ostride;
        store_row<T, CW>(o + c0, acc[k]);
        if (ostride > DD && c0 == 0) {  // padding after the values: zeros, or a block of 16 ones
            constexpr int OE = 16 / sizeof(T);
            for (int c = DD; c < ostride; c += OE) {
                float v[OE];
#pragma unroll
                for (int e = 0; e < OE; ++e)
                    v[e] = ones_col >= 0 && c + e >= ones_col && c + e < ones_col + 16 ? 1.f : 0.f;
                store_row<T, OE>(o + c, v);
            }
        }
    }
}

// ------------------------------------------------------------ cache append
//
// One CTA per sequence (so its length can be updated at the end).  Thread ch
// owns the Eq. 1 chains (kv, g, c) -- output c of KV head g of the keys
// (kv = 0) or values (kv = 1) -- and keeps that column of W in registers.
// Positions that leave the window in this call are staged up to kAppRows at a
// time in shared memory (from the ring for old occupants, from k_new/v_new for
// new tokens that leave at once); every chain thread runs its fixed-order
// chains over the staged rows and writes the pages.  After all ring reads, the
// new tokens that stay in the window are copied into their ring slots, then
// the length is updated.  Loads that do not depend on the length (W columns,
// the last new rows) are issued at entry, so a one-token step costs about two
// round trips to memory.
constexpr int kAppThreads = 512;
constexpr int kAppRows = 8;  // rows staged per round (fewer for many heads)
constexpr int kAppStageBytes = 96 << 10;

template <typename T>
__host__ __device__ inline int app_rows(int Hkv)
{
    const int per_row = 2 * Hkv * kHeadDim * (int)sizeof(T);
    const int r = kAppStageBytes / per_row;
    return r < 1 ? 1 : r > kAppRows ? kAppRows : r;
}

// Whether sequence lengths L and L + nb are ones an append can take (DAR_OK, or the status to report).
__device__ __forceinline__ int append_error(int L, int nb, const AppendArgs &a)
{
    const long long Lnew = (long long)L + nb;
    if (L < 0 || nb < 0 || nb > a.n)
        return DAR_ERR_INVALID_ARG;
    if (Lnew - a.w > (long long)a.maxp * kPage || Lnew > 0x7fffffffLL)
        return DAR_ERR_CAPACITY;
    return DAR_OK;
}

template <typename T, int DD>
__device__ __forceinline__ void append_sequence(const AppendArgs &a)
{
    constexpr int E = Granule<T>::kElems;
    constexpr int GPR = kHeadDim / E;  // 16-byte granules per 64-element row
    extern __shared__ __align__(16) unsigned char app_smem[];
    T *s_x = reinterpret_cast<T *>(app_smem);  // [rows][kv][Hkv][64]
    __shared__ int s_L, s_nb, s_ok;
    __shared__ int s_pid[kAppRows];  // page of each staged row (-1: invalid)

    const int b = blockIdx.x, tid = threadIdx.x;
    const int Hkv = a.Hkv, n = a.n, w = a.w;
    const int nchains = 2 * Hkv * DD;
    const int R = app_rows<T>(Hkv);
    const T *knew = static_cast<const T *>(a.k_new);
    const T *vnew = static_cast<const T *>(a.v_new);
    T *wk = static_cast<T *>(a.win_k);
    T *wv = static_cast<T *>(a.win_v);
    T *pk = static_cast<T *>(a.pool_kd);
    T *pv = static_cast<T *>(a.pool_vd);

    // ---- issued at entry: the length, this thread's first W column and one
    // granule of the last min(n, w) new rows (those land in the ring when the
    // sequence appends all n)
    if (tid == 0) {
        s_L = a.seq_lens[b];
        s_nb = a.n_per_seq ? a.n_per_seq[b] : n;
    }
    float wc[kHeadDim];
    auto load_w = [&](int ch) {
        const int kv = ch / (Hkv * DD), g = (ch / DD) % Hkv, c = ch % DD;
        const float *W = (kv ? a.Dv : a.Dk) + (size_t)g * kHeadDim * DD + c;
#pragma unroll
        for (int t = 0; t < kHeadDim; ++t)
            wc[t] = __ldg(W + (size_t)t * DD);
    };
    if (tid < nchains)
        load_w(tid);
    // granule i of the rows j0, j0 + 1, ... of k_new / v_new (i runs over
    // [row][kv][g][granule])
    auto new_granule = [&](int i, int j0) {
        const int q = i % GPR, rest = i / GPR;
        const int g = rest % Hkv, kv = (rest / Hkv) & 1, j = j0 + rest / (2 * Hkv);
        return (kv ? vnew : knew) + (((size_t)b * Hkv + g) * n + j) * kHeadDim + q * E;
    };
    const int pre_rows = min(n, w);
    uint4 pre = make_uint4(0u, 0u, 0u, 0u);
    if (tid < 2 * Hkv * pre_rows * GPR)
        pre = *reinterpret_cast<const uint4 *>(new_granule(tid, n - pre_rows));
    __syncthreads();
    if (tid == 0) {
        const int e = append_error(s_L, s_nb, a);
        if (e != DAR_OK)
            report(a.status, e);
        s_ok = e == DAR_OK;
    }
    __syncthreads();
    if (!s_ok || s_nb == 0)
        return;
    const int L = s_L, nb = s_nb, Lnew = L + nb;

    // ---- positions leaving the window: [p_lo, p_hi)
    const int p_lo = max(0, L - w), p_hi = max(0, Lnew - w);
    for (int m0 = p_lo; m0 < p_hi; m0 += R) {
        const int nr = min(R, p_hi - m0);
        for (int i = tid; i < nr * 2 * Hkv * GPR; i += blockDim.x) {  // stage [row][kv][g][64]
            const int q = i % GPR, rest = i / GPR;
            const int g = rest % Hkv, kv = (rest / Hkv) & 1, r = rest / (2 * Hkv);
            const int p = m0 + r;
            const T *src = p < L ? (kv ? wv : wk) + (((size_t)b * Hkv + g) * w + p % w) * kHeadDim
                                 : (kv ? vnew : knew) + (((size_t)b * Hkv + g) * n + (p - L)) * kHeadDim;
            reinterpret_cast<uint4 *>(s_x)[i] = *reinterpret_cast<const uint4 *>(src + q * E);
        }
        if (tid < nr) {
            const int lp = (m0 + tid) / kPage;
            const int id = lp < a.maxp ? a.block_table[(size_t)b * a.maxp + lp] : -1;
            const bool valid = id >= 0 && id < a.num_pages;
            if (!valid)
                report(a.status, DAR_ERR_CAPACITY);
            s_pid[tid] = valid ? id : -1;
        }
        __syncthreads();
        for (int ch0 = 0; ch0 < nchains; ch0 += blockDim.x) {
            const int ch = ch0 + tid;
            if (ch >= nchains)
                break;
            if (ch0 > 0)
                load_w(ch);
            const int kv = ch / (Hkv * DD), g = (ch / DD) % Hkv, c = ch % DD;
            T *pool = kv ? pv : pk;
            for (int r = 0; r < nr; ++r) {
                const uint4 *x4 = reinterpret_cast<const uint4 *>(s_x + ((size_t)(r * 2 + kv) * Hkv + g) * kHeadDim);
                float acc = 0.0f;  // Eq. 1: one fp32 FMA chain over t = 0..63
#pragma unroll
                for (int q = 0; q < GPR; ++q) {
                    float xf[E];
                    unpack(x4[q], xf, T());
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        acc = __fmaf_rn(xf[e], wc[q * E + e], acc);
                }
                const int id = s_pid[r], p = m0 + r;
                if (id >= 0)
                    pool[(((size_t)id * Hkv + g) * kPage + p % kPage) * DD + c] = from_f32<T>(acc);
            }
        }
        // the first chain group's W columns are needed again in the next round
        if (nchains > (int)blockDim.x && m0 + R < p_hi && tid < nchains)
            load_w(tid);
        __syncthreads();
    }

    // ---- new tokens that stay in the window: rows j_lo .. nb-1 (positions
    // L + j); every ring read above is complete
    const int j_lo = max(0, nb - w);
    const int granules = 2 * Hkv * (nb - j_lo) * GPR;
    const bool use_pre = nb == n;  // then the prefetched granules are exactly these
    for (int i = tid; i < granules; i += blockDim.x) {
        const int q = i % GPR, rest = i / GPR;
        const int g = rest % Hkv, kv = (rest / Hkv) & 1, j = j_lo + rest / (2 * Hkv);
        const uint4 v = (use_pre && i == tid) ? pre : *reinterpret_cast<const uint4 *>(new_granule(i, j_lo));
        T *dst = (kv ? wv : wk) + (((size_t)b * Hkv + g) * w + (L + j) % w) * kHeadDim + q * E;
        *reinterpret_cast<uint4 *>(dst) = v;
    }
    __syncthreads();
    if (tid == 0)
        a.seq_lens[b] = Lnew;
}

template <typename T, int DD>
__global__ void __launch_bounds__(kAppThreads) cache_append_kernel(AppendArgs a)
{
    append_sequence<T, DD>(a);
}

// The append of a decode step with the decode's query-side set-up (dar_prep.cuh)
// in further blocks: neither needs the other, and host time bounds a step over
// short contexts (one sequence of 101 tokens, 8 heads: 23.5 us with three launches,
// 20.9 with two; 32 sequences of 4096, 12 heads, on the device 31.2 and 30.5).
template <typename T, int DD>
__global__ void __launch_bounds__(kAppThreads) step_front_kernel(AppendArgs a, DecodeArgs d)
{
    sm100::grid_dep_launch();  // the stream kernel may start its set-up now
    if ((int)blockIdx.x < a.B)
        append_sequence<T, DD>(a);
    else
        prep_rows<T, DD, kAppThreads>(d, blockIdx.x - a.B, gridDim.x - a.B);
}

// ------------------------------------------------------- cache append, bulk
//
// The same append for calls with many tokens per sequence (a prompt or a chunk
// of one), spread over the chip: the kernel above runs one CTA per sequence,
// eight rows at a time, and leaves most SMs idle (32 prompts of 1000 to 4096
// tokens, 12 KV heads, d_down 16: 2740 us).  Here a CTA takes R consecutive new
// tokens of one (sequence, KV head, keys or values).  New token j (position
// L + j) pushes position m = L + j - w out of the window; the CTA that holds j
// projects that row -- from ring slot m % w, or from the new rows when m >= L
// -- into its page, and then overwrites ring slot (L + j) % w = m % w (j < w)
// with the last new token that lands there.  A ring slot therefore has one
// reader and one writer, in one CTA, and no order between CTAs is needed.  The
// length is advanced by a second kernel once every CTA has read it.  The FMA
// chains bound it: the same prompts take 122 us a call (2.0 G FMA, 50 us at the
// chip's fp32 rate; 329 MB, 49 us at the copy rate).
template <typename T, int DD, int RPT, int NR>
__device__ __forceinline__ void append_tile(const AppendArgs &a, int tiles)
{
    constexpr int R = RPT * NR, NT = NR * slices<DD>();
    constexpr int CW = cols_per_thread<DD>();
    constexpr int E = Granule<T>::kElems;
    constexpr int CPR = kHeadDim / E;
    __shared__ __align__(16) unsigned char rows[R * kHeadDim * sizeof(T)];
    __shared__ __align__(16) float Ws[kHeadDim * DD];
    const int tid = threadIdx.x, kv = blockIdx.y;
    const int bg = blockIdx.x / tiles, j0 = (blockIdx.x % tiles) * R;
    const int b = bg / a.Hkv, g = bg % a.Hkv;
    const int n = a.n, w = a.w;
    const int L = a.seq_lens[b], nb = a.n_per_seq ? a.n_per_seq[b] : n;
    if (append_error(L, nb, a) != DAR_OK || j0 >= nb)
        return;
    const T *xnew = static_cast<const T *>(kv ? a.v_new : a.k_new) + (size_t)bg * n * kHeadDim;
    T *ring = static_cast<T *>(kv ? a.win_v : a.win_k) + (size_t)bg * w * kHeadDim;
    const int nr = min(R, nb - j0);
    const bool any = (long long)L + j0 + nr > w;  // the tile's last token pushes a position out
    if (any) {
        const uint32_t rows_s = sm100::smem_u32(rows);
        for (int i = tid; i < nr * CPR; i += NT) {
            const int r = i / CPR, c = i % CPR, m = L + j0 + r - w;
            if (m >= 0) {
                const T *src = m < L ? ring + (size_t)(m % w) * kHeadDim : xnew + (size_t)(m - L) * kHeadDim;
                sm100::cp_async16(rows_s + (r * CPR + (c ^ (r & 7))) * 16, src + c * E);
            }
        }
        const float *W = (kv ? a.Dv : a.Dk) + (size_t)g * kHeadDim * DD;
        for (int i = tid; i < kHeadDim * DD / 4; i += NT)
            reinterpret_cast<float4 *>(Ws)[i] = __ldg(reinterpret_cast<const float4 *>(W) + i);
        const int r0 = tid % NR, c0 = slices<DD>() > 1 ? tid / NR * CW : 0;  // this thread's rows r0 + k * NR and columns
        int id[RPT];  // page of each of this thread's rows (-1: not a row that leaves, or no page)
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
            const int r = r0 + k * NR, m = L + j0 + r - w;
            id[k] = -1;
            if (r < nr && m >= 0) {
                const int e = a.block_table[(size_t)b * a.maxp + m / kPage];
                if (e >= 0 && e < a.num_pages)
                    id[k] = e;
                else
                    report(a.status, DAR_ERR_CAPACITY);
            }
        }
        sm100::cp_async_wait_all();
        __syncthreads();  // every ring row this CTA reads is in shared memory
        if (r0 - (tid & 31) < nr) {  // (a warp past the last row has nothing to do)
            float acc[RPT][CW];
            project_rows<T, DD, CW, RPT>(rows, Ws + c0, r0, NR, acc);
            T *pool = static_cast<T *>(kv ? a.pool_vd : a.pool_kd);
#pragma unroll
            for (int k = 0; k < RPT; ++k) {
                const int m = L + j0 + r0 + k * NR - w;
                if (id[k] >= 0)
                    store_row<T, CW>(pool + (((size_t)id[k] * a.Hkv + g) * kPage + m % kPage) * DD + c0, acc[k]);
            }
        }
    }
    // ring slots (L + j) % w, j < min(nb, w): the last new token of each
    const int slots = min(nb, w) - j0;
    for (int i = tid; i < min(slots, R) * CPR; i += NT) {
        const int c = i % CPR, j = j0 + i / CPR, last = j + (nb - 1 - j) / w * w;
        *reinterpret_cast<uint4 *>(ring + (size_t)((L + j) % w) * kHeadDim + c * E) =
            *reinterpret_cast<const uint4 *>(xnew + (size_t)last * kHeadDim + c * E);
    }
}

template <typename T, int DD, int RPT, int NR>
__global__ void __launch_bounds__(NR *slices<DD>()) append_bulk_kernel(AppendArgs a, int tiles)
{
    append_tile<T, DD, RPT, NR>(a, tiles);
    sm100::grid_dep_wait();  // launched beside the kernel before it: end after that one
}

// Advances the lengths (and reports refused sequences) after append_bulk_kernel.
__global__ void append_lens_kernel(AppendArgs a)
{
    sm100::grid_dep_wait();  // every CTA of the append has read the lengths
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= a.B)
        return;
    const int L = a.seq_lens[b], nb = a.n_per_seq ? a.n_per_seq[b] : a.n;
    const int e = append_error(L, nb, a);
    if (e != DAR_OK)
        report(a.status, e);
    else
        a.seq_lens[b] = L + nb;
}

// ----------------------------------------------------------------- launchers

// Big tiles (several rows per thread, so that one read of W feeds them all)
// once they give every SM two; otherwise one row per thread.  Measured on the
// prefill, big / small, us: 8 tiles (fp32, 4 heads x N 256) 20.2 / 17.3; 128
// tiles (16 heads x N 1000) 22.3 / 20.8; 512 tiles (32 heads x N 2000, d_down
// 64) 92 / 101; 1024 tiles (64 heads x N 2047) 82.6 / 85.3.
constexpr int kBulkSmallRows = 64;
constexpr long long kProjectBigCtas = kSms * 2;

template <typename T, int DD>
static cudaError_t down_project_dd(const BulkArgs &a, int B, int nz, cudaStream_t s)
{
    constexpr int R = rows_bulk<T>(), RPT = rows_per_thread<DD>(), NR = R / RPT, SR = kBulkSmallRows;
    if ((long long)(a.n + R - 1) / R * B * a.Hkv * nz >= kProjectBigCtas)
        down_project_kernel<T, DD, RPT, NR><<<dim3((a.n + R - 1) / R, B * a.Hkv, nz), NR * slices<DD>(), 0, s>>>(a);
    else
        down_project_kernel<T, DD, 1, SR><<<dim3((a.n + SR - 1) / SR, B * a.Hkv, nz), SR * slices<DD>(), 0, s>>>(a);
    return cudaGetLastError();
}

template <typename T>
static cudaError_t down_project_t(int dd, const BulkArgs &a, int B, int nz, cudaStream_t s)
{
    switch (dd) {
    case 8: return down_project_dd<T, 8>(a, B, nz, s);
    case 16: return down_project_dd<T, 16>(a, B, nz, s);
    case 32: return down_project_dd<T, 32>(a, B, nz, s);
    case 64: return down_project_dd<T, 64>(a, B, nz, s);
    default: return cudaErrorInvalidValue;
    }
}

static cudaError_t down_project_any(dar_dtype dt, int dd, const BulkArgs &a, int B, int nz, cudaStream_t s)
{
    if (a.n == 0 || B == 0)
        return cudaSuccess;
    return dt == DAR_F32 ? down_project_t<float>(dd, a, B, nz, s) : down_project_t<bf16>(dd, a, B, nz, s);
}

cudaError_t launch_down_project(dar_dtype dt, int dd, const void *x, const float *W, void *out,
                                int B, int Hkv, int n, int ostride, cudaStream_t s)
{
    BulkArgs a = {{x, x}, {W, W}, {out, out}, Hkv, n, {ostride, ostride}, {-1, -1}};
    return down_project_any(dt, dd, a, B, 1, s);
}

cudaError_t launch_down_project_kv(dar_dtype dt, int dd, const void *k, const void *v, const float *Dk,
                                   const float *Dv, void *kd, void *vd, int B, int Hkv, int n, int kstride,
                                   int vstride, int v_ones_col, cudaStream_t s)
{
    BulkArgs a = {{k, v}, {Dk, Dv}, {kd, vd}, Hkv, n, {kstride, vstride}, {-1, v_ones_col}};
    return down_project_any(dt, dd, a, B, 2, s);
}

// d: the decode whose query-side set-up joins the launch, or nullptr.
template <typename T, int DD>
static cudaError_t cache_append_dd(const AppendArgs &a, const DecodeArgs *d, cudaStream_t s)
{
    static PerDeviceOnce once;  // opt-in to more than 48 KB of shared memory, once per device
    const cudaError_t e = per_device_once(once, [](int) {
        const cudaError_t e2 = cudaFuncSetAttribute(cache_append_kernel<T, DD>,
                                                    cudaFuncAttributeMaxDynamicSharedMemorySize, kAppStageBytes);
        return e2 != cudaSuccess ? e2
                                 : cudaFuncSetAttribute(step_front_kernel<T, DD>,
                                                        cudaFuncAttributeMaxDynamicSharedMemorySize, kAppStageBytes);
    });
    if (e != cudaSuccess)
        return e;
    const size_t smem = (size_t)app_rows<T>(a.Hkv) * 2 * a.Hkv * kHeadDim * sizeof(T);
    if (d) {
        constexpr int warps = kAppThreads / 32;
        // A row's reads of Uk (one 16-byte word of each of its d_down lines at a time)
        // keep an SM's L1 busy for about 16 d_down cycles: wide rows go to more blocks
        // than their warps fill, as long as there are SMs.
        constexpr int per = DD > 16 ? 256 / DD : warps;
        const int rows = d->B * d->Hq, full = (rows + warps - 1) / warps;
        const int prep = min(2 * kSms, max(full, min((rows + per - 1) / per, kSms - a.B)));
        step_front_kernel<T, DD><<<a.B + prep, kAppThreads, smem, s>>>(a, *d);
    } else {
        cache_append_kernel<T, DD><<<a.B, kAppThreads, smem, s>>>(a);
    }
    return cudaGetLastError();
}

template <typename T>
static cudaError_t cache_append_t(int dd, const AppendArgs &a, const DecodeArgs *d, cudaStream_t s)
{
    switch (dd) {
    case 8: return cache_append_dd<T, 8>(a, d, s);
    case 16: return cache_append_dd<T, 16>(a, d, s);
    case 32: return cache_append_dd<T, 32>(a, d, s);
    case 64: return cache_append_dd<T, 64>(a, d, s);
    default: return cudaErrorInvalidValue;
    }
}

template <typename T, int DD, int RPT, int NR>
static cudaError_t append_bulk_launch(const AppendArgs &a, bool beside_prev, cudaStream_t s)
{
    const int tiles = (a.n + RPT * NR - 1) / (RPT * NR);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.B * a.Hkv * tiles), 2);
    cfg.blockDim = dim3(NR * slices<DD>());
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = beside_prev ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, append_bulk_kernel<T, DD, RPT, NR>, a, tiles);
    if (e != cudaSuccess)
        return e;
    cfg.gridDim = dim3((a.B + 127) / 128);
    cfg.blockDim = dim3(128);
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, append_lens_kernel, a);
}

// Here big tiles pay once they fill the chip a few times over, if their last rows
// are not mostly past the call's end (64 sequences, 32 heads, d_down 64, n = 9: 199 us
// with big tiles, 45 with small ones; 512 sequences, 4 heads, d_down 16: 47 and 19).
constexpr long long kBulkBigCtas = kSms * 6 * 2;

template <typename T, int DD>
static cudaError_t append_bulk(const AppendArgs &a, bool beside_prev, cudaStream_t s)
{
    constexpr int R = rows_bulk<T>();
    const long long tiles = (a.n + R - 1) / R, small = (a.n + kBulkSmallRows - 1) / kBulkSmallRows;
    if (tiles * a.B * a.Hkv * 2 >= kBulkBigCtas && 4 * tiles * R <= 5 * small * kBulkSmallRows)
        return append_bulk_launch<T, DD, rows_per_thread<DD>(), R / rows_per_thread<DD>()>(a, beside_prev, s);
    return append_bulk_launch<T, DD, 1, kBulkSmallRows>(a, beside_prev, s);
}

template <typename T>
static cudaError_t append_bulk_t(int dd, const AppendArgs &a, bool beside_prev, cudaStream_t s)
{
    switch (dd) {
    case 8: return append_bulk<T, 8>(a, beside_prev, s);
    case 16: return append_bulk<T, 16>(a, beside_prev, s);
    case 32: return append_bulk<T, 32>(a, beside_prev, s);
    case 64: return append_bulk<T, 64>(a, beside_prev, s);
    default: return cudaErrorInvalidValue;
    }
}

// More tokens than one round of the one-CTA-per-sequence kernel: the bulk
// kernel.  Measured (d_down 16, w 128, context 500), one CTA per sequence / bulk:
//   n = 8:  B 1, 8 heads 7.8 / 6.2 us; B 32, 12 heads 9.6 / 8.0; B 64, 8 heads 8.2 / 9.3
//   n = 9:               9.0 / 6.6;                                             9.5 / 8.7
//   n = 64:             38.0 / 8.5;                                            38.3 / 11.9
// and at n = 1 the bulk kernel's second launch costs 2 to 4 us.  It takes a CTA per
// (sequence, head, tensor) however few the tokens, so with many of those the other
// kernel keeps the calls of up to 32 tokens that it does faster: it costs about
// 0.6 us per token, 512 chains and wave of sequences, the bulk kernel 1.2 + 0.15
// d_down ns per CTA.  Measured, one CTA per sequence / bulk at n = 9, 16 and 24:
//   B 128, 16 heads, d_down 32:  19 / 32, 27 / 32, 37 / 33;   B 256, 8, 16:  18 / 19, 24 / 19, 32 / 20
//   B 256, 16 heads, d_down 64:  55 / 82, 83 / 83, 122 / 84;  B 152, 8, 32:  12 / 20, 16 / 20, 21 / 21
//   B 512, 16 heads, d_down 16:  47 / 62, 74 / 62, 113 / 65;  B 512, 4, 16:  26 / 19, 32 / 19, 45 / 20
//   B 64, 32 heads, d_down 64:   50 / 45, 77 / 46, 110 / 46;  B 512, 8, 8:   30 / 23, 40 / 23, 52 / 24
// (A cache with so many heads that not one row of them fits the staging area stays
// with the kernel that refuses it; so does a call whose CTAs a grid cannot count.)
constexpr int kBulkMinTokens = kAppRows + 1, kBulkAlwaysTokens = 33;

static bool use_bulk(dar_dtype dt, int dd, const AppendArgs &a)
{
    const long long row = 2ll * a.Hkv * kHeadDim * (dt == DAR_F32 ? 4 : 2);
    const long long tiles = ((long long)a.n + kBulkSmallRows - 1) / kBulkSmallRows;
    if (a.n < kBulkMinTokens || row > kAppStageBytes || tiles * a.B * a.Hkv > 0x7fffffffLL)
        return false;
    const long long groups = (2ll * a.Hkv * dd + kAppThreads - 1) / kAppThreads, waves = (a.B + kSms - 1) / kSms;
    return a.n >= kBulkAlwaysTokens || 2ll * a.B * a.Hkv * (8 + dd) < 4000ll * a.n * groups * waves;
}

cudaError_t launch_cache_append(dar_dtype dt, int dd, const AppendArgs &a, cudaStream_t s, bool beside_prev)
{
    if (a.B == 0)
        return cudaSuccess;
    if (use_bulk(dt, dd, a))
        return dt == DAR_F32 ? append_bulk_t<float>(dd, a, beside_prev, s) : append_bulk_t<bf16>(dd, a, beside_prev, s);
    return dt == DAR_F32 ? cache_append_t<float>(dd, a, nullptr, s) : cache_append_t<bf16>(dd, a, nullptr, s);
}

cudaError_t launch_step_front(dar_dtype dt, int dd, const AppendArgs &a, const DecodeArgs &d, cudaStream_t s,
                              bool *done)
{
    *done = !use_bulk(dt, dd, a);
    if (!*done)
        return launch_cache_append(dt, dd, a, s);
    return dt == DAR_F32 ? cache_append_t<float>(dd, a, &d, s) : cache_append_t<bf16>(dd, a, &d, s);
}

}  // namespace dar
