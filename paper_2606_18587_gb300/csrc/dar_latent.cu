// dar_latent.cu -- DAR attention in the paper's own latent form (Sec. 2,
// Eq. 1-4 on hidden states, with the cache scheme of Sec. 5 "Compute and
// memory efficiency"): every token keeps ONE bottleneck c_j = h_j W_down,
// shared by all heads and by keys and values; a head g reaches a distant token
// through k'_j = (c_j W_up) W_K^g and v'_j = (c_j W_up) W_V^g.  With W_up
// absorbed (A_K^g = W_up W_K^g, A_V^g = W_up W_V^g, d_lat x d each):
//   global score   scale * q_i . k'_j = scale * (q_i A_K^gT) . c_j = scale * q~_i . c_j
//   global value   sum_j p_ij v'_j  = (sum_j p_ij c_j) A_V^g
// so a decode step streams each distant token's d_lat-vector once for all Hq
// heads (an MLA-like contraction: heads x d_lat against tokens x d_lat),
// while the last w tokens keep full keys and values per KV head.
//
// Kernels:
//  - latent_append: Eq. 1 (c = h W_down, one fp32 FMA chain over the D
//    inputs per element, rounded once to bf16) into the page of every new
//    token; new keys/values into the ring; then the lengths.
//  - latent_absorb: A_K, A_V (fp32 chains over D).
//  - decode: prep (q~ = q A_K^T, bf16), main (a persistent kernel: work
//    items are latent units of four pages and windows of one KV head; their
//    64-token tiles come through a TMA ring, four warps compute S = A B^T and
//    O += P V on mma.sync tensor cores with one online softmax per head and
//    write one partial record per segment),
//    merge (exact log-sum-exp combination of the partial records, then
//    o = (O_loc + O_lat A_V) / l).
#include <cuda.h>

#include <mutex>

#include "dar_common.cuh"
#include "dar_launch.h"
#include "dar_sm100.cuh"

namespace dar {
namespace lat {

using namespace sm100;

constexpr int kTok = DAR_PAGE_SIZE;  // tokens per page
constexpr int kPagesPerSplit = 4;
constexpr int kSplitTok = kTok * kPagesPerSplit;

struct Args {
    const void *q;  // [B][Hq][64]
    void *out;      // [B][Hq][64]
    const void *win_k, *win_v;
    const int32_t *block_table, *seq_lens;
    int32_t *status;
    const float *Ak, *Av;  // [Hkv][64][DL] (transposed), [Hkv][DL][64]
    bf16 *qt;              // [B][Hq][DL]
    float *rec_lat;        // [B][Hq][nspl][DL + 2]
    float *rec_win;        // [B][Hq][66]
    int B, Hq, Hkv, G, w, maxp, num_pages, nspl;
    float c2;  // scale * log2(e)
};

// ---------------------------------------------------------------- append

struct AppendArgs {
    const void *h;  // [B][n][D]
    const void *k_new, *v_new;  // [B][Hkv][n][64]
    const float *Wdown;         // [D][DL]
    void *win_k, *win_v, *pool_c;
    const int32_t *block_table, *n_per_seq;
    int32_t *seq_lens, *status;
    int B, Hkv, n, D, DL, w, maxp, num_pages;
};

// What an append does with sequence b: its length and count, or the status to report.
__device__ __forceinline__ int append_counts(const AppendArgs &a, int b, int &L, int &nb)
{
    nb = a.n_per_seq ? __ldg(a.n_per_seq + b) : a.n;
    L = a.seq_lens[b];
    if (nb < 0 || nb > a.n || L < 0)
        return DAR_ERR_INVALID_ARG;
    return (long long)L + nb > (long long)a.maxp * kTok && nb > 0 ? DAR_ERR_CAPACITY : DAR_OK;
}

constexpr int kAppTok = 4;  // tokens per block

// Block (token group, b): c = round_bf16(chain_k h[k] Wdown[k][c]) for the
// group's tokens, written to their pages; ring rows of the tokens that stay in
// the window.  The lengths are read here and advanced by latent_lens_kernel.
__global__ void __launch_bounds__(256) latent_append_kernel(AppendArgs a)
{
    extern __shared__ float hs[];  // [kAppTok][D]
    const int b = blockIdx.y, r0 = blockIdx.x * kAppTok;
    int L, nb;
    const int e = append_counts(a, b, L, nb);
    if (e != DAR_OK) {
        if (threadIdx.x == 0 && blockIdx.x == 0)
            report(a.status, e);
        return;
    }
    if (r0 >= nb)
        return;
    const int Lnew = L + nb;
    const int nt = min(kAppTok, nb - r0);
    const bf16 *h = static_cast<const bf16 *>(a.h) + ((size_t)b * a.n + r0) * a.D;
    for (int i = threadIdx.x; i < nt * a.D; i += blockDim.x)
        hs[i] = __bfloat162float(h[i]);
    // ring rows of the tokens that are still inside the window after the append
    for (int i = threadIdx.x; i < nt * a.Hkv * 8; i += blockDim.x) {  // 16-byte chunks of 64-wide rows
        const int t = i / (a.Hkv * 8), g = (i / 8) % a.Hkv, ch = i % 8;
        const int p = L + r0 + t;
        if (p < Lnew - a.w)
            continue;
        const size_t src = (((size_t)b * a.Hkv + g) * a.n + r0 + t) * 64 + ch * 8;
        const size_t dst = (((size_t)b * a.Hkv + g) * a.w + p % a.w) * 64 + ch * 8;
        reinterpret_cast<uint4 *>(a.win_k)[dst / 8] = reinterpret_cast<const uint4 *>(a.k_new)[src / 8];
        reinterpret_cast<uint4 *>(a.win_v)[dst / 8] = reinterpret_cast<const uint4 *>(a.v_new)[src / 8];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nt * a.DL; i += blockDim.x) {
        const int t = i / a.DL, c = i % a.DL;
        const int p = L + r0 + t;
        const int pid = __ldg(a.block_table + (size_t)b * a.maxp + p / kTok);
        if (pid < 0 || pid >= a.num_pages) {
            report(a.status, DAR_ERR_CAPACITY);
            continue;
        }
        float acc = 0.f;  // Eq. 1: one fp32 chain over e = 0..D-1 from +0
        for (int k = 0; k < a.D; ++k)
            acc = fmaf(hs[t * a.D + k], __ldg(a.Wdown + (size_t)k * a.DL + c), acc);
        static_cast<bf16 *>(a.pool_c)[((size_t)pid * kTok + p % kTok) * a.DL + c] = __float2bfloat16_rn(acc);
    }
}

// The same append as a matrix product, for D a multiple of 8 (rows of h that
// start on 16 bytes): rows are the B n tokens in memory order, whatever their
// sequence; a CTA takes ROWS rows and COLS columns and walks D in pieces of K
// through a ring of cp.async stages.  A thread holds the fp32 chains of TPT
// rows and CPT columns, two per instruction, in the order of the kernel above.
// The chains bound it (a chain cannot be split over threads, and no tensor core
// rounds like one): 8 prompts of 500 to 1000 tokens, D 2048, DL 256, are 3.1 G
// FMA, 85 us at the chip's fp32 rate: 844 us with the kernel above, 169 with
// this one (FMA pipe 63 % busy; 2.5 CTAs per SM on average, 3 on the fullest).
// WIDE tiles (8 rows x 4 columns per thread) read 6 operands per 32 products;
// narrow ones, for few tokens, take one column per thread, so that a warp's read
// of W is one wavefront and the chip's SMs share the columns.
constexpr int kTileThreads = 128, kTileStages = 3;

template <int TPT, int CPT>
struct Tile {
    static constexpr bool WIDE = CPT > 1;
    static constexpr int LC = WIDE ? 8 : 32;            // lanes side by side over the columns
    static constexpr int CW = WIDE ? 2 : 1;             // warps side by side over the columns
    static constexpr int GROUPS = 4 / CW * (32 / LC);   // threads that share a column
    static constexpr int ROWS = GROUPS * TPT, COLS = CW * LC * CPT;
    static constexpr int K = WIDE ? 64 : 128;
    static constexpr int W_BYTES = K * COLS * 4;
    static constexpr int STAGE = W_BYTES + ROWS * K * 2;
    static constexpr int TOTAL = kTileStages * STAGE;
};

template <int TPT, int CPT>
__global__ void __launch_bounds__(kTileThreads) latent_append_tiled_kernel(AppendArgs a)
{
    using T = Tile<TPT, CPT>;
    constexpr int NT = kTileThreads, ROWS = T::ROWS, COLS = T::COLS, K = T::K;
    extern __shared__ __align__(128) unsigned char tile[];
    __shared__ long long s_dst[ROWS];   // element offset of the row's bottleneck in the pool (-1: none)
    __shared__ int s_b[ROWS], s_slot[ROWS], s_j[ROWS];  // sequence, ring slot (-1: not kept), index in the call
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ncol = a.DL / COLS, c0 = (int)(blockIdx.x % ncol) * COLS;
    const long long rows = (long long)a.B * a.n, r0 = (long long)(blockIdx.x / ncol) * ROWS;
    bool live = false;
    for (int r = tid; r < ROWS; r += NT) {
        s_dst[r] = -1;
        s_slot[r] = -1;
        if (r0 + r >= rows)
            continue;
        const int b = (int)((r0 + r) / a.n), j = (int)((r0 + r) % a.n);
        int L, nb;
        const int e = append_counts(a, b, L, nb);
        if (e != DAR_OK) {
            if (j == 0 && c0 == 0)
                report(a.status, e);
            continue;
        }
        if (j >= nb)
            continue;
        live = true;
        const int p = L + j;
        s_b[r] = b;
        s_j[r] = j;
        s_slot[r] = j >= nb - a.w ? p % a.w : -1;
        const int pid = __ldg(a.block_table + (size_t)b * a.maxp + p / kTok);
        if (pid < 0 || pid >= a.num_pages)
            report(a.status, DAR_ERR_CAPACITY);
        else
            s_dst[r] = ((long long)pid * kTok + p % kTok) * a.DL + c0;
    }
    if (!__syncthreads_or(live))
        return;

    const bf16 *h = static_cast<const bf16 *>(a.h) + r0 * a.D;
    const int nr = (int)min((long long)ROWS, rows - r0), steps = (a.D + K - 1) / K;
    const uint32_t base = smem_u32(tile);
    auto load = [&](int st) {
        if (st < steps) {
            const int k0 = st * K, nk = min(K, a.D - k0);
            const uint32_t wb = base + st % kTileStages * T::STAGE, hb = wb + T::W_BYTES;
            for (int i = tid; i < nk * (COLS / 4); i += NT) {
                const int k = i / (COLS / 4), c = i % (COLS / 4);
                cp_async16(wb + i * 16, a.Wdown + (size_t)(k0 + k) * a.DL + c0 + c * 4);
            }
            for (int i = tid; i < nr * (K / 8); i += NT) {
                const int r = i / (K / 8), c = i % (K / 8);
                if (c * 8 < nk)
                    cp_async16(hb + r * (K * 2) + ((c ^ (r & 7)) << 4), h + (size_t)r * a.D + k0 + c * 8);
            }
        }
        cp_async_commit();
    };
#pragma unroll
    for (int st = 0; st < kTileStages - 1; ++st)
        load(st);

    // ring rows of the tokens that stay in the window, shared out over the column tiles
    for (int i = (int)(blockIdx.x % ncol) * NT + tid; i < nr * a.Hkv * 8; i += ncol * NT) {
        const int r = i / (a.Hkv * 8), g = i / 8 % a.Hkv, ch = i % 8;
        if (s_slot[r] < 0)
            continue;
        const size_t bg = (size_t)s_b[r] * a.Hkv + g;
        const size_t src = (bg * a.n + s_j[r]) * 8 + ch, dst = (bg * a.w + s_slot[r]) * 8 + ch;
        reinterpret_cast<uint4 *>(a.win_k)[dst] = reinterpret_cast<const uint4 *>(a.k_new)[src];
        reinterpret_cast<uint4 *>(a.win_v)[dst] = reinterpret_cast<const uint4 *>(a.v_new)[src];
    }

    // this thread's rows tg + GROUPS i and columns cg CPT ..
    const int cg = warp % T::CW * T::LC + lane % T::LC, tg = warp / T::CW * (32 / T::LC) + lane / T::LC;
    float acc[TPT][CPT];
#pragma unroll
    for (int i = 0; i < TPT; ++i)
#pragma unroll
        for (int c = 0; c < CPT; ++c)
            acc[i][c] = 0.f;
#pragma unroll 1
    for (int st = 0; st < steps; ++st) {
        cp_async_wait<kTileStages - 2>();
        __syncthreads();  // stage st has landed, and everyone is done with the one that load() overwrites
        load(st + kTileStages - 1);
        const unsigned char *ws = tile + st % kTileStages * T::STAGE, *hs = ws + T::W_BYTES;
        const int nq = min(K, a.D - st * K) / 8;
#pragma unroll 2
        for (int q = 0; q < nq; ++q) {
            uint4 x4[TPT];
#pragma unroll
            for (int i = 0; i < TPT; ++i) {
                const int r = tg + T::GROUPS * i;
                x4[i] = *reinterpret_cast<const uint4 *>(hs + r * (K * 2) + ((q ^ (r & 7)) << 4));
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                float x[TPT];
#pragma unroll
                for (int i = 0; i < TPT; ++i) {
                    const uint32_t u = e < 2 ? x4[i].x : e < 4 ? x4[i].y : e < 6 ? x4[i].z : x4[i].w;
                    x[i] = e & 1 ? bf16hi(u) : bf16lo(u);
                }
                const float *wr = reinterpret_cast<const float *>(ws) + (q * 8 + e) * COLS + cg * CPT;
                if constexpr (T::WIDE) {
                    const float4 w4 = *reinterpret_cast<const float4 *>(wr);
#pragma unroll
                    for (int i = 0; i < TPT; ++i) {
                        ffma2(acc[i][0], acc[i][1], x[i], x[i], w4.x, w4.y, acc[i][0], acc[i][1]);
                        ffma2(acc[i][2], acc[i][3], x[i], x[i], w4.z, w4.w, acc[i][2], acc[i][3]);
                    }
                } else if constexpr (TPT > 1) {
#pragma unroll
                    for (int i = 0; i < TPT; i += 2)
                        ffma2(acc[i][0], acc[i + 1][0], x[i], x[i + 1], *wr, *wr, acc[i][0], acc[i + 1][0]);
                } else {
                    acc[0][0] = fmaf(x[0], *wr, acc[0][0]);
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < TPT; ++i) {
        const long long dst = s_dst[tg + T::GROUPS * i];
        if (dst < 0)
            continue;
        bf16 *o = static_cast<bf16 *>(a.pool_c) + dst + cg * CPT;
        if constexpr (T::WIDE)
            *reinterpret_cast<uint2 *>(o) =
                make_uint2(cvt_bf16x2(acc[i][0], acc[i][1]), cvt_bf16x2(acc[i][2], acc[i][3]));
        else
            *o = __float2bfloat16_rn(acc[i][0]);
    }
}

__global__ void latent_lens_kernel(AppendArgs a)
{
    grid_dep_wait();  // every CTA of the append has read the lengths
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    int L, nb;
    if (b < a.B && append_counts(a, b, L, nb) == DAR_OK)
        a.seq_lens[b] = L + nb;
}

// A[g][c][t] = chain_e Wup[c][e] W[g][e][t] (fp32), for A_K (stored as
// [g][t][c]) and A_V (stored as [g][c][t]).
__global__ void latent_absorb_kernel(const float *Wup, const float *WK, const float *WV, float *Ak, float *Av, int D,
                                     int DL)
{
    const int g = blockIdx.y, c = blockIdx.x, t = threadIdx.x;  // 64 threads
    const float *wk = WK + (size_t)g * D * 64, *wv = WV + (size_t)g * D * 64;
    float ak = 0.f, av = 0.f;
    for (int e = 0; e < D; ++e) {
        const float u = __ldg(Wup + (size_t)c * D + e);
        ak = fmaf(u, __ldg(wk + (size_t)e * 64 + t), ak);
        av = fmaf(u, __ldg(wv + (size_t)e * 64 + t), av);
    }
    Ak[((size_t)g * 64 + t) * DL + c] = ak;  // [Hkv][d][d_lat]: the prep kernel reads rows of d_lat
    Av[((size_t)g * DL + c) * 64 + t] = av;  // [Hkv][d_lat][d]: the merge reads rows of d
}

// ---------------------------------------------------------------- decode: prep

// q~[b][h][c] = sum_t q[b][h][t] A_K[g][t][c] (fp32, stored as bf16).  Block
// (g, a few rows of KV head g): A_K^g staged in shared memory by one bulk copy,
// then one warp per row, lanes over c.  It starts the main kernel's launch at once: that
// kernel stages its first pages before it waits for q~.
constexpr int kRowsPerBlock = 8;  // at most: rows (one per warp) of one KV head per block
constexpr int kRowThreads = 32 * kRowsPerBlock;

// One bulk asynchronous copy of `bytes` (a multiple of 16) from global to
// shared memory, waited for by the whole block (bounded; on a timeout the
// status is flagged and false returned).
__device__ __forceinline__ bool stage_matrix(void *dst, const void *src, unsigned bytes, uint64_t *bar,
                                             int32_t *status)
{
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        mbar_init_fence();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        mbar_expect_tx(bar, bytes);
        for (unsigned off = 0; off < bytes; off += 16384u)  // in copies of at most 16 KB
            bulk_g2s(static_cast<char *>(dst) + off, static_cast<const char *>(src) + off,
                     bytes - off < 16384u ? bytes - off : 16384u, bar);
    }
    const bool ok = mbar_wait(bar, 0, nullptr);
    if (!ok && threadIdx.x == 0)
        report(status, DAR_ERR_DEVICE);
    return __syncthreads_and(ok) != 0;
}

template <int DL>
__global__ void __launch_bounds__(kRowThreads) latent_prep_kernel(Args a)
{
    extern __shared__ __align__(16) float aks[];  // [64][DL], then the barrier
    grid_dep_launch();
    const int g = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (!stage_matrix(aks, a.Ak + (size_t)g * 64 * DL, 64 * DL * 4, reinterpret_cast<uint64_t *>(aks + 64 * DL),
                      a.status))
        return;
    const int nrows = a.B * a.G;
    if (const int r = blockIdx.y * (blockDim.x >> 5) + warp; r < nrows) {
        const int row = (r / a.G) * a.Hq + g * a.G + r % a.G;
        const bf16 *qr = static_cast<const bf16 *>(a.q) + (size_t)row * 64;
        const float q0 = __bfloat162float(qr[lane]), q1 = __bfloat162float(qr[lane + 32]);
        float acc[DL / 32];
#pragma unroll
        for (int e = 0; e < DL / 32; ++e)
            acc[e] = 0.f;
#pragma unroll 8
        for (int t = 0; t < 64; ++t) {
            const float qv = __shfl_sync(0xffffffffu, t < 32 ? q0 : q1, t & 31);
#pragma unroll
            for (int e = 0; e < DL / 32; ++e)
                acc[e] = fmaf(qv, aks[t * DL + 32 * e + lane], acc[e]);
        }
#pragma unroll
        for (int e = 0; e < DL / 32; ++e)
            a.qt[(size_t)row * DL + 32 * e + lane] = __float2bfloat16_rn(acc[e]);
    }
}

// ---------------------------------------------------------------- decode: main

// Shared-memory tiles are rows of 128 bytes (64 bf16) with the 16-byte chunk
// index XOR (row % 8), the layout the 128-byte TMA swizzle writes; a W-wide
// row is W / 64 such blocks of rows.
__device__ __forceinline__ uint32_t swz(uint32_t base, int row, int chunk)
{
    return base + (uint32_t)(row * 128 + ((chunk ^ (row & 7)) << 4));
}

constexpr int kConsumerThreads = 128;  // warps 0-3: tensor-core work

// Persistent main kernel.  Work items, enumerated the same way by every
// thread: first the latent units (sequence b, up to four 64-token pages of its
// distant part), then the windows (sequence b, KV head g: the last min(L_b, w)
// tokens' full keys and values, in 64-token tiles).  A CTA takes a run of
// consecutive items of about equal estimated time; the units of one sequence in
// its run form one segment with one partial record (kept in the slot of its
// first unit; the other slots are marked empty).  The items' pages and tiles come
// through a ring of NST stages by TMA, and warps 0-3 run each stage on the tensor
// cores.
//
// Latency bounds it: two CTAs of four consumer warps share an SM (an SM holds
// six 32 KB stages), and the steps of a stage form a chain.  So the rows' A
// fragments stay in registers over a segment, a CTA writes one record for many
// pages, and a stage takes two barriers (row maxima, weights).  Warp 4 issues the
// copies, except at d_lat 256 with two row tiles, where a tenth warp on the SM
// would leave the others 168 registers: there thread 0 refills a stage at the
// next one's first barrier, when every warp is done with it (62 us for 64
// sequences of 1024 to 8192 tokens, 32 heads, d_lat 256; 72 with the warp; at 8
// heads, d_lat 128, 26 with the warp, 29 without).  Measured, prep to merge,
// against round-robin items with a record per unit and the rows read from shared
// memory: those 64 sequences 88 -> 64 us; 32 sequences of 4096, 12 heads, d_lat
// 192 28 -> 22; one sequence of 8192, 32 heads, d_lat 256 22 -> 18.
template <int DL, int MT>
struct MainLayout {
    static constexpr bool kProducer = !(DL == 256 && MT == 2);
    static constexpr int THREADS = kConsumerThreads + (kProducer ? 32 : 0);
    static constexpr uint32_t CST = DL >= 128 ? DL / 64 * 8192 : 16384;  // a latent page, or a window K + V tile
    static constexpr int NST = DL <= 128 ? 6 : DL == 192 ? 4 : 3;
    static constexpr uint32_t STG = 0;
    static constexpr uint32_t P = STG + NST * CST;                        // [MT*16][128 B]
    static constexpr uint32_t RED = P + MT * 16 * 128;                    // [4 warps][16] floats
    static constexpr uint32_t PREF = RED + 4 * 16 * 4;                    // [B + 1] ints (B <= 1024)
    static constexpr uint32_t BAR = PREF + (DAR_DECODE_MAX_BATCH + 1) * 4 + 4;
    static constexpr uint32_t TOTAL = (BAR + 16 * NST + 16 + 15) / 16 * 16;
};

// A latent segment (units of one sequence) or a window.
struct Segment {
    bool latent;
    int b, part;  // latent: first unit of the sequence; window: KV head
    int units;    // items it covers
    int npg;      // pages / tiles
};

constexpr float kMaxDrop = 16.f;  // log2 units: a unit further below weighs less than the rounding of the others

__device__ __forceinline__ void consumer_sync()
{
    asm volatile("bar.sync 1, %0;" ::"n"(kConsumerThreads) : "memory");
}

// What the warps hold of MT m-tiles (16 rows each) of W-wide rows.  Scores:
// warp `warp` takes m-tile warp % MT and 16 MT of a stage's 64 tokens, with the
// rows' A fragments in registers; values: W / 4 columns of every m-tile.
template <int W, int MT>
struct Rows {
    uint32_t a[W / 16][4];
    float o[MT][W / 32][4];
    float m[MT][2];  // reference of the weights (log2 units) of rows grp, grp + 8 of each m-tile
    float top[MT][2];  // the largest it has been
    float l[2];      // sums of this warp's weights, rows of its own m-tile

    // x: `n` rows of stride W (rows past n: zero)
    __device__ __forceinline__ void start(const bf16 *x, int n, int warp, int lane)
    {
        const int r0 = warp % MT * 16 + (lane >> 2), k0 = 2 * (lane & 3);
#pragma unroll
        for (int kk = 0; kk < W / 16; ++kk)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int r = r0 + 8 * (e & 1);
                a[kk][e] = r < n ? *reinterpret_cast<const uint32_t *>(x + (size_t)r * W + kk * 16 + 8 * (e >> 1) + k0)
                                 : 0u;
            }
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
#pragma unroll
            for (int nt = 0; nt < W / 32; ++nt)
                o[mt][nt][0] = o[mt][nt][1] = o[mt][nt][2] = o[mt][nt][3] = 0.f;
            m[mt][0] = m[mt][1] = top[mt][0] = top[mt][1] = -INFINITY;
        }
        l[0] = l[1] = 0.f;
    }

    // One stage: S = A B^T (B: the key-side tile), masks past ntok, one
    // online-softmax step per row (maxima exchanged through `red`), P into shared
    // memory, O += P V (V: the value-side tile).  refill() runs once every warp is
    // done with the stage before.  fresh: the weights' reference starts anew at this
    // tile's maximum, which may be the lower one (by kMaxDrop at most, so that the
    // sums stay finite).  A weight is rounded to bf16 relative to its reference, and
    // the token that sets it has a weight of exactly 1: a reference per unit keeps
    // the error of separate records per unit (against 64 bits, 64 sequences of 1024
    // to 8192 tokens, 32 heads: 0.002368 both; 0.002373 with one maximum over a
    // segment, which is 2 us faster, 65 us; separate records take 79).
    template <typename F>
    __device__ __forceinline__ void stage(uint32_t ktile, uint32_t vtile, unsigned char *sm_p, float *red, int ntok,
                                          float c2, bool fresh, int warp, int lane, F &&refill)
    {
        constexpr int NTS = 2 * MT, NT = W / 32;
        const int grp = lane >> 2, tig = lane & 3, own = warp % MT, tok0 = 16 * MT * (warp / MT);
        float sc[NTS][4];
#pragma unroll
        for (int nt = 0; nt < NTS; ++nt)
            sc[nt][0] = sc[nt][1] = sc[nt][2] = sc[nt][3] = 0.f;
        {
            const int tok = tok0 + (lane & 7) + ((lane >> 4) << 3), khalf = (lane >> 3) & 1;
#pragma unroll
            for (int kk = 0; kk < W / 16; ++kk) {
                const int ch = 2 * kk + khalf;
#pragma unroll
                for (int np = 0; np < MT; ++np) {
                    uint32_t bfr[4];
                    ldsm_x4(swz(ktile + (ch / 8) * 8192, tok + 16 * np, ch % 8), bfr);
                    mma_bf16_16816(sc[2 * np], a[kk], bfr[0], bfr[1]);
                    mma_bf16_16816(sc[2 * np + 1], a[kk], bfr[2], bfr[3]);
                }
            }
        }
        if (ntok < kTok)
#pragma unroll
            for (int nt = 0; nt < NTS; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (tok0 + 8 * nt + 2 * tig + (e & 1) >= ntok)
                        sc[nt][e] = -INFINITY;
#pragma unroll
        for (int hr = 0; hr < 2; ++hr) {
            float mx = -INFINITY;
#pragma unroll
            for (int nt = 0; nt < NTS; ++nt)
                mx = max3(mx, sc[nt][2 * hr], sc[nt][2 * hr + 1]);
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            if (tig == 0)
                red[warp * 16 + grp + 8 * hr] = mx;
        }
        consumer_sync();
        refill();
        float alpha[MT][2], mo[2];
        bool moved = false;
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int hr = 0; hr < 2; ++hr) {
                float mx = -INFINITY;
#pragma unroll
                for (int w2 = mt; w2 < 4; w2 += MT)
                    mx = fmaxf(mx, red[w2 * 16 + grp + 8 * hr]);
                const float mnew = fmaxf(fresh ? top[mt][hr] - kMaxDrop : m[mt][hr], mx * c2);
                top[mt][hr] = fmaxf(top[mt][hr], mnew);
                moved |= mnew != m[mt][hr];
                alpha[mt][hr] = m[mt][hr] == -INFINITY ? 0.f : ex2_approx(m[mt][hr] - mnew);
                m[mt][hr] = mnew;
                if (mt == own) {
                    l[hr] *= alpha[mt][hr];
                    mo[hr] = mnew;
                }
            }
#pragma unroll
        for (int hr = 0; hr < 2; ++hr) {
            const int row = own * 16 + grp + 8 * hr;
#pragma unroll
            for (int nt = 0; nt < NTS; ++nt) {
                const float x0 = sc[nt][2 * hr], x1 = sc[nt][2 * hr + 1];
                const float p0 = x0 == -INFINITY ? 0.f : ex2_approx(fmaf(x0, c2, -mo[hr]));
                const float p1 = x1 == -INFINITY ? 0.f : ex2_approx(fmaf(x1, c2, -mo[hr]));
                const uint32_t pk = cvt_bf16x2(p0, p1);
                l[hr] += bf16lo(pk) + bf16hi(pk);  // the weights the PV product uses
                *reinterpret_cast<uint32_t *>(sm_p + row * 128 + ((((tok0 >> 3) + nt) ^ (row & 7)) << 4) + 4 * tig) =
                    pk;
            }
        }
        if (__any_sync(0xffffffffu, moved)) {
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int hr = 0; hr < 2; ++hr)
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt) {
                        o[mt][nt][2 * hr] *= alpha[mt][hr];
                        o[mt][nt][2 * hr + 1] *= alpha[mt][hr];
                    }
        }
        consumer_sync();
        const uint32_t pbase = smem_u32(sm_p);
#pragma unroll
        for (int kk = 0; kk < kTok / 16; ++kk) {
            uint32_t afr[MT][4];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
                ldsm_x4(swz(pbase, mt * 16 + (lane & 15), 2 * kk + (lane >> 4)), afr[mt]);
            const int krow = 16 * kk + (lane & 7) + (((lane >> 3) & 1) << 3);
#pragma unroll
            for (int np = 0; np < NT / 2; ++np) {
                const int n0 = warp * (W / 4) + 16 * np + ((lane >> 4) << 3);
                uint32_t bfr[4];
                ldsm_x4_t(swz(vtile + (n0 / 64) * 8192, krow, (n0 % 64) / 8), bfr);
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    mma_bf16_16816(o[mt][2 * np], afr[mt], bfr[0], bfr[1]);
                    mma_bf16_16816(o[mt][2 * np + 1], afr[mt], bfr[2], bfr[3]);
                }
            }
        }
    }

    // Records (O, m, l) of rows 0 .. n - 1, after a stage: rec(row) points at W + 2 floats.
    template <typename F>
    __device__ __forceinline__ void finish(float *red, int n, int warp, int lane, F &&rec)
    {
        const int grp = lane >> 2, tig = lane & 3;
#pragma unroll
        for (int hr = 0; hr < 2; ++hr) {
            l[hr] += __shfl_xor_sync(0xffffffffu, l[hr], 1);
            l[hr] += __shfl_xor_sync(0xffffffffu, l[hr], 2);
        }
        // (`red` is free: its maxima were read before the last stage's second barrier)
        if (tig == 0) {
            red[warp * 16 + grp] = l[0];
            red[warp * 16 + grp + 8] = l[1];
        }
        consumer_sync();
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int hr = 0; hr < 2; ++hr) {
                const int row = mt * 16 + grp + 8 * hr;
                if (row >= n)
                    continue;
                float *r = rec(row);
#pragma unroll
                for (int nt = 0; nt < W / 32; ++nt)
                    *reinterpret_cast<float2 *>(r + warp * (W / 4) + 8 * nt + 2 * tig) =
                        make_float2(o[mt][nt][2 * hr], o[mt][nt][2 * hr + 1]);
                if (warp == 0 && tig == 0) {
                    float ls = 0.f;
#pragma unroll
                    for (int w2 = mt; w2 < 4; w2 += MT)
                        ls += red[w2 * 16 + grp + 8 * hr];
                    r[W] = m[mt][hr];
                    r[W + 1] = ls;
                }
            }
        consumer_sync();  // the sums are read: the next segment may write its maxima
    }
};

template <int DL, int MT>
__global__ void __launch_bounds__(MainLayout<DL, MT>::THREADS, 2)
    latent_main_kernel(const __grid_constant__ CUtensorMap tmC, const __grid_constant__ CUtensorMap tmK,
                       const __grid_constant__ CUtensorMap tmV, Args a)
{
    using Ly = MainLayout<DL, MT>;
    constexpr int NST = Ly::NST;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *sm = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                          ~uintptr_t(1023));
    const uint32_t sbase = smem_u32(sm);
    uint64_t *full = reinterpret_cast<uint64_t *>(sm + Ly::BAR);
    uint64_t *empty = full + NST;  // (with a producer warp)
    volatile int *abort_flag = reinterpret_cast<volatile int *>(empty + NST);
    float *red = reinterpret_cast<float *>(sm + Ly::RED);
    int *pref = reinterpret_cast<int *>(sm + Ly::PREF);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    grid_dep_launch();  // the merge kernel may launch; it waits for this grid to finish

    // lengths -> latent units per sequence, prefix sums (every CTA, the same)
    const int B = a.B, cap = a.maxp * kTok;
    auto len_of = [&](int b) {
        const int L = __ldg(a.seq_lens + b);
        return (L < 0 || L > cap) ? 0 : L;  // reported below; such a sequence gets no items
    };
    for (int b = tid; b < B; b += blockDim.x) {
        const int L = __ldg(a.seq_lens + b);
        if ((L < 0 || L > cap) && blockIdx.x == 0)
            report(a.status, DAR_ERR_CAPACITY);
        const int Lg = len_of(b) > a.w ? len_of(b) - a.w : 0;
        pref[b + 1] = (Lg + kSplitTok - 1) / kSplitTok;
    }
    __syncthreads();
    if (warp == 0) {
        int run = 0;
        for (int c0 = 0; c0 < B; c0 += 32) {
            int v = c0 + lane < B ? pref[c0 + lane + 1] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o)
                    v += u;
            }
            if (c0 + lane < B)
                pref[c0 + lane + 1] = run + v;
            run += __shfl_sync(0xffffffffu, v, 31);
        }
        if (lane == 0)
            pref[0] = 0;
    }
    if (tid == 0) {
        for (int st = 0; st < NST; ++st) {
            mbar_init(&full[st], 1);
            mbar_init(&empty[st], 4);  // one arrival per consumer warp
        }
        *abort_flag = 0;
        mbar_init_fence();
    }
    __syncthreads();
    // This CTA's run [k0, k1) of the items: those whose estimated start falls in
    // its share of the total (a page costs its width plus a stage's fixed part).
    // Measured, us, cw's factor 2 / 3 / 5 and 3 without the 2 in cu: 64 sequences of
    // 1024 to 8192 tokens, 8 KV heads, d_lat 256, w 256: 67 / 67 / 73 / 73; 32 of 4096,
    // 12, 192, 128: 31 / 29 / 29 / 29; 64 of 500 to 4000, 32, 128, 1024: 104 / 117 /
    // 168 / 195; 64 of 2000 to 8000, 1, 256, 16: 61 / 51 / 48 / 48; 48 of 1000 to 3000,
    // 16, 64, 700: 36 / 37 / 43 / 62.
    const int n_lat = pref[B];
    int k0, k1;
    {
        const long long cu = kPagesPerSplit * (DL / 64 + 2), cw = 3 * ((a.w + kTok - 1) / kTok + 1);
        const long long lat = n_lat * cu, total = lat + (long long)B * a.Hkv * cw;
        auto first = [&](long long c) {  // the first item that starts at c or later
            return (int)(c <= lat ? (c + cu - 1) / cu : n_lat + (c - lat + cw - 1) / cw);
        };
        // No more items than CTAs: one each (us, shares of the cost / one each: 3 sequences
        // of 2128 to 5765 tokens, 16 KV heads, d_lat 256, w 950 22.1 / 18.8; 20 of 100 to
        // 800, 8, 192, 64 20.7 / 17.7; 30 of 100 to 500, 8, 128, 40 16.8 / 15.8).
        if (const int items = n_lat + B * a.Hkv; items <= (int)gridDim.x) {
            k0 = min(items, (int)blockIdx.x);
            k1 = min(items, k0 + 1);
        } else {
            const long long share = (total + gridDim.x - 1) / gridDim.x;
            k0 = first(min(total, share * blockIdx.x));
            k1 = first(min(total, share * (blockIdx.x + 1)));
        }
    }
    auto segment_of = [&](int k) {
        Segment it;
        if (k < n_lat) {
            int lo = 0, hi = B - 1;  // the last b with pref[b] <= k
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (pref[mid] <= k)
                    lo = mid;
                else
                    hi = mid - 1;
            }
            it.latent = true;
            it.b = lo;
            it.part = k - pref[lo];
            it.units = min(k1, pref[lo + 1]) - k;
            const int L = len_of(lo), Lg = L > a.w ? L - a.w : 0;
            const int t0 = it.part * kSplitTok, t1 = min(Lg, t0 + it.units * kSplitTok);
            it.npg = (t1 - t0 + kTok - 1) / kTok;
        } else {
            const int r = k - n_lat;
            it.latent = false;
            it.b = r / a.Hkv;
            it.part = r % a.Hkv;
            it.units = 1;
            const int nwin = min(len_of(it.b), a.w);
            it.npg = (nwin + kTok - 1) / kTok;
        }
        return it;
    };

    // One thread: the next page or tile of the run into its stage of the ring.  The
    // page's index is loaded a call ahead.
    int pk = k0, pp = 0, pi = 0, pid = 0;
    Segment pit{};
    auto look_ahead = [&] {  // (pit, pp) is the page to fetch next; moves on past finished segments
        while (pp == pit.npg) {
            if (pk >= k1) {
                pit.npg = -1;
                return;
            }
            pit = segment_of(pk);
            pk += pit.units;
            pp = 0;
        }
        if (pit.latent)
            pid = __ldg(a.block_table + (size_t)pit.b * a.maxp + pit.part * kPagesPerSplit + pp);
    };
    auto fetch = [&] {
        const int st = pi++ % NST;
        unsigned char *dst = sm + Ly::STG + st * Ly::CST;
        if (pit.latent) {
            if (pid < 0 || pid >= a.num_pages) {
                report(a.status, DAR_ERR_CAPACITY);
                pid = 0;
            }
            mbar_expect_tx(&full[st], kTok * DL * 2);
#pragma unroll
            for (int cb = 0; cb < DL / 64; ++cb)
                tma_load_2d(dst + cb * 8192, &tmC, cb * 64, pid * kTok, &full[st]);
        } else {
            const int row = (pit.b * a.Hkv + pit.part) * a.w + pp * kTok;
            mbar_expect_tx(&full[st], 2 * 8192);
            tma_load_2d(dst, &tmK, 0, row, &full[st]);
            tma_load_2d(dst + 8192, &tmV, 0, row, &full[st]);
        }
        ++pp;
        look_ahead();
    };
    const int producer = Ly::kProducer ? kConsumerThreads : 0;  // the thread that issues the copies
    if (tid == producer) {
        prefetch_tensormap(&tmC);
        prefetch_tensormap(&tmK);
        prefetch_tensormap(&tmV);
        look_ahead();
        while (pit.npg >= 0 && pi < NST)
            fetch();
        if constexpr (Ly::kProducer)
            while (pit.npg >= 0 && mbar_wait(&empty[pi % NST], (pi / NST - 1) & 1, abort_flag))
                fetch();
    }
    if (warp == 4)
        return;

    grid_dep_wait();  // q~ comes from the prep kernel
    int gp = 0;
    // A wait that gives up sets the abort flag, after which every later one gives
    // up soon: the loops run on (the barriers keep their counts) and the CTA
    // reports the error at its end.
    bool ok = true;
    // wait for a stage and zero its rows past the segment's last token (their P
    // is 0; 0 * NaN must not arise; the barriers in stage() order the writes)
    auto stage_wait = [&](int st, int ntok, int width) {
        ok = mbar_wait(&full[st], (gp / NST) & 1, abort_flag) && ok;
        if (ntok < kTok) {
            unsigned char *t = sm + Ly::STG + st * Ly::CST;
            for (int i = tid; i < (kTok - ntok) * (width / 8); i += kConsumerThreads) {
                const int r = ntok + i / (width / 8), ch = i % (width / 8);
                *reinterpret_cast<uint4 *>(t + (ch / 8) * 8192 + r * 128 + (((ch % 8) ^ (r & 7)) << 4)) =
                    make_uint4(0u, 0u, 0u, 0u);
            }
            fence_proxy_async_smem();  // these writes precede the stage's next TMA fill
        }
    };
    auto run = [&](auto &rows, const Segment &it, int tokens, int width, uint32_t voff) {
        for (int p = 0; p < it.npg; ++p, ++gp) {
            const int st = gp % NST, ntok = min(kTok, tokens - p * kTok);
            stage_wait(st, ntok, width);
            const uint32_t t = sbase + Ly::STG + st * Ly::CST;
            rows.stage(t, t + voff, sm + Ly::P, red, ntok, a.c2, it.latent && p % kPagesPerSplit == 0, warp, lane,
                       [&] {
                if (!Ly::kProducer && tid == 0 && gp > 0 && pit.npg >= 0)
                    fetch();  // into the stage of gp - 1
            });
            if constexpr (Ly::kProducer) {
                __syncwarp();
                if (lane == 0)
                    mbar_arrive(&empty[st]);
            }
        }
    };
    for (int k = k0; k < k1;) {
        const Segment it = segment_of(k);
        k += it.units;
        if (it.npg == 0)
            continue;
        const int L = len_of(it.b), Lg = L > a.w ? L - a.w : 0, nwin = min(L, a.w);
        if (it.latent) {
            Rows<DL, MT> rows;
            rows.start(a.qt + (size_t)it.b * a.Hq * DL, a.Hq, warp, lane);
            run(rows, it, Lg - it.part * kSplitTok, DL, 0);
            // records of one (b, h) are consecutive over the units
            auto rec = [&](int row) {
                return a.rec_lat + (((size_t)it.b * a.Hq + row) * a.nspl + it.part) * (DL + 2);
            };
            rows.finish(red, a.Hq, warp, lane, rec);
            for (int i = tid; i < (it.units - 1) * a.Hq; i += kConsumerThreads)  // the other units' slots: empty
                *reinterpret_cast<float2 *>(rec(i % a.Hq) + (i / a.Hq + 1) * (DL + 2) + DL) =
                    make_float2(-INFINITY, 0.f);
        } else {
            // K block of a stage at +0, V block at +8192
            auto window = [&](auto &rows) {
                rows.start(static_cast<const bf16 *>(a.q) + ((size_t)it.b * a.Hq + it.part * a.G) * 64, a.G, warp,
                           lane);
                run(rows, it, nwin, 128, 8192);
                rows.finish(red, a.G, warp, lane, [&](int row) {
                    return a.rec_win + ((size_t)it.b * a.Hq + it.part * a.G + row) * 66;
                });
            };
            if constexpr (MT > 1) {
                if (a.G > 16) {
                    Rows<64, MT> rows;
                    window(rows);
                    continue;
                }
            }
            Rows<64, 1> rows;
            window(rows);
        }
    }
    if (!ok && lane == 0)
        report(a.status, DAR_ERR_DEVICE);
}

// ---------------------------------------------------------------- decode: merge

// A load the compiler keeps in place (a batch of them is issued before the first
// use; with the registers for it, see the launch bounds, the merge of 31 records of
// 32 heads took 10 us, 25 without).  Zeros, and no load, when !on.
__device__ __forceinline__ float2 ld_early_f2(const float *p, bool on)
{
    float2 r;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %3, 0;\n\t"
        "mov.b32 %0, 0;\n\t"
        "mov.b32 %1, 0;\n\t"
        "@p ld.global.v2.f32 {%0, %1}, [%2];\n\t}"
        : "=&f"(r.x), "=&f"(r.y)
        : "l"(p), "r"((uint32_t)on));
    return r;
}

// Block (g, a few rows of KV head g): A_V^g staged in shared memory by one bulk
// copy (before the dependency wait: it does not come from the main kernel),
// then one warp per row: combine the window record and the sequence's latent splits
// (log-sum-exp, one split per lane), lift the latent sum with A_V, divide.
template <int DL>
__global__ void __launch_bounds__(kRowThreads, 2) latent_merge_kernel(Args a)
{
    extern __shared__ __align__(16) float msm[];
    float *avs = msm;                  // [DL][64]
    float *olat = avs + DL * 64;       // [warps][DL]
    uint64_t *bar = reinterpret_cast<uint64_t *>(olat + kRowsPerBlock * DL);
    const int g = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (!stage_matrix(avs, a.Av + (size_t)g * DL * 64, DL * 64 * 4, bar, a.status))
        return;
    grid_dep_wait();  // the main kernel's records
    const int nrows = a.B * a.G;
    if (const int r = blockIdx.y * (blockDim.x >> 5) + warp; r < nrows) {
        const int b = r / a.G, h = g * a.G + r % a.G, row = b * a.Hq + h;
        int L = __ldg(a.seq_lens + b);
        if (L < 0 || L > a.maxp * kTok)
            L = 0;  // reported by the main kernel; the output is undefined then
        const int Lg = L > a.w ? L - a.w : 0;
        const int ns = (Lg + kSplitTok - 1) / kSplitTok;
        const float *rw = a.rec_win + (size_t)row * 66;
        const float *rl0 = a.rec_lat + (size_t)row * a.nspl * (DL + 2);  // this row's splits, consecutive
        const float mw = L > 0 ? rw[64] : -INFINITY;
        // the splits' maxima and sums, one slot per lane (32 at a time); the
        // weighted sum of their O with every load of a batch issued before it is used
        float M = mw;
        for (int s2 = lane; s2 < ns; s2 += 32)
            M = fmaxf(M, rl0[s2 * (DL + 2) + DL]);
#pragma unroll
        for (int o = 16; o; o >>= 1)
            M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
        float l = 0.f;
        float acc[DL / 32];
#pragma unroll
        for (int e = 0; e < DL / 32; ++e)
            acc[e] = 0.f;
        for (int s0 = 0; s0 < ns; s0 += 32) {
            float f = 0.f;
            if (s0 + lane < ns) {
                const float *rl = rl0 + (s0 + lane) * (DL + 2);
                f = ex2_approx(rl[DL] - M);
                l += f * rl[DL + 1];
            }
            // slots with a weight (empty ones hold no O), in batches of 8
            for (unsigned left = __ballot_sync(0xffffffffu, f != 0.f); left;) {
                const float *src[8];
                bool on[8];
                float fj[8];
                float2 x[8][DL / 64];
#pragma unroll
                for (int j = 0; j < 8; ++j) {  // past the last slot: 0 times 0 (a record may hold an infinity)
                    on[j] = left != 0u;
                    const int at = on[j] ? __ffs(left) - 1 : 0;
                    const float fa = __shfl_sync(0xffffffffu, f, at);
                    fj[j] = on[j] ? fa : 0.f;
                    src[j] = rl0 + (s0 + at) * (DL + 2) + 2 * lane;
                    left &= left - 1;
                }
#pragma unroll
                for (int j = 0; j < 8; ++j)
#pragma unroll
                    for (int e = 0; e < DL / 64; ++e)
                        x[j][e] = ld_early_f2(src[j] + 64 * e, on[j]);
#pragma unroll
                for (int j = 0; j < 8; ++j)
#pragma unroll
                    for (int e = 0; e < DL / 64; ++e) {
                        acc[2 * e] = fmaf(fj[j], x[j][e].x, acc[2 * e]);
                        acc[2 * e + 1] = fmaf(fj[j], x[j][e].y, acc[2 * e + 1]);
                    }
            }
        }
#pragma unroll
        for (int o = 16; o; o >>= 1)
            l += __shfl_xor_sync(0xffffffffu, l, o);
        const float fw = L > 0 ? ex2_approx(mw - M) : 0.f;
        if (L > 0)
            l += fw * rw[65];
#pragma unroll
        for (int e = 0; e < DL / 64; ++e)  // columns 2 lane + 64 e, + 1
            *reinterpret_cast<float2 *>(olat + warp * DL + 2 * lane + 64 * e) = make_float2(acc[2 * e], acc[2 * e + 1]);
        __syncwarp();
        float o0 = L > 0 ? fw * rw[lane] : 0.f, o1 = L > 0 ? fw * rw[lane + 32] : 0.f;
#pragma unroll 16
        for (int c = 0; c < DL; ++c) {
            const float x = olat[warp * DL + c];
            o0 = fmaf(x, avs[c * 64 + lane], o0);
            o1 = fmaf(x, avs[c * 64 + lane + 32], o1);
        }
        const float inv = l > 0.f ? 1.f / l : 0.f;
        bf16 *out = static_cast<bf16 *>(a.out) + (size_t)row * 64;
        out[lane] = __float2bfloat16_rn(o0 * inv);
        out[lane + 32] = __float2bfloat16_rn(o1 * inv);
        __syncwarp();
    }
}

// ---------------------------------------------------------------- host side

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

static bool encode_2d(CUtensorMap *tm, const void *base, unsigned long long rows, int cols)
{
    EncodeTiledFn enc = encode_fn();
    if (!enc)
        return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
    const cuuint32_t box[2] = {64, (cuuint32_t)kTok};
    const cuuint32_t estr[2] = {1, 1};
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int DL, int MT>
static cudaError_t decode_t(const Args &a, const void *pool_c, const void *win_k, const void *win_v, cudaStream_t s)
{
    using Ly = MainLayout<DL, MT>;
    const size_t smem = 1024 + Ly::TOTAL;
    constexpr size_t prep_smem = (size_t)64 * DL * sizeof(float) + 16;
    constexpr size_t merge_smem = ((size_t)DL * 64 + kRowsPerBlock * DL) * sizeof(float) + 16;
    static PerDeviceOnce once;  // records the SM count
    int sms = 0;
    cudaError_t e = per_device_once(
        once,
        [&](int dev) {
            cudaError_t e2 = cudaFuncSetAttribute(latent_main_kernel<DL, MT>,
                                                  cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e2 == cudaSuccess)
                e2 = cudaFuncSetAttribute(latent_prep_kernel<DL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)prep_smem);
            if (e2 == cudaSuccess)
                e2 = cudaFuncSetAttribute(latent_merge_kernel<DL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)merge_smem);
            int n = 0;
            if (e2 == cudaSuccess)
                e2 = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
            once.value[dev] = n;
            return e2;
        },
        &sms);
    if (e != cudaSuccess)
        return e;
    CUtensorMap tm[3];
    if (!encode_2d(&tm[0], pool_c, (unsigned long long)a.num_pages * kTok, DL) ||
        !encode_2d(&tm[1], win_k, (unsigned long long)a.B * a.Hkv * a.w, 64) ||
        !encode_2d(&tm[2], win_v, (unsigned long long)a.B * a.Hkv * a.w, 64))
        return cudaErrorInvalidValue;
    // prep starts after all earlier work on the stream; main and merge are
    // launched programmatically (each waits in-kernel for what it reads)
    // prep and merge: few rows are spread over the chip, many share a staged
    // matrix (4 sequences, 4 KV heads, G 4: 16.5 us with 2 rows a block, 17.7 with
    // 8; 64 sequences, 8 KV heads, G 4: 4 rows a block cost 3 us more than 8).  The
    // merge takes two blocks per SM before rows share one, except at d_lat 64, where
    // its small blocks find room beside the main kernel's; the prep, beside which the
    // main kernel has to start, one (calls, us, merge at one / two blocks per SM, then
    // both at two: 32 sequences of 4096 tokens, 12 heads, d_lat 192 24.5 / 21.9 / 21.9;
    // 61 of 340 to 484, 12, 256 23.6 / 22.4 / 22.7; 10 of 4000 to 8000, 32, 256 40.4 /
    // 38.2 / 40.5; 64 of 300 to 900, 8, 64 11.7 / 12.8 / 12.4; 64 of 16384, 8, 64 47 / 51).
    const auto rows_for = [&](int blocks) {
        int rows = 2;
        while (rows < kRowsPerBlock && a.Hkv * ((a.B * a.G + rows - 1) / rows) > blocks)
            rows *= 2;
        return rows;
    };
    int rows = rows_for(sms);
    latent_prep_kernel<DL><<<dim3(a.Hkv, (a.B * a.G + rows - 1) / rows), 32 * rows, prep_smem, s>>>(a);
    cudaLaunchAttribute pdl[1];
    pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = s;
    cfg.attrs = pdl;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3(2 * (sms > 0 ? sms : 1));  // persistent: two CTAs per SM
    cfg.blockDim = dim3(Ly::THREADS);
    cfg.dynamicSmemBytes = smem;
    e = cudaLaunchKernelEx(&cfg, latent_main_kernel<DL, MT>, tm[0], tm[1], tm[2], a);
    if (e != cudaSuccess)
        return e;
    rows = rows_for(DL > 64 ? 2 * sms : sms);
    cfg.gridDim = dim3(a.Hkv, (a.B * a.G + rows - 1) / rows);
    cfg.blockDim = dim3(32 * rows);
    cfg.dynamicSmemBytes = merge_smem;
    e = cudaLaunchKernelEx(&cfg, latent_merge_kernel<DL>, a);
    if (e != cudaSuccess)
        return e;
    return cudaGetLastError();
}

template <int DL>
static cudaError_t decode_dl(const Args &a, const void *pool_c, const void *win_k, const void *win_v, cudaStream_t s)
{
    return a.Hq <= 16 ? decode_t<DL, 1>(a, pool_c, win_k, win_v, s) : decode_t<DL, 2>(a, pool_c, win_k, win_v, s);
}

// The tiled append's launch.
template <int TPT, int CPT>
static cudaError_t append_tiled(const AppendArgs &a, cudaStream_t s)
{
    using T = Tile<TPT, CPT>;
    static PerDeviceOnce once;
    const cudaError_t e = per_device_once(once, [](int) {
        return cudaFuncSetAttribute(latent_append_tiled_kernel<TPT, CPT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    T::TOTAL);
    });
    if (e != cudaSuccess)
        return e;
    const long long tiles = ((long long)a.B * a.n + T::ROWS - 1) / T::ROWS;
    latent_append_tiled_kernel<TPT, CPT><<<(unsigned)(tiles * (a.DL / T::COLS)), kTileThreads, T::TOTAL, s>>>(a);
    return cudaGetLastError();
}

// The tile by the number of CTAs it makes: the smallest that does not fill the
// chip several times over (small ones have the shorter chain loop, big ones read
// less shared memory per product).  Measured, us, rows x D x DL, tiles of
// 4 / 8 / 16 rows x 32 columns and 32 / 64 rows x 64 columns:
//     8 x 2048 x 256   22.6   25.4   30.0   48.0   72.1
//    64 x 2048 x 256   23.0   25.4   30.8   51.3   77.8
//   600 x  768 x 192   25.2   17.7   18.8   25.1   36.9
//   520 x 2048 x 256   55.5   44.5   38.1   51.3   78.0
//  2000 x 1024 x 256   84.5   59.7   51.6   40.6   43.9
//  8000 x 2048 x 256    571    386    312    187    169
static cudaError_t append_tiled_any(const AppendArgs &a, cudaStream_t s)
{
    const auto ctas = [&](int rows, int cols) {
        return ((long long)a.B * a.n + rows - 1) / rows * (a.DL / cols);
    };
    if (ctas(4, 32) <= kSms)
        return append_tiled<1, 1>(a, s);
    if (ctas(8, 32) <= kSms * 3)
        return append_tiled<2, 1>(a, s);
    if (ctas(16, 32) <= kSms * 3)
        return append_tiled<4, 1>(a, s);
    if (ctas(32, 64) <= kSms * 4)
        return append_tiled<4, 4>(a, s);
    return append_tiled<8, 4>(a, s);
}

// Advances the lengths once the append has finished.
static cudaError_t append_lens(const AppendArgs &a, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((a.B + 255) / 256);
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, latent_lens_kernel, a);
}

}  // namespace lat

size_t latent_decode_workspace_bytes(int B, int Hq, int DL, int maxp)
{
    auto al = [](size_t x) { return (x + 255) & ~size_t(255); };
    const size_t nspl = (size_t)(maxp + lat::kPagesPerSplit - 1) / lat::kPagesPerSplit;
    return al((size_t)B * Hq * DL * 2) + al((size_t)B * nspl * Hq * (DL + 2) * 4) + al((size_t)B * Hq * 66 * 4);
}

cudaError_t launch_latent_decode(const LatentDecodeArgs &x, void *workspace, cudaStream_t s)
{
    if (x.B == 0)
        return cudaSuccess;
    auto al = [](size_t v) { return (v + 255) & ~size_t(255); };
    lat::Args a;
    a.q = x.q;
    a.out = x.out;
    a.win_k = x.win_k;
    a.win_v = x.win_v;
    a.block_table = x.block_table;
    a.seq_lens = x.seq_lens;
    a.status = x.status;
    a.Ak = x.Ak;
    a.Av = x.Av;
    a.B = x.B;
    a.Hq = x.Hq;
    a.Hkv = x.Hkv;
    a.G = x.Hq / x.Hkv;
    a.w = x.w;
    a.maxp = x.maxp;
    a.num_pages = x.num_pages;
    a.nspl = (x.maxp + lat::kPagesPerSplit - 1) / lat::kPagesPerSplit;
    a.c2 = x.scale * 1.4426950408889634f;
    char *p = static_cast<char *>(workspace);
    a.qt = reinterpret_cast<bf16 *>(p);
    p += al((size_t)x.B * x.Hq * x.DL * 2);
    a.rec_lat = reinterpret_cast<float *>(p);
    p += al((size_t)x.B * a.nspl * x.Hq * (x.DL + 2) * 4);
    a.rec_win = reinterpret_cast<float *>(p);
    switch (x.DL) {
    case 64: return lat::decode_dl<64>(a, x.pool_c, x.win_k, x.win_v, s);
    case 128: return lat::decode_dl<128>(a, x.pool_c, x.win_k, x.win_v, s);
    case 192: return lat::decode_dl<192>(a, x.pool_c, x.win_k, x.win_v, s);
    case 256: return lat::decode_dl<256>(a, x.pool_c, x.win_k, x.win_v, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_latent_append(const LatentAppendArgs &x, cudaStream_t s)
{
    if (x.B == 0 || x.n == 0)
        return cudaSuccess;
    lat::AppendArgs a;
    a.h = x.h;
    a.k_new = x.k_new;
    a.v_new = x.v_new;
    a.Wdown = x.Wdown;
    a.win_k = x.win_k;
    a.win_v = x.win_v;
    a.pool_c = x.pool_c;
    a.block_table = x.block_table;
    a.n_per_seq = x.n_per_seq;
    a.seq_lens = x.seq_lens;
    a.status = x.status;
    a.B = x.B;
    a.Hkv = x.Hkv;
    a.n = x.n;
    a.D = x.D;
    a.DL = x.DL;
    a.w = x.w;
    a.maxp = x.maxp;
    a.num_pages = x.num_pages;
    cudaError_t e;
    if (x.D % 8 == 0 && ((long long)x.B * x.n + 3) / 4 * (x.DL / 32) <= 0x7fffffffLL) {
        e = lat::append_tiled_any(a, s);
        return e != cudaSuccess ? e : lat::append_lens(a, s);
    }
    const size_t smem = (size_t)lat::kAppTok * x.D * sizeof(float);
    static PerDeviceOnce once;
    e = per_device_once(once, [&](int) {
        return cudaFuncSetAttribute(lat::latent_append_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)(lat::kAppTok * 8192 * sizeof(float)));
    });
    if (e != cudaSuccess)
        return e;
    lat::latent_append_kernel<<<dim3((x.n + lat::kAppTok - 1) / lat::kAppTok, x.B), 256, smem, s>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess)
        return e;
    return lat::append_lens(a, s);
}

cudaError_t launch_latent_absorb(const float *Wup, const float *WK, const float *WV, float *Ak, float *Av, int Hkv,
                                 int D, int DL, cudaStream_t s)
{
    lat::latent_absorb_kernel<<<dim3(DL, Hkv), 64, 0, s>>>(Wup, WK, WV, Ak, Av, D, DL);
    return cudaGetLastError();
}

}  // namespace dar
