// Warp-specialised attention-logit kernel for 1- to 4-bit codes (Remark 6.4): one persistent CTA of 20 (or 24)
// warps per SM in which loading, code expansion, the MMAs and the output run concurrently on
// different tiles.
//
//   warp 0        bulk-copies each 128-token tile (codes, norms, factor rows) and each block's right
//                 vectors from global memory into a ring of shared-memory stages
//   warps 2-3     build the query-side operands: W = Pi q once per head, Aq = q V^T once per block
//   warps 4-15    three groups of four: expand a tile's codes to fp16 centroids (byte permutes) and
//                 store them, the factor entries and the row norm into one of four tensor-memory
//                 buffers, one token per thread
//   warp 1        issues the nine MMAs of a tile (A from tensor memory, B from shared memory)
//   warps 16 on   read the accumulators back, apply norm and scale, write the logits (four warps for eight queries, or two
//                 such groups)
//
// The high and the low fp16 plane of a query-side operand are stacked along N (columns g and NQ + g of one
// accumulator).  A pass serves NQ = 8 query vectors, or 16 when there are more than eight: an MMA with A in tensor
// memory takes 50 cycles for N = 16 and for N = 32 alike, and expansion does not depend on N, so a second pass would
// cost as much as the first.
//
// A tile takes some 900 cycles (16 queries against 4096 blocks of two bits: 134 us over and over, 146 with inputs from memory that the L2
// cache does not hold; 186 us with two expander groups, the issuing lane alone in its branch, and one sum at a time in the operand builder, which then
// took longer for a block than its eight tiles).  What is left is the schedulers' issue slots: an expander warp has some
// 400 instructions per tile on each of them, an output warp 110.
#include <algorithm>

#include "eosq_common.cuh"
#include "eosq_sm100.cuh"
#include "eosq_expand.cuh"

namespace eosq {

using namespace sm100;

constexpr int TC_ERR_SCORES_WS_TIMEOUT = 8;

constexpr int WS_STAGES = 5;               // shared-memory stages of WS_TPS tiles each, or as many as fit
constexpr int WS_TPS = 4;                  // tiles per stage: few large copies keep the copy engine's queue short
constexpr int WS_BUFS = 4;                 // tensor-memory buffers, three with sixteen queries
constexpr int WS_EXP_GROUPS = 3;           // a tile takes a group 1 500 to 2 400 cycles, mostly latencies
constexpr int WS_PMAX = 12;                // factor rows staged per tile (rank <= pilot k = 11)
// a stage holds 512 tokens: codes (16 BITS bytes per token), norms, 2 boxes of 12 x 256 factors
constexpr uint32_t WS_ST_CODES = 0;
constexpr uint32_t WS_ST_PBOX = WS_PMAX * 512;
template <int BITS, int NQ> struct WsLayout {
    static constexpr uint32_t ROW = 16 * BITS;                              // code bytes per token
    static constexpr uint32_t ST_NORMS = 512 * ROW, ST_P = ST_NORMS + 1024;
    static constexpr uint32_t STAGE_BYTES = ST_P + 2 * WS_ST_PBOX;         // 29696 (2 bits), 37888 (3 bits)
    static constexpr uint32_t B1 = NQ * 512, B2 = NQ * 256;                // W: hi rows 0 .. NQ - 1, then lo rows, two K boxes; Aq: one
    static constexpr uint32_t REST = 2 * B1 + 2 * B2 + 2 * 4096 + 2 * NQ * D * 4 + 1024;
    static constexpr int FIT = static_cast<int>((226 * 1024 - REST) / STAGE_BYTES), STAGES = FIT < WS_STAGES ? FIT : WS_STAGES;
    static_assert(STAGES >= 3, "the loader runs ahead");
    static constexpr uint32_t OFF_B1 = STAGES * STAGE_BYTES;               // 2 x W
    static constexpr uint32_t OFF_B2 = OFF_B1 + 2 * B1;                    // 2 x Aq
    static constexpr uint32_t OFF_V = OFF_B2 + 2 * B2;                     // 2 x 4096: right vectors (fp16)
    static constexpr uint32_t OFF_Q = OFF_V + 2 * 4096;                    // 2 x (NQ x 128) fp32 queries, by head parity
    static constexpr uint32_t SMEM_BYTES = OFF_Q + 2 * NQ * D * 4 + 1024;
    // tensor memory, per buffer: A 0-63, P 64-71, rho 72, D1 80.., D2
    static constexpr int EPI_GROUPS = NQ / 8, EPI_FIRST = 4 + 4 * WS_EXP_GROUPS, THREADS = 32 * (EPI_FIRST + 4 * EPI_GROUPS);   // (one group of four output warps takes 2 000 cycles per tile for 16 queries)
    static constexpr int BUFS = (NQ == 8) ? WS_BUFS : WS_BUFS - 1;
    static constexpr uint32_t COL_D1 = 80, COL_D2 = 80 + 2 * NQ, BUF_COLS = 80 + 4 * NQ;
    static_assert(BUFS * BUF_COLS <= 512, "the buffers fit tensor memory");
};
constexpr uint32_t WS_TMEM_COLS = 512;
constexpr uint32_t WS_COL_P = 64, WS_COL_RHO = 72;
constexpr float WS_QSCALE = 256.0f;

struct WsArgs {
    eosq_cache_t cache;
    int bph, head_stride, heads;   // blocks per head, block stride between heads, heads
    int n, G, g0;
    int local_w;           // W is made by the CTAs themselves (each touches at most two heads)
    const float *pi_t;
    float scale, inv_code;
    uint32_t lo_tab[4], hi_tab[4];   // low / high bytes of the fp16 centroids times kappa (level k in byte k)
    uint32_t pair_tab[2];            // two bits: the centroids, levels 0, 1 and 2, 3
    const uint8_t *wimg;   // per head: the image of the operand W = Pi q (made by scores_w_kernel)
    const __half *q;
    float *scores;
    int *err;
};

__device__ __forceinline__ void ws_bulk_load(void *smem_dst, const void *gsrc, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :
                 : "r"(smem_u32(smem_dst)), "l"(reinterpret_cast<uint64_t>(gsrc)), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// Byte offset of element (row, k) of a K-major, 128-byte-swizzled operand with 2 NQ rows per 64-wide K box.
template <int NQ>
__device__ __forceinline__ uint32_t ws_b_offset(int row, int k) {
    const int box = k >> 6, kk = k & 63;
    return box * (NQ * 256) + row * 128 + ((((kk >> 3) ^ (row & 7)) << 4) | ((kk & 7) << 1));
}

// Where coordinate k of a row stands along K: the expansion of two-bit codes has an order of its own.
template <int BITS>
__device__ __forceinline__ int ws_place(int k) { return (BITS == 2) ? (k & ~15) | expand_place(k & 15) : k; }

template <int NQ>
__device__ __forceinline__ void ws_split_store(uint8_t *plane, int g, int k, float v) {
    const __half hi = __float2half_rn(v), lo = __float2half_rn(v - __half2float(hi));
    *reinterpret_cast<__half *>(plane + ws_b_offset<NQ>(g, k)) = hi;
    *reinterpret_cast<__half *>(plane + ws_b_offset<NQ>(NQ + g, k)) = lo;
}

// Barrier of the 64 threads of the operand builder that also tells each of them whether any brings
// `failed` (the outcome of a bounded wait, which ends per thread).
__device__ __forceinline__ bool ws_builder_any(bool failed) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "bar.red.or.pred q, 2, 64, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(failed ? 1u : 0u)
        : "memory");
    return r != 0;
}

struct WsBarriers {
    uint64_t st_full[WS_STAGES], st_empty[WS_STAGES];
    uint64_t a_full[WS_BUFS], d_full[WS_BUFS], d_empty[WS_BUFS];
    uint64_t blk_full[2], blk_empty[2], b2_full[2], b2_empty[2], b1_full[2], b1_empty[2];
    uint64_t drain;
};

bool make_factor_tensor_map(const void *P, int64_t nb, int n, int rows, CUtensorMap *out);

// W = Pi q for the (at most NQ) query vectors g0.. of every head, times 2^8, split into a high and a low fp16
// plane and laid out as the score kernel's B operand (rows g and NQ + g of a K-major, 128-byte-swizzled tile of
// 2 NQ rows x 128): one image per head, which the score kernel fetches with one bulk copy.
template <int BITS, int NQ>
__global__ void __launch_bounds__(D) scores_w_kernel(const float *__restrict__ pi_t, const __half *q, int G, int g0,
                                                     uint8_t *wimg) {
    __shared__ float qs[NQ][D];
    const int c = threadIdx.x, hd = blockIdx.x;
    const int gcount = min(NQ, G - g0);
    pdl_wait();
    pdl_trigger();
    for (int g = 0; g < NQ; ++g) qs[g][c] = (g < gcount) ? __half2float(q[(static_cast<long long>(hd) * G + g0 + g) * D + c]) : 0.0f;
    __syncthreads();
    float w[NQ];
#pragma unroll
    for (int g = 0; g < NQ; ++g) w[g] = 0.0f;
#pragma unroll 1
    for (int j0 = 0; j0 < D; j0 += 32) {
        float pv[32];
#pragma unroll
        for (int jj = 0; jj < 32; ++jj) pv[jj] = __ldg(pi_t + (j0 + jj) * D + c);   // 32 loads in flight: the kernel is all L2 latency
#pragma unroll
        for (int jj = 0; jj < 32; ++jj) {
#pragma unroll
            for (int g = 0; g < NQ; ++g) w[g] = fmaf(pv[jj], qs[g][j0 + jj], w[g]);
        }
    }
    uint8_t *img = wimg + static_cast<size_t>(hd) * WsLayout<1, NQ>::B1;
#pragma unroll
    for (int g = 0; g < NQ; ++g) ws_split_store<NQ>(img, g, ws_place<BITS>(c), w[g] * WS_QSCALE);
}

template <int BITS, int NQ>
__global__ void __launch_bounds__(WsLayout<BITS, NQ>::THREADS, 1) scores_ws_kernel(const WsArgs a, const __grid_constant__ CUtensorMap pmap4,
                                                                  const __grid_constant__ CUtensorMap pmap8,
                                                                  const __grid_constant__ CUtensorMap pmap12) {
    using L = WsLayout<BITS, NQ>;
    constexpr int WS_NQ = NQ, WS_THREADS = L::THREADS;
    extern __shared__ uint8_t ws_smem_raw[];
    __shared__ __align__(8) WsBarriers bars;
    __shared__ uint32_t tmem_base_s;
    __shared__ int st_rank[WS_STAGES];
    __shared__ volatile int abort_flag;

    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(ws_smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n = a.n, tiles = (n + 127) / 128;
    const int gcount = min(WS_NQ, a.G - a.g0);

    if (tid == 0) {
        for (int s = 0; s < WS_STAGES; ++s) {
            mbar_init(&bars.st_full[s], 1);
            mbar_init(&bars.st_empty[s], 4 * WS_EXP_GROUPS);   // one arrival per expander warp
        }
        for (int b = 0; b < WS_BUFS; ++b) {
            mbar_init(&bars.a_full[b], 4);             // one arrival per warp: 128 arrivals on one barrier serialise
            mbar_init(&bars.d_full[b], 1);
            mbar_init(&bars.d_empty[b], 4 * L::EPI_GROUPS);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&bars.blk_full[b], 1);
            mbar_init(&bars.blk_empty[b], 1);
            mbar_init(&bars.b2_full[b], 1);
            mbar_init(&bars.b2_empty[b], 1);
            mbar_init(&bars.b1_full[b], 1);
            mbar_init(&bars.b1_empty[b], 1);
        }
        abort_flag = 0;
        fence_mbar_init();
    }
    if (tid == 64) {
        mbar_init(&bars.drain, 1);
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(&tmem_base_s, WS_TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem0 = warp_uniform(tmem_base_s);
    const bool issuer = elect_one();   // of warp 1: the lane that issues

    // (the rotation was uploaded before any kernel of the stream)
    const int c = tid & (D - 1), quarter = (tid >> 7) & 3;   // of Pi, see below
    float pv[32];
    if (a.local_w && tid < 4 * D) {
#pragma unroll
        for (int jj = 0; jj < 32; ++jj) pv[jj] = __ldg(a.pi_t + (32 * quarter + jj) * D + c);
    }
    pdl_wait();
    // Ranks are clamped to the rows a stage holds, as in decode; the library never stores more than the pilot k = 11.
    auto rank_of = [&](long long blk) { return max(0, min(a.cache.rank[blk], WS_PMAX)); };
    // contiguous range of (head, block) items of this CTA; every role walks it in the same order
    const int items = a.heads * a.bph;
    const int ipc = (items + gridDim.x - 1) / gridDim.x;
    const int it0 = min(items, ipc * static_cast<int>(blockIdx.x)), it1 = min(items, it0 + ipc);

    // W of the CTA's own heads (two at most), by everybody before the roles part: thread (c, quarter) takes row c of Pi
    // over a quarter of the queries' coordinates.  Some 4 000 cycles, where a kernel in front costs 4 us of a call
    // that takes 14 in all.
    if (a.local_w && it0 < it1) {
        const int head0 = it0 / a.bph, heads_here = (it1 - 1) / a.bph - head0 + 1;
        float *qs = reinterpret_cast<float *>(base + L::OFF_Q), *parts = reinterpret_cast<float *>(base);   // (the stages are still empty)
        // (code that runs once is kept short: what costs here is fetching it)
        if ((reinterpret_cast<uintptr_t>(a.q) & 15u) == 0) {
#pragma unroll 1
            for (int e = tid; e < heads_here * NQ * D / 8; e += WS_THREADS) {
                const int hx = e / (NQ * D / 8), g = (e / (D / 8)) % NQ, j = e % (D / 8);
                uint4 v = make_uint4(0u, 0u, 0u, 0u);
                if (g < gcount) v = *reinterpret_cast<const uint4 *>(a.q + (static_cast<long long>(head0 + hx) * a.G + a.g0 + g) * D + 8 * j);
                const float2 f0 = __half22float2(*reinterpret_cast<const __half2 *>(&v.x)), f1 = __half22float2(*reinterpret_cast<const __half2 *>(&v.y));
                const float2 f2 = __half22float2(*reinterpret_cast<const __half2 *>(&v.z)), f3 = __half22float2(*reinterpret_cast<const __half2 *>(&v.w));
                float4 *dst = reinterpret_cast<float4 *>(qs + 8 * e);
                dst[0] = make_float4(f0.x, f0.y, f1.x, f1.y);
                dst[1] = make_float4(f2.x, f2.y, f3.x, f3.y);
            }
        } else {
#pragma unroll 1
            for (int e = tid; e < heads_here * NQ * D; e += WS_THREADS) {
                const int hx = e / (NQ * D), g = (e / D) % NQ;
                qs[e] = (g < gcount) ? __half2float(a.q[(static_cast<long long>(head0 + hx) * a.G + a.g0 + g) * D + (e % D)]) : 0.0f;
            }
        }
        __syncthreads();
        if (tid < 4 * D) {
#pragma unroll 1
            for (int hx = 0; hx < heads_here; ++hx) {
#pragma unroll 1
                for (int g = 0; g < gcount; g += 4) {   // four queries at a time (of NQ, a multiple of it), sums of sixteen products side by side
                    const float *q = qs + (hx * NQ + g) * D + 32 * quarter;
                    float w[4][2] = {};
#pragma unroll
                    for (int j = 0; j < 32; j += 4) {
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float4 v = *reinterpret_cast<const float4 *>(q + e * D + j);
                            w[e][0] = fmaf(pv[j + 2], v.z, fmaf(pv[j], v.x, w[e][0]));
                            w[e][1] = fmaf(pv[j + 3], v.w, fmaf(pv[j + 1], v.y, w[e][1]));
                        }
                    }
#pragma unroll
                    for (int e = 0; e < 4; ++e) parts[((hx * NQ + g + e) * 4 + quarter) * D + c] = w[e][0] + w[e][1];
                }
            }
        }
        __syncthreads();
#pragma unroll 1
        for (int e = tid; e < heads_here * NQ * D; e += WS_THREADS) {
            const int hx = e / (NQ * D), g = (e / D) % NQ, k = e % D;
            const float *p = parts + (hx * NQ + g) * 4 * D + k;
            const float w = (g < gcount) ? (p[0] + p[D]) + (p[2 * D] + p[3 * D]) : 0.0f;
            ws_split_store<NQ>(base + L::OFF_B1 + hx * L::B1, g, ws_place<BITS>(k), w * WS_QSCALE);
        }
        fence_proxy_async_smem();
        __syncthreads();
    }

    // loads that this thread has announced: stages, blocks' vectors, heads' images (for the clean-up after a failed wait)
    uint32_t st_fills = 0, blk_fills = 0, b1_fills = 0;
    if (warp == 0) {
        // ---------------------------------------------------------------- loader
        // Lane 0 keeps the protocol (waits, expected byte counts) and fetches the factor rows of a tile with
        // one tensor copy (4, 8 or 12 rows, whichever covers the rank); lane 30 copies the codes, lane 31
        // the norms.
        if (it0 < it1) {
            uint32_t sseq = 0;
            int head = it0 / a.bph, jb = it0 - head * a.bph;
            int rank_next = rank_of(static_cast<long long>(head) * a.head_stride + jb);
            bool alive = true;
            for (int item = it0, bi = 0; item < it1 && alive; ++item, ++bi) {
                const long long gb = static_cast<long long>(head) * a.head_stride + jb;
                const int rank = rank_next;
                int nhead = head, njb = jb + 1;
                if (njb == a.bph) {
                    njb = 0;
                    nhead += 1;
                }
                if (item + 1 < it1) rank_next = rank_of(static_cast<long long>(nhead) * a.head_stride + njb);
                const int vb = bi & 1;
                if (lane == 0) {
                    alive = mbar_wait(&bars.blk_empty[vb], ((bi >> 1) & 1u) ^ 1u, &abort_flag);
                    if (alive) {
                        mbar_arrive_expect_tx(&bars.blk_full[vb], 4096);
                        blk_fills = bi + 1;
                        ws_bulk_load(base + L::OFF_V + vb * 4096, a.cache.V + gb * RMAX * D, 4096, &bars.blk_full[vb]);
                    }
                }
                alive = __shfl_sync(0xffffffffu, alive, 0);
                for (int tile = 0; tile < tiles && alive; tile += WS_TPS, ++sseq) {
                    const int stage = sseq % L::STAGES;
                    const int tok0 = tile * 128;
                    const uint32_t rows = static_cast<uint32_t>(min(128 * WS_TPS, n - tok0));
                    const uint32_t boxes = (rows + 255u) >> 8;
                    const int r4 = (rank + 3) >> 2;
                    if (lane == 0) {
                        alive = mbar_wait(&bars.st_empty[stage], ((sseq / L::STAGES) & 1u) ^ 1u, &abort_flag);
                        if (alive) {
                            st_rank[stage] = rank;
                            st_fills = sseq + 1;
                            mbar_arrive_expect_tx(&bars.st_full[stage], rows * (L::ROW + 2u) + boxes * static_cast<uint32_t>(r4) * 2048u);
                        }
                    }
                    alive = __shfl_sync(0xffffffffu, alive, 0);
                    if (!alive) break;
                    uint8_t *st = base + stage * L::STAGE_BYTES;
                    const size_t t0 = static_cast<size_t>(gb) * n + tok0;
                    if (lane < 2) {
                        if (r4 > 0 && static_cast<uint32_t>(lane) < boxes)
                            tma_load_3d(st + L::ST_P + lane * WS_ST_PBOX, r4 == 1 ? &pmap4 : (r4 == 2 ? &pmap8 : &pmap12), &bars.st_full[stage],
                                        tok0 + 256 * lane, 0, static_cast<int>(gb));
                    } else if (lane == 30)
                        ws_bulk_load(st + WS_ST_CODES, a.cache.codes + t0 * L::ROW, rows * L::ROW, &bars.st_full[stage]);
                    else if (lane == 31)
                        ws_bulk_load(st + L::ST_NORMS, a.cache.norms + t0, rows * 2, &bars.st_full[stage]);
                }
                head = nhead;
                jb = njb;
            }
        }
    } else if (warp == 1) {
        // ---------------------------------------------------------------- MMA issue
        if (it0 < it1) {
            constexpr uint32_t idesc = umma_idesc_f16(128, 2 * NQ, false, false);
            uint32_t seq = 0;
            int head = it0 / a.bph, jb = it0 - head * a.bph, hidx = -1, prev_head = -1;
            bool alive = true;
            for (int item = it0, bi = 0; item < it1 && alive; ++item, ++bi) {
                if (head != prev_head) {
                    hidx += 1;
                    prev_head = head;
                    if (!mbar_wait_warp(&bars.b1_full[hidx & 1], (hidx >> 1) & 1u, &abort_flag)) break;
                }
                const int vb = bi & 1, hb = hidx & 1;
                if (!mbar_wait_warp(&bars.b2_full[vb], (bi >> 1) & 1u, &abort_flag)) break;
                const uint32_t b1 = smem_u32(base + L::OFF_B1 + hb * L::B1), b2 = smem_u32(base + L::OFF_B2 + vb * L::B2);
                uint64_t bdesc[D / 16 + 1];
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks) bdesc[ks] = umma_desc_sw128(b1 + (ks >> 2) * (NQ * 256) + (ks & 3) * 32, 16, 1024);
                bdesc[D / 16] = umma_desc_sw128(b2, 16, 1024);
                for (int tile = 0; tile < tiles; ++tile, ++seq) {
                    const int buf = seq % L::BUFS;
                    const uint32_t u = (seq / L::BUFS) & 1u;
                    // a filled buffer is also a drained one: its expanders waited for the epilogue of its last use
                    if (!mbar_wait_warp(&bars.a_full[buf], u, &abort_flag)) {
                        alive = false;
                        break;
                    }
                    tc_fence_after_sync();
                    const uint32_t tb = tmem0 + buf * L::BUF_COLS;
                    if (issuer) {
#pragma unroll
                        for (int ks = 0; ks < D / 16; ++ks) umma_f16_ts(tb + L::COL_D1, tb + 8 * ks, bdesc[ks], idesc, ks ? 1u : 0u);
                        umma_f16_ts(tb + L::COL_D2, tb + WS_COL_P, bdesc[D / 16], idesc, 0u);
                        umma_commit(&bars.d_full[buf]);   // the one commit of a tile
                    }
                    __syncwarp();
                }
                if (!alive) break;
                if (issuer) umma_commit(&bars.b2_empty[vb]);
                int nhead = head, njb = jb + 1;
                if (njb == a.bph) {
                    njb = 0;
                    nhead += 1;
                }
                if (issuer && (nhead != head || item + 1 == it1)) umma_commit(&bars.b1_empty[hb]);
                __syncwarp();
                head = nhead;
                jb = njb;
            }
        }
    } else if (warp < 4) {
        // ---------------------------------------------------------------- operand builder (64 threads)
        const int bt = tid - 64;
        float *qs_all = reinterpret_cast<float *>(base + L::OFF_Q);
        // Head `hd`, the `hx`-th head of this CTA: its queries into shared memory (for the Aq products) and the
        // prepared image of W = Pi q, by one bulk copy, into the operand buffer of its parity.
        auto build_w = [&](int hd, int hx) -> bool {
            const int hb = hx & 1;
            float *qs = qs_all + hb * WS_NQ * D;
            // (a bounded wait ends per thread: its outcome is made common at the group's next barrier, so
            // that the 64 threads leave together and never one by one)
            const bool ok = mbar_wait(&bars.b1_empty[hb], ((hx >> 1) & 1u) ^ 1u, &abort_flag);
            if (a.local_w) {   // W and the queries are in place
                if (bt == 0 && ok) mbar_arrive(&bars.b1_full[hb]);
                return !ws_builder_any(!ok);
            }
            if (bt == 0 && ok) {
                mbar_arrive_expect_tx(&bars.b1_full[hb], L::B1);
                b1_fills = hx + 1;
                ws_bulk_load(base + L::OFF_B1 + hb * L::B1, a.wimg + static_cast<size_t>(hd) * L::B1, L::B1, &bars.b1_full[hb]);
            }
            for (int e = bt; e < WS_NQ * D; e += 64) {
                const int g = e / D;
                qs[e] = (g < gcount) ? __half2float(a.q[(static_cast<long long>(hd) * a.G + a.g0 + g) * D + (e % D)]) : 0.0f;
            }
            return !ws_builder_any(!ok);
        };
        int head = (it0 < it1) ? it0 / a.bph : 0, jb = it0 - head * a.bph, hidx = -1, prev_head = -1;
        bool first_of_head = false, fresh_q = false;
        constexpr int PARTS = 64 / NQ;
        const int qg = bt / PARTS, part = bt % PARTS;
        float qr[D / PARTS];
        int rank_next = (it0 < it1) ? rank_of(static_cast<long long>(head) * a.head_stride + jb) : 0;
        for (int item = it0, bi = 0; item < it1; ++item, ++bi) {
            if (head != prev_head) {
                hidx += 1;
                prev_head = head;
                first_of_head = fresh_q = true;
                if (hidx == 0 && !build_w(head, 0)) break;   // later heads were built one head ahead (below)
            }
            const float *qs = qs_all + (hidx & 1) * WS_NQ * D;
            const int vb = bi & 1;
            const int rank = rank_next;
            {   // the next block's rank is asked for now: a load on the critical path of every block costs over 1 000 cycles
                int nh = head, nj = jb + 1;
                if (nj == a.bph) {
                    nj = 0;
                    nh += 1;
                }
                if (item + 1 < it1) rank_next = rank_of(static_cast<long long>(nh) * a.head_stride + nj);
            }
            const bool ok = mbar_wait(&bars.blk_full[vb], (bi >> 1) & 1u, &abort_flag) &&
                            mbar_wait(&bars.b2_empty[vb], ((bi >> 1) & 1u) ^ 1u, &abort_flag);
            const __half *vs = reinterpret_cast<const __half *>(base + L::OFF_V + vb * 4096);
            uint8_t *b2 = base + L::OFF_B2 + vb * L::B2;
            // Aq[g][i] = q_g . zeta_i for i < rank, zero elsewhere.  PARTS lanes share a query, a slice of which each keeps in
            // registers for as long as the head lasts (16-byte chunks of the vector dealt round-robin), and read the block's
            // vectors once: the lanes of a warp ask for a few neighbouring chunks at a time.
            if (fresh_q) {
                fresh_q = false;
#pragma unroll
                for (int e = 0; e < D / PARTS; ++e) qr[e] = qs[qg * D + 8 * (part + PARTS * (e >> 3)) + (e & 7)];
            }
            // Four vectors at a time: these two warps compete with the other roles for every instruction, and a sum at a time is all latency.
            // Two sums each: none in fp32 runs over more than sixteen products (one of 32: an error of 1.32e-7 in the scores of
            // sixteen queries and one-bit codes, 1.18e-7 so).
#pragma unroll 1
            for (int i0 = 0; i0 < RMAX; i0 += 4) {
                float dot[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                if (i0 < rank) {
                    float sum[4][2] = {};
#pragma unroll
                    for (int ch = 0; ch < D / PARTS / 8; ++ch)
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const uint4 v = reinterpret_cast<const uint4 *>(vs + (i0 + u) * D)[part + PARTS * ch];
                            const uint32_t vw[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&vw[e]));
                                sum[u][0] = fmaf(qr[8 * ch + 2 * e], f.x, sum[u][0]);
                                sum[u][1] = fmaf(qr[8 * ch + 2 * e + 1], f.y, sum[u][1]);
                            }
                        }
#pragma unroll
                    for (int u = 0; u < 4; ++u) dot[u] = sum[u][0] + sum[u][1];
#pragma unroll
                    for (int o = 1; o < PARTS; o <<= 1)
#pragma unroll
                        for (int u = 0; u < 4; ++u) dot[u] += __shfl_xor_sync(0xffffffffu, dot[u], o);
                }
                // (rows of V beyond the rank are whatever the memory held)
                const float mine = (part & 2) ? ((part & 1) ? dot[3] : dot[2]) : ((part & 1) ? dot[1] : dot[0]);
                const int i = i0 + (part & 3);
                if (part < 4) ws_split_store<NQ>(b2, qg, i, (i < rank) ? mine * WS_QSCALE : 0.0f);
            }
            fence_proxy_async_smem();
            if (ws_builder_any(!ok)) break;   // a thread whose wait gave up has built from stale vectors: nothing is handed on
            if (bt == 0) {
                mbar_arrive(&bars.b2_full[vb]);
                mbar_arrive(&bars.blk_empty[vb]);
            }
            if (first_of_head) {
                first_of_head = false;
                if ((head + 1) * a.bph < it1 && !build_w(head + 1, hidx + 1)) break;
            }
            jb += 1;
            if (jb == a.bph) {
                jb = 0;
                head += 1;
            }
        }
    }
    else if (warp < L::EPI_FIRST) {
        // ---------------------------------------------------------------- expanders (groups of 128 threads)
        const int grp = (warp - 4) >> 2;
        const int wt = ((warp - 4) & 3) * 32 + lane;   // token within the tile = tensor-memory lane
        const uint32_t lane_base = static_cast<uint32_t>(32 * (warp & 3)) << 16;
        uint32_t seq0 = 0, sseq = 0;   // the stage's first tile, the stage
        int next = grp;                // this group's next tile, from there
        bool alive = true;
        // Groups take turns on the tiles.  Every group waits for every stage and releases it, whether it has a tile in it or not: one
        // that skipped a phase of the stage's barrier could mistake the phase before the last for the one it waits for next.  (A
        // buffer's d_empty it may skip: when it comes to a tile, its own tile before that one has found its buffer free, and the
        // epilogue empties them in order.)
        for (int item = it0; item < it1 && alive; ++item) {
            for (int tile0 = 0; tile0 < tiles && alive; tile0 += WS_TPS, ++sseq) {
                const int here = min(WS_TPS, tiles - tile0), stage = sseq % L::STAGES;
                if (!mbar_wait_warp(&bars.st_full[stage], (sseq / L::STAGES) & 1u, &abort_flag)) {
                    alive = false;
                    break;
                }
                const uint8_t *st = base + stage * L::STAGE_BYTES;
                const int rank = st_rank[stage];
                auto release = [&] {   // every lane has its copy of the stage's bytes in registers
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bars.st_empty[stage]);
                };
                if (next >= here) release();
                for (; next < here; next += WS_EXP_GROUPS) {
                    const uint32_t seq = seq0 + next;
                    const int tile = tile0 + next, buf = seq % L::BUFS;
                    const bool valid = tile * 128 + wt < n;
                    const int st_tok = next * 128 + wt;   // token within the stage
                    uint32_t cw[4 * BITS];   // the token's 128 codes
#pragma unroll
                    for (int w = 0; w < BITS; ++w) {
                        const uint4 v = *reinterpret_cast<const uint4 *>(st + WS_ST_CODES + st_tok * L::ROW + 16 * w);
                        cw[4 * w] = v.x;
                        cw[4 * w + 1] = v.y;
                        cw[4 * w + 2] = v.z;
                        cw[4 * w + 3] = v.w;
                    }
                    unsigned short rho_raw = *reinterpret_cast<const unsigned short *>(st + L::ST_NORMS + st_tok * 2);
                    const uint8_t *pcol = st + L::ST_P + (st_tok >> 8) * WS_ST_PBOX + (st_tok & 255) * 2;
                    uint32_t pw[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) pw[i] = 0u;
                    // factors four at a time, as many as were copied; those beyond the rank are whatever the memory held
#pragma unroll
                    for (int i = 0; i < WS_PMAX; i += 4) {
                        if (i < rank) {
                            uint32_t v[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e) v[e] = *reinterpret_cast<const unsigned short *>(pcol + (i + e) * 512);
                            const int live = rank - i;
                            pw[i >> 1] = v[0] | ((live > 1) ? v[1] << 16 : 0u);
                            pw[(i >> 1) + 1] = (live > 2) ? (v[2] | ((live > 3) ? v[3] << 16 : 0u)) : 0u;
                        }
                    }
                    if (next + WS_EXP_GROUPS >= here) release();
                    if (!valid) {   // rows past the end of the block were not copied: the stage holds stale bytes there
#pragma unroll
                        for (int w = 0; w < 4 * BITS; ++w) cw[w] = 0u;
                        rho_raw = 0;
#pragma unroll
                        for (int i = 0; i < 8; ++i) pw[i] = 0u;
                    }
                    const uint32_t u = (seq / L::BUFS) & 1u;
                    // the epilogue has read the last use of this buffer, hence its MMAs are over too
                    if (!mbar_wait_warp(&bars.d_empty[buf], u ^ 1u, &abort_flag)) {
                        alive = false;
                        break;
                    }
                    tc_fence_after_sync();
                    const uint32_t tb = tmem0 + lane_base + buf * L::BUF_COLS;
                    {
                        uint32_t av[32];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            if constexpr (BITS == 2) expand16_2bit_placed(cw[q], a.pair_tab, &av[8 * q]);
                            else expand16_codes<BITS>(cw, q, a.lo_tab, a.hi_tab, &av[8 * q]);
                        }
                        tmem_st32(tb, av);
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            if constexpr (BITS == 2) expand16_2bit_placed(cw[4 + q], a.pair_tab, &av[8 * q]);
                            else expand16_codes<BITS>(cw + 2 * BITS, q, a.lo_tab, a.hi_tab, &av[8 * q]);
                        }
                        tmem_st32(tb + 32, av);
                    }
                    tmem_st8(tb + WS_COL_P, pw);
                    {
                        uint32_t rv[8];
                        rv[0] = __float_as_uint(__half2float(__ushort_as_half(rho_raw)));
#pragma unroll
                        for (int i = 1; i < 8; ++i) rv[i] = 0u;
                        tmem_st8(tb + WS_COL_RHO, rv);
                    }
                    tmem_st_wait();
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bars.a_full[buf]);
                }
                next -= here;
                seq0 += here;
            }
        }
    } else {
        // ---------------------------------------------------------------- epilogue (groups of 128 threads)
        const int wt = (warp & 3) * 32 + lane, grp = (warp - L::EPI_FIRST) >> 2;
        const uint32_t lane_base = static_cast<uint32_t>(32 * (warp & 3)) << 16;
        const float f2 = a.scale * (1.0f / WS_QSCALE);
        const size_t qstride = static_cast<size_t>(a.bph) * n;
        uint32_t seq = 0;
        bool alive = true;
        int head = (it0 < it1) ? it0 / a.bph : 0, jb = it0 - head * a.bph;
        for (int item = it0; item < it1 && alive; ++item) {
            float *out_row = a.scores + (static_cast<size_t>(head) * a.G + a.g0 + 8 * grp) * qstride + static_cast<size_t>(jb) * n + wt;
            for (int tile = 0; tile < tiles; ++tile, ++seq) {
                const int buf = seq % L::BUFS;
                if (!mbar_wait_warp(&bars.d_full[buf], (seq / L::BUFS) & 1u, &abort_flag)) {
                    alive = false;
                    break;
                }
                tc_fence_after_sync();
                const uint32_t tb = tmem0 + lane_base + buf * L::BUF_COLS;
                // this group's eight queries: high planes, low planes.  (Groups split the queries and not the tiles: with three
                // buffers, groups that took turns would skip phases of a buffer's barriers, and a parity cannot tell
                // a phase from the one two later.)
                float v[8];
                {
                    uint32_t c[16], p[16], rv[8];
                    if constexpr (NQ == 8) {
                        tmem_ld16(tb + L::COL_D1, c);
                        tmem_ld16(tb + L::COL_D2, p);
                    } else {
                        tmem_ld8(tb + L::COL_D1 + 8 * grp, *reinterpret_cast<uint32_t(*)[8]>(&c[0]));
                        tmem_ld8(tb + L::COL_D1 + NQ + 8 * grp, *reinterpret_cast<uint32_t(*)[8]>(&c[8]));
                        tmem_ld8(tb + L::COL_D2 + 8 * grp, *reinterpret_cast<uint32_t(*)[8]>(&p[0]));
                        tmem_ld8(tb + L::COL_D2 + NQ + 8 * grp, *reinterpret_cast<uint32_t(*)[8]>(&p[8]));
                    }
                    tmem_ld8(tb + WS_COL_RHO, rv);
                    tmem_ld_wait();
                    const float f1 = a.scale * __uint_as_float(rv[0]) * a.inv_code;
#pragma unroll
                    for (int g = 0; g < 8; ++g)
                        v[g] = fmaf(f1, __uint_as_float(c[g]) + __uint_as_float(c[8 + g]), f2 * (__uint_as_float(p[g]) + __uint_as_float(p[8 + g])));
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars.d_empty[buf]);
                if (tile * 128 + wt < n) {
                    float *p = out_row + tile * 128;
#pragma unroll
                    for (int g = 0; g < 8; ++g) {
                        if (8 * grp + g < gcount) *p = v[g];
                        p += qstride;
                    }
                }
            }
            jb += 1;
            if (jb == a.bph) {
                jb = 0;
                head += 1;
            }
        }
    }

    __syncthreads();
    if (abort_flag) {
        if (tid == 0) atomicOr(a.err, TC_ERR_SCORES_WS_TIMEOUT);
        // Copies and MMAs that are still in flight must land before shared and tensor memory are given back.  Each thread waits for
        // the last loads it announced, as many as there are places for them (one that has landed is waited for in no time).
        volatile int scratch = 0;
        const bool issued = warp == 1 && issuer;
        if (issued) umma_commit(&bars.drain);   // (a commit follows the MMAs of its own thread)
#pragma unroll 1
        for (int kind = 0; kind < 4; ++kind) {
            uint64_t *const first = (kind == 0) ? bars.st_full : (kind == 1) ? bars.blk_full : (kind == 2) ? bars.b1_full : &bars.drain;
            const uint32_t places = (kind == 0) ? L::STAGES : (kind == 3) ? 1u : 2u;
            const uint32_t fills = (kind == 0) ? st_fills : (kind == 1) ? blk_fills : (kind == 2) ? b1_fills : issued ? 1u : 0u;
#pragma unroll 1
            for (uint32_t f = (fills > places) ? fills - places : 0u; f < fills; ++f) mbar_wait(&first[f % places], (f / places) & 1u, &scratch);
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc(tmem0, WS_TMEM_COLS);
    }
}

template <int BITS, int NQ>
static bool launch_scores_ws_as(WsArgs &a, int G, int grid, const CUtensorMap &m4, const CUtensorMap &m8, const CUtensorMap &m12,
                                uint8_t *wimg, int64_t *kernels, cudaStream_t s) {
    if (!ensure_dynamic_smem(reinterpret_cast<const void *>(scores_ws_kernel<BITS, NQ>), WsLayout<BITS, NQ>::SMEM_BYTES)) return false;
    for (int g0 = 0; g0 < G; g0 += NQ) {
        a.g0 = g0;
        if (!a.local_w) {
            launch_dependent(scores_w_kernel<(BITS == 2) ? 2 : 1, NQ>, static_cast<unsigned>(a.heads), D, 0, s, a.pi_t, a.q, G, g0, wimg);
            *kernels += 1;
        }
        launch_dependent(scores_ws_kernel<BITS, NQ>, static_cast<unsigned>(grid), WsLayout<BITS, NQ>::THREADS, WsLayout<BITS, NQ>::SMEM_BYTES, s, a, m4, m8, m12);
        *kernels += 1;
    }
    return true;
}

bool launch_scores_ws(const eosq_cache_t &cache, int bits, int64_t heads, int64_t bph, int64_t head_stride, int n, const Rotation &rot,
                      const uint16_t (&table)[16], float kappa, const __half *q, int G, float scale, float *scores, int *err,
                      int sm_count, void **scratch, size_t *scratch_bytes, int64_t *kernels, cudaStream_t s) {
    if (heads * bph > 0x7fffffff || head_stride > 0x7fffffff || bits < 1 || bits > 4) return false;
    WsArgs a;
    a.cache = cache;
    a.bph = static_cast<int>(bph);
    a.head_stride = static_cast<int>(head_stride);
    a.heads = static_cast<int>(heads);
    a.n = n;
    a.G = G;
    a.scale = scale;
    a.inv_code = 1.0f / (kappa * WS_QSCALE);
    for (int w = 0; w < 4; ++w) a.lo_tab[w] = a.hi_tab[w] = 0u;
    for (int k = 0; k < (1 << bits); ++k) {
        a.lo_tab[k >> 2] |= static_cast<uint32_t>(table[k] & 0xFFu) << (8 * (k & 3));
        a.hi_tab[k >> 2] |= static_cast<uint32_t>(table[k] >> 8) << (8 * (k & 3));
    }
    for (int h = 0; h < 2; ++h) a.pair_tab[h] = static_cast<uint32_t>(table[2 * h]) | (static_cast<uint32_t>(table[2 * h + 1]) << 16);
    const int grid = static_cast<int>(std::min<int64_t>(heads * bph, sm_count));
    const int nq = (G > 8) ? 16 : 8;
    a.pi_t = rot.pi_t;
    // A CTA whose run of blocks is no longer than a head's touches two heads at most and makes their W itself.
    a.local_w = (heads * bph + grid - 1) / grid <= bph;
    if (!a.local_w) {
        // one operand image per head, in a buffer the context keeps and grows (earlier work that still reads the old
        // buffer is waited for by cudaFree)
        const size_t need = static_cast<size_t>(heads) * nq * 512;
        if (*scratch_bytes < need) {
            cudaFree(*scratch);
            *scratch = nullptr;
            *scratch_bytes = 0;
            if (cudaMalloc(scratch, need) != cudaSuccess) return false;
            *scratch_bytes = need;
        }
    }
    a.wimg = static_cast<const uint8_t *>(*scratch);
    a.q = q;
    a.scores = scores;
    a.err = err;
    const int64_t nb_total = (heads - 1) * head_stride + bph;
    CUtensorMap m4, m8, m12;
    if (!make_factor_tensor_map(cache.P, nb_total, n, 4, &m4) || !make_factor_tensor_map(cache.P, nb_total, n, 8, &m8) ||
        !make_factor_tensor_map(cache.P, nb_total, n, 12, &m12))
        return false;
    uint8_t *wimg = static_cast<uint8_t *>(*scratch);
    switch (bits * 32 + nq) {
        case 1 * 32 + 8: return launch_scores_ws_as<1, 8>(a, G, grid, m4, m8, m12, wimg, kernels, s);
        case 2 * 32 + 8: return launch_scores_ws_as<2, 8>(a, G, grid, m4, m8, m12, wimg, kernels, s);
        case 3 * 32 + 8: return launch_scores_ws_as<3, 8>(a, G, grid, m4, m8, m12, wimg, kernels, s);
        case 4 * 32 + 8: return launch_scores_ws_as<4, 8>(a, G, grid, m4, m8, m12, wimg, kernels, s);
        case 1 * 32 + 16: return launch_scores_ws_as<1, 16>(a, G, grid, m4, m8, m12, wimg, kernels, s);
        case 2 * 32 + 16: return launch_scores_ws_as<2, 16>(a, G, grid, m4, m8, m12, wimg, kernels, s);
        case 3 * 32 + 16: return launch_scores_ws_as<3, 16>(a, G, grid, m4, m8, m12, wimg, kernels, s);
        default: return launch_scores_ws_as<4, 16>(a, G, grid, m4, m8, m12, wimg, kernels, s);
    }
}

}  // namespace eosq
