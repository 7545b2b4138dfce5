// Tensor-core decode for 1- to 4-bit codes (Algorithm 1 DeQuant + the stored low-rank part):
//   x_t = rho_t (z_t Pi) + sum_i P[t][i] zeta_i,     z_t = centroids of the codes of token t.
//
// One persistent, warp-specialised CTA of 18 warps per SM holds the rotation once, as the B operand of
//   D1[128 tokens][128] = Z[128][128] (fp16 centroids) x Pi      (Pi scaled by 2^12 and split
//                                                                  into a high and a low fp16 plane),
//   D2[128 tokens][128] = P_tile[128][16] x V[16][128]            (stored fp16 factors: exact products),
// both accumulated in fp32 in tensor memory, two buffers of 128 + 128 columns.
//   warp 0        bulk-copies each tile's codes, norms and factor rows into a ring of raw stages
//   warp 1        issues the 17 MMAs of a tile
//   warps 2-9     expand the codes into a K-major, 128-byte-swizzled A tile (byte permutes, 64 codes per thread) and put
//                 the factor entries and, per block, the right vectors into theirs (two A tiles)
//   warps 10-17   turn 64 columns of one token into rho D1 / (kappa 2^12) + D2, stage them and store them by tensor
//                 stores, each half of the columns with its own 16 KB stage
// so that a tile's expansion, the next one's copies, the previous one's MMAs and the one before's output run side by
// side.  Bound by HBM: 32 KB (fp16) or 64 KB out and about 7 KB in per tile, 1 750 cycles of an SM's share; the MMAs
// take 1 090.  (Two independent halves that each went through these steps one after another took 4 000 cycles per
// tile: 0.91 ms for 8192 blocks of 1024 tokens at three bits.)
// Work is dealt out in tiles (TileRuns), so that 16 blocks occupy 128 SMs and no SM is left with one block more than
// the others.
#include <algorithm>
#include <cstdint>
#include <cstring>

#include "eosq_common.cuh"
#include "eosq_expand.cuh"
#include "eosq_sm100.cuh"

namespace eosq {

using namespace sm100;

constexpr int TC_ERR_DECODE_TIMEOUT = 16;

constexpr int DT_THREADS = 576, DT_EXP_FIRST = 2, DT_EXP_WARPS = 8, DT_EPI_FIRST = 10;
constexpr float DT_PSCALE = 4096.0f;                  // keeps the low plane of Pi in fp16's normal range
constexpr uint32_t DT_BOX = 128 * 128;                // 128 rows x 64 fp16 of K
// shared memory: Pi's planes, two A tiles, one box with the K = 16 operands (32 bytes of each 128-byte row: the factor
// entries of the two tiles, the right vectors of two blocks), two output stages, the raw stages
constexpr uint32_t DT_OFF_PI_HI = 0, DT_OFF_PI_LO = 2 * DT_BOX, DT_OFF_A = 4 * DT_BOX, DT_OFF_K16 = 8 * DT_BOX, DT_OFF_OUT = 9 * DT_BOX,
                   DT_OFF_RAW = 11 * DT_BOX;
// a raw stage: packed codes (128 tokens x 16 BITS bytes), norms, up to 12 factor rows of 128 fp16
constexpr int DT_PMAX = 12, DT_RAW_STAGES = 3;
constexpr uint32_t DT_RAW_BYTES = 128 * 64 + 256 + DT_PMAX * 256;
static_assert(KPILOT < DT_PMAX, "every kept factor is staged");
constexpr size_t DT_SMEM = DT_OFF_RAW + DT_RAW_STAGES * DT_RAW_BYTES + 1024;
static_assert(DT_SMEM <= 226 * 1024, "fits the shared memory of an SM next to the barriers");
constexpr uint32_t DT_TMEM_COLS = 512;                // per buffer: D1 128 columns, D2 128 columns

// Byte offset of the 16-byte chunk `jc` (8 fp16 of K) of row `row` in a K-major, 128-byte-swizzled
// operand of 128 rows: 64-wide K boxes of 16 KB, 8-row groups of 1 KB, chunks XOR-ed with the row.
__device__ __forceinline__ uint32_t dt_offset(int row, int jc) {
    return (jc >> 3) * DT_BOX + (row >> 3) * 1024 + (row & 7) * 128 + (((jc & 7) ^ (row & 7)) << 4);
}

// Barrier of the 128 threads of one output half that also tells each of them whether any brings `failed`.  A
// bounded wait ends per thread, so one thread may give up where its neighbour just succeeds: the outcome is
// made common at the next barrier, and the half leaves its loop as a whole (a thread that left alone would let
// the barrier wait for ever).
__device__ __forceinline__ bool dt_out_any(int half, bool failed) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "bar.red.or.pred q, %2, 128, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(failed ? 1u : 0u), "r"(1 + half)
        : "memory");
    return r != 0;
}

struct DtBars {
    uint64_t raw_full[DT_RAW_STAGES], raw_empty[DT_RAW_STAGES];
    uint64_t a_full[2];    // operands of a tile are written (one arrival per expander warp)
    uint64_t done[2];      // its MMAs are over: accumulators ready, A tile free
    uint64_t d_empty[2];   // its accumulators are read (one arrival per output warp)
    uint64_t drain;
};

struct DecodeArgs {
    eosq_cache_t cache;
    int nb, n;
    float inv_scale;            // 1 / (kappa 2^12)
    uint32_t lo_tab[4], hi_tab[4];   // low / high bytes of the fp16 centroids times kappa (level k in byte k)
    const float *pi_t;          // pi_t[j][c] = Pi[c][j]
    int *err;
};

__device__ __forceinline__ void dt_bulk_load(void *smem_dst, const void *gsrc, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :
                 : "r"(smem_u32(smem_dst)), "l"(reinterpret_cast<uint64_t>(gsrc)), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

bool make_block_tensor_map(const void *blocks, int64_t nb, int n, CUtensorMap *out);
bool make_f32_block_tensor_map(const void *blocks, int64_t nb, int n, CUtensorMap *out);

// `omap`: the output as [nb][n][128] with boxes of 128 tokens x 128 bytes (64 fp16 or 32 fp32 coordinates), 128-byte swizzle.
template <typename Tout, int BITS>
__global__ void __launch_bounds__(DT_THREADS, 1) decode_tc_kernel(const DecodeArgs a, const __grid_constant__ CUtensorMap omap) {
    static_assert(BITS >= 1 && BITS <= 4, "code widths of the format");
    extern __shared__ uint8_t dt_smem_raw[];
    __shared__ __align__(8) DtBars bars;
    __shared__ uint32_t tmem_base_s;
    __shared__ float rho_s[4][128];   // rho / (kappa 2^12) of the last tiles: the slot of tile t is free once tile t + 2's MMAs are over
    __shared__ uint32_t fills[DT_RAW_STAGES], drains[DT_RAW_STAGES];
    __shared__ volatile int abort_flag;

    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(dt_smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n = a.n, tiles = (n + 127) / 128;
    constexpr uint32_t ROW = 16 * BITS, RAW_NORMS = 128 * ROW, RAW_P = RAW_NORMS + 256;

    if (tid == 0) {
        for (int s = 0; s < DT_RAW_STAGES; ++s) {
            mbar_init(&bars.raw_full[s], 1);
            mbar_init(&bars.raw_empty[s], DT_EXP_WARPS);
            fills[s] = 0;
            drains[s] = 0;
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&bars.a_full[b], DT_EXP_WARPS);
            mbar_init(&bars.done[b], 1);
            mbar_init(&bars.d_empty[b], 8);
        }
        mbar_init(&bars.drain, 1);
        abort_flag = 0;
        fence_mbar_init();
        tma_prefetch_desc(&omap);
    }
    if (warp == 1) {
        tmem_alloc(&tmem_base_s, DT_TMEM_COLS);
        tmem_relinquish();
    }
    // B operand of D1, once per CTA: row j (output coordinate), K = c: Pi[c][j] 2^12 as high + low fp16
    for (int chunk = tid; chunk < D * (D / 8); chunk += DT_THREADS) {
        const int j = chunk >> 4, jc = chunk & 15;
        const float4 p0 = __ldg(reinterpret_cast<const float4 *>(a.pi_t + j * D + 8 * jc));
        const float4 p1 = __ldg(reinterpret_cast<const float4 *>(a.pi_t + j * D + 8 * jc + 4));
        const float m[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
        uint32_t h[4], l[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float x0 = m[2 * e] * DT_PSCALE, x1 = m[2 * e + 1] * DT_PSCALE;
            const __half h0 = __float2half_rn(x0), h1 = __float2half_rn(x1);
            const __half l0 = __float2half_rn(x0 - __half2float(h0)), l1 = __float2half_rn(x1 - __half2float(h1));
            h[e] = static_cast<uint32_t>(__half_as_ushort(h0)) | (static_cast<uint32_t>(__half_as_ushort(h1)) << 16);
            l[e] = static_cast<uint32_t>(__half_as_ushort(l0)) | (static_cast<uint32_t>(__half_as_ushort(l1)) << 16);
        }
        const uint32_t off = dt_offset(j, jc);
        *reinterpret_cast<uint4 *>(base + DT_OFF_PI_HI + off) = make_uint4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<uint4 *>(base + DT_OFF_PI_LO + off) = make_uint4(l[0], l[1], l[2], l[3]);
    }
    fence_proxy_async_smem();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem0 = warp_uniform(tmem_base_s);
    const bool issuer = elect_one();   // of warp 1: the lane that issues
    pdl_wait();   // (the rotation was uploaded before any kernel of the stream)

    const TileRuns runs(a.nb, tiles, blockIdx.x, gridDim.x);
    const int count = runs.total();
    // every role walks the runs in the same order
    struct Place {
        int run, blk, tile, end;
    };
    auto first_place = [&](Place &p) {
        p.run = 0;
        runs.get(0, p.blk, p.tile, p.end);
    };
    auto advance = [&](Place &p) -> bool {   // true when a new block begins
        if (++p.tile < p.end) return false;
        p.run += 1;
        if (p.run < runs.count) runs.get(p.run, p.blk, p.tile, p.end);
        return true;
    };
    auto next_block = [&](const Place &p) { return (p.run + 1 < runs.count) ? runs.block(p.run + 1) : a.nb; };
    // Ranks are clamped to the rows a raw stage holds; the library never stores more than the pilot k = 11.
    auto rank_of = [&](int blk) { return (blk < a.nb) ? max(0, min(a.cache.rank[blk], DT_PMAX)) : 0; };

    if (warp == 0) {
        // ------------------------------------------------------------------ raw data, one copy per lane
        // (a thread needs over 100 cycles per copy it issues)
        Place at;
        first_place(at);
        int rank = rank_of(at.blk), rank_next = rank_of(next_block(at));
        for (int t = 0; t < count; ++t) {
            const int s = t % DT_RAW_STAGES, blk = at.blk;
            const int tok0 = at.tile * 128;
            const uint32_t rows = static_cast<uint32_t>(min(128, n - tok0));
            const size_t t0 = static_cast<size_t>(blk) * n + tok0;
            bool ok = true;
            if (lane == 0) {
                ok = mbar_wait(&bars.raw_empty[s], ((t / DT_RAW_STAGES) & 1u) ^ 1u, &abort_flag);
                if (ok) {
                    mbar_arrive_expect_tx(&bars.raw_full[s], rows * (ROW + 2u) + static_cast<uint32_t>(rank) * rows * 2u);
                    fills[s] += 1;
                }
            }
            if (!__shfl_sync(0xffffffffu, ok, 0)) break;   // (also: the byte count is announced before any copy can report completion)
            uint8_t *raw = base + DT_OFF_RAW + s * DT_RAW_BYTES;
            if (lane == 0) dt_bulk_load(raw, a.cache.codes + t0 * ROW, rows * ROW, &bars.raw_full[s]);
            else if (lane == 1) dt_bulk_load(raw + RAW_NORMS, a.cache.norms + t0, rows * 2u, &bars.raw_full[s]);
            else if (lane - 2 < rank)
                dt_bulk_load(raw + RAW_P + (lane - 2) * 256, a.cache.P + (static_cast<size_t>(blk) * RMAX + (lane - 2)) * n + tok0, rows * 2u, &bars.raw_full[s]);
            if (advance(at)) {
                rank = rank_next;
                rank_next = rank_of(next_block(at));   // known long before that block starts
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMAs
        {
            constexpr uint32_t idesc = umma_idesc_f16(128, D, false, false);
            const uint32_t hi0 = smem_u32(base + DT_OFF_PI_HI), lo0 = smem_u32(base + DT_OFF_PI_LO), k16 = smem_u32(base + DT_OFF_K16);
            int vb = 0;
            Place at;
            first_place(at);
            for (int t = 0; t < count; ++t) {
                const int buf = t & 1;
                const uint32_t u = (t >> 1) & 1u;
                if (!mbar_wait_warp(&bars.a_full[buf], u, &abort_flag) || !mbar_wait_warp(&bars.d_empty[buf], u ^ 1u, &abort_flag)) break;
                tc_fence_after_sync();
                const uint32_t a0 = smem_u32(base + DT_OFF_A + buf * 2 * DT_BOX), d1 = tmem0 + 256u * buf;
                if (issuer) {
                    umma_f16(d1 + 128u, umma_desc_sw128(k16 + 32 * buf, 16, 1024), umma_desc_sw128(k16 + 64 + 32 * vb, 16, 1024), idesc, 0u);
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks) {
                        const uint32_t ko = (ks >> 2) * DT_BOX + (ks & 3) * 32;
                        const uint64_t da = umma_desc_sw128(a0 + ko, 16, 1024);
                        umma_f16(d1, da, umma_desc_sw128(hi0 + ko, 16, 1024), idesc, ks ? 1u : 0u);
                        umma_f16(d1, da, umma_desc_sw128(lo0 + ko, 16, 1024), idesc, 1u);
                    }
                    umma_commit(&bars.done[buf]);
                }
                __syncwarp();
                if (advance(at)) vb ^= 1;
            }
        }
    } else if (warp < DT_EPI_FIRST) {
        // ------------------------------------------------------------------ expansion: token r, codes [64 box, 64 box + 64)
        const int et = tid - 32 * DT_EXP_FIRST, r = et & 127, box = et >> 7;
        Place at;
        first_place(at);
        int vb = 0, rank = rank_of(at.blk), rank_next = rank_of(next_block(at));
        bool fresh = true;   // the block's right vectors are not in place yet
        // Row j = r of V's operand, K = i: zeta_i[j] (zero beyond the rank), entries 8 box .. 8 box + 7; asked for a whole
        // tile before they are needed.
        unsigned short vr[8];
        auto fetch_v = [&](int b, int rk) {
#pragma unroll
            for (int e = 0; e < 8; ++e)
                vr[e] = (8 * box + e < rk) ? a.cache.V[(static_cast<size_t>(b) * RMAX + 8 * box + e) * D + r] : static_cast<unsigned short>(0);
        };
        fetch_v(at.blk, rank);
        for (int t = 0; t < count; ++t) {
            const int s = t % DT_RAW_STAGES, buf = t & 1;
            uint32_t vw[4];
            if (fresh) {
#pragma unroll
                for (int e = 0; e < 4; ++e) vw[e] = static_cast<uint32_t>(vr[2 * e]) | (static_cast<uint32_t>(vr[2 * e + 1]) << 16);
            }
            if (at.tile == at.end - 1 && t + 1 < count) fetch_v(next_block(at), rank_next);
            if (!mbar_wait_warp(&bars.raw_full[s], (t / DT_RAW_STAGES) & 1u, &abort_flag)) break;
            if (et == 0) drains[s] += 1;
            const uint8_t *raw = base + DT_OFF_RAW + s * DT_RAW_BYTES;
            const bool valid = at.tile * 128 + r < n;   // rows past the end of the block were not copied
            uint32_t cw[2 * BITS];
#pragma unroll
            for (int w = 0; w < BITS; ++w) {
                const uint2 v = *reinterpret_cast<const uint2 *>(raw + r * ROW + 8 * BITS * box + 8 * w);
                cw[2 * w] = valid ? v.x : 0u;
                cw[2 * w + 1] = valid ? v.y : 0u;
            }
            uint32_t rho_raw = 0u, pw[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) pw[i] = 0u;
            if (box == 0 && valid) {
                rho_raw = *reinterpret_cast<const unsigned short *>(raw + RAW_NORMS + 2 * r);
#pragma unroll
                for (int i = 0; i < DT_PMAX; ++i)
                    if (i < rank) pw[i >> 1] |= static_cast<uint32_t>(*reinterpret_cast<const unsigned short *>(raw + RAW_P + i * 256 + 2 * r)) << (16 * (i & 1));
            }
            __syncwarp();   // every lane has its copy of the stage's bytes in registers
            if (lane == 0) mbar_arrive(&bars.raw_empty[s]);
            uint32_t o[4][8];
#pragma unroll
            for (int q = 0; q < 4; ++q) expand16_codes<BITS>(cw, q, a.lo_tab, a.hi_tab, o[q]);
            // the MMAs that read this A tile last are over (and with them, see rho_s, the output of the tile before)
            if (!mbar_wait_warp(&bars.done[buf], ((t >> 1) & 1u) ^ 1u, &abort_flag)) break;
            uint8_t *A = base + DT_OFF_A + buf * 2 * DT_BOX, *K16 = base + DT_OFF_K16;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                *reinterpret_cast<uint4 *>(A + dt_offset(r, 8 * box + 2 * q)) = make_uint4(o[q][0], o[q][1], o[q][2], o[q][3]);
                *reinterpret_cast<uint4 *>(A + dt_offset(r, 8 * box + 2 * q + 1)) = make_uint4(o[q][4], o[q][5], o[q][6], o[q][7]);
            }
            if (box == 0) {
                *reinterpret_cast<uint4 *>(K16 + dt_offset(r, 2 * buf)) = make_uint4(pw[0], pw[1], pw[2], pw[3]);
                *reinterpret_cast<uint4 *>(K16 + dt_offset(r, 2 * buf + 1)) = make_uint4(pw[4], pw[5], pw[6], pw[7]);
                rho_s[t & 3][r] = __half2float(__ushort_as_half(static_cast<unsigned short>(rho_raw))) * a.inv_scale;
            }
            // (this place was read last by MMAs of the block before the previous one, two tiles ago at least)
            if (fresh) *reinterpret_cast<uint4 *>(K16 + dt_offset(r, 4 + 2 * vb + box)) = make_uint4(vw[0], vw[1], vw[2], vw[3]);
            fence_proxy_async_smem();   // the operands were written by ordinary stores and are read by the tensor core
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars.a_full[buf]);
            fresh = false;
            if (advance(at)) {
                vb ^= 1;
                fresh = true;
                rank = rank_next;
                rank_next = rank_of(next_block(at));
            }
        }
    } else {
        // ------------------------------------------------------------------ output: token r, columns [64 half, 64 half + 64)
        const int r = 32 * (warp & 3) + lane, half = (warp - DT_EPI_FIRST) >> 2;
        const bool leader = (warp - DT_EPI_FIRST) % 4 == 0 && lane == 0;
        const uint32_t lane_off = static_cast<uint32_t>(32 * (warp & 3)) << 16;   // a warp reaches lanes 32 (warp % 4)..
        uint8_t *stage = base + DT_OFF_OUT + half * DT_BOX;
        Place at;
        first_place(at);
        for (int t = 0; t < count; ++t) {
            const int buf = t & 1, blk = at.blk, tile = at.tile;
            // (a thread whose wait gave up works on with whatever it reads, up to the half's next barrier)
            const bool ok = mbar_wait(&bars.done[buf], (t >> 1) & 1u, &abort_flag);
            tc_fence_after_sync();
            const float f = rho_s[t & 3][r];
            const uint32_t d1 = tmem0 + 256u * buf + lane_off + 64u * half;
            auto release = [&] {   // the accumulators are read
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars.d_empty[buf]);
            };
            bool failed = false;
            if (sizeof(Tout) == 2) {
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    uint32_t v1[32], v2[32];
                    tmem_ld32(d1 + 32u * c, v1);
                    tmem_ld32(d1 + 128u + 32u * c, v2);
                    tmem_ld_wait();
                    if (c == 1) release();
                    if (c == 0) {
                        if (leader) bulk_wait_read_all();   // the copy engine has read the store before
                        if (dt_out_any(half, !ok)) {
                            failed = true;
                            break;
                        }
                    }
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        uint32_t pk[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const __half2 h = __floats2half2_rn(fmaf(f, __uint_as_float(v1[8 * e + 2 * q]), __uint_as_float(v2[8 * e + 2 * q])),
                                                                fmaf(f, __uint_as_float(v1[8 * e + 2 * q + 1]), __uint_as_float(v2[8 * e + 2 * q + 1])));
                            pk[q] = *reinterpret_cast<const uint32_t *>(&h);
                        }
                        *reinterpret_cast<uint4 *>(stage + dt_offset(r, 4 * c + e)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                    }
                }
                if (!failed) {
                    fence_proxy_async_smem();   // the stage was written by ordinary stores and is read by the copy engine
                    dt_out_any(half, false);
                    if (leader) {   // rows past the end of the block are clipped
                        tma_store_3d(&omap, stage, 64 * half, tile * 128, blk);
                        bulk_commit_group();
                    }
                }
            } else {
#pragma unroll
                for (int c = 0; c < 2; ++c) {   // 32 columns fill the stage
                    uint32_t v1[32], v2[32];
                    tmem_ld32(d1 + 32u * c, v1);
                    tmem_ld32(d1 + 128u + 32u * c, v2);
                    tmem_ld_wait();
                    if (c == 1) release();
                    if (leader) bulk_wait_read_all();
                    if (dt_out_any(half, !ok)) {
                        failed = true;
                        break;
                    }
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        *reinterpret_cast<float4 *>(stage + dt_offset(r, e)) =
                            make_float4(fmaf(f, __uint_as_float(v1[4 * e]), __uint_as_float(v2[4 * e])),
                                        fmaf(f, __uint_as_float(v1[4 * e + 1]), __uint_as_float(v2[4 * e + 1])),
                                        fmaf(f, __uint_as_float(v1[4 * e + 2]), __uint_as_float(v2[4 * e + 2])),
                                        fmaf(f, __uint_as_float(v1[4 * e + 3]), __uint_as_float(v2[4 * e + 3])));
                    fence_proxy_async_smem();
                    dt_out_any(half, false);
                    if (leader) {
                        tma_store_3d(&omap, stage, 64 * half + 32 * c, tile * 128, blk);
                        bulk_commit_group();
                    }
                }
            }
            if (failed) break;
            advance(at);
        }
        if (leader) bulk_wait_all();
    }

    __syncthreads();
    if (abort_flag) {
        if (tid == 0) atomicOr(a.err, TC_ERR_DECODE_TIMEOUT);
        // copies and MMAs that are still in flight must land before shared and tensor memory are given back
        if (tid == 0) {
            volatile int scratch = 0;
            for (int s = 0; s < DT_RAW_STAGES; ++s)
                if (fills[s] != drains[s]) mbar_wait(&bars.raw_full[s], (fills[s] - 1u) & 1u, &scratch);
        }
        if (warp == 1 && issuer) {
            volatile int scratch = 0;
            umma_commit(&bars.drain);
            mbar_wait(&bars.drain, 0, &scratch);
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc(tmem0, DT_TMEM_COLS);
    }
}

float best_table_scale(const Codebook &cb, uint16_t (&table)[16]);

bool decode_tc_supported(const eosq_cache_t &cache, int bits, const void *out_blocks) {
    auto aligned = [](const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };   // bulk copies and tensor stores
    return bits >= 1 && bits <= 4 && aligned(cache.codes) && aligned(cache.norms) && aligned(cache.P) && aligned(out_blocks);
}

template <typename Tout, int BITS>
static bool launch_decode_tc_as(const DecodeArgs &a, const CUtensorMap &omap, int grid, cudaStream_t s) {
    if (!ensure_dynamic_smem(reinterpret_cast<const void *>(decode_tc_kernel<Tout, BITS>), DT_SMEM)) return false;
    launch_dependent(decode_tc_kernel<Tout, BITS>, static_cast<unsigned>(grid), DT_THREADS, DT_SMEM, s, a, omap);
    return true;
}

bool launch_decode_tc(const eosq_cache_t &cache, int64_t nb, int n, const Rotation &rot, const Codebook &cb, void *out_blocks,
                      int out_dtype, int *err, int sm_count, cudaStream_t s) {
    // the centroid table depends only on the codebook: search its scale once per code width
    static uint16_t table[5][16];
    static float kappa[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    const int bits = cb.bits;
    if (bits < 1 || bits > 4) return false;
    if (kappa[bits] == 0.0f) kappa[bits] = best_table_scale(cb, table[bits]);
    DecodeArgs a;
    a.cache = cache;
    a.nb = static_cast<int>(nb);
    a.n = n;
    a.inv_scale = 1.0f / (kappa[bits] * DT_PSCALE);
    for (int w = 0; w < 4; ++w) a.lo_tab[w] = a.hi_tab[w] = 0u;
    for (int k = 0; k < (1 << bits); ++k) {
        a.lo_tab[k >> 2] |= static_cast<uint32_t>(table[bits][k] & 0xFFu) << (8 * (k & 3));
        a.hi_tab[k >> 2] |= static_cast<uint32_t>(table[bits][k] >> 8) << (8 * (k & 3));
    }
    a.pi_t = rot.pi_t;
    a.err = err;
    const int grid = static_cast<int>(std::min<int64_t>(nb * ((n + 127) / 128), sm_count));
    CUtensorMap omap;
    if (out_dtype == EOSQ_F32) {
        if (!make_f32_block_tensor_map(out_blocks, nb, n, &omap)) return false;
        switch (bits) {
            case 1: return launch_decode_tc_as<float, 1>(a, omap, grid, s);
            case 2: return launch_decode_tc_as<float, 2>(a, omap, grid, s);
            case 3: return launch_decode_tc_as<float, 3>(a, omap, grid, s);
            default: return launch_decode_tc_as<float, 4>(a, omap, grid, s);
        }
    }
    if (!make_block_tensor_map(out_blocks, nb, n, &omap)) return false;
    switch (bits) {
        case 1: return launch_decode_tc_as<__half, 1>(a, omap, grid, s);
        case 2: return launch_decode_tc_as<__half, 2>(a, omap, grid, s);
        case 3: return launch_decode_tc_as<__half, 3>(a, omap, grid, s);
        default: return launch_decode_tc_as<__half, 4>(a, omap, grid, s);
    }
}

}  // namespace eosq
