// The exact-arithmetic path: the Gram matrix in double precision (fp32 blocks, short fp16 blocks, and the
// second pass over fp16 blocks whose spectrum the half-precision tensor-core Gram matrix cannot resolve),
// and residual + rotation + quantisation + packing of fp32 blocks as tiled FMA loops in shared memory.
#include <algorithm>

#include "eosq_common.cuh"

namespace eosq {

// ------------------------------------------------------------------------------------------
// G = S^T S on the fp64 tensor instruction: products of fp16 or fp32 inputs are exact in double, so the only
// rounding is the double accumulation, token after token in the same order whatever the launch.  Bound by that
// instruction: 136 of them per four tokens, 17 400 cycles of an SM per 128 tokens (the plain multiply-adds this
// replaces ran at half of that rate, on the whole square).
// Both operands of a product of 8 x 8 tiles are columns of S: lane (m, k) takes column 8 I + m of token k, so the
// values a warp holds for tile rows I serve as A and as B, and a square of Q x Q tiles needs 2 Q values per four
// tokens and lane, straight from global memory (L1 serves the repeats), the next ones on their way meanwhile.
// Q = 4: ten squares (one warp each) cover the lower half, a CTA is a block.  Q = 2: 36 squares, four of them a
// CTA, for launches that would otherwise leave SMs idle.
// ------------------------------------------------------------------------------------------
template <typename Tin, int Q>
__global__ void __launch_bounds__(Q == 4 ? 320 : 128, Q == 4 ? 2 : 4) gram_exact_kernel(const Tin *blocks, int n, double *gram,
                                                                                       int nb, const int *list, const int *count) {
    constexpr int SQ = GRAM_TILE_ROWS / Q, WARPS = (Q == 4) ? 10 : 4, AHEAD = (Q == 4) ? 2 : 4;
    static_assert(Q == 4 ? SQ * (SQ + 1) / 2 == WARPS : SQ * (SQ + 1) / 2 % WARPS == 0, "a warp per square");
    const int lane = threadIdx.x & 31, m = lane >> 2, k = lane & 3;
    const int unit = blockIdx.y * WARPS + (threadIdx.x >> 5);
    int si = 0;
    while ((si + 1) * (si + 2) / 2 <= unit) ++si;
    const int sj = unit - si * (si + 1) / 2;
    pdl_wait();
    const int total = list ? *count : nb;
    for (int li = blockIdx.x; li < total; li += gridDim.x) {
        const int blk = list ? list[li] : li;
        const Tin *src = blocks + (static_cast<size_t>(blk) * n + k) * D + m;
        double acc[Q][Q][2];
#pragma unroll
        for (int i = 0; i < Q; ++i)
#pragma unroll
            for (int j = 0; j < Q; ++j) acc[i][j][0] = acc[i][j][1] = 0.0;
        Tin ra[AHEAD][Q], rb[AHEAD][Q];
        auto fetch = [&](Tin (&a)[Q], Tin (&b)[Q], int step) {
            const Tin *p = src + static_cast<size_t>(step) * 4 * D;
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                a[q] = p[8 * (Q * si + q)];
                b[q] = p[8 * (Q * sj + q)];
            }
        };
        const int steps = n / 4;   // n is a multiple of 8
#pragma unroll
        for (int e = 0; e < AHEAD; ++e) fetch(ra[e], rb[e], min(e, steps - 1));
#pragma unroll 1
        for (int s = 0; s < steps; s += AHEAD) {
#pragma unroll
            for (int e = 0; e < AHEAD; ++e) {
                if (s + e >= steps) break;
                double a[Q], b[Q];
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    a[q] = static_cast<double>(to_float(ra[e][q]));
                    b[q] = static_cast<double>(to_float(rb[e][q]));
                }
                fetch(ra[e], rb[e], min(s + e + AHEAD, steps - 1));
#pragma unroll
                for (int i = 0; i < Q; ++i)
#pragma unroll
                    for (int j = 0; j < Q; ++j) dmma(acc[i][j], a[i], b[j]);
            }
        }
        double *G = gram + static_cast<size_t>(blk) * GRAM_ELEMS + tile_off(m, 2 * k);
#pragma unroll
        for (int i = 0; i < Q; ++i)
#pragma unroll
            for (int j = 0; j < Q; ++j) {
                const int ti = Q * si + i, tj = Q * sj + j;
                if (tj <= ti) *reinterpret_cast<double2 *>(G + tile_index(ti, tj) * TILE_ELEMS) = make_double2(acc[i][j][0], acc[i][j][1]);
            }
    }
}

template <typename Tin>
static void launch_gram_exact_as(const Tin *blocks, int64_t nb, int n, double *gram, const int *list, const int *count, int sm_count, cudaStream_t s) {
    // squares of 2 x 2 tiles as long as the blocks alone do not fill the SMs (two CTAs of squares of 4 x 4 each)
    if (nb >= 2 * static_cast<int64_t>(sm_count)) {
        launch_dependent(gram_exact_kernel<Tin, 4>, dim3(static_cast<unsigned>(std::min<int64_t>(nb, 2 * static_cast<int64_t>(sm_count)))), 320, 0, s, blocks, n, gram,
                         static_cast<int>(nb), list, count);
    } else {
        launch_dependent(gram_exact_kernel<Tin, 2>, dim3(static_cast<unsigned>(nb), 9), 128, 0, s, blocks, n, gram, static_cast<int>(nb), list, count);
    }
}

void launch_gram_exact(const void *blocks, int in_dtype, int64_t nb, int n, double *gram, const int *list, const int *count, int sm_count, cudaStream_t s) {
    if (in_dtype == EOSQ_F32) launch_gram_exact_as(static_cast<const float *>(blocks), nb, n, gram, list, count, sm_count, s);
    else launch_gram_exact_as(static_cast<const __half *>(blocks), nb, n, gram, list, count, sm_count, s);
}

// ------------------------------------------------------------------------------------------
// 32 x 128 by 128 x 128 tile product of the quantiser:
// warp w owns rows 4w..4w+3 of the tile, lane l owns columns 4l..4l+3.
// ------------------------------------------------------------------------------------------
constexpr int TILE_ROWS = 32;

__device__ __forceinline__ void tile_gemm(const float (*tile)[D], const float *Bm, int warp, int lane,
                                          float acc[4][4]) {
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = 0.0f;
#pragma unroll 2
    for (int j = 0; j < D; j += 4) {
        float av[4][4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float4 a = *reinterpret_cast<const float4 *>(&tile[4 * warp + r][j]);
            av[r][0] = a.x;
            av[r][1] = a.y;
            av[r][2] = a.z;
            av[r][3] = a.w;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 bv = *reinterpret_cast<const float4 *>(Bm + (j + q) * D + 4 * lane);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                acc[r][0] = fmaf(av[r][q], bv.x, acc[r][0]);
                acc[r][1] = fmaf(av[r][q], bv.y, acc[r][1]);
                acc[r][2] = fmaf(av[r][q], bv.z, acc[r][2]);
                acc[r][3] = fmaf(av[r][q], bv.w, acc[r][3]);
            }
        }
    }
}

// ------------------------------------------------------------------------------------------
// Residual, norm, rotation, code, pack (Algorithm 3 lines 4-9; Algorithm 1).
// The residual is never formed: rows of Y = R Pi^T are computed as S M with
//   M[j][c] = Pi[c][j] - sum_i coef_i zeta_i[j] (Pi zeta_i)[c],
// rho_t = ||y_t|| (Pi is orthogonal), z = y / rho, code = #thresholds below z.
//
// With few blocks (the calls this kernel is for) the chain to M is what bounds it.  Pi^T comes into shared memory
// while the kernel before is still running, and M is made in place: a thread has one column of W in registers
// and takes four rows at a time, so that no load of its chain waits for another (one element after the other, Pi from
// global memory: 39 us for two blocks of 256 tokens, now 21).
// ------------------------------------------------------------------------------------------
constexpr size_t QUANT_DYN_SMEM = sizeof(float) * (D * D + TILE_ROWS * D + 2 * RMAX * D);

__global__ void __launch_bounds__(256) quant_plain_kernel(const float *blocks, int n, Workspace ws,
                                                          const float *__restrict__ pi_t, Codebook cb,
                                                          eosq_cache_t out, long long block0) {
    extern __shared__ __align__(16) float qs[];
    float *M = qs;                                                         // [D][D]   M[j][c]
    float(*tile)[D] = reinterpret_cast<float(*)[D]>(qs + D * D);           // [32][D]
    float *Vc = qs + D * D + TILE_ROWS * D;                                // [RMAX][D] coef_i zeta_i[j]
    float *W = Vc + RMAX * D;                                              // [RMAX][D] (Pi zeta_i)[c]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = blockIdx.x;
    const long long gb = block0 + b;
#pragma unroll
    for (int e = tid; e < D * D / 4; e += 256) reinterpret_cast<float4 *>(M)[e] = __ldg(reinterpret_cast<const float4 *>(pi_t) + e);
    pdl_wait();
    const int rank = ws.rank[b];
    const float *S = blocks + static_cast<size_t>(gb) * n * D;

    // everything that has to come from memory is asked for at once: the first tile of tokens, V (zero beyond the rank), the coefficients
    auto fetch_tile = [&](int r0) {
#pragma unroll
        for (int e = tid; e < TILE_ROWS * D / 4; e += 256) {
            const int r = e / (D / 4), j = 4 * (e % (D / 4));
            if (r0 + r < n) cp_async16(reinterpret_cast<const double *>(&tile[r][j]), reinterpret_cast<const double *>(S + static_cast<size_t>(r0 + r) * D + j));
            else *reinterpret_cast<float4 *>(&tile[r][j]) = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
    };
    const int first_row = blockIdx.y * TILE_ROWS;
    if (first_row < n) fetch_tile(first_row);
    float coef[RMAX * D / 256];
#pragma unroll
    for (int k = 0; k < RMAX * D / 256; ++k) coef[k] = ws.coef[static_cast<size_t>(b) * RMAX + (tid + 256 * k) / D];
#pragma unroll
    for (int e = tid; e < RMAX * D; e += 256) Vc[e] = ws.vr[static_cast<size_t>(b) * RMAX * D + e];
    __syncthreads();
    const int c = tid & (D - 1), half = tid >> 7;
    {   // W[i][c] = sum_j Pi[c][j] zeta_i[j]
        float w[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] = 0.0f;
        if (8 * half < rank) {
#pragma unroll 4
            for (int j = 0; j < D; j += 4) {
                const float p0 = M[j * D + c], p1 = M[(j + 1) * D + c], p2 = M[(j + 2) * D + c], p3 = M[(j + 3) * D + c];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float4 v = *reinterpret_cast<const float4 *>(Vc + (8 * half + i) * D + j);
                    w[i] = fmaf(p3, v.w, fmaf(p2, v.z, fmaf(p1, v.y, fmaf(p0, v.x, w[i]))));
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) W[(8 * half + i) * D + c] = w[i];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < RMAX * D / 256; ++k) Vc[tid + 256 * k] *= coef[k];
    __syncthreads();
    {
        float w[RMAX];
#pragma unroll
        for (int i = 0; i < RMAX; ++i) w[i] = W[i * D + c];
#pragma unroll 2
        for (int j = half * (D / 2); j < (half + 1) * (D / 2); j += 4) {
            float m0 = M[j * D + c], m1 = M[(j + 1) * D + c], m2 = M[(j + 2) * D + c], m3 = M[(j + 3) * D + c];
#pragma unroll
            for (int i0 = 0; i0 < RMAX; i0 += 4)
                if (i0 < rank) {   // (factors past the rank are zeros)
#pragma unroll
                    for (int i = i0; i < i0 + 4; ++i) {
                        const float4 v = *reinterpret_cast<const float4 *>(Vc + i * D + j);
                        m0 = fmaf(-v.x, w[i], m0);
                        m1 = fmaf(-v.y, w[i], m1);
                        m2 = fmaf(-v.z, w[i], m2);
                        m3 = fmaf(-v.w, w[i], m3);
                    }
                }
            M[j * D + c] = m0;
            M[(j + 1) * D + c] = m1;
            M[(j + 2) * D + c] = m2;
            M[(j + 3) * D + c] = m3;
        }
    }

    const int nthr = (1 << cb.bits) - 1;
    const int chunk_bits = 4 * cb.bits;       // bits contributed by one lane (4 coordinates)
    const int row_words = 4 * cb.bits;        // 128 * bits / 32
    for (int r0 = first_row; r0 < n; r0 += gridDim.y * TILE_ROWS) {
        if (r0 > first_row) {
            __syncthreads();
            fetch_tile(r0);
        }
        cp_async_wait_all();
        __syncthreads();
        float acc[4][4];
        tile_gemm(tile, M, warp, lane, acc);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int row = r0 + 4 * warp + r;
            float ss = acc[r][0] * acc[r][0] + acc[r][1] * acc[r][1] + acc[r][2] * acc[r][2] + acc[r][3] * acc[r][3];
            ss = warp_sum(ss);
            const float rho = sqrtf(ss);
            unsigned chunk = 0u;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float z = (rho > 0.0f) ? acc[r][c] / rho : 0.0f;
                unsigned code = 0u;
                for (int t = 0; t < nthr; ++t) code += (cb.threshold[t] < z) ? 1u : 0u;
                chunk |= code << (c * cb.bits);
            }
            // lane l holds bits [l*chunk_bits, (l+1)*chunk_bits) of the row; lane w assembles word w
            unsigned word = 0u;
            const int first = (32 * lane) / chunk_bits;
#pragma unroll
            for (int s = 0; s < 9; ++s) {
                const int src = first + s;
                const unsigned other = __shfl_sync(0xffffffffu, chunk, src & 31);
                const int pos = src * chunk_bits - 32 * lane;
                if (src < 32 && pos < 32) word |= (pos >= 0) ? (other << pos) : (other >> (-pos));
            }
            if (row < n) {
                if (lane < row_words)
                    reinterpret_cast<unsigned *>(out.codes)[(static_cast<size_t>(gb) * n + row) * row_words + lane] = word;
                if (lane == 0) out.norms[static_cast<size_t>(gb) * n + row] = __half_as_ushort(__float2half_rn(rho));
            }
        }
        // left factors P[i][t] = coef_i <s_t, zeta_i>
        for (int e = tid; e < TILE_ROWS * RMAX; e += 256) {
            const int i = e / TILE_ROWS, r = e % TILE_ROWS;
            if (i < rank && r0 + r < n) {
                float p[4] = {0.0f, 0.0f, 0.0f, 0.0f};   // (four sums side by side)
#pragma unroll 2
                for (int j = 0; j < D; j += 4)
#pragma unroll
                    for (int q = 0; q < 4; ++q) {   // (a different column per row: the rows start in the same bank)
                        const int jr = (j + q + r) & (D - 1);
                        p[q] = fmaf(tile[r][jr], Vc[i * D + jr], p[q]);
                    }
                out.P[(static_cast<size_t>(gb) * RMAX + i) * n + r0 + r] = __half_as_ushort(__float2half_rn((p[0] + p[1]) + (p[2] + p[3])));
            }
        }
    }
}

void launch_quant_plain(const float *blocks, int64_t nb, int n, const Workspace &ws,
                        const Rotation &rot, const Codebook &cb, const eosq_cache_t &out, int64_t block0, int sm_count,
                        cudaStream_t s) {
    ensure_dynamic_smem(reinterpret_cast<const void *>(quant_plain_kernel), QUANT_DYN_SMEM);
    // few blocks: their tiles are dealt out to several CTAs each (every one builds the block's matrix M for itself,
    // which costs about as much as two tiles) as long as that fills SMs that would stay idle
    const int64_t tiles = (n + TILE_ROWS - 1) / TILE_ROWS;
    const unsigned parts = static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>(tiles, 2 * static_cast<int64_t>(sm_count) / nb)));
    const dim3 grid(static_cast<unsigned>(nb), parts);
    launch_dependent(quant_plain_kernel, grid, 256, QUANT_DYN_SMEM, s, blocks, n, ws, rot.pi_t, cb, out, static_cast<long long>(block0));
}

}  // namespace eosq
