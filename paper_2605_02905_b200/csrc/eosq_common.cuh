// Shared declarations of the eosq CUDA library (sm_100a): constants, the context, the
// workspace view and the kernel launchers implemented in the other translation units.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <vector>

#include "eosq.h"
#include "eosq_fp64.cuh"

namespace eosq {

constexpr int D = 128;         // head dimension the kernels are written for
constexpr int RMAX = EOSQ_RMAX;
constexpr int KPILOT = 11;     // floor(128^(1/2.01)), checked against eosq_pilot_k at create time
constexpr int NMAX = 4096;

// Lloyd-Max codebook as kernel parameter (fp32 copies of the host doubles).
struct Codebook {
    float centroid[16];
    float threshold[15];
    int bits;
};

// Device copies of one seeded rotation.
struct Rotation {
    uint64_t seed = 0;
    float *pi = nullptr;     // [c][j]  z_c = sum_j pi[c][j] u_j
    float *pi_t = nullptr;   // [j][c]
};

// Scratch of one chunk of blocks, carved out of the caller's workspace.
struct Workspace {
    double *gram;   // [C][136][64] lower half of the Gram matrix in 8 x 8 tiles (eosq_fp64.cuh); the band reduction leaves its
                    //             panels' reflectors V there, two panels to a tile column
    double *band;   // [C][32][32] the band matrix (bandwidth 4)
    double *tmat;   // [C][16][64] T of each pair of panels (Q = I - V T V^T)
    double *q2;     // [C][136][64] reflectors of the bulge chasing (sweep_offset)
    double *diag;   // [C][D]      tridiagonal diagonal
    double *off;    // [C][D]      tridiagonal off-diagonal (D-1 used)
    double *lam;    // [C][D]      eigenvalues, descending
    float *vr;      // [C][RMAX][D] right vectors as used for the residual
    float *coef;    // [C][RMAX]   phi_i / sigma_i
    int *rank;      // [C]
    int *redo_list; // [C]         blocks whose spectrum the tensor-core Gram matrix cannot resolve
    int *redo_count;// [1]
};

constexpr size_t WS_PER_BLOCK = sizeof(double) * (2 * GRAM_ELEMS + BAND_ELEMS + GRAM_TILE_ROWS * TILE_ELEMS + 3 * D) + sizeof(float) * (RMAX * D + RMAX) + 64 + 8;
// A block is redone with the exact (double precision) Gram matrix when its smallest eigenvalue is
// below this fraction of its largest: the tensor-core Gram matrix carries an absolute error of
// about 1e-8 of the largest eigenvalue, which would move smaller singular values by more than
// 5e-5 relative.
constexpr double REDO_RATIO = 1e-4;
// Blocks of at most this many tokens take the exact Gram matrix at once: the shorter a block, the closer its smallest
// singular values are to zero, and on caches with strong outliers nearly every block of up to 208 tokens, four
// fifths of those of 256 and a quarter of those of 320 would come back for the second pass, whose
// tridiagonalisation costs five times what the exact Gram matrix of such a block does.
constexpr int EXACT_GRAM_MAX_N = 320;
constexpr int64_t CHUNK_BLOCKS = 18944;  // 128 per SM on 148 SMs.  Every kernel here gives a block to one CTA, team or warp whose
                                        // steps are chains of latencies, so throughput comes from blocks in flight: a 16384-block
                                        // cache went from 18.9 ms in chunks of 1184 to 17.1 ms in one chunk (3.2 GB of scratch now).

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Raises a kernel's dynamic shared-memory limit, once per kernel and device (the attribute belongs
// to the device's copy of the function, so a second GPU in the same process needs its own call).
// Implemented in eosq_api.cu.
bool ensure_dynamic_smem(const void *kernel, size_t bytes);

// Launches a kernel that may start while its predecessor on the stream drains (programmatic dependent launch): its
// set-up runs ahead, and pdl_wait() holds it until the predecessor has finished and its results are visible.  Every
// thread of such a kernel calls pdl_wait() before it touches anything the stream's earlier work reads or writes; a
// kernel therefore runs no earlier than its predecessor's predecessor has finished.  What earlier work writes is read by
// ordinary loads through pointers that are not __restrict__: read-only loads and restricted pointers promise that nobody
// else writes the memory meanwhile, and the compiler may move them across the wait.  The successor may start when
// every CTA has ended or called pdl_trigger().  Only kernels whose successor holds one CTA per SM call that early:
// smaller CTAs would be packed onto the few SMs that are free at that moment and stay there (it made a call over
// 4096 blocks 5 % slower).  (An encode is a dozen dependent kernels: the gaps between them were 25 us of a
// 16-block call's 390.)
template <typename... P, typename... A>
inline void launch_dependent(void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t s, A &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);   // an error stays in cudaGetLastError
}
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif

// Carve the scratch arrays of one chunk (capacity `cap` blocks) out of `base`; returns the bytes
// used.  With base = nullptr only the size is computed.
inline size_t carve(void *base, int64_t cap, Workspace *ws) {
    char *p = static_cast<char *>(base);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        void *q = p ? p + off : nullptr;
        off = align_up(off + bytes, 256);
        return q;
    };
    Workspace w;
    w.gram = static_cast<double *>(take(sizeof(double) * cap * GRAM_ELEMS));
    w.band = static_cast<double *>(take(sizeof(double) * cap * BAND_ELEMS));
    w.tmat = static_cast<double *>(take(sizeof(double) * cap * GRAM_TILE_ROWS * TILE_ELEMS));
    w.q2 = static_cast<double *>(take(sizeof(double) * cap * GRAM_ELEMS));
    w.diag = static_cast<double *>(take(sizeof(double) * cap * D));
    w.off = static_cast<double *>(take(sizeof(double) * cap * D));
    w.lam = static_cast<double *>(take(sizeof(double) * cap * D));
    w.vr = static_cast<float *>(take(sizeof(float) * cap * RMAX * D));
    w.coef = static_cast<float *>(take(sizeof(float) * cap * RMAX));
    w.rank = static_cast<int *>(take(sizeof(int) * cap));
    w.redo_list = static_cast<int *>(take(sizeof(int) * cap));
    w.redo_count = static_cast<int *>(take(sizeof(int)));
    if (ws) *ws = w;
    return off;
}

}  // namespace eosq

enum Stage { ST_GRAM = 0, ST_TRIDIAG_A, ST_TRIDIAG_B, ST_TRIDIAG_C, ST_EIGVALS, ST_SPECTRAL, ST_QUANT, ST_DECODE, ST_SCORES, ST_REDO, ST_OTHER };

struct eosq_ctx {
    struct Timed {
        int stage;
        cudaEvent_t start, stop;
    };
    int device = 0;
    int sm_count = 148;
    int *dev_err = nullptr;   // device word: bits raised by kernels whose bounded waits gave up
    std::vector<eosq::Rotation> rotations;
    eosq::Codebook codebooks[5] = {};   // by code width; bits == 0: not made yet
    std::string last_error;
    int64_t launches = 0;
    uint32_t profile_mask = 0;   // bit i set: launches of stage i are bracketed by events
    std::vector<Timed> timed;
    std::vector<cudaEvent_t> free_events;
    void *scores_w = nullptr;        // score path: per-head images of the operand W = Pi q (grown on demand)
    size_t scores_w_bytes = 0;
    // host-buffer path: copy streams and hand-over events of its two arena slots (created on first use)
    cudaStream_t copy_in = nullptr, copy_out = nullptr;
    cudaEvent_t ev_start = nullptr, ev_in[2] = {nullptr, nullptr}, ev_done[2] = {nullptr, nullptr}, ev_out[2] = {nullptr, nullptr};
};

namespace eosq {

// The launch sequence of the encode path for blocks [b0, b0 + nb) of `blocks` (implemented with
// the C entry points; shared by eosq_encode and eosq_encode_static).
int encode_chunk(eosq_ctx *ctx, const void *blocks, int in_dtype, int64_t b0, int64_t nb, int n, int bits,
                 const Rotation &rot, const Codebook &cb, const eosq_cache_t &out_all, const Workspace &ws,
                 cudaStream_t s);

// The codebook of a code width, made once per context (the Lloyd iteration takes up to 0.2 ms of host time).
int get_codebook(eosq_ctx *ctx, int d, int bits, Codebook *cb);

// ---- launchers (each enqueues one kernel on `stream`) ---------------------------------------
// Gram matrix G = S^T S of each block, accumulated in double from exact products.
// With `list` given, the blocks list[0 .. *count) are worked on (same for the spectral launchers below): grids are
// those of a full launch, an empty list ends them at once.
void launch_gram_exact(const void *blocks, int in_dtype, int64_t nb, int n, double *gram, const int *list, const int *count, int sm_count,
                       cudaStream_t s);
// Same result from the tensor cores (fp16 blocks only); also empties the queue of blocks for the second pass.  The chunk starts `block0` blocks into
// `blocks_all`.  Returns false if the launch could not be set up (no kernel was enqueued).
bool launch_gram_tc(const void *blocks_all, int64_t block0, int64_t nb, int n, double *gram, int *redo_count,
                    int *err, int sm_count, cudaStream_t s);
// Full matrix -> band (in place: the panels' reflectors overwrite it; in band_launches() launches, part 0, 1, ..) -> tridiagonal.
int band_launches(int64_t nb, bool listed, int sm_count);
void launch_band(int part, int64_t nb, const Workspace &ws, const int *list, const int *count, int sm_count, cudaStream_t s);
void launch_chase(int64_t nb, const Workspace &ws, const int *list, const int *count, int sm_count, cudaStream_t s);
// Eigenvalues of each tridiagonal matrix: with `full` all of them, otherwise the 32 to 34 largest (what Algorithm 2
// reads one by one).  Every block whose eigenvalue range exceeds 1 / REDO_RATIO goes to `mark_list`, if there is one.
void launch_eigvals(int64_t nb, const Workspace &ws, const int *list, const int *count, int *mark_list, bool full, int sm_count, cudaStream_t s);
// Bulk edge, rank, imputed spectrum, D-transform and shrinkage; kept eigenvectors.
void launch_spectral(int64_t nb, int n, const Workspace &ws, const eosq_cache_t &out, int64_t block0, bool full, int sm_count,
                     cudaStream_t s);
// Residual, norm, rotation, codes, packing and left factors of fp32 blocks.
void launch_quant_plain(const float *blocks, int64_t nb, int n, const Workspace &ws,
                        const Rotation &rot, const Codebook &cb, const eosq_cache_t &out, int64_t block0, int sm_count,
                        cudaStream_t s);
// Same outputs from the tensor cores (fp16 blocks only); `out` is already offset to the chunk.
bool launch_quant_tc(const void *blocks_all, int64_t block0, int64_t nb, int n, const Workspace &ws, const Rotation &rot,
                     const Codebook &cb, const eosq_cache_t &out, int *err, int sm_count, cudaStream_t s);
bool decode_tc_supported(const eosq_cache_t &cache, int bits, const void *out_blocks);
bool launch_decode_tc(const eosq_cache_t &cache, int64_t nb, int n, const Rotation &rot, const Codebook &cb, void *out_blocks,
                      int out_dtype, int *err, int sm_count, cudaStream_t s);
// Attention logits on the tensor cores; `supported` checks the 16-byte alignment the kernel's bulk copies
// need, the launcher returns false if nothing was enqueued.
bool scores_tc_supported(const eosq_cache_t &cache, int bits, int n);
bool launch_scores_tc(const eosq_cache_t &cache, int64_t heads, int64_t bph, int64_t head_stride, int n, const Rotation &rot,
                      const Codebook &cb, const __half *q, int G, float scale, float *scores, int *err, int sm_count,
                      void **scratch, size_t *scratch_bytes, int64_t *kernels, cudaStream_t s);

// ---- work shares ------------------------------------------------------------------------------
// The tiles of `nb` blocks of `tiles` tiles each, dealt out to `ctas` CTAs as runs of tiles [t0, t1) of one block.  First
// whole blocks in turn (neighbouring CTAs work on neighbouring blocks), as long as every CTA gets one; what is left,
// less than a block per CTA, in equal shares of consecutive tiles.  (Whole blocks to the end would leave most
// SMs idle on few blocks and some with one block more than the others on many: 512 blocks of 32 tiles lose 15 %.)
struct TileRuns {
    int tiles, cta, ctas, whole, count, rest_block;
    long long g_first, g_end;   // share of the rest, in tiles from the start of block `rest_block`'s round
#ifdef __CUDACC__
    __device__ __forceinline__ TileRuns(int nb, int tiles_, int cta_, int ctas_) : tiles(tiles_), cta(cta_), ctas(ctas_) {
        whole = nb / ctas;
        const int base = whole * ctas;
        const long long rest = static_cast<long long>(nb - base) * tiles;
        g_first = rest * cta / ctas;
        g_end = rest * (cta + 1) / ctas;
        rest_block = base + static_cast<int>(g_first / tiles);
        count = whole + ((g_end > g_first) ? base + static_cast<int>((g_end - 1) / tiles) - rest_block + 1 : 0);
        g_first -= static_cast<long long>(rest_block - base) * tiles;   // relative to rest_block's first tile
        g_end -= static_cast<long long>(rest_block - base) * tiles;
    }
    __device__ __forceinline__ int block(int i) const { return (i < whole) ? i * ctas + cta : rest_block + (i - whole); }
    __device__ __forceinline__ void get(int i, int &b, int &t0, int &t1) const {
        b = block(i);
        t0 = 0;
        t1 = tiles;
        if (i >= whole) {
            const int start = (i - whole) * tiles;   // (the rest is less than ctas blocks)
            t0 = max(static_cast<int>(g_first) - start, 0);
            t1 = min(static_cast<int>(g_end) - start, tiles);
        }
    }
    __device__ __forceinline__ int total() const { return whole * tiles + static_cast<int>(g_end - g_first); }
#endif
};

// ---- small device helpers -------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ float to_float(float v) { return v; }
__device__ __forceinline__ float to_float(__half v) { return __half2float(v); }

void launch_wait_timeout(int *err, uint32_t polls, cudaStream_t s);

}  // namespace eosq
