// Double-precision pieces shared by the spectral kernels: the 8 x 8 tile layout of the Gram matrices, the
// fp64 tensor-core instruction, and the two reciprocals that sit on every reflector's critical path.
#pragma once

#include <cstdint>

namespace eosq {

// ---- tile layout ------------------------------------------------------------------------------
// A symmetric d x d matrix is kept as the 8 x 8 tiles (I, J), I >= J, of its lower half, tile (I, J) at
// index I (I + 1) / 2 + J, 64 doubles each.  Inside a tile the rows and the halves of a row are permuted so
// that shared memory serves every way the tensor instruction's operands are read without bank conflicts:
// lane (m, k) = (lane / 4, lane % 4) takes columns 2k, 2k + 1 of row m (16 bytes), or column k or 4 + k of
// row m, or column m of row k or 4 + k (8 bytes).
constexpr int TILE_DIM = 8, TILE_ELEMS = 64, GRAM_TILE_ROWS = 128 / TILE_DIM;
constexpr int GRAM_TILES = GRAM_TILE_ROWS * (GRAM_TILE_ROWS + 1) / 2;   // 136
constexpr int GRAM_ELEMS = GRAM_TILES * TILE_ELEMS;                     // 8704 doubles, 68 KB
__host__ __device__ __forceinline__ int tile_row(int r) { return (r ^ ((r >> 1) & 1)) * 8; }
__host__ __device__ __forceinline__ int tile_flip(int r) { return r & 2; }   // XOR on a row's 16-byte chunks
__host__ __device__ __forceinline__ int tile_off(int r, int c) { return tile_row(r) + ((((c >> 1) ^ tile_flip(r)) << 1) | (c & 1)); }
__host__ __device__ __forceinline__ int tile_index(int ti, int tj) { return ti * (ti + 1) / 2 + tj; }

// ---- the band ---------------------------------------------------------------------------------
// Bandwidth 4: block p (rows and columns 4p .. 4p + 3) has its 4 x 4 diagonal block at 32 p and the 4 x 4 block
// below it (upper triangular) at 32 p + 16, both row-major.
constexpr int BAND_W = 4, BAND_BLOCKS = 128 / BAND_W, BAND_ELEMS = BAND_BLOCKS * 32;

// ---- reflectors of the bulge chasing -------------------------------------------------------------
// Sweep s, hop h has one reflector on rows s + 1 + 4 h .. s + 4 + 4 h.  They are packed by sweep in chunks of
// eight rows (two hops): the sweeps with the same (s + 2) / 8 have the same number of chunks, 8700 doubles in
// all.  Within chunk q row r (0 .. 7) sits at sweep_pos: the 16-byte pieces are permuted with q so that
// 32 lanes, two per chunk, read a sweep from shared memory without bank conflicts, 16 bytes at a time.
constexpr int SWEEPS = 126;
__host__ __device__ __forceinline__ int sweep_chunks(int s) { return GRAM_TILE_ROWS - ((s + 2) >> 3); }
__host__ __device__ __forceinline__ int sweep_group_offset(int g) { return 64 * (g * GRAM_TILE_ROWS - g * (g - 1) / 2); }
__host__ __device__ __forceinline__ int sweep_offset(int s) {
    const int g = (s + 2) >> 3;
    return sweep_group_offset(g) + ((s + 2) & 7) * 8 * (GRAM_TILE_ROWS - g);
}
__host__ __device__ __forceinline__ int sweep_pos(int q, int r) { return (((r >> 1) ^ ((q >> 1) & 3)) << 1) | (r & 1); }

#ifdef __CUDACC__
// D += A B of an 8 x 4 and a 4 x 8 matrix in double precision.  Lane (m, k) = (lane / 4, lane % 4) gives A[m][k]
// and B[k][m] and holds D[m][2k], D[m][2k + 1]: element by element an accumulator is a valid A operand of
// the next product (columns in the order 0 2 4 6, then 1 3 5 7).  It runs at the rate of the plain
// multiply-adds (64 per clock and SM, measured) with an eighth of the instructions and no operand traffic
// between lanes, and a dependent one follows after 26 cycles, which beats a shuffle and an addition (43)
// even for sums over a warp.
__device__ __forceinline__ void dmma(double (&c)[2], double a, double b) {
    asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};" : "+d"(c[0]), "+d"(c[1]) : "d"(a), "d"(b));
}

// 16 bytes from global to shared memory without a register in between.
__device__ __forceinline__ void cp_async16(const double *dst, const double *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait_group() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The two refinements below start from the hardware's estimates, good to about 2^-20, and add the next two terms of a
// power series in their residual e (Householder's iterations of third order), so that what is left is of order e^3, below
// the rounding:
//   1 / x        = r / (1 - e),        e = 1 - x r:    r (1 + e + e^2)             next term e^3         2^-60
//   1 / sqrt(x)  = y (1 - e)^(-1/2),   e = 1 - x y^2:  y (1 + e / 2 + 3 e^2 / 8)   next term 5 e^3 / 16  2^-58
// They are shorter than CUDA's division and rsqrt, and sit on chains of dependent operations.  The estimates flush subnormal
// numbers to zero.
__device__ __forceinline__ double sp_rcp(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

// The normalised reflector H = I - u u^T (u . u = 2) that takes x to beta e_1: from alpha = x_1 and
// ss = sum of the other squares, beta = -sign(alpha) ||x||, u_1 = (alpha - beta) g, u_j = x_j g.  g = 0 (H = I)
// when there is nothing to annihilate, or nothing whose square is a normal number (the chasing's fill-in can decay by
// any factor from hop to hop).  The second root's estimate is started from the first one's, so that the two table
// look-ups overlap the refinements.
__device__ __forceinline__ void make_reflector(double alpha, double ss, double &beta, double &g, double &amb) {
    const double aa = fabs(alpha);
    const double sq = fma(alpha, alpha, ss);
    double y0, z0;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y0) : "d"(sq));
    const double n0 = sq * y0;
    const double w0 = fma(aa, n0, sq);
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(z0) : "d"(w0));
    const double e = fma(-n0, y0, 1.0);
    const double nrm = fma(n0 * e, fma(0.375, e, 0.5), n0);
    const double w = fma(aa, nrm, sq);              // beta (beta - alpha)
    const double e2 = fma(-w * z0, z0, 1.0);
    const double gg = fma(z0 * e2, fma(0.375, e2, 0.5), z0);
    const bool live = ss > 0.0 && sq >= 2.2250738585072014e-308;   // the smallest normal number
    const double sb = __hiloint2double(__double2hiint(nrm) | (~__double2hiint(alpha) & 0x80000000), __double2loint(nrm));   // -sign(alpha) nrm
    beta = live ? sb : alpha;
    g = live ? gg : 0.0;
    amb = alpha - beta;
}
#endif

}  // namespace eosq
