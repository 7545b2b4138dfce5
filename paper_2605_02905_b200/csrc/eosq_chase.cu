// Second half of the tridiagonalisation: bandwidth 4 -> tridiagonal by bulge chasing, in double precision,
// with the whole band in registers.
//
// Sweep s annihilates column s below its first off-diagonal entry with a reflector on rows s + 1 .. s + 4 and
// chases the fill-in down the band in hops of four rows.  Hop h of sweep s works on the window i0 = s + 1 + 4 h:
// with the reflector u of rows i0 .. i0 + 3,
//     D <- H D H           (D: rows and columns i0 .. i0 + 3)
//     B <- B H             (B: rows i0 + 4 .. i0 + 7, the same columns)
//     v from B's first column,  B <- H_v B,  v goes to hop h + 1.
// Hop h of sweep s needs hop h - 1 of the same sweep (its reflector) and hop h + 1 of sweep s - 1 (what has
// become final next to its window), so hop h runs sweep s at time step 2 s + h: some 250 steps per matrix
// instead of 2000 hops one after the other.
//
// Mapping.  A lane owns hops 2 g and 2 g + 1 (one runs at even steps, the other at odd ones), sixteen lanes a
// matrix, a warp two: the 4 x 4 blocks D (lower half) and B of a hop are one thread's registers, so a hop
// has no reductions over lanes, no shared memory and no barriers, and a lane's share of the band never
// leaves its registers.  When the window moves on by a row its entries move by one register, which the last
// update of a hop does by writing its results one place up; what comes in at the edge is the first column
// of D, and the first entry of B, that hop h + 1 left behind one step earlier (five shuffles, and four for
// the reflector that goes the other way).  The first reflector of the next sweep is worked out in the odd steps
// next to another hop, off every chain.
//
// A zero-padded matrix needs no bounds: reflectors of zero vectors are zero.
#include <algorithm>
#include <type_traits>

#include "eosq_common.cuh"
#include "eosq_fp64.cuh"

namespace eosq {

namespace {

constexpr int CH_WARPS = 2, CH_LANES = 16, CH_HOPS = D / BAND_W;   // 32 hops

// The state of one hop: its window, shifted for the sweep to come (the entries that are still to come from
// the neighbour are missing), and what it hands on.
struct ChHop {
    double d[4][4];   // lower half: d[a][b], b <= a
    double b[4][4];
    double x[4];      // first column of D that the last sweep left
    double beta;      // first entry of B that it left
};

// One hop with reflector u; `xn`, `bn`: the neighbour's x and beta.  v: the reflector for the next hop.
__device__ __forceinline__ void ch_hop(ChHop &H, const double (&u)[4], const double (&xn)[4], double bn, double (&v)[4]) {
    double d[4][4], b[4][4];
    // the window, complete
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (j <= i) d[i][j] = H.d[i][j];
            b[i][j] = H.b[i][j];
        }
    d[3][3] = xn[0];
#pragma unroll
    for (int i = 0; i < 3; ++i) b[i][3] = xn[i + 1];
    b[3][0] = b[3][1] = b[3][2] = 0.0;
    b[3][3] = bn;
    // B <- B H
    double w[4];
#pragma unroll
    for (int i = 0; i < 3; ++i) w[i] = fma(b[i][1], u[1], b[i][0] * u[0]) + fma(b[i][3], u[3], b[i][2] * u[2]);
    w[3] = b[3][3] * u[3];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
        for (int i = 0; i < 3; ++i) b[i][j] = fma(-w[i], u[j], b[i][j]);
        b[3][j] = (j == 3) ? fma(-w[3], u[3], b[3][3]) : -w[3] * u[j];
    }
    // v from the first column
    const double ss = fma(b[3][0], b[3][0], fma(b[2][0], b[2][0], b[1][0] * b[1][0]));
    double beta, g, amb;
    make_reflector(b[0][0], ss, beta, g, amb);
    // D <- H D H (in the shadow of the roots)
    double p[4];
    p[0] = fma(d[1][0], u[1], d[0][0] * u[0]) + fma(d[3][0], u[3], d[2][0] * u[2]);
    p[1] = fma(d[1][1], u[1], d[1][0] * u[0]) + fma(d[3][1], u[3], d[2][1] * u[2]);
    p[2] = fma(d[2][1], u[1], d[2][0] * u[0]) + fma(d[3][2], u[3], d[2][2] * u[2]);
    p[3] = fma(d[3][1], u[1], d[3][0] * u[0]) + fma(d[3][3], u[3], d[3][2] * u[2]);
    const double k2 = -0.5 * (fma(p[1], u[1], p[0] * u[0]) + fma(p[3], u[3], p[2] * u[2]));
    double q[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) q[i] = fma(k2, u[i], p[i]);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j <= i; ++j) d[i][j] = fma(-q[i], u[j], fma(-u[i], q[j], d[i][j]));
    // B <- H_v B
    double f[4];
#pragma unroll
    for (int j = 1; j < 4; ++j) {
        const double t = fma(b[3][0], b[3][j], fma(b[2][0], b[2][j], b[1][0] * b[1][j]));
        f[j] = g * fma(amb, b[0][j], t);
    }
    v[0] = amb * g;
#pragma unroll
    for (int i = 1; i < 4; ++i) v[i] = b[i][0] * g;
    // results one place up
#pragma unroll
    for (int i = 0; i < 4; ++i) H.x[i] = d[i][0];
    H.beta = beta;
#pragma unroll
    for (int i = 1; i < 4; ++i)
#pragma unroll
        for (int j = 1; j <= i; ++j) H.d[i - 1][j - 1] = d[i][j];
#pragma unroll
    for (int j = 1; j < 4; ++j) {
        H.d[3][j - 1] = fma(-v[0], f[j], b[0][j]);
#pragma unroll
        for (int i = 1; i < 4; ++i) H.b[i - 1][j - 1] = fma(-v[i], f[j], b[i][j]);
    }
}

// The window of hop h before sweep 0 (rows and columns 4 h ..), from the band.
__device__ __forceinline__ void ch_load(ChHop &H, const double *__restrict__ band, int h) {
    double d[4][4], r[4][4];
    const double2 *src = reinterpret_cast<const double2 *>(band + 32 * h);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const double2 a = src[2 * i + q];
            const double2 b = (h < CH_HOPS - 1) ? src[8 + 2 * i + q] : make_double2(0.0, 0.0);
            d[i][2 * q] = a.x;
            d[i][2 * q + 1] = a.y;
            r[i][2 * q] = (2 * q >= i) ? b.x : 0.0;
            r[i][2 * q + 1] = (2 * q + 1 >= i) ? b.y : 0.0;
        }
#pragma unroll
    for (int i = 0; i < 4; ++i) H.x[i] = d[i][0];
    H.beta = r[0][0];
#pragma unroll
    for (int i = 1; i < 4; ++i)
#pragma unroll
        for (int j = 1; j <= i; ++j) H.d[i - 1][j - 1] = d[i][j];
#pragma unroll
    for (int j = 1; j < 4; ++j) {
        H.d[3][j - 1] = r[0][j];
#pragma unroll
        for (int i = 1; i < 4; ++i) H.b[i - 1][j - 1] = r[i][j];
    }
}

__global__ void __launch_bounds__(32 * CH_WARPS) chase_kernel(const double *band, double *q2, double *diag,
                                                              double *off, int nb, const int *list,
                                                              const int *count) {
    const int lane = threadIdx.x & 31, g = lane & (CH_LANES - 1);
    pdl_wait();
    const int total = list ? *count : nb;
    const int slots = (total + 1) / 2;
    for (int w = blockIdx.x * CH_WARPS + (threadIdx.x >> 5); w < slots; w += gridDim.x * CH_WARPS) {
        // (an odd last matrix is done twice: both halves of the warp write the same values)
        const int li = min(2 * w + (lane >> 4), total - 1);
        const int blk = list ? list[li] : li;
        double *const Q = q2 + static_cast<size_t>(blk) * GRAM_ELEMS;
        double *const dd = diag + static_cast<size_t>(blk) * D, *const ee = off + static_cast<size_t>(blk) * D;
        const int pos0 = sweep_pos(g, 0), pos1 = sweep_pos(g, 2), pos2 = sweep_pos(g, 4), pos3 = sweep_pos(g, 6);
        ChHop A, B;   // hops 2 g and 2 g + 1
        ch_load(A, band + static_cast<size_t>(blk) * BAND_ELEMS, 2 * g);
        ch_load(B, band + static_cast<size_t>(blk) * BAND_ELEMS, 2 * g + 1);
        double ua[4] = {0.0, 0.0, 0.0, 0.0}, ub[4] = {0.0, 0.0, 0.0, 0.0};   // reflectors for A's and B's next hop
        // Column s + 1 as hop 0 of sweep s left it: its diagonal entry is final, the rest (D's first column and beta)
        // gives the first reflector of the next sweep.
        auto start = [&](int s, double (&u)[4]) {
            double beta, gg, amb;
            make_reflector(A.x[1], fma(A.beta, A.beta, fma(A.x[3], A.x[3], A.x[2] * A.x[2])), beta, gg, amb);
            u[0] = amb * gg;
            u[1] = A.x[2] * gg;
            u[2] = A.x[3] * gg;
            u[3] = A.beta * gg;
            if (g == 0) {
                dd[s + 1] = A.x[0];
                ee[s + 1] = beta;
            }
        };
        start(-1, ua);
        // Steps 2 k and 2 k + 1: this lane's hops are at sweep s = k - g.  `row`: where sweep s's reflectors of this
        // lane's chunk of eight rows go, while the sweep has that chunk (the piece past its last hop is a zero).
        // GUARD: the sweeps before every lane has started, where a lane that has not must keep its state.  Afterwards
        // there is nothing to guard (a window past the end of the matrix is all zeros and stays so), the two hops are
        // one straight piece of code, and what a hop does off its chain runs under the next hop's.
        auto double_step = [&](int k, auto guard) {
            constexpr bool GUARD = decltype(guard)::value;
            const int s = k - g;
            const bool started = !GUARD || s >= 0;
            const bool store = started && g < sweep_chunks(s);
            double *const row = Q + (started ? sweep_offset(s) : 0) + 8 * g;
            double v[4] = {0.0, 0.0, 0.0, 0.0}, xn[4], bn, u0[4];
            // even step: hop 2 g, its edge from this lane's odd hop
            if (store) {
                *reinterpret_cast<double2 *>(row + pos0) = make_double2(ua[0], ua[1]);
                *reinterpret_cast<double2 *>(row + pos1) = make_double2(ua[2], ua[3]);
            }
            if (started) ch_hop(A, ua, B.x, B.beta, ub);
            // odd step: hop 2 g + 1, its edge from the next lane's even hop; its reflector goes to that lane
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                xn[i] = __shfl_down_sync(0xffffffffu, A.x[i], 1, CH_LANES);
                xn[i] = (g == CH_LANES - 1) ? 0.0 : xn[i];
            }
            bn = __shfl_down_sync(0xffffffffu, A.beta, 1, CH_LANES);
            bn = (g == CH_LANES - 1) ? 0.0 : bn;
            if (store) {
                *reinterpret_cast<double2 *>(row + pos2) = make_double2(ub[0], ub[1]);
                *reinterpret_cast<double2 *>(row + pos3) = make_double2(ub[2], ub[3]);
            }
            if (started) ch_hop(B, ub, xn, bn, v);
            start(s, u0);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const double up = __shfl_up_sync(0xffffffffu, v[i], 1, CH_LANES);
                ua[i] = (g == 0) ? u0[i] : up;
            }
        };
#pragma unroll 1
        for (int k = 0; k < CH_LANES - 1; ++k) double_step(k, std::true_type());
#pragma unroll 1
        for (int k = CH_LANES - 1; k < SWEEPS; ++k) double_step(k, std::false_type());
        // hop 0 has passed the last sweep: the window's second entry is the last of the diagonal
        if (g == 0) {
            dd[D - 1] = A.d[0][0];
            ee[D - 1] = 0.0;
        }
    }
}

}  // namespace

void launch_chase(int64_t nb, const Workspace &ws, const int *list, const int *count, int sm_count, cudaStream_t s) {
    const int64_t grid = std::min<int64_t>((nb + 2 * CH_WARPS - 1) / (2 * CH_WARPS), 6 * static_cast<int64_t>(sm_count));
    launch_dependent(chase_kernel, static_cast<unsigned>(std::max<int64_t>(grid, 1)), 32 * CH_WARPS, 0, s, ws.band, ws.q2, ws.diag, ws.off, static_cast<int>(nb), list, count);
}

}  // namespace eosq
