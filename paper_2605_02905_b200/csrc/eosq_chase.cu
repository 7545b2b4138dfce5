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
struct ChD {
    double d[4][4];   // lower half: d[a][b], b <= a; the last row's first three entries come from B
    double x[4];      // first column of D that the last sweep left
};
struct ChB {
    double b[4][4];
    double beta;      // first entry of B that it left
};

// B's part of one hop with reflector u, the chain from hop to hop: B <- B H in `b`, v for the next hop.  `xn` (entries 1 .. 3), `bn`: the
// neighbour's x and beta.
__device__ __forceinline__ void ch_hop_chain(ChB &H, const double (&u)[4], const double (&xn)[4], double bn, double (&b)[4][4], double (&v)[4]) {
    // the window, complete
#pragma unroll
    for (int i = 0; i < 3; ++i) {
#pragma unroll
        for (int j = 0; j < 3; ++j) b[i][j] = H.b[i][j];
        b[i][3] = xn[i + 1];
    }
    b[3][3] = bn;
    // B <- B H
    double w[4];
#pragma unroll
    for (int i = 0; i < 3; ++i) w[i] = fma(b[i][3], u[3], fma(b[i][2], u[2], fma(b[i][1], u[1], b[i][0] * u[0])));
    w[3] = b[3][3] * u[3];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
        for (int i = 0; i < 3; ++i) b[i][j] = fma(-w[i], u[j], b[i][j]);
        b[3][j] = (j == 3) ? fma(-w[3], u[3], b[3][3]) : -w[3] * u[j];
    }
    // v from the first column
    const double ss = fma(b[3][0], b[3][0], fma(b[2][0], b[2][0], b[1][0] * b[1][0]));
    double g, amb;
    make_reflector(b[0][0], ss, H.beta, g, amb);
    v[0] = amb * g;
#pragma unroll
    for (int i = 1; i < 4; ++i) v[i] = b[i][0] * g;
}
// The rest of it, off the chain: B <- H_v B, results one place up; row: B's first row, for D's last one.
__device__ __forceinline__ void ch_hop_rest(ChB &H, const double (&b)[4][4], const double (&v)[4], double (&row)[3]) {
#pragma unroll
    for (int j = 1; j < 4; ++j) {
        const double f = fma(v[3], b[3][j], fma(v[2], b[2][j], fma(v[1], b[1][j], v[0] * b[0][j])));
        row[j - 1] = fma(-v[0], f, b[0][j]);
#pragma unroll
        for (int i = 1; i < 4; ++i) H.b[i - 1][j - 1] = fma(-v[i], f, b[i][j]);
    }
}

// D's part: D <- H D H, results one place up; xn0: the neighbour's x[0].
__device__ __forceinline__ void ch_hop_d(ChD &H, const double (&u)[4], double xn0) {
    double d[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j <= i; ++j) d[i][j] = (i < 3 || j < 3) ? H.d[i][j] : xn0;
    double p[4];
    p[0] = fma(d[3][0], u[3], fma(d[2][0], u[2], fma(d[1][0], u[1], d[0][0] * u[0])));
    p[1] = fma(d[3][1], u[3], fma(d[2][1], u[2], fma(d[1][1], u[1], d[1][0] * u[0])));
    p[2] = fma(d[3][2], u[3], fma(d[2][2], u[2], fma(d[2][1], u[1], d[2][0] * u[0])));
    p[3] = fma(d[3][3], u[3], fma(d[3][2], u[2], fma(d[3][1], u[1], d[3][0] * u[0])));
    const double k2 = -0.5 * fma(p[3], u[3], fma(p[2], u[2], fma(p[1], u[1], p[0] * u[0])));
    double q[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) q[i] = fma(k2, u[i], p[i]);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j <= i; ++j) d[i][j] = fma(-q[i], u[j], fma(-u[i], q[j], d[i][j]));
#pragma unroll
    for (int i = 0; i < 4; ++i) H.x[i] = d[i][0];
#pragma unroll
    for (int i = 1; i < 4; ++i)
#pragma unroll
        for (int j = 1; j <= i; ++j) H.d[i - 1][j - 1] = d[i][j];
}

// The window of hop h before sweep 0 (rows and columns 4 h ..), from the band.
__device__ __forceinline__ void ch_load(ChD &HD, ChB &HB, const double *band, int h) {
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
    for (int i = 0; i < 4; ++i) HD.x[i] = d[i][0];
    HB.beta = r[0][0];
#pragma unroll
    for (int i = 1; i < 4; ++i)
#pragma unroll
        for (int j = 1; j <= i; ++j) HD.d[i - 1][j - 1] = d[i][j];
#pragma unroll
    for (int j = 1; j < 4; ++j) {
        HD.d[3][j - 1] = r[0][j];
#pragma unroll
        for (int i = 1; i < 4; ++i) HB.b[i - 1][j - 1] = r[i][j];
    }
}

// Column s + 1 as hop 0 of sweep s left it (`x`, `beta`): the reflector u that starts the next sweep; returns the off-diagonal entry.
__device__ __forceinline__ double ch_start(const double (&x)[4], double beta, double (&u)[4]) {
    double e, g, amb;
    make_reflector(x[1], fma(beta, beta, fma(x[3], x[3], x[2] * x[2])), e, g, amb);
    u[0] = amb * g;
    u[1] = x[2] * g;
    u[2] = x[3] * g;
    u[3] = beta * g;
    return e;
}

__device__ __forceinline__ void ch_store(double *row, int pos, double a, double b) { *reinterpret_cast<double2 *>(row + pos) = make_double2(a, b); }

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
        ChD AD, BD;   // hops 2 g and 2 g + 1
        ChB AB, BB;
        ch_load(AD, AB, band + static_cast<size_t>(blk) * BAND_ELEMS, 2 * g);
        ch_load(BD, BB, band + static_cast<size_t>(blk) * BAND_ELEMS, 2 * g + 1);
        double ua[4] = {0.0, 0.0, 0.0, 0.0}, ub[4] = {0.0, 0.0, 0.0, 0.0};   // reflectors for A's and B's next hop
        // Column s + 1's diagonal entry is final after hop 0 of sweep s.
        auto start = [&](int s, double (&u)[4]) {
            const double e = ch_start(AD.x, AB.beta, u);
            if (g == 0) {
                dd[s + 1] = AD.x[0];
                ee[s + 1] = e;
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
                ch_store(row, pos0, ua[0], ua[1]);
                ch_store(row, pos1, ua[2], ua[3]);
            }
            double last[3], b[4][4];   // last: D's last row, which is B's first
            if (started) {
                ch_hop_chain(AB, ua, BD.x, BB.beta, b, ub);
                ch_hop_rest(AB, b, ub, last);
                ch_hop_d(AD, ua, BD.x[0]);
#pragma unroll
                for (int j = 0; j < 3; ++j) AD.d[3][j] = last[j];
            }
            // odd step: hop 2 g + 1, its edge from the next lane's even hop; its reflector goes to that lane
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                xn[i] = __shfl_down_sync(0xffffffffu, AD.x[i], 1, CH_LANES);
                xn[i] = (g == CH_LANES - 1) ? 0.0 : xn[i];
            }
            bn = __shfl_down_sync(0xffffffffu, AB.beta, 1, CH_LANES);
            bn = (g == CH_LANES - 1) ? 0.0 : bn;
            if (store) {
                ch_store(row, pos2, ub[0], ub[1]);
                ch_store(row, pos3, ub[2], ub[3]);
            }
            if (started) {
                ch_hop_chain(BB, ub, xn, bn, b, v);
                ch_hop_rest(BB, b, v, last);
                ch_hop_d(BD, ub, xn[0]);
#pragma unroll
                for (int j = 0; j < 3; ++j) BD.d[3][j] = last[j];
            }
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
            dd[D - 1] = AD.d[0][0];
            ee[D - 1] = 0.0;
        }
    }
}

// The same for few matrices, where one matrix's own time counts: two warps share a pair of matrices, one with the B windows, one with
// the D windows, the reflectors' stores and the starts of the sweeps.  A hop's chain runs through B alone, and most of what a lone
// warp spends on it is issuing the rest.  They meet once per step; what one step writes to shared memory the next one reads, so
// a barrier between them is all it takes.  Entry by entry the arithmetic is that of chase_kernel.  A hop takes 390 cycles so, 600 in one
// warp; the two warps are equally busy, at 3.6 cycles per instruction of which 1.5 are dependences and 0.4 the wait for the other.
// (A hop's last row is not needed before that hop's next turn.)
struct ChShared {
    double2 ua[2][2 * CH_LANES + 2], ub[2][2 * CH_LANES];   // reflectors for the even and the odd hops (the lane's, halves)
    double xa[4][2 * CH_LANES + 1], xb[4][2 * CH_LANES];    // x of the even hops, and the zeros next to the last one; of the odd hops
    double ra[3][2 * CH_LANES], rb[3][2 * CH_LANES];        // last rows of D
    double beta[2 * CH_LANES + 1];                          // of the even hops, and a zero
};

__global__ void __launch_bounds__(64) chase_split_kernel(const double *band, double *q2, double *diag, double *off, int nb, const int *list, const int *count) {
    __shared__ __align__(16) ChShared sh;
    const int lane = threadIdx.x & 31, g = lane & (CH_LANES - 1);
    const bool first = g == 0, end = g == CH_LANES - 1;
    const int up = lane + (lane >> 4);   // the lane's slot of sh.ua: a matrix's seventeenth takes what leaves its last lane
    const int next = end ? 2 * CH_LANES : lane + 1;
    if (threadIdx.x < 5) ((threadIdx.x < 4) ? sh.xa[threadIdx.x & 3] : sh.beta)[2 * CH_LANES] = 0.0;   // (seen after the first barrier)
    auto meet = [] { asm volatile("bar.sync 1, 64;" ::: "memory"); };   // (the two warps meet in different places of the code)
    pdl_wait();
    const int total = list ? *count : nb;
    const int slots = (total + 1) / 2;
    for (int w = blockIdx.x; w < slots; w += gridDim.x) {
        // (an odd last matrix is done twice: both halves of the warps write the same values)
        const int li = min(2 * w + (lane >> 4), total - 1);
        const int blk = list ? list[li] : li;
        ChD AD, BD;   // hops 2 g and 2 g + 1
        ChB AB, BB;
        ch_load(AD, AB, band + static_cast<size_t>(blk) * BAND_ELEMS, 2 * g);
        ch_load(BD, BB, band + static_cast<size_t>(blk) * BAND_ELEMS, 2 * g + 1);
        if (threadIdx.x < 32) {
            // ---------------------------------------------------------------- B
            meet();
            // What a hop does off the chain is left for the next step, under the other hop's chain.
            double ba[4][4], bb[4][4], ub[4] = {0.0, 0.0, 0.0, 0.0}, v[4] = {0.0, 0.0, 0.0, 0.0}, last[3];
            auto double_step = [&](int k, auto guard) {
                constexpr bool GUARD = decltype(guard)::value;
                const bool started = !GUARD || k >= g;
                double xn[4];
                const double2 u0 = sh.ua[0][up], u1 = sh.ua[1][up];
                const double ua[4] = {u0.x, u0.y, u1.x, u1.y};
#pragma unroll
                for (int i = 1; i < 4; ++i) xn[i] = sh.xb[i][lane];
                if (!GUARD || k > g) {
                    ch_hop_rest(BB, bb, v, last);
#pragma unroll
                    for (int j = 0; j < 3; ++j) sh.rb[j][lane] = last[j];
                }
                if (started) ch_hop_chain(AB, ua, xn, BB.beta, ba, ub);
                sh.ub[0][lane] = make_double2(ub[0], ub[1]);
                sh.ub[1][lane] = make_double2(ub[2], ub[3]);
                sh.beta[lane] = AB.beta;
                meet();
#pragma unroll
                for (int i = 1; i < 4; ++i) xn[i] = sh.xa[i][next];
                const double bn = sh.beta[next];
                if (started) {
                    ch_hop_rest(AB, ba, ub, last);
#pragma unroll
                    for (int j = 0; j < 3; ++j) sh.ra[j][lane] = last[j];
                    ch_hop_chain(BB, ub, xn, bn, bb, v);
                }
                sh.ua[0][up + 1] = make_double2(v[0], v[1]);
                sh.ua[1][up + 1] = make_double2(v[2], v[3]);
                meet();
            };
#pragma unroll 1
            for (int k = 0; k < CH_LANES; ++k) double_step(k, std::true_type());
#pragma unroll 1
            for (int k = CH_LANES; k < SWEEPS; ++k) double_step(k, std::false_type());
        } else {
            // ---------------------------------------------------------------- D
            double *const Q = q2 + static_cast<size_t>(blk) * GRAM_ELEMS;
            double *const dd = diag + static_cast<size_t>(blk) * D, *const ee = off + static_cast<size_t>(blk) * D;
            const int pos0 = sweep_pos(g, 0), pos1 = sweep_pos(g, 2), pos2 = sweep_pos(g, 4), pos3 = sweep_pos(g, 6);
            auto start = [&](int s, double beta) {
                double u[4];
                const double e = ch_start(AD.x, beta, u);
                if (first) {
                    dd[s + 1] = AD.x[0];
                    ee[s + 1] = e;
                    sh.ua[0][up] = make_double2(u[0], u[1]);
                    sh.ua[1][up] = make_double2(u[2], u[3]);
                }
            };
            start(-1, AB.beta);
            if (!first) sh.ua[0][up] = sh.ua[1][up] = make_double2(0.0, 0.0);
#pragma unroll
            for (int i = 0; i < 4; ++i) sh.xb[i][lane] = BD.x[i];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                sh.ra[j][lane] = AD.d[3][j];
                sh.rb[j][lane] = BD.d[3][j];
            }
            meet();
            auto double_step = [&](int k, auto guard) {
                constexpr bool GUARD = decltype(guard)::value;
                const int s = k - g;
                const bool started = !GUARD || s >= 0;
                const bool store = started && g < sweep_chunks(s);
                double *const row = Q + (started ? sweep_offset(s) : 0) + 8 * g;
                const double2 a0 = sh.ua[0][up], a1 = sh.ua[1][up];
                const double ua[4] = {a0.x, a0.y, a1.x, a1.y};
#pragma unroll
                for (int j = 0; j < 3; ++j) AD.d[3][j] = sh.ra[j][lane];
                if (started) ch_hop_d(AD, ua, BD.x[0]);
#pragma unroll
                for (int i = 0; i < 4; ++i) sh.xa[i][lane] = AD.x[i];
                if (store) {
                    ch_store(row, pos0, ua[0], ua[1]);
                    ch_store(row, pos1, ua[2], ua[3]);
                }
                meet();
                const double2 b0 = sh.ub[0][lane], b1 = sh.ub[1][lane];
                const double ub[4] = {b0.x, b0.y, b1.x, b1.y};
                const double xn0 = sh.xa[0][next];
#pragma unroll
                for (int j = 0; j < 3; ++j) BD.d[3][j] = sh.rb[j][lane];
                if (started) ch_hop_d(BD, ub, xn0);
#pragma unroll
                for (int i = 0; i < 4; ++i) sh.xb[i][lane] = BD.x[i];
                start(s, sh.beta[lane]);
                if (store) {
                    ch_store(row, pos2, ub[0], ub[1]);
                    ch_store(row, pos3, ub[2], ub[3]);
                }
                meet();
            };
#pragma unroll 1
            for (int k = 0; k < CH_LANES - 1; ++k) double_step(k, std::true_type());
#pragma unroll 1
            for (int k = CH_LANES - 1; k < SWEEPS; ++k) double_step(k, std::false_type());
            if (first) {
                dd[D - 1] = AD.d[0][0];
                ee[D - 1] = 0.0;
            }
        }
        __syncthreads();   // the shared state is reused by the next pair
    }
}

}  // namespace

// Two warps per pair of matrices as long as every pair has its warps at once (six CTAs of either kind fit an SM): 52 us against 76 for up to 128
// blocks, 55 against 78 for 592, 76 against 86 for 1184, 103 against 119 for 1776.  Beyond, one warp per pair: 123 us against
// 140 for 2368 blocks, and 0.83 ms for 16384.
void launch_chase(int64_t nb, const Workspace &ws, const int *list, const int *count, int sm_count, cudaStream_t s) {
    const int n = static_cast<int>(nb);
    if (nb <= 12 * static_cast<int64_t>(sm_count))
        launch_dependent(chase_split_kernel, static_cast<unsigned>((nb + 1) / 2), 64, 0, s, ws.band, ws.q2, ws.diag, ws.off, n, list, count);
    else {
        const int64_t grid = std::min<int64_t>((nb + 2 * CH_WARPS - 1) / (2 * CH_WARPS), 6 * static_cast<int64_t>(sm_count));
        launch_dependent(chase_kernel, static_cast<unsigned>(grid), 32 * CH_WARPS, 0, s, ws.band, ws.q2, ws.diag, ws.off, n, list, count);
    }
}

}  // namespace eosq
