// First half of the tridiagonalisation of the d x d Gram matrices (the symmetric eigen-decomposition that
// stands in for the block's SVD, Sec. 2.3 and Algorithm 2 REQUIRE line): full matrix -> bandwidth 4, in
// double precision on the fp64 tensor instruction.
//
// Why two halves.  Reducing straight to tridiagonal form is a chain of 126 steps, each a matrix-vector
// product and a rank-2 update with two team-wide reductions between them: the matrix is read and written
// once per step for three multiply-adds per element, and the step waits for latencies most of the time
// (256-thread teams, two matrices per SM: 15 % of the fp64 rate).  Reducing to a band first takes the
// reflectors in panels of four: a panel's reflectors come from the panel alone (one warp, no matrix in the
// chain), and the matrix sees the four together, as products of 8 x 8 tiles.  eosq_chase.cu takes the band
// to tridiagonal form with little arithmetic.  Bandwidth 4 and not 8, although the tile products would then
// be used in full: a chasing hop of length 4 fits one thread's registers (1 ms against 4 ms per 16384
// matrices).
//
// Panel p (columns 4p .. 4p + 3, rows from 4p + 4; the even panels are the left halves of the tile columns J
// and start in the middle of the diagonal tile, the odd ones the right halves):
//   1. P = QR by Householder reflectors H_c = I - v_c v_c^T;  Q = H_0 .. H_3 = I - V T V^T,
//      T^-1 = I + strictly upper part of V^T V;
//   2. W = A V T,  S = T^T V^T W,  Z = W - V S / 2            (A: the trailing matrix)
//   3. A <- A - V Z^T - Z V^T                                  ( = Q^T A Q)
//
// Mapping.  A CTA per matrix: the tiles below the diagonal in shared memory (120 tiles, 60 KB at first), the
// diagonal ones in registers as accumulators.  W product warps do steps 2 and 3: warp w owns tile rows w and
// 2 W - 1 - w, and with four rows each 2 W + w and 4 W - 1 - w too (equal shares of the lower half), their products A V and
// the updates of their tiles.  Tile (I, J) is read as it is for row I and transposed for row J, both straight from
// shared memory in operand layout.  One more warp does step 1, one panel ahead: as soon as step 3 has brought the next panel's
// columns up to date it starts, while the rest of the matrix is being updated.  It holds rows l, l + 32, .. of
// the four columns in lane l; the norm of a column and its products with the three others are summed over
// the warp in one go on the tensor instruction.
#include <algorithm>

#include "eosq_common.cuh"
#include "eosq_fp64.cuh"

namespace eosq {

namespace {

constexpr int BD_PV = TILE_DIM * BAND_W;   // 32 doubles: eight rows of a panel

// The shape of one launch: the trailing matrix of TR tile rows, W product warps of RW tile rows each.
template <int TR_, int RW_>
struct BdShape {
    static constexpr int TR = TR_, RW = RW_, W = TR / RW, THREADS = 32 * (W + 1), FIRST = GRAM_TILE_ROWS - TR;   // FIRST: its first tile row
    static constexpr int OFFDIAG = TR * (TR - 1) / 2;   // tiles strictly below the diagonal
    // Parts that V^T W is summed from, each written by one warp: tile rows p and 15 - p of the whole matrix, or that row alone if
    // there are eight rows or less.  The same in every launch, and so is their order, so that a block's bits do not depend on the
    // launch's shape, which is chosen by how many blocks came with it.
    static constexpr int PARTS = (TR > 8) ? 8 : TR, GROUPS = (TR > 8) ? RW / 2 : RW;   // GROUPS: parts of one warp
    static_assert(TR <= 8 || (TR == 16 && RW >= 2 && W == 2 * PARTS / RW), "a warp owns both rows of a part");
    // dynamic shared memory in doubles: the tiles, V of the left and the right panel, W, the parts of V^T W,
    // T of the two panels, a diagonal tile, a tile of zeros
    static constexpr int VSIZE = TR * BD_PV, OFF_V = OFFDIAG * TILE_ELEMS, OFF_Z = OFF_V + 2 * VSIZE, OFF_U = OFF_Z + VSIZE, OFF_T = OFF_U + PARTS * 16,
                         OFF_D = OFF_T + 32, OFF_0 = OFF_D + TILE_ELEMS, DOUBLES = OFF_0 + TILE_ELEMS;
    static constexpr size_t SMEM = sizeof(double) * DOUBLES;
};
static_assert(3 * (BdShape<16, 4>::SMEM + 1024) <= 228 * 1024, "three CTAs per SM");

__device__ __forceinline__ int bd_tile(int i, int j) { return (i * (i - 1) / 2 + j) * TILE_ELEMS; }   // i > j
// tile rows of warp w, ascending in a: w, 2 W - 1 - w, 2 W + w, 4 W - 1 - w
template <class S>
__device__ __forceinline__ int bd_row(int warp, int a) { return (a >> 1) * 2 * S::W + ((a & 1) ? 2 * S::W - 1 - warp : warp); }

// Barriers: the product warps among themselves; the next panel's columns are up to date (the product warps
// arrive, the QR warp waits); V is there, T is there (the other way round; at V the product warps also wait for each other's updates).
template <class S>
__device__ __forceinline__ void bd_sync_products() { asm volatile("bar.sync 1, %0;" ::"n"(32 * S::W) : "memory"); }
template <class S>
__device__ __forceinline__ void bd_arrive_panel() { asm volatile("bar.arrive 2, %0;" ::"n"(S::THREADS) : "memory"); }
template <class S>
__device__ __forceinline__ void bd_wait_panel() { asm volatile("bar.sync 2, %0;" ::"n"(S::THREADS) : "memory"); }
template <class S>
__device__ __forceinline__ void bd_arrive_v() { asm volatile("bar.arrive 3, %0;" ::"n"(S::THREADS) : "memory"); }
template <class S>
__device__ __forceinline__ void bd_wait_v() { asm volatile("bar.sync 3, %0;" ::"n"(S::THREADS) : "memory"); }
template <class S>
__device__ __forceinline__ void bd_arrive_t() { asm volatile("bar.arrive 4, %0;" ::"n"(S::THREADS) : "memory"); }
template <class S>
__device__ __forceinline__ void bd_wait_t() { asm volatile("bar.sync 4, %0;" ::"n"(S::THREADS) : "memory"); }

// Sums over the warp, in every lane, of N <= 4 values.  First stage: value v of all lanes meets a matrix that is one
// on the rows with parity v, so rows 0 2 4 6 of the accumulator hold value 0 summed over the lanes of equal
// lane % 4 and rows 1 3 5 7 value 1; second stage: the accumulator as B operand against ones.  Value 0 comes first.
template <int N>
__device__ __forceinline__ void bd_sums(double (&v)[N], double even, double odd) {
    double a[2] = {0.0, 0.0}, b[2] = {0.0, 0.0}, c[2] = {0.0, 0.0}, d[2] = {0.0, 0.0};
    dmma(a, (N == 1) ? 1.0 : even, v[0]);
    if (N > 1) dmma(a, odd, v[1 % N]);
    if (N > 2) dmma(b, even, v[2 % N]);
    if (N > 3) dmma(b, odd, v[3 % N]);
    dmma(c, 1.0, a[0] + a[1]);
    if (N > 2) dmma(d, 1.0, b[0] + b[1]);
    v[0] = c[0];
    if (N > 1) v[1 % N] = c[1];
    if (N > 2) v[2 % N] = d[0];
    if (N > 3) v[3 % N] = d[1];
}

// Sum over a lane's rows of x[q] y[q], with x0 in place of x[0].
template <int Q>
__device__ __forceinline__ double bd_dot(const double (&P)[Q][4], int cx, int cy, double x0) {
    if constexpr (Q == 1) return x0 * P[0][cy];
    else if constexpr (Q == 2) return fma(P[1 % Q][cx], P[1 % Q][cy], x0 * P[0][cy]);
    else return fma(P[3 % Q][cx], P[3 % Q][cy], P[2 % Q][cx] * P[2 % Q][cy]) + fma(P[1 % Q][cx], P[1 % Q][cy], x0 * P[0][cy]);
}

// Column C of the panel's QR: the reflector of column C, applied to the columns after it.  ss: the column's sum of
// squares below the pivot; on return that of the next column.  The chain from one column to the next runs through
// the next column alone (its update, its norm, the roots); the products with the columns after it and their
// updates go in the shadow.
template <int Q, int C, int PO>
__device__ __forceinline__ void bd_panel_column(double (&P)[Q][4], int lane, double even, double odd, double &ss, double *__restrict__ rout) {
    constexpr int N = 3 - C, PL = PO + C;
    double pr[4], tot[4];
    const double x0 = (lane > PL) ? P[0][C] : 0.0;
#pragma unroll
    for (int k = 0; k <= N; ++k) pr[k] = __shfl_sync(0xffffffffu, P[0][C + k], PL);
    if (N > 0) {
        double d[N > 0 ? N : 1];
#pragma unroll
        for (int k = 0; k < N; ++k) d[k] = bd_dot(P, C, C + 1 + k, x0);
        bd_sums<(N > 0 ? N : 1)>(d, even, odd);
#pragma unroll
        for (int k = 0; k < N; ++k) tot[k + 1] = d[k];
    }
    double beta, g, amb;
    make_reflector(pr[0], ss, beta, g, amb);
    double v[Q];
    v[0] = ((lane == PL) ? amb : x0) * g;
#pragma unroll
    for (int q = 1; q < Q; ++q) v[q] = P[q][C] * g;
    if (N > 0) {
        const double f = g * fma(amb, pr[1], tot[1]);   // v_C . P[:, C + 1]
#pragma unroll
        for (int q = 0; q < Q; ++q) P[q][(C + 1) & 3] = fma(-v[q], f, P[q][(C + 1) & 3]);
        const double y0 = (lane > PL + 1) ? P[0][(C + 1) & 3] : 0.0;
        double n[1];
        {
            const double keep = P[0][(C + 1) & 3];
            P[0][(C + 1) & 3] = y0;
            n[0] = bd_dot(P, (C + 1) & 3, (C + 1) & 3, y0);
            P[0][(C + 1) & 3] = keep;
        }
        bd_sums<1>(n, even, odd);
        ss = n[0];
    }
#pragma unroll
    for (int k = 2; k <= N; ++k) {
        const double f = g * fma(amb, pr[k], tot[k]);
#pragma unroll
        for (int q = 0; q < Q; ++q) P[q][C + k] = fma(-v[q], f, P[q][C + k]);
    }
    if (lane >= PO && lane <= PL) rout[(lane - PO) * 4 + C] = (lane == PL) ? beta : P[0][C];
#pragma unroll
    for (int q = 0; q < Q; ++q) P[q][C] = v[q];
}

// QR of a panel by one warp.  Its rows start at row PO (4 or 0) of tile row f = J + (ODD ? 1 : 0); an even panel
// takes those of the diagonal tile from shared memory.  V goes to shared memory (zero above the panel) and to G, T (4 x 4,
// row-major) to shared memory, R (row-major) to `rout`; the other warps are let go as soon as V is there.  Tj: T of
// the pair of panels in global memory.  Tile rows count from S::FIRST here, in G from 0.
template <class S, bool ODD>
__device__ __forceinline__ void bd_panel_qr(double *__restrict__ sm, int J, int lane, double *__restrict__ G, double *__restrict__ rout, double *__restrict__ Tj) {
    constexpr int PO = ODD ? 0 : 4, Q = S::TR / 4, F = S::FIRST;   // Q: rows of the panel per lane
    const double *const tiles = sm, *const sD = sm + S::OFF_D;
    double *const sV = sm + S::OFF_V + (ODD ? S::VSIZE : 0), *const sT = sm + S::OFF_T + (ODD ? 16 : 0);
    const int f = ODD ? J + 1 : J, t = S::TR - f;
    const int r8 = lane & 7, half = tile_row(r8) + (((ODD ? 2 : 0) ^ tile_flip(r8)) << 1);   // the panel's four columns of this lane's tile row
    const double even = (lane & 4) ? 0.0 : 1.0, odd = 1.0 - even;
    double P[Q][4];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int rel = (lane >> 3) + 4 * q;   // tile of the panel
        const double *src = (!ODD && rel == 0) ? sD + half : tiles + bd_tile(f + ((rel < t) ? rel : (ODD ? 0 : 1)), J) + half;
        const bool in = rel < t && !(PO && q == 0 && lane < PO);
        double2 v0 = make_double2(0.0, 0.0), v1 = v0;
        if (in) {
            v0 = reinterpret_cast<const double2 *>(src)[0];
            v1 = reinterpret_cast<const double2 *>(src)[1];
        }
        P[q][0] = v0.x;
        P[q][1] = v0.y;
        P[q][2] = v1.x;
        P[q][3] = v1.y;
    }
    double ss;
    {
        const double keep = P[0][0], y0 = (lane > PO) ? keep : 0.0;
        P[0][0] = y0;
        double n[1] = {bd_dot(P, 0, 0, y0)};
        P[0][0] = keep;
        bd_sums<1>(n, even, odd);
        ss = n[0];
    }
    bd_panel_column<Q, 0, PO>(P, lane, even, odd, ss, rout);
    bd_panel_column<Q, 1, PO>(P, lane, even, odd, ss, rout);
    bd_panel_column<Q, 2, PO>(P, lane, even, odd, ss, rout);
    bd_panel_column<Q, 3, PO>(P, lane, even, odd, ss, rout);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int rel = (lane >> 3) + 4 * q;
        if (rel < t) {
            double2 *dv = reinterpret_cast<double2 *>(sV + (f + rel) * BD_PV + r8 * BAND_W);
            dv[0] = make_double2(P[q][0], P[q][1]);
            dv[1] = make_double2(P[q][2], P[q][3]);
        }
    }
    __syncwarp();
    bd_arrive_v<S>();
    // T, column by column: -T[:, < c] (V^T v_c), 1 on the diagonal; lane l holds row l % 4
    double Trow[4];
    {
        double g6[4] = {bd_dot(P, 0, 1, P[0][0]), bd_dot(P, 0, 2, P[0][0]), bd_dot(P, 1, 2, P[0][1]), bd_dot(P, 0, 3, P[0][0])};
        double h6[2] = {bd_dot(P, 1, 3, P[0][1]), bd_dot(P, 2, 3, P[0][2])};
        bd_sums<4>(g6, even, odd);
        bd_sums<2>(h6, even, odd);
        const int r = lane & 3;
        Trow[0] = (r == 0) ? 1.0 : 0.0;
        Trow[1] = (r == 1) ? 1.0 : -Trow[0] * g6[0];
        Trow[2] = (r == 2) ? 1.0 : fma(-Trow[1], g6[2], -Trow[0] * g6[1]);
        Trow[3] = (r == 3) ? 1.0 : fma(-Trow[2], h6[1], fma(-Trow[1], h6[0], -Trow[0] * g6[3]));
    }
    if (lane < 4) {
        double2 *dst = reinterpret_cast<double2 *>(sT + lane * 4);
        dst[0] = make_double2(Trow[0], Trow[1]);
        dst[1] = make_double2(Trow[2], Trow[3]);
    }
    __syncwarp();
    bd_arrive_t<S>();
    // off the chain: V and T to global memory
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int rel = (lane >> 3) + 4 * q;
        if (rel < t) {
            double2 *dv = reinterpret_cast<double2 *>(G + tile_index(F + f + rel, F + J) * TILE_ELEMS + half);
            dv[0] = make_double2(P[q][0], P[q][1]);
            dv[1] = make_double2(P[q][2], P[q][3]);
        }
    }
    const double2 z = make_double2(0.0, 0.0);
    if (!ODD) {
        if (lane < 8) {   // the diagonal tile of V has nothing in the right panel's columns; T of the left panel
            double2 *dv = reinterpret_cast<double2 *>(G + tile_index(F + J, F + J) * TILE_ELEMS + (half ^ 4));
            dv[0] = z;
            dv[1] = z;
            double2 *dt = reinterpret_cast<double2 *>(Tj + half);
            dt[0] = (lane < 4) ? make_double2(Trow[0], Trow[1]) : z;
            dt[1] = (lane < 4) ? make_double2(Trow[2], Trow[3]) : z;
            if (F + J == GRAM_TILE_ROWS - 1) {
                dt = reinterpret_cast<double2 *>(Tj + (half ^ 4));
                dt[0] = z;
                dt[1] = z;
            }
        }
    } else {
        // T of the pair, right half: -T_left (V_left^T V_right) T_right above T_right
        const double *const sVl = sm + S::OFF_V, *const sTl = sm + S::OFF_T;
        double x[4][4];   // (V_left^T V_right)[e][c], then times T_right
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int c = 0; c < 4; ++c) x[e][c] = 0.0;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int rel = (lane >> 3) + 4 * q;
            if (rel < t) {
                const double2 *lv = reinterpret_cast<const double2 *>(sVl + (f + rel) * BD_PV + r8 * BAND_W);
                const double2 l0 = lv[0], l1 = lv[1];
                const double l[4] = {l0.x, l0.y, l1.x, l1.y};
#pragma unroll
                for (int e = 0; e < 4; ++e)
#pragma unroll
                    for (int c = 0; c < 4; ++c) x[e][c] = fma(l[e], P[q][c], x[e][c]);
            }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) bd_sums<4>(x[e], even, odd);
        const int r = (lane >> 2) & 3, c = lane & 3;
        double y = 0.0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            double xt = 0.0;
#pragma unroll
            for (int e = 0; e < 4; ++e) xt = fma(x[q][e], sT[e * 4 + c], xt);
            y = fma(-sTl[r * 4 + q], xt, y);
        }
        Tj[tile_off((lane < 16) ? r : 4 + r, 4 + c)] = (lane < 16) ? y : sT[r * 4 + c];
    }
}

struct BdLane {
    int m, k;
    int o_c;              // accumulator: row m, columns 2k, 2k + 1
    int o_d0, o_d1;       // operand as it is: row m, columns k and 4 + k
    int o_t;              // operand transposed: rows k (and 4 + k, 32 doubles on), column m
    int o_v, o_vt, o_vp;  // rows of V and W: [m][k]; [k][m / 2] (rows 4 + k: 16 doubles on); [2k][m / 2] (2k + 1: 4 on)
};

// Y = A V for the last R of the warp's rows over the tile columns [f, TR): tiles left of the diagonal as they are,
// those below it transposed, zeros in place of the diagonal tile, which sits in registers and comes last.  The
// operands of the next column are fetched under the products of this one, at addresses found without
// branches (a branch per tile tripled the time).  Only four of the eight columns of a product are used: column 2c and
// 2c + 1 are both V's column c, so that the first entry of an accumulator is column k of row m, an operand of the next product.
// Plain multiply-adds would save the repetition, and run on a pipe of their own beside the tensor instruction's (127
// multiply-adds per clock and SM together, 64 each), but V's rows then come as 128-bit reads, four per tile column, that the warp
// stalls on: 4.07 ms per 16384 matrices against 3.76 (half of the tile rows that way: 4.10).
template <class S, int R>
__device__ __forceinline__ void bd_multiply(const double *__restrict__ sm, const double *__restrict__ sV, int warp, int f, const BdLane &L,
                                            const double (&dg)[S::RW][2], double (&Y)[S::RW][2]) {
    int row[R];
    double x0[R], x1[R], yb[R][2];
#pragma unroll
    for (int a = 0; a < R; ++a) {
        row[a] = bd_row<S>(warp, S::RW - R + a);
        yb[a][0] = yb[a][1] = 0.0;
    }
    auto fetch = [&](int jj, double (&p)[R], double (&q)[R], double &v, double &w) {
        v = sV[jj * BD_PV + L.o_vt];
        w = sV[jj * BD_PV + L.o_vt + 16];
#pragma unroll
        for (int a = 0; a < R; ++a) {
            const bool left = jj < row[a];
            const int as_is = bd_tile(row[a], 0) + jj * TILE_ELEMS + L.o_d0, transposed = bd_tile(jj, 0) + row[a] * TILE_ELEMS + L.o_t;
            const int at = (jj == row[a]) ? S::OFF_0 : (left ? as_is : transposed);
            p[a] = sm[at];
            q[a] = sm[at + (left ? L.o_d1 - L.o_d0 : 32)];
        }
    };
    double v, w;
    fetch(f, x0, x1, v, w);
#pragma unroll 2
    for (int jj = f; jj < S::TR; ++jj) {
        double p[R], q[R], nv, nw;
        fetch(min(jj + 1, S::TR - 1), p, q, nv, nw);
#pragma unroll
        for (int a = 0; a < R; ++a) dmma(Y[S::RW - R + a], x0[a], v);
#pragma unroll
        for (int a = 0; a < R; ++a) dmma(yb[a], x1[a], w);
#pragma unroll
        for (int a = 0; a < R; ++a) {
            x0[a] = p[a];
            x1[a] = q[a];
        }
        v = nv;
        w = nw;
    }
#pragma unroll
    for (int a = 0; a < R; ++a) dmma(Y[S::RW - R + a], dg[S::RW - R + a][0], sV[row[a] * BD_PV + L.o_vp]);
#pragma unroll
    for (int a = 0; a < R; ++a) dmma(yb[a], dg[S::RW - R + a][1], sV[row[a] * BD_PV + L.o_vp + 4]);
#pragma unroll
    for (int a = 0; a < R; ++a) Y[S::RW - R + a][0] += yb[a][0];
}

// The same for those of the warp's rows that the panel has (its last R at most).
template <class S, int R>
__device__ __forceinline__ void bd_multiply_active(const double *__restrict__ sm, const double *__restrict__ sV, int warp, int f, const BdLane &L,
                                                   const double (&dg)[S::RW][2], double (&Y)[S::RW][2]) {
    if (bd_row<S>(warp, S::RW - R) >= f) bd_multiply<S, R>(sm, sV, warp, f, L, dg, Y);
    else if constexpr (R > 1) bd_multiply_active<S, R - 1>(sm, sV, warp, f, L, dg, Y);
}

// A -= V Z^T + Z V^T on the tiles of the last R of the warp's rows in the tile columns [j0, j1), all left of the diagonal.
template <class S, int R>
__device__ __forceinline__ void bd_update(double *__restrict__ tiles, const double *__restrict__ zv, const double *__restrict__ vv, int warp,
                                          const double (&nv)[S::RW], const double (&nz)[S::RW], int j0, int j1, int o_c) {
    if (j0 >= j1) return;
    double2 *p[R];
    double2 C[R];
#pragma unroll
    for (int a = 0; a < R; ++a) {
        p[a] = reinterpret_cast<double2 *>(tiles + bd_tile(bd_row<S>(warp, S::RW - R + a), j0) + o_c);
        C[a] = p[a][0];
    }
    double z = zv[j0 * BD_PV], v = vv[j0 * BD_PV];
#pragma unroll 2
    for (int jj = j0; jj < j1; ++jj) {
        const int nx = min(jj + 1, j1 - 1), step = (nx - jj) * (TILE_ELEMS / 2);
        const double nzv = zv[nx * BD_PV], nvv = vv[nx * BD_PV];
        double c[R][2];
#pragma unroll
        for (int a = 0; a < R; ++a) {
            c[a][0] = C[a].x;
            c[a][1] = C[a].y;
            C[a] = p[a][step];
        }
#pragma unroll
        for (int a = 0; a < R; ++a) dmma(c[a], nv[S::RW - R + a], z);
#pragma unroll
        for (int a = 0; a < R; ++a) dmma(c[a], nz[S::RW - R + a], v);
#pragma unroll
        for (int a = 0; a < R; ++a) {
            p[a][0] = make_double2(c[a][0], c[a][1]);
            p[a] += step;
        }
        z = nzv;
        v = nvv;
    }
}

// Tile column f, of those of the warp's rows that lie below it.
template <class S, int R>
__device__ __forceinline__ void bd_update_first(double *__restrict__ tiles, const double *__restrict__ zv, const double *__restrict__ vv, int warp,
                                                const double (&nv)[S::RW], const double (&nz)[S::RW], int f, int o_c) {
    if (bd_row<S>(warp, S::RW - R) > f) bd_update<S, R>(tiles, zv, vv, warp, nv, nz, f, f + 1, o_c);
    else if constexpr (R > 1) bd_update_first<S, R - 1>(tiles, zv, vv, warp, nv, nz, f, o_c);
}
// The tile columns from j0 up to the diagonal.
template <class S, int R>
__device__ __forceinline__ void bd_update_rest(double *__restrict__ tiles, const double *__restrict__ zv, const double *__restrict__ vv, int warp,
                                               const double (&nv)[S::RW], const double (&nz)[S::RW], int j0, int o_c) {
    const int j1 = bd_row<S>(warp, S::RW - R);
    bd_update<S, R>(tiles, zv, vv, warp, nv, nz, j0, j1, o_c);
    if constexpr (R > 1) bd_update_rest<S, R - 1>(tiles, zv, vv, warp, nv, nz, max(j0, j1), o_c);
}

// Steps 2 and 3 for the panel whose V (tile rows f ..) and T are in shared memory.
template <class S, bool ODD>
__device__ __forceinline__ void bd_apply(double *__restrict__ sm, int J, int warp, const BdLane &L, double (&dg)[S::RW][2]) {
    double *const tiles = sm, *const sV = sm + S::OFF_V + (ODD ? S::VSIZE : 0), *const sz = sm + S::OFF_Z, *const sU = sm + S::OFF_U, *const sD = sm + S::OFF_D;
    const double *const sT = sm + S::OFF_T + (ODD ? 16 : 0);
    const int f = ODD ? J + 1 : J;
    double Y[S::RW][2] = {};
    bd_multiply_active<S, S::RW>(sm, sV, warp, f, L, dg, Y);
    bd_wait_t<S>();
    // W = Y T, and this warp's parts of U = V^T W (rows w and 15 - w: its first and its last); columns in pairs throughout
    const double tb = sT[L.o_vt];
    double W[S::RW][2], U[S::GROUPS][2] = {};
#pragma unroll
    for (int a = 0; a < S::RW; ++a) {
        const int i = bd_row<S>(warp, a);
        W[a][0] = W[a][1] = 0.0;
        if (i < f) continue;
        dmma(W[a], (!ODD && i == J && L.m < 4) ? 0.0 : Y[a][0], tb);   // (the diagonal tile's first rows are above the panel)
        sz[i * BD_PV + L.o_v] = W[a][0];
    }
    __syncwarp();
    double nv[S::RW];   // -V of the own rows
#pragma unroll
    for (int a = 0; a < S::RW; ++a) {
        const int i = bd_row<S>(warp, a);
        nv[a] = 0.0;
        if (i < f) continue;
        const double *vt = sV + i * BD_PV + L.o_vt, *wt = sz + i * BD_PV + L.o_vt;
        const int g = (a < S::GROUPS) ? a : S::RW - 1 - a;
        dmma(U[g], vt[0], wt[0]);
        dmma(U[g], vt[16], wt[16]);
        nv[a] = -sV[i * BD_PV + L.o_v];
    }
#pragma unroll
    for (int g = 0; g < S::GROUPS; ++g)
        if (!(L.m & 1)) sU[bd_row<S>(warp, g) * 16 + (L.m >> 1) * 4 + L.k] = U[g][0];
    bd_sync_products<S>();
    // S = T^T U, which is symmetric: S^T = U^T T as accumulator is S as operand.  The update as A - V W^T - (W - V S) V^T, so that
    // S enters through the own rows alone: nz = -(W - V S)
    double nz[S::RW];
    {
        double u[2] = {0.0, 0.0};
#pragma unroll
        for (int p = 0; p < S::PARTS; ++p) u[p & 1] += sU[(S::TR > 8 ? p : S::PARTS - 1 - p) * 16 + L.o_vt];   // (a part above the panel is zero)
        double St[2] = {0.0, 0.0};
        dmma(St, u[0] + u[1], tb);
#pragma unroll
        for (int a = 0; a < S::RW; ++a) {
            dmma(W[a], nv[a], St[0]);
            nz[a] = -W[a][0];
        }
    }
    // own rows: first tile column f, which holds the next panel
    const double *const zv = sz + L.o_v, *const vv = sV + L.o_v;
    bd_update_first<S, S::RW>(tiles, zv, vv, warp, nv, nz, f, L.o_c);
#pragma unroll
    for (int a = 0; a < S::RW; ++a)
        if (bd_row<S>(warp, a) == f) {
            dmma(dg[a], nv[a], zv[f * BD_PV]);
            dmma(dg[a], nz[a], -nv[a]);
            if (ODD) *reinterpret_cast<double2 *>(sD + L.o_c) = make_double2(dg[a][0], dg[a][1]);
        }
    bd_arrive_panel<S>();
#pragma unroll
    for (int a = 0; a < S::RW; ++a)
        if (bd_row<S>(warp, a) > f) dmma(dg[a], nv[a], zv[bd_row<S>(warp, a) * BD_PV]);
#pragma unroll
    for (int a = 0; a < S::RW; ++a)
        if (bd_row<S>(warp, a) > f) dmma(dg[a], nz[a], -nv[a]);
    bd_update_rest<S, S::RW>(tiles, zv, vv, warp, nv, nz, f + 1, L.o_c);
}

// gram: [nb][136 tiles] in, the panels' V out; band and tmat as described at Workspace.  Tile columns S::FIRST + [0, JEND);
// what is left of the matrix goes back to gram for the next launch.
template <class S, int JEND, int MINB>
__global__ void __launch_bounds__(S::THREADS, MINB) band_kernel(double *gram, double *band, double *tmat,
                                                                int nb, const int *list, const int *count) {
    extern __shared__ __align__(16) double bd_smem[];
    constexpr int F = S::FIRST;
    constexpr bool LAST = JEND == S::TR;
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // (known to be the same in all lanes)
    BdLane L;
    L.m = lane >> 2;
    L.k = lane & 3;
    L.o_c = tile_off(L.m, 2 * L.k);
    L.o_d0 = tile_off(L.m, L.k);
    L.o_d1 = tile_off(L.m, 4 + L.k);
    L.o_t = tile_off(L.k, L.m);
    L.o_v = L.m * BAND_W + L.k;
    L.o_vt = L.k * BAND_W + (L.m >> 1);
    L.o_vp = 2 * L.k * BAND_W + (L.m >> 1);
    if (tid < TILE_ELEMS) bd_smem[S::OFF_0 + tid] = 0.0;
    pdl_wait();
    const int total = list ? *count : nb;
    for (int li = blockIdx.x; li < total; li += gridDim.x) {
        const int blk = list ? list[li] : li;
        double *const G = gram + static_cast<size_t>(blk) * GRAM_ELEMS;
        double *const Bd = band + static_cast<size_t>(blk) * BAND_ELEMS + 64 * F;
        double dg[S::RW][2];
        // the rows of tiles: those below the diagonal to shared memory, the diagonal ones to their owner's registers
#pragma unroll 1
        for (int i = 1 + warp; i < S::TR; i += S::W + 1) {
            const double *src = G + tile_index(F + i, F) * TILE_ELEMS + 2 * lane;
            const double *dst = bd_smem + bd_tile(i, 0) + 2 * lane;
#pragma unroll 4
            for (int e = 0; e < i; ++e) cp_async16(dst + e * TILE_ELEMS, src + e * TILE_ELEMS);
        }
        if (warp < S::W) {
#pragma unroll
            for (int a = 0; a < S::RW; ++a) {
                const int i = bd_row<S>(warp, a);
                const double2 v = *reinterpret_cast<const double2 *>(G + tile_index(F + i, F + i) * TILE_ELEMS + L.o_c);
                dg[a][0] = v.x;
                dg[a][1] = v.y;
                if (i == 0) *reinterpret_cast<double2 *>(bd_smem + S::OFF_D + L.o_c) = v;
            }
        }
        cp_async_wait_all();
        __syncthreads();
        if (warp < S::W) {
#pragma unroll 1
            for (int J = 0; J < JEND; ++J) {
                bd_wait_v<S>();
                bd_apply<S, false>(bd_smem, J, warp, L, dg);
                if (LAST && J == S::TR - 1) break;
                bd_wait_v<S>();
                bd_apply<S, true>(bd_smem, J, warp, L, dg);
            }
            // the band's diagonal blocks, and what is left
#pragma unroll
            for (int a = 0; a < S::RW; ++a) {
                const int i = bd_row<S>(warp, a);
                if (i < JEND) {
                    if ((L.m < 4) == (L.k < 2))
                        *reinterpret_cast<double2 *>(Bd + 64 * i + ((L.m < 4) ? L.m * 4 + 2 * L.k : 32 + (L.m - 4) * 4 + 2 * L.k - 4)) = make_double2(dg[a][0], dg[a][1]);
                } else {
                    double *const row = G + tile_index(F + i, F) * TILE_ELEMS + L.o_c;
                    *reinterpret_cast<double2 *>(row + i * TILE_ELEMS) = make_double2(dg[a][0], dg[a][1]);
#pragma unroll 4
                    for (int e = JEND; e < i; ++e) *reinterpret_cast<double2 *>(row + e * TILE_ELEMS) = *reinterpret_cast<const double2 *>(bd_smem + bd_tile(i, e) + L.o_c);
                }
            }
        } else {
            double *const T = tmat + static_cast<size_t>(blk) * GRAM_TILE_ROWS * TILE_ELEMS + F * TILE_ELEMS;
#pragma unroll 1
            for (int J = 0; J < JEND; ++J) {
                if (J > 0) bd_wait_panel<S>();
                bd_panel_qr<S, false>(bd_smem, J, lane, G, Bd + 64 * J + 16, T + J * TILE_ELEMS);
                bd_wait_panel<S>();
                if (LAST && J == S::TR - 1) break;
                bd_panel_qr<S, true>(bd_smem, J, lane, G, Bd + 64 * J + 48, T + J * TILE_ELEMS);
            }
            if (!LAST) bd_wait_panel<S>();
        }
        __syncthreads();   // the tiles are reused by the next matrix
    }
}

template <class S, int JEND, int MINB>
void launch_band_part(int64_t nb, const Workspace &ws, const int *list, const int *count, int sm_count, cudaStream_t s) {
    ensure_dynamic_smem(reinterpret_cast<const void *>(band_kernel<S, JEND, MINB>), S::SMEM);
    const int64_t grid = std::min<int64_t>(nb, MINB * static_cast<int64_t>(sm_count));
    launch_dependent(band_kernel<S, JEND, MINB>, static_cast<unsigned>(std::max<int64_t>(grid, 1)), S::THREADS, S::SMEM, s, ws.gram, ws.band, ws.tmat, static_cast<int>(nb), list, count);
}

}  // namespace

// Up to two blocks per SM every block has a CTA at once and what counts is one matrix's own time: eight product warps, one or two
// tile rows each, and a launch of its own for the second half, whose CTAs have less to go through (an encode of 2 to 128 blocks: 6 us less than with one
// launch for all columns; 183 us of two blocks of 512 tokens).  With more blocks the SM's other matrices fill the gaps of one, so what
// counts is how many are in flight: four product warps each and three CTAs per SM while the matrix is large (3.75 ms per 16384 matrices; eight warps on two
// CTAs took 9 % more), and a new launch with more CTAs per SM whenever it has
// halved (64 left: four CTAs of four product warps, a fifth less than six of two; from 32 left eight of two,
// together 1.01 ms).  A launch at 96 left would give 1 % more.  Measured at the ends of the two ranges; between 297 and some
// 900 blocks, where the number of rounds counts, the line has not been searched.
// The second pass works through a list whose length the host does not know.  It is empty for most caches, and then a launch
// costs 1.2 us, but it holds every block of a cache whose outlier channels are strong enough.  So it is one launch where that counts,
// up to twelve blocks per SM (lists of all blocks of 328 tokens, the whole call: 16 blocks 336 us against 330 in two launches, 592 blocks 857
// against 824 in three, 1776 blocks 2042 against 1978; empty lists, 512 tokens: 189 against 191, 423 against 427), and the launches of the
// first pass beyond (4096 blocks 4.50 ms against 4.67 in one, with an empty list the same to 0.2 %).
static bool band_in_one(int64_t nb, bool listed, int sm_count) { return listed && nb <= 12 * static_cast<int64_t>(sm_count); }
int band_launches(int64_t nb, bool listed, int sm_count) {
    return band_in_one(nb, listed, sm_count) ? 1 : ((nb <= 2 * static_cast<int64_t>(sm_count)) ? 2 : 3);
}

void launch_band(int part, int64_t nb, const Workspace &ws, const int *list, const int *count, int sm_count, cudaStream_t s) {
    const bool one = band_in_one(nb, list != nullptr, sm_count);
    if (nb <= 2 * static_cast<int64_t>(sm_count)) {
        if (one) launch_band_part<BdShape<16, 2>, 16, 2>(nb, ws, list, count, sm_count, s);
        else if (part == 0) launch_band_part<BdShape<16, 2>, 8, 2>(nb, ws, list, count, sm_count, s);
        else launch_band_part<BdShape<8, 1>, 8, 2>(nb, ws, list, count, sm_count, s);
    } else if (one) launch_band_part<BdShape<16, 4>, 16, 3>(nb, ws, list, count, sm_count, s);
    else if (part == 0) launch_band_part<BdShape<16, 4>, 8, 3>(nb, ws, list, count, sm_count, s);
    else if (part == 1) launch_band_part<BdShape<8, 2>, 4, 4>(nb, ws, list, count, sm_count, s);
    else launch_band_part<BdShape<4, 2>, 4, 8>(nb, ws, list, count, sm_count, s);
}

}  // namespace eosq
