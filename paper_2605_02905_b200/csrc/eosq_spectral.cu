// Spectral stage of eosq_encode: symmetric eigen-decomposition of the d x d Gram matrix
// (the block's singular values and right singular vectors, Sec. 2.3) and Algorithm 2
// (bulk edge, rank, imputed noise spectrum, D-transform estimators, Frobenius shrinker).
//
// All arithmetic here is double precision: the bulk eigenvalues sit two to three orders of
// magnitude below the largest outlier, and the rank test and the shrunk values must agree with a
// double-precision reference to 1e-4 relative or better.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "eosq_common.cuh"

namespace eosq {

// ------------------------------------------------------------------------------------------
// Eigenvalues of a symmetric tridiagonal matrix from Sturm sequences: with
//   p_0 = 1, p_1 = d_0 - x, p_{i+1} = (d_i - x) p_i - e_{i-1}^2 p_{i-1},
// the number of sign changes in p_0 .. p_d is the number of eigenvalues below x, and p_d(x) is the
// characteristic polynomial.
// One procedure for every eigenvalue, whichever kernel runs it and however many lanes share it, so that a block's
// eigenvalues, and all that follows from them, do not depend on how many blocks came with it (ev_bracket, ev_root):
//   1. counts at EV_GRID points spaced geometrically below the Gershgorin bound (the spectrum of a Gram matrix spans
//      many decades) bracket it;
//   2. bisection on the counts until the bracket holds one eigenvalue and is 0.5 % wide, or is 1e-8 relative wide (2e-15 of the
//      matrix scale for the smallest ones: then its middle is reported);
//   3. Laguerre's iteration on p_d, p_d' and p_d'' inside the bracket.  It converges with the cube of the error, towards the
//      one root of the bracket from either side.
// ------------------------------------------------------------------------------------------
constexpr double EV_E2_FLOOR = 1e-60;   // keeps the recurrence alive across an exactly decoupled entry
constexpr int EV_MAX_ITER = 96;
constexpr int EV_GRID = 96;             // points of the first pass: three per lane where a warp has a block to itself

// The recurrences run from both ends to the middle, rows 0 .. 63 downwards and 127 .. 64 upwards, side by side: half as many
// steps follow one another, and each leaves room for the other's (one chain of 128 rows: 27 us for the eigenvalues of 16 blocks
// and 470 for 16384, so 23 and 446).  With p_i the leading and r_i the trailing minors (r_128 = 1, rows i ..),
//   det(T - x I) = p_64 r_64 - e_63^2 p_63 r_65,
// and the twisted factorisation counts: the sign changes of p_0 .. p_63 and of r_128 .. r_64, and one more if
// the middle pivot det / (p_63 r_64) is negative.
constexpr int EV_HALF = D / 2, EV_GROUP = 2, EV_CHECK = 16;   // steps; fetched together; between two range checks
static_assert(EV_HALF % EV_CHECK == 0 && EV_CHECK % EV_GROUP == 0, "whole groups");

// The entries of steps j .. j + EV_GROUP - 1: rows j from the top and 127 - j from the bottom.  (One group past the middle is fetched and not used.)
struct EvRows {
    double2 top[EV_GROUP], bottom[EV_GROUP];
    __device__ __forceinline__ void fetch(const double2 *__restrict__ sde, int j) {
#pragma unroll
        for (int i = 0; i < EV_GROUP; ++i) {
            top[i] = sde[j + i];
            bottom[i] = sde[D - 1 - j - i];
        }
    }
};

// sde[i] = (d_i, e_{i-1}^2) with e_{-1} = 0, scaled so that every entry is at most 1 in magnitude.  Returns the count of
// eigenvalues below x.  The entries of the next group are fetched before the current group's chain of dependent multiply-adds
// starts, and a pair of minors is brought back to within 2^+-170 of one every sixteen steps: they
// move it by at most 2^48 upwards and, even with full cancellation in every step, 2^-848 downwards.  Rows that are small themselves
// leave that range only if sixteen in a row have |d - x| below 5e-20, in a singular matrix with x as close to zero; no bracket is
// narrowed below 2e-15, so that a count which goes wrong there moves an eigenvalue by no more than the search does anyway.
__device__ __forceinline__ int sturm_count(const double2 *__restrict__ sde, double x) {
    double p0 = 0.0, p1 = 1.0, r0 = 0.0, r1 = 1.0, e2 = 0.0;   // e2: the square that couples the row below
    unsigned sp = 0u, sr = 0u;   // signs, the latest in bit 0
    int cnt = 0;
    auto sign = [](double v) { return static_cast<unsigned>(__double2hiint(v)); };
    auto check = [](double &a, double &b) {
        const int ea = (__double2hiint(a) >> 20) & 0x7ff, eb = (__double2hiint(b) >> 20) & 0x7ff;
        const int em = max(ea, eb);
        if (static_cast<unsigned>(em - 853) > 340u) {
            if (em == 0) {   // both vanished: restart with the current sign
                a = 0.0;
                b = (__double2hiint(b) < 0) ? -1.0 : 1.0;
            } else if (em < 2047) {
                const double sc = __hiloint2double((2046 - em) << 20, 0);   // 2^(1023 - em)
                a *= sc;
                b *= sc;
            }
        }
    };
    EvRows cur, nxt;
    cur.fetch(sde, 0);
#pragma unroll 1
    for (int j = 0; j < EV_HALF; j += EV_CHECK) {
#pragma unroll
        for (int g = 0; g < EV_CHECK; g += EV_GROUP) {
            nxt.fetch(sde, j + g + EV_GROUP);
#pragma unroll
            for (int i = 0; i < EV_GROUP; ++i) {
                const double p2 = fma(cur.top[i].x - x, p1, -(cur.top[i].y * p0));
                const double r2 = fma(cur.bottom[i].x - x, r1, -(e2 * r0));
                e2 = cur.bottom[i].y;
                sp = __funnelshift_l(sign(p2), sp, 1);
                sr = __funnelshift_l(sign(r2), sr, 1);
                p0 = p1;
                p1 = p2;
                r0 = r1;
                r1 = r2;
            }
            cur = nxt;
        }
        constexpr unsigned MASK = (1u << EV_CHECK) - 1u;
        cnt += __popc((sp ^ (sp >> 1)) & MASK) + __popc((sr ^ (sr >> 1)) & MASK);
        check(p0, p1);
        check(r0, r1);
    }
    // the last change of the upper chain gives way to the sign of the middle pivot
    const double det = fma(p1, r1, -((e2 * p0) * r0));
    const unsigned last = (sp ^ (sp >> 1)) & 1u, middle = ((sign(det) >> 31) ^ (sp >> 1) ^ sr) & 1u;
    return cnt - static_cast<int>(last) + static_cast<int>(middle);
}

// Which eigenvalues are resolved.  Algorithm 2 reads individually only lambda_1 .. lambda_{k+r+1} and
// lambda_{2k+1}, lambda_{2k+r+1} (Steps 1 and 2; r <= k); the rest of the spectrum enters through sums
// that the spectral kernel takes from the characteristic polynomial.  The kernels resolve the
// EV_EXPL = 32 largest and lambda_{2k+r+1} (index 32 or 33) for the rare ranks 10 and 11 (the kernel with one warp per
// block in a second round), or every eigenvalue (the optional `eig` output).
constexpr int EV_EXPL = 32;
constexpr int EV_TOP = 3 * KPILOT + 1;   // entries of lam the spectral kernel may read without the full spectrum
static_assert(2 * KPILOT + 9 < EV_EXPL && EV_TOP <= EV_EXPL + 2, "ranks up to 9 find lambda_{2k+r+1} among the first 32");

// Sums over the whole spectrum from the characteristic polynomial p(x) = det(T - x I) and its first
// two derivatives, by the three-term recurrences
//   p_{i+1} = (d_i - x) p_i - e_{i-1}^2 p_{i-1},   p'_{i+1} = (d_i - x) p'_i - p_i - e_{i-1}^2 p'_{i-1},
//   p''_{i+1} = (d_i - x) p''_i - 2 p'_i - e_{i-1}^2 p''_{i-1}   (kept as p'' / 2, which saves the doubling):
//   s1 = sum_j 1 / (lambda_j - x) = -p'/p,   s2 = sum_j 1 / (lambda_j - x)^2 = (p'/p)^2 - p''/p.
// From both ends as for the Sturm counts, sde likewise; det and its derivatives by the product rule.  A chain's six running
// values are brought back to within range together every sixteen rows (the ratios do not change).
// Returns the number of sign bits of p (0 or 1).
struct EvChain {
    double p0 = 0.0, p1 = 1.0, q0 = 0.0, q1 = 0.0, r0 = 0.0, r1 = 0.0;
    __device__ __forceinline__ void row(double t, double e2) {
        const double p2 = fma(t, p1, -e2 * p0);
        const double q2 = fma(t, q1, fma(-e2, q0, -p1));
        const double r2 = fma(t, r1, fma(-e2, r0, -q1));
        p0 = p1;
        p1 = p2;
        q0 = q1;
        q1 = q2;
        r0 = r1;
        r1 = r2;
    }
    __device__ __forceinline__ void rescale() {
        const int ea = (__double2hiint(p0) >> 20) & 0x7ff, eb = (__double2hiint(p1) >> 20) & 0x7ff;
        const int em = max(ea, eb);
        if (em > 0 && em < 2047) {
            const double sc = __hiloint2double((2046 - em) << 20, 0);   // 2^(1023 - em)
            p0 *= sc;
            p1 *= sc;
            q0 *= sc;
            q1 *= sc;
            r0 *= sc;
            r1 *= sc;
        }
    }
};
__device__ __forceinline__ unsigned charpoly_sums(const double2 *__restrict__ sde, double x, double &s1, double &s2) {
    EvChain a, b;
    double e2 = 0.0;
#pragma unroll 1
    for (int j = 0; j < EV_HALF; j += EV_CHECK) {
#pragma unroll
        for (int i = 0; i < EV_CHECK; ++i) {
            const double2 top = sde[j + i], bottom = sde[D - 1 - j - i];
            a.row(top.x - x, top.y);
            b.row(bottom.x - x, e2);
            e2 = bottom.y;
        }
        a.rescale();
        b.rescale();
    }
    auto coupled = [&](double main, double other) { return fma(-e2, other, main); };
    const double f = coupled(a.p1 * b.p1, a.p0 * b.p0);
    const double f1 = coupled(fma(a.p1, b.q1, a.q1 * b.p1), fma(a.p0, b.q0, a.q0 * b.p0));
    const double f2 = coupled(fma(a.p1, b.r1, fma(a.q1, b.q1, a.r1 * b.p1)), fma(a.p0, b.r0, fma(a.q0, b.q0, a.r0 * b.p0)));
    const double ip = sp_rcp(f);
    s1 = -f1 * ip;
    s2 = fma(s1, s1, -2.0 * f2 * ip);
    return static_cast<unsigned>(__double2hiint(f)) >> 31;
}

// The last step: below 1e-7 relative, and below a thousandth of the step before.  Near its root the iteration's error goes
// with its cube, e' = C e^3, so C e^2 was about 1e-3 at the step before and e' is below 1e-9 e.  Its size alone tells
// nothing about a root with a close neighbour: while e is above their distance a step covers only two thirds of e (a
// stop at 1e-7 left up to 0.1 of the distance in the eigenvalue of a pair 1e-7 apart, and as much of its neighbour in the vector).
constexpr double EV_LAGUERRE_STEP = 1e-7, EV_LAGUERRE_RATIO = 1e-3;
// Width of a bracket at which Laguerre's iteration takes over.  An evaluation of it costs half as much again as a count, and the
// closest two of a warp's eigenvalues need about six levels of bisection anyway: the others go on meanwhile (taking over
// as soon as a bracket holds one eigenvalue costs 3.5 us more per 16 blocks, at 2 % it costs 4 % more per 16384).
constexpr double EV_SETTLED = 0.005;

// Grid point t: geometric below ghi when ghi > 0 (nine decades), else uniform.
__device__ __forceinline__ double ev_point(int t, double glo, double ghi) {
    if (ghi > 0.0) return ghi * exp2(-(9.0 * 3.321928094887362 / (EV_GRID - 1)) * static_cast<double>(EV_GRID - 1 - t));
    return fma(static_cast<double>(t + 1) * (1.0 / EV_GRID), ghi - glo, glo);
}

struct EvGrid {
    double x[EV_GRID];   // kept: working a point out again takes longer than the search for it
    int cnt[EV_GRID];    // eigenvalues below it
};
__device__ __forceinline__ void ev_grid_point(EvGrid &grid, const double2 *__restrict__ sde, int t, double glo, double ghi) {
    const double x = ev_point(t, glo, ghi);
    grid.x[t] = x;
    grid.cnt[t] = sturm_count(sde, x);
}

struct EvBracket {
    double lo, hi;
    int below, inside;   // eigenvalues below lo, and in the bracket
};

// The settled bracket of the eigenvalue with ascending index `target`, in the scaled units of sde.  LANES lanes of a
// warp share it (`sub`: this lane's number): four look at two levels of bisection at once.  A lane whose bracket is
// settled keeps it while it keeps the others of its warp company, so nothing depends on those.
template <int LANES>
__device__ __forceinline__ EvBracket ev_bracket(const double2 *__restrict__ sde, const EvGrid &grid, int target, int sub, double glo, double ghi) {
    static_assert(LANES == 1 || LANES == 4, "one or two levels of bisection at a time");
    int t = -1;                      // largest grid index with count <= target
#pragma unroll
    for (int step = 64; step > 0; step >>= 1)
        if (t + step < EV_GRID && grid.cnt[t + step] <= target) t += step;
    double lo = (t >= 0) ? grid.x[t] : glo, hi = (t + 1 < EV_GRID) ? grid.x[t + 1] : ghi;
    if (t == EV_GRID - 1) lo = hi;   // cannot happen (every eigenvalue is below the last point); keeps the bracket sane
    int clo = (t >= 0) ? grid.cnt[t] : 0, chi = (t + 1 < EV_GRID) ? grid.cnt[t + 1] : D;
    auto settled = [&] {
        const double mid = fabs(0.5 * (lo + hi)), width = hi - lo;
        return (chi - clo == 1 && width <= fmax(1e-8, EV_SETTLED * mid)) || width <= fmax(2e-15, 1e-8 * mid);
    };
    auto halve = [&](double x, int c) {
        if (settled()) return;
        if (c > target) {
            hi = x;
            chi = c;
        } else {
            lo = x;
            clo = c;
        }
    };
    for (int it = 0; it < EV_MAX_ITER; it += (LANES == 1) ? 1 : 2) {
        if (__all_sync(0xffffffffu, settled())) break;
        const double x = 0.5 * (lo + hi);
        if (LANES == 1) {
            halve(x, sturm_count(sde, x));
        } else {
            const double xl = 0.5 * (lo + x), xh = 0.5 * (x + hi);
            const int c = sturm_count(sde, (sub == 0) ? xl : ((sub == 1) ? x : xh));
            const int c1 = __shfl_sync(0xffffffffu, c, 1, LANES);
            const int c2 = __shfl_sync(0xffffffffu, c, (c1 > target) ? 0 : 2, LANES);
            halve(x, c1);
            halve((c1 > target) ? xl : xh, c2);
        }
    }
    EvBracket b;
    b.lo = lo;
    b.hi = hi;
    b.below = clo;
    b.inside = chi - clo;
    return b;
}

// The eigenvalue in a settled bracket (lanes without one: inside = 0).
__device__ __forceinline__ double ev_root(const double2 *__restrict__ sde, const EvBracket &b) {
    double lo = b.lo, hi = b.hi;
    double x = 0.5 * (lo + hi), last = hi - lo;
    bool done = b.inside != 1;       // (several eigenvalues within 1e-8: their middle)
    for (int it = 0; it < EV_MAX_ITER; ++it) {
        if (__all_sync(0xffffffffu, done)) break;
        double s1, s2;
        const unsigned negative = charpoly_sums(sde, x, s1, s2);
        if (!done) {
            const bool root_above = negative == (static_cast<unsigned>(b.below) & 1u);   // p_d(x) = prod (lambda - x): its sign is that at lo
            if (root_above) lo = x;
            else hi = x;
            const double disc = fmax((D - 1) * fma(static_cast<double>(D), s2, -s1 * s1), 0.0);
            const double root = sqrt(disc);
            const double dx = static_cast<double>(D) / (root_above ? s1 + root : s1 - root);
            const double xn = x + dx;
            done = !(fabs(dx) > fmax(2e-15, fmin(EV_LAGUERRE_STEP * fabs(x), EV_LAGUERRE_RATIO * last))) || (hi - lo) <= fmax(2e-15, 1e-14 * fabs(x));
            last = fabs(dx);
            if (xn >= lo && xn <= hi) x = xn;
            else if (!done) x = 0.5 * (lo + hi);
        }
    }
    return x;
}

// A row of the scaled matrix: its entry of sde and its Gershgorin disc.  s = 1 / the largest magnitude; `before`: the
// off-diagonal entry of the row before (0 for row 0).
__device__ __forceinline__ double2 ev_row(int i, double d, double e, double before, double s, double &glo, double &ghi) {
    const double sd = d * s, se = fabs(e * s), sp = fabs(before * s);
    glo = fmin(glo, sd - se - sp);
    ghi = fmax(ghi, sd + se + sp);
    return make_double2(sd, (i > 0) ? fmax(sp * sp, EV_E2_FLOOR) : 0.0);
}
__device__ __forceinline__ void ev_widen(double &glo, double &ghi) {
    glo = fma(-1e-10, fabs(glo) + 1.0, glo);
    ghi = fma(1e-10, fabs(ghi) + 1.0, ghi);
}

// Step 1 of Algorithm 2: the bulk edge from lambda_{k+1} and lambda_{2k+1}, and whether an eigenvalue passes it.
struct EdgeRule {
    double edge_c, cut;   // 1 / (4^(1/3) - 1), d^(-1/3)
};
__device__ __forceinline__ double bulk_edge(double l_k, double l_2k, const EdgeRule &r) { return fma(r.edge_c, l_k - l_2k, l_k); }
__device__ __forceinline__ bool above_edge(double l, double edge, const EdgeRule &r) { return l / edge - 1.0 > r.cut; }

// With `mark_list` set (first pass over tensor-core Gram matrices), a block whose smallest eigenvalue is not at least
// REDO_RATIO of the largest (this includes non-finite spectra) is queued in mark_list[atomicAdd(mark_count)] for a
// second pass with the exact Gram matrix.

// A CTA of NT threads per block, for calls with too few blocks to fill the SMs with one warp each and for caches that ask
// for the `eig` output (WANTED = D): LANES threads per eigenvalue, the WANTED largest.  A count is a chain of 128
// rows taken from both ends, 64 steps, so where threads are to spare two levels of bisection share one (see launch_eigvals).
template <int LANES, int NT, int WANTED>
__device__ __forceinline__ void eigvals_block(const double *__restrict__ diag, const double *__restrict__ off, double *__restrict__ lam, int blk,
                                              int *__restrict__ mark_list, int *__restrict__ mark_count) {
    constexpr int NWARP = NT / 32;
    __shared__ __align__(16) double2 sde[D];
    __shared__ double s_red[3][NWARP];
    __shared__ EvGrid grid;
    static_assert(NT >= EV_GRID && NT >= D && NT >= LANES * WANTED, "threads for the grid points, the rows and the eigenvalues");
    const int tid = threadIdx.x;
    const size_t base = static_cast<size_t>(blk) * D;
    const bool row = tid < D;
    const double dv = row ? diag[base + tid] : 0.0, ev = (tid < D - 1) ? off[base + tid] : 0.0, ev_prev = (row && tid > 0) ? off[base + tid - 1] : 0.0;
    double m = fmax(fabs(dv), fabs(ev));
    const bool nonfinite = !(fabs(dv) < 1e300) || !(fabs(ev) < 1e300);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((tid & 31) == 0) s_red[0][tid >> 5] = m;
    // a non-finite entry anywhere poisons the whole spectrum: report NaN instead of a bracket
    const int bad = __syncthreads_or(nonfinite);
    m = s_red[0][0];
#pragma unroll
    for (int w = 1; w < NWARP; ++w) m = fmax(m, s_red[0][w]);
    if (bad || m == 0.0) {
        if (row) lam[base + tid] = bad ? nan("") : 0.0;
        if (bad && mark_list && tid == 0) mark_list[atomicAdd(mark_count, 1)] = blk;
        return;
    }
    double glo = 1e300, ghi = -1e300;
    if (row) sde[tid] = ev_row(tid, dv, ev, ev_prev, 1.0 / m, glo, ghi);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        glo = fmin(glo, __shfl_xor_sync(0xffffffffu, glo, o));
        ghi = fmax(ghi, __shfl_xor_sync(0xffffffffu, ghi, o));
    }
    if ((tid & 31) == 0) {
        s_red[1][tid >> 5] = glo;
        s_red[2][tid >> 5] = ghi;
    }
    __syncthreads();
    glo = s_red[1][0];
    ghi = s_red[2][0];
#pragma unroll
    for (int w = 1; w < NWARP; ++w) {
        glo = fmin(glo, s_red[1][w]);
        ghi = fmax(ghi, s_red[2][w]);
    }
    ev_widen(glo, ghi);
    if (tid < EV_GRID) ev_grid_point(grid, sde, tid, glo, ghi);
    __syncthreads();
    // thread t brackets eigenvalue t / LANES (descending); spare threads keep the last one company
    EvBracket b = ev_bracket<LANES>(sde, grid, D - 1 - min(tid / LANES, WANTED - 1), tid % LANES, glo, ghi);
    if constexpr (LANES > 1) {
        // a lane per eigenvalue from here on: the lanes that shared one would only repeat each other
        __shared__ EvBracket s_bracket[WANTED];
        if (tid % LANES == 0 && tid / LANES < WANTED) s_bracket[tid / LANES] = b;
        __syncthreads();
        if (tid >= 32 * ((WANTED + 31) / 32)) return;
        b.inside = 0;
        if (tid < WANTED) b = s_bracket[tid];
    }
    const double x = ev_root(sde, b);
    if (tid < WANTED) lam[base + tid] = x * m;
    if (mark_list && tid < 32) {
        const double x_top = __shfl_sync(0xffffffffu, x, 0);
        const int below = sturm_count(sde, REDO_RATIO * x_top);
        if (tid == 0 && (below > 0 || !(x_top > 0.0))) mark_list[atomicAdd(mark_count, 1)] = blk;
    }
}

template <int LANES, int NT, int WANTED>
__global__ void __launch_bounds__(NT, 640 / NT) eigvals_kernel(const double *diag, const double *off,
                                                               double *lam, int nb, const int *list,
                                                               const int *count, int *mark_list,
                                                               int *mark_count) {
    pdl_wait();
    const int total = list ? *count : nb;
    for (int li = blockIdx.x; li < total; li += gridDim.x) {
        eigvals_block<LANES, NT, WANTED>(diag, off, lam, list ? list[li] : li, mark_list, mark_count);
        __syncthreads();   // the shared state is reused by the next block
    }
}

// One warp per block, lane t resolves lambda_{t+1}, for calls with many blocks: nothing beyond the 32 largest
// eigenvalues is resolved unless the rank turns out to be 10 or 11.
constexpr int EVT_WARPS = 4;     // blocks per CTA

struct EvtShared {
    double2 sde[D];
    EvGrid grid;
};

__global__ void __launch_bounds__(32 * EVT_WARPS, 5) eigvals_top_kernel(const double *diag, const double *off,
                                                                     double *lam, int nb, const int *list,
                                                                     const int *count, int *mark_list,
                                                                     int *mark_count, EdgeRule edge) {
    __shared__ __align__(16) EvtShared shs[EVT_WARPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    EvtShared &sh = shs[warp];
    pdl_wait();
    const int total = list ? *count : nb;
    for (int li = blockIdx.x * EVT_WARPS + warp; li < total; li += gridDim.x * EVT_WARPS) {
        const int blk = list ? list[li] : li;
        const size_t base = static_cast<size_t>(blk) * D;
        double dv[4], ev[4], m = 0.0;
        bool nonfinite = false;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = lane + 32 * q;
            dv[q] = diag[base + i];
            ev[q] = (i < D - 1) ? off[base + i] : 0.0;
            m = fmax(m, fmax(fabs(dv[q]), fabs(ev[q])));
            nonfinite |= !(fabs(dv[q]) < 1e300) || !(fabs(ev[q]) < 1e300);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        const bool bad = __any_sync(0xffffffffu, nonfinite);
        if (bad || m == 0.0) {
            // a non-finite entry poisons the whole spectrum (NaN, and a second pass if there is one); a zero matrix has a zero spectrum
            lam[base + lane] = bad ? nan("") : 0.0;
            if (lane < 2) lam[base + EV_EXPL + lane] = bad ? nan("") : 0.0;
            if (bad && mark_list && lane == 0) mark_list[atomicAdd(mark_count, 1)] = blk;
            continue;
        }
        __syncwarp();   // the previous block's last reads of sde are over
        double glo = 1e300, ghi = -1e300;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = lane + 32 * q;
            double before = __shfl_up_sync(0xffffffffu, ev[q], 1);
            if (lane == 0) before = (q > 0) ? off[base + i - 1] : 0.0;
            sh.sde[i] = ev_row(i, dv[q], ev[q], before, 1.0 / m, glo, ghi);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            glo = fmin(glo, __shfl_xor_sync(0xffffffffu, glo, o));
            ghi = fmax(ghi, __shfl_xor_sync(0xffffffffu, ghi, o));
        }
        ev_widen(glo, ghi);
        __syncwarp();
#pragma unroll 1
        for (int t = lane; t < EV_GRID; t += 32) ev_grid_point(sh.grid, sh.sde, t, glo, ghi);
        __syncwarp();
        const double x = ev_root(sh.sde, ev_bracket<1>(sh.sde, sh.grid, D - 1 - lane, 0, glo, ghi));
        const double l = x * m;
        lam[base + lane] = l;
        // Is the smallest eigenvalue below REDO_RATIO of the largest?  One count tells.
        if (mark_list) {
            const double x_top = __shfl_sync(0xffffffffu, x, 0);
            const int below = sturm_count(sh.sde, REDO_RATIO * x_top);
            if (lane == 0 && (below > 0 || !(x_top > 0.0))) mark_list[atomicAdd(mark_count, 1)] = blk;
        }
        // Ranks 10 and 11 make Step 2 read lambda_{2k+r+1}, index 32 or 33: resolve both then.
        const double lam_plus = bulk_edge(__shfl_sync(0xffffffffu, l, KPILOT), __shfl_sync(0xffffffffu, l, 2 * KPILOT), edge);
        const unsigned passing = __ballot_sync(0xffffffffu, lane <= KPILOT && above_edge(l, lam_plus, edge));
        if (__popc(passing) >= 10) {
            const double x2 = ev_root(sh.sde, ev_bracket<1>(sh.sde, sh.grid, D - 1 - (EV_EXPL + (lane & 1)), 0, glo, ghi));
            if (lane < 2) lam[base + EV_EXPL + lane] = x2 * m;
        }
    }
}

// ------------------------------------------------------------------------------------------
// Algorithm 2 on the spectrum, then the kept eigenvectors from the twisted factorisation of the
// tridiagonal matrix and back-transformation through the stored reflectors.
// ------------------------------------------------------------------------------------------
//
// Every phase here is a chain of dependent latencies (a pivot after a pivot, a reflector after a
// reflector) that leaves most of the CTA idle, so the kernel is laid out for four CTAs of four warps
// per SM, whose chains overlap.  That is what shared memory holds: 46 KB of dynamic memory (12 columns of factor storage,
// as the rank never exceeds the pilot k = 11, in two arrays that the vectors and the ring of reflector stages take over in
// turn) and 8 KB of static, checked below.
constexpr int SP_THREADS = 128, SP_WARPS = SP_THREADS / 32;
constexpr int FAC_LANES = 12;
static_assert(KPILOT < FAC_LANES && KPILOT <= 3 * SP_WARPS, "one factor column and one warp slot per kept vector");

// Back-transformation x = Q1 Q2 y of the kept vectors, normalisation, and the stores of the right singular
// vectors.  Both sets of reflectors are staged through a ring of four places in shared memory, three stages ahead.
//   Q2, the bulge chasing's, sweep after sweep backwards: the reflectors of a sweep act on disjoint groups
//       of four rows, so a lane owns the rows of a hop, a warp a vector (vectors w, w + 4, w + 8 side by side: a reflector is read
//       once for all of them); from sweep to sweep the groups move by one row, which is one shuffle (the registers
//       move by writing the update's results one place up).
//   Q1, the band reduction's panels, two at a time, as products of 8 x 8 tiles on the fp64 tensor instruction:
//       X^T (eight vectors at a time) stays in registers as accumulators, which are operands too.
// dynamic shared memory: the ratios and vectors [D][12], and the ring, two places of which are the second
// factor array [D][12] until they are needed.
constexpr int BT_STAGE = 64 * (GRAM_TILE_ROWS + 1);   // doubles per stage: eight sweeps, or a column of tiles of V and its T
constexpr int BT_STAGES = 2 * GRAM_TILE_ROWS, BT_RING = 4;   // four in shared memory: three on their way cover the latency of the memory
constexpr size_t SPECTRAL_DYN_SMEM = sizeof(double) * (D * FAC_LANES + BT_RING * BT_STAGE);
static_assert(4 * (SPECTRAL_DYN_SMEM + 8 * 1024 + 1024) <= 228 * 1024, "four CTAs per SM (8 KB static, 1 KB of the system's each)");
static_assert(KPILOT <= 3 * SP_WARPS, "three vectors per warp");
static_assert(D * FAC_LANES >= 16 * TILE_ELEMS && 2 * BT_STAGE >= D * FAC_LANES, "the second factor array fits two places of the ring");
// the first two stages go to the places that the second factor array does not take
__device__ __forceinline__ double *bt_place(double *ring, int n) { return ring + ((n + 2) & (BT_RING - 1)) * BT_STAGE; }

// Stage n of the back-transformation: sweeps with (s + 2) / 8 = 15 - n, then tile column 31 - n of V.  A column goes
// in groups of four tile rows, with zeros above its first tile: the tile of row i at 1 + i - 4 (j / 4), T at 0.
__device__ __forceinline__ void bt_fetch(double *ring, int n, const double *__restrict__ q2, const double *__restrict__ tiles,
                                         const double *__restrict__ tmat, int warp, int lane) {
    double *const dst = bt_place(ring, n) + 2 * lane;
    if (n < GRAM_TILE_ROWS) {
        const int g = GRAM_TILE_ROWS - 1 - n;
        const double *src = q2 + sweep_group_offset(g) + 2 * lane;
#pragma unroll 1
        for (int q = warp; q < GRAM_TILE_ROWS - g; q += SP_WARPS) cp_async16(dst + q * TILE_ELEMS, src + q * TILE_ELEMS);
    } else if (n < BT_STAGES) {
        const int j = BT_STAGES - 1 - n, i0 = j & ~3;
        if (warp == 0) cp_async16(dst, tmat + j * TILE_ELEMS + 2 * lane);
#pragma unroll 1
        for (int i = i0 + warp; i < GRAM_TILE_ROWS; i += SP_WARPS) {
            double *d = dst + (i - i0 + 1) * TILE_ELEMS;
            if (i < j) *reinterpret_cast<double2 *>(d) = make_double2(0.0, 0.0);
            else cp_async16(d, tiles + tile_index(i, j) * TILE_ELEMS + 2 * lane);
        }
    }
    cp_async_commit();
}

// The reflectors of one sweep (u: this lane's) applied to N vectors.  x[v][k] of lane hl is row s + 1 + 4 hl + k before
// sweep s and row s + 4 hl + k after it; the last row goes to the next lane.  The last lane's last row is past the end of the matrix,
// and its reflector has a zero there: the entry s that enters at lane 0 (`top`) starts from that place and comes round with the
// same shuffle.  A sweep waits for the one before through x[0] alone, which therefore comes last in the sum.
constexpr int BT_VECTORS = 3;   // of one warp, at most
template <int N>
__device__ __forceinline__ void bt_sweep(double (&x)[BT_VECTORS][4], const double2 (&u)[2], const double (&top)[BT_VECTORS], int hl) {
    double g[BT_VECTORS];
#pragma unroll
    for (int v = 0; v < N; ++v) {
        if (hl == 31) x[v][3] = top[v];
        g[v] = fma(u[1].y, x[v][3], fma(u[1].x, x[v][2], u[0].y * x[v][1]));
    }
#pragma unroll
    for (int v = 0; v < N; ++v) {
        g[v] = fma(u[0].x, x[v][0], g[v]);
        const double up = __shfl_sync(0xffffffffu, fma(-g[v], u[1].y, x[v][3]), (hl + 31) & 31);
        x[v][3] = fma(-g[v], u[1].x, x[v][2]);
        x[v][2] = fma(-g[v], u[0].y, x[v][1]);
        x[v][1] = fma(-g[v], u[0].x, x[v][0]);
        x[v][0] = up;
    }
}

// The sweeps of a stage, last one first (eight, or six of the very last stage).  p, q: the two pieces of this lane's reflector of the last
// sweep, `stride` 16-byte pieces per sweep; pt: the first vector's entry that enters after it (the others' 4 and 8 further on).
template <int N>
__device__ __forceinline__ void bt_sweeps(double (&x)[BT_VECTORS][4], const double2 *__restrict__ p, const double2 *__restrict__ q, int stride,
                                          const double *__restrict__ pt, int hl, bool six) {
    double2 u[2] = {*p, *q}, w[2];
    double top[BT_VECTORS], next[BT_VECTORS];
#pragma unroll
    for (int v = 0; v < N; ++v) top[v] = pt[4 * v];
#pragma unroll
    for (int e = 7; e >= 0; --e) {
        if (e == 1 && six) break;
        if (e > 0) {
            p -= stride;
            q -= stride;
            w[0] = *p;
            w[1] = *q;
            const int back = ((e <= 2 && six) ? 5 : 8 - e) * FAC_LANES;
#pragma unroll
            for (int v = 0; v < N; ++v) next[v] = pt[4 * v - back];
        }
        bt_sweep<N>(x, u, top, hl);
#pragma unroll
        for (int h = 0; h < 2; ++h) u[h] = w[h];
#pragma unroll
        for (int v = 0; v < N; ++v) top[v] = next[v];
    }
}

// Stage n of Q1 for tile rows w, w + 4, .. of which the last 4 - A0 have tiles of V in this column (j = the column, 4 A0 <= j < 4 A0 + 4).
// The warps' parts meet in shared memory; what else has to happen there comes with `meet`.
template <int A0, bool TWO, typename F>
__device__ __forceinline__ void bt_column(F &&meet, double (&X)[2][4][2], const double *__restrict__ T, const double *__restrict__ st, double *__restrict__ part, int warp,
                                          int o_row, int o_c0, int o_c1) {
    double wa[2][2] = {{0.0, 0.0}, {0.0, 0.0}}, wb[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
    double v0[4], v1[4];
#pragma unroll
    for (int a = A0; a < 4; ++a) {
        v0[a] = st[4 * a * TILE_ELEMS + o_c0];
        v1[a] = st[4 * a * TILE_ELEMS + o_c1];
    }
#pragma unroll
    for (int a = A0; a < 4; ++a) {
        dmma(wa[0], X[0][a][0], v0[a]);
        if (TWO) dmma(wa[1], X[1][a][0], v0[a]);
        dmma(wb[0], X[0][a][1], v1[a]);
        if (TWO) dmma(wb[1], X[1][a][1], v1[a]);
    }
#pragma unroll
    for (int h = 0; h < (TWO ? 2 : 1); ++h)
        *reinterpret_cast<double2 *>(part + (4 * h + warp) * TILE_ELEMS + o_row) = make_double2(wa[h][0] + wb[h][0], wa[h][1] + wb[h][1]);
    const double2 tr = *reinterpret_cast<const double2 *>(T + o_row);
    double2 v[4];
#pragma unroll
    for (int a = A0; a < 4; ++a) v[a] = *reinterpret_cast<const double2 *>(st + 4 * a * TILE_ELEMS + o_row);
    meet();
    double w[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll
    for (int h = 0; h < (TWO ? 2 : 1); ++h) {
        double2 q[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) q[e] = *reinterpret_cast<const double2 *>(part + (4 * h + e) * TILE_ELEMS + o_row);
        dmma(w[h], -((q[0].x + q[1].x) + (q[2].x + q[3].x)), tr.x);
        dmma(w[h], -((q[0].y + q[1].y) + (q[2].y + q[3].y)), tr.y);
    }
#pragma unroll
    for (int h = 0; h < (TWO ? 2 : 1); ++h) {
#pragma unroll
        for (int a = A0; a < 4; ++a) dmma(X[h][a], w[h][0], v[a].x);
#pragma unroll
        for (int a = A0; a < 4; ++a) dmma(X[h][a], w[h][1], v[a].y);
    }
}

template <bool MEET_ONCE>
__device__ __forceinline__ void sp_back_transform(const double *__restrict__ q2, const double *__restrict__ tiles, const double *__restrict__ tmat,
                                                  double *__restrict__ yv, double *__restrict__ ring, const double *__restrict__ zeros, int rank, int tid,
                                                  float *__restrict__ vr, const eosq_cache_t &out, long long gb) {
    const int lane = tid & 31, warp = tid >> 5;
    bt_fetch(ring, 2, q2, tiles, tmat, warp, lane);
    {
        const int count = (rank - warp + SP_WARPS - 1) / SP_WARPS;   // vectors warp, warp + 4, warp + 8
        double x[BT_VECTORS][4];
#pragma unroll
        for (int v = 0; v < BT_VECTORS; ++v)
#pragma unroll
            for (int k = 0; k < 4; ++k) x[v][k] = (lane == 0 && k < 2 && v < count) ? yv[(D - 2 + k) * FAC_LANES + warp + 4 * v] : 0.0;
        const int chunk = lane >> 1, swz = (chunk >> 1) & 3, p0 = (2 * (lane & 1)) ^ swz, p1 = (2 * (lane & 1) + 1) ^ swz;
#pragma unroll 1
        for (int n = 0; n < GRAM_TILE_ROWS; ++n) {
            const int g = GRAM_TILE_ROWS - 1 - n, nh = GRAM_TILE_ROWS - g;
            cp_async_wait_group<2>();
            __syncthreads();   // stage n is there, and everybody is done with stage n - 1
            bt_fetch(ring, n + 3, q2, tiles, tmat, warp, lane);
            if (count > 0) {
                // sweep s of the stage at (s + 2 - 8 g) * 8 nh; a lane beyond the last chunk reads zeros.  All eight sweeps in
                // one piece, their operands fetched one sweep ahead.
                const bool mine = chunk < nh, six = n == GRAM_TILE_ROWS - 1;
                const int stride = mine ? 4 * nh : 0;
                const double2 *p = reinterpret_cast<const double2 *>(mine ? bt_place(ring, n) + 8 * chunk : zeros) + 7 * stride;
                const double *pt = yv + (8 * g + 5) * FAC_LANES + warp;
                if (count == 3) bt_sweeps<3>(x, p + p0, p + p1, stride, pt, lane, six);
                else if (count == 2) bt_sweeps<2>(x, p + p0, p + p1, stride, pt, lane, six);
                else bt_sweeps<1>(x, p + p0, p + p1, stride, pt, lane, six);
            }
        }
#pragma unroll
        for (int v = 0; v < BT_VECTORS; ++v)
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (v < count) yv[(4 * lane + k) * FAC_LANES + warp + 4 * v] = x[v][k];
    }
    __syncthreads();
    // Q1 as X^T <- X^T - ((X^T V) T^T) V^T.  Warp w has the tile rows w, w + 4, w + 8, w + 12 of X^T (eight
    // vectors, and another eight if the rank is above eight); the warps' parts of X^T V meet in shared memory.
    const int m = lane >> 2, k = lane & 3;
    const int o_row = tile_off(m, 2 * k), o_c0 = tile_off(2 * k, m), o_c1 = tile_off(2 * k + 1, m);
    const bool two = rank > 8;
    double X[2][4][2];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int vi = 8 * h + m;
                X[h][a][e] = (vi < rank) ? yv[(8 * (warp + 4 * a) + 2 * k + e) * FAC_LANES + vi] : 0.0;
            }
    if constexpr (MEET_ONCE) cp_async_wait_group<2>();
    __syncthreads();   // yv's place is taken by the parts: [parity of the stage][h][warp][64] (and, meeting once per stage, the first is there)
    double *const parts = yv;
#pragma unroll 1
    for (int n = GRAM_TILE_ROWS; n < BT_STAGES; ++n) {
        const int j = BT_STAGES - 1 - n;
        if constexpr (!MEET_ONCE) {
            cp_async_wait_group<2>();
            __syncthreads();   // stage n is there, and everybody is done with stage n - 1
            bt_fetch(ring, n + 3, q2, tiles, tmat, warp, lane);
        }
        auto meet = [&] {
            // one barrier per stage: the parts of stage n and the whole of stage n + 1 are there, and everybody is done with stage n - 1
            if constexpr (MEET_ONCE) cp_async_wait_group<1>();
            __syncthreads();
            if constexpr (MEET_ONCE) bt_fetch(ring, n + 3, q2, tiles, tmat, warp, lane);
        };
        const double *const T = bt_place(ring, n), *const st = T + (1 + warp - (j & ~3)) * TILE_ELEMS;   // tile of row warp + 4 a at st + 256 a
        double *const part = parts + (n & 1) * 8 * TILE_ELEMS;
        auto column = [&](auto a0) {
            if (two) bt_column<decltype(a0)::value, true>(meet, X, T, st, part, warp, o_row, o_c0, o_c1);
            else bt_column<decltype(a0)::value, false>(meet, X, T, st, part, warp, o_row, o_c0, o_c1);
        };
        switch (j >> 2) {
            case 0: column(std::integral_constant<int, 0>()); break;
            case 1: column(std::integral_constant<int, 1>()); break;
            case 2: column(std::integral_constant<int, 2>()); break;
            default: column(std::integral_constant<int, 3>()); break;
        }
    }
    // norms: the warps' sums of squares of the sixteen vectors
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        double nn = 0.0;
#pragma unroll
        for (int a = 0; a < 4; ++a) nn = fma(X[h][a][0], X[h][a][0], fma(X[h][a][1], X[h][a][1], nn));
        nn += __shfl_xor_sync(0xffffffffu, nn, 1);
        nn += __shfl_xor_sync(0xffffffffu, nn, 2);
        if (k == 0) parts[(8 * h + m) * 4 + warp] = nn;
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int vi = 8 * h + m;
        if (vi >= rank) continue;
        const double nn = (parts[vi * 4] + parts[vi * 4 + 1]) + (parts[vi * 4 + 2] + parts[vi * 4 + 3]);
        const double rn = (nn > 0.0) ? rsqrt(nn) : 0.0;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int row = 8 * (warp + 4 * a) + 2 * k;
            const float f0 = static_cast<float>(X[h][a][0] * rn), f1 = static_cast<float>(X[h][a][1] * rn);
            *reinterpret_cast<float2 *>(vr + vi * D + row) = make_float2(f0, f1);
            *reinterpret_cast<uint32_t *>(out.V + (gb * RMAX + vi) * D + row) =
                static_cast<uint32_t>(__half_as_ushort(__float2half_rn(f0))) | (static_cast<uint32_t>(__half_as_ushort(__float2half_rn(f1))) << 16);
            if (out.vr32) *reinterpret_cast<float2 *>(out.vr32 + (gb * RMAX + vi) * D + row) = make_float2(f0, f1);
        }
    }
}

// Constants of Algorithm 2, from the host: the edge rule's, and (1 - (j / k)^(2/3)) / (4^(1/3) - 1) for j = 1 .. k.
struct SpectralConstants {
    EdgeRule edge;
    double imputed[KPILOT];
};

template <bool MEET_ONCE>
__global__ void __launch_bounds__(SP_THREADS, 4) spectral_kernel(int n, Workspace ws, eosq_cache_t out, long long block0, bool full, SpectralConstants cst) {
    __shared__ double lam[D], dd[D], ee[D], atoms[D];
    __shared__ __align__(16) double2 sde[D];  // (d_i, e_{i-1}^2) of the scaled matrix, for the characteristic polynomial
    __shared__ double st1[6 * KPILOT], st2[6 * KPILOT];   // weighted samples of the tail sums around each kept eigenvalue
    __shared__ double s_max[SP_WARPS];
    __shared__ double s_phi[RMAX], s_sig[RMAX];
    __shared__ unsigned s_flags;
    __shared__ int s_twist[FAC_LANES];
    __shared__ double s_imputed[KPILOT], s_ms[KPILOT], s_msp[KPILOT];
    __shared__ __align__(16) double s_zero[8];
    extern __shared__ __align__(16) double dyn[];
    double *yv = dyn;                        // e_i / D+_i, then the vectors                       [D][12]
    double *fb = dyn + D * FAC_LANES;         // e_i / D-_{i+1}                                     [D][12]
    double *ring = dyn + D * FAC_LANES;       // the back-transformation's stages (fb takes two places of four until they are needed)

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = blockIdx.x;
    const long long gb = block0 + b;
    const size_t base = static_cast<size_t>(b) * D;
    pdl_wait();
    pdl_trigger();   // (the quantiser: one CTA per SM, its set-up fits next to the last CTAs here)
    {
        // lam[EV_TOP .. D-2] holds eigenvalues only when the full spectrum was asked for
        lam[tid] = (full || tid < EV_TOP) ? ws.lam[base + tid] : 0.0;   // (indices 32, 33: only meaningful, and only read, for ranks 10, 11)
        dd[tid] = ws.diag[base + tid];
        ee[tid] = ws.off[base + tid];
        double mx = fmax(fabs(dd[tid]), fabs(ee[tid]));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane == 0) s_max[warp] = mx;
    }
    if (tid < RMAX) {
        s_phi[tid] = 0.0;
        s_sig[tid] = 0.0;
    }
    const double *const bq2 = ws.q2 + static_cast<size_t>(b) * GRAM_ELEMS, *const bv = ws.gram + static_cast<size_t>(b) * GRAM_ELEMS,
                 *const bt = ws.tmat + static_cast<size_t>(b) * GRAM_TILE_ROWS * TILE_ELEMS;
    bt_fetch(ring, 0, bq2, bv, bt, warp, lane);
    bt_fetch(ring, 1, bq2, bv, bt, warp, lane);
    if (tid < 8) s_zero[tid] = 0.0;
    if (tid < KPILOT) s_imputed[tid] = cst.imputed[tid];
    if (tid == 0) s_flags = 0u;
    __syncthreads();
    const double mscale = fmax(fmax(s_max[0], s_max[1]), fmax(s_max[2], s_max[3]));

    // Step 1: bulk edge from lambda_{k+1}, lambda_{2k+1} (1-based) and the rank test.
    const double lam_plus = bulk_edge(lam[KPILOT], lam[2 * KPILOT], cst.edge);
    const bool pass = (tid <= KPILOT) && above_edge(lam[tid], lam_plus, cst.edge);
    int rank = __syncthreads_count(pass);
    if (tid == 0) {
        unsigned f = 0u;
        if (!(lam[0] == lam[0]) || !(lam[0] < 1e300) || !(lam_plus == lam_plus)) f |= EOSQ_BLOCK_NONFINITE;
        if (rank > KPILOT) f |= EOSQ_BLOCK_NONFINITE;
        if (f) atomicOr(&s_flags, f);
    }
    if (rank > KPILOT) rank = KPILOT;

    if (rank > 0) {
        // Step 2: k imputed atoms behind the outliers; the observed eigenvalues after them are known
        // one by one up to lambda_EV_EXPL, the rest (the tail) only through sums.
        {
            double a = 0.0;
            if (tid >= rank + KPILOT && tid < EV_EXPL) a = lam[tid];
            else if (tid >= rank && tid < rank + KPILOT) {
                const int jj = tid - rank + 1;
                const double bs = lam[KPILOT + rank];
                const double gap = bs - lam[2 * KPILOT + rank];
                a = fma(s_imputed[jj - 1], gap, bs);
            }
            atoms[tid] = a;
        }
        const double floor_piv = 1.2e-16 * fmax(fabs(lam[0]), 1e-280), inv_floor = 1.0 / floor_piv;
        {
            const double is = (mscale > 0.0) ? 1.0 / mscale : 0.0;
            const double se = (tid > 0) ? fabs(ee[tid - 1] * is) : 0.0;
            sde[tid] = make_double2(dd[tid] * is, (tid > 0) ? fmax(se * se, EV_E2_FLOOR) : 0.0);
        }
        __syncthreads();
        // Tail sums  sum_{j > EV_EXPL} 1 / (lambda_j - z)  and  sum 1 / (lambda_j - z)^2  at z = lambda_i:
        // the sums over the whole spectrum have a pole at z, so they are taken at six points
        // z + m h, m = -3 .. 3 without 0, the known eigenvalues are subtracted there, and what is left
        // (smooth: the tail lies well below z) is interpolated to z, exact for polynomials of degree 5.
        // h = z / 64, or a little less when a known eigenvalue would sit on a sample point.
        // Warps 1 .. 3 take these sums and Step 3 while warp 0 factorises for the eigenvectors below.
        if (warp > 0) {
            const int e = tid - 32;
            if (e < 6 * rank) {
                const int i = e / 6, m6 = e % 6;
                const int mm = (m6 < 3) ? m6 - 3 : m6 - 2;   // -3, -2, -1, 1, 2, 3
                const double z = lam[i];
                // A known eigenvalue right at a sample point would be subtracted with a large
                // cancellation error: shrink h until every other known eigenvalue keeps a quarter
                // step away from all six points (the six threads of a vector find the same h).
                // (Only neighbours within three and a half steps matter: they are looked for outwards from i.)
                double h = z * (1.0 / 64.0);
#pragma unroll 1
                for (int attempt = 0; attempt < 8; ++attempt) {
                    const double reach = 3.5 * h, ih = sp_rcp(h);
                    bool near = false;
                    auto look = [&](double dist) {   // true while there may be more
                        if (!(dist < reach)) return false;
                        const double t = dist * ih;
                        near |= t >= 0.5 && fabs(t - rint(t)) < 0.25;
                        return true;
                    };
#pragma unroll 1
                    for (int j = i - 1; j >= 0 && look(lam[j] - z); --j) {}
#pragma unroll 1
                    for (int j = i + 1; j < EV_EXPL && look(z - lam[j]); ++j) {}
                    if (!near) break;
                    h *= 0.8125;
                }
                const double x = fma(static_cast<double>(mm), h, z);
                const double is = sp_rcp(mscale);
                double f1, f2;
                charpoly_sums(sde, x * is, f1, f2);
                f1 *= is;
                f2 *= is * is;
#pragma unroll 8
                for (int j = 0; j < EV_EXPL; ++j) {
                    const double inv = sp_rcp(lam[j] - x);
                    f1 -= inv;
                    f2 = fma(-inv, inv, f2);
                }
                const int am = (mm < 0) ? -mm : mm;
                const double w = (am == 1) ? 15.0 / 20.0 : ((am == 2) ? -6.0 / 20.0 : 1.0 / 20.0);
                st1[e] = w * f1;
                st2[e] = w * f2;
            }
            asm volatile("bar.sync 1, 96;" ::: "memory");
            // Step 3: Stieltjes transforms of F_e at z = lambda_i, a warp each ..
            for (int i = warp - 1; i < rank; i += SP_WARPS - 1) {
                const int j = rank + lane;
                const double inv = (j < EV_EXPL) ? sp_rcp(atoms[min(j, EV_EXPL - 1)] - lam[i]) : 0.0;
                double ms = inv, msp = inv * inv;
                if (lane < 6) {
                    ms += st1[6 * i + lane];
                    msp += st2[6 * i + lane];
                }
                ms = warp_sum(ms);
                msp = warp_sum(msp);
                if (lane == 0) {
                    s_ms[i] = ms;
                    s_msp[i] = msp;
                }
            }
            asm volatile("bar.sync 1, 96;" ::: "memory");
            // .. D-transform, Eq. 9, Eq. 6, a lane each.
            if (warp == 1 && lane < rank) {
                const int i = lane;
                const double z = lam[i];
                const double nn = static_cast<double>(D - rank);
                const double ms = s_ms[i] / nn, msp = s_msp[i] / nn;
                const double ratio = static_cast<double>(D) / static_cast<double>(n);
                const double m1 = ratio * ms - (1.0 - ratio) / z;  // n x n side: n - d extra zeros
                const double m1p = ratio * msp + (1.0 - ratio) / (z * z);
                const double m2 = ms, m2p = msp;                   // d x d side
                const double T = z * m1 * m2;
                const double Tp = m1 * m2 + z * (m1p * m2 + m1 * m2p);
                const double dh = 1.0 / sqrt(T);
                const double a1 = m1 / (dh * dh * Tp), a2 = m2 / (dh * dh * Tp);
                double ph = dh * sqrt(a1 * a2);
                const double sg = sqrt(z);
                if (!(ph >= 0.0) || !(ph < 1e300)) {
                    ph = 0.0;
                    atomicOr(&s_flags, EOSQ_BLOCK_CLAMPED);
                } else if (ph > sg) {
                    ph = sg;
                    atomicOr(&s_flags, EOSQ_BLOCK_CLAMPED);
                }
                s_phi[i] = ph;
                s_sig[i] = sg;
                if (i > 0 && (lam[i - 1] - z) < 1e-9 * lam[i - 1]) atomicOr(&s_flags, EOSQ_BLOCK_CLUSTERED);
            }
        }

        // Kept eigenvectors of the tridiagonal matrix from its twisted factorisation: with the
        // pivots of T - mu I = L+ D+ L+^T taken from the top,  D+_{i+1} = (d_{i+1} - mu) - e_i^2 / D+_i,
        // and of U- D- U-^T taken from the bottom,  D-_i = (d_i - mu) - e_i^2 / D-_{i+1},
        // gamma_i = D+_i + D-_i - (d_i - mu) is the residual of the vector z that starts with z_r = 1
        // at index r and runs  z_i = -(e_i / D+_i) z_{i+1}  upwards and  z_{i+1} = -(e_i / D-_{i+1}) z_i
        // downwards: (T - mu I) z = gamma_r e_r.  r = argmin |gamma| gives a residual of the order of
        // the error of mu, which is at rounding level here, so one such vector is as good as inverse
        // iteration converged.  Lanes c and c + 16 of warp 0 take the two directions for vector c side by side
        // and leave the ratios (column c of the arrays), from which the pivots follow.
        if (warp == 0 && (lane & 15) < rank) {
            const int c = lane & 15;
            const bool down = lane >= 16;
            const double mu = lam[c];
            double *const ratio = (down ? fb + (D - 2) * FAC_LANES : yv) + c;
            const double *const pe = ee + (down ? D - 2 : 0), *const pd = dd + (down ? D - 2 : 1);
            const int step = down ? -1 : 1;
            double piv = dd[down ? D - 1 : 0] - mu;
#pragma unroll 4
            for (int i = 0; i < D - 1; ++i) {
                const double e = pe[i * step], next = pd[i * step] - mu;
                const bool small = !(fabs(piv) >= floor_piv);
                const double r = small ? ((piv < 0.0) ? -inv_floor : inv_floor) : sp_rcp(piv);
                const double q = e * r;
                ratio[i * step * FAC_LANES] = q;
                piv = fma(-q, e, next);
            }
        }
    }
    __syncthreads();
    if (rank > 0) {
        // Twist index of every vector (a warp each): gamma_i = (d_i - mu) - e_{i-1} (e_{i-1} / D+_{i-1}) - e_i (e_i / D-_{i+1}),
        // the smallest by the upper bits of its magnitude (to 1e-4, ties to the higher index), the index in the lower ones.
        for (int c = warp; c < rank; c += SP_WARPS) {
            const double mu = lam[c];
            unsigned best = 0xffffffffu;
#pragma unroll
            for (int q = 0; q < D / 32; ++q) {
                const int i = lane + 32 * q;
                const int above = max(i - 1, 0), here = min(i, D - 2);
                const double ea = ee[above], eh = ee[here], ra = yv[above * FAC_LANES + c], rh = fb[here * FAC_LANES + c];
                double gam = dd[i] - mu;
                gam = fma((i > 0) ? -ea : 0.0, ra, gam);
                gam = fma((i < D - 1) ? -eh : 0.0, rh, gam);
                best = min(best, (static_cast<unsigned>(__double2hiint(gam)) & 0x7fffff80u) | static_cast<unsigned>(D - 1 - i));
            }
            best = __reduce_min_sync(0xffffffffu, best);
            if (lane == 0) s_twist[c] = D - 1 - static_cast<int>(best & 127u);
        }
    }
    __syncthreads();
    // The vectors, left unnormalised (the back-transformation normalises at the end): lane 2 c upwards, lane 2 c + 1
    // downwards from the twist.  (One chain of up to 127 products; split over the four warps, each working out the product of its 32 factors
    // first: 39 us against 38 for 16 and 128 blocks, 74.3 against 73.3 for 592, the same for 2 and for 16384.)
    if (warp == 0 && (lane >> 1) < rank) {
        const int c = lane >> 1, r = s_twist[c];
        const bool up = !(lane & 1);
        const int count = up ? r : D - 1 - r, step = up ? -FAC_LANES : FAC_LANES;
        const double *src = (up ? yv + (r - 1) * FAC_LANES : fb + r * FAC_LANES) + c;
        double *dst = yv + (up ? r - 1 : r + 1) * FAC_LANES + c;
        double z = 1.0, ss = 0.0, f[8];
        if (up) yv[r * FAC_LANES + c] = 1.0;
        // (reads past the end are clamped, not skipped: a branch per entry would cost more than the entry)
#pragma unroll
        for (int q = 0; q < 8; ++q) f[q] = -src[min(q, count - 1) * step];
#pragma unroll 1
        for (int i = 0; i < count; i += 8) {
            double nx[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) nx[q] = -src[min(i + 8 + q, count - 1) * step];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                z *= f[q];
                const bool in = i + q < count;
                if (in) dst[(i + q) * step] = z;
                const double zz = in ? z : 0.0;
                ss = fma(zz, zz, ss);
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) f[q] = nx[q];
        }
        if (!(ss < 1e300)) atomicOr(&s_flags, EOSQ_BLOCK_NOT_CONVERGED);
    }
    __syncthreads();

    // Back-transformation of the kept vectors (its stages take the place of the factorisations, which
    // are no longer needed after the barrier above).
    float *vr = ws.vr + static_cast<size_t>(b) * RMAX * D;
    if (rank > 0) sp_back_transform<MEET_ONCE>(bq2, bv, bt, yv, ring, s_zero, rank, tid, vr, out, gb);
    else cp_async_wait_all();   // (the stages asked for ahead must have landed before the CTA leaves)
    // rows >= rank of V are zero; scalars
    for (int e = tid; e < RMAX * D; e += SP_THREADS) {
        if (e / D >= rank) {
            out.V[gb * RMAX * D + e] = 0;
            vr[e] = 0.0f;
            if (out.vr32) out.vr32[gb * RMAX * D + e] = 0.0f;
        }
    }
    if (tid < RMAX) {
        const float sg = static_cast<float>(s_sig[tid]);
        const float ph = static_cast<float>(s_phi[tid]);
        const float cf = (tid < rank && s_sig[tid] > 0.0) ? static_cast<float>(s_phi[tid] / s_sig[tid]) : 0.0f;
        out.sigma[gb * RMAX + tid] = sg;
        out.phi[gb * RMAX + tid] = ph;
        ws.coef[static_cast<size_t>(b) * RMAX + tid] = cf;
        if (out.coef) out.coef[gb * RMAX + tid] = cf;
    }
    if (full && out.eig) out.eig[gb * D + tid] = static_cast<float>(lam[tid]);
    if (tid == 0) {
        out.rank[gb] = rank;
        ws.rank[b] = rank;
        out.status[gb] = static_cast<int32_t>(s_flags);
        if (out.lambda_plus) out.lambda_plus[gb] = static_cast<float>(lam_plus);
    }
}

// Blocks that a launch over a list has CTAs for (it loops over longer lists): the list is almost always empty, and
// thousands of CTAs that find nothing to do would cost more than the launch.
constexpr int64_t LIST_BLOCKS = 2368;
static const SpectralConstants &spectral_constants() {
    static const SpectralConstants cst = [] {
        SpectralConstants c;
        c.edge.edge_c = 1.0 / (std::cbrt(4.0) - 1.0);
        c.edge.cut = 1.0 / std::cbrt(static_cast<double>(D));
        for (int j = 1; j <= KPILOT; ++j) c.imputed[j - 1] = (1.0 - std::pow(static_cast<double>(j) / KPILOT, 2.0 / 3.0)) * c.edge.edge_c;
        return c;
    }();
    return cst;
}

// Which kernel runs changes the time only.  Up to four blocks per SM a CTA of 160 threads per block, four of which fit an SM:
// 23 us for 16 blocks and 43 for 592, where one warp per block takes a third to a half more (its second round, for ranks 10
// and 11, doubles its chain).  Beyond, the warps' lower total wins: 54 us for 700 blocks, 58 for 1184, 446 for 16384, where the wide kernel
// takes as much for 593, 1.4 times that for 1200 and 2.4 times for 16384.  The whole spectrum with four threads per eigenvalue: no faster for two blocks, 10 % of an
// encode slower for 304.
void launch_eigvals(int64_t nb, const Workspace &ws, const int *list, const int *count, int *mark_list, bool full, int sm_count, cudaStream_t s) {
    const int64_t work = list ? std::min<int64_t>(nb, LIST_BLOCKS) : nb;
    const int n = static_cast<int>(nb);
    if (full)
        launch_dependent(eigvals_kernel<1, D, D>, static_cast<unsigned>(work), D, 0, s, ws.diag, ws.off, ws.lam, n, list, count, mark_list, ws.redo_count);
    else if (nb <= 4 * static_cast<int64_t>(sm_count))
        launch_dependent(eigvals_kernel<4, 160, EV_TOP>, static_cast<unsigned>(work), 160, 0, s, ws.diag, ws.off, ws.lam, n, list, count, mark_list, ws.redo_count);
    else
        launch_dependent(eigvals_top_kernel, static_cast<unsigned>((work + EVT_WARPS - 1) / EVT_WARPS), 32 * EVT_WARPS, 0, s, ws.diag, ws.off, ws.lam, n, list, count,
                         mark_list, ws.redo_count, spectral_constants().edge);
}

// One barrier per stage of the panels' back-transformation shortens the chain, but waits for a stage's copies a stage ahead, which costs
// once the SM's other blocks fill the gaps anyway: 33 us against 35 for 2 blocks, 74 against 76 for 592, 235 against 237 for 2368, the same
// for 2960, 1.58 ms against 1.54 for 16384.  So: up to twenty blocks per SM.  The bits are the same.
void launch_spectral(int64_t nb, int n, const Workspace &ws, const eosq_cache_t &out, int64_t block0, bool full, int sm_count,
                     cudaStream_t s) {
    const auto kernel = (nb <= 20 * static_cast<int64_t>(sm_count)) ? spectral_kernel<true> : spectral_kernel<false>;
    ensure_dynamic_smem(reinterpret_cast<const void *>(kernel), SPECTRAL_DYN_SMEM);
    launch_dependent(kernel, static_cast<unsigned>(nb), SP_THREADS, SPECTRAL_DYN_SMEM, s, n, ws, out, static_cast<long long>(block0), full, spectral_constants());
}

}  // namespace eosq
