// fwd_sweeps64.cuh -- FP64 2D split step as two sweep passes (Eq. swe, Sec.
// 5; Roe-type f-wave solver per edge, Sec. 6), with or without the wet/dry
// option.
//
// The FP64 units bound this step (ops64.cuh), so it is laid out for the
// fewest FP64 operations per cell.  A pass sweeps along one direction; each
// lane walks a segment of one line of cells (a row in the x-pass, a column in
// the y-pass) and solves, limits and updates in registers, so every edge is
// solved and limited once but for the ends of segments.  No halo rows are
// swept twice (a 32 x 4 tile with halos solved the x-edges 2.2 times and
// limited every edge twice), and the passes' extra trip through memory costs
// nothing beside the arithmetic.  What needs no FP64 operation takes none:
// signs, comparisons, minima and halvings work on the words of a double, and
// the divisions of the CFL number by dx and dy are left to the end (a
// division by a positive constant is monotone under rounding, so the largest
// quotient is the quotient of the largest).
// The x-pass reads buffer cur and writes the x-swept state to the other one,
// the y-pass reads that and writes the new state back to buffer cur.
// Measured, us per step, tiles / sweeps with quotients and roots of 3 and 6
// FP64 operations / so (none): 512^2 (waves over 60 %) 721 / 216 / 154, 2048^2
// 10400 / 2050 / 1448; 511 x 350 with wet/dry (a third land) 672 / 300 / 244.
// The FP64 units stay what bounds it, with about 95 operations a cell and pass
// (the cell's products formed once, not for both its edges: 3 % of it).
//
// Every rounding operation is the FP64 reference's, in its order (an exact
// zero is not added), so the state keeps the reference's bits.
#pragma once
#include "fwd_kernels.cuh"
#include "ops64.cuh"

namespace swadj {
namespace s64 {

constexpr int kThreads = 128;
using namespace d64;

// A cell in the frame of a sweep (mn the momentum normal to the edges).
struct Cell {
    double h, mn, mt, eta, un, ut, sq, b;
    double fn, ft, wn, wt;   // mn un, mn ut and sq un, sq ut, one product for both edges
};

// A solved edge: wave speeds, the vectors of waves 1 and 3, the strength of
// the shear wave (0, 0, b2), the fluctuations to the left and right cell.
// A shore edge (wet/dry) has no waves for its neighbours' limiters.
struct Edge {
    double s1, s2, s3, z1[3], z3[3], b2, am[3], ap[3];
    bool shore;
};

// Velocities and sqrt(h) of a cell.  moving = false: its momenta are zero in
// every lane of the warp, and sqrt(h) is left to an edge that needs it.  A 1D
// grid (TWO_D false) has no tangential momentum.
template <bool WD, bool TWO_D = true>
__device__ __forceinline__ Cell derive(double tol, double h, double mn, double mt, double eta,
                                       double b, bool moving) {
    Cell c;
    c.h = h; c.mn = mn; c.mt = mt; c.eta = eta; c.b = b;
    c.un = 0.0; c.ut = 0.0; c.sq = 0.0;
    c.fn = 0.0; c.ft = 0.0; c.wn = 0.0; c.wt = 0.0;
    if (moving && (!WD || h > tol)) {
        const Recip r = recip(h);
        c.un = div(mn, r);
        c.sq = root(h);
        c.fn = mn * c.un;
        c.wn = c.sq * c.un;
        if (TWO_D) {
            c.ut = div(mt, r);
            c.ft = mn * c.ut;
            c.wt = c.sq * c.ut;
        }
    }
    return c;
}

// The part of wave vector component z, of a wave of speed s, that goes left
// (right): all, nothing, or half at speed 0.
__device__ __forceinline__ double to_left(double s, double z) {
    return is_zero(s) ? half_of(z) : (__double2hiint(s) < 0 ? z : 0.0);
}
__device__ __forceinline__ double to_right(double s, double z) {
    return is_zero(s) ? half_of(z) : (__double2hiint(s) < 0 ? 0.0 : z);
}

// shore_edge: a dry cell, or u - c or u + c rising through zero.  A flow
// clearly slower than its waves on both sides is neither.
__device__ __forceinline__ bool is_shore(double g, double tol, const Cell &L, const Cell &R) {
    if (!(L.h > tol) || !(R.h > tol)) return true;
    const float c = 0.999f * sqrtf((float)g);
    if (fabsf((float)L.un) < c * (float)L.sq && fabsf((float)R.un) < c * (float)R.sq) return false;
    const double cL = root(g * L.h), cR = root(g * R.h);
    return (negative(L.un - cL) && positive(R.un - cR)) ||
           (negative(L.un + cL) && positive(R.un + cR));
}

// shore_fluct with this file's operations (a dry cell's velocities are zero).
__device__ __forceinline__ void shore(double g, const Cell &L, const Cell &R, double am[3],
                                      double ap[3]) {
    const double Bm = L.b > R.b ? L.b : R.b;
    double hLs = L.eta - Bm, hRs = R.eta - Bm;
    if (negative(hLs)) hLs = 0.0;
    if (negative(hRs)) hRs = 0.0;
    const double hg = half_of(g);
    const double pL = hg * (L.h * L.h), pR = hg * (R.h * R.h);
    const double pLs = hg * (hLs * hLs), pRs = hg * (hRs * hRs);
    double F[3] = {0.0, 0.0, 0.0};
    if (positive(hLs) || positive(hRs)) {
        const double cL = root(g * hLs), cR = root(g * hRs);
        const double lL = L.un - cL, lR = R.un - cR, rL = L.un + cL, rR = R.un + cR;
        const double sL = lL < lR ? lL : lR, sR = rL > rR ? rL : rR;
        const double QL[3] = {hLs, hLs * L.un, hLs * L.ut}, QR[3] = {hRs, hRs * R.un, hRs * R.ut};
        const double FL[3] = {QL[1], QL[1] * L.un + pLs, QL[1] * L.ut};
        const double FR[3] = {QR[1], QR[1] * R.un + pRs, QR[1] * R.ut};
        const Recip w = recip(sR - sL);
#pragma unroll
        for (int m = 0; m < 3; m++) {
            if (!negative(sL)) F[m] = FL[m];
            else if (!positive(sR)) F[m] = FR[m];
            else F[m] = div(sR * FL[m] - sL * FR[m] + sL * sR * (QR[m] - QL[m]), w);
        }
    }
    const double fL[3] = {L.mn, L.fn + pL, L.ft};
    const double fR[3] = {R.mn, R.fn + pR, R.ft};
    am[0] = F[0] - fL[0]; am[1] = (F[1] + (pL - pLs)) - fL[1]; am[2] = F[2] - fL[2];
    ap[0] = fR[0] - F[0]; ap[1] = fR[1] - (F[1] + (pR - pRs)); ap[2] = fR[2] - F[2];
}

// Whether the edge between L and R carries nothing: no momentum on either
// side, and one surface (or, wet/dry, bare land on both sides).
template <bool WD>
__device__ __forceinline__ bool is_still(double tol, const Cell &L, const Cell &R) {
    if (!is_zero(L.mn) || !is_zero(L.mt) || !is_zero(R.mn) || !is_zero(R.mt)) return false;
    const bool level = __double_as_longlong(L.eta) == __double_as_longlong(R.eta) ||
                       (is_zero(L.eta) && is_zero(R.eta));
    if (!WD) return level;
    return (level && L.h > tol && R.h > tol) || (is_zero(L.h) && is_zero(R.h));
}

// Waves and fluctuations of the edge between L and R (the expressions of
// fwave_roe, wave_vec and edge_flux).
template <bool WD>
__device__ __forceinline__ Edge solve(double g, double tol, const Cell &L, const Cell &R) {
    Edge e;
    e.shore = WD && is_shore(g, tol, L, R);
    if (WD && e.shore) {
        e.s1 = -1.0; e.s2 = 0.0; e.s3 = 1.0; e.b2 = 0.0;
#pragma unroll
        for (int m = 0; m < 3; m++) { e.z1[m] = 0.0; e.z3[m] = 0.0; }
        shore(g, L, R, e.am, e.ap);
        return e;
    }
    const double gh = g * half_of(L.h + R.h);
    const Recip den = recip(L.sq + R.sq);
    const double uh = div(L.wn + R.wn, den);
    const double vh = div(L.wt + R.wt, den);
    const double ch = root(gh);
    e.s1 = uh - ch; e.s2 = uh; e.s3 = uh + ch;
    const double df1 = R.mn - L.mn;
    const double df2 = (R.fn - L.fn) + gh * (R.eta - L.eta);
    const double df3 = R.ft - L.ft;
    const Recip w = recip(e.s3 - e.s1);
    const double b1 = div(e.s3 * df1 - df2, w), b3 = div(df2 - e.s1 * df1, w);
    e.b2 = df3 - vh * df1;
    e.z1[0] = b1; e.z1[1] = b1 * e.s1; e.z1[2] = b1 * vh;
    e.z3[0] = b3; e.z3[1] = b3 * e.s3; e.z3[2] = b3 * vh;
    const double l2 = to_left(uh, e.b2), r2 = to_right(uh, e.b2);
    if (negative(e.s1) && positive(e.s3)) {   // subsonic
        e.am[0] = e.z1[0]; e.am[1] = e.z1[1]; e.am[2] = e.z1[2] + l2;
        e.ap[0] = e.z3[0]; e.ap[1] = e.z3[1]; e.ap[2] = r2 + e.z3[2];
    } else {
#pragma unroll
        for (int m = 0; m < 3; m++) {
            double a = to_left(e.s1, e.z1[m]), p = to_right(e.s1, e.z1[m]);
            if (m == 2) { a += l2; p += r2; }
            e.am[m] = a + to_left(e.s3, e.z3[m]);
            e.ap[m] = p + to_right(e.s3, e.z3[m]);
        }
    }
    return e;
}

// phi(theta) of the MC limiter, theta = dot / zz (0 where zz = 0).
__device__ __forceinline__ double limiter(double dot, double zz) {
    if (is_zero(zz) || !positive(dot)) return 0.0;   // zz >= 0
    const double th = div(dot, recip(zz));
    return min_pos(twice(th), min_pos(half_of(1.0 + th), 2.0));
}

// (sign(s) / 2) (1 - nu |s|) phi, the factor of a wave in the correction.
__device__ __forceinline__ double factor(double s, double nu, double phi) {
    if (is_zero(s)) return 0.0;
    return flip_if(__double2hiint(s) < 0, half_of(1.0 - nu * fabs(s))) * phi;
}

// MC-limited correction F of edge w from its left (l) and right (r)
// neighbour edges (each wave's upwind one).
__device__ __forceinline__ void correct(const Edge &l, const Edge &w, const Edge &r, double nu,
                                        double F[3]) {
    const bool p1 = positive(w.s1), p3 = positive(w.s3);
    double u[3];
#pragma unroll
    for (int m = 0; m < 3; m++) u[m] = p1 ? l.z1[m] : r.z1[m];
    const double f1 = factor(
        w.s1, nu,
        limiter(u[0] * w.z1[0] + u[1] * w.z1[1] + u[2] * w.z1[2],
                w.z1[0] * w.z1[0] + w.z1[1] * w.z1[1] + w.z1[2] * w.z1[2]));
    const double f2 =
        factor(w.s2, nu, limiter((positive(w.s2) ? l.b2 : r.b2) * w.b2, w.b2 * w.b2));
#pragma unroll
    for (int m = 0; m < 3; m++) u[m] = p3 ? l.z3[m] : r.z3[m];
    const double f3 = factor(
        w.s3, nu,
        limiter(u[0] * w.z3[0] + u[1] * w.z3[1] + u[2] * w.z3[2],
                w.z3[0] * w.z3[0] + w.z3[1] * w.z3[1] + w.z3[2] * w.z3[2]));
    F[0] = f1 * w.z1[0] + f3 * w.z3[0];
    F[1] = f1 * w.z1[1] + f3 * w.z3[1];
    F[2] = (f1 * w.z1[2] + f2 * w.b2) + f3 * w.z3[2];
}

// One pass: YPASS false sweeps rows (lines along x), true columns and ends
// the step (CFL maximum and clock).  Resident warps take units from a
// counter: unit u is segment u / groups (seg cells) of the 32 lines of group u
// % groups; the x-pass's units end with the gauges of a recorded step.
// Where a whole warp's edge is still (the ocean at rest, bare land) it is
// not solved and a cell between two such edges keeps its state, which is
// what the arithmetic gives exactly.
template <bool YPASS, bool WD, int ORD>
__global__ void __launch_bounds__(kThreads, 2)
    fwd_f64_sweep(FwdParams<double> p, int seg, int nunits) {
    volatile DevClock *clk = p.clk;
    const double t = clk->t;
    double dt = clk->dt_cfl;
    if (p.t_end - t < dt) dt = p.t_end - t;
    if (!(dt > 0.0)) return;   // clock already at t_end: no-op step
    const int cur = clk->cur, src = YPASS ? cur ^ 1 : cur;
    const int nx = p.nx, lane = threadIdx.x & 31;
    const double g = p.g, tol = p.dry_tol;
    const double *q0 = p.q[src][0], *qn = p.q[src][YPASS ? 2 : 1], *qt = p.q[src][YPASS ? 1 : 2];
    double *o0 = p.q[src ^ 1][0], *on = p.q[src ^ 1][YPASS ? 2 : 1],
           *ot = p.q[src ^ 1][YPASS ? 1 : 2];
    const int lines = YPASS ? nx : p.ny, n = YPASS ? p.ny : nx;
    const int groups = (lines + 31) / 32;
    const int bc_lo = YPASS ? p.bc.lo_y : p.bc.lo_x, bc_hi = YPASS ? p.bc.hi_y : p.bc.hi_x;
    const double nu = dt / (YPASS ? p.dy : p.dx);
    const int ngroups = !YPASS && p.gauges.n > 0 ? (p.gauges.n + 31) / 32 : 0;
    unsigned int *work = YPASS ? &p.clk->work2 : &p.clk->work;
    double mx = 0.0, my = 0.0;   // max |u| + c, |v| + c
    bool bad = false;
    for (;;) {   // warp-uniform
        int unit = 0;
        if (lane == 0) unit = (int)atomicAdd(work, 1u);
        unit = __shfl_sync(0xffffffffu, unit, 0);
        if (unit >= nunits) {
            if (unit >= nunits + ngroups) break;
            record_gauge_group<double>(p.gauges, q0, p.bath, nx, p.ny, 1, p.clk, unit - nunits);
            continue;
        }
        const int s0 = unit / groups * seg, s1 = (s0 + seg < n ? s0 + seg : n) - 1;
        int line = unit % groups * 32 + lane;
        const bool valid = line < lines;
        if (!valid) line = lines - 1;
        auto at = [&](int i) { return YPASS ? (size_t)i * nx + line : (size_t)line * nx + i; };
        double rh, rn, rt, rb;   // the next cell
        auto load = [&](int i) {
            bool flip;
            const size_t o = at(ghost_index(i, n, bc_lo, bc_hi, &flip));
            rh = q0[o]; rn = qn[o]; rt = qt[o]; rb = p.bath[o];
            rn = flip ? -rn : rn;
        };
        Cell A = {}, C = {};     // cells i-2 (state only), i-1
        Edge W1 = {}, W2 = {};   // edges (i-3|i-2), (i-2|i-1)
        double ap1[3] = {}, F1[3] = {};   // of the edge below cell i-2
        bool bare = false;                // C's sqrt(h) is not formed yet
        bool still1 = false, still2 = false;   // W1, W2 carry nothing in any lane
        load(s0 - 2);
#pragma unroll 1
        for (int i = s0 - 2; i <= s1 + 2; i++) {
            const bool moving =
                !__all_sync(0xffffffffu, is_zero(rn) && is_zero(rt));
            Cell D = derive<WD>(tol, rh, rn, rt, rh + rb, rb, moving);
            if (i <= s1 + 1) load(i + 1);
            Edge Wn = {};
            bool still = false, bared = !moving;
            if (i >= s0 - 1) {   // edge (i-1|i)
                still = __all_sync(0xffffffffu, is_still<WD>(tol, C, D));
                if (!still) {
                    if (bare && (!WD || C.h > tol)) C.sq = root(C.h);
                    if (bared && (!WD || D.h > tol)) D.sq = root(D.h);
                    bared = false;
                    Wn = solve<WD>(g, tol, C, D);
                }
            }
            double F[3] = {0.0, 0.0, 0.0};
            if (ORD >= 2 && i >= s0 + 1 && !still2 && (!WD || !W2.shore))
                correct(W1, W2, Wn, nu, F);
            if (i >= s0 + 2) {   // cell i-2 takes the edges (i-3|i-2), (i-2|i-1)
                double q[3] = {A.h, A.mn, A.mt};
                const bool kept = still1 && still2;
                if (!kept) {
#pragma unroll
                    for (int m = 0; m < 3; m++) {
                        double d = -nu * (ap1[m] + W2.am[m]);
                        if (ORD >= 2) d = d - nu * (F[m] - F1[m]);
                        q[m] = q[m] + d;
                    }
                }
                const bool dry = WD && !(q[0] > tol);
                if (dry) {   // a dry cell keeps no momentum, no negative depth
                    if (q[0] < 0.0) q[0] = 0.0;
                    q[1] = 0.0;
                    q[2] = 0.0;
                }
                if (valid) {
                    const size_t o = at(i - 2);
                    o0[o] = q[0];
                    on[o] = q[1];
                    ot[o] = q[2];
                    if (YPASS) {
                        bad |= !(WD ? q[0] >= 0.0 : q[0] > 0.0) || !isfinite(q[1]) ||
                               !isfinite(q[2]);
                        if (!dry) {
                            const double c = root(g * q[0]);
                            double ax = c, ay = c;
                            if (!kept) {
                                const Recip r = recip(q[0]);
                                ax = fabs(div(q[2], r)) + c;
                                ay = fabs(div(q[1], r)) + c;
                            }
                            if (!is_nan(ax)) {
                                mx = max_pos(mx, ax);
                                if (!is_nan(ay)) my = max_pos(my, ay);
                            }
                        }
                    }
                }
            }
            A = C; C = D;
            bare = bared;
            W1 = W2; W2 = Wn;
            still1 = still2; still2 = still;
#pragma unroll
            for (int m = 0; m < 3; m++) { ap1[m] = W1.ap[m]; F1[m] = F[m]; }
        }
    }
    if (!YPASS) return;
    if (bad) atomicOr(p.err, ERR_UNSTABLE);
    // block max -> partial, the last block reduces and advances the clock
    __shared__ double red[32];
    __shared__ int am_last;
    const double sx = mx / p.dx, sy = my / p.dy;
    const double bm = block_max<kThreads>(sx > sy ? sx : sy, red);
    const int tid = threadIdx.x;
    if (tid == 0) {
        p.partial[blockIdx.x] = bm;
        __threadfence();
        am_last = atomicAdd((unsigned int *)&p.clk->ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (am_last) {
        __threadfence();
        double m = 0.0;
        for (int k = tid; k < (int)gridDim.x; k += kThreads) {
            const double v = __ldcg(p.partial + k);
            m = v > m ? v : m;
        }
        m = block_max<kThreads>(m, red);
        if (tid == 0) {
            clk->t = t + dt;
            clk->smax = m;
            clk->dt_cfl = p.cfl / m;
            clk->nsteps = clk->nsteps + 1;
            clk->ticket = 0u;
            clk->work = 0u;
            clk->work2 = 0u;
            if (p.gauges.n > 0) *p.gauges.row += 1;
        }
    }
}

// ------------------------------------------------------------- 1D grids
// One step of a 1D grid: a warp per 28 output cells (32 with two halo cells
// each side), a cell and the edge to its right per lane, neighbours by
// shuffles.  A 1D grid has few cells, so what counts is how long one warp
// takes: about 115 FP64 operations a lane (the tiled kernel: about 360, each
// edge limited twice), with warps spread over as many schedulers as there
// are.
// Measured, us per step, tiles / strips: 100 cells 28.8 / 10.2, 2000 31.1 / 12.0
// (1.8 more when not chained), 8000 31.3 / 11.7; 2000 with wet/dry 50 / 18.6.
__device__ __forceinline__ double dn(double x) { return __shfl_down_sync(0xffffffffu, x, 1); }
__device__ __forceinline__ double up(double x) { return __shfl_up_sync(0xffffffffu, x, 1); }

constexpr int kLineOut = 28;
template <bool WD, int ORD>
__global__ void __launch_bounds__(32) fwd_f64_line(FwdParams<double> p) {
    chain_begin();
    volatile DevClock *clk = p.clk;
    const double t = clk->t;
    double dt = clk->dt_cfl;
    if (p.t_end - t < dt) dt = p.t_end - t;
    if (!(dt > 0.0)) return;   // clock already at t_end: no-op step
    const int cur = clk->cur, lane = threadIdx.x;
    const double *q0 = p.q[cur][0], *q1 = p.q[cur][1];
    const double g = p.g, tol = p.dry_tol, nu = dt / p.dx;
    double mx = 0.0;   // max |u| + c
    bool bad = false;
    const int units = (p.nx + kLineOut - 1) / kLineOut;
    const int ngroups = p.gauges.n > 0 ? (p.gauges.n + 31) / 32 : 0;
    for (int unit = blockIdx.x; unit < units + ngroups; unit += gridDim.x) {
        if (unit >= units) {
            record_gauge_group<double>(p.gauges, q0, p.bath, p.nx, p.ny, 0, p.clk, unit - units);
            continue;
        }
        const int i = unit * kLineOut - 2 + lane;
        bool flip;
        const int o = ghost_index(i, p.nx, p.bc.lo_x, p.bc.hi_x, &flip);
        const double h = q0[o], b = p.bath[o];
        const double m = flip ? -q1[o] : q1[o];
        const Cell c = derive<WD, false>(tol, h, m, 0.0, h + b, b, true);
        Cell r;
        r.h = dn(c.h); r.mn = dn(c.mn); r.mt = 0.0; r.eta = dn(c.eta); r.un = dn(c.un);
        r.ut = 0.0; r.sq = dn(c.sq); r.b = dn(c.b);
        r.fn = dn(c.fn); r.wn = dn(c.wn); r.ft = 0.0; r.wt = 0.0;
        const bool still = __all_sync(0xffffffffu, is_still<WD>(tol, c, r));
        Edge w = {};
        if (!still) w = solve<WD>(g, tol, c, r);   // edge (i|i+1)
        double F[3] = {0.0, 0.0, 0.0};
        if (ORD >= 2) {
            Edge wl = {}, wr = {};
#pragma unroll
            for (int k = 0; k < 2; k++) {
                wl.z1[k] = up(w.z1[k]); wl.z3[k] = up(w.z3[k]);
                wr.z1[k] = dn(w.z1[k]); wr.z3[k] = dn(w.z3[k]);
            }
            if (!still && (!WD || !w.shore)) correct(wl, w, wr, nu, F);
        }
        double q[2] = {c.h, c.mn};
#pragma unroll
        for (int k = 0; k < 2; k++) {
            const double apl = up(w.ap[k]), Fl = up(F[k]);
            if (!still) {
                double d = -nu * (apl + w.am[k]);
                if (ORD >= 2) d = d - nu * (F[k] - Fl);
                q[k] = q[k] + d;
            }
        }
        const bool dry = WD && !(q[0] > tol);
        if (dry) {   // a dry cell keeps no momentum, no negative depth
            if (q[0] < 0.0) q[0] = 0.0;
            q[1] = 0.0;
        }
        if (lane >= 2 && lane < 30 && i < p.nx) {
            p.q[cur ^ 1][0][i] = q[0];
            p.q[cur ^ 1][1][i] = q[1];
            bad |= !(WD ? q[0] >= 0.0 : q[0] > 0.0) || !isfinite(q[1]);
            if (!dry) {
                const double ax = fabs(div(q[1], recip(q[0]))) + root(g * q[0]);
                if (!is_nan(ax)) mx = max_pos(mx, ax);
            }
        }
    }
    if (bad) atomicOr(p.err, ERR_UNSTABLE);
    mx = mx / p.dx;
    for (int s = 16; s > 0; s >>= 1) {
        const double v = __shfl_xor_sync(0xffffffffu, mx, s);
        mx = v > mx ? v : mx;
    }
    int last = 0;
    if (lane == 0) {
        p.partial[blockIdx.x] = mx;
        __threadfence();
        last = atomicAdd((unsigned int *)&p.clk->ticket, 1u) == gridDim.x - 1;
    }
    if (!__shfl_sync(0xffffffffu, last, 0)) return;
    __threadfence();
    mx = 0.0;
    for (int k = lane; k < (int)gridDim.x; k += 32) {
        const double v = __ldcg(p.partial + k);
        mx = v > mx ? v : mx;
    }
    for (int s = 16; s > 0; s >>= 1) {
        const double v = __shfl_xor_sync(0xffffffffu, mx, s);
        mx = v > mx ? v : mx;
    }
    if (lane == 0) {
        clk->t = t + dt;
        clk->smax = mx;
        clk->dt_cfl = p.cfl / mx;
        clk->cur = cur ^ 1;
        clk->nsteps = clk->nsteps + 1;
        clk->ticket = 0u;
        clk->work = 0u;
        clk->work2 = 0u;
        if (p.gauges.n > 0) *p.gauges.row += 1;
    }
}

}  // namespace s64
}  // namespace swadj
