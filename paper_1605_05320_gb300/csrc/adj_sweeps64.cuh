// adj_sweeps64.cuh -- FP64 2D adjoint step as two sweep passes (Sec. 4, the
// time-reversed linear adjoint of adj_kernels.cuh, dimensionally split y then
// x), laid out like the FP64 forward step (fwd_sweeps64.cuh): the FP64 units
// bound it, each lane walks a segment of one line of cells, and every edge is
// solved and limited once but for the ends of segments (a 32 x 4 tile solved
// them 1.8 times and limited every edge twice).  The y-pass reads the state
// and writes the y-swept one to the other buffer, the x-pass writes the new
// state (and its snapshot) back.  An edge with zero data on both sides in
// every lane has no waves and is not solved: far from the target the adjoint
// is still exactly zero.
// Measured, us per step early and late in the solve, tiles / sweeps: 512^2 212
// and 223 / 57 and 82, 2048^2 3110 and 3120 / 261 and 335.
//
// Every rounding operation is the FP64 reference's, in its order (an exact
// zero is not added), so the state keeps the reference's bits.
#pragma once
#include "adj_kernels.cuh"
#include "ops64.cuh"

namespace swadj {
namespace a64 {

using namespace d64;

constexpr int kThreads = 32;   // one warp a block: blocks balance over the schedulers

// A cell: eta~, the normal component, c = sqrt(g hbar) (0 where dry), g hbar.
struct Cell {
    double e, m, c, gh;
};

// A solved edge: its two wave vectors (speeds -cl and cr); wall: a wet/dry
// edge, no second-order correction.
struct Edge {
    double z1[2], z2[2], cl, cr;
    bool wall;
};

// adj_riemann
__device__ __forceinline__ Edge solve(Cell L, Cell R) {
    Edge w = {};
    const bool dL = !positive(L.c), dR = !positive(R.c);
    w.wall = dL || dR;
    if (dL && dR) return w;
    if (dL) { L = R; L.m = -R.m; }
    if (dR) { R = L; R.m = -L.m; }
    const double d1 = L.gh * L.m - R.gh * R.m, d2 = L.e - R.e;
    const Recip s = recip(L.c + R.c);
    const double b1 = div(d1 + R.c * d2, s), b2 = div(L.c * d2 - d1, s);
    w.cl = L.c;
    w.cr = R.c;
    w.z1[0] = b1 * L.c; w.z1[1] = b1;
    w.z2[0] = -b2 * R.c; w.z2[1] = b2;
    return w;
}

// (1 - nu c) / 2 phi(theta), the factor of wave vector z with upwind vector u
__device__ __forceinline__ double factor(const double z[2], const double u[2], double c,
                                         double nu) {
    const double zz = z[0] * z[0] + z[1] * z[1], dot = u[0] * z[0] + u[1] * z[1];
    if (is_zero(zz) || !positive(dot)) return 0.0;
    const double th = div(dot, recip(zz));
    return half_of(1.0 - nu * c) * min_pos(twice(th), min_pos(half_of(1.0 + th), 2.0));
}

// One pass: XPASS false sweeps columns (eta~, gamma~), true rows (eta~, mu~)
// and writes the snapshot.  Warp u takes segment u / groups (seg cells) of
// the 32 lines of group u % groups.
template <bool XPASS, int ORD>
__global__ void __launch_bounds__(kThreads) adj_f64_sweep(AdjParams<double> p, int seg) {
    const int nx = p.nx, lane = threadIdx.x & 31, unit = blockIdx.x;
    // y-pass: src -> dst; x-pass: dst -> src
    const double *const *q = XPASS ? const_cast<const double *const *>(p.dst) : p.src;
    const double *qe = q[0], *qm = q[XPASS ? 1 : 2], *qt = q[XPASS ? 2 : 1];
    double *oe, *om, *ot;
    if (XPASS) {
        oe = const_cast<double *>(p.src[0]); om = const_cast<double *>(p.src[1]);
        ot = const_cast<double *>(p.src[2]);
    } else {
        oe = p.dst[0]; om = p.dst[2]; ot = p.dst[1];
    }
    const int lines = XPASS ? p.ny : nx, n = XPASS ? nx : p.ny, groups = (lines + 31) / 32;
    const int s0 = unit / groups * seg, s1 = (s0 + seg < n ? s0 + seg : n) - 1;
    int line = unit % groups * 32 + lane;
    const bool valid = line < lines;
    if (!valid) line = lines - 1;
    const int bc_lo = XPASS ? p.bc.lo_x : p.bc.lo_y, bc_hi = XPASS ? p.bc.hi_x : p.bc.hi_y;
    const double nu = XPASS ? p.nux : p.nuy;
    auto at = [&](int i) { return XPASS ? (size_t)line * nx + i : (size_t)i * nx + line; };
    double re, rm, rt, rh;   // the next cell (rh its hbar)
    auto load = [&](int i) {
        bool flip;
        const size_t o = at(ghost_index(i, n, bc_lo, bc_hi, &flip));
        re = qe[o]; rm = qm[o]; rt = qt[o]; rh = p.c[o];
        rm = flip ? -rm : rm;
    };
    auto speed = [&](Cell &x) {   // from hbar, kept in x.gh until needed
        const double hb = x.gh;
        x.gh = hb > p.dry_tol ? p.g * hb : 0.0;
        x.c = hb > p.dry_tol ? root(x.gh) : 0.0;
    };
    Cell A = {}, C = {};             // cells i-2, i-1
    double tA = 0.0, tC = 0.0;       // their passive component
    Edge W1 = {}, W2 = {};           // edges (i-3|i-2), (i-2|i-1)
    double F1[2] = {0.0, 0.0};       // of the edge below cell i-2
    bool bare = true, still1 = false, still2 = false;   // C's speed not formed; W1, W2 carry nothing
    load(s0 - 2);
#pragma unroll 1
    for (int i = s0 - 2; i <= s1 + 2; i++) {
        Cell D;
        D.e = re; D.m = rm; D.gh = rh; D.c = 0.0;
        const double tD = rt;
        if (i <= s1 + 1) load(i + 1);
        Edge Wn = {};
        bool still = false, bared = true;
        if (i >= s0 - 1) {   // edge (i-1|i)
            still = __all_sync(0xffffffffu, is_zero(C.e) && is_zero(C.m) && is_zero(D.e) &&
                                                is_zero(D.m));
            if (!still) {
                if (bare) speed(C);
                speed(D);
                bare = bared = false;
                Wn = solve(C, D);
            }
        }
        double F[2] = {0.0, 0.0};
        if (ORD >= 2 && i >= s0 + 1 && !still2 && !W2.wall) {   // edge (i-2|i-1)
            const double k1 = -factor(W2.z1, Wn.z1, W2.cl, nu), k2 = factor(W2.z2, W1.z2, W2.cr, nu);
            F[0] = k1 * W2.z1[0] + k2 * W2.z2[0];
            F[1] = k1 * W2.z1[1] + k2 * W2.z2[1];
        }
        if (i >= s0 + 2) {   // cell i-2 takes the edges (i-3|i-2), (i-2|i-1)
            double e = A.e, m = A.m;
            if (!(still1 && still2) && positive(A.c)) {
                double d0 = -nu * (W1.z2[0] + W2.z1[0]), d1 = -nu * (W1.z2[1] + W2.z1[1]);
                if (ORD >= 2) {
                    d0 = d0 - nu * (F[0] - F1[0]);
                    d1 = d1 - nu * (F[1] - F1[1]);
                }
                e = e + d0;
                m = m + d1;
            }
            if (valid) {
                const size_t o = at(i - 2);
                oe[o] = e;
                om[o] = m;
                ot[o] = tA;
                if (XPASS && p.snap_f) {
                    p.snap_f[o] = (float)e;
                    p.snap_f[p.snap_comp_stride + o] = (float)m;
                    p.snap_f[2 * p.snap_comp_stride + o] = (float)tA;
                } else if (XPASS && p.snap_d) {
                    p.snap_d[o] = e;
                    p.snap_d[p.snap_comp_stride + o] = m;
                    p.snap_d[2 * p.snap_comp_stride + o] = tA;
                }
            }
        }
        A = C; C = D;
        tA = tC; tC = tD;
        W1 = W2; W2 = Wn;
        bare = bared;
        still1 = still2; still2 = still;
        F1[0] = F[0]; F1[1] = F[1];
    }
    if (XPASS && (p.snap_f || p.snap_d) && unit == 0 && lane == 0) *p.tau_dev = p.tau_val;
}

}  // namespace a64
}  // namespace swadj
