// ctu_strips.cuh -- the FP32 unsplit 2D step with transverse waves
// (ctu_kernels.cuh states the method) as warp strips.
//
// A warp owns 32 columns (28 of them its output) and walks its rows
// downwards, as in the split step (strips.cuh): x-edges are solved and
// limited across the warp with shuffles, y-edges in registers over a window
// of rows, every edge once; its two fluctuations are split transversely once,
// as the halves of packed operations, and each half goes to the cell it
// enters.  Row j brings the x-edges of row j and the y-edge (j-1|j); with the
// latter the transverse corrections of row j - 1's x-edges are known, and the
// y-edge (j-2|j-1) with its limiter completes row j - 2.  The tiled kernel
// this replaces staged waves and per-cell terms through shared memory in four
// phases between barriers.
// What bounds it is the number of instructions issued.  Measured, us per step
// near the start of a run and with waves everywhere, tiles / strips: 64^2
// 15.2 / 11.4 both, 512^2 33.9 / 14.9 and 34.9 / 18.7, 2048^2 338 / 44.8 and
// 358 / 105.
#pragma once
#include "strips.cuh"

namespace swadj {
namespace strip {

// Transverse parts of an edge's two fluctuations (x half: A-dQ, y half:
// A+dQ), split by the tangential flux Jacobian at the edge's Roe state:
// speeds vh - ch, vh, vh + ch, vectors (1, uh, vh - ch), (0, 1, 0), (1, uh,
// vh + ch) in the edge's frame.  n: the part moving in the negative
// tangential direction, p: in the positive one.  SUB: |vh| < ch.
struct Trans {
    fp::f2 n[3], p[3];
};
template <bool SUB>
__device__ __forceinline__ Trans transverse(const fp::Edge &w, const fp::Fluct &a) {
    using namespace fp;
    const float m0 = sub(w.vh, w.ch), m2 = add(w.vh, w.ch);
    const float k0 = mul(m0, w.hr), k2 = mul(m2, w.hr), q = mul(k0, m2);
    // wave strengths times speeds
    const f2 c0 = fma(a.a2, dup(-k0), mul(a.a0, dup(q)));
    const f2 c2 = fma(a.a0, dup(-q), mul(a.a2, dup(k2)));
    const f2 c1 = mul(dup(w.vh), fma(a.a0, dup(-w.uh), a.a1));
    const bool neg = w.vh < 0.f;
    const f2 z = dup(0.f), sn = neg ? c1 : z, sp = neg ? z : c1;
    Trans t;
    if (SUB) {
        t.n[0] = c0;
        t.n[1] = fma(c0, dup(w.uh), sn);
        t.n[2] = mul(c0, dup(m0));
        t.p[0] = c2;
        t.p[1] = fma(c2, dup(w.uh), sp);
        t.p[2] = mul(c2, dup(m2));
    } else {
        const f2 c0n = m0 < 0.f ? c0 : z, c0p = m0 < 0.f ? z : c0;
        const f2 c2n = m2 < 0.f ? c2 : z, c2p = m2 < 0.f ? z : c2;
        t.n[0] = add(c0n, c2n);
        t.n[1] = fma(t.n[0], dup(w.uh), sn);
        t.n[2] = fma(c0n, dup(m0), mul(c2n, dup(m2)));
        t.p[0] = add(c0p, c2p);
        t.p[1] = fma(t.p[0], dup(w.uh), sp);
        t.p[2] = fma(c0p, dup(m0), mul(c2p, dup(m2)));
    }
    return t;
}

// Subsonic in both directions, so that both SUB forms hold.
__device__ __forceinline__ bool slow(const fp::Edge &w) {
    return fp::subsonic(w.s1, w.s3) && fabsf(w.vh) < w.ch;
}

// One strip, as strip_unit.  Components 0, 1, 2 are eta, hu, hv throughout;
// an x-edge's frame is (h, hu, hv), a y-edge's (h, hv, hu).
template <int ORD>
__device__ __forceinline__ void ctu_unit(const View &v, int x0, int y0, int rows, float nux,
                                         float nuy, float g, Ring &R, float &smax, bool &bad) {
    using namespace fp;
    const int lane = threadIdx.x & 31;
    const int ylast = (y0 + rows < v.ny ? y0 + rows : v.ny) - 1;
    const int gi = x0 - 2 + lane;
    bool fx;
    const int col = ghost_index(gi, v.nx, v.bc.lo_x, v.bc.hi_x, &fx);
    const bool out = lane >= 2 && lane < kLanes - 2 && gi < v.nx;
    const float gh = 0.5f * g, kt = mul(0.5f, mul(nux, nuy));
    const bool yin = y0 - 2 >= 0 && ylast + 2 < v.ny;
    const int jend = ylast + 2;
    int jn = y0 - 2, sn = 0, sc = 0;   // next row to fetch, its ring slot, the slot to read
    auto fetch = [&]() {
        if (jn <= jend) {
            bool fy;
            const int row = yin ? jn : ghost_index(jn, v.ny, v.bc.lo_y, v.bc.hi_y, &fy);
            fetch_row(R, sn, v, col, row, lane);
        }
        cp_commit();
        jn++;
        sn = (sn + 1) & (kRing - 1);
    };
    auto turned = [](const Cell &c) {   // the cell in a y-edge's frame
        Cell t = c;
        t.mn = c.mt; t.mt = c.mn; t.su = c.sv; t.sv = c.su;
        t.P = mul(c.sv, c.sv);
        return t;
    };
#pragma unroll
    for (int k = 0; k < kRing - 1; k++) fetch();
    // rows before the strip's window stand in as water at rest: their values
    // are finite and reach no output row
    Cell B = {};                       // row j-1
    B.h = 1.f; B.sq = 1.f;
    Edge W1 = solve<true>(gh, B, B), W2 = W1;   // y-edges (j-3|j-2), (j-2|j-1)
    float xb[3] = {}, py[3] = {}, my[3] = {};   // row j-1: its x-edges' net and transverse sums
    float py1[3] = {};                 // row j-2's upward sums
    float px2[3] = {}, mx2[3] = {};    // transverse parts of the y-edge (j-2|j-1)'s upward half
    float q1[3] = {}, h1 = 1.f;        // row j-2 with its x-edges applied
    float nr[3] = {}, t1[3] = {};      // of the y-edge (j-3|j-2): R of its net, its transverse sum
#pragma unroll 1
    for (int j = y0 - 2; j <= jend; j++) {
        fetch();
        cp_wait<kRing - 1>();   // row j has landed
        bool fy = false;
        if (!yin) ghost_index(j, v.ny, v.bc.lo_y, v.bc.hi_y, &fy);
        const float eta = R.v[sc][0][lane], mu = R.v[sc][1][lane], mv = R.v[sc][2][lane];
        const float hb = R.v[sc][3][lane];
        sc = (sc + 1) & (kRing - 1);
        const Cell c = derive(eta, add(eta, hb), fx ? -mu : mu, fy ? -mv : mv);
        const Edge w = xsolve<true>(c, gh);
        const Edge Wn = j > y0 - 2 ? solve<true>(gh, turned(B), turned(c)) : W2;   // y-edge (j-1|j)
        float nb[3], np[3], nm[3], nx[3];   // row j: net, sums; row j-1: transverse x-correction
        Net N;
        auto row = [&](auto form) {
            constexpr bool SUB = decltype(form)::value;
            const Fluct f = fluct<SUB>(w);
            const Net n = xnet<SUB, ORD>(w, nux, f);
            nb[0] = mul(-nux, add(up(n.R0), n.L0));
            nb[1] = mul(-nux, add(up(n.R1), n.L1));
            nb[2] = mul(-nux, add(up(n.R2), n.L2));
            const Trans t = transverse<SUB>(w, f);
#pragma unroll
            for (int m = 0; m < 3; m++) {
                np[m] = add(t.p[m].x, up(t.p[m].y));
                nm[m] = add(t.n[m].x, up(t.n[m].y));
            }
            const Trans s = transverse<SUB>(Wn, fluct<SUB>(Wn));
#pragma unroll
            for (int m = 0; m < 3; m++) {
                const int k = m == 0 ? 0 : 3 - m;   // y-edge frame (h, hv, hu)
                const float px = add(px2[m], s.p[k].x), mx = add(mx2[m], s.n[k].x);
                const float tx = add(px, dn(mx));   // of row j-1's x-edge (l|l+1)
                nx[m] = sub(tx, up(tx));
                px2[m] = s.p[k].y;
                mx2[m] = s.n[k].y;
            }
            N = net3(W1, W2, Wn, nuy, ORD, SUB);
        };
        if (__all_sync(kFull, (lane < 1 || lane > kLanes - 3 || slow(w)) &&
                                  (lane < 1 || lane > kLanes - 2 || (slow(Wn) && slow(W2)))))
            row(std::true_type());
        else
            row(std::false_type());
        const float L[3] = {N.L0, N.L2, N.L1};
        float d[3], t2[3];
#pragma unroll
        for (int m = 0; m < 3; m++) {
            t2[m] = add(py1[m], my[m]);   // of the y-edge (j-2|j-1)
            d[m] = fma(kt, sub(t2[m], t1[m]), mul(-nuy, add(nr[m], L[m])));
            t1[m] = t2[m];
        }
        if (j >= y0 + 2 && out) {   // row j-2 is complete
            const float ne = add(q1[0], d[0]), nmu = add(q1[1], d[1]), nmv = add(q1[2], d[2]);
            const size_t o = (size_t)(j - 2) * v.nx + gi;
            v.o0[o] = ne;
            v.o1[o] = nmu;
            v.o2[o] = nmv;
            const float h = add(h1, d[0]);
            bad |= !(h > 0.f) || !isfinite(nmu) || !isfinite(nmv);
            smax = fmaxf(smax, cfl_f32(h, nmu, nmv, g, v.rdx, v.rdy, 1));
        }
        // row j-1 takes its x-edges
        const float x0d = fma(kt, nx[0], xb[0]);
        q1[0] = add(B.eta, x0d);
        h1 = add(B.h, x0d);
        q1[1] = add(B.mn, fma(kt, nx[1], xb[1]));
        q1[2] = add(B.mt, fma(kt, nx[2], xb[2]));
#pragma unroll
        for (int m = 0; m < 3; m++) { py1[m] = py[m]; py[m] = np[m]; my[m] = nm[m]; xb[m] = nb[m]; }
        nr[0] = N.R0; nr[1] = N.R2; nr[2] = N.R1;
        B = c;
        W1 = W2; W2 = Wn;
    }
}

}  // namespace strip
}  // namespace swadj
