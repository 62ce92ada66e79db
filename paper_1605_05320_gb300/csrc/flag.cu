// flag.cu -- adjoint-weighted flagging (Sec. 4.1, 4.2, Sec. 6) and gauges.
//
// For the forward state at its device time t and q = (eta, hu, hv) the pass
// computes m = max over tau in [t, T] of |q^(tau) . q|, T = min(t + (t_f -
// t_s), t_f), the window clipped to the stored snapshot times, with q^
// bilinear in space (component by component, clamped at the outermost
// adjoint cell centres) and either linear in time (INTERP: the maximum of a
// piecewise-linear function sits at a window end or at a snapshot time inside
// it) or taken over every bracketing snapshot (BRACKET, Eq. ip_timepoint).
// m = 0 where the forward cell is dry or a positively weighted adjoint cell
// is dry (Sec. 6).  The pass streams each snapshot once per cell: it is
// bandwidth bound, so the snapshot loop is written for coalesced loads.
#include <type_traits>

#include "flag.cuh"
#include "gauge.cuh"

namespace swadj {

struct Window {
    int empty;
    int k0, k1;          // snapshots read: k0..k1 inclusive
    int ki0, ki1;        // snapshots strictly inside the window (INTERP), or
                         // the whole read range (BRACKET)
    int kh, kl;          // INTERP: bracket index at hi and at lo
    int exact_h, exact_l;
    double ah, al;       // weights on snapshot kh (resp. kl) at hi (lo)
    double lo, hi;
};

// Index k of the snapshot interval holding s: the first k (from 0) whose
// successor is no later than s, i.e. tau[k+1] <= s (K-1 if none).
__device__ __forceinline__ int bracket_index(const double *tau, int K, double s) {
    int a = 1, b = K;  // first j in [1, K) with tau[j] <= s, else K
    while (a < b) {
        const int m = (a + b) >> 1;
        if (tau[m] > s) a = m + 1;
        else b = m;
    }
    return a - 1;
}

__device__ Window make_window(const double *tau, int K, double t, double t_s,
                              double t_f, int mode) {
    Window w;
    double T = t + (t_f - t_s);
    if (T > t_f) T = t_f;
    double lo = t, hi = T;
    w.empty = 1;
    w.k0 = 0; w.k1 = -1; w.ki0 = 0; w.ki1 = -1;
    w.kh = -2; w.kl = -2; w.exact_h = 1; w.exact_l = 1;
    w.ah = 1.0; w.al = 1.0;
    if (K < 1) return w;
    if (lo < tau[K - 1]) lo = tau[K - 1];
    if (hi > tau[0]) hi = tau[0];
    w.lo = lo; w.hi = hi;
    if (lo > hi || t > t_f) return w;
    w.empty = 0;
    if (mode == SWA_FLAG_BRACKET) {
        int kb = K - 1, ke = 0;
        for (int k = 0; k < K; k++) if (tau[k] <= lo) { kb = k; break; }
        for (int k = K - 1; k >= 0; k--) if (tau[k] >= hi) { ke = k; break; }
        w.k0 = ke; w.k1 = kb;
        w.ki0 = ke; w.ki1 = kb;
        return w;
    }
    const int kh = bracket_index(tau, K, hi);
    const int kl = bracket_index(tau, K, lo);
    w.kh = kh; w.kl = kl;
    w.exact_h = (kh + 1 >= K || tau[kh] == hi);
    w.exact_l = (kl + 1 >= K || tau[kl] == lo);
    if (!w.exact_h) w.ah = (hi - tau[kh + 1]) / (tau[kh] - tau[kh + 1]);
    if (!w.exact_l) w.al = (lo - tau[kl + 1]) / (tau[kl] - tau[kl + 1]);
    w.k0 = kh;
    w.k1 = w.exact_l ? kl : kl + 1;
    if (w.k1 < w.k0) w.k1 = w.k0;
    // tau[k] in (lo, hi) exactly for k in [kh + 1, kl], minus an end that
    // coincides with lo or hi
    w.ki0 = kh + 1;
    w.ki1 = kl;
    while (w.ki0 <= w.ki1 && !(tau[w.ki0] < hi)) w.ki0++;
    while (w.ki1 >= w.ki0 && !(tau[w.ki1] > lo)) w.ki1--;
    return w;
}

// The window of a pass, formed by thread 0 of a block of 256 from a copy of
// the snapshot times in shared memory (its searches are chains of dependent
// loads: a few microseconds from global memory in every pass).
constexpr int kTauMax = 512;
__device__ __forceinline__ void block_window(Window &sw, const double *tau, int K,
                                             const DevClock *clk, double t_s, double t_f,
                                             int mode) {
    __shared__ double stau[kTauMax];
    for (int k = threadIdx.x; k < K && K <= kTauMax; k += 256) stau[k] = tau[k];
    __syncthreads();
    if (threadIdx.x == 0)
        sw = make_window(K <= kTauMax ? stau : tau, K, clk->t, t_s, t_f, mode);
    __syncthreads();
}

// Arithmetic of the flag products.  In float every rounding is fixed in the
// source (fmaf and unfused multiplies), so the pruned and the full variant
// form the same numbers; double keeps the plain expressions.
__device__ __forceinline__ float acc(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double acc(double a, double b, double c) { return a * b + c; }
__device__ __forceinline__ float dot3(float a, float x, float b, float y, float c, float z) {
    return fmaf(c, z, fmaf(b, y, __fmul_rn(a, x)));
}
__device__ __forceinline__ double dot3(double a, double x, double b, double y, double c,
                                       double z) {
    return a * x + b * y + c * z;
}
__device__ __forceinline__ float lerp2(float a, float x, float b, float y) {
    return fmaf(a, x, __fmul_rn(b, y));
}
__device__ __forceinline__ double lerp2(double a, double x, double b, double y) {
    return a * x + b * y;
}

// Products are accumulated in float when both the forward state and the
// snapshots are float (the bandwidth-bound FP32 path; GB300's FP64 rate is a
// small fraction of its FP32 rate) and in double otherwise.
//
// A block takes `cells` cells at a time (a power of 2 up to 256), 256 / cells
// threads each: on a small grid the snapshots of a cell are shared among
// threads, so that the pass does not wait for one thread's walk through the
// whole window.  Every product is formed as by one thread, and the maximum
// does not depend on the order.
// Measured, us per pass: 2000 cells in 1D with 701 FP64 snapshots 185 with one
// thread a cell, 26 so.
// The FP32 pass on one grid waits for memory, so a thread has several snapshots
// in flight.  Measured, us per pass, one / so: 511 x 509 with about 40 snapshots in
// the window 59 / 34, 1001 x 999 142 / 101, 1D 10^6 cells 55 / 39.  The blocks per
// SM are those whose registers hold that: 5 for FP32 (48 registers) 52 at 511 x
// 509, and for FP64, which its units bound, 4 (56 registers) left 401 x 399 in blocks
// of 256 cells in two rounds, 104 against 96.  On another grid the compiler's own 63
// registers stand: a bound of 4 made it 64, and 332 x 1139 over 83 x 284 22.9 to 23.4.
template <typename R, typename S, bool SAME>
__global__ void __launch_bounds__(256, !SAME ? 0 : sizeof(R) + sizeof(S) == 8 ? 4 : 5)
    flag_kernel(FlagParams<R, S> p, int cells) {
    using A = typename std::conditional<sizeof(R) == 4 && sizeof(S) == 4, float,
                                        double>::type;
    __shared__ Window sw;
    block_window(sw, p.tau, p.K, p.clk, p.t_s, p.t_f, p.mode);
    const Window &w = sw;
    const int cur = p.clk->cur;
    const R *q0 = p.q[cur][0], *q1 = p.q[cur][1], *q2 = p.q[cur][2];
    const size_t n = (size_t)p.nx * p.ny;
    const int segs = 256 / cells, seg = threadIdx.x / cells, ci = threadIdx.x - seg * cells;
    __shared__ A s_m[256], s_end[4][128];   // per thread, per cell (dh0, dh1, dl0, dl1)
    int f = 0;
    // persistent grid: each block walks cells i, i + gridDim.x * cells, ...
    for (size_t i0 = (size_t)blockIdx.x * cells; i0 < n; i0 += (size_t)gridDim.x * cells) {
        const bool in = i0 + ci < n;
        const size_t i = in ? i0 + ci : n - 1;
        A m = A(0);
        const R a = q0[i], b = p.bath[i];
        R h, eta;
        if (sizeof(R) == 4) { eta = a; h = a + b; }
        else { h = a; eta = a + b; }
        const A qe = (A)eta, qu = (A)q1[i];
        const A qv = p.two_d ? (A)q2[i] : A(0);
        bool dry = !(h > p.dry_tol);
        size_t st[4] = {i, i, i, i};
        A wt[4] = {A(1), A(0), A(0), A(0)};
        if (!SAME && sizeof(A) == 4 && p.two_d) {
            // FP32 pass: the stencil from the float map (FP64 is a small
            // fraction of the FP32 rate on this GPU)
            const int ix = (int)(i % p.nx), jy = (int)(i / p.nx);
            float fx = fmaf((float)ix + 0.5f, p.frx, p.fcx);
            fx = fminf(fmaxf(fx, 0.f), (float)(p.anx - 1));
            int i0 = (int)floorf(fx);
            if (i0 > p.anx - 2) i0 = p.anx - 2;
            if (i0 < 0) i0 = 0;
            float ax = fx - (float)i0;
            const int i1 = p.anx > 1 ? i0 + 1 : i0;
            if (p.anx == 1) ax = 0.f;
            float fy = fmaf((float)jy + 0.5f, p.fry, p.fcy);
            fy = fminf(fmaxf(fy, 0.f), (float)(p.any - 1));
            int j0 = (int)floorf(fy);
            if (j0 > p.any - 2) j0 = p.any - 2;
            if (j0 < 0) j0 = 0;
            float ay = fy - (float)j0;
            const int j1 = p.any > 1 ? j0 + 1 : j0;
            if (p.any == 1) ay = 0.f;
            st[0] = (size_t)j0 * p.anx + i0; wt[0] = (A)__fmul_rn(1.f - ax, 1.f - ay);
            st[1] = (size_t)j0 * p.anx + i1; wt[1] = (A)__fmul_rn(ax, 1.f - ay);
            st[2] = (size_t)j1 * p.anx + i0; wt[2] = (A)__fmul_rn(1.f - ax, ay);
            st[3] = (size_t)j1 * p.anx + i1; wt[3] = (A)__fmul_rn(ax, ay);
        } else if (!SAME) {
            const int ix = (int)(i % p.nx), jy = (int)(i / p.nx);
            const double x = p.x_lo + ((double)ix + 0.5) * p.dx;
            const double y = p.y_lo + ((double)jy + 0.5) * p.dy;
            double fx = (x - p.ax_lo) / p.adx - 0.5;
            fx = fx < 0.0 ? 0.0 : (fx > (double)(p.anx - 1) ? (double)(p.anx - 1) : fx);
            int i0 = (int)floor(fx);
            if (i0 > p.anx - 2) i0 = p.anx - 2;
            if (i0 < 0) i0 = 0;
            double ax = fx - (double)i0;
            const int i1 = p.anx > 1 ? i0 + 1 : i0;
            if (p.anx == 1) ax = 0.0;
            if (!p.two_d) {
                st[0] = i0; st[1] = i1;
                wt[0] = (A)(1.0 - ax); wt[1] = (A)ax;
            } else {
                double fy = (y - p.ay_lo) / p.ady - 0.5;
                fy = fy < 0.0 ? 0.0 : (fy > (double)(p.any - 1) ? (double)(p.any - 1) : fy);
                int j0 = (int)floor(fy);
                if (j0 > p.any - 2) j0 = p.any - 2;
                if (j0 < 0) j0 = 0;
                double ay = fy - (double)j0;
                const int j1 = p.any > 1 ? j0 + 1 : j0;
                if (p.any == 1) ay = 0.0;
                st[0] = (size_t)j0 * p.anx + i0; wt[0] = (A)((1.0 - ax) * (1.0 - ay));
                st[1] = (size_t)j0 * p.anx + i1; wt[1] = (A)(ax * (1.0 - ay));
                st[2] = (size_t)j1 * p.anx + i0; wt[2] = (A)((1.0 - ax) * ay);
                st[3] = (size_t)j1 * p.anx + i1; wt[3] = (A)(ax * ay);
            }
        }
#pragma unroll
        for (int c = 0; c < 4; c++)
            if (wt[c] > A(0) && !p.awet[st[c]]) dry = true;
        A mm = A(0), e0 = A(0), e1 = A(0), e2 = A(0), e3 = A(0);
        if (!w.empty && !dry) {
            A dh0 = A(0), dh1 = A(0), dl0 = A(0), dl1 = A(0);
            auto snapshot = [&](int k) {
                const S *s = p.snaps + (size_t)k * p.snap_stride;
                A v0, v1, v2 = A(0);
                if (SAME) {
                    v0 = (A)s[i];
                    v1 = (A)s[p.na + i];
                    if (p.ncomp == 3) v2 = (A)s[2 * p.na + i];
                } else {
                    v0 = A(0); v1 = A(0);
#pragma unroll
                    for (int c = 0; c < 4; c++) {
                        v0 = acc(wt[c], (A)s[st[c]], v0);
                        v1 = acc(wt[c], (A)s[p.na + st[c]], v1);
                        if (p.ncomp == 3) v2 = acc(wt[c], (A)s[2 * p.na + st[c]], v2);
                    }
                }
                const A d = dot3(v0, qe, v1, qu, v2, qv);
                if (k >= w.ki0 && k <= w.ki1) m = fabs(d) > m ? fabs(d) : m;
                if (k == w.kh) dh0 = d;
                if (k == w.kh + 1) dh1 = d;
                if (k == w.kl) dl0 = d;
                if (k == w.kl + 1) dl1 = d;
            };
            if constexpr (SAME && sizeof(A) == 4) {
                if (p.ncomp == 3) {
#pragma unroll 4
                    for (int k = w.k0 + seg; k <= w.k1; k += segs) snapshot(k);
                } else {   // 8 at a time, a short last batch repeating its first
                    for (int k = w.k0 + seg; k <= w.k1; k += 8 * segs)
#pragma unroll
                        for (int j = 0; j < 8; j++)
                            snapshot(k + j * segs <= w.k1 ? k + j * segs : k);
                }
            } else {
                for (int k = w.k0 + seg; k <= w.k1; k += segs) snapshot(k);
            }
            if (segs > 1) {   // the threads of a cell meet in shared memory
                s_m[threadIdx.x] = m;
                const int ks[4] = {w.kh, w.kh + 1, w.kl, w.kl + 1};
                const A ds[4] = {dh0, dh1, dl0, dl1};
#pragma unroll
                for (int e = 0; e < 4; e++)
                    if (ks[e] >= w.k0 && ks[e] <= w.k1 && (ks[e] - w.k0) % segs == seg)
                        s_end[e][ci] = ds[e];
            }
            mm = m;
            e0 = dh0; e1 = dh1; e2 = dl0; e3 = dl1;
        }
        if (segs > 1) {
            __syncthreads();
            if (seg == 0 && !w.empty && !dry) {
                for (int k = 1; k < segs; k++) {
                    const A v = s_m[k * cells + ci];
                    mm = v > mm ? v : mm;
                }
                const bool two_h = w.kh + 1 <= w.k1, two_l = w.kl + 1 <= w.k1;
                if (p.mode != SWA_FLAG_BRACKET) {
                    e0 = s_end[0][ci]; e2 = s_end[2][ci];
                    if (two_h) e1 = s_end[1][ci];
                    if (two_l) e3 = s_end[3][ci];
                }
            }
            __syncthreads();
        }
        if (seg == 0 && in) {
            if (!w.empty && !dry && p.mode != SWA_FLAG_BRACKET) {
                const A ah = (A)w.ah, al = (A)w.al;
                const A vh = w.exact_h ? e0 : lerp2(ah, e0, A(1) - ah, e1);
                const A vl = w.exact_l ? e2 : lerp2(al, e2, A(1) - al, e3);
                mm = fabs(vh) > mm ? fabs(vh) : mm;
                mm = fabs(vl) > mm ? fabs(vl) : mm;
            }
            const int fi = (!w.empty && !dry && mm >= (A)p.tol) ? 1 : 0;
            p.flags[i] = (uint8_t)fi;
            if (p.maxip) p.maxip[i] = (float)mm;
            f += fi;
        }
    }
    int cnt = f;
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(p.count, (unsigned long long)cnt);
}

// FP32 forward state and FP32 snapshots on the same grid: the bandwidth-bound
// case.  Each thread takes 4 consecutive cells with 16-byte loads; the window
// (index ranges and end weights) is computed once per block, so the per-cell
// loop has no FP64 work at all.
//
// PRUNE (no maxip output requested, envelope present): a group of snapshots
// is read only where it can matter.  For a cell with forward state q and a
// group whose per-component maxima over the cell's quad are (Me, Mu, Mv),
// every product satisfies |q^ . q| <= Me |eta| + Mu |hu| + Mv |hv| =: bnd.
// If bnd < tol (1 - 1e-5) for every wet cell of the quad, no product of the
// group can reach tol even after float rounding (the products and bnd carry
// relative errors of a few 1e-7), and neither can a time-interpolated end
// value built from two such products; the group is skipped.  An end value
// (INTERP) is computed from both of its snapshots whenever either of their
// groups is read.  Every product that is formed is the one the unpruned pass
// forms, so the flags and the count are identical to the unpruned pass; only
// m differs (it may omit values below tol), hence PRUNE only without maxip.
// Ahead of the forward wave q = 0 exactly: such a quad reads its state only.
// On one grid a warp's loads are consecutive at every stage and its warps need
// not wait for one another, so a thread keeps its quad from state to flags.
// The phases of the other-grid pass below were up to 25 % faster here where
// many groups matter (160 / 128 us at 2048^2), but up to 45 % slower where
// all cells move and few groups do (27 / 39, 68 / 85).
template <bool PRUNE>
__global__ void __launch_bounds__(256, 4) flag_kernel_f32x4(FlagParams<float, float> p) {
    __shared__ Window sw;
    block_window(sw, p.tau, p.K, p.clk, p.t_s, p.t_f, p.mode);
    const Window &w = sw;   // read from shared memory where used
    const int cur = p.clk->cur;
    const size_t n4 = ((size_t)p.nx * p.ny) >> 2;
    const bool interp = p.mode != SWA_FLAG_BRACKET;
    const float tol = (float)p.tol;
    const float tolp = (float)(p.tol * (1.0 - 1e-5));
    const int gb0 = w.k0 / kEnvGroup, gb1 = w.k1 / kEnvGroup;
    const size_t cs = p.na >> 2, ks = p.snap_stride >> 2;
    int f = 0;
    // persistent grid: each block walks quads i, i + gridDim.x * 256, ...
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4;
         i += (size_t)gridDim.x * blockDim.x) {
        const float4 e = reinterpret_cast<const float4 *>(p.q[cur][0])[i];
        const float4 u = reinterpret_cast<const float4 *>(p.q[cur][1])[i];
        const float4 v = reinterpret_cast<const float4 *>(p.q[cur][2])[i];
        const float4 hb = reinterpret_cast<const float4 *>(p.bath)[i];
        const uchar4 wet = reinterpret_cast<const uchar4 *>(p.awet)[i];
        const float dt = p.dry_tol;
        const bool ok0 = e.x + hb.x > dt && wet.x, ok1 = e.y + hb.y > dt && wet.y;
        const bool ok2 = e.z + hb.z > dt && wet.z, ok3 = e.w + hb.w > dt && wet.w;
        float4 m = make_float4(0.f, 0.f, 0.f, 0.f);
        float4 dh0 = m, dh1 = m, dl0 = m, dl1 = m;
        // envelope test of group gb (PRUNE only): true when no product of the
        // group can reach tol in any wet cell of the quad
        auto skip = [&](int gb) -> bool {
            const float *eg = p.env + (size_t)gb * 3 * n4;
            const float Me = __ldg(eg + i), Mu = __ldg(eg + n4 + i), Mv = __ldg(eg + 2 * n4 + i);
            const float b0 = Me * fabsf(e.x) + Mu * fabsf(u.x) + Mv * fabsf(v.x);
            const float b1 = Me * fabsf(e.y) + Mu * fabsf(u.y) + Mv * fabsf(v.y);
            const float b2 = Me * fabsf(e.z) + Mu * fabsf(u.z) + Mv * fabsf(v.z);
            const float b3 = Me * fabsf(e.w) + Mu * fabsf(u.w) + Mv * fabsf(v.w);
            return (!ok0 || b0 < tolp) && (!ok1 || b1 < tolp) && (!ok2 || b2 < tolp) &&
                   (!ok3 || b3 < tolp);
        };
        // PRUNE: a quad whose forward state is exactly zero (the ocean at rest
        // ahead of the wave) has every product exactly zero, m = 0 as in the
        // full pass, so even its envelope is not read
        const bool rest = e.x == 0.f && e.y == 0.f && e.z == 0.f && e.w == 0.f &&
                          u.x == 0.f && u.y == 0.f && u.z == 0.f && u.w == 0.f &&
                          v.x == 0.f && v.y == 0.f && v.z == 0.f && v.w == 0.f;
        if (!w.empty && (!PRUNE || ((ok0 || ok1 || ok2 || ok3) && !rest))) {
            const float4 *s0 = reinterpret_cast<const float4 *>(p.snaps) + i;
            // skip bits of the first 32 groups of the window (256 snapshots),
            // their loads issued independently of one another
            unsigned mask = 0u;
            if (PRUNE) {
                const int ng = gb1 - gb0 + 1 < 32 ? gb1 - gb0 + 1 : 32;
#pragma unroll 2
                for (int j = 0; j < ng; j++)
                    if (skip(gb0 + j)) mask |= 1u << j;
            }
            // groups past the first 32 of the window are always read
            auto skipped = [&](int gb) -> bool {
                const int j = gb - gb0;
                return j < 32 && ((mask >> j) & 1u) != 0u;
            };
            bool need_h = true, need_l = true;
            if (PRUNE && interp) {
                const int kh1 = w.exact_h ? w.kh : w.kh + 1;
                const int kl1 = w.exact_l ? w.kl : w.kl + 1;
                need_h = !(skipped(w.kh / kEnvGroup) && skipped(kh1 / kEnvGroup));
                need_l = !(skipped(w.kl / kEnvGroup) && skipped(kl1 / kEnvGroup));
            }
            for (int gb = gb0; gb <= gb1; gb++) {
                const bool gs = PRUNE && skipped(gb);
                const int ka = w.k0 > gb * kEnvGroup ? w.k0 : gb * kEnvGroup;
                const int kb = w.k1 < gb * kEnvGroup + kEnvGroup - 1 ? w.k1
                                                                    : gb * kEnvGroup + kEnvGroup - 1;
                if (gs) {
                    // a skipped group can only supply the snapshots of a
                    // needed end pair
                    const bool hh = need_h && w.kh <= kb && w.kh + 1 >= ka;
                    const bool ll = need_l && w.kl <= kb && w.kl + 1 >= ka;
                    if (!interp || !(hh || ll)) continue;
                }
#pragma unroll 2
                for (int k = ka; k <= kb; k++) {
                    if (gs && !((need_h && (k == w.kh || k == w.kh + 1)) ||
                                (need_l && (k == w.kl || k == w.kl + 1))))
                        continue;
                    const float4 a = __ldcs(s0 + (size_t)k * ks);
                    const float4 b = __ldcs(s0 + (size_t)k * ks + cs);
                    const float4 c = __ldcs(s0 + (size_t)k * ks + 2 * cs);
                    float4 d;
                    // rounding fixed in the source, identical in both variants
                    d.x = fmaf(c.x, v.x, fmaf(b.x, u.x, __fmul_rn(a.x, e.x)));
                    d.y = fmaf(c.y, v.y, fmaf(b.y, u.y, __fmul_rn(a.y, e.y)));
                    d.z = fmaf(c.z, v.z, fmaf(b.z, u.z, __fmul_rn(a.z, e.z)));
                    d.w = fmaf(c.w, v.w, fmaf(b.w, u.w, __fmul_rn(a.w, e.w)));
                    if (k >= w.ki0 && k <= w.ki1) {
                        m.x = fmaxf(m.x, fabsf(d.x)); m.y = fmaxf(m.y, fabsf(d.y));
                        m.z = fmaxf(m.z, fabsf(d.z)); m.w = fmaxf(m.w, fabsf(d.w));
                    }
                    if (k == w.kh) dh0 = d;
                    if (k == w.kh + 1) dh1 = d;
                    if (k == w.kl) dl0 = d;
                    if (k == w.kl + 1) dl1 = d;
                }
            }
            if (interp) {
                const float ah = (float)w.ah, al = (float)w.al;
                const float bh = 1.f - ah, bl = 1.f - al;
#define SWADJ_ENDS(c)                                                          \
    {                                                                          \
        const float vh = w.exact_h ? dh0.c : fmaf(ah, dh0.c, __fmul_rn(bh, dh1.c)); \
        const float vl = w.exact_l ? dl0.c : fmaf(al, dl0.c, __fmul_rn(bl, dl1.c)); \
        m.c = fmaxf(m.c, fmaxf(fabsf(vh), fabsf(vl)));                         \
    }
                SWADJ_ENDS(x) SWADJ_ENDS(y) SWADJ_ENDS(z) SWADJ_ENDS(w)
#undef SWADJ_ENDS
            }
        }
        const int f0 = (!w.empty && ok0 && m.x >= tol), f1 = (!w.empty && ok1 && m.y >= tol);
        const int f2 = (!w.empty && ok2 && m.z >= tol), f3 = (!w.empty && ok3 && m.w >= tol);
        reinterpret_cast<uchar4 *>(p.flags)[i] = make_uchar4(f0, f1, f2, f3);
        if (!PRUNE && p.maxip) {
            const float4 mm = make_float4(ok0 ? m.x : 0.f, ok1 ? m.y : 0.f,
                                          ok2 ? m.z : 0.f, ok3 ? m.w : 0.f);
            reinterpret_cast<float4 *>(p.maxip)[i] = w.empty ? make_float4(0.f, 0.f, 0.f, 0.f) : mm;
        }
        f += f0 + f1 + f2 + f3;
    }
    int cnt = f;
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(p.count, (unsigned long long)cnt);
}

// The pruned pass with the adjoint on another grid: FP32 state and FP32
// snapshots of a 2D adjoint with an envelope, no maxip output.  A group of
// snapshots is read for a cell only where it can matter: for
// a cell with forward state q and a group whose per-component maxima over the
// envelope quads that hold its stencil are (Me, Mu, Mv), every product
// satisfies |q^ . q| <= Me |eta| + Mu |hu| + Mv |hv| =: bnd (an interpolated
// component is a convex combination of its stencil's).  If bnd < tol (1 -
// 1e-5) for every wet cell of a quad of 4 cells, no product of the group can
// reach tol even after float rounding (the products and bnd carry relative
// errors of a few 1e-7), and neither can a time-interpolated end value built
// from two such products; the group is skipped.  An end value (INTERP) is
// computed from both of its snapshots whenever either of their groups is
// read.  Every product that is formed is the one the full pass forms, so the
// flags and the count are identical to the full pass; only m differs (it may
// omit values below tol), hence no maxip.  Where q = 0 exactly (the ocean at
// rest ahead of the wave) nothing but the state is read.
//
// What bounds it is the latency of dependent loads (state, envelope, then
// snapshots), with work in few places.  A block therefore takes a tile of up to 256
// quads in phases: it loads the states, packs the quads that move into a
// list, tests (quad, group) pairs spread over its threads, packs those that
// can matter into a second list, and spreads these over its threads again,
// each forming the products of up to 8 snapshots; the maxima meet in shared
// memory.  (One quad per thread from its state to its last snapshot left most
// lanes of a warp waiting for its busiest quad; tiles of one warp were slower
// on grids of few tiles, where the groups of a quad want many threads.)
// Measured, us per pass, before / so (waves over a tenth and a third of the
// domain): 512^2 over a 2048^2 adjoint with 401
// snapshots 147 / 69 and 138 / 92; 4096^2 over 1024^2 237 / 147 and 427 / 313;
// 1001 x 700 over 252 x 176 19.6 / 16.6 and 27.8 / 24.5.  Reading the group
// with the largest bound first, to leave the others of a flagged cell, was
// slower (its extra phases cost more than the reads: 122 and 418 us).
// A grid of few tiles takes smaller ones, with the same threads: the fewest quads
// (32 to 256) whose tiles are still one wave of blocks.  Measured, us per pass,
// all cells moving, 256 / 128 / 64 / 32 quads: 128^2 over 192^2, 150 snapshots 51 / 32 /
// 23 / 18 (253 tiles of 32 at 180^2: 47 / 31 / 22 / 19); 256^2 over 384^2 41 / 27 / 22 /
// 23 (512 tiles of 32); 700^2 over 1048^2 62 / 62 / 77 / 90.
constexpr int kTile = 256;      // quads per tile at most, threads per block
constexpr int kChunk = 32;      // snapshot groups tested at a time
struct FlagTile {
    float q[3][4][kTile];       // eta, hu, hv of the packed quads' cells
    int m[4][kTile];            // max |q^ . q| so far, as the bits of a float >= 0
    unsigned off[kTile];                          // first cell of the packed quad
    int ix[kTile], jy[kTile];                     // its column and row
    unsigned char ok[kTile];                      // wet cells
    unsigned char need_h[kTile], need_l[kTile];   // the window's ends can matter
    unsigned short item[kTile * kChunk];          // packed quad | group << 8
    int nact, nitem;
};

// Adjoint stencil of forward cell (ix, jy) in float: first cell and weights.
struct Stencil {
    int i0, j0, di, dj;
    float w[4];
};
__device__ __forceinline__ Stencil stencil_f32(const FlagParams<float, float> &p, int ix, int jy) {
    Stencil t;
    float fx = fmaf((float)ix + 0.5f, p.frx, p.fcx);
    fx = fminf(fmaxf(fx, 0.f), (float)(p.anx - 1));
    int i0 = (int)floorf(fx);
    if (i0 > p.anx - 2) i0 = p.anx - 2;
    if (i0 < 0) i0 = 0;
    float ax = fx - (float)i0;
    if (p.anx == 1) ax = 0.f;
    float fy = fmaf((float)jy + 0.5f, p.fry, p.fcy);
    fy = fminf(fmaxf(fy, 0.f), (float)(p.any - 1));
    int j0 = (int)floorf(fy);
    if (j0 > p.any - 2) j0 = p.any - 2;
    if (j0 < 0) j0 = 0;
    float ay = fy - (float)j0;
    if (p.any == 1) ay = 0.f;
    t.i0 = i0; t.j0 = j0;
    t.di = p.anx > 1 ? 1 : 0;
    t.dj = p.any > 1 ? 1 : 0;
    t.w[0] = __fmul_rn(1.f - ax, 1.f - ay);
    t.w[1] = __fmul_rn(ax, 1.f - ay);
    t.w[2] = __fmul_rn(1.f - ax, ay);
    t.w[3] = __fmul_rn(ax, ay);
    return t;
}

// VEC: nx % 4 == 0 (quads never straddle a row, 16-byte loads).
template <bool VEC>
__global__ void __launch_bounds__(kTile, 3)
    flag_pruned_kernel(FlagParams<float, float> p, int tile) {
    __shared__ Window sw;
    __shared__ FlagTile T;
    const int t = threadIdx.x, lane = t & 31;
    const unsigned below = (1u << lane) - 1u;
    block_window(sw, p.tau, p.K, p.clk, p.t_s, p.t_f, p.mode);
    const Window &w = sw;
    const int cur = p.clk->cur;
    const float *q0 = p.q[cur][0], *q1 = p.q[cur][1], *q2 = p.q[cur][2];
    const int nq = (p.nx + 3) / 4;
    const unsigned quads = (unsigned)nq * (unsigned)p.ny;
    const bool interp = p.mode != SWA_FLAG_BRACKET;
    const float tol = (float)p.tol, tolp = (float)(p.tol * (1.0 - 1e-5));
    const int gb0 = w.k0 / kEnvGroup, gb1 = w.k1 / kEnvGroup;
    const int kh1 = w.exact_h ? w.kh : w.kh + 1, kl1 = w.exact_l ? w.kl : w.kl + 1;
    const int gh0 = w.kh / kEnvGroup, gh1 = kh1 / kEnvGroup;
    const int gl0 = w.kl / kEnvGroup, gl1 = kl1 / kEnvGroup;
    const size_t na = p.na, na4 = na >> 2;
    int f = 0;
    for (unsigned q0th = blockIdx.x * tile; q0th < quads; q0th += gridDim.x * tile) {
        if (t == 0) { T.nact = 0; T.nitem = 0; }
        __syncthreads();
        // 1) states; every flag starts at 0
        const unsigned quad = q0th + t;
        unsigned ok = 0;
        float e[4], u[4], v[4];
        int jy = 0, ix = 0;
        unsigned o = 0;
        if (t < tile && quad < quads) {
            jy = (int)(quad / (unsigned)nq);
            ix = 4 * (int)(quad - (unsigned)jy * (unsigned)nq);
            o = (unsigned)jy * (unsigned)p.nx + (unsigned)ix;
            float hb[4];
            if (VEC) {
                const float4 a = *reinterpret_cast<const float4 *>(q0 + o);
                const float4 b = *reinterpret_cast<const float4 *>(q1 + o);
                const float4 c = *reinterpret_cast<const float4 *>(q2 + o);
                const float4 d = *reinterpret_cast<const float4 *>(p.bath + o);
                e[0] = a.x; e[1] = a.y; e[2] = a.z; e[3] = a.w;
                u[0] = b.x; u[1] = b.y; u[2] = b.z; u[3] = b.w;
                v[0] = c.x; v[1] = c.y; v[2] = c.z; v[3] = c.w;
                hb[0] = d.x; hb[1] = d.y; hb[2] = d.z; hb[3] = d.w;
                *reinterpret_cast<uchar4 *>(p.flags + o) = make_uchar4(0, 0, 0, 0);
            } else {
#pragma unroll
                for (int c = 0; c < 4; c++) {
                    const bool in = ix + c < p.nx;
                    e[c] = in ? q0[o + c] : 0.f;
                    u[c] = in ? q1[o + c] : 0.f;
                    v[c] = in ? q2[o + c] : 0.f;
                    hb[c] = in ? p.bath[o + c] : 0.f;
                    if (in) p.flags[o + c] = 0;
                }
            }
            if (!w.empty) {
#pragma unroll
                for (int c = 0; c < 4; c++) {
                    if (e[c] == 0.f && u[c] == 0.f && v[c] == 0.f) continue;
                    bool wet = e[c] + hb[c] > p.dry_tol;
                    if (wet) {
                        const Stencil s = stencil_f32(p, ix + c, jy);
                        const uint8_t *a = p.awet + (size_t)s.j0 * p.anx + s.i0;
                        const uint8_t *b = a + (size_t)s.dj * p.anx;
                        wet = !((s.w[0] > 0.f && !a[0]) || (s.w[1] > 0.f && !a[s.di]) ||
                                (s.w[2] > 0.f && !b[0]) || (s.w[3] > 0.f && !b[s.di]));
                    }
                    ok |= wet ? 1u << c : 0u;
                }
            }
        }
        const unsigned vote = __ballot_sync(0xffffffffu, ok != 0);
        if (vote) {
            int at = 0;
            if (lane == 0) at = atomicAdd(&T.nact, __popc(vote));
            at = __shfl_sync(0xffffffffu, at, 0) + __popc(vote & below);
            if (ok) {
#pragma unroll
                for (int c = 0; c < 4; c++) {
                    T.q[0][c][at] = e[c];
                    T.q[1][c][at] = u[c];
                    T.q[2][c][at] = v[c];
                    T.m[c][at] = 0;
                }
                T.off[at] = o;
                T.ix[at] = ix;
                T.jy[at] = jy;
                T.ok[at] = (unsigned char)ok;
                T.need_h[at] = T.need_l[at] = 0;
            }
        }
        __syncthreads();
        const int nact = T.nact;
        if (nact == 0) continue;   // block-uniform
        // threads per quad in the group test: 256 / P, P >= nact a power of 2
        int logP = 5;
        while ((1 << logP) < nact) logP++;
        // product of the packed quad's cell c (all its cells) with snapshot k
        auto dot_cell = [&](const Stencil &s, int a, int c, int k) {
            const float *x = p.snaps + (size_t)k * p.snap_stride + (size_t)s.j0 * p.anx + s.i0;
            const float *y = x + (size_t)s.dj * p.anx;
            float d[3];
#pragma unroll
            for (int m = 0; m < 3; m++, x += na, y += na) {
                float r = fmaf(s.w[0], __ldg(x), 0.f);
                r = fmaf(s.w[1], __ldg(x + s.di), r);
                r = fmaf(s.w[2], __ldg(y), r);
                d[m] = fmaf(s.w[3], __ldg(y + s.di), r);
            }
            return dot3(d[0], T.q[0][c][a], d[1], T.q[1][c][a], d[2], T.q[2][c][a]);
        };
        for (int gc = gb0; gc <= gb1; gc += kChunk) {
            const int ng = gb1 - gc + 1 < kChunk ? gb1 - gc + 1 : kChunk;
            // 2) which (quad, group) can matter
            const int a2 = t & ((1 << logP) - 1), a = a2 < nact ? a2 : nact - 1;
            const unsigned oka = a2 < nact ? T.ok[a] : 0u;
            float ae[4], au[4], av[4];
#pragma unroll
            for (int c = 0; c < 4; c++) {   // a dry cell takes part with zeros
                const bool in = (oka >> c) & 1;
                ae[c] = in ? fabsf(T.q[0][c][a]) : 0.f;
                au[c] = in ? fabsf(T.q[1][c][a]) : 0.f;
                av[c] = in ? fabsf(T.q[2][c][a]) : 0.f;
            }
            // envelope quads x0 .. x1 and y0 .. y1 of the stencil's two rows
            unsigned x0, x1, y0, y1;
            const int ix = T.ix[a], jy = T.jy[a];
            const Stencil s0 = stencil_f32(p, ix, jy);
            const Stencil s1 = stencil_f32(p, ix + 3 < p.nx ? ix + 3 : p.nx - 1, jy);
            const unsigned r0 = (unsigned)s0.j0 * (unsigned)p.anx;
            const unsigned r1 = r0 + (unsigned)(s0.dj * p.anx);
            x0 = (r0 + s0.i0) >> 2; x1 = (r0 + s1.i0 + s1.di) >> 2;
            y0 = (r1 + s0.i0) >> 2; y1 = (r1 + s1.i0 + s1.di) >> 2;
            const unsigned xm = x1 - x0 > y1 - y0 ? x1 - x0 : y1 - y0;
            const int gstep = kTile >> logP;   // the same for all lanes of a warp
#pragma unroll 2
            for (int g = t >> logP; g < ng; g += gstep) {   // warp-uniform
                const float *eg = p.env + (size_t)(gc + g) * 3 * na4;
                float Me = __ldg(eg + x0), Mu = __ldg(eg + na4 + x0), Mv = __ldg(eg + 2 * na4 + x0);
                Me = fmaxf(Me, __ldg(eg + y0));
                Mu = fmaxf(Mu, __ldg(eg + na4 + y0));
                Mv = fmaxf(Mv, __ldg(eg + 2 * na4 + y0));
                for (unsigned k = 1; k <= xm; k++) {
                    const unsigned x = x0 + k < x1 ? x0 + k : x1, y = y0 + k < y1 ? y0 + k : y1;
                    Me = fmaxf(Me, fmaxf(__ldg(eg + x), __ldg(eg + y)));
                    Mu = fmaxf(Mu, fmaxf(__ldg(eg + na4 + x), __ldg(eg + na4 + y)));
                    Mv = fmaxf(Mv, fmaxf(__ldg(eg + 2 * na4 + x), __ldg(eg + 2 * na4 + y)));
                }
                bool need = false;
#pragma unroll
                for (int c = 0; c < 4; c++)
                    need = need || !(Me * ae[c] + Mu * au[c] + Mv * av[c] < tolp);
                need = need && oka != 0;
                const unsigned b = __ballot_sync(0xffffffffu, need);
                int at = 0;
                if (lane == 0 && b) at = atomicAdd(&T.nitem, __popc(b));
                at = __shfl_sync(0xffffffffu, at, 0) + __popc(b & below);
                if (need) {
                    T.item[at] = (unsigned short)(a | g << 8);
                    const int gg = gc + g;
                    if (interp && (gg == gh0 || gg == gh1)) T.need_h[a] = 1;
                    if (interp && (gg == gl0 || gg == gl1)) T.need_l[a] = 1;
                }
            }
            __syncthreads();
            const int nitem = T.nitem;
            // 3) the products of those groups strictly inside the window
            for (int it = t; it < 4 * nitem; it += kTile) {
                const int item = T.item[it >> 2], a = item & 255, c = it & 3;
                const int g = gc + (item >> 8);
                const int ka = w.ki0 > g * kEnvGroup ? w.ki0 : g * kEnvGroup;
                const int kb = w.ki1 < g * kEnvGroup + kEnvGroup - 1 ? w.ki1
                                                                    : g * kEnvGroup + kEnvGroup - 1;
                // a cell that is flagged already needs no other group
                if (!((T.ok[a] >> c) & 1) || __int_as_float(T.m[c][a]) >= tol) continue;
                const Stencil s = stencil_f32(p, T.ix[a] + c, T.jy[a]);
                float m = 0.f;
#pragma unroll 2
                for (int k = ka; k <= kb; k++) m = fmaxf(m, fabsf(dot_cell(s, a, c, k)));
                atomicMax(&T.m[c][a], __float_as_int(m));
            }
            __syncthreads();
            if (gc + kChunk <= gb1) {   // another chunk follows
                if (t == 0) T.nitem = 0;
                __syncthreads();
            }
        }
        // 4) the window's ends and the flags (a cell flagged already needs
        // neither end)
        for (int it = t; it < 4 * nact; it += kTile) {
            const int a = it >> 2;
            const size_t o = T.off[a];
            const float ah = (float)w.ah, al = (float)w.al, bh = 1.f - ah, bl = 1.f - al;
            const int c = it & 3;
            if (!((T.ok[a] >> c) & 1)) continue;   // flag 0 already
            const Stencil s = stencil_f32(p, T.ix[a] + c, T.jy[a]);
            float m = __int_as_float(T.m[c][a]);
            if (T.need_h[a] && !(m >= tol)) {
                const float d = dot_cell(s, a, c, w.kh);
                m = fmaxf(m, fabsf(w.exact_h ? d
                                             : fmaf(ah, d, __fmul_rn(bh, dot_cell(s, a, c, w.kh + 1)))));
            }
            if (T.need_l[a] && !(m >= tol)) {
                const float d = dot_cell(s, a, c, w.kl);
                m = fmaxf(m, fabsf(w.exact_l ? d
                                             : fmaf(al, d, __fmul_rn(bl, dot_cell(s, a, c, w.kl + 1)))));
            }
            if (m >= tol) {
                p.flags[o + c] = 1;
                f++;
            }
        }
        __syncthreads();
    }
    for (int o = 16; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
    if (lane == 0 && f) atomicAdd(p.count, (unsigned long long)f);
}

// Envelope of one stored snapshot, folded into its group: one thread per
// quad of 4 consecutive cells.
__global__ void __launch_bounds__(256) env_update_kernel(const float *slot, size_t na,
                                                         float *env, int first) {
    const size_t n4 = na >> 2;
    for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < n4;
         q += (size_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const float4 a = __ldcg(reinterpret_cast<const float4 *>(slot + c * na) + q);
            const float mx = fmaxf(fmaxf(fabsf(a.x), fabsf(a.y)), fmaxf(fabsf(a.z), fabsf(a.w)));
            float *o = env + c * n4 + q;
            *o = first ? mx : fmaxf(*o, mx);
        }
    }
}

int env_launch_update(const float *slot, size_t na, float *env_group, int first,
                      cudaStream_t st) {
    const size_t n4 = na >> 2;
    size_t blocks = (n4 + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    if (blocks < 1) blocks = 1;
    env_update_kernel<<<(unsigned)blocks, 256, 0, st>>>(slot, na, env_group, first);
    return swadj_host::cuda_check(cudaGetLastError(), "env_update_kernel");
}

// Blocks of a persistent flag pass: every SM filled with as many blocks of
// the kernel (256 threads each) as fit, at most `need`.
template <typename K>
static unsigned persistent_blocks(K kernel, int &per_sm, size_t need) {
    static int sms = 0;
    if (sms == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms < 1) sms = 1;
    }
    if (per_sm == 0) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 256, 0);
        if (per_sm < 1) per_sm = 1;
    }
    const size_t b = (size_t)per_sm * (size_t)sms;
    return (unsigned)(need < b ? need : b);
}

template <bool VEC>
static void launch_pruned(const FlagParams<float, float> &p, cudaStream_t st) {
    static int per_sm = 0;
    const size_t quads = (size_t)((p.nx + 3) / 4) * p.ny;
    const size_t wave = persistent_blocks(flag_pruned_kernel<VEC>, per_sm, SIZE_MAX);
    int tile = 32;
    while (tile < kTile && (quads + tile - 1) / tile > wave) tile *= 2;
    const size_t tiles = (quads + tile - 1) / tile;
    flag_pruned_kernel<VEC><<<(unsigned)(tiles < wave ? tiles : wave), kTile, 0, st>>>(p, tile);
}

template <typename R, typename S, bool SAME>
static void launch_full(const FlagParams<R, S> &p, size_t n, cudaStream_t st) {
    static int per_sm = 0;
    const size_t wave = persistent_blocks(flag_kernel<R, S, SAME>, per_sm, SIZE_MAX);
    const size_t sms = wave / per_sm;
    const bool f32 = sizeof(R) + sizeof(S) == 8;
    int cells = 256;
    if (SAME) {
        // fewer cells a block while the grid has under two blocks per SM and every
        // thread keeps 8 snapshots or more.  Measured, us per pass, 256 / 128 cells:
        // FP32 1D 50000 cells (1.3 blocks per SM), 600 snapshots 88 / 56, 100000 (2.6)
        // 18.6 / 19.2
        while (cells > 8 && n / cells < 2 * sms && 16 * (256 / cells) <= p.K) cells /= 2;
    }
    if (!SAME || !f32) {
        // From there the cells of the least rounds times a thread's snapshots and the
        // price of beginning a cell (on another grid every thread of it forms the
        // stencil), and at about the same cost those that fill a round.  FP32 waits
        // for memory, and a round is the resident blocks; FP64 is bound by its units,
        // and a round is a block per SM.
        // Measured, us per pass, 256 / 128 / 64 / 32 cells: FP32 200^2 over 300^2, 180
        // snapshots 150 / 83 / 87 / 71, 300^2 over 75^2, 15 snapshots 14 / 16 / 17 / 24;
        // FP64 230^2 over 57^2, 60 snapshots 138 / 112 / 124 / 148, 256^2 over 64^2, 15
        // snapshots 44 / 52 / 60 / 88; on one grid 351^2, 180 snapshots 193 / 172 / 173 /
        // 171, 391^2 193 / 220 / 201 / 209.
        const double setup = SAME ? 1.5 : f32 ? 8.0 : 4.0;
        const size_t round = f32 ? wave : sms;
        const int most = cells;
        double best = 0.0, margin = 1.0;
        for (int c = most; c >= 8 && (c == most || 4 * (256 / c) <= p.K); c /= 2) {
            const size_t blocks = (n + c - 1) / c, rounds = (blocks + round - 1) / round;
            const double cost = (double)rounds * (setup + (double)p.K * c / 256);
            if (c == most || cost < margin * best) {
                best = cost;
                cells = c;
                margin = !SAME && blocks < round ? 1.05 : 0.97;
            }
        }
    }
    const size_t blocks = (n + cells - 1) / cells;
    flag_kernel<R, S, SAME><<<(unsigned)(blocks < wave ? blocks : wave), 256, 0, st>>>(p, cells);
}

// Cells times snapshots up to which a pass over another grid reads every
// snapshot: the phases of the pruned pass, one waiting for the other, take longer
// than the products then.  Measured, us per pass, full / pruned (waves over a
// tenth and all of the domain): 64^2, 10 snapshots 12 / 12 and 12, 150 snapshots
// 14 / 14 and 20; 300^2, 10 snapshots (0.9 M) 12 / 12 and 14; 180^2, 41 snapshots
// (1.3 M) 14 / 13 and 14, 720^2 adjoint 20 / 13 and 15.
constexpr size_t kFullProducts = 1 << 20;

template <typename R, typename S>
int flag_launch(const FlagParams<R, S> &p, cudaStream_t st) {
    const size_t n = (size_t)p.nx * p.ny;
    cudaError_t e = cudaMemsetAsync(p.count, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return swadj_host::cuda_check(e, "flag count reset");
    const bool f32 = sizeof(R) == 4 && sizeof(S) == 4 && p.two_d;
    const FlagParams<float, float> &pf = *reinterpret_cast<const FlagParams<float, float> *>(&p);
    // four flags, and four values of m, a store
    const bool aligned = ((uintptr_t)p.flags & 3) == 0 && ((uintptr_t)p.maxip & 15) == 0;
    const bool prune = p.env && !p.maxip;
    if (f32 && p.same_grid && (n & 3) == 0 && aligned) {
        const size_t blocks = ((n >> 2) + 255) / 256;
        static int per_sm[2] = {0, 0};
        if (prune)
            flag_kernel_f32x4<true>
                <<<persistent_blocks(flag_kernel_f32x4<true>, per_sm[1], blocks), 256, 0, st>>>(pf);
        else
            flag_kernel_f32x4<false>
                <<<persistent_blocks(flag_kernel_f32x4<false>, per_sm[0], blocks), 256, 0, st>>>(pf);
    } else if (f32 && prune && !p.same_grid && n * p.K > kFullProducts && (float)p.tol > 0.f) {
        // this pass takes m = 0 as no flag, so tol has to be above 0
        if (p.nx % 4 == 0 && aligned) launch_pruned<true>(pf, st);
        else launch_pruned<false>(pf, st);
    } else if (p.same_grid) {
        launch_full<R, S, true>(p, n, st);
    } else {
        launch_full<R, S, false>(p, n, st);
    }
    return swadj_host::cuda_check(cudaGetLastError(), "flag_kernel");
}

template int flag_launch<double, double>(const FlagParams<double, double> &, cudaStream_t);
template int flag_launch<double, float>(const FlagParams<double, float> &, cudaStream_t);
template int flag_launch<float, float>(const FlagParams<float, float> &, cudaStream_t);
template int flag_launch<float, double>(const FlagParams<float, double> &, cudaStream_t);

// |eta| > tol on wet cells, eta stored (float) or h + B (double).
template <typename R>
__global__ void __launch_bounds__(256) surface_kernel(SurfParams<R> p) {
    const int cur = p.clk->cur;
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    int f = 0;
    if (i < p.n) {
        const R a = p.q[cur][0][i], b = p.bath[i];
        R h, eta;
        if (sizeof(R) == 4) { eta = a; h = a + b; }
        else { h = a; eta = a + b; }
        f = (h > p.dry_tol && fabs(eta) > p.tol) ? 1 : 0;
        p.flags[i] = (uint8_t)f;
    }
    const int cnt = __syncthreads_count(f);
    if (threadIdx.x == 0 && cnt) atomicAdd(p.count, (unsigned long long)cnt);
}

template <typename R>
int surface_launch(const SurfParams<R> &p, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(p.count, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return swadj_host::cuda_check(e, "surface count reset");
    surface_kernel<R><<<(unsigned)((p.n + 255) / 256), 256, 0, st>>>(p);
    return swadj_host::cuda_check(cudaGetLastError(), "surface_kernel");
}

template int surface_launch<double>(const SurfParams<double> &, cudaStream_t);
template int surface_launch<float>(const SurfParams<float> &, cudaStream_t);

template <typename R>
__global__ void gauge_kernel(GaugeParams<R> p) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= p.n) return;
    const int cur = p.clk->cur;
    p.out[k] = gauge_eta<R>(p.q[cur][0], p.bath, p.nx, p.ny, p.two_d, p.x_lo, p.y_lo, p.dx,
                            p.dy, p.xy[2 * k], p.xy[2 * k + 1]);
}

template <typename R>
int gauge_launch(const GaugeParams<R> &p, cudaStream_t st) {
    if (p.n <= 0) return 0;
    gauge_kernel<R><<<(p.n + 127) / 128, 128, 0, st>>>(p);
    return swadj_host::cuda_check(cudaGetLastError(), "gauge_kernel");
}

template int gauge_launch<double>(const GaugeParams<double> &, cudaStream_t);
template int gauge_launch<float>(const GaugeParams<float> &, cudaStream_t);

}  // namespace swadj
