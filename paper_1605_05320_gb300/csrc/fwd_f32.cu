// fwd_f32.cu -- FP32 perturbation-form forward step (Eq. swe, Sec. 5; Roe-type
// f-wave solver per edge, Sec. 6) for GB300.
//
// Storage: eta = h + B, hu, hv and hbar = -B in float.  Depth h = eta + hbar
// enters only wave speeds and Roe averages; the surface jump that drives the
// bathymetry-balanced momentum flux is taken from eta directly, so decimetre
// waves on 4000 m are resolved to float precision of eta, not of h.
//
// 2D grids run the warp strips of strips.cuh (per edge the arithmetic of
// fwd_pair.cuh); 1D grids run a one-thread-per-cell kernel with the same
// arithmetic.  The CFL maximum
// is reduced in float (max is exact); the last block to finish turns it into
// the next time step in double.
#include "ctu_strips.cuh"
#include "strips.cuh"

namespace swadj {
namespace f32 {


// 2D grids: persistent warps take work units from the clock's counter, one
// unit a strip of 28 output columns by `rows` rows, in row-major order, then
// the gauges of a recorded step, 32 a unit.
// Where the ocean is at rest a unit costs little (strips.cuh), so units are
// short and taken as warps free up: the active part of the domain spreads
// over every SM instead of over the few warps whose strips it crosses.
// ORD: the order of the scheme (1 or 2), fixed at compile time; CTU: the
// unsplit update with transverse waves (a window at rest stays so under it
// too, with the same CFL terms).
template <int ORD, bool CTU>
__global__ void __launch_bounds__(strip::kThreads, 4)
    fwd_f32_strips(FwdParams<float> p, int rows, int nunits) {
    __shared__ float s_nu[2];
    __shared__ int s_cur, s_run;
    __shared__ float red[strip::kThreads / 32];
    __shared__ int am_last;
    __shared__ strip::Ring ring[strip::kThreads / 32];
    double t_now = 0.0, dt = 0.0;
    if (!fwave::begin_step(p.clk, p.t_end, (double)p.dx, (double)p.dy, s_nu, &s_cur, &s_run,
                           t_now, dt))
        return;
    const int cur = s_cur;
    // with gauge recording, the warps that first run out of strips sample the
    // state the step starts from, 32 gauges each (the strips write the other
    // buffer)
    const int ngroups = p.gauges.n > 0 ? (p.gauges.n + 31) / 32 : 0;
    const int nsx = (p.nx + strip::kOut - 1) / strip::kOut;
    strip::View v;
    v.q0 = p.q[cur][0]; v.q1 = p.q[cur][1]; v.q2 = p.q[cur][2]; v.hb = p.bath;
    v.o0 = p.q[cur ^ 1][0]; v.o1 = p.q[cur ^ 1][1]; v.o2 = p.q[cur ^ 1][2];
    v.nx = p.nx; v.ny = p.ny;
    v.rdx = 1.f / p.dx; v.rdy = 1.f / p.dy;
    v.bc = p.bc;
    float smax = 0.f;
    bool bad = false;
    const int lane = threadIdx.x & 31;
    const bool quiet = p.rest_tab && p.umap && !p.keep_rest;
    // Marks carry the unit height: those of another one (the caller may change
    // it, and a captured step keeps its own) say nothing.
    const int tag = (rows & 63) << 2;
    // the first unit by position, the others from the counter (the counter's
    // first round trip cost 1.1 us of 15.5 at 512^2)
    int next = lane == 0 ? (int)(blockIdx.x * (strip::kThreads / 32) + (threadIdx.x >> 5)) : -1;
    for (;;) {   // warp-uniform
        int u = next;
        if (lane == 0 && u < 0)
            u = (int)(gridDim.x * (strip::kThreads / 32) + atomicAdd(&p.clk->work, 1u));
        u = __shfl_sync(0xffffffffu, u, 0);
        next = -1;
        if (u >= nunits) {
            if (u >= nunits + ngroups) break;
            record_gauge_group<float>(p.gauges, p.q[cur][0], p.bath, p.nx, p.ny, 1, p.clk,
                                      u - nunits);
            continue;
        }
        const int sy = u / nsx, sx = u - sy * nsx;
        if (quiet) {
            const int own = p.umap[u];
            if (own != (tag | UNIT_ACTIVE)) {
                // still among still units: both buffers hold it at rest, and
                // only its CFL terms count (2048^2 at rest but for a small
                // source 35 us with each unit scanned and stored, 29 so;
                // 4096^2 81 and 44)
                if (own == (tag | UNIT_STILL) &&
                    still_around(p.umap, u, sx, nsx, nunits, tag | UNIT_STILL)) {
                    const int yend = (sy + 1) * rows < p.ny ? (sy + 1) * rows : p.ny;
                    for (int j = sy * rows + lane; j < yend; j += 32)
                        smax = fmaxf(smax, p.rest_tab[(size_t)sx * p.ny + j]);
                    continue;
                }
                // the scan alone decides that a unit is at rest; one that has
                // had waves keeps them (the ocean does not return exactly to
                // rest behind a wave) and is not scanned again
                if (strip::quiet_unit<true>(v, p.rest_tab, sx, sx * strip::kOut, sy * rows, rows,
                                            p.g, smax)) {
                    if (lane == 0) p.umap[u] = tag | UNIT_STILL;
                    continue;
                }
                if (lane == 0) p.umap[u] = tag | UNIT_ACTIVE;
            }
        }
        // Units with waves take every row in full: a strip loop that tests
        // rows for waves is slower, and quiet units cover the ocean at rest.
        if (CTU)
            strip::ctu_unit<ORD>(v, sx * strip::kOut, sy * rows, rows, s_nu[0], s_nu[1], p.g,
                                 ring[threadIdx.x >> 5], smax, bad);
        else
            strip::strip_unit<ORD, 2>(v, sx * strip::kOut, sy * rows, rows, s_nu[0], s_nu[1], p.g,
                                      ring[threadIdx.x >> 5], smax, bad);
    }
    // no marks but this step's units': without this, heights changed to and
    // fro would find old marks where the other height has fewer units
    if (p.umap)
        for (int k = (quiet ? nunits : 0) + blockIdx.x * strip::kThreads + threadIdx.x;
             k < p.umap_n; k += gridDim.x * strip::kThreads)
            p.umap[k] = UNIT_UNKNOWN;
    if (bad) atomicOr(p.err, ERR_UNSTABLE);
    fwave::finish_step<strip::kThreads>(p.clk, p.partial, p.nblocks, p.cfl, smax, red, &am_last,
                                        t_now, dt, cur);
    if (ngroups > 0 && threadIdx.x == 0 && am_last) *p.gauges.row += 1;
}

// 1D grids: one thread per cell, solving the four edges it needs itself
// (1D grids are small; the redundancy costs nothing that matters).
__global__ void __launch_bounds__(256) fwd_f32_1d(FwdParams<float> p) {
    __shared__ float s_nu[2];
    __shared__ int s_cur, s_run;
    __shared__ float red[8];
    __shared__ int am_last;
    double t_now = 0.0, dt = 0.0;
    if (!fwave::begin_step(p.clk, p.t_end, (double)p.dx, (double)p.dy, s_nu, &s_cur, &s_run,
                          t_now, dt))
        return;
    const int cur = s_cur;
    if (p.gauges.n > 0 && blockIdx.x == 0)   // the state this step starts from
        record_gauges<float, 256>(p.gauges, p.q[cur][0], p.bath, p.nx, p.ny, 0, t_now);
    const float nux = s_nu[0], g = p.g;
    const float *q0 = p.q[cur][0], *q1 = p.q[cur][1];
    const int i = blockIdx.x * 256 + threadIdx.x;
    float sm = 0.f;
    bool bad = false;
    if (i < p.nx) {
        fp::Cell c[5];
#pragma unroll
        for (int k = 0; k < 5; k++) {
            bool fx;
            const int ci = ghost_index(i - 2 + k, p.nx, p.bc.lo_x, p.bc.hi_x, &fx);
            const float eta = q0[ci], mu = fx ? -q1[ci] : q1[ci];
            c[k] = fp::derive(eta, fp::add(eta, p.bath[ci]), mu, 0.f);
        }
        const float gh = 0.5f * g;
        fp::Edge w[4];
#pragma unroll
        for (int k = 0; k < 4; k++) w[k] = fp::solve(gh, c[k], c[k + 1]);
        const fp::Net n0 =
            fp::net3(w[0], w[1], w[2], nux, p.order, fp::subsonic(w[1].s1, w[1].s3));
        const fp::Net n1 =
            fp::net3(w[1], w[2], w[3], nux, p.order, fp::subsonic(w[2].s1, w[2].s3));
        const float d0 = fp::mul(-nux, fp::add(n0.R0, n1.L0));
        const float ne = fp::add(c[2].eta, d0);
        const float nmu = fp::add(c[2].mn, fp::mul(-nux, fp::add(n0.R1, n1.L1)));
        p.q[cur ^ 1][0][i] = ne;
        p.q[cur ^ 1][1][i] = nmu;
        const float hn = fp::add(c[2].h, d0);
        bad = !(hn > 0.f) || !isfinite(nmu);
        sm = cfl_f32(hn, nmu, 0.f, g, 1.f / p.dx, 1.f / p.dy, 0);
    }
    if (bad) atomicOr(p.err, ERR_UNSTABLE);
    fwave::finish_step<256>(p.clk, p.partial, p.nblocks, p.cfl, sm, red, &am_last, t_now, dt,
                            cur);
}

// The rest CFL table of quiet units (strips.cuh): per strip sx and row j,
// the maximum over the strip's output columns of cfl_f32(hbar, 0, 0), the
// step's CFL term of a cell at rest, with the step's own 1/dx and 1/dy; NaN
// where a column has hbar <= 0.
__global__ void rest_cfl_table(FwdParams<float> p, float *tab) {
    const int nsx = (p.nx + strip::kOut - 1) / strip::kOut;
    const float rdx = 1.f / p.dx, rdy = 1.f / p.dy;
    const size_t n = (size_t)nsx * p.ny;
    for (size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
         k += (size_t)gridDim.x * blockDim.x) {
        const int sx = (int)(k / p.ny), j = (int)(k - (size_t)sx * p.ny);
        const int x1 = (sx + 1) * strip::kOut < p.nx ? (sx + 1) * strip::kOut : p.nx;
        float t = 0.f;
        bool ok = true;
        for (int i = sx * strip::kOut; i < x1; i++) {
            const float hb = p.bath[(size_t)j * p.nx + i];
            ok = ok && hb > 0.f;
            t = fmaxf(t, cfl_f32(hb, 0.f, 0.f, p.g, rdx, rdy, 1));
        }
        tab[k] = ok ? t : __int_as_float(0x7fc00000);
    }
}

}  // namespace f32

// Lowest height of a work unit in rows.
constexpr int kMinUnitRows = 4;

// Entries of the unit map: units of the lowest height.
int fwd_f32_unit_map_bytes(int nx, int ny) {
    return ((nx + strip::kOut - 1) / strip::kOut) * ((ny + kMinUnitRows - 1) / kMinUnitRows);
}

size_t fwd_f32_rest_table_floats(int nx, int ny) {
    return (size_t)((nx + strip::kOut - 1) / strip::kOut) * ny;
}

int fwd_f32_rest_table(const FwdParams<float> &p, float *tab, cudaStream_t st) {
    const size_t n = fwd_f32_rest_table_floats(p.nx, p.ny);
    int blocks = (int)((n + 255) / 256);
    if (blocks > 4096) blocks = 4096;
    f32::rest_cfl_table<<<blocks, 256, 0, st>>>(p, tab);
    return swadj_host::cuda_check(cudaGetLastError(), "rest_cfl_table");
}

// Persistent blocks at most (reduction slots of the grid workspace).
constexpr int kMaxStepBlocks = 4096;


// Blocks of one resident wave of the strip kernel on the current device.
template <bool CTU>
static int resident_blocks() {
    static int blocks = 0;
    if (blocks == 0) {
        int dev = 0, sms = 0, per_sm = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f32::fwd_f32_strips<2, CTU>,
                                                      strip::kThreads, 0);
        blocks = (sms > 0 ? sms : 1) * (per_sm > 0 ? per_sm : 1);
        if (blocks > kMaxStepBlocks) blocks = kMaxStepBlocks;
    }
    return blocks;
}

static int strip_units(int nx, int ny, int rows) {
    return ((nx + strip::kOut - 1) / strip::kOut) * ((ny + rows - 1) / rows);
}

// Rows of a work unit of the FP32 2D step: the requested strip height (16,
// 32 or 64), else the lowest height (at least kMinUnitRows) whose units are
// no more than k times the resident warps, for the smallest k that needs no
// more than kMaxUnitRows rows.  A unit walks its rows one after the other,
// 0.58 us each when its warp is alone on its scheduler, so a grid of fewer
// units than warps is latency-bound and takes the lowest units that still
// fill the warps; a grid of many units wants them high (each walks four
// halo rows more) and a whole number of rounds.  All heights give the same
// results.
// Measured, us per step, 32 rows / this rule (rest outside the source, waves
// everywhere): 64^2 28.7 / 12.3 both; 512^2 26.9 / 15.7 and 28.1 / 18.1; 1024^2
// 30.1 / 23.9 and 32.8 / 28.7; 1500^2 (34 rows) 33.9 / 35.4 and 53.3 / 44.4;
// 2048^2 keeps 32; 4096^2 (36 rows) 84.3 / 86.1 and 258 / 248.
constexpr int kMaxUnitRows = 36;
template <bool CTU>
static int unit_rows(const FwdParams<float> &p) {
    if (p.fwd_rows > 0) return p.fwd_rows;
    const long long warps = (long long)resident_blocks<CTU>() * (strip::kThreads / 32);
    const int nsx = (p.nx + strip::kOut - 1) / strip::kOut;
    long long k = ((long long)nsx + warps - 1) / warps;
    for (;; k++) {
        const long long bands = k * warps / nsx;
        const long long rows = (p.ny + bands - 1) / bands;
        if (rows <= kMaxUnitRows) return rows > kMinUnitRows ? (int)rows : kMinUnitRows;
    }
}

template <bool CTU>
static int launch_strips(FwdParams<float> p, cudaStream_t st) {
    const int rows = unit_rows<CTU>(p);
    const int units = strip_units(p.nx, p.ny, rows);
    constexpr int wpb = strip::kThreads / 32;
    const int blocks = (units + wpb - 1) / wpb, wave = resident_blocks<CTU>();
    p.nblocks = blocks < wave ? blocks : wave;
    return swadj_host::cuda_check(
        launch_chained(p.order == 2 ? f32::fwd_f32_strips<2, CTU> : f32::fwd_f32_strips<1, CTU>,
                       p.nblocks, strip::kThreads, 0, st, p, rows, units),
        "fwd_f32_strips");
}

template <>
int fwd_launch_step<float>(const FwdParams<float> &p0, cudaStream_t st) {
    if (p0.two_d) return launch_strips<false>(p0, st);
    FwdParams<float> p = p0;
    dim3 grid((p.nx + 255) / 256, 1);
    p.nblocks = (int)grid.x;
    return swadj_host::cuda_check(launch_chained(f32::fwd_f32_1d, grid, 256, 0, st, p),
                                  "fwd_f32_1d");
}

template <>
int fwd_step_blocks<float>(const FwdParams<float> &p) {
    // one reduction slot per block: at most one block per 4 units (of the
    // lowest height), at most kMaxStepBlocks
    if (p.two_d) {
        const int b = (strip_units(p.nx, p.ny, kMinUnitRows) + 3) / 4;
        return b < kMaxStepBlocks ? b : kMaxStepBlocks;
    }
    return (p.nx + 255) / 256;
}

// The wet/dry option runs the tiled split step (fwd_kernels.cuh) with the
// shore solver, in the perturbation form.
template <>
int fwd_launch_wd<float>(const FwdParams<float> &p0, cudaStream_t st) {
    FwdParams<float> p = p0;
    // Measured, us per step, plain / chained: 280 x 200 (450 blocks) 28.4 / 26.4, 330 x
    // 240 (660) 28.9 / 31.5, 384 x 260 (780) 31.8 / 31.4, 512 x 400 (1600) 48.9 / 47.6;
    // 1D 90000 cells (704 blocks) 18.4 / 17.0, 120000 (938) 18.6 / 20.7, 130000 20.5 / 20.2
    if (p.two_d) {
        static int wave = 0;
        dim3 grid((p.nx + 31) / 32, (p.ny + 3) / 4);
        p.nblocks = (int)(grid.x * grid.y);
        return swadj_host::cuda_check(
            swadj_host::launch_spread(fwd_step_kernel<float, true, true, 32, 4, true>, wave, 6,
                                      grid, dim3(32, 4), 0, st, p),
            "fwd_step_kernel<float, wet/dry>");
    } else {
        static int wave = 0;
        dim3 grid((p.nx + 127) / 128, 1);
        p.nblocks = (int)grid.x;
        return swadj_host::cuda_check(
            swadj_host::launch_spread(fwd_step_kernel<float, true, false, 128, 1, true>, wave, 6,
                                      grid, dim3(128, 1), 0, st, p),
            "fwd_step_kernel<float, wet/dry>");
    }
}

template <>
int fwd_wd_blocks<float>(const FwdParams<float> &p) {
    if (p.two_d) return ((p.nx + 31) / 32) * ((p.ny + 3) / 4);
    return (p.nx + 127) / 128;
}

template <>
int fwd_launch_ctu<float>(const FwdParams<float> &p, cudaStream_t st) {
    return launch_strips<true>(p, st);
}

template <>
int fwd_ctu_blocks<float>(const FwdParams<float> &p) {
    return fwd_step_blocks<float>(p);
}

template <>
int fwd_launch_clock_init<float>(const FwdParams<float> &p, double t0, const StateSrc *src,
                                 cudaStream_t st) {
    const size_t n = (size_t)p.nx * p.ny;
    int blocks = (int)((n + 255) / 256);
    if (blocks > kInitBlocks) blocks = kInitBlocks;
    if (src)
        clock_init_kernel<float, true, true><<<blocks, 256, 0, st>>>(p, t0, *src);
    else
        clock_init_kernel<float, true, false><<<blocks, 256, 0, st>>>(p, t0, StateSrc{});
    return swadj_host::cuda_check(cudaGetLastError(), "clock_init_kernel<float>");
}

}  // namespace swadj
