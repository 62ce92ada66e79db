// fwd_f64.cu -- FP64 forward-step instantiations.  This translation unit is
// compiled without floating-point contraction (-fmad=false) and the kernels
// evaluate every expression in the same order as the FP64 reference solver,
// so the FP64 path rounds exactly like it.  In (h, hu) form one ulp of a
// 4000 m depth (4.5e-13 m) already moves the momentum by ~1e-11 per step
// through g*hhat*(eta_R - eta_L); matching rounding is what keeps the FP64
// path within 1e-12 of the reference after thousands of steps.
#include "ctu_kernels.cuh"
#include "fwd_sweeps64.cuh"

namespace swadj {

template <bool WD>
static int launch_tiles(FwdParams<double> p, cudaStream_t st) {
    dim3 grid((p.nx + 31) / 32, (p.ny + 3) / 4);
    p.nblocks = (int)(grid.x * grid.y);
    return swadj_host::cuda_check(
        launch_chained(fwd_step_kernel<double, false, true, 32, 4, WD>, grid, dim3(32, 4), 0, st,
                       p),
        "fwd_step_kernel<double>");
}

// Cells per segment of a pass over `lines` lines of n cells.  A warp's FP64
// operations are about 98 per cell and 187 for the ends of its segment; the
// FP64 units (one per scheduler, 4 per SM) finish within about half a unit of
// one another, and part of a running grid is usually still.  Segments of 2 /
// 6 / 14 / 32 cells on 512^2 took 271 / 214 / 262 / 536 us per step (the rule
// takes 7 and 6: 213), on 2048^2 3164 / 2213 / 1994 / 2164 (14: 2006), when a
// cell took 147 operations and its ends 280, in the same proportion.
static int f64_segment(int lines, int n, int sms) {
    const double groups = (lines + 31) / 32, schedulers = 4.0 * sms;
    int best = n;
    double best_cost = 1e300;
    for (int seg = 2; seg < 130; seg++) {
        const double rounds = groups * ((n + seg - 1) / seg) / schedulers;
        const double cost = (rounds > 1.0 ? 0.75 * rounds + 0.5 : 1.2) * (98.0 * seg + 187.0);
        if (cost < best_cost) { best_cost = cost; best = seg; }
        if (seg >= n) break;
    }
    return best;
}

template <bool YPASS, bool WD>
static int launch_sweep(const FwdParams<double> &p, int sms, cudaStream_t st) {
    const int lines = YPASS ? p.nx : p.ny, n = YPASS ? p.ny : p.nx;
    int seg = f64_segment(lines, n, sms);
    const int units = ((lines + 31) / 32) * ((n + seg - 1) / seg);
    const int wpb = s64::kThreads / 32;
    int blocks = (units + wpb - 1) / wpb;
    if (blocks > 2 * sms) blocks = 2 * sms;
    if (p.order == 2)
        s64::fwd_f64_sweep<YPASS, WD, 2><<<blocks, s64::kThreads, 0, st>>>(p, seg, units);
    else
        s64::fwd_f64_sweep<YPASS, WD, 1><<<blocks, s64::kThreads, 0, st>>>(p, seg, units);
    return swadj_host::cuda_check(cudaGetLastError(), "fwd_f64_sweep");
}

// A 2D step runs as sweep passes, except on grids of a few long rows: there
// the x-pass has fewer lines than a warp has lanes and its segments grow, while
// the tiled kernel still takes one wave.
// Measured, us per step with waves everywhere, tiles / sweeps: 1000 x 4 69 / 63
// (segments of 2 cells), 2000 x 4 69 / 79 (4 cells), 4096 x 4 68 / 88 (7 cells;
// wet/dry 137 / 161), 4096 x 8 (two waves of tiles) 107 / 89.
template <bool WD>
static int launch_sweeps(const FwdParams<double> &p, cudaStream_t st) {
    static int sms = 0;
    if (sms == 0) {
        int dev = 0, n = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        sms = n > 0 ? n : 1;
    }
    if (fwd_step_blocks<double>(p) <= sms && f64_segment(p.ny, p.nx, sms) > 3)
        return launch_tiles<WD>(p, st);
    const int rc = launch_sweep<false, WD>(p, sms, st);
    return rc ? rc : launch_sweep<true, WD>(p, sms, st);
}

template <bool WD>
static int launch_line(const FwdParams<double> &p, cudaStream_t st) {
    // at most kInitBlocks blocks (the reduction slots every grid has)
    const int units = (p.nx + s64::kLineOut - 1) / s64::kLineOut;
    const int blocks = units < kInitBlocks ? units : kInitBlocks;
    auto kernel = p.order == 2 ? s64::fwd_f64_line<WD, 2> : s64::fwd_f64_line<WD, 1>;
    return swadj_host::cuda_check(launch_chained(kernel, blocks, 32, 0, st, p), "fwd_f64_line");
}

template <>
int fwd_launch_step<double>(const FwdParams<double> &p, cudaStream_t st) {
    if (p.two_d && p.keep_input) return launch_tiles<false>(p, st);
    if (p.two_d) return launch_sweeps<false>(p, st);
    return launch_line<false>(p, st);
}

template <>
int fwd_step_blocks<double>(const FwdParams<double> &p) {
    if (p.two_d) return ((p.nx + 31) / 32) * ((p.ny + 3) / 4);
    return (p.nx + 127) / 128;
}

template <>
int fwd_launch_wd<double>(const FwdParams<double> &p, cudaStream_t st) {
    if (p.two_d) return launch_sweeps<true>(p, st);
    return launch_line<true>(p, st);
}

template <>
int fwd_wd_blocks<double>(const FwdParams<double> &p) {
    return fwd_step_blocks<double>(p);
}

template <>
int fwd_launch_ctu<double>(const FwdParams<double> &p, cudaStream_t st) {
    return ctu_launch<double, 16, 8>(p, st, "fwd_ctu_kernel<double>");
}

template <>
int fwd_ctu_blocks<double>(const FwdParams<double> &p) {
    return ctu_blocks<16, 8>(p.nx, p.ny);
}

template <>
int fwd_launch_clock_init<double>(const FwdParams<double> &p, double t0, const StateSrc *src,
                                  cudaStream_t st) {
    const size_t n = (size_t)p.nx * p.ny;
    int blocks = (int)((n + 255) / 256);
    if (blocks > kInitBlocks) blocks = kInitBlocks;
    if (src)
        clock_init_kernel<double, false, true><<<blocks, 256, 0, st>>>(p, t0, *src);
    else
        clock_init_kernel<double, false, false><<<blocks, 256, 0, st>>>(p, t0, StateSrc{});
    return swadj_host::cuda_check(cudaGetLastError(), "clock_init_kernel<double>");
}

}  // namespace swadj
