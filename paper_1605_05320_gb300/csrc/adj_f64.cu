// adj_f64.cu -- FP64 adjoint-step instantiations, compiled without
// floating-point contraction (-fmad=false); expressions are evaluated in
// the same order as the FP64 reference solver, so the rounding matches it.
#include "adj_sweeps64.cuh"

namespace swadj {

template <typename R, bool TWO_D, int TX, int TY>
static int launch_adj(const AdjParams<R> &p, cudaStream_t st) {
    dim3 grid((p.nx + TX - 1) / TX, TWO_D ? (p.ny + TY - 1) / TY : 1);
    // Measured, us per step in 1D, plain / chained: 8000 cells 16.1 / 13.4, 85000
    // (665 blocks) 38 / 33, 90000 (704) 37 / 59, 150000 (1172) 55 / 58, 160000 59 / 59
    static int wave = 0;
    return swadj_host::cuda_check(
        swadj_host::launch_spread(adj_step_kernel<R, TWO_D, TX, TY>, wave, 7, grid,
                                  dim3(TX, TY), 0, st, p),
        "adj_step_kernel<double>");
}

static int sm_count() {
    static int sms = 0;
    if (sms == 0) {
        int dev = 0, n = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        sms = n > 0 ? n : 1;
    }
    return sms;
}

// A 2D step runs as sweep passes, except on grids of few tiles (one wave of
// the tiled kernel), where nothing but one step's latency counts.
// Measured, us per step, tiles / sweeps: 64^2 28.9 / 37.1 and 160 x 120 29.0 /
// 37.2 when a quotient took FP64 operations; 200^2 56 / 37, 256 x 200 61 / 41
// (late in the solve).
bool adj_f64_sweeps(int nx, int ny) {
    return (long long)((nx + 31) / 32) * ((ny + 3) / 4) > sm_count();
}

// Cells per segment of a pass over `lines` lines of n cells.  A warp's FP64
// operations are about 52 per cell and 105 for the ends of its segment; the
// FP64 units (one per scheduler, 4 per SM) finish within about half a unit of
// one another, and about half of an adjoint's edges are still.
static int adj_segment(int lines, int n) {
    const double groups = (lines + 31) / 32, schedulers = 4.0 * sm_count();
    int best = n;
    double best_cost = 1e300;
    for (int seg = 2; seg <= 8; seg++) {
        const double rounds = groups * ((n + seg - 1) / seg) / schedulers;
        const double cost = (rounds > 1.0 ? 0.5 * rounds + 0.5 : 1.0) * (52.0 * seg + 105.0);
        if (cost < best_cost) { best_cost = cost; best = seg; }
        if (seg >= n) break;
    }
    return best;
}

template <bool XPASS>
static int launch_pass(const AdjParams<double> &p, cudaStream_t st) {
    const int lines = XPASS ? p.ny : p.nx, n = XPASS ? p.nx : p.ny;
    const int seg = adj_segment(lines, n);
    const int units = ((lines + 31) / 32) * ((n + seg - 1) / seg);
    if (p.order == 2)
        a64::adj_f64_sweep<XPASS, 2><<<units, a64::kThreads, 0, st>>>(p, seg);
    else
        a64::adj_f64_sweep<XPASS, 1><<<units, a64::kThreads, 0, st>>>(p, seg);
    return swadj_host::cuda_check(cudaGetLastError(), "adj_f64_sweep");
}

template <>
int adj_launch_step<double>(const AdjParams<double> &p, cudaStream_t st) {
    if (p.two_d && adj_f64_sweeps(p.nx, p.ny)) {   // y-pass src -> dst, x-pass dst -> src
        const int rc = launch_pass<false>(p, st);
        return rc ? rc : launch_pass<true>(p, st);
    }
    if (p.two_d) return launch_adj<double, true, 32, 4>(p, st);
    return launch_adj<double, false, 128, 1>(p, st);
}

}  // namespace swadj
