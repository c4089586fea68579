// Binary64 cell-local coordinates (HDMC_FP64).
#include "hdmc_export.cuh"
#include "hdmc_kernels.cuh"

namespace hdmc {
constexpr long long kLaneCells = 32768;   // active cells above which one thread per cell is faster

// Lanes per cell: few active cells leave the chip idle and the chain of one
// cell update binds, so its work is spread over a group of lanes; with many
// the instructions bind, of which one thread per cell needs fewest.  Crowded
// cells (most directions have a third disk) keep two lanes, which hold all
// slots in registers.  us per sub-sweep in-step with 8 / 4 / 2 lanes and one
// thread, n_M = 4, then 8:
//       270 active cells    3.14 / 3.37 / 4.35 / 4.98       4.18 / 4.48 / 6.04 / 6.95
//     9,064                 5.18 / 5.15 / 6.45 / 7.03       7.43 / 7.25 / 8.90 / 10.1
//    12,138                 5.18 / 5.30 / 7.03 / 6.96       7.45 / 7.32 / 9.66 / 10.0
//    18,270                 7.84 / 5.31 / 6.97 / 8.74       11.3 / 7.40 / 9.65 / 12.1
//    28,574                 10.3 / 8.55 / 7.16 / 8.92       15.5 / 12.0 / 9.96 / 12.5
//    34,228                 11.8 / 9.29 / 7.29 / 7.24       17.6 / 13.0 / 10.1 / 10.0
//    64,428                 19.6 / 14.4 / 13.5 / 9.35       29.9 / 20.6 / 18.9 / 13.4
//   293,328                 80.3 / 56.4 / 44.4 / 35.7        122 / 83.8 / 65.6 / 55.2
//   crowded, 9,360          5.71 / 5.65 / 8.41 / 19.8       8.10 / 7.97 / 12.3 / 30.5
//   crowded, 22,680         9.22 / 5.93 / 8.81 / 21.9       13.2 / 8.32 / 12.8 / 33.9
//   crowded, 325,503         102 / 71.4 / 59.8 / 91.5        153 /  106 / 92.1 / 173
// (One thread per cell with the draws in the trial loop and the loads first took
// 8.0 at 270, 15.5 at 18,270, 46 at 287,000; crowded 16.2 at 2,340, 90 at 325,000.)
void launch_subsweep_f64(const LaunchCtx& c, void* cells, const SweepDraw* draw, int k) {
    if (c.g.cq <= 12288) return launch_lanes<8>(c, cells, draw, k);
    if (c.g.cq <= 24576) return launch_lanes<4>(c, cells, draw, k);
    if (c.g.cq <= kLaneCells || c.g.dense) return launch_lanes<2>(c, cells, draw, k);
    double* a = reinterpret_cast<double*>(cells);
    const dim3 grid((unsigned)((c.g.hx + 31) / 32), (unsigned)((c.g.hy + 1) / 2)), block(32, 2);
    if (c.g.nsel == 4) launch_on(c, k_subsweep_f64<2, 4>, grid, block, c.g, a, draw, k, c.partial);
    else if (c.g.nsel == 8) launch_on(c, k_subsweep_f64<2, 8>, grid, block, c.g, a, draw, k, c.partial);
    else launch_on(c, k_subsweep_f64<2, 0>, grid, block, c.g, a, draw, k, c.partial);
}
void launch_shift_f64(const LaunchCtx& c, const void* src, void* dst, const SweepDraw* draw) {
    launch_shift_t<double>(c, src, dst, draw);
}
void launch_hist_f64(const LaunchCtx& c, const void* cells) { launch_hist_t<double>(c, cells); }
void launch_psi6_f64(const LaunchCtx& c, const void* cells, double rc2, double* psi, double* partial, double* out) {
    launch_psi6_t<double>(c, cells, rc2, psi, partial, out);
}
void launch_export_f64(const LaunchCtx& c, const void* cells, const ExportCtx& x, unsigned* counts, double* xy, int32_t* cell) {
    launch_export_t<double>(c, cells, x, counts, xy, cell);
}
void launch_check_f64(const LaunchCtx& c, const void* cells, unsigned long long* out) {
    launch_check_t<double>(c, cells, out);
}

// Two lanes per cell for few active cells over all replicas or crowded cells,
// one thread per cell for many, as in a single system.  ms per 64 sweeps at n_M =
// 4, two lanes / one thread (one thread with the loads before the draws, the form
// before the lanes): 18,144 active cells 1.95 / 2.64 (3.46), 27,216 2.18 / 2.78
// (3.65), 36,288 3.65 / 3.00 (4.08), 72,576 5.75 / 5.15 (6.50), 1.35M 82.8 / 62.9
// (78.9); n_M = 8 2.66 / 3.57 (4.63), 2.97 / 3.71, 5.03 / 4.02, 8.02 / 7.07, 114.6
// / 89.0 (107.3); crowded, 147,000 active cells 11.7 / 15.0 (16.0).
void launch_subsweep_f64_batch(const BatchCtx& c, void* arena, const SweepDraw* draws, int j, int k) {
    auto run = [&](auto kernel, int warps) {
        launch_on(c, kernel, dim3(c.sub_blocks), dim3(32, warps), c.reps, c.sub_map, reinterpret_cast<double*>(arena), draws,
                  c.R, j, k, c.partial);
    };
    if (c.dense || (long long)c.sub_blocks * 128 <= kLaneCells) return run(k_subsweep_lanes_batch<2>, 8);
    if (c.nsel == 4) return run(k_subsweep_f64_batch<4>, 4);
    if (c.nsel == 8) return run(k_subsweep_f64_batch<8>, 4);
    run(k_subsweep_f64_batch<0>, 4);
}
}  // namespace hdmc
