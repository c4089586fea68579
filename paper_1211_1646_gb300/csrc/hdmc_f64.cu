// Binary64 cell-local coordinates (HDMC_FP64).
#include "hdmc_export.cuh"
#include "hdmc_kernels.cuh"

namespace hdmc {
// Lanes per cell: few active cells leave the chip idle and the chain of one
// cell update binds, so its work is spread over a group of lanes; with many
// the instructions bind, of which one thread per cell needs fewest.  Crowded
// cells (most directions have a third disk) keep two lanes, which hold all
// slots in registers.  us per sub-sweep in-step at n_M = 4 with 8 / 4 / 2
// lanes and one thread (before: 8.0, 12.8, 16.2, 17.3, 20.5, 47.9; crowded
// 19.1, 43.1), the loads ahead of the draws; with the draws ahead (pdl_wait)
// the chosen forms take 3.2, 5.2, 5.3, 7.3, 14.6, 36.0; crowded 5.7, 30.3:
//       270 active cells   3.7 / 4.3 / 5.7 / 6.7
//     8,976                5.9 / 6.4 / 8.3 / 9.0
//    18,270                8.4 / 6.6 / 8.9 / 10.8
//    36,108               12.9 / 10.7 / 9.3 / 11.2
//    73,332               22.5 / 17.8 / 15.8 / 16.0
//   293,328               79.6 / 57.1 / 45.2 / 37.8
//   crowded, 9,360         6.3 / 6.9 / 10.3 / 17.9
//   crowded, 147,441      47.0 / 34.7 / 31.6 / 40.3
void launch_subsweep_f64(const LaunchCtx& c, void* cells, const SweepDraw* draw, int k) {
    if (c.g.cq <= 12288) return launch_lanes<8>(c, cells, draw, k);
    if (c.g.cq <= 24576) return launch_lanes<4>(c, cells, draw, k);
    if (c.g.cq <= 65536 || c.g.dense) return launch_lanes<2>(c, cells, draw, k);
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
constexpr long long kBatchLaneCells = 32768;
void launch_subsweep_f64_batch(const BatchCtx& c, void* arena, const SweepDraw* draws, int j, int k) {
    auto run = [&](auto kernel, int warps) {
        launch_on(c, kernel, dim3(c.sub_blocks), dim3(32, warps), c.reps, c.sub_map, reinterpret_cast<double*>(arena), draws,
                  c.R, j, k, c.partial);
    };
    if (c.dense || (long long)c.sub_blocks * 128 <= kBatchLaneCells) return run(k_subsweep_lanes_batch<2>, 8);
    if (c.nsel == 4) return run(k_subsweep_f64_batch<4>, 4);
    if (c.nsel == 8) return run(k_subsweep_f64_batch<8>, 4);
    run(k_subsweep_f64_batch<0>, 4);
}
}  // namespace hdmc
