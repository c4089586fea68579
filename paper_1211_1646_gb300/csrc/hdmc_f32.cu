// Binary32 cell-local coordinates (HDMC_FP32_LOCAL).
#include "hdmc_export.cuh"
#include "hdmc_kernels.cuh"

namespace hdmc {
// A binary32 state of up to 64 MB stays in L2 (129 MB, with its other half)
// from one sub-sweep to the next.  Above, the loads come before the draws where
// that measured faster (us per sub-sweep in-step, draws first -> loads first):
// n_M = 4, 1.15M active cells 38.9 -> 37.3; run-time n_M = 12 117.1 -> 114.7;
// crowded, 590,000 active cells, run-time n_M = 5 35.2 -> 34.7, but crowded
// n_M = 4 25.7 -> 25.9, n_M = 8 42.4 -> 43.2, and n_M = 1 30.0 -> 30.5.  The
// other n_M have the one form at every size.
constexpr long long kAheadCells = 2000000;

void launch_subsweep_f32(const LaunchCtx& c, void* cells, const SweepDraw* draw, int k) {
    float* a = reinterpret_cast<float*>(cells);
    // blocks of two set rows of 32 cells: in-step faster than one-row blocks
    // (fewer blocks to schedule) and as fast as four-row blocks
    const dim3 grid((unsigned)((c.g.hx + 31) / 32), (unsigned)((c.g.hy + 1) / 2));
    auto run = [&](auto kernel) { launch_on(c, kernel, grid, dim3(32, 2), c.g, a, draw, k, c.partial); };
    const int nsel = c.g.nsel;
    const bool ahead = c.g.C <= kAheadCells;   // see subsweep_f32, phase 1
    if (c.g.dense) {   // cells that often hold three or four disks
        if (nsel == 4) return run(k_subsweep_f32<2, 4, true>);
        if (nsel == 8) return run(k_subsweep_f32<2, 8, true>);
        return ahead ? run(k_subsweep_f32<2, 0, true>) : run(k_subsweep_f32<2, 0, true, false>);
    }
    if (!ahead && nsel == 4) return run(k_subsweep_f32<2, 4, false, false>);
    if (!ahead && nsel == 8) return run(k_subsweep_f32<2, 8, false, false>);
    if (!ahead && nsel > 8) return run(k_subsweep_f32<2, 0, false, false>);
    // n_M fixed at compile time (directions drawn in one pass, trials
    // unrolled) up to kDirChunk; 100 sweeps of 2,585 active cells at n_M = 7 and
    // their pressure: 2.21 -> 1.70 ms
    switch (nsel) {
        case 1: return run(k_subsweep_f32<2, 1>);
        case 2: return run(k_subsweep_f32<2, 2>);
        case 3: return run(k_subsweep_f32<2, 3>);
        case 4: return run(k_subsweep_f32<2, 4>);
        case 5: return run(k_subsweep_f32<2, 5>);
        case 6: return run(k_subsweep_f32<2, 6>);
        case 7: return run(k_subsweep_f32<2, 7>);
        case 8: return run(k_subsweep_f32<2, 8>);
        default: return run(k_subsweep_f32<2, 0>);
    }
}
void launch_shift_f32(const LaunchCtx& c, const void* src, void* dst, const SweepDraw* draw) {
    launch_shift_t<float>(c, src, dst, draw);
}
void launch_hist_f32(const LaunchCtx& c, const void* cells) { launch_hist_t<float>(c, cells); }
void launch_psi6_f32(const LaunchCtx& c, const void* cells, double rc2, double* psi, double* partial, double* out) {
    launch_psi6_t<float>(c, cells, rc2, psi, partial, out);
}
unsigned psi6_blocks(const Geometry& g) {
    const dim3 grid = set_grid(g, dim3(kPsiBX, kPsiBY));
    return grid.x * grid.y * grid.z;
}
unsigned export_blocks(const Geometry& g) { return (unsigned)((g.C + kExportB - 1) / kExportB); }
void launch_export_f32(const LaunchCtx& c, const void* cells, const ExportCtx& x, unsigned* counts, double* xy, int32_t* cell) {
    launch_export_t<float>(c, cells, x, counts, xy, cell);
}
void launch_check_f32(const LaunchCtx& c, const void* cells, unsigned long long* out) {
    launch_check_t<float>(c, cells, out);
}

void launch_subsweep_f32_batch(const BatchCtx& c, void* arena, const SweepDraw* draws, int j, int k, bool track) {
    float* a = reinterpret_cast<float*>(arena);
#define HDMC_SUB_BATCH(ROWS, TRACK, DENSE, NSEL)                                                           \
    launch_on(c, k_subsweep_f32_batch<ROWS, TRACK, DENSE, NSEL>, dim3(c.sub_blocks), dim3(32, ROWS),      \
              c.reps, c.sub_map, a, draws, c.R, j, k, c.partial, c.msd)
    // crowded cells in every replica: the dense kernel; one n_M shared by
    // every replica (4 or 8): the kernel with n_M fixed (the autotuner's
    // tracking launches keep the general one)
#define HDMC_SUB_BATCH_NSEL(ROWS, DENSE)                                                                   \
    do {                                                                                                   \
        if (c.nsel == 4) HDMC_SUB_BATCH(ROWS, false, DENSE, 4);                                            \
        else if (c.nsel == 8) HDMC_SUB_BATCH(ROWS, false, DENSE, 8);                                       \
        else HDMC_SUB_BATCH(ROWS, false, DENSE, 0);                                                        \
    } while (0)
#define HDMC_SUB_BATCH_ROWS(ROWS)                                                                          \
    do {                                                                                                   \
        if (track) HDMC_SUB_BATCH(ROWS, true, false, 0);                                                   \
        else if (c.dense) HDMC_SUB_BATCH_NSEL(ROWS, true);                                                 \
        else HDMC_SUB_BATCH_NSEL(ROWS, false);                                                             \
    } while (0)
    if (c.rows == 1) HDMC_SUB_BATCH_ROWS(1);
    else if (c.rows == 2) HDMC_SUB_BATCH_ROWS(2);
    else if (c.rows == 8) HDMC_SUB_BATCH_ROWS(8);
    else HDMC_SUB_BATCH_ROWS(4);
#undef HDMC_SUB_BATCH_ROWS
#undef HDMC_SUB_BATCH_NSEL
#undef HDMC_SUB_BATCH
}

void launch_shift_batch(const BatchCtx& c, int prec, const void* src, void* dst, const SweepDraw* draws, int j) {
    const dim3 grid(c.sh_blocks), block(kShiftBX, kShiftBY);
    auto run = [&](auto kernel, auto zero) {
        using T = decltype(zero);
        launch_on(c, kernel, grid, block, c.reps, c.sh_map, static_cast<const T*>(src), static_cast<T*>(dst), draws, c.R, j,
                  c.sts);
    };
    if (prec == 1) run(k_shift_batch<float, false>, 0.0f);
    else if (shift_early<double>((long long)c.sh_blocks * (kShiftBX * kShiftBY))) run(k_shift_batch<double, true>, 0.0);
    else run(k_shift_batch<double, false>, 0.0);
}

void launch_hist_batch(const BatchCtx& c, int prec, const void* arena) {
    if (prec == 1)
        k_hist_batch<float><<<c.hi_blocks, dim3(kHistBX, kHistBY), 0, c.stream>>>(
            c.reps, c.hi_map, reinterpret_cast<const float*>(arena), c.edges2, c.hist);
    else
        k_hist_batch<double><<<c.hi_blocks, dim3(kHistBX, kHistBY), 0, c.stream>>>(
            c.reps, c.hi_map, reinterpret_cast<const double*>(arena), c.edges2, c.hist);
}
}  // namespace hdmc
