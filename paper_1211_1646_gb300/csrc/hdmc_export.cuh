// hdmc_export.cuh -- global coordinates of a state in canonical (cell, slot)
// order, put together on the device: the disks or spheres of every block of
// canonical cells are counted, the counts are summed in front of each block,
// and each block writes its coordinates in order (up to kExportB blocks add the
// counts in front of them up themselves).  What crosses to the host is
// the coordinates alone (16 or 24 bytes a particle) instead of the padded
// cells, and the host does no arithmetic.  Binary32, whole call: 1M disks 33.2
// -> 0.67 ms, 1M spheres 35.5 -> 0.86 ms (the loops over padded cells on one
// host core bound it); 1024 disks 0.06 -> 0.07 ms (three launches and a wait).
#pragma once

#include "hdmc_common.cuh"

namespace hdmc {

// Exclusive prefix sum of v over a block of kExportB threads; total of the block.
__device__ __forceinline__ unsigned block_prefix(unsigned v, unsigned& total) {
    __shared__ unsigned warp_sum[kExportB / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned u = __shfl_up_sync(0xffffffffu, incl, o);
        incl += lane >= o ? u : 0u;
    }
    __syncthreads();   // the sums of an earlier call have been read
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    unsigned before = 0;
    total = 0;
#pragma unroll
    for (int w = 0; w < kExportB / 32; ++w) {
        before += w < warp ? warp_sum[w] : 0u;
        total += warp_sum[w];
    }
    return before + incl - v;
}

// counts[b] -> sum of counts[0..b), counts[nb] = the grand total (one block).
static __global__ void __launch_bounds__(kExportB) k_export_scan(unsigned* __restrict__ counts, unsigned nb) {
    unsigned carry = 0;
    for (unsigned b0 = 0; b0 < nb; b0 += kExportB) {
        const unsigned b = b0 + threadIdx.x;
        const unsigned v = b < nb ? counts[b] : 0u;
        unsigned total;
        const unsigned before = block_prefix(v, total);
        if (b < nb) counts[b] = carry + before;
        carry += total;
    }
    if (threadIdx.x == 0) counts[nb] = carry;
}

// O + (c w + x) wrapped into [0, L), each binary64 operation rounded.
__device__ __forceinline__ double global_coordinate(double origin, int c, double w, double x, double L) {
    const double v = __dadd_rn(origin, __dadd_rn(__dmul_rn((double)c, w), x));
    return __dsub_rn(v, __dmul_rn(L, floor(__ddiv_rn(v, L))));
}

// Canonical cell c of the thread: its position, its cell in storage, its disks.
template <typename T>
__device__ __forceinline__ unsigned export_cell(const Geometry& g, const T* __restrict__ cells, long long c, int& cx, int& cy,
                                                const T*& p) {
    if (c >= g.C) return 0u;
    cy = (int)((unsigned)c / (unsigned)g.mx);
    cx = (int)((unsigned)c - (unsigned)cy * (unsigned)g.mx);
    p = cells + 8 * storage_index(g, cx, cy);
    unsigned n = 0;
#pragma unroll
    for (int j = 0; j < kSlots; ++j) n = is_empty(__ldg(p + j)) ? n : (unsigned)j + 1u;
    return n;
}

template <typename T>
__global__ void __launch_bounds__(kExportB) k_export_count(const Geometry g, const T* __restrict__ cells,
                                                           unsigned* __restrict__ counts) {
    int cx, cy;
    const T* p;
    unsigned total;
    block_prefix(export_cell(g, cells, (long long)blockIdx.x * kExportB + threadIdx.x, cx, cy, p), total);
    if (threadIdx.x == 0) counts[blockIdx.x] = total;
}

template <typename T>
__global__ void __launch_bounds__(kExportB) k_export(const Geometry g, const T* __restrict__ cells,
                                                     unsigned* counts, const ExportCtx x, const DevState* __restrict__ st, double* __restrict__ xy,
                                                     int32_t* __restrict__ cell) {
    int cx, cy;
    const T* q;
    unsigned total;
    const long long c = (long long)blockIdx.x * kExportB + threadIdx.x;
    const unsigned n = export_cell(g, cells, c, cx, cy, q);
    unsigned before;
    if (gridDim.x <= kExportB) {   // no k_export_scan
        block_prefix(threadIdx.x < blockIdx.x ? counts[threadIdx.x] : 0u, before);
    } else {
        before = counts[blockIdx.x];
    }
    unsigned p = before + block_prefix(n, total);
    if (gridDim.x <= kExportB && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) counts[gridDim.x] = before + total;
    for (unsigned j = 0; j < n && p < x.limit; ++j, ++p) {
        if (p < x.first) continue;
        const size_t o = p - x.first;
        xy[2 * o] = global_coordinate(st->origin[0], cx, x.wx, (double)__ldg(q + j), x.Lx);
        xy[2 * o + 1] = global_coordinate(st->origin[1], cy, x.wy, (double)__ldg(q + 4 + j), x.Ly);
        if (cell) cell[o] = (int32_t)c;
    }
}

template <typename T>
inline void launch_export_t(const LaunchCtx& c, const void* cells, const ExportCtx& x, unsigned* counts, double* xy, int32_t* cell) {
    const unsigned nb = export_blocks(c.g);
    const T* a = reinterpret_cast<const T*>(cells);
    k_export_count<T><<<nb, kExportB, 0, c.stream>>>(c.g, a, counts);
    if (nb > (unsigned)kExportB) k_export_scan<<<1, kExportB, 0, c.stream>>>(counts, nb);
    k_export<T><<<nb, kExportB, 0, c.stream>>>(c.g, a, counts, x, c.st, xy, cell);
}

}  // namespace hdmc
