// hdmc_subsweep64.cuh -- the binary64 disk sub-sweep (Alg. 2), with one thread
// per active cell (large systems) or a group of G lanes per active cell
// (small ones, and crowded cells).
//
// Every decision is the exact binary64 expression (trial coordinate p + d*u,
// overlap iff dx*dx + dy*dy < sigma^2, each operation rounded), but binary64
// arithmetic is slow on this GPU (1/64 of the binary32 rate), so binary32
// estimates settle the clear cases first:
//  - in-circle test: u, v from their high words (|error| < 2^-23); cases with
//    the estimate of u^2 + v^2 within 2^-18 of 1 are decided in binary64;
//  - overlap test: positions truncated to binary32 (relative error <= 2^-23),
//    the squared distance estimated with binary32 pair arithmetic (error
//    below 3e-6 sigma^2 where it matters, r^2 < 1.3 sigma^2); a candidate counts
//    as certainly overlapping below sigma^2 (1 - 2^-15) and certainly clear above
//    sigma^2 (1 + 2^-15) (pair_bands); those in between are decided in binary64,
//    slot by slot.
// What is left on the binary64 pipe is one fused multiply-add per variate and
// one addition per trial coordinate.
#pragma once

#include "hdmc_common.cuh"
#include "hdmc_subsweep.cuh"

namespace hdmc {

constexpr float kCircleBand = 0x1p-18f;
constexpr int kDir2 = 8;   // trial directions drawn ahead per cell

// v 2^-52 on the integer pipe (v > 0; exact).
__device__ __forceinline__ double times_2m52(double v) {
    const int hi = __double2hiint(v);
    if (hi < (54 << 20)) return __dmul_rn(v, 0x1p-52);
    return __hiloint2double(hi - (52 << 20), __double2loint(v));
}

// Is the attempt that these words hold inside the unit circle (u*u + v*v < 1)?
__device__ __forceinline__ bool in_circle(const uint4 r) {
    const float uf = (float)(int)(r.x ^ 0x80000000u) * 0x1p-31f, vf = (float)(int)(r.z ^ 0x80000000u) * 0x1p-31f;
    const float e = __fmaf_rn(uf, uf, __fmul_rn(vf, vf));
    if (fabsf(e - 1.0f) > kCircleBand) return e < 1.0f;
    const double a = sym52(r.x, r.y), b = sym52(r.z, r.w);
    return __dadd_rn(__dmul_rn(a, a), __dmul_rn(b, b)) < 1.0;
}

// RN(d u) of the variate u = m 2^-52 that these words hold, d52 = d 2^-52:
// fma(d52, 2^52 + |m|, -d) with m's sign -- the product is exactly
// d + d |m| 2^-52, so one instruction of the binary64 pipe rounds d u.
__device__ __forceinline__ double displacement(double d, double d52, double words) {
    const double v = sym52_offset((uint32_t)__double2hiint(words), (uint32_t)__double2loint(words));
    const long long s = __double_as_longlong(v) & (1ll << 63);
    return __fma_rn(d52, v, __longlong_as_double(__double_as_longlong(d) ^ (s ^ (1ll << 63))));
}

__device__ __forceinline__ bool inside64(double p, double w) { return Prm<double>::ge0(p) && Prm<double>::lt(p, w); }
__device__ __forceinline__ bool hit64(const Geometry& g, double dx, double dy) {
    return __double_as_longlong(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy))) < __double_as_longlong(g.sig2);
}

// ---- one thread per active cell ------------------------------------------------------
// As the binary32 sub-sweep (hdmc_subsweep.cuh): neighbours in registers,
// directions drawn ahead, n_M fixed at compile time where NSEL > 0.
constexpr int kDirRows64 = 12;   // rows of the directions buffer: at least kDirChunk and straight_blocks(n_M)
// Blocks drawn without a loop for n_M directions (one attempt each, kept with
// probability pi/4): nearly every warp has a lane that needs them.  One block
// more: 36.1 instead of 35.8 us at 293k active cells and n_M = 4, 62.4 instead
// of 55.5 us at n_M = 8; two more: 35.7 and 61.0.
__host__ __device__ constexpr int straight_blocks(int nsel) { return nsel + nsel / 4; }

template <int ROWS, int NSEL>
__device__ __forceinline__ void subsweep_f64(const Geometry& g, double* __restrict__ cells,
                                             const SweepDraw* __restrict__ draw, int k, int bx, int by,
                                             unsigned long long* __restrict__ bpart,
                                             uint4 (*__restrict__ sdir)[32 * ROWS]) {
    static_assert(NSEL <= kDirChunk && kDirRows64 >= kDirChunk && kDirRows64 >= straight_blocks(kDirChunk), "sdir rows");
    const int nsel = NSEL > 0 ? NSEL : g.nsel;
    const int tid = threadIdx.y * 32 + threadIdx.x;
    int Q;
    uint32_t sweep;
    set_and_sweep(draw, k, Q, sweep);
    const int hx = bx * 32 + threadIdx.x, hy = by * ROWS + threadIdx.y;
    const int cx = 2 * hx + (Q & 1), cy = 2 * hy + (Q >> 1);
    const bool live = hx < g.hx && hy < g.hy && cy >= g.ylo && cy <= g.yhi;
    const Neighbourhood nbh(g, Q, hx, hy, live);

    // trial directions: the words of kept attempts (attempt a = block a)
    const uint32_t cell = (uint32_t)(cy + g.row0) * (uint32_t)g.mx + (uint32_t)cx;   // global cell number
    const uint32_t setbits = (uint32_t)Q << 24, c2 = (kDomTrial << 28) | setbits;
    const PhiloxKeys K(g.key0, g.key1);
    uint32_t blk = 0;
    int have = 0;
    auto attempt = [&](uint32_t b) {
        const uint4 r = philox_rk<false>(make_uint4(sweep, cell, c2, b), K);
        if (in_circle(r)) sdir[have++][tid] = r;
    };
    if constexpr (NSEL > 0) {
#pragma unroll
        for (int b = 0; b < straight_blocks(NSEL); ++b) attempt((uint32_t)b);
        for (uint32_t b = straight_blocks(NSEL); have < NSEL; ++b) attempt(b);
    } else {
        for (const int want = min(kDirChunk, nsel); have < want; ++blk) attempt(blk);
    }
    pdl_wait();   // what comes before depends on the draw table alone

    Cell<double> own;
#pragma unroll
    for (int j = 0; j < 4; ++j) own.x[j] = own.y[j] = kEmpty;
    double* ownp = cell_at(cells, nbh.own(g, hx, hy));
    if (live) load_cell(ownp, own);
    // slots 0, 1 of the neighbours as packed binary32 pairs in this cell's
    // frame; directions with a third disk flagged (all 24 loads ahead of the
    // first use need registers that spill: 37.8 -> 40.0 us)
    f2x qx[8], qy[8];
    uint32_t mine = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        qx[c] = pk(kFar, kFar);
        qy[c] = 0;
        if (live) {
            const double2* p = reinterpret_cast<const double2*>(cell_at(cells, nbh.index(g, c, hx, hy)));
            const double2 x01 = p[0], y01 = p[2];
            const double x2 = reinterpret_cast<const double*>(p + 1)[0];
            const float sx = (float)dir_dx(c) * g.wxf, sy = (float)dir_dy(c) * g.wyf;
            qx[c] = add2(pk(pos_or_far(x01.x), pos_or_far(x01.y)), pk(sx, sx));
            qy[c] = add2(pk(approx_pos(y01.x), approx_pos(y01.y)), pk(sy, sy));
            mine |= is_empty(x2) ? 0u : 1u << c;
        }
    }

    const int n = !is_empty(own.x[0]) + !is_empty(own.x[1]) + !is_empty(own.x[2]) + !is_empty(own.x[3]);
    const uint32_t dir23 = __reduce_or_sync(0xffffffffu, mine);
    const bool own23 = __any_sync(0xffffffffu, n >= 3);
    unsigned int n_tr = 0, n_acc = 0, n_leave = 0;
    if (n > 0) {
        if (n >= 2 && !(g.flags & kNoParticleShuffle)) {
            WordStream s(g.key0, g.key1, sweep, cell, (kDomShuffle << 28) | setbits);
            shuffle_slots(own.x, own.y, n, s.bounded(factorial(n)));
        }
        float ofx[4], ofy[4];   // binary32 truncations of the own slots
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            ofx[j] = pos_or_far(own.x[j]);
            ofy[j] = approx_pos(own.y[j]);
        }
        // slot pair (2,3) of the first flagged direction; further flagged
        // directions (rare) are read in the trial loop
        f2x fx23 = 0, fy23 = 0;
        const uint32_t more23 = dir23 & (dir23 - 1);
        auto pair23 = [&](int c, f2x& x, f2x& y) {
            const double2* p = reinterpret_cast<const double2*>(cell_at(cells, nbh.index(g, c, hx, hy)));
            const double2 x23 = p[1], y23 = p[3];
            const float sx = (float)dir_dx(c) * g.wxf, sy = (float)dir_dy(c) * g.wyf;
            x = add2(pk(pos_or_far(x23.x), pos_or_far(x23.y)), pk(sx, sx));
            y = add2(pk(approx_pos(y23.x), approx_pos(y23.y)), pk(sy, sy));
        };
        if (dir23) pair23(__ffs(dir23) - 1, fx23, fy23);
        const double d = g.d, d52 = times_2m52(d);
        const f2x lo2 = pk(g.lim, g.lim), band2 = pk(-g.bands, -g.bands);   // certainly overlapping below 0, possibly below 2 bands

        int i = 0;
        auto trial = [&](int tt, auto slots) {
            constexpr unsigned M = decltype(slots)::value;
            const uint4 w = sdir[tt][tid];
            const double tx = __dadd_rn(pick_in<M>(own.x, i), displacement(d, d52, __hiloint2double((int)w.x, (int)w.y)));
            const double ty = __dadd_rn(pick_in<M>(own.y, i), displacement(d, d52, __hiloint2double((int)w.z, (int)w.w)));
            const bool inside = inside64(tx, g.wx) && inside64(ty, g.wy);
            const float txf = approx_pos(tx), tyf = approx_pos(ty);
            const f2x tx2 = pk(txf, txf), ty2 = pk(tyf, tyf);
            uint32_t sure = 0, maybe = 0;   // sign bits: certainly / possibly overlapping
            auto own_pair = [&](int j, bool m0, bool m1) {   // slots j, j + 1 unless masked
                const f2x z = zpair(tx2, ty2, pk(ofx[j], ofx[j + 1]), pk(ofy[j], ofy[j + 1]), lo2), y = add2(z, band2);
                sure |= (m0 ? 0u : lo32(z)) | (m1 ? 0u : hi32(z));
                maybe |= (m0 ? 0u : lo32(y)) | (m1 ? 0u : hi32(y));
            };
            own_pair(0, (M & 1u) && i == 0, (M & 2u) && i == 1);
            if (own23) own_pair(2, (M & 4u) && i == 2, (M & 8u) && i == 3);
            auto pair = [&](f2x x, f2x y) {
                const f2x z = zpair(tx2, ty2, x, y, lo2), h = add2(z, band2);
                sure |= lo32(z) | hi32(z);
                maybe |= lo32(h) | hi32(h);
            };
#pragma unroll
            for (int c = 0; c < 8; ++c) pair(qx[c], qy[c]);
            if (dir23) pair(fx23, fy23);
            for (uint32_t m = more23; m; m &= m - 1) {   // warp-uniform, rarely taken
                f2x x, y;
                pair23(__ffs(m) - 1, x, y);
                pair(x, y);
            }
            bool hit = (sure >> 31) != 0;
            if (!hit && inside && (maybe >> 31)) {
                // some disk is too close to contact for the estimates: decide those in binary64
                uint32_t close = 0;   // bits 2c, 2c + 1: slots 0, 1 of direction c
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const f2x y = add2(zpair(tx2, ty2, qx[c], qy[c], lo2), band2);
                    close |= ((lo32(y) >> 31) << (2 * c)) | ((hi32(y) >> 31) << (2 * c + 1));
                }
                // Without branches on the outcome: with "occupied && hit" here and
                // n_M = 8, lanes of one warp that decided the same trial differently
                // were compiled onto paths that never met again (once in 6M
                // trials; checked_warp).  4M disks 157.1 -> 158.2 us, 1M the same.
                auto slot_hit = [&](int c, int j, bool known) {   // known: the slot holds a disk
                    const double* q = cell_at(cells, nbh.index(g, c, hx, hy)) + j;
                    return (known | !is_empty(q[0])) &
                           hit64(g, __dsub_rn(tx, __dadd_rn(q[0], (double)dir_dx(c) * g.wx)),
                                 __dsub_rn(ty, __dadd_rn(q[4], (double)dir_dy(c) * g.wy)));
                };
                for (; close; close &= close - 1) {
                    const int b = __ffs(close) - 1;
                    hit |= slot_hit(b >> 1, b & 1, true);
                }
                for (uint32_t m = dir23; m; m &= m - 1) {
                    const int c = __ffs(m) - 1;
                    hit |= slot_hit(c, 2, false) | slot_hit(c, 3, false);
                }
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (j != i && j < n) hit |= hit64(g, __dsub_rn(tx, own.x[j]), __dsub_rn(ty, own.y[j]));
            }
            const bool ok = inside && !hit;
            put_in<M>(own.x, i, tx, ok);
            put_in<M>(own.y, i, ty, ok);
            put_in<M>(ofx, i, txf, ok);
            put_in<M>(ofy, i, tyf, ok);
            n_acc += ok;
            n_leave += !inside;
            i = (i + 1 == n) ? 0 : i + 1;
        };
        if constexpr (NSEL > 0) {
            unrolled_trials(trial, std::make_integer_sequence<int, NSEL>{});
        } else {
            for (int t0 = 0; t0 < nsel; t0 += kDirChunk) {
                const int want = min(kDirChunk, nsel - t0);
                if (t0 > 0)
                    for (have = 0; have < want; ++blk) attempt(blk);
#pragma unroll 1
                for (int tt = 0; tt < want; ++tt) trial(tt, std::integral_constant<unsigned, 0xFu>{});
            }
        }
        n_tr = (unsigned)nsel;
        store_cell(ownp, own);
    }
    checked_warp(g.check);
    add_block_counters<ROWS>(n_tr, n_acc, n_leave, bpart);
}

template <int ROWS, int NSEL>
static __global__ void __launch_bounds__(32 * ROWS, 16 / ROWS)
k_subsweep_f64(const Geometry g, double* __restrict__ cells, const SweepDraw* __restrict__ draw, int k,
               unsigned long long* __restrict__ partial) {
    pdl_release();
    __shared__ uint4 sdir[kDirRows64][32 * ROWS];
    // counters of the tile that holds this block (shared: atomic adds)
    subsweep_f64<ROWS, NSEL>(g, cells, draw, k, blockIdx.x, blockIdx.y,
                             partial + 4 * ((long long)(blockIdx.y * ROWS / kCounterRows) * gridDim.x + blockIdx.x), sdir);
}

// ---- G lanes per active cell -----------------------------------------------------------
// Each lane keeps 8 / G neighbour cells in registers and tests every trial
// position against them; a vote of the group decides the trial.  The group's
// lanes draw the trial directions together, one Philox block per lane and
// round.
//
// Shared memory of one warp's cells; the cell last: the lanes of a warp read
// neighbouring banks.
template <int G> struct Warp2 {
    static constexpr int kCells = 32 / G;
    static constexpr int kRing = 16;
    static_assert(kRing >= kDir2 - 1 + G, "fewer than kDir2 directions left over, G more per round");
    double dir[kRing][2][kCells];     // kept attempts, a ring: their words, then d u
    double own[kSlots][2][kCells];    // own disks, slot order before the shuffle
};

// Updates the cells of one warp: 32 / G consecutive cells of set row hy
// starting at column hx0.
template <int G>
__device__ __forceinline__ void subsweep_lanes(const Geometry& g, double* __restrict__ cells,
                                               const SweepDraw* __restrict__ draw, int k, int hx0, int hy,
                                               unsigned long long* __restrict__ bpart, Warp2<G>& sw) {
    using W = Warp2<G>;
    constexpr int NC = 8 / G;                 // neighbour cells of a lane
    constexpr int NO = G < 4 ? 4 / G : 1;     // own slots a lane loads and stores
    constexpr unsigned kFull = 0xFFFFFFFFu;
    const int lane = threadIdx.x, grp = lane / G, L = lane % G, gb = grp * G;
    const unsigned gm = ((1u << G) - 1u) << gb;          // lanes of my group
    const unsigned below = gm & ((1u << lane) - 1u);      // those before me
    int Q;
    uint32_t sweep;
    set_and_sweep(draw, k, Q, sweep);
    const int hx = hx0 + grp;
    const int cx = 2 * hx + (Q & 1), cy = 2 * hy + (Q >> 1);
    const bool live = hx < g.hx && hy < g.hy && cy >= g.ylo && cy <= g.yhi;
    const Neighbourhood nbh(g, Q, hx, hy, live);

    // Trial directions: attempt a = block a of the trial stream, u = sym52(w0,
    // w1), v = sym52(w2, w3), kept iff u*u + v*v < 1; trial t takes the t-th
    // kept attempt.
    const uint32_t cell = (uint32_t)(cy + g.row0) * (uint32_t)g.mx + (uint32_t)cx;   // global cell number
    const uint32_t setbits = (uint32_t)Q << 24;
    const double d = g.d, d52 = times_2m52(d);
    unsigned have = 0, used = 0;   // directions kept so far, blocks used
    auto attempt = [&](bool need, uint32_t dom, uint32_t block) {
        const uint4 r = philox4x32_10(make_uint4(sweep, cell, dom, block), g.key0, g.key1);
        const bool kept = in_circle(r) && need;
        const unsigned b = __ballot_sync(kFull, kept);
        if (kept) {
            const unsigned pos = (have + __popc(b & below)) % W::kRing;
            sw.dir[pos][0][grp] = __hiloint2double((int)r.x, (int)r.y);
            sw.dir[pos][1][grp] = __hiloint2double((int)r.z, (int)r.w);
        }
        have += __popc(b & gm);
        return r.x;
    };
    // directions t0 .. t0 + want - 1, as d u
    auto fill = [&](int t0, int want) {
#pragma unroll 1
        for (;;) {
            const bool need = live && have < (unsigned)(t0 + want);
            if (!__any_sync(kFull, need)) break;
            attempt(need, (kDomTrial << 28) | setbits, used + L);
            used += need ? G : 0;
        }
        __syncwarp();
#pragma unroll 1
        for (int i = L; i < 2 * want; i += G) {
            double& w = sw.dir[(unsigned)(t0 + (i >> 1)) % W::kRing][i & 1][grp];
            w = displacement(d, d52, w);
        }
        __syncwarp();
    };
    // first round: the group's last lane draws the first word of the shuffle stream instead
    const bool shuf = L == G - 1;
    uint32_t word = attempt(live && !shuf, ((shuf ? kDomShuffle : kDomTrial) << 28) | setbits, shuf ? 0u : (uint32_t)L);
    used = G - 1;
    word = __shfl_sync(kFull, word, gb + G - 1);
    fill(0, min(kDir2, g.nsel));
    pdl_wait();   // what comes before depends on the draw table alone

    // own slots L, L + G and my neighbour cells (slots 2, 3 where used)
    double* const ownp = cell_at(cells, nbh.own(g, hx, hy));
    double own[NO][2];
#pragma unroll
    for (int r = 0; r < NO; ++r) {
        own[r][0] = own[r][1] = kEmpty;
        if (live && L + r * G < 4) {
            own[r][0] = ownp[L + r * G];
            own[r][1] = ownp[4 + L + r * G];
        }
    }
    f2x qx[NC][2], qy[NC][2];
    uint32_t has2 = 0;   // bit j: my j-th neighbour has a third disk
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        const int c = j * G + L;
        qx[j][0] = qx[j][1] = pk(kFar, kFar);
        qy[j][0] = qy[j][1] = 0;
        if (live) {
            const double2* q = reinterpret_cast<const double2*>(cell_at(cells, nbh.index(g, c, hx, hy)));
            const float sx = (float)dir_dx(c) * g.wxf, sy = (float)dir_dy(c) * g.wyf;
            const double2 x01 = q[0], x23 = q[1], y01 = q[2];
            qx[j][0] = add2(pk(pos_or_far(x01.x), pos_or_far(x01.y)), pk(sx, sx));
            qy[j][0] = add2(pk(approx_pos(y01.x), approx_pos(y01.y)), pk(sy, sy));
            if (!is_empty(x23.x)) {
                const double2 y23 = q[3];
                qx[j][1] = add2(pk(approx_pos(x23.x), pos_or_far(x23.y)), pk(sx, sx));
                qy[j][1] = add2(pk(approx_pos(y23.x), approx_pos(y23.y)), pk(sy, sy));
                has2 |= 1u << j;
            }
        }
    }

    // own cell
    int n = 0;
#pragma unroll
    for (int r = 0; r < NO; ++r) {
        n += __popc(__ballot_sync(kFull, !is_empty(own[r][0])) & gm);
        if (L + r * G < 4) {
            sw.own[L + r * G][0][grp] = own[r][0];
            sw.own[L + r * G][1][grp] = own[r][1];
        }
    }
    __syncwarp();
    // shuffle (Alg. 1): slot j of the shuffled cell is old slot (perm >> 4j) & 3
    unsigned perm = 0x3210u;
    if (n >= 2 && !(g.flags & kNoParticleShuffle)) {
        const uint32_t range = factorial(n);
        const unsigned long long m = (unsigned long long)word * range;   // 32-bit Lemire draw in [0, n!)
        uint32_t kk = (uint32_t)(m >> 32);
        if ((uint32_t)m < range) {   // as good as never: the stream from its start
            WordStream s(g.key0, g.key1, sweep, cell, (kDomShuffle << 28) | setbits);
            kk = s.bounded(range);
        }
        auto swap = [&](unsigned j, unsigned r) {
            const unsigned x = ((perm >> (4 * j)) ^ (perm >> (4 * r))) & 3u;   // 0 when j == r
            perm ^= (x << (4 * j)) ^ (x << (4 * r));
        };
        if (n >= 4) {
            swap(3u, kk & 3u);
            kk >>= 2;
        }
        if (n >= 3) {   // kk < 6
            swap(2u, kk >= 3u ? kk - 3u : kk);
            kk = kk >= 3u ? 1u : 0u;
        }
        swap(1u, kk & 1u);
    }
    uint32_t any23 = 0;   // warp-uniform: j-th neighbours with a third disk in some lane
    if (NC == 1) any23 = __any_sync(kFull, has2) ? 1u : 0u;
    else any23 = __reduce_or_sync(kFull, has2);
    const bool crowd = __any_sync(kFull, n >= 2), crowdG = G < kSlots && __any_sync(kFull, n > G);

    // g.lim and g.bands; with two lanes a cell made from sigma^2 here (17.15 us a
    // sub-sweep of 73,720 crowded cells, read from the parameters 17.30; with eight
    // lanes and 16,500 cells 5.32 and 5.24)
    const float bands = G == 2 ? fmaxf(g.sig2f, kBandFloor) * 0x1p-14f : g.bands;
    const float lim = G == 2 ? 0.5f * bands - g.sig2f : g.lim;
    const f2x lo2 = pk(lim, lim), band2 = pk(-bands, -bands);   // certainly overlapping below 0, possibly below 2 bands
    unsigned n_ac = 0, n_lf = 0;
    int i = 0, cur = (int)(perm & 3u);
    double px = sw.own[cur][0][grp], py = sw.own[cur][1][grp];   // disk `cur` before its trial
#pragma unroll 1
    for (int t = 0; t < g.nsel; ++t) {
        if (t > 0 && t % kDir2 == 0) fill(t, min(kDir2, g.nsel - t));
        // the next trial's disk, read ahead (another one than this trial's unless it is alone)
        i = i + 1 >= n ? 0 : i + 1;
        const int next = (int)((perm >> (4 * i)) & 3u);
        const double nx = sw.own[next][0][grp], ny = sw.own[next][1][grp];
        const double tx = __dadd_rn(px, sw.dir[(unsigned)t % W::kRing][0][grp]);
        const double ty = __dadd_rn(py, sw.dir[(unsigned)t % W::kRing][1][grp]);
        const bool inside = inside64(tx, g.wx) && inside64(ty, g.wy);
        const float txf = approx_pos(tx), tyf = approx_pos(ty);
        const f2x tx2 = pk(txf, txf), ty2 = pk(tyf, tyf);
        uint32_t sure = 0, maybe = 0;   // sign bits: certainly / possibly overlapping
#pragma unroll
        for (int j = 0; j < NC; ++j) {
            const f2x z = zpair(tx2, ty2, qx[j][0], qy[j][0], lo2), y = add2(z, band2);
            sure |= lo32(z) | hi32(z);
            maybe |= lo32(y) | hi32(y);
            if (any23 & (1u << j)) {
                const f2x z3 = zpair(tx2, ty2, qx[j][1], qy[j][1], lo2), y3 = add2(z3, band2);
                sure |= lo32(z3) | hi32(z3);
                maybe |= lo32(y3) | hi32(y3);
            }
        }
        bool hit = (sure >> 31) != 0;
        if (crowd) {   // the other disks of the cell
            auto own_hit = [&](int j) {
                const double ox = sw.own[j][0][grp], oy = sw.own[j][1][grp];
                const float ex = __fsub_rn(txf, approx_pos(ox)), ey = __fsub_rn(tyf, approx_pos(oy));
                const float z = __fmaf_rn(ex, ex, __fmaf_rn(ey, ey, lim));
                if (z < 0.f || z >= bands) return z < 0.f;
                return hit64(g, __dsub_rn(tx, ox), __dsub_rn(ty, oy));
            };
            if (L < n && L != cur) hit |= own_hit(L);
            if (crowdG)
                for (int j = L + G; j < n; j += G)
                    if (j != cur) hit |= own_hit(j);
        }
        if (!hit && inside && (maybe >> 31)) {
            // some slot is too close to contact for the estimates: decide those in binary64
            unsigned close = 0;   // bits 4j + s: slot s of my j-th neighbour
#pragma unroll
            for (int j = 0; j < NC; ++j)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const f2x y = add2(zpair(tx2, ty2, qx[j][h], qy[j][h], lo2), band2);
                    close |= ((lo32(y) >> 31) << (4 * j + 2 * h)) | ((hi32(y) >> 31) << (4 * j + 2 * h + 1));
                }
            while (close) {
                const int b = __ffs(close) - 1;
                close &= close - 1u;
                const int c = (b >> 2) * G + L;
                const double* q = cell_at(cells, nbh.index(g, c, hx, hy)) + (b & 3);
                hit |= hit64(g, __dsub_rn(tx, __dadd_rn(q[0], (double)dir_dx(c) * g.wx)),
                             __dsub_rn(ty, __dadd_rn(q[4], (double)dir_dy(c) * g.wy)));
            }
        }
        checked_warp(g.check);
        const bool overlap = (__ballot_sync(kFull, hit) & gm) != 0;
        const bool ok = n > 0 && inside && !overlap;
        if (ok && L == 0) {
            sw.own[cur][0][grp] = tx;
            sw.own[cur][1][grp] = ty;
        }
        n_ac += ok;
        n_lf += !inside;
        px = n > 1 ? nx : (ok ? tx : px);
        py = n > 1 ? ny : (ok ? ty : py);
        cur = next;
        __syncwarp();
    }
    // the shuffled slots back; unused slots keep their sentinels
#pragma unroll
    for (int r = 0; r < NO; ++r) {
        const int j = L + r * G;
        if (j < n) {
            const unsigned o = (perm >> (4 * j)) & 3u;
            ownp[j] = sw.own[o][0][grp];
            ownp[4 + j] = sw.own[o][1][grp];
        }
    }
    checked_warp(g.check);
    const bool count = L == 0 && n > 0;
    add_block_counters<1>(count ? (unsigned)g.nsel : 0u, count ? n_ac : 0u, count ? n_lf : 0u, bpart);
}

// One warp per 32 / G cells of a set row, four rows per block (one counter
// tile high).
template <int G>
static __global__ void __launch_bounds__(32 * kCounterRows, 5)
k_subsweep_lanes(const Geometry g, double* __restrict__ cells, const SweepDraw* __restrict__ draw, int k, int tiles,
                 unsigned long long* __restrict__ partial) {
    pdl_release();
    __shared__ Warp2<G> sw[kCounterRows];
    const int hx0 = (int)blockIdx.x * (32 / G), hy = (int)blockIdx.y * kCounterRows + (int)threadIdx.y;
    // counters of the tile (32 columns x kCounterRows rows, `tiles` in a row) that holds these cells
    subsweep_lanes<G>(g, cells, draw, k, hx0, hy, partial + 4 * ((long long)blockIdx.y * tiles + hx0 / 32), sw[threadIdx.y]);
}

template <int G>
inline void launch_lanes(const LaunchCtx& c, void* cells, const SweepDraw* draw, int k) {
    const int per = 32 / G;
    launch_on(c, k_subsweep_lanes<G>,
              dim3((unsigned)((c.g.hx + per - 1) / per), (unsigned)((c.g.hy + kCounterRows - 1) / kCounterRows)),
              dim3(32, kCounterRows), c.g, reinterpret_cast<double*>(cells), draw, k, (c.g.hx + 31) / 32, c.partial);
}

}  // namespace hdmc
