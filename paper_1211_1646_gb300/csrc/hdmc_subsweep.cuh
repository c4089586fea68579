// hdmc_subsweep.cuh -- the binary32 sub-sweep (Alg. 2) with one thread per
// active cell (hdmc_subsweep64.cuh has the form with several lanes per cell).
//
// Every floating-point operation that decides an acceptance is written with
// an explicit round-to-nearest operation, so the result does not depend on
// compiler contraction: trial coordinate fma(d, u, p), overlap iff
// fma(dx, dx, fma(dy, dy, -sigma^2)) < 0.
#pragma once

#include "hdmc_common.cuh"

namespace hdmc {

// ---- binary32 sub-sweep: the cell updates of Alg. 1 / Alg. 2 ---------------------------
// One thread per active cell of set Q = draw->perm[k]; block 32 x ROWS over
// the set's half-resolution grid.  Phases:
//   1. draw the trial directions of the cell's stream (kept attempts staged
//      in shared memory, kDirChunk at a time).  They depend on the draw table
//      alone, so with AHEAD they come before pdl_wait: as a programmatic
//      dependent the kernel draws them while the previous kernel's last blocks
//      run.  Where the state does not fit L2 the loads may go first, the draws
//      covering their latency (launch_subsweep_f32).  us per sub-sweep in-step
//      at n_M = 4, loads first -> draws first: 270 active cells 1.84 -> 1.69, 9k
//      3.6 -> 2.6, 73k 4.05 -> 3.2, 293k 10.6 either way (n_M = 8 16.4 -> 15.8),
//      1.15M (147 MB) 37.3 -> 38.9; crowded 9k 4.0 -> 2.7.  Draws first only in
//      the blocks of the first wave: 11.0 at 293k;
//   2. load the own cell and the 8 neighbouring cells (they belong to other
//      sets and are not written by this launch);
//   3. shuffle the disks with the draw in field 0 of the stream's first block,
//      translate neighbour slot pair (0,1) into this cell's frame as packed
//      binary32 pairs, flag (warp-uniformly) the directions where some lane
//      has a third disk;
//   4. n_M trial moves, visiting the shuffled slots cyclically.
// NSEL > 0 fixes n_M at compile time (the trial loop is then unrolled).
// With TRACK, the block also adds the net squared displacement of its disks
// over the cell update (final minus start position, summed over the disks)
// to *msd: a sampling-efficiency measure used by the batch autotuner.
template <int ROWS>
__device__ __forceinline__ void draw_directions(const Geometry& g, uint32_t sweep, uint32_t cell, uint32_t c2,
                                                uint32_t F[6], uint32_t& blk, int& pnext, int want,
                                                float2 (*__restrict__ sdir)[32 * ROWS], int tid) {
    int have = 0;
    for (;;) {
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            if (p >= pnext && have < want) {
                const float u = sym21(F[2 * p]), v = sym21(F[2 * p + 1]);
                if (__fmaf_rn(u, u, __fmul_rn(v, v)) < 1.0f) {
                    sdir[have][tid] = make_float2(u, v);
                    ++have;
                }
                pnext = p + 1;
            }
        }
        if (have >= want) break;
        ++blk;
        fields21(philox4x32_10(make_uint4(sweep, cell, c2, blk), g.key0, g.key1), F);
        pnext = 0;
    }
}

// Philox4x32-10 (the library's philox4x32_10, the same function) with the
// round keys of one key computed once per thread.  WIDE forms each round's
// two products as 32 x 32 -> 64-bit multiplies, otherwise as separate high
// and low products (measured: the wide form is faster in the n_M = 8
// kernels, the separate one in the n_M = 4 kernels).
struct PhiloxKeys {
    uint32_t k0[10], k1[10];
    __device__ __forceinline__ PhiloxKeys(uint32_t a, uint32_t b) {
#pragma unroll
        for (int r = 0; r < 10; ++r) {
            k0[r] = a + (uint32_t)r * 0x9E3779B9u;
            k1[r] = b + (uint32_t)r * 0xBB67AE85u;
        }
    }
};
template <bool WIDE>
__device__ __forceinline__ uint4 philox_rk(uint4 c, const PhiloxKeys& K) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        uint32_t hi0, lo0, hi1, lo1;
        if constexpr (WIDE) {
            const uint64_t p0 = (uint64_t)0xD2511F53u * c.x, p1 = (uint64_t)0xCD9E8D57u * c.z;
            hi0 = (uint32_t)(p0 >> 32);
            lo0 = (uint32_t)p0;
            hi1 = (uint32_t)(p1 >> 32);
            lo1 = (uint32_t)p1;
        } else {
            hi0 = __umulhi(0xD2511F53u, c.x);
            lo0 = 0xD2511F53u * c.x;
            hi1 = __umulhi(0xCD9E8D57u, c.z);
            lo1 = 0xCD9E8D57u * c.z;
        }
        c = make_uint4(hi1 ^ c.y ^ K.k0[r], lo1, hi0 ^ c.w ^ K.k1[r], lo0);
    }
    return c;
}

// All WANT <= kDirChunk directions of a cell update in one pass, in the
// stream order of draw_directions: the two attempts of block 0 (field pairs
// 1 and 2), blocks 1 and 2 without a loop (every lane needs block 1 and
// nearly every warp has a lane that needs block 2), then block after block
// while the lane has fewer than WANT kept attempts.  A lane may keep more
// than WANT (at most max(8, WANT + 2) <= kDirRows), in rows of sdir that no
// trial reads; the stream is not continued.
template <int ROWS, int WANT> struct DrawOnce {
    static_assert(WANT <= kDirChunk && kDirRows >= kDirChunk + 2 && kDirRows >= 8, "sdir rows");
    static constexpr uint32_t kOnce = WANT == 1 ? 2 : 3;   // blocks without a loop
    const PhiloxKeys K;
    uint32_t sweep, cell, c2;
    float2 (*sdir)[32 * ROWS];
    int tid, have;
    __device__ __forceinline__ DrawOnce(const Geometry& g, uint32_t sweep_, uint32_t cell_, uint32_t c2_,
                                        float2 (*sdir_)[32 * ROWS], int tid_)
        : K(g.key0, g.key1), sweep(sweep_), cell(cell_), c2(c2_), sdir(sdir_), tid(tid_), have(0) {}
    __device__ __forceinline__ void attempt(uint32_t a, uint32_t b) {
        const float u = sym21(a), v = sym21(b);
        if (__fmaf_rn(u, u, __fmul_rn(v, v)) < 1.0f) {
            sdir[have][tid] = make_float2(u, v);
            ++have;
        }
    }
    // The attempts of one block; returns its field 0 (block 0: the shuffle draw).
    __device__ __forceinline__ uint32_t block(uint32_t blk) {
        uint32_t F[6];
        fields21(philox_rk<(WANT > 4)>(make_uint4(sweep, cell, c2, blk), K), F);
        if (blk != 0u) attempt(F[0], F[1]);
        attempt(F[2], F[3]);
        attempt(F[4], F[5]);
        return F[0];
    }
    __device__ __forceinline__ uint32_t all() {   // returns field 0 of block 0
        const uint32_t f0 = block(0u);
#pragma unroll
        for (uint32_t blk = 1; blk < kOnce; ++blk) block(blk);
        for (uint32_t blk = kOnce; have < WANT; ++blk) block(blk);
        return f0;
    }
};

// Phases 3 and 4 for a warp whose cells hold at most two disks each: nearly
// every warp with cells of about sigma (none of a 256^2-disk fluid at phi =
// 0.716 held three).  Trial t moves slot t mod n, so even trials move slot 0
// without a select, odd ones slot n - 1, and the shuffle is one conditional
// exchange (bit 20 of field 0: the 21-bit Lemire draw in [0, 2)).  N = 1M, phi
// = 0.70, in-step: 11.31 -> 10.60 us at n_M = 4, 17.88 -> 16.31 us at n_M = 8.  (Bounding the 16 neighbour slots
// through |t|^2 + (|q|^2 - sigma^2) - 2 t.q first, two packed multiply-adds
// and a three-input minimum per pair with a band that falls back on the
// method's expression, was slower: 11.77 us.)
template <int ROWS, int NSEL>
__device__ __forceinline__ void trials_of_two(const Geometry& g, const float* __restrict__ cells, const Neighbourhood& nbh,
                                              int hx, int hy, Cell<float>& own, int n, uint32_t f0, const float4 (&n01)[8],
                                              uint32_t dir23, const float2 (*__restrict__ sdir)[32 * ROWS], int tid,
                                              unsigned int& n_acc, unsigned int& n_leave) {
    const bool two = n == 2;
    float x0 = own.x[0], y0 = own.y[0], x1 = own.x[1], y1 = own.y[1];
    if (two && !(f0 >> 20) && !(g.flags & kNoParticleShuffle)) {
        x0 = own.x[1];
        y0 = own.y[1];
        x1 = own.x[0];
        y1 = own.y[0];
    }
    const f2x ns2 = pk(-g.sig2f, -g.sig2f);
    f2x qx[8], qy[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const float sx = (float)dir_dx(c) * g.wxf, sy = (float)dir_dy(c) * g.wyf;
        qx[c] = add2(pk(n01[c].x, n01[c].y), pk(sx, sx));
        qy[c] = add2(pk(n01[c].z, n01[c].w), pk(sy, sy));
    }
    // slot pair (2,3) of flagged direction c, translated
    auto pair23 = [&](int c, f2x& x, f2x& y) {
        const float2* p = reinterpret_cast<const float2*>(cell_at(cells, nbh.index(g, c, hx, hy)));
        const float2 x23 = p[1], y23 = p[3];
        const float sx = (float)dir_dx(c) * g.wxf, sy = (float)dir_dy(c) * g.wyf;
        x = add2(pk(x23.x, x23.y), pk(sx, sx));
        y = add2(pk(y23.x, y23.y), pk(sy, sy));
    };
    f2x fx23 = 0, fy23 = 0;
    const uint32_t more23 = dir23 & (dir23 - 1);
    if (dir23) pair23(__ffs(dir23) - 1, fx23, fy23);
    const float df = g.df;
#pragma unroll
    for (int t = 0; t < NSEL; ++t) {
        const bool second = (t & 1) && two;   // moves slot 1
        const float2 uv = sdir[t][tid];
        const float tx = __fmaf_rn(df, uv.x, second ? x1 : x0);
        const float ty = __fmaf_rn(df, uv.y, second ? y1 : y0);
        // 0 <= t < w as one unsigned compare of the bit patterns (w > 0; fma(d, u, p) with d*u != 0 is never -0)
        const bool inside = __float_as_uint(tx) < __float_as_uint(g.wxf) && __float_as_uint(ty) < __float_as_uint(g.wyf);
        const f2x tx2 = pk(tx, tx), ty2 = pk(ty, ty);
        // the other own slot (empty unless two), by the method's expression
        const float ex = __fsub_rn(tx, second ? x0 : x1), ey = __fsub_rn(ty, second ? y0 : y1);
        uint32_t acc = __float_as_uint(__fmaf_rn(ex, ex, __fmaf_rn(ey, ey, -g.sig2f)));
        if (dir23) {
            const f2x z = zpair(tx2, ty2, fx23, fy23, ns2);
            acc |= lo32(z) | hi32(z);
        }
        for (uint32_t m = more23; m; m &= m - 1) {   // warp-uniform, rarely taken
            f2x x, y;
            pair23(__ffs(m) - 1, x, y);
            const f2x z = zpair(tx2, ty2, x, y, ns2);
            acc |= lo32(z) | hi32(z);
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const f2x z = zpair(tx2, ty2, qx[c], qy[c], ns2);
            acc |= lo32(z) | hi32(z);
        }
        const bool ok = inside && !(acc >> 31);
        if (t & 1) {
            const bool ok1 = ok && two, ok0 = ok && !two;
            x1 = ok1 ? tx : x1;
            y1 = ok1 ? ty : y1;
            x0 = ok0 ? tx : x0;
            y0 = ok0 ? ty : y0;
        } else {
            x0 = ok ? tx : x0;
            y0 = ok ? ty : y0;
        }
        n_acc += ok;
        n_leave += !inside;
    }
    own.x[0] = x0;
    own.y[0] = y0;
    own.x[1] = x1;
    own.y[1] = y1;
}

// DENSE (cells that often hold three or four disks, as with the paper's
// cells just below sqrt(2) sigma): slot pairs (2,3) of all 8 neighbours stay
// in registers and every trial tests all of them, instead of the flagged
// directions' pairs being read again in every trial.
template <int ROWS, int NSEL, bool TRACK, bool DENSE, bool AHEAD>
__device__ __forceinline__ void subsweep_f32(const Geometry& g, float* __restrict__ cells,
                                             const SweepDraw* __restrict__ draw, int k, int bx, int by,
                                             unsigned long long* __restrict__ bpart,
                                             float2 (*__restrict__ sdir)[32 * ROWS], double* msd = nullptr) {
    const int nsel = NSEL > 0 ? NSEL : g.nsel;
    const int tid = threadIdx.y * 32 + threadIdx.x;
    int Q;
    uint32_t sweep;
    set_and_sweep(draw, k, Q, sweep);
    const int hx = bx * 32 + threadIdx.x;
    const int hy = by * ROWS + threadIdx.y;
    const int cx = 2 * hx + (Q & 1), cy = 2 * hy + (Q >> 1);
    const bool live = hx < g.hx && hy < g.hy && cy >= g.ylo && cy <= g.yhi;
    const Neighbourhood nbh(g, Q, hx, hy, live);
    const uint32_t cell = (uint32_t)(cy + g.row0) * (uint32_t)g.mx + (uint32_t)cx;   // global cell number
    const uint32_t c2 = (kDomTrial << 28) | ((uint32_t)Q << 24);
    uint32_t f0;   // shuffle draw: field 0 of block 0
    constexpr bool kFixed = NSEL > 0 && NSEL <= kDirChunk;
    DrawOnce<ROWS, kFixed ? NSEL : 1> D(g, sweep, cell, c2, sdir, tid);
    uint32_t F[6];
    uint32_t blk = 0;
    int pnext = 1;               // next attempt: field pair 1 of block 0 (fields 2,3)
    auto draw_first = [&] {
        if constexpr (kFixed) {
            f0 = D.all();
        } else {
            fields21(philox4x32_10(make_uint4(sweep, cell, c2, 0u), g.key0, g.key1), F);
            f0 = F[0];
            draw_directions<ROWS>(g, sweep, cell, c2, F, blk, pnext, min(kDirChunk, nsel), sdir, tid);   // refills F
        }
    };
    if (AHEAD) draw_first();
    pdl_wait();

    // 2. loads
    Cell<float> own;
#pragma unroll
    for (int j = 0; j < 4; ++j) own.x[j] = own.y[j] = (float)kEmpty;
    float* ownp = cell_at(cells, nbh.own(g, hx, hy));
    if (live) load_cell(ownp, own);
    float4 n01[8];   // slots 0,1 of the neighbours (x0 x1 y0 y1); slot 2 only to flag its use
    float n2[8];
    float4 n23[DENSE ? 8 : 1];   // DENSE: slots 2,3 of the neighbours (x2 x3 y2 y3)
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        n01[c] = make_float4((float)kEmpty, (float)kEmpty, (float)kEmpty, (float)kEmpty);
        n2[c] = (float)kEmpty;
        if (DENSE) n23[c] = n01[c];
        if (live) {
            const float* p = cell_at(cells, nbh.index(g, c, hx, hy));
            Cell<float> a;
            load_cell(p, a);   // one 256-bit load; slots 0, 1 and x2 are used
            n01[c] = make_float4(a.x[0], a.x[1], a.y[0], a.y[1]);
            n2[c] = a.x[2];
            if (DENSE) n23[c] = make_float4(a.x[2], a.x[3], a.y[2], a.y[3]);
        }
    }

    if (!AHEAD) draw_first();   // covers the latency of the loads

    // 3. cell contents
    const int n = (own.x[0] >= 0.f) + (own.x[1] >= 0.f) + (own.x[2] >= 0.f) + (own.x[3] >= 0.f);
    uint32_t dir23 = 0;   // warp-uniform: directions where some lane has a third disk
    {
        uint32_t mine = 0;
#pragma unroll
        for (int c = 0; c < 8; ++c) mine |= (n2[c] >= 0.f) ? (1u << c) : 0u;
        dir23 = __reduce_or_sync(0xffffffffu, mine);
    }
    const bool own23 = __any_sync(0xffffffffu, n >= 3);

    unsigned int n_tr = 0, n_acc = 0, n_leave = 0;
    float net2 = 0.f;
    if constexpr (!DENSE && !TRACK && NSEL > 0 && NSEL <= kDirChunk) {
        if (!own23) {   // warp-uniform
            if (n > 0) {
                trials_of_two<ROWS, NSEL>(g, cells, nbh, hx, hy, own, n, f0, n01, dir23, sdir, tid, n_acc, n_leave);
                n_tr = (unsigned)NSEL;
                store_cell(ownp, own);
            }
            checked_warp(g.check);
            add_block_counters<ROWS>(n_tr, n_acc, n_leave, bpart);
            return;
        }
    }
    if (n > 0) {
        // shuffle of the cell's disks (Alg. 1): one draw in [0, n!) by 21-bit Lemire on field 0
        if (n >= 2 && !(g.flags & kNoParticleShuffle)) {
            const uint32_t range = factorial(n);
            const uint32_t m = f0 * range;
            const uint32_t thr = n == 4 ? 8u : (n == 3 ? 2u : 0u);   // 2^21 mod n!
            uint32_t kk = m >> 21;
            if ((m & 0x1FFFFFu) < thr) {   // rejected: draw from the shuffle stream instead
                WordStream s(g.key0, g.key1, sweep, cell, (kDomShuffle << 28) | ((uint32_t)Q << 24));
                kk = s.bounded(range);
            }
            shuffle_slots(own.x, own.y, n, kk);
        }
        float sx0[4], sy0[4];
        if (TRACK) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                sx0[j] = own.x[j];
                sy0[j] = own.y[j];
            }
        }
        f2x qx01[8], qy01[8];
        f2x qx23[DENSE ? 8 : 1], qy23[DENSE ? 8 : 1];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const float sx = (float)dir_dx(c) * g.wxf, sy = (float)dir_dy(c) * g.wyf;
            qx01[c] = add2(pk(n01[c].x, n01[c].y), pk(sx, sx));
            qy01[c] = add2(pk(n01[c].z, n01[c].w), pk(sy, sy));
            if (DENSE) {
                qx23[c] = add2(pk(n23[c].x, n23[c].y), pk(sx, sx));
                qy23[c] = add2(pk(n23[c].z, n23[c].w), pk(sy, sy));
            }
        }
        // slot pair (2,3) of the first flagged direction, translated; further
        // flagged directions (rare) are read in the trial loop
        f2x fx23 = 0, fy23 = 0;
        const uint32_t more23 = DENSE ? 0u : dir23 & (dir23 - 1);
        if (!DENSE && dir23) {
            const int c = __ffs(dir23) - 1;
            const float2* p = reinterpret_cast<const float2*>(cell_at(cells, nbh.index(g, c, hx, hy)));
            const float2 x23 = p[1], y23 = p[3];
            const float sx = (float)dir_dx(c) * g.wxf, sy = (float)dir_dy(c) * g.wyf;
            fx23 = add2(pk(x23.x, x23.y), pk(sx, sx));
            fy23 = add2(pk(y23.x, y23.y), pk(sy, sy));
        }
        const float df = g.df;
        const f2x ns2 = pk(-g.sig2f, -g.sig2f);

        // 4. trials; trial tt of the current chunk uses direction sdir[tt]
        // and slot i, which lies in the slot set M
        int i = 0;
        auto trial = [&](int tt, auto slots) {
            constexpr unsigned M = decltype(slots)::value;
            {
                const float2 uv = sdir[tt][tid];
                const float tx = __fmaf_rn(df, uv.x, pick_in<M>(own.x, i));
                const float ty = __fmaf_rn(df, uv.y, pick_in<M>(own.y, i));
                // tx >= 0 && tx < w as one unsigned compare of the bit
                // patterns (w > 0); exact because fma(d, u, p) with
                // d*u != 0 is never -0, the one value read differently
                const bool inside = __float_as_uint(tx) < __float_as_uint(g.wxf) &&
                                    __float_as_uint(ty) < __float_as_uint(g.wyf);
                const f2x tx2 = pk(tx, tx), ty2 = pk(ty, ty);
                // own cell: every other occupied slot (slot i excluded)
                f2x z = zpair(tx2, ty2, pk(own.x[0], own.x[1]), pk(own.y[0], own.y[1]), ns2);
                uint32_t acc = ((M & 1u) && i == 0 ? 0u : lo32(z)) | ((M & 2u) && i == 1 ? 0u : hi32(z));
                if (DENSE || own23) {
                    z = zpair(tx2, ty2, pk(own.x[2], own.x[3]), pk(own.y[2], own.y[3]), ns2);
                    acc |= ((M & 4u) && i == 2 ? 0u : lo32(z)) | ((M & 8u) && i == 3 ? 0u : hi32(z));
                }
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    z = zpair(tx2, ty2, qx01[c], qy01[c], ns2);
                    acc |= lo32(z) | hi32(z);
                    if (DENSE) {
                        z = zpair(tx2, ty2, qx23[c], qy23[c], ns2);
                        acc |= lo32(z) | hi32(z);
                    }
                }
                if (!DENSE && dir23) {
                    z = zpair(tx2, ty2, fx23, fy23, ns2);
                    acc |= lo32(z) | hi32(z);
                }
                for (uint32_t m = more23; m; m &= m - 1) {   // warp-uniform, rarely taken
                    const int c = __ffs(m) - 1;
                    const float2* p = reinterpret_cast<const float2*>(cell_at(cells, nbh.index(g, c, hx, hy)));
                    const float2 x23 = p[1], y23 = p[3];
                    const float sx = (float)dir_dx(c) * g.wxf, sy = (float)dir_dy(c) * g.wyf;
                    z = zpair(tx2, ty2, add2(pk(x23.x, x23.y), pk(sx, sx)), add2(pk(y23.x, y23.y), pk(sy, sy)), ns2);
                    acc |= lo32(z) | hi32(z);
                }
                const bool ok = inside && !(acc & 0x80000000u);
                put_in<M>(own.x, i, tx, ok);
                put_in<M>(own.y, i, ty, ok);
                n_acc += ok;
                n_leave += !inside;
                i = (i + 1 == n) ? 0 : i + 1;
            }
        };
        if constexpr (NSEL > 0 && NSEL <= kDirChunk) {
            unrolled_trials(trial, std::make_integer_sequence<int, NSEL>{});
        } else {
            for (int t0 = 0; t0 < nsel; t0 += kDirChunk) {
                const int want = min(kDirChunk, nsel - t0);
                if (t0 > 0) draw_directions<ROWS>(g, sweep, cell, c2, F, blk, pnext, want, sdir, tid);
#pragma unroll 1
                for (int tt = 0; tt < want; ++tt) trial(tt, std::integral_constant<unsigned, 0xFu>{});
            }
        }
        n_tr = (unsigned)nsel;
        store_cell(ownp, own);
        if (TRACK) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float ex = own.x[j] - sx0[j], ey = own.y[j] - sy0[j];
                net2 += ex * ex + ey * ey;
            }
        }
    }
    checked_warp(g.check);
    if (TRACK) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) net2 += __shfl_xor_sync(0xffffffffu, net2, o);
        if (threadIdx.x == 0) atomicAdd(msd, (double)net2);
    }
    add_block_counters<ROWS>(n_tr, n_acc, n_leave, bpart);
}

template <int ROWS, int NSEL, bool DENSE = false, bool AHEAD = true>
static __global__ void __launch_bounds__(32 * ROWS, DENSE ? 16 / ROWS : 20 / ROWS)
k_subsweep_f32(const Geometry g, float* __restrict__ cells, const SweepDraw* __restrict__ draw, int k,
               unsigned long long* __restrict__ partial) {
    pdl_release();
    __shared__ float2 sdir[kDirRows][32 * ROWS];
    // counters of the tile that holds this block (shared by the blocks of a
    // tile: atomic adds)
    const long long slot = (long long)(blockIdx.y * ROWS / kCounterRows) * gridDim.x + blockIdx.x;
    subsweep_f32<ROWS, NSEL, false, DENSE, AHEAD>(g, cells, draw, k, blockIdx.x, blockIdx.y, partial + 4 * slot, sdir);
}

}  // namespace hdmc
