// hdmc3_subsweep.cuh -- the three-dimensional sub-sweep (Alg. 1 and Alg. 2
// with eight checkerboard sets): a group of G lanes per active cell.  Each
// lane keeps slots 0 and 1 of its share of the 26 neighbour cells in
// registers, as packed binary32 pairs, and tests every trial position against
// them; a vote of the group decides the trial.  The group's lanes draw the
// trial directions together, one Philox block (binary64: three) per lane and
// round, and the first round also draws the shuffle.  Third spheres of a cell
// are rare (flagged per warp, read when present).
//
// What binds it: with few active cells the chain of one cell update (loads,
// Philox, n_M dependent trials), which wide groups shorten; with many latency at
// 10 to 12 warps per SM (168 registers) beside the instructions, and in binary64
// also the binary64 pipe, which has two instructions per trial coordinate.  One
// thread per cell, which first gathered the neighbours within reach of its trials
// into shared memory, took (us per sub-sweep in-step, n_M = 4, phi = 0.47, before
// -> now):
//     216 active cells (N = 2048)       binary32 14.4 ->  3.9   binary64  47.6 ->  4.9
//   2,197             (N = 16384)                14.3 ->  4.6             46.6 ->  6.8
//  32,768             (N = 256,000)              16.5 -> 11.7             53.4 -> 23.4
// 140,608             (N = 1,048,576)            39.5 -> 30.8            166.5 -> 76.6
#pragma once

#include "hdmc3_device.cuh"

namespace hdmc {

// Is (hi:lo, ...) an attempt inside the unit ball?  The definition is the
// binary64 test (u0*u0 + u1*u1) + u2*u2 < 1 on the three sym52 variates.  A
// binary32 estimate from the high words (each within 6.1e-8 of its variate,
// so the estimate of the sum within 1e-6) decides whenever it lies farther
// than 2^-16 from 1; the rest are decided in binary64.
__device__ __forceinline__ bool inside_ball(const uint32_t (&w)[6]) {
    const float a = (float)(int32_t)(w[0] ^ 0x80000000u) * 0x1p-31f;
    const float b = (float)(int32_t)(w[2] ^ 0x80000000u) * 0x1p-31f;
    const float c = (float)(int32_t)(w[4] ^ 0x80000000u) * 0x1p-31f;
    const float s = a * a + b * b + c * c;
    if (s < 1.0f - 0x1p-16f) return true;
    if (s > 1.0f + 0x1p-16f) return false;
    const double u0 = sym52(w[0], w[1]), u1 = sym52(w[2], w[3]), u2 = sym52(w[4], w[5]);
    return (u0 * u0 + u1 * u1) + u2 * u2 < 1.0;
}

// Precision-specific parts of a cell update.
//
// Trial directions, uniform in the unit ball by rejection from (-1,1)^3:
//   binary64: consecutive words of the trial stream, six per attempt, three
//             sym52 variates u = m 2^-52 (m odd, |m| < 2^52); a lane takes
//             three Philox blocks, two attempts.  The words of a kept
//             attempt are stored, then made into displacements: each variate is
//             the binary64 with m's sign and magnitude 2^52 + |m| (sym52_offset),
//             and d u is RN(d u) = fma(d 2^-52, 2^52 + |m|, -d), with the
//             sign of m: the product is exactly d + d |m| 2^-52, so one
//             instruction of the slow binary64 pipe rounds d u correctly.
//   binary32: each Philox block of the trial stream cut into six 21-bit
//             fields, two attempts of three sym21 variates per block, kept
//             when fma(u, u, fma(v, v, s*s)) < 1; a lane takes one block.
//
// Overlap test of a trial position with two slots at once, on binary32
// coordinates.  binary32: the method's own test.  binary64: the coordinates
// are truncated copies and r^2 is estimated; every difference is within
// 6e-7 sigma of the binary64 one (truncations 2 x 1.7e-7, the offset's and
// the sums' roundings 2.6e-7, coordinates below 1.42 sigma), r^2 near
// contact within 2.4e-6 sigma^2, and the band of 2^-16 sigma^2 on either side
// is decided in binary64.
template <typename T> struct Sub3;

template <> struct Sub3<float> {
    static constexpr bool kExact = true;   // the pair test decides
    struct Draw {
        float u[2][3];
        bool keep[2];
    };
    static __device__ __forceinline__ uint32_t attempts(const G3& g, uint32_t sweep, uint32_t c, uint32_t dom,
                                                        uint32_t lane_block, Draw& d) {
        uint32_t f[6];
        const uint4 r = philox4x32_10(make_uint4(sweep, c, dom, lane_block), g.key0, g.key1);
        fields21(r, f);
#pragma unroll
        for (int a = 0; a < 2; ++a) {
#pragma unroll
            for (int q = 0; q < 3; ++q) d.u[a][q] = sym21(f[3 * a + q]);
            d.keep[a] = fmaf(d.u[a][0], d.u[a][0], fmaf(d.u[a][1], d.u[a][1], d.u[a][2] * d.u[a][2])) < 1.0f;
        }
        return r.x;
    }
    static __device__ __forceinline__ float trial(const G3& g, float x, float u) { return fmaf(g.df, u, x); }
    static __device__ __forceinline__ bool inside(float p, float w) { return p >= 0.0f && p < w; }
    static __device__ __forceinline__ float est(float v) { return v; }
    static __device__ __forceinline__ float est_or_far(float v) { return v; }   // an empty slot's sentinel is far away
};

template <> struct Sub3<double> {
    static constexpr bool kExact = false;
    struct Draw {
        double u[2][3];
        bool keep[2];
    };
    static __device__ __forceinline__ uint32_t attempts(const G3& g, uint32_t sweep, uint32_t c, uint32_t dom,
                                                        uint32_t lane_block, Draw& d) {
        uint32_t w[12];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const uint4 r = philox4x32_10(make_uint4(sweep, c, dom, 3 * lane_block + b), g.key0, g.key1);
            w[4 * b] = r.x;
            w[4 * b + 1] = r.y;
            w[4 * b + 2] = r.z;
            w[4 * b + 3] = r.w;
        }
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const uint32_t v[6] = {w[6 * a], w[6 * a + 1], w[6 * a + 2], w[6 * a + 3], w[6 * a + 4], w[6 * a + 5]};
            d.keep[a] = inside_ball(v);
#pragma unroll
            for (int q = 0; q < 3; ++q) d.u[a][q] = __hiloint2double((int)v[2 * q], (int)v[2 * q + 1]);
        }
        return w[0];
    }
    static __device__ __forceinline__ double displacement(const G3& g, double words) {
        const double v = sym52_offset((uint32_t)__double2hiint(words), (uint32_t)__double2loint(words));
        const double c = __longlong_as_double(__double_as_longlong(g.d) ^
                                              ((__double_as_longlong(v) & (1ll << 63)) ^ (1ll << 63)));   // -d with v's sign
        return __fma_rn(g.d52, v, c);
    }
    static __device__ __forceinline__ double trial(const G3&, double x, double du) { return __dadd_rn(x, du); }
    static __device__ __forceinline__ bool inside(double p, double w) {
        return Prm<double>::ge0(p) && Prm<double>::lt(p, w);
    }
    static __device__ __forceinline__ float est(double v) { return approx_pos(v); }
    static __device__ __forceinline__ float est_or_far(double v) { return pos_or_far(v); }
};

// Slots 0 and 1 of a cell, moved by (sx, sy, sz), as packed pairs, and
// whether slot 2 is occupied.  Slots 2 and 3 likewise (OFF = 2).
struct Pair3 {
    f2x x, y, z;
};
template <typename T>
__device__ __forceinline__ void ld2(const T* p, T& a, T& b);
template <> __device__ __forceinline__ void ld2(const float* p, float& a, float& b) {
    const float2 v = *reinterpret_cast<const float2*>(p);
    a = v.x;
    b = v.y;
}
template <> __device__ __forceinline__ void ld2(const double* p, double& a, double& b) {
    const double2 v = *reinterpret_cast<const double2*>(p);
    a = v.x;
    b = v.y;
}
template <typename T>
__device__ __forceinline__ Pair3 pair_at(const T* p, float sx, float sy, float sz, T& x2) {
    T x0, x1, y0, y1, z0, z1;
    if constexpr (sizeof(T) == 4) {
        const float4 v = *reinterpret_cast<const float4*>(p);
        x0 = v.x;
        x1 = v.y;
        x2 = v.z;
    } else {
        ld2(p, x0, x1);
        x2 = p[2];
    }
    ld2(p + 4, y0, y1);
    ld2(p + 8, z0, z1);
    Pair3 r;
    r.x = add2(pk(Sub3<T>::est_or_far(x0), Sub3<T>::est_or_far(x1)), pk(sx, sx));
    r.y = add2(pk(Sub3<T>::est(y0), Sub3<T>::est(y1)), pk(sy, sy));
    r.z = add2(pk(Sub3<T>::est(z0), Sub3<T>::est(z1)), pk(sz, sz));
    return r;
}

template <typename T>
__device__ __forceinline__ Pair3 pair23_at(const T* p, float sx, float sy, float sz) {
    T x0, x1, y0, y1, z0, z1;
    ld2(p + 2, x0, x1);
    ld2(p + 6, y0, y1);
    ld2(p + 10, z0, z1);
    Pair3 r;
    r.x = add2(pk(Sub3<T>::est_or_far(x0), Sub3<T>::est_or_far(x1)), pk(sx, sx));
    r.y = add2(pk(Sub3<T>::est(y0), Sub3<T>::est(y1)), pk(sy, sy));
    r.z = add2(pk(Sub3<T>::est(z0), Sub3<T>::est(z1)), pk(sz, sz));
    return r;
}

// fma(dx, dx, fma(dy, dy, fma(dz, dz, ns2))) for both slots of a pair.
__device__ __forceinline__ f2x ztriple(const Pair3& q, f2x px, f2x py, f2x pz, f2x ns2) {
    const f2x dx = sub2(px, q.x), dy = sub2(py, q.y), dz = sub2(pz, q.z);
    return fma2(dx, dx, fma2(dy, dy, fma2(dz, dz, ns2)));
}

// Where a cell's neighbours are: the storage index of the neighbour at offset
// (dx, dy, dz) is x[dx + 1] + y[dy + 1] + z[dz + 1] (the set number and the
// half-grid position both separate by axis; periodic).
struct Axes3 {
    unsigned x[3], y[3], z[3];
    __device__ __forceinline__ static void axis(int i, int q, int h, unsigned stride, unsigned set, unsigned (&v)[3]) {
        int lo = i - 1 + q, hi = i + q;
        lo = lo < 0 ? h - 1 : lo;
        hi = hi >= h ? 0 : hi;
        v[0] = (unsigned)lo * stride + (unsigned)(q ^ 1) * set;
        v[1] = (unsigned)i * stride + (unsigned)q * set;
        v[2] = (unsigned)hi * stride + (unsigned)(q ^ 1) * set;
    }
    __device__ __forceinline__ Axes3(const G3& g, int Q, int ix, int iy, int iz) {
        axis(ix, Q & 1, g.h[0], 1u, g.cq, x);
        axis(iy, (Q >> 1) & 1, g.h[1], (unsigned)g.h[0], 2u * g.cq, y);
        axis(iz, Q >> 2, g.h[2], (unsigned)g.h[0] * (unsigned)g.h[1], 4u * g.cq, z);
    }
    // Neighbours 0..25: 3 row + (dx + 1) for the eight x-rows (dy, dz) != (0, 0)
    // in the order (dz, dy), then dx = -1 and dx = 1 of the cell's own row.
    __device__ __forceinline__ unsigned at(const G3& g, int num, int& dx, int& dy, int& dz) const {
        int row = (num * 11) >> 5;   // num / 3 for num < 32
        dx = num >= 24 ? 2 * (num - 24) : num - 3 * row;
        row = num >= 24 ? 4 : row + (row >= 4);   // 4: the own row
        dz = (row * 11) >> 5;
        dy = row - 3 * dz;
        const unsigned i = (dx == 0 ? x[0] : dx == 1 ? x[1] : x[2]) + (dy == 0 ? y[0] : dy == 1 ? y[1] : y[2]) +
                           (dz == 0 ? z[0] : dz == 1 ? z[1] : z[2]);
        --dx;
        --dy;
        --dz;
        return (unsigned)checked_cell(g.check, i, g.C);
    }
};

// The method's test of the trial position against slots first..last of one
// neighbour cell, up to its first empty slot.
template <typename T>
__device__ __forceinline__ bool slots_hit(const G3& g, const T* cells, unsigned sn, int dx, int dy, int dz, int first, int last,
                                          const T* p) {
    using A = Ar3<T>;
    const T sx = (T)dx * A::w(g, 0), sy = (T)dy * A::w(g, 1), sz = (T)dz * A::w(g, 2);
    bool hit = false;
    for (int j = first; j <= last; ++j) {
        const T* q = slot3(cells, g, sn, j);
        if (is_empty(q[0])) break;
        hit |= A::hit(g, p[0] - (q[0] + sx), p[1] - (q[4] + sy), p[2] - (q[8] + sz));
    }
    return hit;
}

constexpr int kSubB3 = 32;     // threads of a sub-sweep block: one warp, no block barrier (blocks of 4 warps: 41 instead of 37 us at 132,651 active cells)
constexpr int kDir3 = 8;       // trial directions drawn ahead per cell

// Shared memory of one warp's cells.
template <typename T, int G> struct Warp3 {
    static constexpr int kCells = 32 / G;
    // kept directions, a ring: fewer than kDir3 left over, 2 G more per round
    static constexpr int kRing = G <= 4 ? 16 : G <= 8 ? 32 : 128;
    static_assert(kRing >= kDir3 - 1 + 2 * G, "direction ring");
    // the cell last: the lanes of a warp read neighbouring banks
    T dir[kRing][3][kCells];
    T own[kSlots3][3][kCells];   // own spheres, slot order before the shuffle
    T trial[3][kCells];          // the current trial position
};

// One sub-sweep: every cell of set Q = table[jd].perm[k] (Alg. 1, Alg. 2).
template <typename T, int G>
__device__ __forceinline__ void sub3_cells(const G3& g, T* __restrict__ cells, const Draw3* __restrict__ table, int jd,
                                           int k, unsigned long long* __restrict__ ctr) {
    using S = Sub3<T>;
    using A = Ar3<T>;
    using W = Warp3<T, G>;
    constexpr int NC = G <= 8 ? 24 / G + 1 : 1;    // neighbour cells of a lane
    static_assert(G == 2 || G == 4 || G == 8 || G == 32, "lanes per cell");
    constexpr unsigned kFull = 0xFFFFFFFFu;
    __shared__ W warps[kSubB3 / 32];
    W& sw = warps[threadIdx.x / 32];
    const int lane = threadIdx.x & 31, grp = lane / G, L = lane % G, gb = grp * G;
    const unsigned gm = (G == 32 ? kFull : ((1u << G) - 1u) << gb);   // lanes of my group
    const unsigned below = gm & ((1u << lane) - 1u);                    // those before me
    // the draw table, read through L2 ahead of pdl_wait
    const Draw3* dr = table + jd;
    const uint32_t sweep = __ldcg(&dr->sweep);
    const int Q = (int)((__ldcg(reinterpret_cast<const uint32_t*>(dr->perm) + (k >> 2)) >> (8 * (k & 3))) & 0xFFu);
    const unsigned s = (blockIdx.x * (kSubB3 / 32) + threadIdx.x / 32) * W::kCells + grp;
    const bool live = s < g.cq;
    const unsigned r1 = g.div0(s), ix = s - r1 * (unsigned)g.h[0];
    const unsigned iz = g.div1(r1), iy = r1 - iz * (unsigned)g.h[1];
    const Axes3 ax(g, Q, (int)ix, (int)iy, (int)iz);
    const int cx = 2 * (int)ix + (Q & 1), cy = 2 * (int)iy + ((Q >> 1) & 1), cz = 2 * (int)iz + (Q >> 2);
    const uint32_t c = ((uint32_t)cz * (uint32_t)g.m[1] + (uint32_t)cy) * (uint32_t)g.m[0] + (uint32_t)cx;
    const unsigned sown = (unsigned)checked_cell(g.check, live ? ax.x[1] + ax.y[1] + ax.z[1] : 0u, g.C);

    // the first trial directions, while the previous kernel's last blocks run
    const uint32_t setbits = (uint32_t)Q << 24;
    unsigned have = 0, used = 0;   // directions kept so far, lane blocks used
    auto keep = [&](bool need, const typename S::Draw& d) {
        const bool k0 = need && d.keep[0], k1 = need && d.keep[1];
        const unsigned b0 = __ballot_sync(kFull, k0), b1 = __ballot_sync(kFull, k1);
        const unsigned pos = have + __popc(b0 & below) + __popc(b1 & below);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            if (k0) sw.dir[pos % W::kRing][q][grp] = d.u[0][q];
            if (k1) sw.dir[(pos + k0) % W::kRing][q][grp] = d.u[1][q];
        }
        have += __popc(b0 & gm) + __popc(b1 & gm);
    };
    // directions t0 .. t0 + want - 1 (binary64: as displacements d u)
    auto draw = [&](int t0, int want) {
#pragma unroll 1
        for (;;) {
            const bool need = live && have < (unsigned)(t0 + want);
            if (!__any_sync(kFull, need)) break;
            typename S::Draw d;
            S::attempts(g, sweep, c, (kDomTrial << 28) | setbits, used + L, d);
            keep(need, d);
            used += need ? G : 0;
        }
        __syncwarp();
        if constexpr (!S::kExact) {
#pragma unroll 1
            for (int i = L; i < 3 * want; i += G) {
                T& w = sw.dir[(unsigned)(t0 + i / 3) % W::kRing][i % 3][grp];
                w = S::displacement(g, w);
            }
            __syncwarp();
        }
    };
    // first round: the group's last lane draws the first word of the shuffle
    // stream instead, the others the first G - 1 lane blocks
    uint32_t word;
    {
        typename S::Draw d;
        const bool last = L == G - 1;
        word = S::attempts(g, sweep, c, ((last ? kDomShuffle : kDomTrial) << 28) | setbits, last ? 0u : (uint32_t)L, d);
        keep(live && !last, d);
        used = G - 1;
        word = __shfl_sync(kFull, word, gb + G - 1);
    }
    draw(0, min(kDir3, g.nsel));
    pdl_wait();   // what comes before depends on the draw table alone

    // own spheres: the primary half's slots L, L + G
    constexpr int NO = G < 4 ? 4 / G : 1;
    T own[NO][3];
#pragma unroll
    for (int r = 0; r < NO; ++r) {
        own[r][0] = (T)kEmpty;
        own[r][1] = own[r][2] = (T)0;
        if (live && L + r * G < 4) {
            const T* p = cells + primary3(sown) + (L + r * G);
            own[r][0] = p[0];
            own[r][1] = p[4];
            own[r][2] = p[8];
        }
    }
    // my neighbour cells: slots 0 and 1 in registers; has2: bit c set when
    // the c-th of them has a third sphere
    Pair3 nb[NC];
    unsigned has2 = 0;
    // the number (Axes3::at) of my j-th neighbour: whole x-rows, then one of the own row
    auto number = [&](int j) { return G > 8 ? j * G + L : j < 3 * (8 / G) ? 3 * (L + (j / 3) * G) + j % 3 : 24 + L; };
    auto neighbour = [&](int j, unsigned sn, float sx, float sy, float sz) {
        T x2;
        nb[j] = pair_at(cells + primary3(sn), sx, sy, sz, x2);
        has2 |= !is_empty(x2) ? 1u << j : 0u;
    };
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        nb[j].x = pk(kFar, kFar);
        nb[j].y = nb[j].z = 0;
    }
    if (live) {
        if constexpr (G <= 8) {
#pragma unroll
            for (int r = 0; r < 8 / G; ++r) {
                const int num = 3 * (L + r * G);
                int dx, dy, dz;
                const unsigned row = ax.at(g, num, dx, dy, dz) - ax.x[0];
                const float sy = (float)dy * g.wf[1], sz = (float)dz * g.wf[2];
#pragma unroll
                for (int e = 0; e < 3; ++e)
                    neighbour(3 * r + e, (unsigned)checked_cell(g.check, row + ax.x[e], g.C), (float)(e - 1) * g.wf[0], sy, sz);
            }
            if (L < 2) {
                int dx, dy, dz;
                const unsigned sn = ax.at(g, 24 + L, dx, dy, dz);
                neighbour(NC - 1, sn, (float)dx * g.wf[0], 0.0f, 0.0f);
            }
        } else if (L < 26) {
            int dx, dy, dz;
            const unsigned sn = ax.at(g, L, dx, dy, dz);
            neighbour(0, sn, (float)dx * g.wf[0], (float)dy * g.wf[1], (float)dz * g.wf[2]);
        }
    }

    // own cell: number of spheres, slots 4..7 when slot 3 is occupied
    int n = 0;
#pragma unroll
    for (int r = 0; r < NO; ++r) {
        n += __popc(__ballot_sync(kFull, !is_empty(own[r][0])) & gm);
        if (L + r * G < 4) {
#pragma unroll
            for (int q = 0; q < 3; ++q) sw.own[L + r * G][q][grp] = own[r][q];
        }
    }
    if (__any_sync(kFull, n == 4)) {
        int more4 = 0;
        if (n == 4)
            for (int j = L; j < 4; j += G) {
                const T* p = cells + secondary3(g, sown) + j;
                if (is_empty(p[0])) break;
                sw.own[4 + j][0][grp] = p[0];
                sw.own[4 + j][1][grp] = p[4];
                sw.own[4 + j][2][grp] = p[8];
                ++more4;
            }
#pragma unroll
        for (int o = 1; o < (G < 4 ? G : 4); o <<= 1) more4 += __shfl_xor_sync(kFull, more4, o);
        n += __shfl_sync(kFull, more4, gb);
    }
    // shuffle (Alg. 1): slot j of the shuffled cell is old slot (perm >> 4j) & 7
    unsigned perm = 0x76543210u;
    if (n >= 2 && !(g.flags & kNoParticleShuffle)) {
        const uint32_t range = factorial8(n);
        const unsigned long long m = (unsigned long long)word * range;
        uint32_t kk = (uint32_t)(m >> 32);
        if ((uint32_t)m < range) {   // as good as never: WordStream::bounded from the start
            WordStream ws(g.key0, g.key1, sweep, c, (kDomShuffle << 28) | setbits);
            kk = ws.bounded(range);
        }
#pragma unroll 1
        for (int j = n - 1; j >= 3; --j) {   // swap slots j and kk mod (j+1)
            const unsigned qt = kk / (uint32_t)(j + 1), r = kk - qt * (uint32_t)(j + 1);
            kk = qt;
            const unsigned x = ((perm >> (4 * j)) ^ (perm >> (4 * r))) & 7u;   // 0 when j == r
            perm ^= (x << (4 * j)) ^ (x << (4 * r));
        }
        if (n >= 3) {   // kk < 6: slots 2 and kk mod 3
            const unsigned r = kk >= 3u ? kk - 3u : kk;
            kk = kk >= 3u ? 1u : 0u;
            const unsigned x = ((perm >> 8) ^ (perm >> (4 * r))) & 7u;
            perm ^= (x << 8) ^ (x << (4 * r));
        }
        if (kk == 0u) {   // kk < 2: slots 1 and kk
            const unsigned x = ((perm >> 4) ^ perm) & 7u;
            perm ^= (x << 4) ^ x;
        }
    }
    // slots 2 and 3 of the first flagged neighbour cell; further flagged cells
    // and slots 4..7 (rare) are read in the trial loop
    Pair3 f23;
    f23.x = pk(kFar, kFar);
    f23.y = f23.z = 0;
    const bool any23 = __any_sync(kFull, has2 != 0);
    unsigned more = has2 & (has2 - 1u);   // bit 31: slots 4..7 of the first flagged cell may be occupied
    if (has2) {
        int dx, dy, dz;
        const T* p = cells + primary3(ax.at(g, number(__ffs(has2) - 1), dx, dy, dz));
        f23 = pair23_at(p, (float)dx * g.wf[0], (float)dy * g.wf[1], (float)dz * g.wf[2]);
        more |= !is_empty(p[3]) ? 0x80000000u : 0u;
    }
    const bool crowd = __any_sync(kFull, n >= 2), crowdG = G < kSlots3 && __any_sync(kFull, n > G);
    __syncwarp();

    // Binary32: every lane computes the trial position.  Binary64, where the
    // slow pipe's instructions count: lane L computes coordinate L (all three
    // in every lane: 8.4 instead of 7.0 us at 2,197 active cells).
    constexpr bool kAll = S::kExact;
    static_assert(kAll || G >= 4, "one lane per coordinate");
    const int a0 = L < 3 ? L : 0;
    const T w0 = A::w(g, 0), w1 = A::w(g, 1), w2 = A::w(g, 2);
    const T wa = a0 == 0 ? w0 : a0 == 1 ? w1 : w2;
    const f2x lo2 = S::kExact ? pk(-g.sig2f, -g.sig2f) : pk(-g.band_lo, -g.band_lo);
    const f2x band2 = pk(g.band_lo - g.band_hi, g.band_lo - g.band_hi);
    unsigned n_ac = 0, n_lf = 0;
    int i = 0;
#pragma unroll 1
    for (int t = 0; t < g.nsel; ++t) {
        if (t > 0 && t % kDir3 == 0) draw(t, min(kDir3, g.nsel - t));
        const int cur = (int)((perm >> (4 * i)) & 7u);
        T(&me)[3][W::kCells] = sw.own[cur];
        const T(&u)[3][W::kCells] = sw.dir[(unsigned)t % W::kRing];
        float px, py, pz;   // estimates of the trial position (binary32: the position)
        bool inside;
        T tp[3];
        if constexpr (kAll) {
#pragma unroll
            for (int q = 0; q < 3; ++q) tp[q] = S::trial(g, me[q][grp], u[q][grp]);
            inside = S::inside(tp[0], w0) && S::inside(tp[1], w1) && S::inside(tp[2], w2);
            px = S::est(tp[0]);
            py = S::est(tp[1]);
            pz = S::est(tp[2]);
        } else {
            const T p = S::trial(g, me[a0][grp], u[a0][grp]);
            const float pf = S::est(p);
            px = __shfl_sync(kFull, pf, gb);
            py = __shfl_sync(kFull, pf, gb + 1);
            pz = __shfl_sync(kFull, pf, gb + 2);
            inside = ((__ballot_sync(kFull, S::inside(p, wa)) >> gb) & 7u) == 7u;
            if (L < 3) sw.trial[L][grp] = p;
            __syncwarp();
        }
        auto position = [&](int q) { return kAll ? tp[q] : sw.trial[q][grp]; };   // the exact one
        const f2x px2 = pk(px, px), py2 = pk(py, py), pz2 = pk(pz, pz);
        uint32_t sure = 0, maybe = 0;   // sign bits: certainly / possibly overlapping
#pragma unroll
        for (int j = 0; j < NC; ++j) {
            const f2x z = ztriple(nb[j], px2, py2, pz2, lo2);
            sure |= lo32(z) | hi32(z);
            if (!S::kExact) {
                const f2x y = add2(z, band2);
                maybe |= lo32(y) | hi32(y);
            }
        }
        if (any23) {
            const f2x z = ztriple(f23, px2, py2, pz2, lo2);
            sure |= lo32(z) | hi32(z);
            if (!S::kExact) {
                const f2x y = add2(z, band2);
                maybe |= lo32(y) | hi32(y);
            }
        }
        bool hit = (sure >> 31) != 0;
        // own cell: the other spheres, one per lane
        if (crowd) {
            auto own_hit = [&](int j) {
                const T q[3] = {sw.own[j][0][grp], sw.own[j][1][grp], sw.own[j][2][grp]};
                if constexpr (S::kExact) {
                    return A::hit(g, px - q[0], py - q[1], pz - q[2]);
                } else {
                    const float ex = px - S::est(q[0]), ey = py - S::est(q[1]), ez = pz - S::est(q[2]);
                    const float r2 = fmaf(ex, ex, fmaf(ey, ey, ez * ez));
                    if (r2 < g.band_lo || r2 > g.band_hi) return r2 < g.band_lo;
                    return A::hit(g, position(0) - q[0], position(1) - q[1], position(2) - q[2]);
                }
            };
            if (L < n && L != cur) hit |= own_hit(L);
            if (crowdG)
                for (int j = L + G; j < n; j += G)
                    if (j != cur) hit |= own_hit(j);
        }
        if (!S::kExact && !hit && inside && (maybe >> 31)) {
            // some slot is too close to contact for the estimates: decide those slots in binary64
            unsigned close = 0;   // bits 2j, 2j+1: slots 0, 1 of neighbour j; bits 30, 31: the flagged pair
#pragma unroll
            for (int j = 0; j < NC; ++j) {
                const f2x y = add2(ztriple(nb[j], px2, py2, pz2, lo2), band2);
                close |= ((lo32(y) >> 31) << (2 * j)) | ((hi32(y) >> 31) << (2 * j + 1));
            }
            const f2x y = add2(ztriple(f23, px2, py2, pz2, lo2), band2);
            close |= ((lo32(y) >> 31) << 30) | (hi32(y) & 0x80000000u);
            const T at[3] = {position(0), position(1), position(2)};
            while (close) {
                const int b = __ffs(close) - 1;
                close &= close - 1u;
                const int j = b >= 30 ? __ffs(has2) - 1 : b >> 1, slot = b >= 30 ? b - 28 : b & 1;
                int dx, dy, dz;
                const unsigned sn = ax.at(g, number(j), dx, dy, dz);
                hit |= slots_hit(g, cells, sn, dx, dy, dz, slot, slot, at);
            }
        }
        if (more && !hit && inside) {   // rare: slots 2..7 of further flagged cells, slots 4..7 of the first
            for (unsigned m = more; m; m &= m - 1u) {
                const int b = __ffs(m) - 1;
                int dx, dy, dz;
                const unsigned sn = ax.at(g, number(b == 31 ? __ffs(has2) - 1 : b), dx, dy, dz);
                const T at[3] = {position(0), position(1), position(2)};
                hit |= slots_hit(g, cells, sn, dx, dy, dz, b == 31 ? 4 : 2, kSlots3 - 1, at);
            }
        }
        checked_warp(g.check);
        const bool overlap = (__ballot_sync(kFull, hit) & gm) != 0;
        if (n > 0 && inside && !overlap) {
            if (L == 0) {
#pragma unroll
                for (int q = 0; q < 3; ++q) me[q][grp] = position(q);
            }
            ++n_ac;
        }
        n_lf += !inside;
        __syncwarp();
        i = i + 1 >= n ? 0 : i + 1;
    }
    // the shuffled slots back; unused slots keep their sentinels
#pragma unroll 1
    for (int j = L; j < n; j += G) {
        const unsigned o = (perm >> (4 * j)) & 7u;
        T* p = cells + (j < 4 ? primary3(sown) + j : secondary3(g, sown) + (j - 4));
        p[0] = sw.own[o][0][grp];
        p[4] = sw.own[o][1][grp];
        p[8] = sw.own[o][2][grp];
    }
    // counters: one lane per cell
    checked_warp(g.check);
    const bool count = L == 0 && n > 0;
    add_block_counters<1>(count ? (unsigned)g.nsel : 0u, count ? n_ac : 0u, count ? n_lf : 0u,
                          ctr + 4 * (blockIdx.x % kCtr3));
}

template <typename T, int G>
__global__ void __launch_bounds__(kSubB3, G == 2 ? 12 : G == 4 ? 16 : G == 8 ? 20 : 24) k_sub3(const G3 g, T* __restrict__ cells, const Draw3* __restrict__ table, int jd,
                                                 int k, unsigned long long* __restrict__ ctr) {
    pdl_release();
    sub3_cells<T, G>(g, cells, table, jd, k, ctr);
}

}  // namespace hdmc
