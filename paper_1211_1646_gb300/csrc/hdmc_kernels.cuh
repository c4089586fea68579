// hdmc_kernels.cuh -- cell-shift, contact-histogram, batched-replica and
// snapshot-check kernels, and the launchers.  Included once by each
// precision's translation unit.
//
// Every floating-point operation that decides an ownership or a histogram
// bin is written with an explicit round-to-nearest operation.
#pragma once

#include "hdmc_common.cuh"
#include "hdmc_subsweep64.cuh"
#include "hdmc_subsweep.cuh"

namespace hdmc {

// ---- cell shift: Alg. 4 ----------------------------------------------------------------
// Every disk is translated by -f*ds (equivalently the grid moves by +f*ds).
// One thread per new cell; grid (set row, set column, set).  New cell c = the
// disks of old c that stay inside c (old slot order), then the disks of old
// c+f that leave c+f, re-expressed in c's frame (+f*w).  The ownership test
// is the same computation in the two threads that see a disk, so every disk
// lands in exactly one cell (Sec. 3.2).  A re-expressed value that rounds
// onto the upper edge is clamped below it.
//
// The cells are read with plain loads (src is not __restrict__): the assembler
// may move read-only loads ahead of pdl_wait.
//
// Grid origin O += f*ds (one thread per shift), binary64: ds added or
// subtracted (the same rounding as adding -ds).  Kept out of line so that
// the binary64 instruction stays in that one thread.
static __device__ __noinline__ void add_origin(DevState* __restrict__ st, int ax, int sgn, double ds) {
    st->origin[ax] = sgn > 0 ? __dadd_rn(st->origin[ax], ds) : __dsub_rn(st->origin[ax], ds);
}

// Per-launch constants of the moving coordinate and the evaluation of the
// disks seen by one new cell: stayer() for a disk of old c (does it stay, and
// its new coordinate if it does), migrant() for a disk of old c + f (does it
// leave c + f, and its coordinate in c's frame if it does).  Both apply the
// same ownership test to a disk, so the two threads that see it agree.
template <typename T> struct ShiftParams;

// binary64 path: dp = x - sgn ds; stays iff 0 <= dp < w; a migrant's new
// coordinate dp + sgn w, clamped into [0, w).
template <> struct ShiftParams<double> {
    double sd, w, sw, wprev;
    const SweepDraw* draw;
    __device__ ShiftParams(const Geometry& g, const SweepDraw& r, int ax, int sgn) {
        draw = &r;
        w = ax ? g.wy : g.wx;
        sd = sgn > 0 ? r.ds : -r.ds;
        sw = sgn > 0 ? w : -w;
        wprev = Prm<double>::prev(w);
    }
    __device__ __forceinline__ double origin_ds() const { return draw->ds; }
    __device__ __forceinline__ void stayer(double x, bool& stay, double& v) const {
        v = __dsub_rn(x, sd);
        stay = Prm<double>::ge0(v) && Prm<double>::lt(v, w);
    }
    __device__ __forceinline__ void migrant(double x, bool& leave, double& v) const {
        const double dp = __dsub_rn(x, sd);
        leave = !(Prm<double>::ge0(dp) && Prm<double>::lt(dp, w));
        v = __dadd_rn(dp, sw);
        v = Prm<double>::lt(v, w) ? v : wprev;
        v = Prm<double>::ge0(v) ? v : 0.0;
    }
};

// binary32 rounding of the real number s + t + eta, |eta| <= mu, |s| >= |t|
// (s, t binary32): r = RN32(s + t), and s + t = r + rho exactly (Fast2Sum).
// All reals within mu of s + t round to r when r is positive, not a power
// of two, and rho stays more than mu inside its rounding interval (half an
// ulp on either side); otherwise ok is cleared.
__device__ __forceinline__ float rn32_certified(float s, float t, float mu, bool& ok) {
    const float r = __fadd_rn(s, t);
    const float rho = __fsub_rn(t, __fsub_rn(r, s));
    const uint32_t rb = __float_as_uint(r);
    const float h = __uint_as_float((rb & 0x7F800000u) - (24u << 23));   // half an ulp of r
    ok = (rb & 0x7FFFFFu) != 0u && rb > (25u << 23) && rb < 0x7F800000u && __fadd_rn(fabsf(rho), mu) < h;
    return r;
}

// binary32 path, remapped in binary64 on the binary32 width W = wf:
// dp = RN64(x - sgn ds); stays iff 0 <= dp < W; the stored coordinate is
// RN32(dp) for a stayer and RN32(RN64(dp + sgn W)) for a migrant, clamped
// below wf.  binary64 arithmetic is slow on this GPU, so the result is
// computed in binary32 without rounding error where that is possible and
// certified: sgn ds = d1 + d2 + d3 (d1 = RN32(sgn ds), d2 = RN32(sgn ds -
// d1), |d3| <= 2^-48 ds); s = RN32(x - d1) with its exact error e
// (TwoSum); t = RN32(e - d2); then x - sgn ds = s + t + eta with
// |eta| <= 2^-46 W.  Where s is farther than 2^-20 W from 0 and from W the
// ownership is decided by s, and rn32_certified rounds the stayer's s + t,
// the +f migrant's (s + W) + t (Fast2Sum, exact) or the -f migrant's
// (s - W) + t (s - W exact, Sterbenz) with the bound mu = 2^-43 W on eta,
// the binary32 rounding of the tails and the binary64 roundings of the
// remap.  The rest, about one disk in 10^5, is evaluated with binary64
// instructions; only that branch touches the binary64 constants.
template <> struct ShiftParams<float> {
    float d1, d2, wf, wprev, tau, mu;
    int sgn;
    bool fast;   // the bounds need cell widths far above the binary32 underflow range
    const SweepDraw* draw;
    __device__ ShiftParams(const Geometry& g, const SweepDraw& r, int ax, int sgn_) {
        sgn = sgn_;
        wf = ax ? g.wyf : g.wxf;
        wprev = Prm<float>::prev(wf);
        d1 = sgn > 0 ? r.dsf : -r.dsf;
        d2 = sgn > 0 ? r.dsf2 : -r.dsf2;
        tau = __fmul_rn(wf, 0x1p-20f);
        mu = __fmul_rn(wf, 0x1p-43f);
        fast = wf > 0x1p-60f;
        draw = &r;
    }
    __device__ __forceinline__ double origin_ds() const { return draw->ds; }
    // s = RN32(x - d1) and t: x - sgn ds = s + t + eta; sw = RN32(s - W)
    __device__ __forceinline__ void split(float x, float& s, float& t, float& sw, bool& sure) const {
        s = __fsub_rn(x, d1);
        const float bb = __fsub_rn(s, x);   // TwoSum(x, -d1): s + e = x - d1 exactly
        const float e = __fadd_rn(__fsub_rn(x, __fsub_rn(s, bb)), __fsub_rn(-d1, bb));
        t = __fsub_rn(e, d2);
        sw = __fsub_rn(s, wf);
        sure = fast && fabsf(s) > tau && fabsf(sw) > tau;   // the ownership test is decided by s
    }
    // binary64 instructions.  The conversion of W is a volatile asm, and ds
    // is added or subtracted rather than negated: binary64 operations on the
    // loop invariants would otherwise be hoisted out of this rare branch and
    // issued by every warp (the binary64 pipe is 1/64 of binary32 here).
    __device__ __forceinline__ void exact(float x, bool& stay, float& v) const {
        double W;
        asm volatile("cvt.f64.f32 %0, %1;" : "=d"(W) : "f"(wf));
        const double xd = (double)x, ds = draw->ds;
        const double dp = sgn > 0 ? __dsub_rn(xd, ds) : __dadd_rn(xd, ds);
        stay = Prm<double>::ge0(dp) && Prm<double>::lt(dp, W);
        v = __double2float_rn(stay ? dp : (sgn > 0 ? __dadd_rn(dp, W) : __dsub_rn(dp, W)));
    }
    __device__ __forceinline__ void stayer(float x, bool& stay, float& v) const {
        float s, t, sw;
        bool sure, ok;
        split(x, s, t, sw, sure);
        stay = s > 0.0f && sw < 0.0f;
        v = rn32_certified(s, t, mu, ok);
        if (!sure || (stay && !ok)) exact(x, stay, v);
        v = v < wf ? v : wprev;   // v >= 0, or -0 from a -0 stayer as the binary64 rule gives
    }
    __device__ __forceinline__ void migrant(float x, bool& leave, float& v) const {
        float s, t, sw;
        bool sure, ok;
        split(x, s, t, sw, sure);
        leave = !(s > 0.0f && sw < 0.0f);
        if (sgn > 0) {   // (s + W) + t, s + W by Fast2Sum (warp-uniform branch)
            const float s2 = __fadd_rn(s, wf);
            v = rn32_certified(s2, __fadd_rn(__fsub_rn(s, __fsub_rn(s2, wf)), t), mu, ok);
        } else {         // (s - W) + t, s - W exact
            v = rn32_certified(sw, t, mu, ok);
        }
        if (!sure || (leave && !ok)) {
            bool stay;
            exact(x, stay, v);
            leave = !stay;
        }
        v = v < wf ? v : wprev;
    }
};

// EARLY reads the own cell before the draw is known: faster where the latency of
// the two reads binds (binary64, few cells), slower where the reads themselves do
// and the cell of the other read is close by (us per shift in-step, both reads
// after the draw -> EARLY): binary64 1024 disks 2.27 -> 2.22, 65,536 5.90 -> 5.70,
// 115,850 6.03 -> 5.95, but 1M 29.2 -> 29.4, crowded 570,000 10.2 -> 11.3;
// binary32 65,536 2.94 -> 2.98, 1M 10.95 -> 11.13, 4M 51.2 -> 52.5.
constexpr long long kShiftEarlyCells = 200000;
template <typename T>
__host__ __device__ constexpr bool shift_early(long long cells) {
    return sizeof(T) == 8 && cells <= kShiftEarlyCells;
}

template <typename T, bool EARLY>
__device__ __forceinline__ void shift_cells(const Geometry& g, const T* src, T* dst,
                                            const SweepDraw* __restrict__ draw, DevState* __restrict__ st, int bx,
                                            int by, int q) {
    const int hx = bx * kShiftBX + threadIdx.x;
    const int hy = by * kShiftBY + threadIdx.y;
    const int cx = 2 * hx + (q & 1), cy = 2 * hy + (q >> 1);
    const bool live = hx < g.hx && hy < g.hy && cy >= g.slo && cy <= g.shi;   // a strip's halo rows are not its own
    const long long idx = (long long)q * g.cq + (long long)hy * g.hx + hx;
    Cell<T> o, b, r;
    if (EARLY && live) load_cell(src + 8 * idx, o);
    const int fdir = draw->fdir;
    const int ax = fdir >> 1;
    const int sgn = (fdir & 1) ? -1 : 1;
    const ShiftParams<T> P(g, *draw, ax, sgn);
    if (hx == 0 && hy == 0 && q == 0) add_origin(st, ax, sgn, P.origin_ds());
    if (!live) return;
    const int ncx = ax ? cx : wrap(cx + sgn, g.mx);
    const int ncy = ax ? wrap(cy + sgn, g.my) : cy;
    if (!EARLY) load_cell(src + 8 * idx, o);
    load_cell(src + 8 * storage_index(g, ncx, ncy), b);
#pragma unroll
    for (int j = 0; j < 4; ++j) r.x[j] = r.y[j] = T(kEmpty);
    int kept = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {   // stayers of old c (occupied slots form a prefix)
        if (Prm<T>::ge0(o.x[j])) {
            bool stay;
            T v;
            P.stayer(ax ? o.y[j] : o.x[j], stay, v);
            const T vx = ax ? o.x[j] : v, vy = ax ? v : o.y[j];
#pragma unroll
            for (int s = 0; s <= j; ++s) {
                r.x[s] = (stay && kept == s) ? vx : r.x[s];
                r.y[s] = (stay && kept == s) ? vy : r.y[s];
            }
            kept += stay;
        }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {   // migrants of old c + f
        if (Prm<T>::ge0(b.x[j])) {
            bool leave;
            T v;
            P.migrant(ax ? b.y[j] : b.x[j], leave, v);
            const T vx = ax ? b.x[j] : v, vy = ax ? v : b.y[j];
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                r.x[s] = (leave && kept == s) ? vx : r.x[s];
                r.y[s] = (leave && kept == s) ? vy : r.y[s];
            }
            kept += leave;
        }
    }
    if (kept > 4) atomicOr(&st->error, kErrOverflow);
    store_cell(dst + 8 * idx, r);
}

template <typename T, bool EARLY>
__global__ void __launch_bounds__(kShiftBX * kShiftBY)
k_shift(const Geometry g, const T* src, T* dst, const SweepDraw* __restrict__ draw,
        DevState* __restrict__ st) {
    pdl_release();
    pdl_wait();
    // the four sets of one tile are adjacent blocks (set = blockIdx.x & 3), so
    // the old cells a block reads from the neighbouring set are read by that
    // set's block at about the same time: the second read hits L2 even when
    // the state does not fit there
    shift_cells<T, EARLY>(g, src, dst, draw, st, blockIdx.x >> 2, blockIdx.y, blockIdx.x & 3);
}

// ---- contact histogram: Sec. 4 ------------------------------------------------------
// Ordered pairs (i, j != i) at distance r in [sigma, sigma + 200 dr), in bins
// [sigma + b dr, sigma + (b+1) dr) decided on the binary64 r^2 against the
// squared bin edges; distances from cell-local coordinates over the 5x5
// neighbourhood (w >= sigma, so two rings reach past 1.02 sigma).  A binary32
// estimate of r^2 with a wide margin selects the candidates (about 0.7 per
// disk); each warp queues its candidates in shared memory and computes the
// binary64 distance and bin of 32 queued pairs at a time, so the (slow)
// binary64 instructions run with every lane busy.  Non-negative doubles
// order like their bit patterns read as signed integers, so the bin search
// compares integers.
//
// The estimates bind the kernel, so each is made once for the two orders of a
// pair: a cell looks at itself and at the 12 cells ahead of it (dy > 0, or dy
// = 0 and dx > 0), and a candidate is queued in both orders, each evaluated
// with its own roundings.  A cell two steps away is looked at only if some
// lane has a disk within reach of it (a band of 0.02 sigma with cells of
// sigma, nowhere with the paper's cells), its corners never.  What is left on
// the binary64 pipe is seven instructions per queued pair.  A block does a tile
// of 32 x 8 cells, in large binary32 systems two, before it adds its bins to the
// global ones.  One histogram with its launch, each pair estimated in both orders
// -> now: 65,536 disks binary32 18.7 -> 10.5 us, binary64 29.2 -> 14.2; 1M 119 ->
// 56, 245 -> 91; the paper's cells (N = 1520^2) 189 -> 73, 289 -> 90.
__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(double v) { return approx_f32(v); }

// Exact binary32 -> binary64 on the integer pipe (conversions run on the
// binary64 pipe); subnormal binary32 values, not met in earnest, convert.
__device__ __forceinline__ double widen(float v) {
    const uint32_t u = __float_as_uint(v), m = u & 0x7FFFFFFFu;
    if (m < 0x00800000u && m != 0u) return (double)v;
    const uint32_t hi = (u & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u);
    return __hiloint2double((int)hi, (int)(u << 29));
}
__device__ __forceinline__ double widen(double v) { return v; }

constexpr int kHistQueue = 96;   // per-warp candidate queue (< 32 pending + 64 appended)

// Tiles of kHistBY set rows of a block.  Fewer blocks add fewer bins, more fill
// the chip: us with one / two / four tiles, binary32 65,536 disks 10.5 / 14.5 /
// 22.7, 360,000 26.8 / 27.8 / 30.1, 640,000 41.0 / 37.8 / 43.3, 1M 61.0 / 56.1 /
// 63.3; binary64 65,536 14.2 / 18.6 / 26.4, 1M 90.7 / 96.7 / 103.2.
constexpr long long kHistTwoCells = 500000;   // binary32: two tiles above

struct HistShared {
    unsigned int bins[kHistBins];
    long long edge[kHistBins + 1];   // bit patterns of the squared edges
    uint32_t queue[kHistBY][kHistQueue];
    double sx[5], sy[5];             // cell offsets (k - 2) wx, (k - 2) wy
};

template <typename T>
__device__ __forceinline__ void hist_begin(const Geometry& g, const double* __restrict__ edges2, HistShared& S) {
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    for (int b = tid; b < kHistBins; b += blockDim.x * blockDim.y) S.bins[b] = 0u;
    for (int b = tid; b <= kHistBins; b += blockDim.x * blockDim.y) S.edge[b] = __double_as_longlong(edges2[b]);
    if (tid < 10) {
        const int k = tid % 5;
        (tid < 5 ? S.sx : S.sy)[k] = (double)(k - 2) * (tid < 5 ? (double)Prm<T>::wx(g) : (double)Prm<T>::wy(g));
    }
    __syncthreads();
}

__device__ __forceinline__ void hist_end(HistShared& S, unsigned long long* __restrict__ hist) {
    __syncthreads();
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    for (int b = tid; b < kHistBins; b += blockDim.x * blockDim.y)
        if (S.bins[b]) atomicAdd(&hist[b], (unsigned long long)S.bins[b]);
}

// Candidate entry: source lane (5 bits), its slot i (2), the neighbour's slot
// j (2), dx + 2 (3), dy (2), 1 if the neighbour's disk comes first (1).
__device__ __forceinline__ uint32_t hist_entry(int lane, int b, int dx, int dy, int back) {
    return (uint32_t)lane | ((uint32_t)(b >> 2) << 5) | ((uint32_t)(b & 3) << 7) | ((uint32_t)(dx + 2) << 9) |
           ((uint32_t)dy << 12) | ((uint32_t)back << 14);
}

// Bins the first `count` queued pairs, one per lane (warp-uniform call).
template <typename T>
__device__ __forceinline__ void hist_flush(const Geometry& g, const T* __restrict__ cells, HistShared& S, const uint32_t* sq,
                                           int count, int q, int bx, int hy, float sigf, float inv_drf) {
    const int lane = threadIdx.x;
    if (lane >= count) return;
    const uint32_t e = sq[lane];
    const int src = e & 31, i = (e >> 5) & 3, j = (e >> 7) & 3;
    const int dx = (int)((e >> 9) & 7) - 2, dy = (int)((e >> 12) & 3), back = (int)((e >> 14) & 1);
    const int hx = bx * kHistBX + src;
    const int cx = 2 * hx + (q & 1), cy = 2 * hy + (q >> 1);
    const T* own = cells + 8 * ((long long)q * g.cq + (long long)hy * g.hx + hx) + i;
    const T* nb = cells + 8 * storage_index(g, wrap(cx + dx, g.mx), wrap(cy + dy, g.my)) + j;
    const T* p = back ? nb : own;
    const T* r = back ? own : nb;
    const double ex = __dadd_rn(widen(__ldg(r)), S.sx[(back ? -dx : dx) + 2]);
    const double ey = __dadd_rn(widen(__ldg(r + 4)), S.sy[(back ? -dy : dy) + 2]);
    const double ddx = __dsub_rn(widen(__ldg(p)), ex), ddy = __dsub_rn(widen(__ldg(p + 4)), ey);
    const double r2 = __dadd_rn(__dmul_rn(ddx, ddx), __dmul_rn(ddy, ddy));
    const long long r2i = __double_as_longlong(r2);   // r2 >= +0
    if (r2i >= S.edge[0] && r2i < S.edge[kHistBins]) {
        // bin b: edge[b] <= r2 < edge[b+1]; start from a binary32 estimate
        const float r2f = approx_f32(r2);
        int bb = (int)((r2f * rsqrtf(r2f) - sigf) * inv_drf);
        bb = bb < 0 ? 0 : (bb > kHistBins - 1 ? kHistBins - 1 : bb);
        while (bb > 0 && r2i < S.edge[bb]) --bb;
        while (bb < kHistBins - 1 && r2i >= S.edge[bb + 1]) ++bb;
        atomicAdd(&S.bins[bb], 1u);
    }
}

// The pairs of one tile of kHistBX x kHistBY cells of set q.
template <typename T>
__device__ __forceinline__ void hist_tile(const Geometry& g, const T* __restrict__ cells, HistShared& S, int bx, int by, int q) {
    const int lane = threadIdx.x;
    const int hx = bx * kHistBX + threadIdx.x;
    const int hy = by * kHistBY + threadIdx.y;
    const int cx = 2 * hx + (q & 1), cy = 2 * hy + (q >> 1);
    // first disks lie in rows slo..shi; a strip's two halo rows below its own
    // are looked at for the pairs whose first disk is the one ahead
    const bool live = hx < g.hx && hy < g.hy && cy >= max(g.slo - 2, 0) && cy <= g.shi;
    const bool mine = live && cy >= g.slo;
    uint32_t* sq = S.queue[threadIdx.y];
    Cell<T> own;
#pragma unroll
    for (int j = 0; j < 4; ++j) own.x[j] = own.y[j] = T(kEmpty);
    if (live) load_cell_ro(cells + 8 * ((long long)q * g.cq + (long long)hy * g.hx + hx), own);
    if (!__any_sync(0xffffffffu, Prm<T>::ge0(own.x[0]))) return;
    const bool own23 = __any_sync(0xffffffffu, Prm<T>::ge0(own.x[2]));
    const float wxf = g.wxf, wyf = g.wyf;
    const float sigf = (float)g.sigma, inv_drf = 1.0f / ((float)kHistDr * sigf);
    const float rmax = sigf * (1.0f + kHistBins * (float)kHistDr) * (1.0f + 1.0e-6f);
    const float thr = rmax * rmax * 1.001f;   // binary32 estimate margin (estimate error < 1e-6)
    const f2x nt = pk(-thr, -thr);
    float ox[4], oy[4];
    float minx = 3.0e38f, maxx = -3.0e38f, maxy = -3.0e38f;
    uint32_t occupied = 0;   // bits 4i..4i+3 set when own slot i holds a disk
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        ox[i] = to_f32(own.x[i]);
        oy[i] = to_f32(own.y[i]);
        if (Prm<T>::ge0(own.x[i])) {
            occupied |= 0xFu << (4 * i);
            minx = fminf(minx, ox[i]);
            maxx = fmaxf(maxx, ox[i]);
            maxy = fmaxf(maxy, oy[i]);
        }
    }
    // is a cell two steps away within reach of some lane's disks (margin far above the binary32 roundings)
    const float reach = rmax * (1.0f + 1.0e-4f);
    const bool left2 = __any_sync(0xffffffffu, minx + wxf < reach);
    const bool right2 = __any_sync(0xffffffffu, 2.0f * wxf - maxx < reach);
    const bool up2 = __any_sync(0xffffffffu, 2.0f * wyf - maxy < reach);
    int qn = 0;   // queued candidates of this warp (warp-uniform)
    for (int dy = 0; dy <= (up2 ? 2 : 1); ++dy) {
        const int ny = wrap(cy + dy, g.my);
        const bool theirs = ny >= g.slo && ny <= g.shi;
        // corner cells begin sqrt(wx^2 + wy^2) >= 1.41 sigma away
        const int dx0 = dy == 0 ? 0 : (left2 && dy < 2 ? -2 : -1), dx1 = right2 && dy < 2 ? 2 : 1;
        for (int dx = dx0; dx <= dx1; ++dx) {
            Cell<T> c;
#pragma unroll
            for (int j = 0; j < 4; ++j) c.x[j] = c.y[j] = T(kEmpty);
            if (live) load_cell_ro(cells + 8 * storage_index(g, wrap(cx + dx, g.mx), ny), c);
            const float sxf = (float)dx * wxf, syf = (float)dy * wyf;
            const f2x qx01 = add2(pk(to_f32(c.x[0]), to_f32(c.x[1])), pk(sxf, sxf));
            const f2x qx23 = add2(pk(to_f32(c.x[2]), to_f32(c.x[3])), pk(sxf, sxf));
            const f2x qy01 = add2(pk(to_f32(c.y[0]), to_f32(c.y[1])), pk(syf, syf));
            const f2x qy23 = add2(pk(to_f32(c.y[2]), to_f32(c.y[3])), pk(syf, syf));
            const bool c23 = __any_sync(0xffffffffu, Prm<T>::ge0(c.x[2]));
            uint32_t cand = 0;   // bit 4i+j: pair (own i, neighbour slot j) passes the estimate
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (i >= 2 && !own23) continue;
                const f2x tx2 = pk(ox[i], ox[i]), ty2 = pk(oy[i], oy[i]);
                f2x z = zpair(tx2, ty2, qx01, qy01, nt);
                cand |= ((lo32(z) >> 31) << (4 * i)) | ((hi32(z) >> 31) << (4 * i + 1));
                if (c23) {
                    z = zpair(tx2, ty2, qx23, qy23, nt);
                    cand |= ((lo32(z) >> 31) << (4 * i + 2)) | ((hi32(z) >> 31) << (4 * i + 3));
                }
            }
            // empty own slots are excluded (two empty slots sit one cell offset
            // apart), and no disk is paired with itself; pairs inside the cell
            // appear in both orders already
            cand &= occupied;
            const bool self = dx == 0 && dy == 0;
            if (self) cand &= ~0x8421u;
            for (;;) {   // queue the candidates, one per lane and round
                const bool more = cand != 0;
                if (!__any_sync(0xffffffffu, more)) break;
                const unsigned fwd = __ballot_sync(0xffffffffu, more && mine);
                const unsigned rev = __ballot_sync(0xffffffffu, more && theirs && !self);
                if (more) {
                    const int b = __ffs(cand) - 1;
                    cand &= cand - 1;
                    const unsigned below = (1u << lane) - 1u;
                    if (mine) sq[qn + __popc(fwd & below)] = hist_entry(lane, b, dx, dy, 0);
                    if (theirs && !self) sq[qn + __popc(fwd) + __popc(rev & below)] = hist_entry(lane, b, dx, dy, 1);
                }
                qn += __popc(fwd) + __popc(rev);
                while (qn >= 32) {
                    __syncwarp();
                    hist_flush<T>(g, cells, S, sq + (qn - 32), 32, q, bx, hy, sigf, inv_drf);
                    qn -= 32;
                    __syncwarp();
                }
            }
        }
    }
    __syncwarp();
    hist_flush<T>(g, cells, S, sq, qn, q, bx, hy, sigf, inv_drf);
    __syncwarp();
}

template <typename T, int TILES>
__global__ void __launch_bounds__(kHistBX * kHistBY)
k_hist(const Geometry g, const T* __restrict__ cells, const double* __restrict__ edges2,
       unsigned long long* __restrict__ hist) {
    __shared__ HistShared S;
    hist_begin<T>(g, edges2, S);
#pragma unroll 1
    for (int t = 0; t < TILES; ++t) hist_tile<T>(g, cells, S, blockIdx.x, blockIdx.y * TILES + t, blockIdx.z);
    hist_end(S, hist);
}

// ---- bond-orientational order psi_6 (Sec. 3.3's order parameter) -------------------------
// Neighbours k of disk j: the other disks closer than r_cut (r_cut <= 2 w, so
// the 5x5 neighbourhood holds them); psi_6(j) = (1/n_j) sum_k z^6 / (|z|^2)^3,
// z = dx + i dy from cell-local coordinates as in the histogram, 0 without
// neighbours.  Pairs in the order dy, dx, slot and every binary64 operation
// explicitly rounded, so psi_6(j) is the same number whatever the launch.
//
// The binary64 pipe binds this kernel (1/64 of the binary32 rate, about 50
// binary64 instructions per neighbour), so it is given only neighbours, and
// full warps of them: a binary32 estimate with a margin above its error
// selects each disk's candidates (6 of the 23 disks of 25 cells at r_cut =
// 1.4 sigma) into a list per lane; the lists of a warp are laid end to end
// and evaluated 32 at a time, and each lane then adds its own terms up in
// list order, which is the order dy, dx, slot.  Coordinates are widened to
// binary64 on the integer pipe.  N = 1M, phi = 0.716, r_cut = 1.4 sigma,
// binary32, psi_6 alone: 3.21 -> 0.80 ms (the pair loop
// in binary64 over every disk of the 25 cells had 18.7 of 32 lanes active).
// One thread per cell, one warp per 32 cells of a set row; block sums of
// {re, im, |psi_6|, n} in a fixed order to partial[4 * block]; k_psi6_sum adds
// them up, so that the host reads four numbers.
constexpr int kPsiBX = 32, kPsiBY = 4;
constexpr int kPsiList = 32;    // candidates a lane holds; a cell adds at most 16
constexpr int kPsiFlat = 256;   // terms evaluated between two rounds of sums

// 2 v exactly as __dmul_rn(2.0, v) gives it, on the integer pipe (v finite
// and far below overflow; a subnormal v, not met in earnest, is multiplied).
__device__ __forceinline__ double twice(double v) {
    const uint32_t hi = (uint32_t)__double2hiint(v), e = hi & 0x7FF00000u;
    if (e == 0u) return __dmul_rn(2.0, v);
    return __hiloint2double((int)(hi + 0x00100000u), __double2loint(v));
}

struct PsiShared {
    uint16_t list[kPsiList][kPsiBX];   // entry: own slot (2 bits), slot (2), dx + 2 (3), dy + 2 (3)
    uint32_t flat[kPsiFlat];           // entry | lane << 10, bit 31 set once found within r_cut
    double2 term[kPsiFlat];            // z^6 / |z|^6
};

// Evaluates the warp's listed candidates and adds each lane's terms to its
// disks' sums in list order (warp-uniform call).
template <typename T>
__device__ __forceinline__ void psi6_flush(const Geometry& g, const T* __restrict__ cells, PsiShared& s, int count,
                                           long long own0, int cx0, int cy, double rc2, const double* shx,
                                           const double* shy, double are[4], double aim[4], int nb[4]) {
    const int lane = threadIdx.x;
    int first = count;   // exclusive prefix sum of the counts
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, first, o);
        first += lane >= o ? v : 0;
    }
    const int total = __shfl_sync(0xffffffffu, first, 31);
    first -= count;
    for (int base = 0; base < total; base += kPsiFlat) {
        const int k0 = max(0, base - first), k1 = min(count, base + kPsiFlat - first);   // my share of this part
        for (int k = k0; k < k1; ++k) s.flat[first + k - base] = (uint32_t)s.list[k][lane] | ((uint32_t)lane << 10);
        __syncwarp();
        const int n = min(kPsiFlat, total - base);
        for (int f = lane; f < n; f += 32) {
            const uint32_t e = s.flat[f];
            const int i = e & 3, j = (e >> 2) & 3, dx = (int)((e >> 4) & 7) - 2, dy = (int)((e >> 7) & 7) - 2;
            const int src = (e >> 10) & 31;
            const T* own = cells + 8 * (own0 + src);
            const T* q = cells + 8 * storage_index(g, wrap(cx0 + 2 * src + dx, g.mx), wrap(cy + dy, g.my));
            const double ddx = __dsub_rn(widen(__ldg(own + i)), __dadd_rn(widen(__ldg(q + j)), shx[dx + 2]));
            const double ddy = __dsub_rn(widen(__ldg(own + 4 + i)), __dadd_rn(widen(__ldg(q + 4 + j)), shy[dy + 2]));
            const double xx = __dmul_rn(ddx, ddx), yy = __dmul_rn(ddy, ddy);
            const double r2 = __dadd_rn(xx, yy);
            // r2 >= +0 and rc2 > 0: their bit patterns order as they do
            if (__double_as_longlong(r2) < __double_as_longlong(rc2)) {
                const double ar = __dsub_rn(xx, yy);   // z^2
                const double ai = twice(__dmul_rn(ddx, ddy));
                const double br = __dsub_rn(__dmul_rn(ar, ddx), __dmul_rn(ai, ddy));   // z^3
                const double bi = __dadd_rn(__dmul_rn(ar, ddy), __dmul_rn(ai, ddx));
                const double zr = __dsub_rn(__dmul_rn(br, br), __dmul_rn(bi, bi));   // z^6
                const double zi = twice(__dmul_rn(br, bi));
                const double r6 = __dmul_rn(__dmul_rn(r2, r2), r2);
                s.term[f] = make_double2(__ddiv_rn(zr, r6), __ddiv_rn(zi, r6));
                s.flat[f] = e | 0x80000000u;
            }
        }
        __syncwarp();
        for (int k = k0; k < k1; ++k) {
            const uint32_t e = s.flat[first + k - base];
            if (e >> 31) {
                const int i = e & 3;
                const double2 t = s.term[first + k - base];
                const double r = __dadd_rn(pick(are, i), t.x), m = __dadd_rn(pick(aim, i), t.y);
                put_if(are, i, r, true);
                put_if(aim, i, m, true);
                put_if(nb, i, pick(nb, i) + 1, true);
            }
        }
        __syncwarp();
    }
}

template <typename T>
__global__ void __launch_bounds__(kPsiBX * kPsiBY)
k_psi6(const Geometry g, const T* __restrict__ cells, double rc2, double* __restrict__ psi,
       double* __restrict__ partial) {
    __shared__ PsiShared sh[kPsiBY];
    __shared__ double red[kPsiBY][3];
    __shared__ int redn[kPsiBY];
    __shared__ double shx[5], shy[5];   // cell offsets (dx - 2) wx, (dy - 2) wy
    const int lane = threadIdx.x;
    const int q = blockIdx.z;
    const int hx = blockIdx.x * kPsiBX + lane, hy = blockIdx.y * kPsiBY + threadIdx.y;
    if (threadIdx.y == 0 && lane < 10) {
        const int k = lane % 5;
        const double w = lane < 5 ? (double)Prm<T>::wx(g) : (double)Prm<T>::wy(g);
        (lane < 5 ? shx : shy)[k] = (double)(k - 2) * w;
    }
    __syncthreads();
    const bool live = hx < g.hx && hy < g.hy;
    const int cx = 2 * hx + (q & 1), cy = 2 * hy + (q >> 1);
    const long long own0 = (long long)q * g.cq + (long long)hy * g.hx + (long long)blockIdx.x * kPsiBX;
    Cell<T> own;
#pragma unroll
    for (int j = 0; j < 4; ++j) own.x[j] = own.y[j] = T(kEmpty);
    if (live) load_cell_ro(cells + 8 * (own0 + lane), own);
    double are[4] = {0, 0, 0, 0}, aim[4] = {0, 0, 0, 0};
    int nb[4] = {0, 0, 0, 0};
    if (__any_sync(0xffffffffu, Prm<T>::ge0(own.x[0]))) {
        PsiShared& s = sh[threadIdx.y];
        const float wxf = (float)Prm<T>::wx(g), wyf = (float)Prm<T>::wy(g);
        // estimate: |error of a difference| < 1e-6 (wx + wy), below the margin on r_cut
        const float rcf = sqrtf((float)rc2) * 1.00001f + 1.0e-5f * (wxf + wyf);
        const f2x nt = pk(-rcf * rcf, -rcf * rcf);
        const bool own23 = __any_sync(0xffffffffu, Prm<T>::ge0(own.x[2]));
        const bool corners = rcf * rcf > wxf * wxf + wyf * wyf;   // cells (+-2, +-2) start sqrt(wx^2 + wy^2) away
        float ox[4], oy[4];
        uint32_t occupied = 0;   // bits 4i..4i+3 set when own slot i holds a disk
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            ox[i] = to_f32(own.x[i]);
            oy[i] = to_f32(own.y[i]);
            occupied |= Prm<T>::ge0(own.x[i]) ? (0xFu << (4 * i)) : 0u;
        }
        int count = 0;
        for (int dy = -2; dy <= 2; ++dy) {
            const int ny = wrap(cy + dy, g.my);
            for (int dx = -2; dx <= 2; ++dx) {
                if (!corners && (dx == -2 || dx == 2) && (dy == -2 || dy == 2)) continue;
                Cell<T> c;
#pragma unroll
                for (int j = 0; j < 4; ++j) c.x[j] = c.y[j] = T(kEmpty);
                if (live) load_cell_ro(cells + 8 * storage_index(g, wrap(cx + dx, g.mx), ny), c);
                const float sxf = (float)dx * wxf, syf = (float)dy * wyf;
                const f2x qx01 = add2(pk(to_f32(c.x[0]), to_f32(c.x[1])), pk(sxf, sxf));
                const f2x qx23 = add2(pk(to_f32(c.x[2]), to_f32(c.x[3])), pk(sxf, sxf));
                const f2x qy01 = add2(pk(to_f32(c.y[0]), to_f32(c.y[1])), pk(syf, syf));
                const f2x qy23 = add2(pk(to_f32(c.y[2]), to_f32(c.y[3])), pk(syf, syf));
                const bool c23 = __any_sync(0xffffffffu, Prm<T>::ge0(c.x[2]));
                uint32_t cand = 0, there = 0;   // bit 4i+j: pair (own i, neighbour slot j)
#pragma unroll
                for (int j = 0; j < 4; ++j) there |= Prm<T>::ge0(c.x[j]) ? (0x1111u << j) : 0u;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (i >= 2 && !own23) continue;
                    const f2x tx2 = pk(ox[i], ox[i]), ty2 = pk(oy[i], oy[i]);
                    f2x z = zpair(tx2, ty2, qx01, qy01, nt);
                    cand |= ((lo32(z) >> 31) << (4 * i)) | ((hi32(z) >> 31) << (4 * i + 1));
                    if (c23) {
                        z = zpair(tx2, ty2, qx23, qy23, nt);
                        cand |= ((lo32(z) >> 31) << (4 * i + 2)) | ((hi32(z) >> 31) << (4 * i + 3));
                    }
                }
                cand &= occupied & there;
                if (dx == 0 && dy == 0) cand &= ~0x8421u;
                const uint32_t tag = ((uint32_t)(dx + 2) << 4) | ((uint32_t)(dy + 2) << 7);
                while (cand) {
                    const int b = __ffs(cand) - 1;
                    cand &= cand - 1;
                    s.list[count++][lane] = (uint16_t)(tag | (uint32_t)(b >> 2) | ((uint32_t)(b & 3) << 2));
                }
                if (__any_sync(0xffffffffu, count > kPsiList - 16)) {
                    psi6_flush<T>(g, cells, s, count, own0, cx - 2 * lane, cy, rc2, shx, shy, are, aim, nb);
                    count = 0;
                }
            }
        }
        psi6_flush<T>(g, cells, s, count, own0, cx - 2 * lane, cy, rc2, shx, shy, are, aim, nb);
    }
    // psi_6 of the warp's disks, laid end to end so that the divisions and
    // square roots run with full warps too
    double t[3] = {0, 0, 0};   // re, im, |psi_6|
    int tn = 0;                // neighbours
    {
        PsiShared& s = sh[threadIdx.y];
        int total = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const bool used = Prm<T>::ge0(own.x[i]);
            const unsigned m = __ballot_sync(0xffffffffu, used);
            if (used) {
                const int k = total + __popc(m & ((1u << lane) - 1u));
                s.term[k] = make_double2(are[i], aim[i]);
                s.flat[k] = (uint32_t)lane | ((uint32_t)i << 5) | ((uint32_t)nb[i] << 8);
                tn += nb[i];
            }
            total += __popc(m);
        }
        __syncwarp();
        for (int k = lane; k < total; k += 32) {
            const uint32_t e = s.flat[k];
            const double2 a = s.term[k];
            const int n = (int)(e >> 8);
            double pr = 0.0, pi = 0.0;
            if (n > 0) {
                pr = __ddiv_rn(a.x, (double)n);
                pi = __ddiv_rn(a.y, (double)n);
                t[0] = __dadd_rn(t[0], pr);
                t[1] = __dadd_rn(t[1], pi);
                t[2] = __dadd_rn(t[2], __dsqrt_rn(__dadd_rn(__dmul_rn(pr, pr), __dmul_rn(pi, pi))));
            }
            if (psi) {
                const long long cc = (long long)cy * g.mx + (cx - 2 * lane + 2 * (int)(e & 31));
                const int i = (int)((e >> 5) & 3);
                psi[(4 * cc + i) * 2] = pr;
                psi[(4 * cc + i) * 2 + 1] = pi;
            }
        }
        if (psi && live) {   // unused slots
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (!Prm<T>::ge0(own.x[i])) {
                    const long long cc = (long long)cy * g.mx + cx;
                    psi[(4 * cc + i) * 2] = 0.0;
                    psi[(4 * cc + i) * 2 + 1] = 0.0;
                }
        }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k)
        for (int o = 16; o > 0; o >>= 1) t[k] = __dadd_rn(t[k], __shfl_down_sync(0xffffffffu, t[k], o));
    tn = __reduce_add_sync(0xffffffffu, tn);
    if (lane == 0) {
        for (int k = 0; k < 3; ++k) red[threadIdx.y][k] = t[k];
        redn[threadIdx.y] = tn;
    }
    __syncthreads();
    if (lane < 4 && threadIdx.y == 0) {
        const long long b = ((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
        double v = 0.0;
        int n = 0;
        for (int w = 0; w < kPsiBY; ++w) {
            if (lane < 3) v = __dadd_rn(v, red[w][lane]);
            n += redn[w];
        }
        partial[4 * b + lane] = lane < 3 ? v : (double)n;
    }
}

// Sums of the nb block sums into out[0..3], in an order fixed by nb alone
// (one block; out does not overlap the partials).
static __global__ void __launch_bounds__(256) k_psi6_sum(const double* __restrict__ partial, unsigned nb,
                                                         double* __restrict__ out) {
    __shared__ double red[256];
    const int k = threadIdx.x & 3;
    double v = 0.0;
    for (unsigned b = threadIdx.x >> 2; b < nb; b += 64) v = __dadd_rn(v, partial[4 * (size_t)b + k]);
    red[threadIdx.x] = v;
    for (int o = 128; o >= 4; o >>= 1) {
        __syncthreads();
        if (threadIdx.x < o) red[threadIdx.x] = __dadd_rn(red[threadIdx.x], red[threadIdx.x + o]);
    }
    if (threadIdx.x < 4) out[k] = red[k];
}

// ---- batched replicas ------------------------------------------------------------------
// Every stage is one launch over all replicas of a batch: the launch's flat
// block index is mapped to (replica, local block) by a per-stage table, and
// each replica keeps its own geometry, cells, draws, device state,
// counters and histogram.  Replica r's cells start at cell rd.cell_off of
// the arena; its sweep draws of chunk position j sit at draws[j*R + r].
// NSEL > 0: every replica makes NSEL trial moves per cell update.
// Launched as programmatic dependents like the single system's kernels, the
// directions drawn ahead: 64 sweeps of the 64-replica workload at n_M = 8 28.6
// -> 25.9 ms (27.1 with the loads first), of 16 replicas of 1024 to 8192 disks
// 1.37 -> 1.08 ms.
template <int ROWS, bool TRACK, bool DENSE = false, int NSEL = 0>
static __global__ void __launch_bounds__(32 * ROWS, DENSE ? (16 / ROWS > 0 ? 16 / ROWS : 1) : 20 / ROWS)
k_subsweep_f32_batch(const ReplicaDesc* __restrict__ reps, const unsigned short* __restrict__ map,
                     float* __restrict__ arena, const SweepDraw* __restrict__ draws, int R, int j, int k,
                     unsigned long long* __restrict__ partial, double* __restrict__ msd) {
    pdl_release();
    __shared__ float2 sdir[kDirRows][32 * ROWS];
    const int r = map[blockIdx.x];
    const ReplicaDesc* rd = reps + r;
    const int local = (int)blockIdx.x - rd->sub_block0;
    const int by = local / rd->sub_gx, bx = local - by * rd->sub_gx;
    subsweep_f32<ROWS, NSEL, TRACK, DENSE, true>(rd->g, arena + 8 * rd->cell_off, draws + (size_t)j * R + r, k, bx, by,
                                     partial + 4 * (rd->part_off + local), sdir, msd + r);
}

// Binary64: G lanes per cell, a block of G warps per set row and four rows; or
// one thread per cell (launch_subsweep_f64_batch).
template <int G>
static __global__ void __launch_bounds__(128 * G)
k_subsweep_lanes_batch(const ReplicaDesc* __restrict__ reps, const unsigned short* __restrict__ map,
                     double* __restrict__ arena, const SweepDraw* __restrict__ draws, int R, int j, int k,
                     unsigned long long* __restrict__ partial) {
    pdl_release();
    __shared__ Warp2<G> sw[4 * G];
    const int r = map[blockIdx.x];
    const ReplicaDesc* rd = reps + r;
    const int local = (int)blockIdx.x - rd->sub_block0;
    const int by = local / rd->sub_gx, bx = local - by * rd->sub_gx;
    const int row = threadIdx.y / G, part = threadIdx.y % G;
    subsweep_lanes<G>(rd->g, arena + 8 * rd->cell_off, draws + (size_t)j * R + r, k, bx * 32 + part * (32 / G),
                              by * 4 + row, partial + 4 * (rd->part_off + local), sw[threadIdx.y]);
}

template <int NSEL>
static __global__ void __launch_bounds__(128, 4)
k_subsweep_f64_batch(const ReplicaDesc* __restrict__ reps, const unsigned short* __restrict__ map,
                     double* __restrict__ arena, const SweepDraw* __restrict__ draws, int R, int j, int k,
                     unsigned long long* __restrict__ partial) {
    pdl_release();
    __shared__ uint4 sdir[kDirRows64][128];
    const int r = map[blockIdx.x];
    const ReplicaDesc* rd = reps + r;
    const int local = (int)blockIdx.x - rd->sub_block0;
    const int by = local / rd->sub_gx, bx = local - by * rd->sub_gx;
    subsweep_f64<4, NSEL>(rd->g, arena + 8 * rd->cell_off, draws + (size_t)j * R + r, k, bx, by,
                          partial + 4 * (rd->part_off + local), sdir);
}

template <typename T, bool EARLY>
__global__ void __launch_bounds__(kShiftBX * kShiftBY)
k_shift_batch(const ReplicaDesc* __restrict__ reps, const unsigned short* __restrict__ map,
              const T* src, T* dst, const SweepDraw* __restrict__ draws, int R, int j,
              DevState* __restrict__ sts) {
    pdl_release();
    pdl_wait();
    const int r = map[blockIdx.x];
    const ReplicaDesc* rd = reps + r;
    const int local = (int)blockIdx.x - rd->sh_block0;
    const int q = local & 3, rem = local >> 2;   // the four sets of a tile in adjacent blocks
    const int by = rem / rd->sh_gx, bx = rem - by * rd->sh_gx;
    shift_cells<T, EARLY>(rd->g, src + 8 * rd->cell_off, dst + 8 * rd->cell_off, draws + (size_t)j * R + r, sts + r, bx,
                   by, q);
}

template <typename T>
__global__ void __launch_bounds__(kHistBX * kHistBY)
k_hist_batch(const ReplicaDesc* __restrict__ reps, const unsigned short* __restrict__ map,
             const T* __restrict__ arena, const double* __restrict__ edges2, unsigned long long* __restrict__ hist) {
    const int r = map[blockIdx.x];
    const ReplicaDesc* rd = reps + r;
    const int local = (int)blockIdx.x - rd->hi_block0;
    const int per_set = rd->hi_gx * rd->hi_gy;
    const int q = local / per_set, rem = local - q * per_set;
    const int by = rem / rd->hi_gx, bx = rem - by * rd->hi_gx;
    __shared__ HistShared S;
    hist_begin<T>(rd->g, edges2, S);
    hist_tile<T>(rd->g, arena + 8 * rd->cell_off, S, bx, by, q);
    hist_end(S, hist + (size_t)r * kHistBins);
}

// ---- launchers ---------------------------------------------------------------------
inline dim3 set_grid(const Geometry& g, dim3 block) {
    return dim3((unsigned)((g.hx + block.x - 1) / block.x), (unsigned)((g.hy + block.y - 1) / block.y), 4u);
}

template <typename T>
void launch_shift_t(const LaunchCtx& c, const void* src, void* dst, const SweepDraw* draw) {
    const dim3 block(kShiftBX, kShiftBY);
    const dim3 sg = set_grid(c.g, block);
    auto run = [&](auto kernel) {
        launch_on(c, kernel, dim3(4 * sg.x, sg.y, 1), block, c.g, reinterpret_cast<const T*>(src),
                  reinterpret_cast<T*>(dst), draw, c.st);
    };
    if constexpr (sizeof(T) == 8) {
        if (shift_early<T>(c.g.C)) return run(k_shift<T, true>);
    }
    run(k_shift<T, false>);
}

template <typename T>
void launch_psi6_t(const LaunchCtx& c, const void* cells, double rc2, double* psi, double* partial, double* out) {
    const dim3 block(kPsiBX, kPsiBY);
    const dim3 grid = set_grid(c.g, block);
    const unsigned nb = grid.x * grid.y * grid.z;
    k_psi6<T><<<grid, block, 0, c.stream>>>(c.g, reinterpret_cast<const T*>(cells), rc2, psi, partial);
    k_psi6_sum<<<1, 256, 0, c.stream>>>(partial, nb, out);
}

template <typename T>
void launch_hist_t(const LaunchCtx& c, const void* cells) {
    const dim3 block(kHistBX, kHistBY);
    const dim3 sg = set_grid(c.g, block);
    const T* a = reinterpret_cast<const T*>(cells);
    if constexpr (sizeof(T) == 4) {
        if (c.g.C > kHistTwoCells) {
            k_hist<T, 2><<<dim3(sg.x, (sg.y + 1) / 2, sg.z), block, 0, c.stream>>>(c.g, a, c.edges2, c.hist);
            return;
        }
    }
    k_hist<T, 1><<<sg, block, 0, c.stream>>>(c.g, a, c.edges2, c.hist);
}

// ---- snapshot check ---------------------------------------------------------------------
// Checks every cell of an incoming image (any storage order): occupied slots
// form a prefix, occupied coordinates lie in [0,wx) x [0,wy) of the
// coordinate type, unused slots hold kEmpty in both coordinates.  out[0]
// accumulates the number of disks, out[1] becomes non-zero on a bad cell.
template <typename T>
__global__ void __launch_bounds__(256) k_check_cells(const Geometry g, const T* __restrict__ cells,
                                                     unsigned long long* __restrict__ out) {
    const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
    unsigned n = 0;
    bool bad = false;
    if (i < g.C) {
        Cell<T> c;
        load_cell_ro(cells + 8 * i, c);
        bool empty_seen = false;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (c.x[j] == T(kEmpty) && c.y[j] == T(kEmpty)) {
                empty_seen = true;
            } else {
                bad |= empty_seen || !(c.x[j] >= T(0) && c.x[j] < Prm<T>::wx(g)) ||
                       !(c.y[j] >= T(0) && c.y[j] < Prm<T>::wy(g));
                ++n;
            }
        }
    }
    const unsigned tot = __reduce_add_sync(0xffffffffu, n);
    if (threadIdx.x % 32 == 0 && tot) atomicAdd(out, (unsigned long long)tot);
    if (bad) atomicOr(out + 1, 1ull);
}

template <typename T>
void launch_check_t(const LaunchCtx& c, const void* cells, unsigned long long* out) {
    const unsigned blocks = (unsigned)((c.g.C + 255) / 256);
    k_check_cells<T><<<blocks, 256, 0, c.stream>>>(c.g, reinterpret_cast<const T*>(cells), out);
}

}  // namespace hdmc
