// Tile binning without any depth order.
//
// The paper removes depth sorting because the blending sums of Eq. 2 commute
// (Sec. 2, Eq. 1 discussion; Sec. 3.1).  The lists built here are keyed by
// tile only -- a counting sort by tile:
//
//   0. the work plan, at the start of k_bin_count: every warp of the binning
//      grid (at most one 512-thread CTA per SM) takes an equal contiguous share
//      of the cost numbering of all rectangle rows, cut at row boundaries.
//      Preprocessing has summed the rows' costs (kRowCost plus the row's width
//      in tiles) per group of 32 consecutive Gaussians; each group adds a fixed
//      visit charge.
//   1. k_bin_count: each warp resolves its rows, 32 at a time (one per lane):
//      the tiles of a rectangle row that pass the FP32 tile test form one
//      interval (row_tiles), which is added to a per-CTA shared-memory
//      difference array (+1 at its first tile, -1 after its last); a prefix
//      sum per tile row turns those into the CTA's tile counts, and one
//      global atomicAdd per (CTA, tile) reserves the CTA's block inside the
//      tile and returns its base.
//   2. k_scan_order: exclusive scan of the per-tile totals -> tile offsets,
//      and the rasterisation order (longest lists first).
//   3. k_bin_scatter: the same warps resolve the same rows again and write
//      the rows' tiles (lane by lane, or spread over the warp when a batch
//      holds a long row) at offset[tile] + base[c][tile] + (shared-memory
//      rank).
//
// A pair is listed only if the FP32 tile test (tile_may_hit) allows an
// included pixel in the tile; its rectangle alone (the 3-sigma bounding
// square) would list many tiles a thin ellipse never reaches.  Resolving a
// row costs a handful of test evaluations instead of one per tile (the test
// is monotone along the row up to its vertex, see row_tiles).  Order within a
// tile follows the atomics and is not reproducible; the rasteriser does not
// depend on it beyond FP32 rounding.
#include <algorithm>

#include "mgs_internal.cuh"

namespace mgs {
namespace {

constexpr int kScanThreads = 1024;
// Count and scatter run one 512-thread CTA per SM at 64 registers a thread:
// half of the register file, so that the previous frame's rasteriser keeps
// two CTAs on the SM meanwhile.  Alone, more threads bin faster (600k at 1600x1063,
// 512 / 768 / 1024: count 0.052 / 0.041 / 0.040 ms, scatter 0.121 / 0.116 / 0.116),
// but frames in flight on several streams render faster this way (1030 / 1024 / 1026
// FPS, served 870 / 858 / 860 views/s).
constexpr int kBinThreads = 512;
constexpr int kBand = 32768;          // words per shared-memory band (128 KB)

__device__ __forceinline__ void rect_of(const uint2 r, int &x0, int &y0, int &w, int &h) {
    x0 = r.x & 0xFFFF;
    y0 = r.y & 0xFFFF;
    w = (int)(r.x >> 16) - x0;
    h = (int)((r.y & ~kRectWide) >> 16) - y0;
}

// FP32-contract tile test: may Gaussian (m, l) include a pixel centre of tile
// (tx, ty)?  Slab bounds at the tile centre with half extent 7.5 and a 2^-18
// relative margin, one correctly rounded operation per step (the oracle
// evaluates the identical sequence, so both build the same lists).  A tile
// that fails holds no pixel with q <= 9.
__device__ __forceinline__ bool tile_may_hit(float mx, float my, float l11, float l21, float l22,
                                             int tx, int ty) {
    const float h = 7.5f;
    const float bx = (float)(tx * kTile + 8), by = (float)(ty * kTile + 8);
    const float dxb = __fsub_rn(bx, mx);
    const float dyb = __fsub_rn(by, my);
    const float e1c = fabsf(__fmaf_rn(l11, dxb, __fmul_rn(l21, dyb)));
    const float h1 = __fmaf_rn(fabsf(l11), h, __fmul_rn(fabsf(l21), h));
    const float u2 = __fadd_rn(fabsf(dyb), h);
    const float s1 = __fadd_rn(__fmul_rn(fabsf(l11), __fadd_rn(fabsf(dxb), h)), __fmul_rn(fabsf(l21), u2));
    const float m1 = __fmul_rn(3.814697265625e-06f, __fadd_rn(s1, 4.0f));
    const float e2c = fabsf(__fmul_rn(l22, dyb));
    const float h2 = __fmul_rn(fabsf(l22), h);
    const float m2 = __fmul_rn(3.814697265625e-06f, __fadd_rn(__fmul_rn(fabsf(l22), u2), 4.0f));
    return __fsub_rn(e1c, h1) <= __fadd_rn(3.0f, m1) && __fsub_rn(e2c, h2) <= __fadd_rn(3.0f, m2);
}

// Row constants of the FP32 tile test for one tile row of one Gaussian:
// along the row only dxb = (tile centre x) - m_x changes.
struct RowTest {
    float mx, l11, P, h1, s12;   // P = l21 dyb, h1 = |l11| h + |l21| h, s12 = |l21| (|dyb| + h)
};
// e1c - h1 of tile tx (left-hand side of the test's first slab)
__device__ __forceinline__ float row_lhs(const RowTest &r, int tx) {
    const float dxb = __fsub_rn((float)(tx * kTile + 8), r.mx);
    return __fsub_rn(fabsf(__fmaf_rn(r.l11, dxb, r.P)), r.h1);
}
// l11 dxb + P of tile tx (its sign changes once along the row)
__device__ __forceinline__ float row_e1(const RowTest &r, int tx) {
    return __fmaf_rn(r.l11, __fsub_rn((float)(tx * kTile + 8), r.mx), r.P);
}
// 3 + m1 for |dxb| = adx (right-hand side of the first slab)
__device__ __forceinline__ float row_rhs(const RowTest &r, float adx) {
    const float s1 = __fadd_rn(__fmul_rn(fabsf(r.l11), __fadd_rn(adx, 7.5f)), r.s12);
    return __fadd_rn(3.0f, __fmul_rn(3.814697265625e-06f, __fadd_rn(s1, 4.0f)));
}
__device__ __forceinline__ int clamp_tile(float v, int lo, int hi) {
    return (int)fminf(fmaxf(v, (float)lo), (float)hi);   // NaN -> lo
}

// Smallest t in [lo, hi] with row_lhs(t) <= K, starting from `guess`; the
// predicate is false ... false true ... true on [lo, hi] and true at hi.
// A few steps from a good guess, else bisection.  *v: row_lhs at the result.
__device__ __forceinline__ int row_first(const RowTest &r, float K, int lo, int hi, int guess,
                                         float &v) {
    int t = min(max(guess, lo), hi);
    v = row_lhs(r, t);
    if (v <= K) {
        for (int s = 0; s < 4 && t > lo; ++s) {
            const float u = row_lhs(r, t - 1);
            if (!(u <= K)) return t;
            --t;
            v = u;
        }
        if (t == lo) return t;
        hi = t;
    } else {
        for (int s = 0; s < 4; ++s) {
            ++t;
            v = row_lhs(r, t);
            if (v <= K) return t;
        }
        lo = t + 1;
    }
    while (lo < hi) {   // bisection on [lo, hi], predicate true at hi
        const int m = (lo + hi) >> 1;
        if (row_lhs(r, m) <= K) hi = m;
        else lo = m + 1;
    }
    v = row_lhs(r, lo);
    return lo;
}
// Largest t in [lo, hi] with row_lhs(t) <= K (true ... true false ... false,
// true at lo).
__device__ __forceinline__ int row_last(const RowTest &r, float K, int lo, int hi, int guess,
                                        float &v) {
    int t = min(max(guess, lo), hi);
    v = row_lhs(r, t);
    if (v <= K) {
        for (int s = 0; s < 4 && t < hi; ++s) {
            const float u = row_lhs(r, t + 1);
            if (!(u <= K)) return t;
            ++t;
            v = u;
        }
        if (t == hi) return t;
        lo = t;
    } else {
        for (int s = 0; s < 4; ++s) {
            --t;
            v = row_lhs(r, t);
            if (v <= K) return t;
        }
        hi = t - 1;
    }
    while (lo < hi) {   // bisection on [lo, hi], predicate true at lo
        const int m = (lo + hi + 1) >> 1;
        if (row_lhs(r, m) <= K) lo = m;
        else hi = m - 1;
    }
    v = row_lhs(r, lo);
    return lo;
}

// The tiles of tile row ty inside rectangle columns [x0, x1) that pass
// tile_may_hit, as one interval [a, b] (a > b: none).  Returns false when it
// cannot establish that they form one interval; the caller then tests every
// tile of the row.
//
// Why an interval: along the row the test is  |l11 dxb + P| - h1 <= 3 + m1
// with dxb = fl(x - m_x).  Every operation is a correctly rounded, hence
// monotone, function of its inputs, so fl(l11 dxb + P) is monotone in the
// tile index, its absolute value falls and then rises, and for any fixed
// bound K the tiles with  fl(|.| - h1) <= K  form an interval.  The margin m1
// grows with |dxb| only, so on the rectangle it lies between its value at
// |dxb| = 0 and its value at the farther end: the tiles passing with the
// larger bound form an interval I_max, those passing with the smaller one an
// interval I_min inside it, and only the tiles of I_max \ I_min (none in
// practice: the bounds differ by 2^-18 relative) are tested one by one.  The
// second slab |l22 dyb| - h2 <= 3 + m2 is the same for the whole row.
// Most rows are settled by a certificate: the two tiles nearest the real
// crossings pass with the smaller bound and their outer neighbours fail with
// the larger one, so I_min = I_max = the tiles between them.
__device__ __forceinline__ bool row_tiles(float mx, float my, float l11, float l21, float l22, int x0,
                                       int x1, int ty, int &a, int &b) {
    a = 1;
    b = 0;
    const float h = 7.5f;
    const float dyb = __fsub_rn((float)(ty * kTile + 8), my);
    const float u2 = __fadd_rn(fabsf(dyb), h);
    const float e2c = fabsf(__fmul_rn(l22, dyb));
    const float h2 = __fmul_rn(fabsf(l22), h);
    const float m2 = __fmul_rn(3.814697265625e-06f, __fadd_rn(__fmul_rn(fabsf(l22), u2), 4.0f));
    if (!(__fsub_rn(e2c, h2) <= __fadd_rn(3.0f, m2))) return true;   // no tile of the row
    RowTest r;
    r.mx = mx;
    r.l11 = l11;
    r.P = __fmul_rn(l21, dyb);
    r.h1 = __fmaf_rn(fabsf(l11), h, __fmul_rn(fabsf(l21), h));
    r.s12 = __fmul_rn(fabsf(l21), u2);
    const int xl = x0, xr = x1 - 1;
    if (!(fabsf(l11) > 0.0f && fabsf(l11) < 3.0e38f && fabsf(r.P) < 3.0e38f && fabsf(mx) < 3.0e38f))
        return false;
    const float Kmin = row_rhs(r, 0.0f);
    const float Kmax = row_rhs(r, fmaxf(fabsf(__fsub_rn((float)(xl * kTile + 8), mx)),
                                        fabsf(__fsub_rn((float)(xr * kTile + 8), mx))));
    // real-valued crossings |l11 dxb + P| = h1 + Kmax around the vertex tz
    const float tz = (mx - 8.0f - r.P / l11) * 0.0625f;
    const float span = (r.h1 + Kmax) / fabsf(l11) * 0.0625f;
    {   // fast path: the tiles gl, gr pass and their outer neighbours fail, so
        // (I_max being an interval) I_max = [gl, gr]
        const int gl = clamp_tile(floorf(tz - span) + 1.0f, xl, xr);
        const int gr = clamp_tile(floorf(tz + span), xl, xr);
        if (gl <= gr) {
            const float vl = row_lhs(r, gl), vr = row_lhs(r, gr);
            const bool out_l = gl == xl || !(row_lhs(r, gl - 1) <= Kmax);
            const bool out_r = gr == xr || !(row_lhs(r, gr + 1) <= Kmax);
            if (vl <= Kmin && vr <= Kmin && out_l && out_r) {   // and I_min = I_max
                a = gl;
                b = gr;
                return true;
            }
        }
    }
    // vertex: the first tile t in [xl, xr + 1] at which l11 dxb + P has the
    // sign of l11 (xr + 1 counts as such); |.| is smallest at t or t - 1
    const float sg = l11 > 0.0f ? 1.0f : -1.0f;
    int t = clamp_tile(floorf(tz) + 1.0f, xl, xr + 1);
    if (t <= xr && row_e1(r, t) * sg >= 0.0f) {
        int s = 0;
        while (t > xl && row_e1(r, t - 1) * sg >= 0.0f) {
            --t;
            if (++s > 8) return false;
        }
    } else {
        int s = 0;
        while (t <= xr && !(row_e1(r, t) * sg >= 0.0f)) {
            ++t;
            if (++s > 8) return false;
        }
    }
    int tm;
    float vm;
    if (t > xr) {
        tm = xr;
        vm = row_lhs(r, xr);
    } else if (t == xl) {
        tm = xl;
        vm = row_lhs(r, xl);
    } else {
        const float v1 = row_lhs(r, t), v0 = row_lhs(r, t - 1);
        tm = v1 <= v0 ? t : t - 1;
        vm = fminf(v1, v0);
    }
    if (!(vm <= Kmax)) return true;   // the lowest point fails even the larger bound
    // I_max from guesses at the real crossings
    float va, vb;
    const int a2 = row_first(r, Kmax, xl, tm, clamp_tile(floorf(tz - span) + 1.0f, xl, tm), va);
    const int b2 = row_last(r, Kmax, tm, xr, clamp_tile(floorf(tz + span), tm, xr), vb);
    if (va <= Kmin && vb <= Kmin) {   // I_min = I_max: every tile of [a2, b2] passes
        a = a2;
        b = b2;
        return true;
    }
    // band tiles: test them one by one; together with I_min they must form one run
    if (b2 - a2 > 64) return false;
    int first = -1, last = -2, runs = 0;
    bool prev = false;
    for (int x = a2; x <= b2; ++x) {
        const float v = row_lhs(r, x);
        const bool p = v <= Kmin || (v <= Kmax && tile_may_hit(mx, my, l11, l21, l22, x, ty));
        if (p && !prev) {
            ++runs;
            if (first < 0) first = x;
        }
        if (p) last = x;
        prev = p;
    }
    if (runs > 1) return false;
    if (runs == 1) {
        a = first;
        b = last;
    }
    return true;
}

// Plan cost of a rectangle row: kRowCost plus its width (mgs_internal.cuh), summed per
// group by preprocessing.

// Cost of a group in the work plan beyond its rows: a fixed charge for
// visiting it (loading its 32 rectangles, the scans and the row split), so
// that shares over sparse stretches of the scene (many Gaussians with one
// or two rows each) stay short.  Measured on the 600k benchmark view with the
// row certificate: a visit charge of 1024 with a row cost of 3 balanced the
// warps best among 256 ... 1536 and 3 ... 8 (a visit costs about as much as a
// hundred rows).
constexpr int kGroupCost = 1024;

// A lane's Gaussian of a group: rectangle and cull geometry, loaded together
// (the geometry of a Gaussian without a rectangle is loaded but never used),
// one group ahead of its use.
struct GroupLoad {
    uint2 r;
    float4 a;
    float l22;
};
__device__ __forceinline__ GroupLoad load_group(const uint2 *__restrict__ rect,
                                                const ProjRec *__restrict__ rec, int64_t n,
                                                int64_t g0) {
    GroupLoad L{make_uint2(0u, 0u), make_float4(0.f, 0.f, 0.f, 0.f), 0.f};
    const int64_t i = g0 + (threadIdx.x & 31);
    if (i < n) {
        L.r = __ldg(&rect[i]);
        L.a = __ldg(&rec[i].a);
        L.l22 = __ldg(&rec[i].b.x);
    }
    return L;
}

// One row handed to a row callback: Gaussian gid, tile row ty, rectangle
// columns [x0, x1), cull geometry, wide flag.
struct RowItem {
    uint32_t gid;
    int ty, x0, x1;
    float mx, my, l11, l21, l22;
    bool wide;
};

// Rows wait in a per-warp queue in shared memory (kQueue slots)
// until 32 of them fill a batch, so that sparse groups (a few visible
// Gaussians with one or two rows) still give every lane a row.
constexpr int kQueue = 64;

// A queued row: {gid, ty | wide << 31, x0 | x1 << 16, l22} and {m_x, m_y, l11, l21}.
struct RowSlot {
    uint4 u;
    float4 g;
};

// Calls f(active, item) with queued rows [qh, qh + cnt) (cnt <= 32), one per
// lane; every lane calls f.
template <class F>
__device__ __forceinline__ void run_rows(const RowSlot *q, int qh, int cnt, F &&f) {
    const int lane = threadIdx.x & 31;
    RowItem it{};
    const bool active = lane < cnt;
    if (active) {
        const RowSlot e = q[(qh + lane) & (kQueue - 1)];
        it.gid = e.u.x;
        it.ty = (int)(e.u.y & 0x7FFFFFFFu);
        it.wide = (e.u.y >> 31) != 0u;
        it.x0 = (int)(e.u.z & 0xFFFFu);
        it.x1 = (int)(e.u.z >> 16);
        it.l22 = __uint_as_float(e.u.w);
        it.mx = e.g.x;
        it.my = e.g.y;
        it.l11 = e.g.z;
        it.l21 = e.g.w;
    }
    f(active, it);
}

// Queues the rows of the group at g0 (Gaussians g0 .. g0 + 31, one per lane)
// whose start cost lies in [ca, cb) of the group's row cost numbering
// (Gaussian after Gaussian, rows top to bottom, row k of Gaussian i starting
// at cost excl_i + k (kRowCost + w_i)), and runs every full batch of 32.
template <class F>
__device__ __forceinline__ void warp_rows(const GroupLoad &L, int64_t g0, int ca, int cb,
                                          RowSlot *q, int &qh, int &qn, F &&f) {
    const int lane = threadIdx.x & 31;
    int x0 = 0, y0 = 0, w = 0, h = 0;
    rect_of(L.r, x0, y0, w, h);
    const bool wide = (L.r.y & kRectWide) != 0;
    const int rc = kRowCost + w;
    const int c = (w > 0 && h > 0) ? h * rc : 0;
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    const int excl = incl - c;
    // rows k with ca <= excl + k rc < cb
    int r0 = 0, nr = 0;
    if (c > 0) {
        r0 = ca > excl ? (ca - excl + rc - 1) / rc : 0;
        const int r1 = cb >= incl ? h : (cb > excl ? min((cb - excl + rc - 1) / rc, h) : 0);
        nr = max(r1 - r0, 0);
    }
    int rincl = nr;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, rincl, o);
        if (lane >= o) rincl += y;
    }
    const int rexcl = rincl - nr;
    const int R = __shfl_sync(0xffffffffu, rincl, 31);
    const int ybase = y0 + r0 - rexcl;   // row of index p for this lane: ybase + p
    for (int base = 0; base < R; base += 32) {
        const int p = base + lane;
        // owner: the largest lane whose exclusive prefix is <= p
        int lo = 0;
#pragma unroll
        for (int step = 16; step > 0; step >>= 1) {
            const int e = __shfl_sync(0xffffffffu, rexcl, lo + step);
            if (e <= p) lo += step;
        }
        const int ty = __shfl_sync(0xffffffffu, ybase, lo) + p;
        const uint32_t xw = __shfl_sync(0xffffffffu, (uint32_t)x0 | ((uint32_t)(x0 + w) << 16) |
                                                         (wide ? 0x80000000u : 0u), lo);
        RowSlot e;
        e.u = make_uint4((uint32_t)(g0 + lo), (uint32_t)ty | (xw & 0x80000000u), xw & 0x7FFFFFFFu,
                         __float_as_uint(__shfl_sync(0xffffffffu, L.l22, lo)));
        e.g = make_float4(__shfl_sync(0xffffffffu, L.a.x, lo), __shfl_sync(0xffffffffu, L.a.y, lo),
                          __shfl_sync(0xffffffffu, L.a.z, lo), __shfl_sync(0xffffffffu, L.a.w, lo));
        if (p < R) q[(qh + qn + lane) & (kQueue - 1)] = e;
        __syncwarp();
        qn += min(32, R - base);
        if (qn >= 32) {
            run_rows(q, qh, 32, f);
            qh = (qh + 32) & (kQueue - 1);
            qn -= 32;
            __syncwarp();
        }
    }
}

// A warp's share of the cost numbering: len costs from c0 on.  The group it starts
// in begins `before` costs earlier (less than one group's cost).
struct Share {
    unsigned long long c0;
    long long len;
    uint32_t before;
    int group;
};

// What k_bin_count hands to k_bin_scatter: plan[0] is the total cost C, plan[1 + w]
// the {group, before} of warp w.  At most one share per group, so that the plan
// fits its scratch of groups + 1 entries.
__device__ __forceinline__ Share share_of(unsigned long long C, int groups) {
    const unsigned long long all = (unsigned long long)gridDim.x * (blockDim.x >> 5);
    const unsigned long long W = all < (unsigned long long)groups ? all : (unsigned long long)groups;
    const unsigned long long w = (unsigned long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    Share sh{0ull, 0, 0u, 0};
    if (w < W) {
        sh.c0 = C * w / W;
        sh.len = (long long)(C * (w + 1) / W - sh.c0);
    }
    return sh;
}

// Calls f(active, item) for the rows of this warp's share of the work plan: a
// group's visit charge comes first and then its row costs, and a row belongs to
// the share holding its start cost.  The groups' costs are read 32 at a time
// (the next 32 ahead) and groups without rows (all Gaussians culled) are skipped
// without loading them; each group with rows is loaded while the previous one is
// processed.
template <class F>
__device__ __forceinline__ void warp_share_rows(const uint2 *__restrict__ rect,
                                                const ProjRec *__restrict__ rec, int64_t n,
                                                const uint32_t *__restrict__ cost, int groups,
                                                const Share &sh, RowSlot *q, F &&f) {
    const int lane = threadIdx.x & 31;
    int qh = 0, qn = 0;   // queued rows: slots [qh, qh + qn) mod kQueue
    if (sh.len <= 0) return;
    long long e = -(long long)sh.before;   // cost at which group gb starts, from c0 on
    uint32_t v_n = sh.group + lane < groups ? cost[sh.group + lane] : 0u;
    for (int gb = sh.group; gb < groups; gb += 32) {
        const int gl = gb + lane;
        const long long v = gl < groups ? (long long)v_n + kGroupCost : 0;
        v_n = gl + 32 < groups ? cost[gl + 32] : 0u;
        long long e1l = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, e1l, o);
            if (lane >= o) e1l += y;
        }
        e1l += e;
        const long long e0l = e1l - v;
        e = __shfl_sync(0xffffffffu, e1l, 31);
        // groups of this chunk with rows whose row costs meet the share
        unsigned m = __ballot_sync(0xffffffffu, v > kGroupCost && e1l > 0 && e0l + kGroupCost < sh.len);
        const bool done = __ballot_sync(0xffffffffu, gl >= groups || e1l >= sh.len) != 0u;
        if (m) {
            int j = __ffs(m) - 1;
            m &= m - 1;
            GroupLoad cur = load_group(rect, rec, n, (int64_t)(gb + j) * 32);
            for (;;) {
                const int jn = m ? __ffs(m) - 1 : -1;
                GroupLoad nxt{};
                if (jn >= 0) nxt = load_group(rect, rec, n, (int64_t)(gb + jn) * 32);   // in flight meanwhile
                const long long e0 = __shfl_sync(0xffffffffu, e0l, j) + kGroupCost;   // row costs start
                const long long nc = __shfl_sync(0xffffffffu, e1l, j) - e0;
                const long long ca = max(0ll, -e0);
                const long long cb = min(nc, sh.len - e0);
                if (ca < cb) warp_rows(cur, (int64_t)(gb + j) * 32, (int)ca, (int)cb, q, qh, qn, f);
                if (jn < 0) break;
                j = jn;
                m &= m - 1;
                cur = nxt;
            }
        }
        if (done) break;
    }
    if (qn > 0) run_rows(q, qh, qn, f);
}

// The CTA's shares.  Every CTA sums all group costs by chunks (4 bytes per 32
// Gaussians, from L2), scans the chunks' sums in shared memory, and each warp
// looks its start up: chunk by the scan, then group inside the chunk.  Bound: the
// latency of these dependent loads; in each CTA it costs 1 us (50k Gaussians), 5 us
// (600k) or 65 us (6M) of the count.  One CTA that scans for all (7, 14 and 85 us) is
// a launch more and leaves every warp three dependent searches in the count and in
// the scatter: 50k at 640x480 65.2 us a frame with it, 63.4 without; depth of 300k
// 479.6 and 474.5 us; 600k at 1600x1063 1039 and 1034.5 us.
constexpr int kPlanChunk = 128;      // groups per chunk, doubled until they fit
constexpr int kPlanChunks = 2048;
struct PlanSmem {
    unsigned long long pre[kPlanChunks + 1];   // costs before each chunk, total last
    unsigned long long warp_sums[kBinThreads / 32];
};
static_assert(kPlanChunks == 4 * kBinThreads, "four chunks per thread in the scan");

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ Share plan_shares(const uint32_t *__restrict__ cost, int groups,
                                             PlanSmem &sm, unsigned long long *__restrict__ plan) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int size = kPlanChunk;
    while ((int64_t)size * kPlanChunks < groups) size *= 2;
    const int chunks = (groups - 1) / size + 1;
#pragma unroll 4
    for (int c = warp; c < chunks; c += kBinThreads / 32) {
        unsigned long long sum = 0;
        const int end = (int)min((int64_t)groups, (int64_t)(c + 1) * size);
        for (int g = c * size + lane; g < end; g += kPlanChunk) {
            uint32_t v[kPlanChunk / 32];
#pragma unroll
            for (int k = 0; k < kPlanChunk / 32; ++k) v[k] = g + 32 * k < end ? cost[g + 32 * k] : 0u;
#pragma unroll
            for (int k = 0; k < kPlanChunk / 32; ++k)
                sum += (unsigned long long)v[k] + (g + 32 * k < end ? kGroupCost : 0);
        }
        sum = warp_sum(sum);
        if (lane == 0) sm.pre[c] = sum;
    }
    __syncthreads();
    // exclusive scan of the chunks
    unsigned long long v[4], local = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        v[k] = 4 * tid + k < chunks ? sm.pre[4 * tid + k] : 0ull;
        local += v[k];
    }
    unsigned long long incl = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) sm.warp_sums[warp] = incl;
    __syncthreads();
    unsigned long long run = incl - local, C = 0;
    for (int w = 0; w < kBinThreads / 32; ++w) {
        if (w < warp) run += sm.warp_sums[w];
        C += sm.warp_sums[w];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (4 * tid + k < chunks) sm.pre[4 * tid + k] = run;
        run += v[k];
    }
    if (tid == 0) sm.pre[chunks] = C;
    __syncthreads();

    Share sh = share_of(C, groups);
    if (blockIdx.x == 0 && tid == 0) plan[0] = C;
    if (sh.len > 0) {
        int lo = 0, hi = chunks;   // pre[lo] <= c0 < pre[hi]
        while (hi - lo > 1) {
            const int step = (hi - lo + 31) / 32;
            const int p = lo + step * (lane + 1);
            const unsigned le = __ballot_sync(0xffffffffu, p < hi && sm.pre[p] <= sh.c0);
            lo += step * __popc(le);
            if (lo + step < hi) hi = lo + step;
        }
        unsigned long long e = sm.pre[lo];
        // the group inside the chunk: it exists, c0 < pre[lo + 1]
        for (int g = lo * size; g < groups; g += 32) {
            const unsigned long long c = g + lane < groups ? (unsigned long long)cost[g + lane] + kGroupCost : 0ull;
            unsigned long long end = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long y = __shfl_up_sync(0xffffffffu, end, o);
                if (lane >= o) end += y;
            }
            const unsigned long long total = __shfl_sync(0xffffffffu, end, 31);
            if (e + total > sh.c0) {
                const int k = __popc(__ballot_sync(0xffffffffu, e + end <= sh.c0));   // lanes before it
                sh.group = g + k;
                sh.before = (uint32_t)(sh.c0 - e - __shfl_sync(0xffffffffu, end - c, k));
                break;
            }
            e += total;
        }
        if (lane == 0)
            plan[1 + blockIdx.x * (kBinThreads / 32) + warp] =
                (unsigned long long)sh.group << 32 | sh.before;
    }
    return sh;
}

// The same share, as k_bin_count stored it.
__device__ __forceinline__ Share stored_share(const unsigned long long *plan, int groups) {
    Share sh = share_of(plan[0], groups);
    if (sh.len > 0) {
        const unsigned long long p = plan[1 + blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)];
        sh.group = (int)(p >> 32);
        sh.before = (uint32_t)p;
    }
    return sh;
}

// Tile rows per shared-memory band: the count's difference array takes
// tiles_x + 1 words per tile row.
__host__ __device__ __forceinline__ int band_rows(int tiles_x, int tiles_y) {
    const int r = kBand / (tiles_x + 1);
    return r < tiles_y ? r : tiles_y;
}

// Counts per tile; with `tc` (tensor-core rasteriser) and a frame that has
// wide Gaussians, also sets kTileWide in tile_count[] of every tile that
// lists one (per-CTA counts stay below 2^31, so the flag never meets a carry).
// Shared memory: the band's difference array (band_rows x (tiles_x + 1)
// ints), then one wide-flag byte per tile of the band.
__global__ void __launch_bounds__(kBinThreads, 2) k_bin_count(const uint2 *__restrict__ rect,
                                                           const ProjRec *__restrict__ rec,
                                                           int64_t n, int tiles_x, int tiles_y,
                                                           const uint32_t *__restrict__ cost,
                                                           int groups,
                                                           unsigned long long *__restrict__ plan,
                                                           uint32_t *__restrict__ tile_count,
                                                           uint32_t *__restrict__ bases,
                                                           const DevStatus *__restrict__ status,
                                                           bool tc) {
    grid_wait();
    grid_trigger();   // the dependent (the tile scan) is one CTA
    extern __shared__ int diff_s[];
    __shared__ union {
        RowSlot queue[kBinThreads / 32][kQueue];
        PlanSmem plan;
    } sm;
    const Share share = plan_shares(cost, groups, sm.plan, plan);
    __syncthreads();   // the queues take the plan's place
    const int T = tiles_x * tiles_y;
    const int stride = tiles_x + 1;
    const int brows = band_rows(tiles_x, tiles_y);
    unsigned char *wide_s = reinterpret_cast<unsigned char *>(diff_s + brows * stride);
    const bool mark = tc && status->wide_bits != 0u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int ty0 = 0; ty0 < tiles_y; ty0 += brows) {
        const int nrows = min(brows, tiles_y - ty0);
        for (int i = threadIdx.x; i < nrows * stride; i += kBinThreads) diff_s[i] = 0;
        if (mark)
            for (int i = threadIdx.x; i < nrows * tiles_x; i += kBinThreads) wide_s[i] = 0;
        __syncthreads();
        warp_share_rows(rect, rec, n, cost, groups, share, sm.queue[warp], [&](bool active, const RowItem &it) {
            const int ry = it.ty - ty0;
            if (!active || (unsigned)ry >= (unsigned)nrows) return;
            int *d = diff_s + ry * stride;
            int a, b;
            if (row_tiles(it.mx, it.my, it.l11, it.l21, it.l22, it.x0, it.x1, it.ty, a, b)) {
                if (a <= b) {
                    atomicAdd(&d[a], 1);
                    atomicAdd(&d[b + 1], -1);
                    if (mark && it.wide)
                        for (int x = a; x <= b; ++x) wide_s[ry * tiles_x + x] = 1;
                }
            } else {   // not one interval: every tile of the row on its own
                for (int x = it.x0; x < it.x1; ++x)
                    if (tile_may_hit(it.mx, it.my, it.l11, it.l21, it.l22, x, it.ty)) {
                        atomicAdd(&d[x], 1);
                        atomicAdd(&d[x + 1], -1);
                        if (mark && it.wide) wide_s[ry * tiles_x + x] = 1;
                    }
            }
        });
        __syncthreads();
        // prefix sums along each tile row -> this CTA's tile counts; reserve
        // the CTA's block in every tile it lists pairs in
        for (int ry = warp; ry < nrows; ry += kBinThreads / 32) {
            int carry = 0;
            for (int xb = 0; xb < tiles_x; xb += 32) {
                const int x = xb + lane;
                int v = x < tiles_x ? diff_s[ry * stride + x] : 0;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, v, o);
                    if (lane >= o) v += y;
                }
                const int c = carry + v;
                carry += __shfl_sync(0xffffffffu, v, 31);
                if (x < tiles_x) {
                    const int t = (ty0 + ry) * tiles_x + x;
                    if (c > 0)
                        bases[(int64_t)blockIdx.x * T + t] =
                            atomicAdd(&tile_count[t], (uint32_t)c) & kTileMask;
                    if (mark && wide_s[ry * tiles_x + x]) atomicOr(&tile_count[t], kTileWide);
                }
            }
        }
        __syncthreads();
    }
}

// Rows of at most this many listed tiles are written lane by lane; a batch
// holding a longer one spreads its tiles over the warp instead.  So does every
// batch once the sectors being filled (one per CTA and tile) outgrow the L2:
// neighbouring tiles, written together, then meet more of them still there.
// Scatter, lane by lane / spread: 6M at 3840x2160 (158 MB of sectors) 6.73 / 6.21 ms,
// 1M 2.69 / 2.65 and 300k 0.363 / 0.358 at that size; 3M at 2560x1440 (70 MB)
// 1.16 / 1.27, 6M at 1920x1080 (40 MB) 1.29 / 1.96, 600k at 1600x1063 0.121 / 0.129.
// The line lies at the size of GB300's L2 (129 MB); between 70 and 158 MB it was not measured.
constexpr int64_t kOpenSectors = (int64_t)128 << 20 >> 5;
constexpr int kLaneRun = 16;

// Its CTAs may be resident while k_scan_order still runs: what that kernel or the
// count writes is read through plain pointers, so that no load is taken for one of
// data that stay constant for as long as this kernel lives.
__global__ void __launch_bounds__(kBinThreads, 2) k_bin_scatter(
    const uint2 *__restrict__ rect, int64_t n, int tiles_x, int tiles_y,
    const uint32_t *__restrict__ cost, int groups, const unsigned long long *plan,
    const uint32_t *offsets, const uint32_t *bases, uint32_t *gids, uint64_t capacity,
    const DevStatus *status, const ProjRec *__restrict__ rec, uint4 *__restrict__ wt16) {
    grid_wait();
    extern __shared__ uint32_t cur_s[];
    __shared__ RowSlot queue_s[kBinThreads / 32][kQueue];
    if (status->last_pairs > capacity) return;  // overflow: lists are not built
    const Share share = stored_share(plan, groups);
    const int we = (int)((status->wmax_frame_bits >> 23) & 0xFFu) - 127;
    if (wt16 && we >= 14) {   // preprocessing wrote the FP16 weights unscaled; rescale them
        const float scale = __int_as_float((127 + 14 - we) << 23);
        for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < n;
             g += (int64_t)gridDim.x * blockDim.x) {
            const uint2 r = rect[g];
            if (r.x | r.y) wt16[g] = weights_f16(rec[g], scale);
        }
    }
    const int T = tiles_x * tiles_y;
    const unsigned lane_run = (int64_t)gridDim.x * T > kOpenSectors ? 0u : (unsigned)kLaneRun;
    const int brows = band_rows(tiles_x, tiles_y);
    const int lane = threadIdx.x & 31;
    for (int ty0 = 0; ty0 < tiles_y; ty0 += brows) {
        const int nrows = min(brows, tiles_y - ty0);
        const int t0 = ty0 * tiles_x, bn = nrows * tiles_x;
        // entries of tiles this CTA has no pairs in are never read
        for (int i = threadIdx.x; i < bn; i += kBinThreads)
            cur_s[i] = offsets[t0 + i] + bases[(int64_t)blockIdx.x * T + t0 + i];
        __syncthreads();
        warp_share_rows(rect, rec, n, cost, groups, share, queue_s[threadIdx.x >> 5], [&](bool active, const RowItem &it) {
            const int ry = it.ty - ty0;
            const bool in = active && (unsigned)ry < (unsigned)nrows;
            int a = 1, b = 0;
            const bool one = in ? row_tiles(it.mx, it.my, it.l11, it.l21, it.l22, it.x0, it.x1,
                                            it.ty, a, b)
                                : true;
            const int L = (in && one && a <= b) ? b - a + 1 : 0;
            if (__reduce_max_sync(0xffffffffu, (unsigned)L) <= lane_run) {
                // short rows: each lane writes its own row's tiles
                for (int x = a; x < a + L; ++x) {
                    const uint32_t slot = atomicAdd(&cur_s[ry * tiles_x + x], 1u);
                    if (slot < capacity) gids[slot] = it.gid;
                }
            } else {
                // a long row among them: the rows' tiles, 32 at a time over the warp
                int incl = L;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                const int ex = incl - L;
                const int total = __shfl_sync(0xffffffffu, incl, 31);
                const int tb = ry * tiles_x + a - ex;   // band tile of pair p of this lane: tb + p
                for (int base = 0; base < total; base += 32) {
                    const int p = base + lane;
                    int lo = 0;   // owner: the largest lane whose exclusive prefix is <= p
#pragma unroll
                    for (int step = 16; step > 0; step >>= 1) {
                        const int e = __shfl_sync(0xffffffffu, ex, lo + step);
                        if (e <= p) lo += step;
                    }
                    const int t = __shfl_sync(0xffffffffu, tb, lo) + p;
                    const uint32_t gid = __shfl_sync(0xffffffffu, it.gid, lo);
                    if (p < total) {
                        const uint32_t slot = atomicAdd(&cur_s[t], 1u);
                        if (slot < capacity) gids[slot] = gid;
                    }
                }
            }
            if (in && !one)   // not one interval: every tile of the row on its own
                for (int x = it.x0; x < it.x1; ++x)
                    if (tile_may_hit(it.mx, it.my, it.l11, it.l21, it.l22, x, it.ty)) {
                        const uint32_t slot = atomicAdd(&cur_s[ry * tiles_x + x], 1u);
                        if (slot < capacity) gids[slot] = it.gid;
                    }
        });
        __syncthreads();
    }
}

// One block over the per-tile totals:
//   * exclusive scan of tile_count[T] into tile_offsets[T+1]; records the
//     pair count and flags capacity overflow;
//   * rasterisation order: tiles by decreasing list length (bucketed by
//     floor(log2(length))), so the longest tiles start first and the tail of
//     the raster launch is made of short tiles;
//   * hands this frame's weight bound to the rasteriser and resets the
//     accumulator (and the wide-Gaussian flag) for the next frame;
//   * carries each tile's kTileWide flag from tile_count[] into its order
//     entry.
// It may be resident while the count still writes tile_count: a plain pointer, as in
// k_bin_scatter.
__global__ void __launch_bounds__(kScanThreads) k_scan_order(const uint32_t *count,
                                                             uint32_t *__restrict__ offsets,
                                                             uint32_t *__restrict__ order, int T,
                                                             uint64_t capacity, DevStatus *status) {
    grid_wait();
    __shared__ unsigned long long warp_sums[kScanThreads / 32];
    __shared__ unsigned long long carry;
    __shared__ uint32_t hist[33], start[33];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        carry = 0;
        status->wmax_frame_bits = status->wmax_bits;
        status->wmax_bits = 0u;
        status->wide_bits = 0u;
        status->last_visible = status->visible;
        status->visible = 0u;
        status->last_wide_tiles = 0u;
    }
    if (tid < 33) hist[tid] = 0u;
    __syncthreads();
    for (int base = 0; base < T; base += kScanThreads * 4) {
        const int i0 = base + tid * 4;
        unsigned long long v[4], local = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = (i0 + k < T) ? (count[i0 + k] & kTileMask) : 0u;
            local += v[k];
            if (i0 + k < T) {
                const uint32_t c = (uint32_t)v[k];
                atomicAdd(&hist[c ? 32 - __clz(c) : 0], 1u);   // bucket 0 (empty) .. 32
            }
        }
        unsigned long long incl = local;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) warp_sums[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            unsigned long long sw = warp_sums[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                unsigned long long y = __shfl_up_sync(0xffffffffu, sw, o);
                if (lane >= o) sw += y;
            }
            warp_sums[lane] = sw;
        }
        __syncthreads();
        unsigned long long run = carry + (incl - local) + (warp > 0 ? warp_sums[warp - 1] : 0ull);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (i0 + k < T) offsets[i0 + k] = (uint32_t)run;
            run += v[k];
        }
        __syncthreads();
        if (tid == kScanThreads - 1) carry = run;
        __syncthreads();
    }
    if (tid == 0) {
        const unsigned long long K = carry;
        offsets[T] = (uint32_t)K;
        status->last_pairs = K;
        atomicMax(&status->max_pairs, K);
        if (K > capacity || K > 0xFFFFFFFFull) atomicOr(&status->overflow, kStatusOverflow);
        uint32_t r = 0;
        for (int bk = 32; bk >= 0; --bk) {      // longest bucket first
            start[bk] = r;
            r += hist[bk];
        }
    }
    __syncthreads();
    grid_trigger();
    for (int t = tid; t < T; t += blockDim.x) {
        const uint32_t cw = count[t], c = cw & kTileMask;
        order[atomicAdd(&start[c ? 32 - __clz(c) : 0], 1u)] = (uint32_t)t | (cw & kTileWide);
        if (cw & kTileWide) atomicAdd(&status->last_wide_tiles, 1u);
    }
}

}  // namespace

// One binning CTA per SM at most: the work plan balances the warps, so a second
// resident CTA would only add per-CTA tile bases.  Below that, one per 512
// Gaussians, a group per warp: small scenes are bound by the latency of a warp's
// walk over its groups.  One CTA per 256 / 512 / 1024 Gaussians: 4k frame at 256x256
// 40.4 / 40.4 / 48.2 us, 50k at 640x480 63.7 / 63.5 / 70.8 us, twelve served views of
// 40k to 160k 1.062 / 1.065 / 1.079 ms.
int bin_ctas(int64_t n, int sm_count) {
    int64_t c = (n + 511) / 512;
    const int64_t cap = (int64_t)sm_count;
    if (c > cap) c = cap;
    return c < 1 ? 1 : (int)c;
}

uint32_t *bin_group_cost(uint32_t *scratch, int64_t n, int64_t T, int sm_count) {
    const int64_t groups = (n + 31) / 32;
    return scratch + (bin_ctas(n, sm_count) * T + 1) / 2 * 2 + 2 * (groups + 1);
}

int64_t bin_scratch_words(int64_t n, int64_t T, int sm_count) {
    return bin_scratch_words_for(bin_ctas(n, sm_count), T, n);
}

cudaError_t launch_binning(const RenderArgs &a, int sm_count, uint32_t *scratch,
                           cudaStream_t stream, const cudaEvent_t *marks, bool grouped) {
    const int tx = a.cam.tiles_x, ty = a.cam.tiles_y;
    const int T = tx * ty;
    const int CL = bin_ctas(a.n, sm_count);   // the scratch's layout
    // Views prepared side by side fill the chip between them, so each takes at most
    // half as many CTAs: less per-CTA work (clearing and scanning T counts, summing the
    // plan).  A burst of twelve views of 160k Gaussians: 1.087 ms with one CTA per SM and
    // view, 1.078 with one per two SMs in a group of views, 1.066 where the lone views of
    // a busy server do the same; a third and a quarter of the SMs are slower (1.071 and
    // 1.108 where half took 1.053).  This is what the plan inside the count had cost the
    // burst (1.06 with a plan kernel of its own), not a gain over it.
    const int C = grouped ? std::min(CL, std::max(sm_count / 2, 1)) : CL;
    const int64_t groups = (a.n + 31) / 32;
    uint32_t *bases = scratch;
    unsigned long long *plan =
        reinterpret_cast<unsigned long long *>(scratch + ((int64_t)CL * T + 1) / 2 * 2);
    const int brows = band_rows(tx, ty);
    const size_t count_smem = ((size_t)brows * (tx + 1) * sizeof(int) + (size_t)brows * tx + 15) / 16 * 16;
    const size_t scatter_smem = (size_t)brows * tx * sizeof(uint32_t);
    cudaError_t e = cudaSuccess;
    if (a.n == 0)   // preprocessing, which clears the counts, did not run
        e = cudaMemsetAsync(a.tile_count, 0, (size_t)T * sizeof(uint32_t), stream);
    if (e != cudaSuccess) return e;
    if (a.n > 0) {
        if ((e = cudaFuncSetAttribute(k_bin_count, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)(kBand * (sizeof(int) + 1)))) != cudaSuccess)
            return e;
        if ((e = cudaFuncSetAttribute(k_bin_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)(kBand * sizeof(uint32_t)))) != cudaSuccess)
            return e;
        if (marks && (e = cudaEventRecord(marks[0], stream)) != cudaSuccess) return e;
        if ((e = launch_dependent(k_bin_count, C, kBinThreads, count_smem, stream, a.rect, a.rec, a.n, tx,
                                  ty, a.group_cost, (int)groups, plan, a.tile_count, bases, a.status, tc_raster(a))) !=
            cudaSuccess)
            return e;
        if (marks && (e = cudaEventRecord(marks[1], stream)) != cudaSuccess) return e;
    } else if (marks) {
        if ((e = cudaEventRecord(marks[0], stream)) != cudaSuccess) return e;
        if ((e = cudaEventRecord(marks[1], stream)) != cudaSuccess) return e;
    }
    if ((e = launch_dependent(k_scan_order, 1, kScanThreads, 0, stream, a.tile_count, a.tile_offsets,
                              a.tile_order, T, a.capacity, a.status)) != cudaSuccess)
        return e;
    if (marks && (e = cudaEventRecord(marks[2], stream)) != cudaSuccess) return e;
    if (a.n == 0) return e;
    return launch_dependent(k_bin_scatter, C, kBinThreads, scatter_smem, stream, a.rect, a.n, tx, ty,
                            a.group_cost, (int)groups, plan, a.tile_offsets, bases, a.gids, a.capacity, a.status, a.rec,
                            tc_raster(a) ? a.wt16 : nullptr);
}

}  // namespace mgs
