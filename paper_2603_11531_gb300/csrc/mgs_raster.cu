// Per-pixel depth-aware, order-independent accumulation (Sec. 3.1, Eq. 2):
//
//   A = sum_i c_i a_i w_i,  B = sum_i a_i w_i,  T = prod_i (1 - a_i)
//   C = (1 - T) A / B + T c_bg          (foreground term 0 when B = 0)
//
// One CTA per 16x16 tile, four warps of 8x8 pixels; the four lanes of a quad
// own one row of eight pixels.  Each warp walks the tile's Gaussian list itself,
// testing each entry against its block with a conservative bound
// (block_may_hit) and compacting (ballot) the candidates into a ring in shared
// memory; the lanes of a quad take different candidates, and their sums are
// added at the end.
//
// FP32 scenes (k_raster): packed FP32x2 arithmetic over pixel pairs, all sums
// on the FMA pipe.
//
// FP16-attribute scenes (k_raster_tc): alpha is computed, tested and multiplied
// into T in FP32 exactly as above (packed over two candidates), but a_i w_i c_i
// and a_i w_i are summed on the tensor cores by
// mma.sync (m16n8k8, FP16 operands, FP32 accumulation) with the weights split
// into FP16 high and low parts, which leaves alpha's FP16 rounding (relative
// 2^-12 per term) as the only extra error; tiles listing a Gaussian outside
// the FP16 weight range take the FP32 code.
//
// No atomics, no sort: every pixel belongs to one quad, and a tile's list is
// accumulated in whatever order binning stored it.
//
// T stops being updated where no further update can change a bit of the image: a
// lane's partial product only shrinks, so once every lane of a warp holds at most
// 2^-38 for each of its pixels, the product over a quad is at most 2^-152, which FP32
// rounds to 0, as it does the product of anything smaller.  With a background of zeros
// T c_bg is 0 whatever T is, and 2^-8 suffices: T <= 2^-32, so that 1 - T rounds to 1.
// A NaN stays NaN, updated or not.  The aux output returns T and keeps the updates.
#include "mgs_internal.cuh"

namespace mgs {
namespace {

constexpr int kThreads = 128;
constexpr int kWarps = kThreads / 32;
constexpr float kZeroT = 3.637978807091713e-12f;   // 2^-38: T is 0
constexpr float kOneMinusT = 0.00390625f;          // 2^-8: 1 - T is 1
constexpr int kFreezeEvery = 128;             // list entries between two checks
constexpr float kLogClamp = -0.014499569695115089f;   // log2(0.99)

typedef unsigned long long f2;  // two packed FP32 lanes

__device__ __forceinline__ f2 pk(float lo, float hi) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void upk(f2 v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
    f2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Staged Gaussian of the FMA sums: five 16-byte words of duplicated pairs, so
// every operand of the packed arithmetic comes straight from one shared-memory
// load.
//   s0 = {m_x, m_x, m_y, m_y}      s1 = {l11, l11, l21, l21}
//   s2 = {l22, l22, log2 o, log2 o} s3 = {-w, -w, -w c_r, -w c_r}
//   s4 = {-w c_g, -w c_g, -w c_b, -w c_b}, depth image: s5 = {-w d, -w d, 0, 0}
constexpr int kGroup = 4;         // candidates per step: one per lane of a quad
constexpr int kRingF = 36;        // slots per warp: 32 + 3 left over, whole groups
template <bool kDepth>
struct FmaSmem {
    ulonglong2 s[kWarps][kDepth ? 6 : 5][kRingF];
};

// The sums of one lane: its row's eight pixels as four pairs.
template <bool kDepth>
struct FmaSums {
    f2 A[4][3], B[4], T[4], AD[kDepth ? 4 : 1];
};

// Accumulates one staged Gaussian (slot k of the warp's ring) into the lane's
// eight pixels.  kClamp: its opacity may exceed 0.99; kLive: T is updated.
template <bool kCount, bool kDepth, bool kClamp, bool kLive>
__device__ __forceinline__ void accumulate(const ulonglong2 (*wb)[kRingF], int k, const f2 (&px)[4],
                                           f2 pyc, f2 kq2, FmaSums<kDepth> &S, int (&cnt)[8]) {
    const ulonglong2 s0 = wb[0][k], s1 = wb[1][k], s2 = wb[2][k];
    // inclusion test (exact FP32 sequence); the row terms are shared by the pairs
    const f2 dy = sub2(pyc, s0.y);
    const f2 ldy = mul2(s1.y, dy);
    const f2 e2 = mul2(s2.x, dy);
    const f2 e2s = mul2(e2, e2);
    const ulonglong2 s3 = wb[3][k], s4 = wb[4][k];
    f2 wd = 0ull;
    if constexpr (kDepth) wd = wb[5][k].x;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const f2 e1 = fma2(s1.x, sub2(px[p], s0.x), ldy);
        const f2 q = fma2(e1, e1, e2s);
        // a = min(0.99, o 2^(-q log2(e) / 2)), kept negated
        const f2 g = fma2(q, kq2, s2.y);
        float q0, q1, g0, g1;
        upk(q, q0, q1);
        upk(g, g0, g1);
        float n0 = -ex2(g0), n1 = -ex2(g1);
        if constexpr (kClamp) {
            n0 = fmaxf(n0, -0.99f);
            n1 = fmaxf(n1, -0.99f);
        }
        n0 = q0 <= 9.0f ? n0 : 0.0f;
        n1 = q1 <= 9.0f ? n1 : 0.0f;
        if constexpr (kCount) {
            cnt[2 * p] += q0 <= 9.0f;
            cnt[2 * p + 1] += q1 <= 9.0f;
        }
        const f2 na = pk(n0, n1);
        S.A[p][0] = fma2(na, s3.y, S.A[p][0]);
        S.A[p][1] = fma2(na, s4.x, S.A[p][1]);
        S.A[p][2] = fma2(na, s4.y, S.A[p][2]);
        S.B[p] = fma2(na, s3.x, S.B[p]);
        if constexpr (kLive) S.T[p] = fma2(na, S.T[p], S.T[p]);
        if constexpr (kDepth) S.AD[p] = fma2(na, wd, S.AD[p]);
    }
}

// Every lane's partial products at most this: T no longer matters (see above).
__device__ __forceinline__ bool zero_bg(const RenderArgs &args) {
    return args.bg[0] == 0.0f && args.bg[1] == 0.0f && args.bg[2] == 0.0f;
}
__device__ __forceinline__ bool all_frozen(const RenderArgs &args, float m) {
    return __all_sync(0xffffffffu, m <= (zero_bg(args) ? kOneMinusT : kZeroT));
}
// May T stop being updated?  0 c_bg is 0 for a finite background only.  The depth image's
// lists rarely reach 2^-38 and only pay for the question (300k at 1280x720: 0.393 ms with
// it, 0.388 without; 0.379 with a background of zeros, which freezes at 2^-8).
template <bool kAux, bool kDepth>
__device__ __forceinline__ bool may_freeze(const RenderArgs &args) {
    if (kAux) return false;
    if (kDepth) return zero_bg(args);
    return fmaxf(fmaxf(fabsf(args.bg[0]), fabsf(args.bg[1])), fabsf(args.bg[2])) < INFINITY;
}

// Writes one pixel's outputs from its sums.
template <bool kAux, bool kCount, bool kDepth>
__device__ __forceinline__ void put_pixel(const RenderArgs &args, int x, int y, float ar, float ag,
                                          float ab, float bb, float tr, int cnt, float ad) {
    const DevCamera &cam = args.cam;
    const int64_t HW = (int64_t)cam.width * cam.height;
    const int64_t p = (int64_t)y * cam.width + x;
    const float fg = bb > 0.0f ? (1.0f - tr) / bb : 0.0f;
    float *out = args.out_rgb + 3 * p;
    out[0] = fmaf(fg, ar, tr * args.bg[0]);
    out[1] = fmaf(fg, ag, tr * args.bg[1]);
    out[2] = fmaf(fg, ab, tr * args.bg[2]);
    if (kAux) {
        args.out_aux[p] = ar;
        args.out_aux[HW + p] = ag;
        args.out_aux[2 * HW + p] = ab;
        args.out_aux[3 * HW + p] = bb;
        args.out_aux[4 * HW + p] = tr;
    }
    if (kCount) args.out_count[p] = cnt;
    if (kDepth) args.out_depth[p] = bb > 0.0f ? ad / bb : 0.0f;
}

// Sum over the quad of a lane's four pixel pairs: lane t of the quad receives
// pair t (reduce-scatter: half of the pairs to the other half of the quad,
// then one to the neighbour).
__device__ __forceinline__ float2 quad_sum(const f2 (&v)[4], int t) {
    float x[4][2];
#pragma unroll
    for (int p = 0; p < 4; ++p) upk(v[p], x[p][0], x[p][1]);
    float y[2][2];
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float send = (t & 2) ? x[p][h] : x[p + 2][h];
            y[p][h] = ((t & 2) ? x[p + 2][h] : x[p][h]) + __shfl_xor_sync(0xffffffffu, send, 2);
        }
    float z[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float send = (t & 1) ? y[0][h] : y[1][h];
        z[h] = ((t & 1) ? y[1][h] : y[0][h]) + __shfl_xor_sync(0xffffffffu, send, 1);
    }
    return make_float2(z[0], z[1]);
}
// The same with products (T).
__device__ __forceinline__ float2 quad_product(const f2 (&v)[4], int t) {
    float2 r = make_float2(1.0f, 1.0f);
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        float x, y;
        upk(v[p], x, y);
        x *= __shfl_xor_sync(0xffffffffu, x, 1);
        y *= __shfl_xor_sync(0xffffffffu, y, 1);
        x *= __shfl_xor_sync(0xffffffffu, x, 2);
        y *= __shfl_xor_sync(0xffffffffu, y, 2);
        if (p == t) r = make_float2(x, y);
    }
    return r;
}

// Rasterises one tile on the FMA pipe (four warps).  Each warp streams the
// tile's list on its own (no block-wide barrier): 32 entries at a time, one per
// lane (list entries are fetched two batches ahead, their records one batch
// ahead), are tested against the warp's block and queued in its ring; groups
// of four candidates are accumulated, one per lane of each quad.
//
// Bound: issue (36 packed operations and about 69 instructions per lane,
// candidate and eight pixels).  With two warps of 16x8 pixels per tile and four
// pixels per lane, every candidate's operands and row terms served four pixels
// instead of eight, 14 % more (block, Gaussian) pairs were evaluated, and small
// images had half the warps: 0.212 ms at 160k Gaussians, 1001x667, against
// 0.167 ms; 29 against 20 us at 4k, 256x256; 0.51 against 0.46 ms for the
// training forward (300k, 1296x840).
template <bool kAux, bool kCount, bool kDepth = false>
__device__ __forceinline__ void raster_tile(const RenderArgs &args, int tile, FmaSmem<kDepth> &sm) {
    const DevCamera &cam = args.cam;
    const int tx = tile % cam.tiles_x, ty = tile / cam.tiles_x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    const int bx0 = tx * kTile + 8 * (warp & 1), by0 = ty * kTile + 8 * (warp >> 1);
    const int py = by0 + g;

    const uint32_t start = args.tile_offsets[tile];
    const uint32_t end = args.tile_offsets[tile + 1];
    const bool no_cull = (args.flags & MGS_FLAG_NO_CULL) != 0;
    const float bcx = (float)bx0 + 4.0f, bcy = (float)by0 + 4.0f;

    f2 px[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) px[p] = pk((float)(bx0 + 2 * p) + 0.5f, (float)(bx0 + 2 * p) + 1.5f);
    const f2 pyc = pk((float)py + 0.5f, (float)py + 0.5f);
    const float kq = -0.72134752044448170f;  // -log2(e) / 2
    const f2 kq2 = pk(kq, kq);
    FmaSums<kDepth> S;
    int cnt[8];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        S.A[p][0] = S.A[p][1] = S.A[p][2] = S.B[p] = 0ull;
        S.T[p] = pk(1.0f, 1.0f);
        if constexpr (kDepth) S.AD[p] = 0ull;
        cnt[2 * p] = cnt[2 * p + 1] = 0;
    }
    ulonglong2(*wb)[kRingF] = sm.s[warp];

    int head = 0, count = 0;   // queued candidates: ring slots [head, head + count) mod kRingF
    int clamp_left = 0;        // queued candidates up to the last whose opacity exceeds 0.99
    bool live = true;          // T is still updated
    const bool freeze = may_freeze<kAux, false>(args);
    auto group = [&]() {
        const int k = head + t;
        if (live) {
            if (clamp_left > 0) accumulate<kCount, kDepth, true, true>(wb, k, px, pyc, kq2, S, cnt);
            else accumulate<kCount, kDepth, false, true>(wb, k, px, pyc, kq2, S, cnt);
        } else if constexpr (!kAux) {
            if (clamp_left > 0) accumulate<kCount, kDepth, true, false>(wb, k, px, pyc, kq2, S, cnt);
            else accumulate<kCount, kDepth, false, false>(wb, k, px, pyc, kq2, S, cnt);
        }
        clamp_left -= kGroup;
        count -= kGroup;
        head += kGroup;
        if (head == kRingF) head = 0;
    };
    float4 a_n = make_float4(0.f, 0.f, 0.f, 0.f), b_n = a_n, c_n = a_n;
    uint32_t gid_nn = 0;
    if (start + lane < end) {
        const uint32_t gid = __ldg(&args.gids[start + lane]);
        a_n = __ldg(&args.rec[gid].a);
        b_n = __ldg(&args.rec[gid].b);
        c_n = __ldg(&args.rec[gid].c);
    }
    if (start + 32 + lane < end) gid_nn = __ldg(&args.gids[start + 32 + lane]);
    for (uint32_t base = start; base < end; base += 32) {
        const uint32_t j = base + lane;
        const float4 a = a_n, b = b_n, c = c_n;
        const bool cand =
            j < end && (no_cull || block_may_hit(a.x, a.y, a.z, a.w, b.x, bcx, bcy, 3.5f, 3.5f));
        if (j + 32 < end) {
            const uint32_t gid = gid_nn;
            a_n = __ldg(&args.rec[gid].a);
            b_n = __ldg(&args.rec[gid].b);
            c_n = __ldg(&args.rec[gid].c);
        }
        if (j + 64 < end) gid_nn = __ldg(&args.gids[j + 64]);
        const unsigned bal = __ballot_sync(0xffffffffu, cand);
        const unsigned cb = __ballot_sync(0xffffffffu, cand && !(b.y <= kLogClamp));
        if (cand) {
            int pos = head + count + __popc(bal & ((1u << lane) - 1u));
            if (pos >= kRingF) pos -= kRingF;
            wb[0][pos] = make_ulonglong2(pk(a.x, a.x), pk(a.y, a.y));
            wb[1][pos] = make_ulonglong2(pk(a.z, a.z), pk(a.w, a.w));
            wb[2][pos] = make_ulonglong2(pk(b.x, b.x), pk(b.y, b.y));
            wb[3][pos] = make_ulonglong2(pk(b.z, b.z), pk(b.w, b.w));
            wb[4][pos] = make_ulonglong2(pk(c.x, c.x), pk(c.y, c.y));
            if constexpr (kDepth) wb[5][pos] = make_ulonglong2(pk(c.w, c.w), 0ull);   // -w d
        }
        if (cb) clamp_left = count + __popc(bal & (0xffffffffu >> __clz(cb)));
        __syncwarp();
        count += __popc(bal);
        while (count >= kGroup) group();
        if (freeze && live && ((base - start) & (kFreezeEvery - 1)) == kFreezeEvery - 32) {
            float m = 0.0f;
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                float x, y;
                upk(S.T[p], x, y);
                m = fmaxf(m, fmaxf(x, y));
            }
            live = !all_frozen(args, m);
        }
        __syncwarp();
    }
    if (count > 0) {   // pad the last group with entries that include no pixel and weigh 0
        if (lane < kGroup - count) {
            int pos = head + count + lane;
            if (pos >= kRingF) pos -= kRingF;
            wb[0][pos] = make_ulonglong2(pk(1e30f, 1e30f), pk(1e30f, 1e30f));
            wb[1][pos] = make_ulonglong2(pk(1.0f, 1.0f), 0ull);
            wb[2][pos] = make_ulonglong2(pk(1.0f, 1.0f), 0ull);
            wb[3][pos] = wb[4][pos] = make_ulonglong2(0ull, 0ull);
            if constexpr (kDepth) wb[5][pos] = make_ulonglong2(0ull, 0ull);
        }
        __syncwarp();
        group();
    }

    // lane t of a quad receives the sums of pixels 2t, 2t + 1
    const f2 Ar[4] = {S.A[0][0], S.A[1][0], S.A[2][0], S.A[3][0]};
    const f2 Ag[4] = {S.A[0][1], S.A[1][1], S.A[2][1], S.A[3][1]};
    const f2 Ab[4] = {S.A[0][2], S.A[1][2], S.A[2][2], S.A[3][2]};
    const float2 ar = quad_sum(Ar, t), ag = quad_sum(Ag, t), ab = quad_sum(Ab, t);
    const float2 bb = quad_sum(S.B, t), tr = quad_product(S.T, t);
    float2 ad = make_float2(0.f, 0.f);
    if constexpr (kDepth) ad = quad_sum(S.AD, t);
    int c2[2] = {0, 0};
    if constexpr (kCount) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            int x = cnt[k];
            x += __shfl_xor_sync(0xffffffffu, x, 1);
            x += __shfl_xor_sync(0xffffffffu, x, 2);
            if ((k >> 1) == t) c2[k & 1] = x;
        }
    }
    const int x = bx0 + 2 * t;
    if (py >= cam.height || x >= cam.width) return;
    put_pixel<kAux, kCount, kDepth>(args, x, py, ar.x, ag.x, ab.x, bb.x, tr.x, c2[0], ad.x);
    if (x + 1 < cam.width)
        put_pixel<kAux, kCount, kDepth>(args, x + 1, py, ar.y, ag.y, ab.y, bb.y, tr.y, c2[1], ad.y);
}

// ---------------------------------------------------------------------------
// Tensor-core accumulation of A and B (FP16-attribute scenes).
//
// One CTA (four warps) per tile; warp w owns the 8x8 block at
// (8 (w % 2), 8 (w / 2)) of the tile.  A warp's 64 pixels are the M = 64 rows
// of four m16n8k8 tiles: lane (g, t) = (lane / 4, lane % 4) owns the eight
// pixels x = 0..7 of the block's row g (rows g and g + 8 of m-tile i are
// pixels 2i and 2i + 1), shared by the four lanes of its quad.  Candidates
// are gathered into chunks of 8 Gaussians (the K dimension); lane t of a
// quad evaluates chunk entries 2t and 2t + 1 at its pixels -- one packed
// FP32x2 operation serves both, and the packed pair of alphas is exactly the
// A fragment the lane holds.  B = the chunk's weights [w c_r, w c_g, w c_b, w]
// as FP16 high parts (columns 0-3) and low parts (columns 4-7), so column c +
// column c + 4 is the sum with a 22-bit weight; preprocessing writes these
// FP16 weights once per Gaussian, and binning rescales them by a power of two
// when the frame's largest weight would overflow FP16 (the scale cancels in
// A / B and is divided out here).  T stays in FP32 FMAs.  Tiles listing a Gaussian
// outside that scale's range (kTileWide) are rasterised by the FMA tile code.
//
// Bound: instruction issue (78 % of the slots used at 600k Gaussians, 1600x1063; a packed
// FP32x2 operation takes two), so the time follows the instructions per pixel: without
// T's two FMAs where T is frozen, and with the weight fragment read by one ldmatrix
// instead of two 16-bit loads and a merge, that frame takes 0.834 ms with a background
// and 0.810 ms on zeros (0.865 never frozen), 3M at 640x480 1.34 and 1.33 ms (1.43), 6M at
// 3840x2160 36.9 and 36.7 ms (40.1); 50k at 640x480, whose lists are too short to
// freeze, 34.1 us (34.2).  Two lanes per record instead of one (cp.async into shared memory)
// saves L1 tag lookups but waits longer: 0.876 ms.
constexpr int kChunk = 8;        // candidates per MMA (K)
constexpr int kRing = 64;        // candidate slots per warp: eight chunks (a power of two)

// Ring slot s stores its geometry in pair-interleaved words, so that lane t
// reads the two entries 2t, 2t + 1 of a chunk with one 16-byte load each:
//   geo[0][s / 2] = {m_x(a), m_x(b), m_y(a), m_y(b)}
//   geo[1][s / 2] = {l11(a), l11(b), l21(a), l21(b)}
//   geo[2][s / 2] = {l22(a), l22(b), log2 o(a), log2 o(b)}   (a = even slot)
struct TcSmem {
    float4 geo[kWarps][3][kRing / 2];
    uint4 wt[kWarps][kRing];            // slot s: its 8 FP16 weight columns
    float2 wd[kWarps][kRing / 2];       // depth image only: w d of slots 2p, 2p + 1
};

__device__ __forceinline__ uint32_t h2bits(float lo, float hi) {
    const __half2 h = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&h);
}

__device__ __forceinline__ void mma_k8(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(b0));
}

// One chunk of 8 candidates starting at ring slot c0 (a multiple of 8): the
// lane's entries 2t, 2t + 1 at its eight pixels (same FP32 sequence as
// accumulate()), T updated, alphas packed to FP16 and summed by four MMAs.
// kLive: T is updated (two of about 17 issue slots per pixel).
// kDepth: also AD[j] += (a, b) * (w d of the two entries), the FP32 numerator
// of the depth image (Eq. 5), kept as two partial sums per pixel.
template <bool kCount, bool kClamp, bool kDepth, bool kLive>
__device__ __forceinline__ void tc_chunk(const float4 (*geo)[kRing / 2], const uint4 *wt,
                                         int c0, int g, int t, const f2 (&pxc)[8], f2 pyc,
                                         f2 kq2, float (&T)[8], float (&D)[4][4], int (&cnt)[8],
                                         const float2 *wd = nullptr, f2 *AD = nullptr) {
    const int pr = (c0 >> 1) + t;
    f2 wdp = 0ull;
    if constexpr (kDepth) wdp = pk(wd[pr].x, wd[pr].y);
    const float4 q0 = geo[0][pr], q1 = geo[1][pr], q2 = geo[2][pr];
    const f2 mx = pk(q0.x, q0.y), my = pk(q0.z, q0.w);
    const f2 l11 = pk(q1.x, q1.y), l21 = pk(q1.z, q1.w);
    const f2 l22 = pk(q2.x, q2.y), lo = pk(q2.z, q2.w);
    const f2 dy = sub2(pyc, my);
    const f2 ldy = mul2(l21, dy);
    const f2 e2 = mul2(l22, dy);
    const f2 e2s = mul2(e2, e2);
    uint32_t a[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const f2 dx = sub2(pxc[j], mx);
        const f2 e1 = fma2(l11, dx, ldy);
        const f2 q = fma2(e1, e1, e2s);
        const f2 gg = fma2(q, kq2, lo);
        float qa, qb, ga, gb;
        upk(q, qa, qb);
        upk(gg, ga, gb);
        float aa = ex2(ga), ab = ex2(gb);
        if (kClamp) {
            aa = fminf(aa, 0.99f);
            ab = fminf(ab, 0.99f);
        }
        aa = qa <= 9.0f ? aa : 0.0f;
        ab = qb <= 9.0f ? ab : 0.0f;
        if (kCount) cnt[j] += (qa <= 9.0f) + (qb <= 9.0f);
        if constexpr (kLive) {
            T[j] = fmaf(-aa, T[j], T[j]);
            T[j] = fmaf(-ab, T[j], T[j]);
        }
        if constexpr (kDepth) AD[j] = fma2(pk(aa, ab), wdp, AD[j]);
        a[j] = h2bits(aa, ab);            // k = 2t (low half), 2t + 1
    }
    uint32_t b0;   // column g, k = 2t, 2t + 1: the chunk's weights transposed
    asm volatile("ldmatrix.sync.aligned.m8n8.x1.trans.shared.b16 {%0}, [%1];"
                 : "=r"(b0)
                 : "r"((uint32_t)__cvta_generic_to_shared(wt + c0 + (threadIdx.x & 7))));
#pragma unroll
    for (int i = 0; i < 4; ++i) mma_k8(D[i], a[2 * i], a[2 * i + 1], b0);   // pixels 2i, 2i + 1
}

template <bool kAux, bool kCount, bool kDepth = false>
__device__ __forceinline__ void raster_tile_tc(const RenderArgs &args, int tile, TcSmem &sm) {
    const DevCamera &cam = args.cam;
    const int tx = tile % cam.tiles_x, ty = tile / cam.tiles_x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    const int bx0 = tx * kTile + 8 * (warp & 1), by0 = ty * kTile + 8 * (warp >> 1);
    const int xb = bx0;
    const int py = by0 + g;
    float4(*geo)[kRing / 2] = sm.geo[warp];
    uint4 *wt = sm.wt[warp];
    float2 *wd = sm.wd[warp];

    const uint32_t start = args.tile_offsets[tile];
    const uint32_t end = args.tile_offsets[tile + 1];
    const bool no_cull = (args.flags & MGS_FLAG_NO_CULL) != 0;
    const float bcx = (float)bx0 + 4.0f, bcy = (float)by0 + 4.0f;
    // weight scale 2^(14 - e) when the frame's largest weight has exponent e >= 14
    const int we = (int)((args.status->wmax_frame_bits >> 23) & 0xFFu) - 127;
    const float wscale = we >= 14 ? __int_as_float((127 + 14 - we) << 23) : 1.0f;

    f2 pxc[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) pxc[j] = pk((float)(xb + j) + 0.5f, (float)(xb + j) + 0.5f);
    const f2 pyc = pk((float)py + 0.5f, (float)py + 0.5f);
    const float kq = -0.72134752044448170f;  // -log2(e) / 2
    const f2 kq2 = pk(kq, kq);
    float T[8];
    float D[4][4];
    int cnt[8];
    f2 AD[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        T[j] = 1.0f;
        cnt[j] = 0;
        AD[j] = 0ull;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) D[i][0] = D[i][1] = D[i][2] = D[i][3] = 0.0f;

    int head = 0, count = 0;          // unprocessed candidates: ring slots [head, head + count)
    uint64_t clamp_mask = 0;          // ring slots whose opacity exceeds 0.99
    const bool freeze = may_freeze<kAux, kDepth>(args);
    bool live = true;                 // T is still updated
    auto chunk = [&]() {
        const bool clamp = ((clamp_mask >> head) & 0xFFull) != 0;
        if (kAux || live) {
            if (clamp)
                tc_chunk<kCount, true, kDepth, true>(geo, wt, head, g, t, pxc, pyc, kq2, T, D, cnt, wd, AD);
            else
                tc_chunk<kCount, false, kDepth, true>(geo, wt, head, g, t, pxc, pyc, kq2, T, D, cnt, wd, AD);
        } else {
            if (clamp)
                tc_chunk<kCount, true, kDepth, false>(geo, wt, head, g, t, pxc, pyc, kq2, T, D, cnt, wd, AD);
            else
                tc_chunk<kCount, false, kDepth, false>(geo, wt, head, g, t, pxc, pyc, kq2, T, D, cnt, wd, AD);
        }
    };
    // prefetch of the next batch: everything the block test and staging need
    float4 a_n = make_float4(0.f, 0.f, 0.f, 0.f);
    float2 b_n = make_float2(0.f, 0.f);
    uint4 w_n = make_uint4(0u, 0u, 0u, 0u);
    float d_n = 0.f;                      // depth image: -w d
    // list entries are fetched two batches ahead and their records one batch
    // ahead, so the dependent record loads never wait on the list load
    uint32_t gid_nn = 0;
    if (start + lane < end) {
        const uint32_t gid = __ldg(&args.gids[start + lane]);
        a_n = __ldg(&args.rec[gid].a);
        b_n = __ldg(reinterpret_cast<const float2 *>(&args.rec[gid].b));
        w_n = __ldg(&args.wt16[gid]);
        if constexpr (kDepth) d_n = __ldg(&args.rec[gid].c.w);
    }
    if (start + 32 + lane < end) gid_nn = __ldg(&args.gids[start + 32 + lane]);
    for (uint32_t base = start; base < end; base += 32) {
        const uint32_t j = base + lane;
        const float4 a = a_n;
        const float2 b = b_n;
        const uint4 wv = w_n;
        const float dv = d_n;
        const bool cand =
            j < end && (no_cull || block_may_hit(a.x, a.y, a.z, a.w, b.x, bcx, bcy, 3.5f, 3.5f));
        if (j + 32 < end) {
            const uint32_t gid = gid_nn;
            a_n = __ldg(&args.rec[gid].a);
            b_n = __ldg(reinterpret_cast<const float2 *>(&args.rec[gid].b));
            w_n = __ldg(&args.wt16[gid]);
            if constexpr (kDepth) d_n = __ldg(&args.rec[gid].c.w);
        }
        if (j + 64 < end) gid_nn = __ldg(&args.gids[j + 64]);
        const unsigned bal = __ballot_sync(0xffffffffu, cand);
        bool clamp = false;
        int pos = 0;
        if (cand) {
            pos = (head + count + __popc(bal & ((1u << lane) - 1u))) & (kRing - 1);
            float *q = reinterpret_cast<float *>(&geo[0][pos >> 1]);
            const int o = pos & 1;
            q[o] = a.x;
            q[2 + o] = a.y;
            q = reinterpret_cast<float *>(&geo[1][pos >> 1]);
            q[o] = a.z;
            q[2 + o] = a.w;
            q = reinterpret_cast<float *>(&geo[2][pos >> 1]);
            q[o] = b.x;
            q[2 + o] = b.y;
            clamp = b.y > kLogClamp;
            wt[pos] = wv;                        // FP16 weights written by preprocessing
            if constexpr (kDepth) reinterpret_cast<float *>(&wd[pos >> 1])[o] = -dv;
        }
        // slots of this batch that need the 0.99 clamp
        const unsigned cb = __ballot_sync(0xffffffffu, clamp);
        if (cb) {
            for (unsigned m = cb; m; m &= m - 1) {
                const int l = __ffs(m) - 1;
                const int p = __shfl_sync(0xffffffffu, pos, l);
                clamp_mask |= 1ull << p;
            }
        }
        __syncwarp();
        count += __popc(bal);
        while (count >= kChunk) {
            chunk();
            clamp_mask &= ~(0xFFull << head);
            head = (head + kChunk) & (kRing - 1);
            count -= kChunk;
        }
        if (freeze && live && ((base - start) & (kFreezeEvery - 1)) == kFreezeEvery - 32) {
            float m = T[0];
#pragma unroll
            for (int k = 1; k < 8; ++k) m = fmaxf(m, T[k]);
            live = !all_frozen(args, m);
        }
        __syncwarp();
    }
    if (count > 0) {
        // pad the last chunk with entries that include no pixel and weigh 0
        if (lane < kChunk - count) {
            const int pos = (head + count + lane) & (kRing - 1);
            const int o = pos & 1;
            float *q = reinterpret_cast<float *>(&geo[0][pos >> 1]);
            q[o] = 1e30f;
            q[2 + o] = 1e30f;
            q = reinterpret_cast<float *>(&geo[1][pos >> 1]);
            q[o] = 1.0f;
            q[2 + o] = 0.0f;
            q = reinterpret_cast<float *>(&geo[2][pos >> 1]);
            q[o] = 1.0f;
            q[2 + o] = 0.0f;
            wt[pos] = make_uint4(0u, 0u, 0u, 0u);
            if constexpr (kDepth) reinterpret_cast<float *>(&wd[pos >> 1])[o] = 0.0f;
        }
        __syncwarp();
        chunk();
    }

    // Quad reduction: columns c and c + 4 (lanes t, t ^ 2), then swap halves
    // (lanes t, t ^ 1); T and counts multiply / add over the four lanes.
    float v[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int k = 0; k < 4; ++k) v[i][k] = D[i][k] + __shfl_xor_sync(0xffffffffu, D[i][k], 2);
    float o[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int k = 0; k < 4; ++k) o[i][k] = __shfl_xor_sync(0xffffffffu, v[i][k], 1);
    float ad[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        if constexpr (kDepth) {
            float x, y;
            upk(AD[k], x, y);
            ad[k] = x + y;
            ad[k] += __shfl_xor_sync(0xffffffffu, ad[k], 1);
            ad[k] += __shfl_xor_sync(0xffffffffu, ad[k], 2);
        }
        T[k] *= __shfl_xor_sync(0xffffffffu, T[k], 1);
        T[k] *= __shfl_xor_sync(0xffffffffu, T[k], 2);
        if (kCount) {
            cnt[k] += __shfl_xor_sync(0xffffffffu, cnt[k], 1);
            cnt[k] += __shfl_xor_sync(0xffffffffu, cnt[k], 2);
        }
    }
    if (py >= cam.height) return;
    const float inv = 1.0f / wscale;
    const int64_t HW = (int64_t)cam.width * cam.height;
    const bool even = (t & 1) == 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (i != t) continue;   // lane t writes pixels 2t, 2t + 1
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int x = xb + 2 * i + h;
            if (x >= cam.width) break;
            // v / o: (A_r, A_g) on even lanes, (A_b, B) on odd lanes; k = 2h, 2h + 1
            const float ar = (even ? v[i][2 * h] : o[i][2 * h]) * inv;
            const float ag = (even ? v[i][2 * h + 1] : o[i][2 * h + 1]) * inv;
            const float ab = (even ? o[i][2 * h] : v[i][2 * h]) * inv;
            const float bb = (even ? o[i][2 * h + 1] : v[i][2 * h + 1]) * inv;
            const float tr = T[2 * i + h];
            const int64_t p = (int64_t)py * cam.width + x;
            const float fg = bb > 0.0f ? (1.0f - tr) / bb : 0.0f;
            float *out = args.out_rgb + 3 * p;
            out[0] = fmaf(fg, ar, tr * args.bg[0]);
            out[1] = fmaf(fg, ag, tr * args.bg[1]);
            out[2] = fmaf(fg, ab, tr * args.bg[2]);
            if (kAux) {
                args.out_aux[p] = ar;
                args.out_aux[HW + p] = ag;
                args.out_aux[2 * HW + p] = ab;
                args.out_aux[3 * HW + p] = bb;
                args.out_aux[4 * HW + p] = tr;
            }
            if (kCount) args.out_count[p] = cnt[2 * i + h];
            // FP32 numerator over the tensor-core B (both unscaled)
            if (kDepth) args.out_depth[p] = bb > 0.0f ? ad[2 * i + h] / bb : 0.0f;
        }
    }
}

// Accumulates one staged Gaussian into a thread's four pixels (two pairs).
template <bool kCount, bool kDepth>
__device__ __forceinline__ void accumulate_wide(const ulonglong2 (*wb)[32], int k, f2 pxa, f2 pxb,
                                           f2 pyc, f2 kq2, f2 (&A)[2][3], f2 (&B)[2],
                                           f2 (&T)[2], f2 (&AD)[2], int (&cnt)[4]) {
    const ulonglong2 s0 = wb[0][k], s1 = wb[1][k], s2 = wb[2][k];
    // inclusion test (exact FP32 sequence); the row terms are shared by both pairs
    const f2 dy = sub2(pyc, s0.y);
    const f2 ldy = mul2(s1.y, dy);
    const f2 e2 = mul2(s2.x, dy);
    const f2 e2s = mul2(e2, e2);
    const f2 dxa = sub2(pxa, s0.x);
    const f2 dxb = sub2(pxb, s0.x);
    const f2 e1a = fma2(s1.x, dxa, ldy);
    const f2 e1b = fma2(s1.x, dxb, ldy);
    const f2 qa = fma2(e1a, e1a, e2s);
    const f2 qb = fma2(e1b, e1b, e2s);
    // a = min(0.99, o 2^(-q log2(e) / 2)), kept negated
    const f2 ga = fma2(qa, kq2, s2.y);
    const f2 gb = fma2(qb, kq2, s2.y);
    float q[4], g[4], n[4];
    upk(qa, q[0], q[1]);
    upk(qb, q[2], q[3]);
    upk(ga, g[0], g[1]);
    upk(gb, g[2], g[3]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        n[i] = q[i] <= 9.0f ? fmaxf(-ex2(g[i]), -0.99f) : 0.0f;
        if (kCount) cnt[i] += q[i] <= 9.0f;
    }
    const ulonglong2 s3 = wb[3][k], s4 = wb[4][k];
    const f2 na[2] = {pk(n[0], n[1]), pk(n[2], n[3])};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        A[h][0] = fma2(na[h], s3.y, A[h][0]);
        A[h][1] = fma2(na[h], s4.x, A[h][1]);
        A[h][2] = fma2(na[h], s4.y, A[h][2]);
        B[h] = fma2(na[h], s3.x, B[h]);
        T[h] = fma2(na[h], T[h], T[h]);
    }
    if (kDepth) {
        const ulonglong2 s5 = wb[5][k];   // {-w d, -w d, 0, 0}
        AD[0] = fma2(na[0], s5.x, AD[0]);
        AD[1] = fma2(na[1], s5.x, AD[1]);
    }
}

// FMA tile code inside the tensor-core kernels: wide tiles of FP16 views and every tile
// of an FP32 view in the batched kernel.  Two warps; warp w owns the 16x8 pixel block of
// rows 8w..8w+7, lane l the four pixels (4 (l & 3) .. +3, l >> 2) of that block.  Each
// warp streams the tile's list on its own (no block-wide barrier): 32 entries at a time,
// one per lane (the next 32 are fetched while the current ones are accumulated), are
// tested against the warp's block, compacted into the warp's shared-memory buffer
// (ballot) and accumulated by all lanes.
//
// raster_tile is 1.27 times as fast where it is a kernel's only code, but its eight
// pixels per lane cost the code around it more than wide tiles, which are rare, can give
// back: in k_raster_tc, where the tensor-core tiles then took 0.861 ms at 600k Gaussians,
// 1600x1063, they took 0.96 ms beside it inlined and 0.876 ms with it out of line.  In
// k_raster_batch it takes 128 registers instead of 112 and gains nothing: bursts of twelve
// FP32 views of 40k to 160k Gaussians 1.238 ms against 1.239 ms here, of 150k to 600k
// 4.05 against 4.08 ms.
template <bool kAux, bool kCount, bool kDepth = false>
__device__ __forceinline__ void raster_tile_wide(const RenderArgs &args, int tile,
                                            ulonglong2 (*buf)[kDepth ? 6 : 5][32]) {
    const DevCamera &cam = args.cam;
    const int tx = tile % cam.tiles_x, ty = tile / cam.tiles_x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int bx0 = tx * kTile, by0 = ty * kTile + 8 * warp;
    const int px = bx0 + 4 * (lane & 3);
    const int py = by0 + (lane >> 2);

    const uint32_t start = args.tile_offsets[tile];
    const uint32_t end = args.tile_offsets[tile + 1];
    const bool no_cull = (args.flags & MGS_FLAG_NO_CULL) != 0;
    const float bx = (float)bx0 + 8.0f, by = (float)by0 + 4.0f;

    const f2 pxa = pk((float)px + 0.5f, (float)px + 1.5f);
    const f2 pxb = pk((float)px + 2.5f, (float)px + 3.5f);
    const f2 pyc = pk((float)py + 0.5f, (float)py + 0.5f);
    const float kq = -0.72134752044448170f;  // -log2(e) / 2
    const f2 kq2 = pk(kq, kq);
    f2 A[2][3] = {{0ull, 0ull, 0ull}, {0ull, 0ull, 0ull}};
    f2 B[2] = {0ull, 0ull};
    f2 T[2] = {pk(1.0f, 1.0f), pk(1.0f, 1.0f)};
    f2 AD[2] = {0ull, 0ull};
    int cnt[4] = {0, 0, 0, 0};
    ulonglong2(*wb)[32] = buf[warp];

    // list entries two batches ahead, their records one batch ahead (the
    // dependent record loads never wait on the list load)
    float4 a_n = make_float4(0.f, 0.f, 0.f, 0.f), b_n = a_n, c_n = a_n;
    uint32_t gid_nn = 0;
    if (start + lane < end) {
        const uint32_t gid = __ldg(&args.gids[start + lane]);
        a_n = __ldg(&args.rec[gid].a);
        b_n = __ldg(&args.rec[gid].b);
        c_n = __ldg(&args.rec[gid].c);
    }
    if (start + 32 + lane < end) gid_nn = __ldg(&args.gids[start + 32 + lane]);
    for (uint32_t base = start; base < end; base += 32) {
        const uint32_t j = base + lane;
        const float4 a = a_n, b = b_n, c = c_n;
        const bool cand =
            j < end && (no_cull || block_may_hit(a.x, a.y, a.z, a.w, b.x, bx, by, 7.5f, 3.5f));
        if (j + 32 < end) {
            const uint32_t gid = gid_nn;
            a_n = __ldg(&args.rec[gid].a);
            b_n = __ldg(&args.rec[gid].b);
            c_n = __ldg(&args.rec[gid].c);
        }
        if (j + 64 < end) gid_nn = __ldg(&args.gids[j + 64]);
        const unsigned bal = __ballot_sync(0xffffffffu, cand);
        if (cand) {
            const int pos = __popc(bal & ((1u << lane) - 1u));
            wb[0][pos] = make_ulonglong2(pk(a.x, a.x), pk(a.y, a.y));
            wb[1][pos] = make_ulonglong2(pk(a.z, a.z), pk(a.w, a.w));
            wb[2][pos] = make_ulonglong2(pk(b.x, b.x), pk(b.y, b.y));
            wb[3][pos] = make_ulonglong2(pk(b.z, b.z), pk(b.w, b.w));
            wb[4][pos] = make_ulonglong2(pk(c.x, c.x), pk(c.y, c.y));
            if (kDepth) wb[5][pos] = make_ulonglong2(pk(c.w, c.w), 0ull);   // -w d
        }
        __syncwarp();
        const int nc = __popc(bal);
#pragma unroll 2
        for (int k = 0; k < nc; ++k)
            accumulate_wide<kCount, kDepth>(wb, k, pxa, pxb, pyc, kq2, A, B, T, AD, cnt);
        __syncwarp();
    }

    if (py >= cam.height) return;
    float ar[4], ag[4], ab[4], bb[4], tt[4], ad[4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        upk(AD[h], ad[2 * h], ad[2 * h + 1]);
        upk(A[h][0], ar[2 * h], ar[2 * h + 1]);
        upk(A[h][1], ag[2 * h], ag[2 * h + 1]);
        upk(A[h][2], ab[2 * h], ab[2 * h + 1]);
        upk(B[h], bb[2 * h], bb[2 * h + 1]);
        upk(T[h], tt[2 * h], tt[2 * h + 1]);
    }
    const int64_t HW = (int64_t)cam.width * cam.height;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int x = px + k;
        if (x >= cam.width) break;
        const int64_t p = (int64_t)py * cam.width + x;
        const float fg = bb[k] > 0.0f ? (1.0f - tt[k]) / bb[k] : 0.0f;
        float *o = args.out_rgb + 3 * p;
        o[0] = fmaf(fg, ar[k], tt[k] * args.bg[0]);
        o[1] = fmaf(fg, ag[k], tt[k] * args.bg[1]);
        o[2] = fmaf(fg, ab[k], tt[k] * args.bg[2]);
        if (kAux) {
            args.out_aux[p] = ar[k];
            args.out_aux[HW + p] = ag[k];
            args.out_aux[2 * HW + p] = ab[k];
            args.out_aux[3 * HW + p] = bb[k];
            args.out_aux[4 * HW + p] = tt[k];
        }
        if (kCount) args.out_count[p] = cnt[k];
        if (kDepth) args.out_depth[p] = bb[k] > 0.0f ? ad[k] / bb[k] : 0.0f;
    }
}

// Tensor-core accumulation is used for FP16-attribute scenes unless the
// caller asks for the FP32 FMA sums.
__host__ __device__ __forceinline__ bool use_tc(const RenderArgs &a) { return tc_raster(a); }

// One CTA per tile, longest tile lists first.
template <bool kAux, bool kCount, bool kDepth = false>
__global__ void __launch_bounds__(kThreads) k_raster(RenderArgs args) {
    grid_wait();
    __shared__ FmaSmem<kDepth> sm;
    if (args.status->last_pairs > args.capacity) return;  // overflowed: lists incomplete
    raster_tile<kAux, kCount, kDepth>(args, (int)(args.tile_order[blockIdx.x] & kTileMask), sm);
}

// Tiles that list a Gaussian whose weight the FP16 sums cannot hold next to
// the others (kTileWide, see kWideWeight) take the FP32 FMA tile code.
template <bool kAux, bool kCount, bool kDepth = false>
__global__ void __launch_bounds__(kThreads) k_raster_tc(RenderArgs args) {
    grid_wait();
    __shared__ union {
        TcSmem tc;
        ulonglong2 buf[2][kDepth ? 6 : 5][32];
    } sm;
    if (args.status->last_pairs > args.capacity) return;  // overflowed: lists incomplete
    const uint32_t ord = args.tile_order[blockIdx.x];
    const int tile = (int)(ord & kTileMask);
    if (ord & kTileWide) {
        if (threadIdx.x < 64) raster_tile_wide<kAux, kCount, kDepth>(args, tile, sm.buf);
    } else {
        raster_tile_tc<kAux, kCount, kDepth>(args, tile, sm.tc);
    }
}

// Persistent, batched: the tiles of several views (different scenes and
// resolutions) form one work list; resident CTAs pull (view, tile) items from
// an atomic counter until the list is exhausted.  Items are numbered view by
// view (prefix[v] = first item of view v), each view's tiles longest first.
// FP16 views use all four warps (tensor-core sums), FP32 views and wide tiles
// (kTileWide) the first two (FMA sums).
__global__ void __launch_bounds__(kThreads) k_raster_batch(const RenderArgs *__restrict__ views,
                                                             const int *__restrict__ prefix,
                                                             int nviews,
                                                             unsigned *__restrict__ counter) {
    __shared__ union {
        ulonglong2 buf[2][5][32];
        TcSmem tc;
    } sm;
    __shared__ int item_s;
    const int total = prefix[nviews];
    for (;;) {
        if (threadIdx.x == 0) item_s = (int)atomicAdd(counter, 1u);
        __syncthreads();
        const int item = item_s;
        __syncthreads();
        if (item >= total) return;
        int lo = 0, hi = nviews - 1;       // last view with prefix[v] <= item
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (prefix[mid] <= item) lo = mid; else hi = mid - 1;
        }
        const RenderArgs &a = views[lo];
        if (a.status->last_pairs > a.capacity) continue;   // that view overflowed
        const uint32_t ord = a.tile_order[item - prefix[lo]];
        const int tile = (int)(ord & kTileMask);
        if (use_tc(a) && !(ord & kTileWide))
            raster_tile_tc<false, false>(a, tile, sm.tc);
        else if (threadIdx.x < 64)
            raster_tile_wide<false, false>(a, tile, sm.buf);
    }
}

template <bool kAux, bool kCount>
cudaError_t launch_t(const RenderArgs &a, cudaStream_t stream) {
    const int T = a.cam.tiles_x * a.cam.tiles_y;
    if (use_tc(a))
        return launch_dependent(k_raster_tc<kAux, kCount>, T, kThreads, 0, stream, a);
    return launch_dependent(k_raster<kAux, kCount>, T, kThreads, 0, stream, a);
}

}  // namespace

cudaError_t launch_raster(const RenderArgs &a, cudaStream_t stream) {
    const bool aux = a.out_aux != nullptr, cnt = a.out_count != nullptr;
    if (a.out_depth) {   // depth image (Eq. 5), no aux / count outputs
        const int T = a.cam.tiles_x * a.cam.tiles_y;
        if (use_tc(a)) return launch_dependent(k_raster_tc<false, false, true>, T, kThreads, 0, stream, a);
        return launch_dependent(k_raster<false, false, true>, T, kThreads, 0, stream, a);
    }
    if (aux && cnt) return launch_t<true, true>(a, stream);
    if (aux) return launch_t<true, false>(a, stream);
    if (cnt) return launch_t<false, true>(a, stream);
    return launch_t<false, false>(a, stream);
}

}  // namespace mgs

namespace mgs {

cudaError_t launch_raster_batch(const RenderArgs *views_dev, const int *prefix_dev, int nviews,
                                unsigned *counter_dev, int sm_count, cudaStream_t stream) {
    cudaError_t e = cudaMemsetAsync(counter_dev, 0, sizeof(unsigned), stream);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_raster_batch, kThreads, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    k_raster_batch<<<sm_count * per_sm, kThreads, 0, stream>>>(views_dev, prefix_dev, nviews,
                                                                 counter_dev);
    return cudaGetLastError();
}

}  // namespace mgs
