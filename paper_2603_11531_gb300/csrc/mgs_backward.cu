// Backward pass: the adjoint of the forward render (Sec. 3.1 Eq. 2-4, Sec. 3.2,
// App. B), for training through torch.autograd.
//
// Per pixel p with C = (1 - T) A / B + T c_bg, r = A / B, G = dL/dC(p):
//   dL/dc_i  += (1 - T)/B * a_i w_i G
//   dL/dw_i  += (1 - T)/B * a_i G.(c_i - r)
//   dL/da_i  += w_i (1 - T)/B G.(c_i - r) - T/(1 - a_i) G.(c_bg - r)
// and through a_i = o_i exp(-q/2) (zero when the 0.99 clamp is active) to
// o_i, the pixel mean and the covariance.  All of these only need (A, B, T) of the
// forward, so the backward is as order-independent as the forward.
//
//   k_raster_bwd      one warp per 8x8 block, lane = Gaussian: a lane sums its
//                     Gaussian's partials over the block's pixels in registers
//                     and adds them to a per-Gaussian gradient record.
//   k_preprocess_bwd  one thread per Gaussian: recomputes the forward, chains
//                     through the EWA covariance, projection, SH colour,
//                     Eq. 3 weight and (warp-cooperatively) the Eq. 4 MLP.
//                     The MLP's deltas and weight gradients are TF32 mma.sync
//                     products (FP32 accumulation); weight gradients stay in
//                     registers across the CTA's rows, are written once per
//                     CTA and reduced in a fixed order by k_mlp_grad_reduce.
#include "mgs_internal.cuh"
#include "mgs_mlp.cuh"

namespace mgs {
namespace {

constexpr int kBwdThreads = 128;  // raster backward: four warps per CTA, one 8x8 block each
constexpr int kBwdWarps = kBwdThreads / 32;
constexpr int kBwdRing = 64;      // candidate slots per warp (a power of two)
constexpr int kGRec = 12;         // per-Gaussian raster gradient record
// layout: dc(3), dw, do, dm(2), M(3), pad(2), with M the second moments of s =
// -2 dL/dq in the whitened coordinates e = L^T (pixel - mean) of the inclusion
// test: sum s e1^2, sum s e1 e2, sum s e2^2.  dL/dSigma_2D = L M L^T / 2 and
// dL/dm = L sum(s e) then have no cancelling terms, which the moments of
// (dx, dy) have for elongated Gaussians.

typedef unsigned long long f2;    // two packed FP32 lanes: two adjacent pixels
__device__ __forceinline__ f2 pk(float lo, float hi) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void upk(f2 v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ float hsum(f2 v) {
    float lo, hi;
    upk(v, lo, hi);
    return lo + hi;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
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
__device__ __forceinline__ float ex2f(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcpf(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// p[0..3] += (a, b, c, d), p 16-byte aligned, without a result
__device__ __forceinline__ void red4(float *p, float a, float b, float c, float d) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c),
                 "f"(d)
                 : "memory");
}

// Shared memory of the rasteriser adjoint, per warp: the constants of the
// block's 32 horizontal pixel pairs (pair 4 y + x / 2), and the candidate ring.
//   px0 = {k_A G_r (2 pixels), k_A G_g (2)}, px1 = {k_A G_b (2), -k_A G.r (2)},
//   px2 = {-T G.(c_bg - r) (2)}
//   ring[0] = {m_x, m_y, l11, l21}, ring[1] = {l22, log2 o, 1 / o, w},
//   ring[2] = {c_r, c_g, c_b, Gaussian index}
struct BwdRaster {
    float4 px0[kBwdWarps][32], px1[kBwdWarps][32];
    float2 px2[kBwdWarps][32];
    float4 ring[kBwdWarps][3][kBwdRing];
};

// How a batch treats the pixels: kFast (every product of an excluded pixel finite,
// no opacity above 0.99: its alpha is 0 and so is everything it adds), kClamped
// (some opacity above 0.99) and kGuarded (a pixel constant is not finite, or some
// candidate's weight or colour is so large, or not finite, that its products with
// the block's pixel constants may leave the FP32 range, where 0 times them is NaN:
// excluded pixels are skipped, so that they add nothing).
enum BwdMode { kFast, kClamped, kGuarded };
constexpr float kSafeProduct = 1e38f;   // FP32's largest number is 3.4e38

__device__ __forceinline__ float warp_max(float v) {   // v >= 0, or NaN
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}

// One batch: lane = one candidate, looping over the warp's 8x8 block at (bx0,
// by0); adds the candidate's ten partials to its gradient record.
//   per pixel with q <= 9 (a = min(a_raw, 0.99), u = k_A (G.c - G.r)):
//     dc  += w a k_A G       dw += a u
//   and, where the clamp is inactive, with s = a (w u - T G.(c_bg - r) / (1 - a)):
//     do  += s / o,  and s e1, s e2, s e1^2, s e1 e2, s e2^2 for the mean and
//     covariance terms (e2 is the same for a row: its moments are taken row by row).
template <int kMode>
__device__ __forceinline__ void bwd_batch(const BwdRaster &sm, int warp, int slot, bool active,
                                          int bx0, int by0, float *__restrict__ gG) {
    const float4 *px0 = sm.px0[warp], *px1 = sm.px1[warp];
    const float2 *px2 = sm.px2[warp];
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = make_float4(0.f, -INFINITY, 0.f, 0.f), c = a;
    if (active) {
        a = sm.ring[warp][0][slot];
        b = sm.ring[warp][1][slot];
        c = sm.ring[warp][2][slot];
    }
    const float my = a.y, l21 = a.w, l22 = b.x;
    const f2 l11 = pk(a.z, a.z), lo = pk(b.y, b.y), w = pk(b.w, b.w);
    const f2 c0 = pk(c.x, c.x), c1 = pk(c.y, c.y), c2 = pk(c.z, c.z);
    const float kq = -0.72134752044448170f;  // -log2(e) / 2
    const f2 kq2 = pk(kq, kq), one = pk(1.0f, 1.0f), mx = pk(a.x, a.x);
    f2 dx[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
        dx[j] = sub2(pk((float)(bx0 + 2 * j) + 0.5f, (float)(bx0 + 2 * j) + 1.5f), mx);
    f2 sc0 = 0ull, sc1 = 0ull, sc2 = 0ull, sw = 0ull, m11 = 0ull;
    float s0 = 0.f, se1 = 0.f, se2 = 0.f, m12 = 0.f, m22 = 0.f;
#pragma unroll 2
    for (int r = 0; r < 8; ++r) {
        const float dy = __fsub_rn((float)(by0 + r) + 0.5f, my);
        const float ldys = __fmul_rn(l21, dy);
        const float e2 = __fmul_rn(l22, dy);
        const float e2q = __fmul_rn(e2, e2);
        const f2 ldy = pk(ldys, ldys), e2s = pk(e2q, e2q);
        f2 r0 = 0ull, r1 = 0ull;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 p0 = px0[4 * r + j], p1 = px1[4 * r + j];
            const float2 p2 = px2[4 * r + j];
            const f2 e1 = fma2(l11, dx[j], ldy);
            const f2 q = fma2(e1, e1, e2s);
            const f2 g = fma2(q, kq2, lo);
            float qa, qb, ga, gb;
            upk(q, qa, qb);
            upk(g, ga, gb);
            float aa = ex2f(ga), ab = ex2f(gb);
            const bool ia = qa <= 9.0f, ib = qb <= 9.0f;
            bool ua = true, ub = true;   // clamp inactive
            if constexpr (kMode != kFast) {
                ua = aa < 0.99f;
                ub = ab < 0.99f;
                aa = fminf(aa, 0.99f);
                ab = fminf(ab, 0.99f);
            }
            aa = ia ? aa : 0.0f;
            ab = ib ? ab : 0.0f;
            const f2 al = pk(aa, ab);
            f2 k0 = pk(p0.x, p0.y), k1 = pk(p0.z, p0.w), k2 = pk(p1.x, p1.y);
            f2 kr = pk(p1.z, p1.w), tg = pk(p2.x, p2.y);
            if constexpr (kMode == kGuarded) {   // excluded pixels: all constants 0
                k0 = pk(ia ? p0.x : 0.f, ib ? p0.y : 0.f);
                k1 = pk(ia ? p0.z : 0.f, ib ? p0.w : 0.f);
                k2 = pk(ia ? p1.x : 0.f, ib ? p1.y : 0.f);
                kr = pk(ia ? p1.z : 0.f, ib ? p1.w : 0.f);
                tg = pk(ia ? p2.x : 0.f, ib ? p2.y : 0.f);
            }
            sc0 = fma2(al, k0, sc0);
            sc1 = fma2(al, k1, sc1);
            sc2 = fma2(al, k2, sc2);
            f2 u = fma2(k0, c0, fma2(k1, c1, fma2(k2, c2, kr)));
            // 1 - a >= 0.01: the fast reciprocal is accurate to a few ulp
            float na, nb;
            upk(sub2(one, al), na, nb);
            const f2 inv = pk(rcpf(na), rcpf(nb));
            f2 s;
            if constexpr (kMode == kGuarded) {
                float u0, u1;
                upk(u, u0, u1);
                u = pk(ia ? u0 : 0.f, ib ? u1 : 0.f);   // a non-finite colour times 0
                sw = fma2(al, u, sw);
                float v0, v1;
                upk(mul2(al, fma2(w, u, mul2(tg, inv))), v0, v1);
                s = pk(ia && ua ? v0 : 0.f, ib && ub ? v1 : 0.f);
            } else {
                sw = fma2(al, u, sw);
                s = mul2(al, fma2(w, u, mul2(tg, inv)));
                if constexpr (kMode == kClamped) {
                    float v0, v1;
                    upk(s, v0, v1);
                    s = pk(ua ? v0 : 0.f, ub ? v1 : 0.f);
                }
            }
            const f2 sx = mul2(s, e1);
            r0 = add2(r0, s);
            r1 = add2(r1, sx);
            m11 = fma2(sx, e1, m11);
        }
        const float t0 = hsum(r0), t1 = hsum(r1), t2 = e2 * t0;
        s0 += t0;
        se1 += t1;
        se2 += t2;
        m12 = fmaf(e2, t1, m12);
        m22 = fmaf(e2, t2, m22);
    }
    if (!active) return;
    // dL/dq = -s / 2 per pixel and q = e^T e with e = L^T (pixel - m): dq/dm = -2 L e
    const float io = b.z;
    float acc[10];
    acc[0] = b.w * hsum(sc0);
    acc[1] = b.w * hsum(sc1);
    acc[2] = b.w * hsum(sc2);
    acc[3] = hsum(sw);
    acc[4] = s0 * io;
    acc[5] = a.z * se1;
    acc[6] = fmaf(l21, se1, l22 * se2);
    acc[7] = hsum(m11);
    acc[8] = m12;
    acc[9] = m22;
    float *rec = gG + (size_t)__float_as_uint(c.w) * kGRec;
    if (acc[0] != 0.f || acc[1] != 0.f || acc[2] != 0.f || acc[3] != 0.f)
        red4(rec, acc[0], acc[1], acc[2], acc[3]);
    if (io > 0.0f) {   // o = 0: no gradient through alpha
        if (acc[4] != 0.f || acc[5] != 0.f || acc[6] != 0.f || acc[7] != 0.f)
            red4(rec + 4, acc[4], acc[5], acc[6], acc[7]);
        if (acc[8] != 0.f || acc[9] != 0.f) red4(rec + 8, acc[8], acc[9], 0.f, 0.f);
    }
}

// Rasteriser adjoint.  `splits` CTAs per tile, each taking an equal share of the
// tile's list; warp w owns the 8x8 block at (8 (w % 2), 8 (w / 2)) and streams
// the share on its own, 32 entries at a time (one per lane), testing them
// against its block and queueing the candidates in its ring.  Every 32
// candidates make a batch in which a lane holds one Gaussian and loops over
// the block's 64 pixels, whose constants all lanes read from shared memory
// by broadcast: the ten partials of a (Gaussian, block) are plain register
// sums, so nothing is reduced across lanes, and the three 16-byte reductions
// per (Gaussian, block) are the only other traffic.
//
// Bound: the FP32 FMA pipe (19 packed operations of two cycles each per pixel
// pair, 0.36 ms for the pairs below) and issue.  Measured at 300k Gaussians,
// 1296x840 (12 M (block, Gaussian) pairs): 0.69 ms, 0.53 G instructions, FMA
// pipe 60 % busy.  The layout it replaced (lane = four pixels of a 16x8 block,
// ten partials per candidate reduced through shared memory, ten scalar
// atomics) took 1.85 ms and 1.52 G instructions; at 30k, 333x251 (336 tiles)
// 0.27 against 0.06 ms, there also because the lists are split over CTAs.
// Bounding each candidate's products takes 0.01 ms of it.  Variants that were
// slower than 0.67 ms without that: 80 registers for six CTAs per SM (0.69 ms,
// spills), pairs unrolled by two instead of four (0.78 ms).
__global__ void __launch_bounds__(kBwdThreads) k_raster_bwd(RenderArgs args,
                                                            const float *__restrict__ dL,
                                                            const float *__restrict__ aux,
                                                            float *__restrict__ gG, int splits) {
    __shared__ BwdRaster sm;
    const DevCamera &cam = args.cam;
    const int tile = (int)(args.tile_order[blockIdx.x / splits] & kTileMask);
    const int split = blockIdx.x % splits;
    const int tx = tile % cam.tiles_x, ty = tile / cam.tiles_x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int bx0 = tx * kTile + 8 * (warp & 1), by0 = ty * kTile + 8 * (warp >> 1);
    if (args.status->last_pairs > args.capacity) return;
    const uint32_t t0 = args.tile_offsets[tile], t1 = args.tile_offsets[tile + 1];
    const uint32_t share = ((t1 - t0 + 31) / 32 + splits - 1) / splits * 32;   // whole batches
    const uint32_t start = min((uint64_t)t0 + (uint64_t)split * share, (uint64_t)t1);
    const uint32_t end = min((uint64_t)start + share, (uint64_t)t1);
    if (start >= end) return;

    // this lane's pixel pair: constants from the forward's (A, B, T) and dL/dC,
    // with k_A = (1 - T) / B and r = A / B (all zero without coverage)
    bool finite = true;
    float k_lane = 0.f, kr_lane = 0.f, tg_lane = 0.f;
    {
        const int64_t HW = (int64_t)cam.width * cam.height;
        const int py = by0 + (lane >> 2), x0 = bx0 + 2 * (lane & 3);
        float k[5][2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
            for (int e = 0; e < 5; ++e) k[e][h] = 0.f;
            if (x0 + h < cam.width && py < cam.height) {
                const int64_t p = (int64_t)py * cam.width + x0 + h;
                const float B = aux[3 * HW + p];
                if (B > 0.0f) {
                    const float T = aux[4 * HW + p];
                    const float inv = 1.0f / B;
                    const float kA = (1.0f - T) * inv;
                    float G[3], r[3];
#pragma unroll
                    for (int ch = 0; ch < 3; ++ch) {
                        G[ch] = dL[3 * p + ch];
                        r[ch] = aux[ch * HW + p] * inv;
                        k[ch][h] = kA * G[ch];
                    }
                    k[3][h] = -kA * (G[0] * r[0] + G[1] * r[1] + G[2] * r[2]);
                    k[4][h] = -T * (G[0] * (args.bg[0] - r[0]) + G[1] * (args.bg[1] - r[1]) +
                                    G[2] * (args.bg[2] - r[2]));
                }
            }
#pragma unroll
            for (int e = 0; e < 5; ++e) finite &= isfinite(k[e][h]);
            k_lane = fmaxf(k_lane, fabsf(k[0][h]) + fabsf(k[1][h]) + fabsf(k[2][h]));
            kr_lane = fmaxf(kr_lane, fabsf(k[3][h]));
            tg_lane = fmaxf(tg_lane, fabsf(k[4][h]));
        }
        sm.px0[warp][lane] = make_float4(k[0][0], k[0][1], k[1][0], k[1][1]);
        sm.px1[warp][lane] = make_float4(k[2][0], k[2][1], k[3][0], k[3][1]);
        sm.px2[warp][lane] = make_float2(k[4][0], k[4][1]);
    }
    const bool px_finite = __all_sync(0xffffffffu, finite);
    // block maxima of |k_A G_r| + |k_A G_g| + |k_A G_b|, |k_A G.r| and |T G.(c_bg - r)|
    // (finite non-negative floats order as unsigned integers)
    const float k_max = warp_max(k_lane), kr_max = warp_max(kr_lane), tg_max = warp_max(tg_lane);
    const float bx = (float)bx0 + 4.0f, by = (float)by0 + 4.0f;
    const float kLogClamp = -0.014499569695115089f;   // log2(0.99)
    float4(*ring)[kBwdRing] = sm.ring[warp];

    int head = 0, count = 0;   // queued candidates: ring slots [head, head + count)
    auto batch = [&](int n) {
        const int slot = (head + lane) & (kBwdRing - 1);
        const bool active = lane < n;
        bool special = false, clamp = false;
        if (active) {
            const float4 b = ring[1][slot], c = ring[2][slot];
            // bounds u and w u + tg of every excluded pixel (1 - a = 1 there), and
            // fails for a NaN
            const float c_max = fmaxf(fmaxf(fabsf(c.x), fabsf(c.y)), fabsf(c.z));
            const float u_max = fmaf(k_max, c_max, kr_max);
            special = !(fmaf(fmaxf(fabsf(b.w), 1.0f), u_max, tg_max) < kSafeProduct &&
                        fabsf(b.w) + fabsf(c.x) + fabsf(c.y) + fabsf(c.z) < INFINITY);
            clamp = !(b.y <= kLogClamp);
        }
        if (!px_finite || __any_sync(0xffffffffu, special))
            bwd_batch<kGuarded>(sm, warp, slot, active, bx0, by0, gG);
        else if (__any_sync(0xffffffffu, clamp))
            bwd_batch<kClamped>(sm, warp, slot, active, bx0, by0, gG);
        else
            bwd_batch<kFast>(sm, warp, slot, active, bx0, by0, gG);
        __syncwarp();
    };
    // list entries two batches ahead, their records one batch ahead
    uint32_t gid_n = 0, gid_nn = 0;
    float4 a_n = make_float4(0.f, 0.f, 0.f, 0.f), b_n = a_n, c_n = a_n;
    if (start + lane < end) {
        gid_n = __ldg(&args.gids[start + lane]);
        a_n = __ldg(&args.rec[gid_n].a);
        b_n = __ldg(&args.rec[gid_n].b);
        c_n = __ldg(&args.rec[gid_n].c);
    }
    if (start + 32 + lane < end) gid_nn = __ldg(&args.gids[start + 32 + lane]);
    for (uint32_t base = start; base < end; base += 32) {
        const uint32_t j = base + lane;
        const uint32_t gid = gid_n;
        const float4 a = a_n, b = b_n, c = c_n;
        const bool cand = j < end && block_may_hit(a.x, a.y, a.z, a.w, b.x, bx, by, 3.5f, 3.5f);
        if (j + 32 < end) {
            gid_n = gid_nn;
            a_n = __ldg(&args.rec[gid_n].a);
            b_n = __ldg(&args.rec[gid_n].b);
            c_n = __ldg(&args.rec[gid_n].c);
        }
        if (j + 64 < end) gid_nn = __ldg(&args.gids[j + 64]);
        const unsigned bal = __ballot_sync(0xffffffffu, cand);
        if (cand) {
            const int pos = (head + count + __popc(bal & ((1u << lane) - 1u))) & (kBwdRing - 1);
            const float w = -b.z, o = exp2f(b.y);
            const float iw = 1.0f / w;
            ring[0][pos] = a;
            // 1 / o (0 when o = 0: no opacity gradient then; nor below FP32's smallest
            // normal number, where alpha is flushed to 0 and 1 / o may be infinite);
            // colour c = (-w c) / (-w)
            ring[1][pos] = make_float4(b.x, b.y, o >= 1.1754943508222875e-38f ? 1.0f / o : 0.0f, w);
            ring[2][pos] = make_float4(-b.w * iw, -c.x * iw, -c.y * iw, __uint_as_float(gid));
        }
        __syncwarp();
        count += __popc(bal);
        if (count >= 32) {
            batch(32);
            head = (head + 32) & (kBwdRing - 1);
            count -= 32;
        }
    }
    if (count > 0) batch(count);
}

// CTAs per tile of the rasteriser adjoint: images with few tiles split their
// lists so that about ten CTAs per SM are in flight.
int bwd_splits(int T, int sm_count) {
    const int s = (10 * sm_count + T - 1) / T;
    return s < 1 ? 1 : (s > 8 ? 8 : s);
}

// ---------------------------------------------------------------------------
// Preprocessing adjoint.
// ---------------------------------------------------------------------------

constexpr int kMlpGrad = kMlpHidden * kMlpIn + kMlpHidden + kMlpHidden * kMlpHidden +
                         kMlpHidden + kMlpOut * kMlpHidden + kMlpOut;  // 5957
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kMlpHidden * kMlpIn, kOffW2 = kOffB1 + kMlpHidden,
              kOffB2 = kOffW2 + kMlpHidden * kMlpHidden, kOffW3 = kOffB2 + kMlpHidden,
              kOffB3 = kOffW3 + kMlpOut * kMlpHidden;

// Row buffers of the MLP adjoint hold the CTA's 128 rows (row = warp * 32 +
// lane).  Strides: 72 floats per delta row make the transposed fragment
// loads of the weight-gradient products conflict-free; 8 per d3 row and 24
// per staged dx row.
constexpr int kRows = kMlpThreads;
constexpr int kDS = 72;
constexpr int kD3S = 8;
constexpr int kDxS = 24;
constexpr int kOnesCol = kMlpHidden;  // h1 column 64 holds 1: its products give dL/db2
constexpr int kXOnesCol = kMlpIn;     // x column 22 holds 1: its products give dL/db1

// About 108 KB, two CTAs per SM: d1 overwrites d2 once the products that
// need d2 are done, and dx reuses h2's space once h2 is no longer read.
struct BwdSmem {
    MlpSmem mlp;                          // weights, BF16 features x, head outputs
    __nv_bfloat16 h1[kRows * kHStride];   // BF16 hidden activations (forward recompute)
    union {
        __nv_bfloat16 h2[kRows * kHStride];
        float dx[kRows * kDxS];           // dL/d(features), staged for the row threads
    };
    float dd[kRows * kDS];                // dL/d(pre-activation 2), then of pre-activation 1
    float d3[kRows * kD3S];               // dL/d(head outputs), columns 5..7 zero
    float b3[kMlpThreads / 32][8];        // per-warp sums of d3
};
static_assert(kRows * kDxS * sizeof(float) <= kRows * kHStride * sizeof(__nv_bfloat16),
              "dx fits in h2's space");

// Weight-gradient accumulators of one lane (m16n8 fragments): warp w owns
// rows 16w..16w+15 of dW2 (nine n-tiles, the last one the b2 column), of dW1
// (three n-tiles; column 22 is b1) and of dW3^T.
struct WGradAcc {
    float w2[9][4];
    float w1[3][4];
    float w3[4];
};

__device__ __forceinline__ uint32_t to_tf32(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}
// A BF16 value as a TF32 operand (exact: BF16 keeps 8 significand bits).
__device__ __forceinline__ uint32_t bf_tf32(const __nv_bfloat16 *p) {
    return (uint32_t)(*reinterpret_cast<const unsigned short *>(p)) << 16;
}
// D += A B, m16n8k8, TF32 operands, FP32 accumulation.  Fragments (g = lane / 4,
// t = lane % 4): a = A[g][t], A[g+8][t], A[g][t+4], A[g+8][t+4]; b = B[t][g],
// B[t+4][g]; d = D[g][2t], D[g][2t+1], D[g+8][2t], D[g+8][2t+1].
__device__ __forceinline__ void mma_tf32(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                         uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ float2 relu_mask(const __nv_bfloat16 *h, float a, float b) {
    const __nv_bfloat162 m = *reinterpret_cast<const __nv_bfloat162 *>(h);
    return make_float2(__low2float(m) > 0.0f ? a : 0.0f, __high2float(m) > 0.0f ? b : 0.0f);
}

// The adjoint of the Eq. 4 MLP for the CTA's 128 rows (d3 in shared memory)
// runs in four steps, with a CTA barrier after each of the first three:
//   1. mlp_d2_warp      d2 = (d3 W3) * [h2 > 0] for the warp's 32 rows;
//   2. mlp_wgrad2_cta   dW2 += d2^T [h1 | 1] and dW3^T += h2^T d3;
//   3. mlp_d1_warp      d1 = (d2 W2) * [h1 > 0] over d2 in place and
//                       dx = d1 W1 into h2's space, for the warp's rows;
//   4. mlp_wgrad1_cta   dW1 += d1^T [x | 1].
// TF32 products, FP32 accumulation.

__device__ __forceinline__ void mlp_d2_warp(BwdSmem &sm, int warp, int lane) {
    const int g = lane >> 2, t = lane & 3;
#pragma unroll 1
    for (int mt = 0; mt < 2; ++mt) {
        const int r0 = warp * 32 + mt * 16 + g, r1 = r0 + 8;
        const uint32_t a0 = to_tf32(sm.d3[r0 * kD3S + t]), a1 = to_tf32(sm.d3[r1 * kD3S + t]);
        const uint32_t a2 = to_tf32(sm.d3[r0 * kD3S + t + 4]);
        const uint32_t a3 = to_tf32(sm.d3[r1 * kD3S + t + 4]);
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
            float c[4] = {0.f, 0.f, 0.f, 0.f};
            mma_tf32(c, a0, a1, a2, a3, bf_tf32(&sm.mlp.w3[t * kW2Stride + nt * 8 + g]),
                     bf_tf32(&sm.mlp.w3[(t + 4) * kW2Stride + nt * 8 + g]));
            const int col = nt * 8 + 2 * t;
            *reinterpret_cast<float2 *>(&sm.dd[r0 * kDS + col]) =
                relu_mask(&sm.h2[r0 * kHStride + col], c[0], c[1]);
            *reinterpret_cast<float2 *>(&sm.dd[r1 * kDS + col]) =
                relu_mask(&sm.h2[r1 * kHStride + col], c[2], c[3]);
        }
    }
}

// The d1 accumulators serve directly as the A fragments of dx = d1 W1,
// taking k = 2t and 2t + 1 of each step for fragment columns t and t + 4
// (B rows follow the same order).
__device__ __forceinline__ void mlp_d1_warp(BwdSmem &sm, int warp, int lane) {
    const int g = lane >> 2, t = lane & 3;
#pragma unroll 1
    for (int mt = 0; mt < 2; ++mt) {
        const int r0 = warp * 32 + mt * 16 + g, r1 = r0 + 8;
        float c[8][4];
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) c[nt][0] = c[nt][1] = c[nt][2] = c[nt][3] = 0.f;
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
            const int k0 = ks * 8;
            const uint32_t a0 = to_tf32(sm.dd[r0 * kDS + k0 + t]);
            const uint32_t a1 = to_tf32(sm.dd[r1 * kDS + k0 + t]);
            const uint32_t a2 = to_tf32(sm.dd[r0 * kDS + k0 + t + 4]);
            const uint32_t a3 = to_tf32(sm.dd[r1 * kDS + k0 + t + 4]);
#pragma unroll
            for (int nt = 0; nt < 8; ++nt)
                mma_tf32(c[nt], a0, a1, a2, a3, bf_tf32(&sm.mlp.w2[(k0 + t) * kW2Stride + nt * 8 + g]),
                         bf_tf32(&sm.mlp.w2[(k0 + t + 4) * kW2Stride + nt * 8 + g]));
        }
        __syncwarp();   // every lane has read this m-tile's d2 rows: overwrite them with d1
        float dx[3][4];
#pragma unroll
        for (int ft = 0; ft < 3; ++ft) dx[ft][0] = dx[ft][1] = dx[ft][2] = dx[ft][3] = 0.f;
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
            const int col = nt * 8 + 2 * t;
            const float2 e0 = relu_mask(&sm.h1[r0 * kHStride + col], c[nt][0], c[nt][1]);
            const float2 e1 = relu_mask(&sm.h1[r1 * kHStride + col], c[nt][2], c[nt][3]);
            *reinterpret_cast<float2 *>(&sm.dd[r0 * kDS + col]) = e0;
            *reinterpret_cast<float2 *>(&sm.dd[r1 * kDS + col]) = e1;
            const uint32_t a0 = to_tf32(e0.x), a1 = to_tf32(e1.x), a2 = to_tf32(e0.y),
                           a3 = to_tf32(e1.y);
#pragma unroll
            for (int ft = 0; ft < 3; ++ft)
                mma_tf32(dx[ft], a0, a1, a2, a3, bf_tf32(&sm.mlp.w1[col * kW1Stride + ft * 8 + g]),
                         bf_tf32(&sm.mlp.w1[(col + 1) * kW1Stride + ft * 8 + g]));
        }
#pragma unroll
        for (int ft = 0; ft < 3; ++ft) {
            const int col = ft * 8 + 2 * t;
            *reinterpret_cast<float2 *>(&sm.dx[r0 * kDxS + col]) = make_float2(dx[ft][0], dx[ft][1]);
            *reinterpret_cast<float2 *>(&sm.dx[r1 * kDxS + col]) = make_float2(dx[ft][2], dx[ft][3]);
        }
    }
}

// Weight gradients of the CTA's 128 rows into this lane's accumulators, each
// a sum over the rows (the K dimension), warp w taking output rows
// 16w..16w+15.
__device__ __forceinline__ void mlp_wgrad2_cta(const BwdSmem &sm, int warp, int lane, WGradAcc &acc) {
    const int g = lane >> 2, t = lane & 3;
    const int m0 = warp * 16 + g, m1 = m0 + 8;
#pragma unroll 2
    for (int ks = 0; ks < kRows / 8; ++ks) {
        const int ra = ks * 8 + t, rb = ra + 4;
        const uint32_t a0 = to_tf32(sm.dd[ra * kDS + m0]), a1 = to_tf32(sm.dd[ra * kDS + m1]);
        const uint32_t a2 = to_tf32(sm.dd[rb * kDS + m0]), a3 = to_tf32(sm.dd[rb * kDS + m1]);
#pragma unroll
        for (int nt = 0; nt < 9; ++nt)
            mma_tf32(acc.w2[nt], a0, a1, a2, a3, bf_tf32(&sm.h1[ra * kHStride + nt * 8 + g]),
                     bf_tf32(&sm.h1[rb * kHStride + nt * 8 + g]));
        mma_tf32(acc.w3, bf_tf32(&sm.h2[ra * kHStride + m0]), bf_tf32(&sm.h2[ra * kHStride + m1]),
                 bf_tf32(&sm.h2[rb * kHStride + m0]), bf_tf32(&sm.h2[rb * kHStride + m1]),
                 to_tf32(sm.d3[ra * kD3S + g]), to_tf32(sm.d3[rb * kD3S + g]));
    }
}

__device__ __forceinline__ void mlp_wgrad1_cta(const BwdSmem &sm, int warp, int lane, WGradAcc &acc) {
    const int g = lane >> 2, t = lane & 3;
    const int m0 = warp * 16 + g, m1 = m0 + 8;
    const __nv_bfloat16 *X = &sm.mlp.x[0][0];
#pragma unroll 2
    for (int ks = 0; ks < kRows / 8; ++ks) {
        const int ra = ks * 8 + t, rb = ra + 4;
        const uint32_t a0 = to_tf32(sm.dd[ra * kDS + m0]), a1 = to_tf32(sm.dd[ra * kDS + m1]);
        const uint32_t a2 = to_tf32(sm.dd[rb * kDS + m0]), a3 = to_tf32(sm.dd[rb * kDS + m1]);
#pragma unroll
        for (int ft = 0; ft < 3; ++ft)
            mma_tf32(acc.w1[ft], a0, a1, a2, a3, bf_tf32(&X[ra * kXStride + ft * 8 + g]),
                     bf_tf32(&X[rb * kXStride + ft * 8 + g]));
    }
}

template <bool kFP16>
__device__ __forceinline__ void load_rec(const void *attrs, int64_t i, float (&v)[kRec]) {
    if constexpr (kFP16) {
        const uint4 *p = reinterpret_cast<const uint4 *>(attrs) + 3 * i;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            uint4 u = __ldg(p + k);
            const __half2 *h = reinterpret_cast<const __half2 *>(&u);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float2 f = __half22float2(h[j]);
                v[8 * k + 2 * j] = f.x;
                v[8 * k + 2 * j + 1] = f.y;
            }
        }
    } else {
        const float4 *p = reinterpret_cast<const float4 *>(attrs) + 6 * i;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            float4 f = __ldg(p + k);
            v[4 * k] = f.x;
            v[4 * k + 1] = f.y;
            v[4 * k + 2] = f.z;
            v[4 * k + 3] = f.w;
        }
    }
}

template <bool kFP16, bool kMLP, bool kResidual>
__global__ void __launch_bounds__(kMlpThreads) k_preprocess_bwd(RenderArgs args,
                                                               const float *__restrict__ gG,
                                                               float *__restrict__ d_attrs,
                                                               float *__restrict__ partials) {
    grid_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    BwdSmem &sm = *reinterpret_cast<BwdSmem *>(smem_raw);
    const DevCamera &cam = args.cam;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if constexpr (kMLP) {
        mlp_load_weights(sm.mlp, args.mlp);
        // h1 columns 64..71: a column of ones (bias gradient b2), then zeros
        for (int e = threadIdx.x; e < kRows * 8; e += blockDim.x)
            sm.h1[(e >> 3) * kHStride + kOnesCol + (e & 7)] =
                __float2bfloat16((e & 7) == 0 ? 1.0f : 0.0f);
    }
    WGradAcc wacc;
    float sb3[kMlpOut];
    if constexpr (kMLP) {
#pragma unroll
        for (int nt = 0; nt < 9; ++nt) wacc.w2[nt][0] = wacc.w2[nt][1] = wacc.w2[nt][2] = wacc.w2[nt][3] = 0.f;
#pragma unroll
        for (int ft = 0; ft < 3; ++ft) wacc.w1[ft][0] = wacc.w1[ft][1] = wacc.w1[ft][2] = wacc.w1[ft][3] = 0.f;
        wacc.w3[0] = wacc.w3[1] = wacc.w3[2] = wacc.w3[3] = 0.f;
#pragma unroll
        for (int k = 0; k < kMlpOut; ++k) sb3[k] = 0.f;
    }
    const float *W = cam.R;
    float cc[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) cc[j] = -(W[j] * cam.t[0] + W[3 + j] * cam.t[1] + W[6 + j] * cam.t[2]);
    const float C0 = 0.28209479177387814f, C1 = 0.4886025119029199f;
    const float limx = 1.3f * (0.5f * (float)cam.width / cam.fx);
    const float limy = 1.3f * (0.5f * (float)cam.height / cam.fy);

    for (int64_t base = (int64_t)blockIdx.x * kMlpThreads; base < args.n;
         base += (int64_t)gridDim.x * kMlpThreads) {
        // the previous iteration's weight-gradient products read every warp's rows
        if constexpr (kMLP) __syncthreads();
        const int64_t i = base + threadIdx.x;
        const bool valid = i < args.n;
        float v[kRec];
#pragma unroll
        for (int k = 0; k < kRec; ++k) v[k] = 0.f;
        bool vis = false;
        if (valid) {
            load_rec<kFP16>(args.attrs, i, v);
            const uint2 r = args.rect[i];
            vis = (r.x != 0u || r.y != 0u) && ((r.x >> 16) > (r.x & 0xFFFF));
        }
        float up[10];
#pragma unroll
        for (int e = 0; e < 10; ++e) up[e] = vis ? gG[(size_t)i * kGRec + e] : 0.f;
        // ---- forward recompute (FP32) ----
        const float qn = sqrtf(v[6] * v[6] + v[7] * v[7] + v[8] * v[8] + v[9] * v[9]);
        const float iqn = vis ? 1.0f / qn : 0.f;
        const float qw = v[6] * iqn, qx = v[7] * iqn, qy = v[8] * iqn, qz = v[9] * iqn;
        float d[3] = {v[0] - cc[0], v[1] - cc[1], v[2] - cc[2]};
        const float dn = sqrtf(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
        const float idn = dn > 0.f ? 1.0f / dn : 0.f;
        const float P[3] = {d[0] * idn, d[1] * idn, d[2] * idn};

        float phi = 1.0f, o = v[10], yv[5] = {1.f, 0.f, 0.f, 0.f, 0.f};
        if constexpr (kMLP) {
            __nv_bfloat16 *xr = &sm.mlp.x[warp][lane * kXStride];
            float f[kMlpK1];
#pragma unroll
            for (int k = 0; k < kMlpK1; ++k) f[k] = 0.f;
            if (valid) {
                f[0] = P[0]; f[1] = P[1]; f[2] = P[2];
                f[3] = v[3]; f[4] = v[4]; f[5] = v[5];
                f[6] = qw; f[7] = qx; f[8] = qy; f[9] = qz;
#pragma unroll
                for (int k = 0; k < 12; ++k) f[10 + k] = v[11 + k];
            }
            f[kXOnesCol] = 1.0f;  // W1's column 22 is zero: the forward is unchanged
#pragma unroll
            for (int k = 0; k < kMlpK1; k += 8) {
                uint4 u;
                u.x = pack_bf16(f[k], f[k + 1]);
                u.y = pack_bf16(f[k + 2], f[k + 3]);
                u.z = pack_bf16(f[k + 4], f[k + 5]);
                u.w = pack_bf16(f[k + 6], f[k + 7]);
                *reinterpret_cast<uint4 *>(xr + k) = u;
            }
            __syncwarp();
            mlp_warp<true>(sm.mlp, warp, lane, sm.h1 + warp * 32 * kHStride, sm.h2 + warp * 32 * kHStride);
            __syncwarp();
#pragma unroll
            for (int k = 0; k < 5; ++k) yv[k] = sm.mlp.out[warp][lane][k];
            phi = fmaxf(yv[0], 0.f);
            o = 1.0f / (1.0f + __expf(-yv[1]));
        }
        // colour
        float cbase[3];
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) {
            cbase[ch] = C0 * v[11 + ch] - C1 * P[1] * v[14 + ch] + C1 * P[2] * v[17 + ch] -
                       C1 * P[0] * v[20 + ch] + 0.5f;
            if constexpr (kResidual) cbase[ch] += yv[2 + ch];
        }
        // projection
        float R[9];
        R[0] = 1.f - 2.f * (qy * qy + qz * qz);
        R[1] = 2.f * (qx * qy - qw * qz);
        R[2] = 2.f * (qx * qz + qw * qy);
        R[3] = 2.f * (qx * qy + qw * qz);
        R[4] = 1.f - 2.f * (qx * qx + qz * qz);
        R[5] = 2.f * (qy * qz - qw * qx);
        R[6] = 2.f * (qx * qz - qw * qy);
        R[7] = 2.f * (qy * qz + qw * qx);
        R[8] = 1.f - 2.f * (qx * qx + qy * qy);
        float t[3];
#pragma unroll
        for (int r = 0; r < 3; ++r) t[r] = W[3 * r] * v[0] + W[3 * r + 1] * v[1] + W[3 * r + 2] * v[2] + cam.t[r];
        const float rz = vis ? 1.0f / t[2] : 0.f;
        const float u = t[0] * rz, vv = t[1] * rz;
        const bool cx_ = fabsf(u) > limx, cy_ = fabsf(vv) > limy;
        const float uc = fminf(fmaxf(u, -limx), limx), vc = fminf(fmaxf(vv, -limy), limy);
        const float J00 = cam.fx * rz, J02 = -cam.fx * uc * rz;
        const float J11 = cam.fy * rz, J12 = -cam.fy * vc * rz;
        float T0[3], T1[3], M[9], V0[3], V1[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            T0[j] = J00 * W[j] + J02 * W[6 + j];
            T1[j] = J11 * W[3 + j] + J12 * W[6 + j];
        }
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int j = 0; j < 3; ++j) M[3 * k + j] = R[3 * k + j] * v[3 + j];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            V0[j] = T0[0] * M[j] + T0[1] * M[3 + j] + T0[2] * M[6 + j];
            V1[j] = T1[0] * M[j] + T1[1] * M[3 + j] + T1[2] * M[6 + j];
        }
        int am = 0;
        float smax = v[3];
        if (v[4] > smax) { smax = v[4]; am = 1; }
        if (v[5] > smax) { smax = v[5]; am = 2; }
        const float es = vis ? expf(smax * rz) : 0.f;

        // ---- backward ----
        const float gcol[3] = {up[0], up[1], up[2]}, gw = up[3], go = up[4];
        float dt[3] = {0.f, 0.f, 0.f}, ds[3] = {0.f, 0.f, 0.f}, dq[4] = {0.f, 0.f, 0.f, 0.f};
        float dP[3] = {0.f, 0.f, 0.f}, dY[12];
        // whitened second moments -> Sigma_2D:  dSigma = L M L^T / 2, with the
        // forward's factors L = [[l11, 0], [l21, l22]]
        float l11 = 0.f, l21 = 0.f, l22 = 0.f;
        if (vis) {
            const float4 ra = __ldg(&args.rec[i].a);
            l11 = ra.z;
            l21 = ra.w;
            l22 = __ldg(&args.rec[i].b.x);
        }
        const float LM00 = l11 * up[7], LM01 = l11 * up[8];   // first row of L M
        const float LM10 = l21 * up[7] + l22 * up[8], LM11 = l21 * up[8] + l22 * up[9];
        const float ga = 0.5f * LM00 * l11, gb = LM00 * l21 + LM01 * l22;   // gb: twice dSigma_01
        const float gc = 0.5f * (LM10 * l21 + LM11 * l22);
        float dV0[3], dV1[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            dV0[j] = 2.0f * ga * V0[j] + gb * V1[j];
            dV1[j] = gb * V0[j] + 2.0f * gc * V1[j];
        }
        float dT0[3], dT1[3], dR[9];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            dT0[k] = dV0[0] * M[3 * k] + dV0[1] * M[3 * k + 1] + dV0[2] * M[3 * k + 2];
            dT1[k] = dV1[0] * M[3 * k] + dV1[1] * M[3 * k + 1] + dV1[2] * M[3 * k + 2];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const float dM = T0[k] * dV0[j] + T1[k] * dV1[j];
                dR[3 * k + j] = dM * v[3 + j];
                ds[j] += dM * R[3 * k + j];
            }
        }
        const float dJ00 = dT0[0] * W[0] + dT0[1] * W[1] + dT0[2] * W[2];
        const float dJ02 = dT0[0] * W[6] + dT0[1] * W[7] + dT0[2] * W[8];
        const float dJ11 = dT1[0] * W[3] + dT1[1] * W[4] + dT1[2] * W[5];
        const float dJ12 = dT1[0] * W[6] + dT1[1] * W[7] + dT1[2] * W[8];
        const float rz2 = rz * rz;
        dt[2] += -dJ00 * cam.fx * rz2 - dJ11 * cam.fy * rz2;
        if (!cx_) {
            dt[0] += -dJ02 * cam.fx * rz2;
            dt[2] += dJ02 * 2.0f * cam.fx * t[0] * rz2 * rz;
        } else {
            dt[2] += dJ02 * cam.fx * uc * rz2;
        }
        if (!cy_) {
            dt[1] += -dJ12 * cam.fy * rz2;
            dt[2] += dJ12 * 2.0f * cam.fy * t[1] * rz2 * rz;
        } else {
            dt[2] += dJ12 * cam.fy * vc * rz2;
        }
        // pixel mean
        dt[0] += up[5] * cam.fx * rz;
        dt[1] += up[6] * cam.fy * rz;
        dt[2] += -(up[5] * cam.fx * t[0] + up[6] * cam.fy * t[1]) * rz2;
        // Eq. 3
        const float dphi = gw * (2.0f * phi + rz2);
        dt[2] += gw * (-2.0f * phi * rz2 * rz - es * smax * rz2);
        ds[am] += gw * es * rz;
        // colour
        float dbase[3];
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) {
            dbase[ch] = cbase[ch] > 0.0f ? gcol[ch] : 0.0f;
            dY[ch] = C0 * dbase[ch];
            dY[3 + ch] = -C1 * P[1] * dbase[ch];
            dY[6 + ch] = C1 * P[2] * dbase[ch];
            dY[9 + ch] = -C1 * P[0] * dbase[ch];
            dP[0] += -C1 * v[20 + ch] * dbase[ch];
            dP[1] += -C1 * v[14 + ch] * dbase[ch];
            dP[2] += C1 * v[17 + ch] * dbase[ch];
        }
        float d_o_stored = 0.0f;
        float dqh[4] = {0.f, 0.f, 0.f, 0.f};
        if constexpr (kMLP) {
            // Eq. 4 head: phi = ReLU(y0), o = sigmoid(y1), residual y2..4
            float d3[5];
            d3[0] = yv[0] > 0.0f ? dphi : 0.0f;
            d3[1] = go * o * (1.0f - o);
            d3[2] = kResidual ? dbase[0] : 0.0f;
            d3[3] = kResidual ? dbase[1] : 0.0f;
            d3[4] = kResidual ? dbase[2] : 0.0f;
            if (!vis) d3[0] = d3[1] = d3[2] = d3[3] = d3[4] = 0.0f;
            const int row = warp * 32 + lane;
#pragma unroll
            for (int k = 0; k < 8; ++k) sm.d3[row * kD3S + k] = k < kMlpOut ? d3[k] : 0.0f;
#pragma unroll
            for (int k = 0; k < kMlpOut; ++k) sb3[k] += d3[k];
            __syncwarp();
            mlp_d2_warp(sm, warp, lane);
            __syncthreads();
            mlp_wgrad2_cta(sm, warp, lane, wacc);
            __syncthreads();
            mlp_d1_warp(sm, warp, lane);
            __syncthreads();
            mlp_wgrad1_cta(sm, warp, lane, wacc);
            float dx[kDxS];
#pragma unroll
            for (int k = 0; k < kDxS; k += 4) {
                const float4 q4 = *reinterpret_cast<const float4 *>(&sm.dx[row * kDxS + k]);
                dx[k] = q4.x;
                dx[k + 1] = q4.y;
                dx[k + 2] = q4.z;
                dx[k + 3] = q4.w;
            }
            dP[0] += dx[0];
            dP[1] += dx[1];
            dP[2] += dx[2];
            ds[0] += dx[3];
            ds[1] += dx[4];
            ds[2] += dx[5];
            dqh[0] += dx[6];
            dqh[1] += dx[7];
            dqh[2] += dx[8];
            dqh[3] += dx[9];
#pragma unroll
            for (int k = 0; k < 12; ++k) dY[k] += dx[10 + k];
        } else {
            d_o_stored = go;
            (void)dphi;
        }
        if (!valid) continue;
        float *out = d_attrs + (size_t)(args.perm ? args.perm[i] : (uint32_t)i) * kRec;
        if (!vis) {
#pragma unroll
            for (int k = 0; k < kRec; ++k) out[k] = 0.f;
            continue;
        }
        // R(q_hat) -> q_hat
        const float w_ = qw, x_ = qx, y_ = qy, z_ = qz;
        dqh[0] += 2.f * (-z_ * dR[1] + y_ * dR[2] + z_ * dR[3] - x_ * dR[5] - y_ * dR[6] + x_ * dR[7]);
        dqh[1] += 2.f * (y_ * dR[1] + z_ * dR[2] + y_ * dR[3] - 2.f * x_ * dR[4] - w_ * dR[5] +
                         z_ * dR[6] + w_ * dR[7] - 2.f * x_ * dR[8]);
        dqh[2] += 2.f * (-2.f * y_ * dR[0] + x_ * dR[1] + w_ * dR[2] + x_ * dR[3] + z_ * dR[5] -
                         w_ * dR[6] + z_ * dR[7] - 2.f * y_ * dR[8]);
        dqh[3] += 2.f * (-2.f * z_ * dR[0] - w_ * dR[1] + x_ * dR[2] + w_ * dR[3] - 2.f * z_ * dR[4] +
                         y_ * dR[5] + x_ * dR[6] + y_ * dR[7]);
        const float qd = qw * dqh[0] + qx * dqh[1] + qy * dqh[2] + qz * dqh[3];
        dq[0] = (dqh[0] - qw * qd) * iqn;
        dq[1] = (dqh[1] - qx * qd) * iqn;
        dq[2] = (dqh[2] - qy * qd) * iqn;
        dq[3] = (dqh[3] - qz * qd) * iqn;
        // t = W mu + t_cam, P = (mu - c) / |mu - c|
        const float pd = P[0] * dP[0] + P[1] * dP[1] + P[2] * dP[2];
        float dmu[3];
#pragma unroll
        for (int j = 0; j < 3; ++j)
            dmu[j] = W[j] * dt[0] + W[3 + j] * dt[1] + W[6 + j] * dt[2] + (dP[j] - P[j] * pd) * idn;
        out[0] = dmu[0];
        out[1] = dmu[1];
        out[2] = dmu[2];
        out[3] = ds[0];
        out[4] = ds[1];
        out[5] = ds[2];
        out[6] = dq[0];
        out[7] = dq[1];
        out[8] = dq[2];
        out[9] = dq[3];
        out[10] = d_o_stored;
#pragma unroll
        for (int k = 0; k < 12; ++k) out[11 + k] = dY[k];
        out[23] = 0.f;
    }
    if constexpr (kMLP) {
        // every element of this CTA's partial row is owned by one (lane, register)
        float *P = partials + (size_t)blockIdx.x * kMlpGrad;
        const int g = lane >> 2, t = lane & 3;
        const int m0 = warp * 16 + g, m1 = m0 + 8;
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
            const int c = nt * 8 + 2 * t;
            P[kOffW2 + m0 * kMlpHidden + c] = wacc.w2[nt][0];
            P[kOffW2 + m0 * kMlpHidden + c + 1] = wacc.w2[nt][1];
            P[kOffW2 + m1 * kMlpHidden + c] = wacc.w2[nt][2];
            P[kOffW2 + m1 * kMlpHidden + c + 1] = wacc.w2[nt][3];
        }
        if (t == 0) {
            P[kOffB2 + m0] = wacc.w2[8][0];
            P[kOffB2 + m1] = wacc.w2[8][2];
        }
#pragma unroll
        for (int ft = 0; ft < 3; ++ft) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int f = ft * 8 + 2 * t + h;
                if (f < kMlpIn) {
                    P[kOffW1 + m0 * kMlpIn + f] = wacc.w1[ft][h];
                    P[kOffW1 + m1 * kMlpIn + f] = wacc.w1[ft][2 + h];
                } else if (f == kXOnesCol) {
                    P[kOffB1 + m0] = wacc.w1[ft][h];
                    P[kOffB1 + m1] = wacc.w1[ft][2 + h];
                }
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = 2 * t + h;
            if (k < kMlpOut) {
                P[kOffW3 + k * kMlpHidden + m0] = wacc.w3[h];
                P[kOffW3 + k * kMlpHidden + m1] = wacc.w3[2 + h];
            }
        }
#pragma unroll
        for (int k = 0; k < kMlpOut; ++k) {
            float x = sb3[k];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            if (lane == 0) sm.b3[warp][k] = x;
        }
        __syncthreads();
        if (threadIdx.x < kMlpOut) {
            float x = 0.f;
            for (int w = 0; w < kMlpThreads / 32; ++w) x += sm.b3[w][threadIdx.x];
            P[kOffB3 + threadIdx.x] = x;
        }
    }
}

// Sums the CTAs' partial weight gradients, in a fixed order: a block takes 32
// elements, each of its eight warps every eighth CTA's row.  (One thread per
// element over all rows was a serial chain of 304 loads: 8.5 us against 3.)
constexpr int kReduceWarps = 8;
__global__ void __launch_bounds__(32 * kReduceWarps) k_mlp_grad_reduce(const float *__restrict__ partials,
                                                                       int nparts,
                                                                       float *__restrict__ out) {
    grid_wait();
    __shared__ float part[kReduceWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int e = blockIdx.x * 32 + lane;
    float s = 0.f;
    if (e < kMlpGrad) {
#pragma unroll 4
        for (int c = warp; c < nparts; c += kReduceWarps) s += partials[(size_t)c * kMlpGrad + e];
    }
    part[warp][lane] = s;
    __syncthreads();
    if (warp == 0 && e < kMlpGrad) {
#pragma unroll
        for (int w = 1; w < kReduceWarps; ++w) s += part[w][lane];
        out[e] = s;
    }
}

template <bool kFP16, bool kMLP, bool kRes>
cudaError_t launch_pre_bwd(const RenderArgs &a, int blocks, const float *gG, float *d_attrs,
                           float *partials, cudaStream_t stream) {
    const size_t smem = kMLP ? sizeof(BwdSmem) : 16;
    auto kern = k_preprocess_bwd<kFP16, kMLP, kRes>;
    if (kMLP) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
    }
    return launch_dependent(kern, (unsigned)blocks, kMlpThreads, smem, stream, a, gG, d_attrs, partials);
}

}  // namespace

int mlp_grad_size() { return kMlpGrad; }
int grad_record_size() { return kGRec; }
int pre_bwd_blocks(int64_t n, int sm_count) {
    int64_t b = (n + kMlpThreads - 1) / kMlpThreads;
    const int64_t cap = 2 * (int64_t)sm_count;
    if (b > cap) b = cap;
    return b < 1 ? 1 : (int)b;
}

cudaError_t launch_backward(const RenderArgs &a, int sm_count, const float *dL_drgb,
                            const float *aux, float *gG, float *d_attrs, float *d_mlp,
                            float *partials, cudaStream_t stream) {
    const int T = a.cam.tiles_x * a.cam.tiles_y;
    cudaError_t e = cudaMemsetAsync(gG, 0, (size_t)a.n * kGRec * sizeof(float), stream);
    if (e != cudaSuccess) return e;
    const int splits = bwd_splits(T, sm_count);
    k_raster_bwd<<<T * splits, kBwdThreads, 0, stream>>>(a, dL_drgb, aux, gG, splits);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int blocks = pre_bwd_blocks(a.n, sm_count);
    const bool fp16 = a.precision == MGS_PREC_FP16;
    if (a.use_mlp) {
        if (a.rgb_residual)
            e = fp16 ? launch_pre_bwd<true, true, true>(a, blocks, gG, d_attrs, partials, stream)
                     : launch_pre_bwd<false, true, true>(a, blocks, gG, d_attrs, partials, stream);
        else
            e = fp16 ? launch_pre_bwd<true, true, false>(a, blocks, gG, d_attrs, partials, stream)
                     : launch_pre_bwd<false, true, false>(a, blocks, gG, d_attrs, partials, stream);
        if (e != cudaSuccess) return e;
        if (d_mlp) {
            e = launch_dependent(k_mlp_grad_reduce, (kMlpGrad + 31) / 32, 32 * kReduceWarps, 0, stream,
                                 partials, blocks, d_mlp);
        }
        return e;
    }
    e = fp16 ? launch_pre_bwd<true, false, false>(a, blocks, gG, d_attrs, partials, stream)
             : launch_pre_bwd<false, false, false>(a, blocks, gG, d_attrs, partials, stream);
    if (e == cudaSuccess && d_mlp)
        e = cudaMemsetAsync(d_mlp, 0, (size_t)kMlpGrad * sizeof(float), stream);
    return e;
}

}  // namespace mgs
