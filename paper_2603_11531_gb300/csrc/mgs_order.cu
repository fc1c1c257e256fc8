// Spatial order of a resident scene.  At load time the Gaussians are sorted
// along a 3D Morton curve of their means (10 bits per axis over the scene's
// bounding box), so that Gaussians stored close together are close in space:
// a binning CTA's contiguous range of Gaussians then covers a compact set of
// tiles, and its list writes stay local.  The image does not depend on the
// storage order (Eq. 2 is a sum); every per-Gaussian output is mapped back to
// the caller's order through perm (stored position -> caller index) and its
// inverse.
//
// The sort is a stable LSD radix sort of the 32-bit keys with their indices,
// four passes of 8 bits: a histogram per block of 4,096 keys, a scan of every
// digit's column over the blocks, and a scatter in which a block first orders
// its keys in shared memory and then writes every digit's run coalesced.
// A pass over 3M Gaussians takes 11 + 5 + 40 us (its 60 MB would take 9 us at the
// measured 6.8 TB/s: the scatter is bound by its ranking and short runs).  Eight
// passes of 4 bits over 64-bit keys, ranked serially per thread and scanned by
// one block, took 107 us each: loading 3M Gaussians from device memory 2.12 ms
// against 0.83 ms, which also saves seven of eleven allocations and a copy.
#include "mgs_internal.cuh"

namespace mgs {
namespace {

constexpr int kOrdThreads = 256;

// float <-> order-preserving unsigned encoding (for atomic min / max)
__device__ __forceinline__ uint32_t f2ord(float f) {
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ord2f(uint32_t u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u);
}

template <bool kFP16>
__device__ __forceinline__ void mean_of(const void *attrs, int64_t i, float (&m)[3]) {
#pragma unroll
    for (int k = 0; k < 3; ++k)
        m[k] = kFP16 ? __half2float(static_cast<const __half *>(attrs)[kRec * i + k])
                     : static_cast<const float *>(attrs)[kRec * i + k];
}

// bounds[0..2] = min, bounds[3..5] = max of the finite means (encoded)
template <bool kFP16>
__global__ void __launch_bounds__(kOrdThreads) k_bounds(const void *attrs, int64_t n,
                                                        uint32_t *bounds) {
    __shared__ uint32_t blk[6];
    if (threadIdx.x < 6) blk[threadIdx.x] = threadIdx.x < 3 ? 0xFFFFFFFFu : 0u;
    __syncthreads();
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        float m[3];
        mean_of<kFP16>(attrs, i, m);
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (isfinite(m[k])) {
                lo[k] = fminf(lo[k], m[k]);
                hi[k] = fmaxf(hi[k], m[k]);
            }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], o));
            hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], o));
        }
        if ((threadIdx.x & 31) == 0) {
            atomicMin(&blk[k], f2ord(lo[k]));
            atomicMax(&blk[3 + k], f2ord(hi[k]));
        }
    }
    __syncthreads();   // one global atomic per block and bound
    if (threadIdx.x < 3) atomicMin(&bounds[threadIdx.x], blk[threadIdx.x]);
    else if (threadIdx.x < 6) atomicMax(&bounds[threadIdx.x], blk[threadIdx.x]);
}

__device__ __forceinline__ uint32_t spread10(uint32_t v) {   // 10 bits -> every third bit
    v &= 0x3FFu;
    v = (v | (v << 16)) & 0x030000FFu;
    v = (v | (v << 8)) & 0x0300F00Fu;
    v = (v | (v << 4)) & 0x030C30C3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}

template <bool kFP16>
__global__ void __launch_bounds__(kOrdThreads) k_morton(const void *attrs, int64_t n,
                                                        const uint32_t *bounds, uint32_t *keys) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float m[3];
    mean_of<kFP16>(attrs, i, m);
    uint32_t key = 0x3FFFFFFFu;   // non-finite means last
    if (isfinite(m[0]) && isfinite(m[1]) && isfinite(m[2])) {
        key = 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float lo = ord2f(bounds[k]), hi = ord2f(bounds[3 + k]);
            const float ext = hi - lo;
            const float u = ext > 0.0f ? (m[k] - lo) / ext : 0.0f;
            const uint32_t q = (uint32_t)fminf(fmaxf(u * 1024.0f, 0.0f), 1023.0f);
            key |= spread10(q) << k;
        }
    }
    keys[i] = key;
}

// ---- radix sort ------------------------------------------------------------
constexpr int kSortThreads = 256;               // one thread per digit value
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortItems = 16;
constexpr int kSortTile = kSortThreads * kSortItems;
constexpr int kDigits = 256;

// hist[d][b]: keys of block b whose digit is d.
__global__ void __launch_bounds__(kSortThreads) k_sort_hist(const uint32_t *__restrict__ keys, int64_t n,
                                                            int shift, int nblocks,
                                                            uint32_t *__restrict__ hist) {
    __shared__ uint32_t h[kDigits];
    h[threadIdx.x] = 0u;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kSortTile;
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) {
        const int64_t idx = base + i * kSortThreads + threadIdx.x;
        if (idx < n) atomicAdd(&h[(keys[idx] >> shift) & (kDigits - 1)], 1u);
    }
    __syncthreads();
    hist[(int64_t)threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

// Inclusive scan over the block's kSortThreads values.
__device__ __forceinline__ uint32_t block_scan(uint32_t x, uint32_t *warp_sums) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[warp] = x;
    __syncthreads();
    uint32_t before = 0;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) before += w < warp ? warp_sums[w] : 0u;
    __syncthreads();
    return x + before;
}

// Block d: exclusive scan of column hist[d][0 .. nblocks) in place, its total in
// total[d].
__global__ void __launch_bounds__(kSortThreads) k_sort_scan(uint32_t *__restrict__ hist, int nblocks,
                                                            uint32_t *__restrict__ total) {
    __shared__ uint32_t warp_sums[kSortWarps];
    __shared__ uint32_t last;
    uint32_t *col = hist + (int64_t)blockIdx.x * nblocks;
    uint32_t carry = 0;
    for (int base = 0; base < nblocks; base += kSortThreads) {
        const int i = base + threadIdx.x;
        const uint32_t v = i < nblocks ? col[i] : 0u;
        const uint32_t incl = block_scan(v, warp_sums);
        if (i < nblocks) col[i] = carry + incl - v;
        if (threadIdx.x == kSortThreads - 1) last = incl;
        __syncthreads();
        carry += last;
        __syncthreads();
    }
    if (threadIdx.x == 0) total[blockIdx.x] = carry;
}

// Stable scatter by one digit; vin null: the values are the indices.
__global__ void __launch_bounds__(kSortThreads) k_sort_scatter(
    const uint32_t *__restrict__ kin, const uint32_t *__restrict__ vin, int64_t n, int shift, int nblocks,
    const uint32_t *__restrict__ hist, const uint32_t *__restrict__ total, uint32_t *__restrict__ kout,
    uint32_t *__restrict__ vout) {
    __shared__ uint32_t cnt[kSortWarps][kDigits];   // per warp: keys so far, then its start in the digit
    __shared__ uint32_t sk[kSortTile], sv[kSortTile];
    __shared__ uint32_t first[kDigits];             // global position of the block's run minus its local one
    __shared__ uint32_t warp_sums[kSortWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t tot = total[tid], before = hist[(int64_t)tid * nblocks + blockIdx.x];
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) cnt[w][tid] = 0u;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kSortTile;
    const int m = (int)(n - base < kSortTile ? n - base : kSortTile);
    uint32_t key[kSortItems], rank[kSortItems];
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) {
        const int p = warp * 32 * kSortItems + i * 32 + lane;
        key[i] = p < m ? kin[base + p] : 0u;
        const uint32_t d = p < m ? (key[i] >> shift) & (kDigits - 1) : (uint32_t)kDigits;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        if (d < kDigits) rank[i] = cnt[warp][d] + __popc(peers & ((1u << lane) - 1u));
        __syncwarp();
        if (d < kDigits && lane == __ffs(peers) - 1) cnt[warp][d] += __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    uint32_t c = 0;   // thread = digit: starts of the warps, the block's count
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) {
        const uint32_t x = cnt[w][tid];
        cnt[w][tid] = c;
        c += x;
    }
    const uint32_t start = block_scan(c, warp_sums) - c;             // local position of the digit
    const uint32_t gbase = block_scan(tot, warp_sums) - tot;         // global position of the digit
    first[tid] = gbase + before - start;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) cnt[w][tid] += start;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) {
        const int p = warp * 32 * kSortItems + i * 32 + lane;
        if (p >= m) continue;
        const uint32_t at = cnt[warp][(key[i] >> shift) & (kDigits - 1)] + rank[i];
        sk[at] = key[i];
        sv[at] = vin ? vin[base + p] : (uint32_t)(base + p);
    }
    __syncthreads();
    for (int p = tid; p < m; p += kSortThreads) {
        const uint32_t k = sk[p];
        const uint32_t at = first[(k >> shift) & (kDigits - 1)] + (uint32_t)p;
        kout[at] = k;
        vout[at] = sv[p];
    }
}

// Records in sorted order, one thread per 16-byte piece (kRow16 per record).
template <int kRow16>
__global__ void __launch_bounds__(kOrdThreads) k_gather(const uint4 *__restrict__ in,
                                                        const uint32_t *__restrict__ order,
                                                        int64_t n, uint4 *__restrict__ out,
                                                        uint32_t *__restrict__ perm,
                                                        uint32_t *__restrict__ iperm) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n * kRow16) return;
    const int64_t j = e / kRow16;
    const int k = (int)(e - j * kRow16);
    const uint32_t src = order[j];
    out[e] = in[(int64_t)src * kRow16 + k];
    if (k == 0) {
        perm[j] = src;
        iperm[src] = (uint32_t)j;
    }
}

__global__ void k_map_ids(const uint32_t *__restrict__ in, const uint32_t *__restrict__ perm,
                          int64_t k, uint32_t *__restrict__ out) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j < k) out[j] = perm[in[j]];
}

}  // namespace

cudaError_t spatial_order(const void *attrs_in, int64_t n, int precision, void *attrs_out,
                          uint32_t *perm, uint32_t *iperm, cudaStream_t stream) {
    if (n <= 0) return cudaSuccess;
    const bool fp16 = precision == MGS_PREC_FP16;
    const int nblocks = (int)((n + kSortTile - 1) / kSortTile);
    // one allocation: bounds, digit totals, histograms, keys and values twice
    const size_t hist_words = (size_t)kDigits * nblocks, N = (size_t)n;
    uint32_t *mem = nullptr;
    cudaError_t e = cudaMalloc(&mem, (8 + kDigits + hist_words + 4 * N) * sizeof(uint32_t));
    if (e != cudaSuccess) return e;
    uint32_t *bounds = mem, *total = mem + 8, *hist = total + kDigits, *k = hist + hist_words, *kt = k + N,
             *v = kt + N, *vt = v + N;
    const uint32_t init[6] = {0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0u, 0u, 0u};
    e = cudaMemcpyAsync(bounds, init, sizeof init, cudaMemcpyHostToDevice, stream);
    const unsigned grid = (unsigned)((n + kOrdThreads - 1) / kOrdThreads);
    if (e == cudaSuccess) {
        const unsigned gb = grid < 1024 ? grid : 1024;
        if (fp16)
            k_bounds<true><<<gb, kOrdThreads, 0, stream>>>(attrs_in, n, bounds);
        else
            k_bounds<false><<<gb, kOrdThreads, 0, stream>>>(attrs_in, n, bounds);
        if (fp16)
            k_morton<true><<<grid, kOrdThreads, 0, stream>>>(attrs_in, n, bounds, k);
        else
            k_morton<false><<<grid, kOrdThreads, 0, stream>>>(attrs_in, n, bounds, k);
        for (int shift = 0; shift < 32; shift += 8) {
            k_sort_hist<<<nblocks, kSortThreads, 0, stream>>>(k, n, shift, nblocks, hist);
            k_sort_scan<<<kDigits, kSortThreads, 0, stream>>>(hist, nblocks, total);
            k_sort_scatter<<<nblocks, kSortThreads, 0, stream>>>(k, shift ? v : nullptr, n, shift, nblocks,
                                                                 hist, total, kt, vt);
            std::swap(k, kt);
            std::swap(v, vt);
        }
        const int row16 = kRec * (fp16 ? 2 : 4) / 16;
        const unsigned gg = (unsigned)((n * row16 + kOrdThreads - 1) / kOrdThreads);
        const uint4 *in = static_cast<const uint4 *>(attrs_in);
        uint4 *out = static_cast<uint4 *>(attrs_out);
        if (fp16)
            k_gather<3><<<gg, kOrdThreads, 0, stream>>>(in, v, n, out, perm, iperm);
        else
            k_gather<6><<<gg, kOrdThreads, 0, stream>>>(in, v, n, out, perm, iperm);
        e = cudaGetLastError();
    }
    const cudaError_t es = cudaStreamSynchronize(stream);
    if (e == cudaSuccess) e = es;
    cudaFree(mem);
    return e;
}

cudaError_t map_ids(const uint32_t *in, const uint32_t *perm, int64_t count, uint32_t *out,
                    cudaStream_t stream) {
    if (count <= 0) return cudaSuccess;
    k_map_ids<<<(unsigned)((count + 255) / 256), 256, 0, stream>>>(in, perm, count, out);
    return cudaGetLastError();
}

}  // namespace mgs
