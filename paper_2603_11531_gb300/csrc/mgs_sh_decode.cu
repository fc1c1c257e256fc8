// Load-time SH decode (Sec. 3.2, Eq. 6): every Gaussian stores a diffuse
// feature h_d and a view-dependent feature h_v (3 values each); two small
// MLPs with one hidden layer of 64 ReLU units and 16-bit parameters (App. C)
// turn them into the degree-0 and degree-1 SH coefficients once, before
// rendering:  f_d = MLP_d(h_d, h_v) -> Y0 rgb,  f_v = MLP_v(h_d, h_v) ->
// Y1 rgb, Y2 rgb, Y3 rgb.  Four Gaussians per thread, FP32 accumulation, the
// parameters (passed by value) staged in shared memory as FP32.
#include <cuda_fp16.h>

#include <cstring>

#include "mgs_internal.cuh"

namespace mgs {
namespace {

constexpr int kDecThreads = 256;

struct DecodeParams {
    __half w1d[64 * 6], b1d[64], w2d[3 * 64], b2d[3];
    __half w1v[64 * 6], b1v[64], w2v[9 * 64], b2v[9];
};

// Weights of one hidden unit pair (unit j of MLP_d and of MLP_v), 16-byte words:
// {w1d[6], b1d, -} {w1v[6], b1v, -} {w2d[3], -} {w2v[9], -, -, -}
struct DecodeSmem {
    float4 u[64][8];
    float b2[12];
};

// x[0..5] of Gaussian i / y[0..11] into columns 11..22.  kVec: h and attrs are
// aligned for the wide accesses (FP16: 4 bytes; FP32: h 8, attrs 16 bytes).
template <bool kFP16, bool kVec>
__device__ __forceinline__ void load_h(const void *h, int64_t i, float (&x)[6]) {
    if constexpr (kFP16 && kVec) {
        const __half2 *p = reinterpret_cast<const __half2 *>(static_cast<const __half *>(h) + 6 * i);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float2 f = __half22float2(__ldg(p + k));
            x[2 * k] = f.x;
            x[2 * k + 1] = f.y;
        }
    } else if constexpr (kVec) {
        const float2 *p = reinterpret_cast<const float2 *>(static_cast<const float *>(h) + 6 * i);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float2 f = __ldg(p + k);
            x[2 * k] = f.x;
            x[2 * k + 1] = f.y;
        }
    } else {
#pragma unroll
        for (int k = 0; k < 6; ++k)
            x[k] = kFP16 ? __half2float(static_cast<const __half *>(h)[6 * i + k])
                         : static_cast<const float *>(h)[6 * i + k];
    }
}
template <bool kFP16, bool kVec>
__device__ __forceinline__ void store_y(void *attrs, int64_t i, const float (&y)[12]) {
    if constexpr (kFP16) {
        __half *o = static_cast<__half *>(attrs) + kRec * i + 11;
        if constexpr (kVec) {
            o[0] = __float2half_rn(y[0]);
#pragma unroll
            for (int k = 1; k < 11; k += 2)
                *reinterpret_cast<__half2 *>(o + k) = __floats2half2_rn(y[k], y[k + 1]);
            o[11] = __float2half_rn(y[11]);
        } else {
#pragma unroll
            for (int k = 0; k < 12; ++k) o[k] = __float2half_rn(y[k]);
        }
    } else {
        float *o = static_cast<float *>(attrs) + kRec * i + 11;
        if constexpr (kVec) {
            o[0] = y[0];
            *reinterpret_cast<float4 *>(o + 1) = make_float4(y[1], y[2], y[3], y[4]);
            *reinterpret_cast<float4 *>(o + 5) = make_float4(y[5], y[6], y[7], y[8]);
            *reinterpret_cast<float2 *>(o + 9) = make_float2(y[9], y[10]);
            o[11] = y[11];
        } else {
#pragma unroll
            for (int k = 0; k < 12; ++k) o[k] = y[k];
        }
    }
}

// kPer Gaussians per thread share every weight load.  Bound: the FMA pipe, 1,536
// FMA per Gaussian (3M: 0.12 ms).  One Gaussian per thread loaded a weight for
// every FMA: 0.42 ms for 3M FP16 Gaussians against 0.23 ms.
constexpr int kPer = 4;
template <bool kFP16, bool kVec>
__global__ void __launch_bounds__(kDecThreads)
    k_decode_sh(int64_t n, const void *__restrict__ h, void *__restrict__ attrs, DecodeParams p) {
    __shared__ DecodeSmem sm;
    for (int e = threadIdx.x; e < 64 * 32; e += blockDim.x) {
        const int j = e / 32, c = e % 32;
        float v = 0.0f;
        if (c < 6) v = __half2float(p.w1d[j * 6 + c]);
        else if (c == 6) v = __half2float(p.b1d[j]);
        else if (c >= 8 && c < 14) v = __half2float(p.w1v[j * 6 + c - 8]);
        else if (c == 14) v = __half2float(p.b1v[j]);
        else if (c >= 16 && c < 19) v = __half2float(p.w2d[(c - 16) * 64 + j]);
        else if (c >= 20 && c < 29) v = __half2float(p.w2v[(c - 20) * 64 + j]);
        reinterpret_cast<float *>(sm.u[j])[c] = v;
    }
    if (threadIdx.x < 12)
        sm.b2[threadIdx.x] = __half2float(threadIdx.x < 3 ? p.b2d[threadIdx.x] : p.b2v[threadIdx.x - 3]);
    __syncthreads();

    const int64_t step = (int64_t)gridDim.x * kDecThreads * kPer;
    for (int64_t i0 = (int64_t)blockIdx.x * kDecThreads * kPer + threadIdx.x; i0 < n; i0 += step) {
        float x[kPer][6], y[kPer][12];
#pragma unroll
        for (int g = 0; g < kPer; ++g) {
            const int64_t i = i0 + g * kDecThreads;
            load_h<kFP16, kVec>(h, i < n ? i : i0, x[g]);
#pragma unroll
            for (int k = 0; k < 12; ++k) y[g][k] = sm.b2[k];
        }
#pragma unroll 1
        for (int j = 0; j < 64; ++j) {
            float w[32];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float4 f = sm.u[j][q];
                w[4 * q] = f.x;
                w[4 * q + 1] = f.y;
                w[4 * q + 2] = f.z;
                w[4 * q + 3] = f.w;
            }
#pragma unroll
            for (int g = 0; g < kPer; ++g) {
                float hd = w[6], hv = w[14];
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    hd = fmaf(w[k], x[g][k], hd);
                    hv = fmaf(w[8 + k], x[g][k], hv);
                }
                hd = fmaxf(hd, 0.0f);
                hv = fmaxf(hv, 0.0f);
#pragma unroll
                for (int k = 0; k < 3; ++k) y[g][k] = fmaf(w[16 + k], hd, y[g][k]);
#pragma unroll
                for (int k = 0; k < 9; ++k) y[g][3 + k] = fmaf(w[20 + k], hv, y[g][3 + k]);
            }
        }
#pragma unroll
        for (int g = 0; g < kPer; ++g) {
            const int64_t i = i0 + g * kDecThreads;
            if (i < n) store_y<kFP16, kVec>(attrs, i, y[g]);
        }
    }
}

bool fill(const uint16_t *src, __half *dst, int count) {
    if (!src) return false;
    memcpy(dst, src, (size_t)count * 2);
    return true;
}

mgs_status bad(mgs_status s, const char *msg) {
    set_last_error(msg);
    return s;
}

}  // namespace
}  // namespace mgs

using namespace mgs;

extern "C" mgs_status mgs_decode_sh(mgs_ctx ctx, int64_t n, int32_t precision, const void *h,
                                    const mgs_sh_mlp *mlp_d, const mgs_sh_mlp *mlp_v,
                                    void *attrs, mgs_stream stream_) {
    if (!ctx || !mlp_d || !mlp_v) return bad(MGS_ERR_INVALID_ARG, "NULL argument");
    if (n < 0) return bad(MGS_ERR_INVALID_ARG, "n < 0");
    if (precision != MGS_PREC_FP32 && precision != MGS_PREC_FP16)
        return bad(MGS_ERR_INVALID_ARG, "unknown precision");
    if (n > 0 && (!h || !attrs)) return bad(MGS_ERR_INVALID_ARG, "h or attrs is NULL");
    DecodeParams p;
    if (!fill(mlp_d->w1, p.w1d, 64 * 6) || !fill(mlp_d->b1, p.b1d, 64) ||
        !fill(mlp_d->w2, p.w2d, 3 * 64) || !fill(mlp_d->b2, p.b2d, 3) ||
        !fill(mlp_v->w1, p.w1v, 64 * 6) || !fill(mlp_v->b1, p.b1v, 64) ||
        !fill(mlp_v->w2, p.w2v, 9 * 64) || !fill(mlp_v->b2, p.b2v, 9))
        return bad(MGS_ERR_INVALID_ARG, "an SH decoder parameter array is NULL");
    if (n == 0) return MGS_OK;
    int prev = 0;
    if (cudaGetDevice(&prev) != cudaSuccess || cudaSetDevice(ctx_device(ctx)) != cudaSuccess)
        return bad(MGS_ERR_CUDA, "cannot select the context's device");
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    int64_t blocks = (n + kDecThreads * kPer - 1) / (kDecThreads * kPer);
    const int64_t cap = (int64_t)ctx_sm_count(ctx) * 8;
    if (blocks > cap) blocks = cap;
    const bool fp16 = precision == MGS_PREC_FP16;
    const uintptr_t hp = reinterpret_cast<uintptr_t>(h), ap = reinterpret_cast<uintptr_t>(attrs);
    const bool vec = fp16 ? ((hp | ap) & 3) == 0 : (hp & 7) == 0 && (ap & 15) == 0;
    auto kern = fp16 ? (vec ? k_decode_sh<true, true> : k_decode_sh<true, false>)
                     : (vec ? k_decode_sh<false, true> : k_decode_sh<false, false>);
    kern<<<(unsigned)blocks, kDecThreads, 0, stream>>>(n, h, attrs, p);
    const cudaError_t e = cudaGetLastError();
    cudaSetDevice(prev);
    if (e != cudaSuccess) return bad(MGS_ERR_CUDA, "SH decode launch failed");
    return MGS_OK;
}
