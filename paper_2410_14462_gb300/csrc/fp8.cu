// FP8-E4M3 storage of feature maps (the precision form's 8-bit variant; the
// format is the OCP 8-bit floating point one): every view v is scaled by
// s_v = max|x| / 448 over the view (1 for an all-zero view), so that its
// largest magnitude lands on the largest finite E4M3 value, and each scaled
// value is rounded to the nearest E4M3 code (ties to even, saturating).
// The uplift of FP8 features (ludvig_uplift_fp8, with the uplift kernels)
// multiplies the codes back by s_v.
//
// Three passes over the features: a per-view maximum of |x| (the float bits
// of non-negative values order like unsigned integers, so atomicMax on them
// is exact), the scales, and the rounding of x / s_v (IEEE division, then the
// hardware's round-to-nearest-even E4M3 conversion).
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "common.cuh"

namespace ludvig {

namespace {

// Both passes take a view's elements in pieces of P x 256 groups of four (float32)
// or eight (bfloat16): 16-byte loads, P = 4 of them in flight per thread, or one where
// the views are too small to give every SM a few pieces of four.  A view that does not
// start on a 16-byte boundary (or whose codes do not start on one of a group's size), and
// the end of a view, go element by element, four at a time.
template <class T>
struct Vec {
    static constexpr int kN = 16 / (int)sizeof(T);
    float x[kN];
};
__device__ __forceinline__ void load_vec(const float* p, Vec<float>& v) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v.x[0] = q.x;
    v.x[1] = q.y;
    v.x[2] = q.z;
    v.x[3] = q.w;
}
__device__ __forceinline__ void load_vec(const __nv_bfloat16* p, Vec<__nv_bfloat16>& v) {
    const uint4 q = *reinterpret_cast<const uint4*>(p);
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        v.x[2 * k] = __uint_as_float(w[k] << 16);
        v.x[2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u);
    }
}
__device__ __forceinline__ float load_x(const float* p, int64_t i) { return p[i]; }
__device__ __forceinline__ float load_x(const __nv_bfloat16* p, int64_t i) { return __bfloat162float(p[i]); }

template <class T, int P>
constexpr int64_t piece_elems() {
    return (int64_t)P * 256 * Vec<T>::kN;
}

// blockIdx.y = view; grid-stride over the view's pieces.
template <class T, int P>
__global__ void __launch_bounds__(256) k_view_absmax(const T* __restrict__ x, int64_t view_elems,
                                                     uint32_t* __restrict__ amax_bits) {
    constexpr int kN = Vec<T>::kN;
    const T* xv = x + (int64_t)blockIdx.y * view_elems;
    const bool vec = (reinterpret_cast<uintptr_t>(xv) & 15) == 0;
    float m = 0.f;
    for (int64_t e0 = (int64_t)blockIdx.x * piece_elems<T, P>(); e0 < view_elems;
         e0 += (int64_t)gridDim.x * piece_elems<T, P>()) {
        if (vec && e0 + piece_elems<T, P>() <= view_elems) {
            Vec<T> v[P];
#pragma unroll
            for (int k = 0; k < P; ++k) load_vec(xv + e0 + (int64_t)(k * 256 + threadIdx.x) * kN, v[k]);
#pragma unroll
            for (int k = 0; k < P; ++k)
#pragma unroll
                for (int q = 0; q < kN; ++q) m = fmaxf(m, fabsf(v[k].x[q]));
        } else {
            const int64_t e1 = min(view_elems, e0 + piece_elems<T, P>());
            for (int64_t e = e0 + threadIdx.x; e < e1; e += 4 * 256) {
                float v[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) v[k] = e + 256 * k < e1 ? load_x(xv, e + 256 * k) : 0.f;
#pragma unroll
                for (int k = 0; k < 4; ++k) m = fmaxf(m, fabsf(v[k]));
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    __shared__ float wm[8];
    if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        float b = wm[0];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) b = fmaxf(b, wm[w]);
        atomicMax(amax_bits + blockIdx.y, __float_as_uint(b));
    }
}

// In place: the maximum's bits become the scale.
__global__ void k_view_scales(float* __restrict__ s, int n_views) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n_views) return;
    const float amax = __uint_as_float(reinterpret_cast<const uint32_t*>(s)[v]);
    s[v] = amax > 0.f ? __fdiv_rn(amax, 448.0f) : 1.0f;
}

__device__ __forceinline__ uint32_t e4m3_of(float x, float s) {
    return (uint32_t)__nv_cvt_float_to_fp8(__fdiv_rn(x, s), __NV_SATFINITE, __NV_E4M3);
}

// blockIdx.y = view, blockIdx.x = piece of it.  Bound by HBM (5 or 3 bytes per
// element): 12 float32 views of 640x480x512 in 1.26 ms = 7.5 TB/s (3.14 ms with a
// 64-bit division and a 4-byte load per element); the maximum 1.24 -> 1.05 ms.
template <class T, int P>
__global__ void __launch_bounds__(256) k_quantize_e4m3(const T* __restrict__ x, const float* __restrict__ scales,
                                                       int64_t view_elems, uint8_t* __restrict__ q) {
    constexpr int kN = Vec<T>::kN;
    const T* xv = x + (int64_t)blockIdx.y * view_elems;
    uint8_t* qv = q + (int64_t)blockIdx.y * view_elems;
    const float s = scales[blockIdx.y];
    const int64_t e0 = (int64_t)blockIdx.x * piece_elems<T, P>();
    const bool vec = ((reinterpret_cast<uintptr_t>(xv) & 15) | (reinterpret_cast<uintptr_t>(qv) & (kN - 1))) == 0;
    if (vec && e0 + piece_elems<T, P>() <= view_elems) {
        Vec<T> v[P];
#pragma unroll
        for (int k = 0; k < P; ++k) load_vec(xv + e0 + (int64_t)(k * 256 + threadIdx.x) * kN, v[k]);
#pragma unroll
        for (int k = 0; k < P; ++k) {
            uint32_t w[kN / 4];
#pragma unroll
            for (int h = 0; h < kN / 4; ++h) {
                w[h] = 0u;
#pragma unroll
                for (int b = 0; b < 4; ++b) w[h] |= e4m3_of(v[k].x[4 * h + b], s) << (8 * b);
            }
            uint8_t* dst = qv + e0 + (int64_t)(k * 256 + threadIdx.x) * kN;
            if constexpr (kN == 4)
                *reinterpret_cast<uint32_t*>(dst) = w[0];
            else
                *reinterpret_cast<uint2*>(dst) = make_uint2(w[0], w[1]);
        }
    } else {
        const int64_t e1 = min(view_elems, e0 + piece_elems<T, P>());
        for (int64_t e = e0 + threadIdx.x; e < e1; e += 4 * 256) {
            float v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = e + 256 * k < e1 ? load_x(xv, e + 256 * k) : 0.f;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (e + 256 * k < e1) qv[e + 256 * k] = (uint8_t)e4m3_of(v[k], s);
        }
    }
}

template <class T, int P>
ludvig_status quantize(const T* x, int n_views, int64_t view_elems, uint8_t* q, float* scales, cudaStream_t st) {
    const int64_t pieces = ceil_div(view_elems, piece_elems<T, P>());
    LV_ARG(pieces <= 0x7fffffff, "view too large");
    k_view_absmax<T, P><<<dim3((unsigned)std::min<int64_t>(pieces, 1024), (unsigned)n_views), 256, 0, st>>>(
        x, view_elems, reinterpret_cast<uint32_t*>(scales));
    LV_LAUNCH();
    k_view_scales<<<(unsigned)ceil_div(n_views, 256), 256, 0, st>>>(scales, n_views);
    LV_LAUNCH();
    k_quantize_e4m3<T, P><<<dim3((unsigned)pieces, (unsigned)n_views), 256, 0, st>>>(x, scales, view_elems, q);
    LV_LAUNCH();
    return LUDVIG_OK;
}

// Pieces of four loads per thread where that gives the GPU a few blocks per SM; else of
// one (3 views of 8235 bfloat16 values, the call 18 -> 14 us).
template <class T>
ludvig_status quantize(const T* x, int n_views, int64_t view_elems, uint8_t* q, float* scales, cudaStream_t st) {
    return ceil_div(view_elems, piece_elems<T, 4>()) * n_views >= 4 * 152
               ? quantize<T, 4>(x, n_views, view_elems, q, scales, st)
               : quantize<T, 1>(x, n_views, view_elems, q, scales, st);
}

}  // namespace

}  // namespace ludvig

using namespace ludvig;

extern "C" ludvig_status ludvig_fp8_quantize(const void* feats, int32_t dtype, int32_t n_views, int64_t view_elems,
                                             uint8_t* q, float* scales, void* stream) {
    LV_ARG(dtype == LUDVIG_F32 || dtype == LUDVIG_BF16, "unknown dtype %d", dtype);
    LV_ARG(n_views >= 0 && n_views <= 65535, "n_views must be in [0, 65535]");
    LV_ARG(view_elems >= 0, "view_elems must be >= 0");
    if (n_views == 0) return LUDVIG_OK;
    LV_ARG(scales != nullptr, "scales is NULL");
    LV_ARG(view_elems == 0 || (feats != nullptr && q != nullptr), "NULL buffer");
    LV_ARG(((uintptr_t)q & 3) == 0, "q must be 4-byte aligned");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    LV_CUDA(cudaMemsetAsync(scales, 0, sizeof(float) * (size_t)n_views, st));
    if (view_elems > 0)
        return dtype == LUDVIG_F32
                   ? quantize(static_cast<const float*>(feats), n_views, view_elems, q, scales, st)
                   : quantize(static_cast<const __nv_bfloat16*>(feats), n_views, view_elems, q, scales, st);
    k_view_scales<<<(unsigned)ceil_div(n_views, 256), 256, 0, st>>>(scales, n_views);
    LV_LAUNCH();
    return LUDVIG_OK;
}
