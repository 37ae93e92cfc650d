// 3x3 layers of a few input channels (a network's first layer) on the FP32 pipe.
//
// The sums of such a layer are short (9 c_in products) and there are many of them: the layer moves more
// than it computes, and the matrix instructions, which take 16 (32) channels at a time, would be mostly
// padding.  It runs dense, with zeros in the pruned places: 2.4 us of packed multiply-adds for 3 -> 64 channels
// at 224x224, where the results alone take 2 us to write.  A lane keeps 16 filters of up to four pixels, and up to four
// neighbouring lanes the 64 filters of a pixel: a weight read from shared memory serves all pixels of a thread, a pixel read
// through L1 16 filters (per channel and tap 8 accesses for 32 packed multiply-adds), and the stores of a warp fill
// whole lines (lanes side by side over pixels, 256 bytes apart, took 32 lines an access and a quarter of the time).
// Against the command stream, us: 3 -> 64 at 224x224 fp32 12.2 -> 8.1, fp16 10.8 -> 7.8, int8 13.5 -> 8.3; 4 -> 64 12.9 -> 10.1, 11.9 -> 9.5,
// 14.6 -> 9.8; 13 images of 20x171, 6 -> 32, fp16 11.3 -> 6.4; 32 of 112x112, 3 -> 32, stride 2, fp32 19.9 -> 8.6; 32x32, 3 -> 32, int8 8.6 -> 2.8.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <vector>

#include "fewconv.h"
#include "patconv_internal.h"

namespace patconv {

constexpr int kFewThreads = 128, kFewWarps = kFewThreads / 32;
constexpr int kFewFilters = 64;                 // filters of a block, at most: four groups of 16
constexpr int kFewPitch = 20;                   // words of a group's 16 weights: four lanes' groups in distinct banks

struct FewParams {
    const void *x; void *y; const void *bias; const float *w;
    int h, wd, ho, wo, c_out, rows;
    int relu, stride;
    int groups, log_groups;                     // groups of 16 filters in a block (1, 2 or 4)
    int vec_y, y32;                             // 16-byte (32-byte) pieces of y are aligned
    unsigned pixels;
};

__device__ __forceinline__ void fma2(float &a0, float &a1, float w0, float w1, float x) {
    asm("{\n .reg .b64 a, b, c;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %4};\n mov.b64 c, {%0, %1};\n fma.rn.f32x2 c, a, b, c;\n mov.b64 {%0, %1}, c;\n}"
        : "+f"(a0), "+f"(a1) : "f"(w0), "f"(w1), "f"(x));
}

template <int DT> __device__ __forceinline__ float few_value(const void *x, size_t i) {
    if constexpr (DT == XGEN_F32) return __ldg(static_cast<const float *>(x) + i);
    else if constexpr (DT == XGEN_F16_F32ACC) return __half2float(__ushort_as_half(__ldg(static_cast<const unsigned short *>(x) + i)));
    else return (float)__ldg(static_cast<const unsigned char *>(x) + i);
}

// The CIN channels of a pixel.  (One by one: accesses of two or four channels at once took a second form of every tap for
// tensors that are not aligned to them, and twice the code: 4 -> 64 at 224x224 fp16 11.2 us, 9.5 one by one.)
template <int DT, int CIN> __device__ __forceinline__ void few_pixel(const FewParams &P, size_t i, float (&v)[CIN]) {
#pragma unroll
    for (int e = 0; e < CIN; ++e) v[e] = few_value<DT>(P.x, i + e);
}

// Store one result.  (ReLU of a NaN is 0, as on the command stream, which the same handle's fused runs and its runs of large images
// with few kernels left take.)
template <int DT> __device__ __forceinline__ void few_store1(const FewParams &P, size_t i, float sum, const void *bias, int c) {
    if constexpr (DT == XGEN_I8_I32) {
        // (the sum is exact, at most 7 x 4 products below 2^15; a bias that takes it past 2^31 wraps, as on the matrix path)
        const int v = (int)((uint32_t)(int)sum + (bias ? static_cast<const uint32_t *>(bias)[c] : 0u));
        static_cast<int *>(P.y)[i] = P.relu ? max(v, 0) : v;
    } else {
        float v = sum + (bias ? static_cast<const float *>(bias)[c] : 0.0f);
        if (P.relu) v = fmaxf(v, 0.0f);
        if constexpr (DT == XGEN_F32) static_cast<float *>(P.y)[i] = v;
        else static_cast<__half *>(P.y)[i] = __float2half_rn(v);
    }
}

// PX pixels of a thread.
template <int DT, int CIN, int PX>
__global__ void __launch_bounds__(kFewThreads, 3) few_kernel(const __grid_constant__ FewParams P) {
    __shared__ __align__(16) float s_w[9 * CIN * 4 * kFewPitch];
    asm volatile("griddepcontrol.launch_dependents;");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n0 = blockIdx.y * kFewFilters, width = P.groups * kFewPitch;
    for (int i = threadIdx.x; i < 9 * CIN * P.groups * 4; i += kFewThreads) {
        const int k = i >> (P.log_groups + 2), f = (i & (P.groups * 4 - 1)) * 4;
        const bool in = n0 + f < P.rows;
        *reinterpret_cast<float4 *>(s_w + k * width + f / 16 * kFewPitch + f % 16) =
            in ? __ldg(reinterpret_cast<const float4 *>(P.w + (size_t)k * P.rows + n0 + f)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int group = lane & (P.groups - 1), c0 = n0 + group * 16;
    const unsigned side = 32u >> P.log_groups;             // pixels of a warp side by side
    const unsigned first = (blockIdx.x * kFewWarps + warp) * (side * PX) + (lane >> P.log_groups);
    if (c0 >= P.c_out) return;
    int iy0[PX], ix0[PX];
    size_t img[PX];
    int at0[PX];                                           // element of the first tap, from the image's first row on
    unsigned in_y[PX], in_x[PX];                           // a bit a row (column) of taps: inside the image
#pragma unroll
    for (int p = 0; p < PX; ++p) {
        const unsigned px = min(first + side * p, P.pixels - 1);
        const unsigned row = px / (unsigned)P.wo, n = row / (unsigned)P.ho;
        ix0[p] = (int)(px - row * (unsigned)P.wo) * P.stride - 1;
        iy0[p] = (int)(row - n * (unsigned)P.ho) * P.stride - 1;
        img[p] = (size_t)n * P.h;
        at0[p] = (int)(img[p] + iy0[p]) * P.wd * CIN + ix0[p] * CIN;          // (x has fewer than 2^31 elements)
        in_y[p] = in_x[p] = 0u;
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            if ((unsigned)(iy0[p] + t) < (unsigned)P.h) in_y[p] |= 1u << t;
            if ((unsigned)(ix0[p] + t) < (unsigned)P.wd) in_x[p] |= 1u << t;
        }
    }
    float acc[PX][16];
#pragma unroll
    for (int p = 0; p < PX; ++p)
#pragma unroll
        for (int f = 0; f < 16; ++f) acc[p][f] = 0.0f;
    const float *const w = s_w + group * kFewPitch;
    // a tap's pixels are asked for while the tap before is multiplied
    float v[2][PX][CIN];
    auto fetch = [&](int t, float (&to)[PX][CIN]) {
#pragma unroll
        for (int p = 0; p < PX; ++p) {
#pragma unroll
            for (int c = 0; c < CIN; ++c) to[p][c] = 0.0f;
            if ((in_y[p] >> (t / 3) & in_x[p] >> (t % 3)) & 1u) few_pixel<DT, CIN>(P, (size_t)(at0[p] + (t / 3 * P.wd + t % 3) * CIN), to[p]);
        }
    };
    fetch(0, v[0]);
#pragma unroll
    for (int t = 0; t < 9; ++t) {
        if (t < 8) fetch(t + 1, v[(t + 1) & 1]);
#pragma unroll
        for (int c = 0; c < CIN; ++c) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 f = *reinterpret_cast<const float4 *>(w + (t * CIN + c) * width + 4 * q);
#pragma unroll
                for (int p = 0; p < PX; ++p) {
                    fma2(acc[p][4 * q], acc[p][4 * q + 1], f.x, f.y, v[t & 1][p][c]);
                    fma2(acc[p][4 * q + 2], acc[p][4 * q + 3], f.z, f.w, v[t & 1][p][c]);
                }
            }
        }
    }
    const bool whole = P.vec_y && c0 + 16 <= P.c_out;
#pragma unroll
    for (int p = 0; p < PX; ++p) {
        const unsigned px = first + side * p;
        if (px >= P.pixels) break;
        const size_t at = (size_t)px * P.c_out + c0;
        if constexpr (DT != XGEN_I8_I32) {
            // A sum that is infinite or NaN may have met an infinity under a pruned weight: it is added up anew from
            // the kept weights alone.
            float odd = 0.0f;
#pragma unroll
            for (int f = 0; f < 16; ++f) odd = fmaf(acc[p][f], 0.0f, odd);
            if (odd != 0.0f) {                          // (NaN)
#pragma unroll 1
                for (int f = 0; f < 16 && c0 + f < P.c_out; ++f) {
                    float sum = 0.0f;
                    const float *wf = s_w + group * kFewPitch + f;
#pragma unroll 1
                    for (int k = 0; k < 9 * CIN; ++k, wf += width) {
                        const int t = k / CIN, iy = iy0[p] + t / 3, ix = ix0[p] + t % 3;
                        if (__float_as_uint(*wf) == 0u) continue;                          // pruned
                        const bool in = (unsigned)iy < (unsigned)P.h && (unsigned)ix < (unsigned)P.wd;
                        sum = fmaf(*wf, in ? few_value<DT>(P.x, ((img[p] + iy) * P.wd + ix) * CIN + (k - t * CIN)) : 0.0f, sum);
                    }
                    few_store1<DT>(P, at + f, sum, P.bias, c0 + f);
                }
                continue;
            }
        }
        if (!whole) {
#pragma unroll
            for (int f = 0; f < 16; ++f)
                if (c0 + f < P.c_out) few_store1<DT>(P, at + f, acc[p][f], P.bias, c0 + f);
            continue;
        }
        uint32_t o[16];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint4 b = P.bias ? __ldg(reinterpret_cast<const uint4 *>(P.bias) + c0 / 4 + q) : make_uint4(0u, 0u, 0u, 0u);
            const uint32_t bb[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if constexpr (DT == XGEN_I8_I32) {
                    const int v = (int)((uint32_t)(int)acc[p][4 * q + e] + bb[e]);
                    o[4 * q + e] = (uint32_t)(P.relu ? max(v, 0) : v);
                } else {
                    float v = acc[p][4 * q + e] + __uint_as_float(bb[e]);
                    if (P.relu) v = fmaxf(v, 0.0f);
                    o[4 * q + e] = __float_as_uint(v);
                }
            }
        }
        constexpr int NW = DT == XGEN_F16_F32ACC ? 8 : 16;
        if constexpr (DT == XGEN_F16_F32ACC) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const __half2 t = __floats2half2_rn(__uint_as_float(o[2 * e]), __uint_as_float(o[2 * e + 1]));
                o[e] = *reinterpret_cast<const uint32_t *>(&t);
            }
        }
        uint32_t *const y = reinterpret_cast<uint32_t *>(static_cast<char *>(P.y) + at * (DT == XGEN_F16_F32ACC ? 2 : 4));
        if (P.y32) {
#pragma unroll
            for (int q = 0; q < NW / 8; ++q)
                asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                             ::"l"(y + 8 * q), "r"(o[8 * q]), "r"(o[8 * q + 1]), "r"(o[8 * q + 2]), "r"(o[8 * q + 3]),
                               "r"(o[8 * q + 4]), "r"(o[8 * q + 5]), "r"(o[8 * q + 6]), "r"(o[8 * q + 7]) : "memory");
        } else {
#pragma unroll
            for (int q = 0; q < NW / 4; ++q) reinterpret_cast<uint4 *>(y)[q] = make_uint4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
        }
    }
}

xgen_status few_upload(FewWeights &fw, xgen_dtype dt, int c_in, int c_out, const int16_t *kpat, const uint32_t *kw4,
                       const uint16_t *masks) {
    fw.dtype = dt; fw.c_in = c_in; fw.c_out = c_out; fw.rows = (c_out + 15) / 16 * 16;
    std::vector<float> w;
    try {
        w.assign((size_t)9 * c_in * fw.rows, 0.0f);
    } catch (const std::bad_alloc &) {
        return XGEN_ERR_ALLOC;
    }
    for (int oc = 0; oc < c_out; ++oc)
        for (int ic = 0; ic < c_in; ++ic) {
            const size_t k = (size_t)oc * c_in + ic;
            if (kpat[k] < 0) continue;
            for (int t = 0, kept = 0; t < 9; ++t)
                if (masks[kpat[k]] >> t & 1) {
                    float v;
                    std::memcpy(&v, kw4 + 4 * k + kept++, 4);
                    w[((size_t)t * c_in + ic) * fw.rows + oc] = v == 0.0f ? -0.0f : v;
                }
        }
    cudaError_t e = cudaMalloc(&fw.dev, w.size() * 4);
    if (e == cudaSuccess) e = cudaMemcpy(fw.dev, w.data(), w.size() * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) return XGEN_OK;
    cudaGetLastError();
    few_free(fw);
    return e == cudaErrorMemoryAllocation ? XGEN_ERR_ALLOC : XGEN_ERR_CUDA;
}
void few_free(FewWeights &fw) {
    if (fw.dev) cudaFree(fw.dev);
    fw = FewWeights();
}

template <int DT, int CIN> static const void *few_kernel_px(int px) {
    return px == 4 ? (const void *)few_kernel<DT, CIN, 4> : px == 2 ? (const void *)few_kernel<DT, CIN, 2> : (const void *)few_kernel<DT, CIN, 1>;
}
template <int DT> static const void *few_kernel_of(int c_in, int px) {
    switch (c_in) {
        case 1: return few_kernel_px<DT, 1>(px);
        case 2: return few_kernel_px<DT, 2>(px);
        case 3: return few_kernel_px<DT, 3>(px);
        case 4: return few_kernel_px<DT, 4>(px);
        case 5: return few_kernel_px<DT, DT == XGEN_F32 ? 4 : 5>(px);
        case 6: return few_kernel_px<DT, DT == XGEN_F32 ? 4 : 6>(px);
        default: return few_kernel_px<DT, DT == XGEN_F32 ? 4 : 7>(px);
    }
}

// Of the current device.
static int sm_count() {
    static std::atomic<int> known[64];
    int device = 0, sms = 148;
    if (cudaGetDevice(&device) != cudaSuccess || device < 0 || device >= 64) return sms;
    if (const int k = known[device].load(std::memory_order_relaxed)) return k;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return 148;
    known[device].store(sms, std::memory_order_relaxed);
    return sms;
}

cudaError_t few_launch(const FewWeights &fw, const void *x, int n, int h, int w, int stride, const void *bias, bool relu, void *y,
                       bool overlap, cudaStream_t st) {
    FewParams P{};
    P.x = x; P.y = y; P.bias = bias; P.w = fw.dev;
    P.h = h; P.wd = w; P.ho = (h - 1) / stride + 1; P.wo = (w - 1) / stride + 1;
    P.c_out = fw.c_out; P.rows = fw.rows; P.relu = relu ? 1 : 0; P.stride = stride;
    P.pixels = (unsigned)((int64_t)n * P.ho * P.wo);
    const int yb = fw.dtype == XGEN_F16_F32ACC ? 2 : 4;
    P.vec_y = (uintptr_t)y % 16 == 0 && (uintptr_t)bias % 16 == 0 && (size_t)fw.c_out * yb % 16 == 0;
    P.y32 = P.vec_y && (uintptr_t)y % 32 == 0 && (size_t)fw.c_out * yb % 32 == 0;
    const int left = std::min(fw.rows, kFewFilters) / 16;
    P.log_groups = left > 2 ? 2 : left > 1 ? 1 : 0;
    P.groups = 1 << P.log_groups;
    // Four pixels a thread where that still gives every scheduler of the GPU two warps, else fewer, so that a small image
    // spreads over it (13 x 20x171, 3 -> 32, fp16: 10.3 us with four, 5.2 with two).
    const int64_t units = ((int64_t)P.pixels + 31) / 32 * ((fw.rows + 15) / 16);
    const int64_t sms = sm_count();
    const int px = units >= 4 * sms * 8 ? 4 : units >= 2 * sms * 8 ? 2 : 1;
    const int per_block = (kFewThreads >> P.log_groups) * px;
    const dim3 grid((unsigned)(((int64_t)P.pixels + per_block - 1) / per_block), (unsigned)((fw.rows + kFewFilters - 1) / kFewFilters));
    const void *kern = fw.dtype == XGEN_F32 ? few_kernel_of<XGEN_F32>(fw.c_in, px)
                     : fw.dtype == XGEN_F16_F32ACC ? few_kernel_of<XGEN_F16_F32ACC>(fw.c_in, px) : few_kernel_of<XGEN_I8_I32>(fw.c_in, px);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = dim3(kFewThreads); cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at; cfg.numAttrs = overlap ? 1 : 0;
    void *args[1] = {&P};
    cudaError_t e = cudaLaunchKernelExC(&cfg, kern, args);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) count_launch();
    return e;
}

}  // namespace patconv
