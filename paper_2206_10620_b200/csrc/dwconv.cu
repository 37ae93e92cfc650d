// libpatconv: depthwise pattern-pruned 3x3 convolution (sm_100a) and its C ABI.
//
// Every channel has one 3x3 kernel that keeps the 4 weights of its pattern.  The layer moves
// two activations per 4 useful multiply-adds, so HBM binds it: the kernel's job is to read x
// once and write y once, with enough loads in flight and few instructions for an element (see
// dwconv_kernel).  Pruned taps carry weight 0 in the packed table [9][channels].
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "dwconv.h"
#include "patconv_internal.h"

struct xgen_dwconv_packed {
    int c = 0, stride = 1;
    xgen_dtype dtype = XGEN_F32;
    int device = -1;
    int64_t surviving = 0;
    std::vector<float> w9;          // [9][c], pruned taps zero
    float *d_w9 = nullptr;
};

namespace dwconv {

struct DParams {
    const void *x; void *y; const float *bias; const float *w9;
    int n, h, w, ho, wo, c;
    int relu;
    int cvs;                        // threads side by side along the channels, c / V
    int strips;                     // strips of TX output pixels per output row
    int segs, seg_rows;             // pieces of an image's rows, rows of a piece
    unsigned threads;
};

// V channels as stored: loaded and stored in one access.
template <int DT, int V> struct Raw { static constexpr int words = DT == XGEN_F32 ? V : (V + 1) / 2; uint32_t r[words]; };

template <int DT, int V> __device__ __forceinline__ Raw<DT, V> load_raw(const void *x, unsigned elem, bool ok) {
    Raw<DT, V> t;
#pragma unroll
    for (int i = 0; i < Raw<DT, V>::words; ++i) t.r[i] = 0u;
    if (!ok) return t;
    const char *p = static_cast<const char *>(x) + (size_t)elem * (DT == XGEN_F32 ? 4 : 2);
    constexpr int bytes = V * (DT == XGEN_F32 ? 4 : 2);
    if constexpr (bytes == 16) { const uint4 u = __ldg(reinterpret_cast<const uint4 *>(p)); t.r[0] = u.x; t.r[1] = u.y; t.r[2] = u.z; t.r[3] = u.w; }
    else if constexpr (bytes == 8) { const uint2 u = __ldg(reinterpret_cast<const uint2 *>(p)); t.r[0] = u.x; t.r[1] = u.y; }
    else if constexpr (bytes == 4) t.r[0] = __ldg(reinterpret_cast<const uint32_t *>(p));
    else t.r[0] = __ldg(reinterpret_cast<const unsigned short *>(p));
    return t;
}
template <int DT, int V> __device__ __forceinline__ void widen(const Raw<DT, V> &t, float (&v)[V]) {
    if constexpr (DT == XGEN_F32) {
#pragma unroll
        for (int i = 0; i < V; ++i) v[i] = __uint_as_float(t.r[i]);
    } else if constexpr (V == 1) {
        v[0] = __half2float(__ushort_as_half((unsigned short)t.r[0]));
    } else {
#pragma unroll
        for (int i = 0; i < V / 2; ++i) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&t.r[i]));
            v[2 * i] = f.x; v[2 * i + 1] = f.y;
        }
    }
}
template <int DT, int V> __device__ __forceinline__ void store_vec(void *y, unsigned elem, const float (&v)[V]) {
    char *p = static_cast<char *>(y) + (size_t)elem * (DT == XGEN_F32 ? 4 : 2);
    if constexpr (DT == XGEN_F32) {
        if constexpr (V == 4) *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
        else if constexpr (V == 2) *reinterpret_cast<float2 *>(p) = make_float2(v[0], v[1]);
        else *reinterpret_cast<float *>(p) = v[0];
    } else if constexpr (V == 1) {
        *reinterpret_cast<__half *>(p) = __float2half_rn(v[0]);
    } else {
        uint32_t o[V / 2];
#pragma unroll
        for (int i = 0; i < V / 2; ++i) {
            const __half2 h = __floats2half2_rn(v[2 * i], v[2 * i + 1]);
            o[i] = *reinterpret_cast<const uint32_t *>(&h);
        }
        if constexpr (V == 4) *reinterpret_cast<uint2 *>(p) = make_uint2(o[0], o[1]);
        else *reinterpret_cast<uint32_t *>(p) = o[0];
    }
}

// acc += w * x per channel; two channels an instruction where V allows it.
template <int V> __device__ __forceinline__ void fma_v(float (&acc)[V], const float (&w)[V], const float (&x)[V]) {
    if constexpr (V == 1) acc[0] = fmaf(w[0], x[0], acc[0]);
    else {
#pragma unroll
        for (int i = 0; i < V; i += 2)
            asm("{\n .reg .b64 a, b, c;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n mov.b64 c, {%0, %1};\n"
                " fma.rn.f32x2 c, a, b, c;\n mov.b64 {%0, %1}, c;\n}"
                : "+f"(acc[i]), "+f"(acc[i + 1]) : "f"(w[i]), "f"(w[i + 1]), "f"(x[i]), "f"(x[i + 1]));
    }
}

// V channels global -> shared, asynchronously; zeros where !ok (nothing is read then).
template <int BYTES> __device__ __forceinline__ void copy_v(uint32_t dst, const char *src, bool ok) {
    if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16u : 0u) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst), "l"(src), "n"(BYTES), "r"(ok ? (uint32_t)BYTES : 0u) : "memory");
}

// Memory binds the layer (4 useful multiply-adds per two activations moved), so the kernel is built to
// keep loads in flight and to spend few instructions on an element.  A thread owns V channels of a
// strip of TX output pixels and walks down a piece of the image's rows: an input row is loaded once
// (the next row while this one is used), widened once, and added to the three output rows that it
// belongs to (stride 2: an odd row is kept for the next output row).  All nine taps run with masked
// weights, two channels an instruction: skipping a tap would save no traffic.  32 images of
// 56x56x128 fp16: 24.2 us with a thread per output strip (each input row loaded and widened
// three times, 825 instructions for 16 results), 16.2 us with rows walked.
// AHEAD (stride 1): rows come kAhead ahead of their use, by asynchronous copies into shared memory that is the thread's
// own, so no thread waits for another and rows on their way hold no registers: 14.7 us (see where it is chosen).
// S = stride, V = channels per thread (4, 2 or 1), TX = output pixels per thread along x.
constexpr int kAhead = 3, kSlots = kAhead + 1;
template <int DT, int S, int V, int TX, bool AHEAD>
__global__ void __launch_bounds__(128) dwconv_kernel(const __grid_constant__ DParams P) {
    constexpr int NC = (TX - 1) * S + 3;            // input columns a strip needs
    constexpr int kBytes = V * (DT == XGEN_F32 ? 4 : 2);
    __shared__ __align__(16) unsigned char ring[AHEAD ? kSlots * NC * 128 * kBytes : 16];
    asm volatile("griddepcontrol.launch_dependents;");
    const unsigned id = blockIdx.x * 128u + threadIdx.x;
    if (id >= P.threads) return;
    unsigned q = id / (unsigned)P.cvs;
    const unsigned ch = (id - q * (unsigned)P.cvs) * V;
    unsigned q2 = q / (unsigned)P.strips;
    const int ox0 = (int)(q - q2 * (unsigned)P.strips) * TX;
    const unsigned n = q2 / (unsigned)P.segs;
    const int oy0 = (int)(q2 - n * (unsigned)P.segs) * P.seg_rows, oy1 = min(P.ho, oy0 + P.seg_rows);
    if (oy0 >= oy1) return;

    float wt[9][V];
#pragma unroll
    for (int t = 0; t < 9; ++t) {
        const Raw<XGEN_F32, V> r = load_raw<XGEN_F32, V>(P.w9, (unsigned)t * (unsigned)P.c + ch, true);
        widen<XGEN_F32, V>(r, wt[t]);
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    float bias[V];
#pragma unroll
    for (int v = 0; v < V; ++v) bias[v] = P.bias ? __ldg(P.bias + ch + v) : 0.0f;

    // Tensors hold fewer than 2^31 elements, so element offsets are 32-bit.
    const unsigned row_elems = (unsigned)P.w * (unsigned)P.c;
    const unsigned x0 = n * (unsigned)P.h * row_elems + ch;
    bool col_ok[NC];
#pragma unroll
    for (int j = 0; j < NC; ++j) col_ok[j] = (unsigned)(ox0 * S + j - 1) < (unsigned)P.w;
    auto fetch = [&](Raw<DT, V> (&raw)[NC], int iy) {
        const bool row_ok = (unsigned)iy < (unsigned)P.h;
        const unsigned at = x0 + (unsigned)iy * row_elems + (unsigned)(ox0 * S - 1) * (unsigned)P.c;
#pragma unroll
        for (int j = 0; j < NC; ++j) raw[j] = load_raw<DT, V>(P.x, at + (unsigned)j * (unsigned)P.c, row_ok && col_ok[j]);
    };
    auto emit = [&](const float (&acc)[TX][V], int oy) {
        const unsigned at = ((n * (unsigned)P.ho + (unsigned)oy) * (unsigned)P.wo + (unsigned)ox0) * (unsigned)P.c + ch;
#pragma unroll
        for (int t = 0; t < TX; ++t) {
            if (ox0 + t >= P.wo) break;
            float o[V];
#pragma unroll
            for (int v = 0; v < V; ++v) {
                o[v] = acc[t][v];
                if (P.relu) o[v] = fmaxf(o[v], 0.0f);
            }
            store_vec<DT, V>(P.y, at + (unsigned)t * (unsigned)P.c, o);
        }
    };
    auto start = [&](float (&acc)[TX][V]) {
#pragma unroll
        for (int t = 0; t < TX; ++t)
#pragma unroll
            for (int v = 0; v < V; ++v) acc[t][v] = bias[v];
    };
    auto add_row = [&](float (&acc)[TX][V], const float (&col)[NC][V], int dy) {
#pragma unroll
        for (int t = 0; t < TX; ++t)
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) fma_v<V>(acc[t], wt[3 * dy + dx], col[t * S + dx]);
    };
    auto widen_row = [&](const Raw<DT, V> (&raw)[NC], float (&col)[NC][V]) {
#pragma unroll
        for (int j = 0; j < NC; ++j) widen<DT, V>(raw[j], col[j]);
    };

    if constexpr (S == 1) {
        float acc[3][TX][V];
        start(acc[1]);
        start(acc[2]);
        Raw<DT, V> raw[NC];
        int next = oy0 - 1;                         // AHEAD: the row that is asked for next
        unsigned put = 0, got = 0;
        const uint32_t mine = (uint32_t)__cvta_generic_to_shared(ring) + threadIdx.x * kBytes;
        auto ask = [&]() {
            const bool row_ok = next <= oy1 && (unsigned)next < (unsigned)P.h;
            const unsigned at = x0 + (unsigned)next * row_elems + (unsigned)(ox0 - 1) * (unsigned)P.c;
            const uint32_t dst = mine + put * (NC * 128 * kBytes);
#pragma unroll
            for (int j = 0; j < NC; ++j) {
                const bool ok = row_ok && col_ok[j];
                copy_v<AHEAD ? kBytes : 16>(dst + j * (128 * kBytes), static_cast<const char *>(P.x) + (ok ? (size_t)(at + (unsigned)j * (unsigned)P.c) * (DT == XGEN_F32 ? 4 : 2) : 0), ok);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            put = put + 1 == kSlots ? 0 : put + 1;
            ++next;
        };
        auto take = [&](float (&col)[NC][V]) {
            ask();
            asm volatile("cp.async.wait_group %0;" ::"n"(kAhead) : "memory");
            const unsigned char *const src = ring + got * (NC * 128 * kBytes) + threadIdx.x * kBytes;
#pragma unroll
            for (int j = 0; j < NC; ++j) {
                Raw<DT, V> t;
                if constexpr (kBytes == 16) { const uint4 u = *reinterpret_cast<const uint4 *>(src + j * (128 * kBytes)); t.r[0] = u.x; t.r[1] = u.y; t.r[2] = u.z; t.r[3] = u.w; }
                else if constexpr (kBytes == 8) { const uint2 u = *reinterpret_cast<const uint2 *>(src + j * (128 * kBytes)); t.r[0] = u.x; t.r[1] = u.y; }
                widen<DT, V>(t, col[j]);
            }
            got = got + 1 == kSlots ? 0 : got + 1;
        };
        if constexpr (AHEAD) {
#pragma unroll
            for (int i = 0; i < kAhead; ++i) ask();
        } else fetch(raw, oy0 - 1);
        // input row r goes to output rows r + 1 (starting it), r, and r - 1 (finishing it); the three
        // accumulators change places, so three steps are written out
        for (int r = oy0 - 1; r <= oy1; r += 3) {
#pragma unroll
            for (int u = 0; u < 3; ++u) {
                if (r + u > oy1) break;
                float col[NC][V];
                if constexpr (AHEAD) take(col);
                else {
                    widen_row(raw, col);
                    if (r + u < oy1) fetch(raw, r + u + 1);
                }
                start(acc[u]);
                add_row(acc[u], col, 0);
                add_row(acc[(u + 2) % 3], col, 1);
                add_row(acc[(u + 1) % 3], col, 2);
                if (r + u - 1 >= oy0) emit(acc[(u + 1) % 3], r + u - 1);
            }
        }
    } else {
        Raw<DT, V> even[NC], odd[NC];
        float above[NC][V], col[NC][V], acc[TX][V];
        fetch(odd, 2 * oy0 - 1);
        fetch(even, 2 * oy0);
        widen_row(odd, above);
        fetch(odd, 2 * oy0 + 1);
        for (int oy = oy0; oy < oy1; ++oy) {
            start(acc);
            add_row(acc, above, 0);
            widen_row(even, col);
            if (oy + 1 < oy1) fetch(even, 2 * oy + 2);
            add_row(acc, col, 1);
            widen_row(odd, above);
            if (oy + 1 < oy1) fetch(odd, 2 * oy + 3);
            add_row(acc, above, 2);
            emit(acc, oy);
        }
    }
}

constexpr int kStrip1 = 4, kStrip2 = 2;     // output pixels per thread at stride 1 / 2

template <int DT> static const void *kernel_dt(int stride, int v, bool ahead) {
    if (stride == 1) {
        if (ahead && v == 4) return (const void *)dwconv_kernel<DT, 1, 4, kStrip1, true>;
        if constexpr (DT == XGEN_F32) if (ahead && v == 2) return (const void *)dwconv_kernel<DT, 1, 2, kStrip1, true>;
        return v == 4 ? (const void *)dwconv_kernel<DT, 1, 4, kStrip1, false> : v == 2 ? (const void *)dwconv_kernel<DT, 1, 2, kStrip1, false>
                                                                                        : (const void *)dwconv_kernel<DT, 1, 1, kStrip1, false>;
    }
    return v == 4 ? (const void *)dwconv_kernel<DT, 2, 4, kStrip2, false> : v == 2 ? (const void *)dwconv_kernel<DT, 2, 2, kStrip2, false>
                                                                                    : (const void *)dwconv_kernel<DT, 2, 1, kStrip2, false>;
}
static const void *kernel_for(xgen_dtype dt, int stride, int v, bool ahead) {
    return dt == XGEN_F32 ? kernel_dt<XGEN_F32>(stride, v, ahead) : kernel_dt<XGEN_F16_F32ACC>(stride, v, ahead);
}

// Blocks of the kernel that the device holds at once (asked for once per kernel and device).
static int resident_blocks(const void *kern, int device) {
    static std::mutex mu;
    static std::vector<std::array<intptr_t, 3>> known;
    std::lock_guard<std::mutex> lock(mu);
    for (auto &k : known)
        if (k[0] == (intptr_t)kern && k[1] == device) return (int)k[2];
    int sms = 148, per_sm = 4;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 128, 0) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        per_sm = 4;
    }
    known.push_back({(intptr_t)kern, device, sms * per_sm});
    return sms * per_sm;
}

static float half_bits_to_float(uint16_t h) {
    const uint32_t sign = (uint32_t)(h >> 15) << 31;
    const int exp = (h >> 10) & 0x1f;
    uint32_t man = h & 0x3ff, bits;
    if (exp == 0) {
        if (man == 0) bits = sign;
        else {
            int e = -1;
            do { ++e; man <<= 1; } while (!(man & 0x400));
            bits = sign | (uint32_t)(127 - 15 - e) << 23 | (man & 0x3ff) << 13;
        }
    } else if (exp == 31) bits = sign | 0x7f800000u | man << 13;
    else bits = sign | (uint32_t)(exp - 15 + 127) << 23 | man << 13;
    float f;
    std::memcpy(&f, &bits, 4);
    return f;
}

}  // namespace dwconv

using namespace dwconv;

extern "C" {

xgen_status xgen_dwconv_pack(const xgen_dwconv_desc *d, const void *dense_w, const int16_t *pid, int device,
                             xgen_dwconv_packed **out) {
    if (!d || !dense_w || !pid || !out || !d->pattern_masks) return XGEN_ERR_INVALID_ARG;
    *out = nullptr;
    if (d->channels < 1) return XGEN_ERR_INVALID_ARG;
    if (d->pad != 1 || (d->stride != 1 && d->stride != 2)) return XGEN_ERR_UNSUPPORTED;
    if (d->dtype != XGEN_F32 && d->dtype != XGEN_F16_F32ACC) return XGEN_ERR_UNSUPPORTED;
    if (d->num_patterns < 1 || d->num_patterns > patconv::kNumAllMasks) return XGEN_ERR_BAD_PATTERN;
    for (int p = 0; p < d->num_patterns; ++p) {
        const uint16_t m = d->pattern_masks[p];
        if (m >= 512 || __builtin_popcount(m) != 4) return XGEN_ERR_BAD_PATTERN;
    }
    xgen_dwconv_packed *h = new (std::nothrow) xgen_dwconv_packed();
    if (!h) return XGEN_ERR_ALLOC;
    try {
        h->c = d->channels; h->stride = d->stride; h->dtype = d->dtype; h->device = device;
        h->w9.assign((size_t)9 * d->channels, 0.0f);
        for (int c = 0; c < d->channels; ++c) {
            const int p = pid[c];
            if (p >= d->num_patterns || p < -1) { delete h; return XGEN_ERR_BAD_PATTERN; }
            if (p < 0) continue;
            ++h->surviving;
            for (int t = 0; t < 9; ++t) {
                if (!((d->pattern_masks[p] >> t) & 1)) continue;
                const size_t i = (size_t)c * 9 + t;
                h->w9[(size_t)t * d->channels + c] = d->dtype == XGEN_F32 ? static_cast<const float *>(dense_w)[i]
                                                                           : half_bits_to_float(static_cast<const uint16_t *>(dense_w)[i]);
            }
        }
    } catch (const std::bad_alloc &) {
        delete h;
        return XGEN_ERR_ALLOC;
    }
    if (device >= 0) {
        int prev = 0;
        cudaGetDevice(&prev);
        xgen_status st = XGEN_OK;
        if (cudaSetDevice(device) != cudaSuccess) st = XGEN_ERR_CUDA;
        if (st == XGEN_OK && cudaMalloc(&h->d_w9, h->w9.size() * 4) != cudaSuccess) st = XGEN_ERR_ALLOC;
        if (st == XGEN_OK && cudaMemcpy(h->d_w9, h->w9.data(), h->w9.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess) st = XGEN_ERR_CUDA;
        cudaSetDevice(prev);
        if (st != XGEN_OK) {
            cudaGetLastError();
            xgen_dwconv_free(h);
            return st;
        }
    }
    *out = h;
    return XGEN_OK;
}

xgen_status xgen_dwconv_run(const xgen_dwconv_packed *h, const void *x, int32_t n, int32_t hh, int32_t ww,
                            const void *bias, int32_t relu, void *y, void *stream) {
    if (!h || !x || !y) return XGEN_ERR_INVALID_ARG;
    const size_t eb = h->dtype == XGEN_F32 ? 4 : 2;
    if (((uintptr_t)x % eb) || ((uintptr_t)y % eb) || ((uintptr_t)bias % 4)) return XGEN_ERR_INVALID_ARG;
    if (n < 1 || hh < 1 || ww < 1) return XGEN_ERR_SHAPE;
    const int ho = (hh + 2 - 3) / h->stride + 1, wo = (ww + 2 - 3) / h->stride + 1;
    const int64_t xe = (int64_t)n * hh * ww * h->c, ye = (int64_t)n * ho * wo * h->c;
    if (xe > 2147483647LL || ye > 2147483647LL) return XGEN_ERR_SHAPE;
    {
        const uintptr_t xa = (uintptr_t)x, xz = xa + (size_t)xe * eb, ya = (uintptr_t)y, yz = ya + (size_t)ye * eb;
        if (xa < yz && ya < xz) return XGEN_ERR_INVALID_ARG;
    }
    if (h->device < 0) return XGEN_ERR_CUDA;
    auto whole = [&](int v) {                                   // v channels are one aligned access everywhere
        return h->c % v == 0 && (uintptr_t)x % (v * eb) == 0 && (uintptr_t)y % (v * eb) == 0;
    };
    const int v = whole(4) ? 4 : whole(2) ? 2 : 1;
    const int tx = h->stride == 1 ? kStrip1 : kStrip2;
    DParams P{};
    P.x = x; P.y = y; P.bias = static_cast<const float *>(bias); P.w9 = h->d_w9;
    P.n = n; P.h = hh; P.w = ww; P.ho = ho; P.wo = wo; P.c = h->c;
    P.relu = relu ? 1 : 0;
    P.cvs = h->c / v;
    P.strips = (wo + tx - 1) / tx;
    // Rows ahead, where a call is long enough for bandwidth to count and accesses are 8 bytes or more (a copy of 4 bytes
    // costs as much), later for pairs of fp32, whose copies carry half of what those of four do.  us without and with: fp16 32x56x56x128 (51 MB) 16.2, 14.7; 123x188x336 (31 MB) 11.6, 11.0;
    // fp32 16x56x56x128 12.8, 10.0; but 11x49x39x112 (9 MB) 5.5, 6.0; 20x14x14x512 4.5, 5.0; single fp32 channels 8x42x42x881 25.0, 27.0;
    // pairs of fp16 8x42x42x882 17.5, 21.5; stride 2, two rows ahead in registers, 8x112x112x64 3.7, 5.0.
    // Around 24 MB fp16 15x56x56x128 9.0, 8.8, 13x56x56x128 (21 MB) 7.3 without; fp32 15x28x28x256 6.5, 5.8; fp32 pairs 36 MB 11x56x56x130
    // 9.8, 10.7; 70 MB 6x75x75x250 16.6, 16.7, 21x56x56x130 17.0, 17.6; 100 MB 9x75x75x250 23.6, 22.6, 31x28x28x510 22.5, 21.0.
    const bool ahead = h->stride == 1 && v * (int)eb >= 8 && (xe + ye) * (int64_t)eb >= (eb == 4 && v == 2 ? 90000000 : 24000000);
    const void *const kern = kernel_for(h->dtype, h->stride, v, ahead);
    // Pieces of an image's rows: a piece loads (and at stride 1 adds up) two rows besides its own and costs
    // about two more to start, so pieces want to be long; but the blocks run in waves of what the GPU holds,
    // and one that is partly filled costs as much as a full one.
    const int64_t columns = (int64_t)n * P.strips * P.cvs;
    const int at_once = resident_blocks(kern, h->device);
    double best = 1e30;
    auto weigh = [&](int rows) {
        const int segs = (ho + rows - 1) / rows;
        rows = (ho + segs - 1) / segs;
        const int64_t waves = ((columns * segs + 127) / 128 + at_once - 1) / at_once;
        const double t = (double)waves * (rows + 4);
        if (t < best * 0.999) { best = t; P.segs = segs; P.seg_rows = rows; }
    };
    for (int segs = 1; segs <= 12 && segs <= ho; ++segs) weigh((ho + segs - 1) / segs);
    for (int rows : {8, 6, 4, 3, 2, 1}) if (rows < ho / 12) weigh(rows);
    const int64_t threads = columns * P.segs;
    if (threads > 0x7FFFFFFFLL) return XGEN_ERR_SHAPE;
    P.threads = (unsigned)threads;
    int prev = h->device;
    cudaGetDevice(&prev);
    if (prev != h->device && cudaSetDevice(h->device) != cudaSuccess) return XGEN_ERR_CUDA;
    void *args[] = {&P};
    xgen_status st = XGEN_OK;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((threads + 127) / 128)); cfg.blockDim = dim3(128); cfg.stream = (cudaStream_t)stream;
    // the kernel waits for its predecessor before it touches x or y
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    if (cudaLaunchKernelExC(&cfg, kern, args) != cudaSuccess) {
        cudaGetLastError();
        st = XGEN_ERR_CUDA;
    } else patconv::count_launch();
    if (prev != h->device) cudaSetDevice(prev);
    return st;
}

xgen_status xgen_dwconv_query(const xgen_dwconv_packed *h, int64_t *kernels_surviving) {
    if (!h || !kernels_surviving) return XGEN_ERR_INVALID_ARG;
    *kernels_surviving = h->surviving;
    return XGEN_OK;
}

void xgen_dwconv_free(xgen_dwconv_packed *h) {
    if (!h) return;
    if (h->device >= 0 && h->d_w9) {
        int prev = 0;
        cudaGetDevice(&prev);
        if (cudaSetDevice(h->device) == cudaSuccess) cudaFree(h->d_w9);
        cudaSetDevice(prev);
    }
    delete h;
}

}  // extern "C"
