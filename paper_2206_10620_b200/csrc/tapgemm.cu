// The pattern-pruned convolution and the block-pruned matrix product on the matrix units.
//
// What is left of a pruned layer is 4/9 x (1 - prune rate) of a dense one, but the matrix units
// are 22 times (fp16) to 44 times (int8) the packed-FMA pipe, 4 times in fp32 (six bf16 products), and the
// command stream reaches 20 to 45 % of that, so the layer is run dense (fp32 layers of 512 channels on few
// pixels are faster on the command stream from 88 % of the kernels pruned on, by 10 % at 90): pruned
// weights are zeros of the operand.  0 x infinity is NaN there, so sums that come out infinite or NaN
// are computed anew from the kept weights alone (tap_repair).
//
// The input of a tile with its halo is staged once per group of channels and serves all nine taps:
// in shared memory a tap is only another start address.  A tile is 128 (256) output pixels, either
// 8 wide and 16 (32) high -- a row of 8 pixels is one row group of the operand, the pitch of the
// staged rows the distance of groups -- or a run of the zero-padded raster of all images (rows one
// entry longer than the image, one row of zeros between images), which wastes one column in w + 1
// where 8-pixel columns would waste up to 7.  Measured: the matrix instructions run at full rate (64
// cycles for 128 x 128 x 16) at every shift.  The other choice, one copy-engine load per tap
// (im2col), moves the tile nine times through L2.
//
// fp16 and int8 pixels are rows of 128 bytes of channels, swizzled; the copy engine delivers them
// (zeros outside the image), one copy a tile or one a row; layers whose channels it cannot address
// are gathered by the producer warps.  fp32 goes through the producer warps, which write planes of
// 16 bytes (8 channels) per pixel and part, unswizzled.
//
// A matrix instruction of 128 x 128 x 16 reads 8 KB of shared memory in its 64 cycles, all that
// shared memory delivers; the weights that stream in slow it down.  So where there are two tiles,
// two blocks work as a pair (cta_group::2): each reads its own rows and half of the filters.
//
// fp32: every operand is split into three bf16 parts (8 + 8 + 8 significand bits, the sum is
// exact) and six of the nine products are taken; what is left out is below 2^-24 of the product.
// The matrix unit truncates when it adds to its accumulator (measured: a chain of 288 steps ends
// 1.5e-5 low, one of 9 steps 1.6e-7), so the leading product is accumulated for one stage only
// (at most 18 steps) and then added, rounded, to sums in registers; the five small products have
// an accumulator of their own, where truncation is 2^-8 of that, and are added the same way.  fp16 chains of
// more than 288 steps are cut every 144 (288) and added, rounded, to sums in tensor memory, by instances of
// their own (CUT): 4096 channels of positive terms came out 7.3e-5 low in one chain, 4.2e-6 now; 512 do 8.5e-6.
// (Time of uncut and cut, 32 images of 14x14 x 1024 -> 1024: 90.8, 97.6 us; 4096 rows x 8192 -> 1024: 57.2, 57.3.)
//
// Roles: 8 or 16 epilogue warps (tensor memory -> registers -> y), 6 producer warps (x), one
// warp that issues the matrix instructions, one that fetches weights with tensor copies.  Blocks are
// persistent; a block keeps its range of filters, and where all of its weights fit they are
// fetched once.  Items that would leave the GPU idle share one reduction between the blocks of a
// cluster, which send each other their sums through distributed shared memory and add them in a fixed order.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstring>
#include <mutex>
#include <utility>
#include <vector>

#include "patconv_internal.h"
#include "ptx.cuh"
#include "tapgemm.h"

namespace patconv {

// Epilogue warps wait for tensor memory and y more than they compute: sixteen where the registers
// allow it; fp32 keeps 64 sums a thread, so eight.
__host__ __device__ constexpr int epi_warps(int dt) { return dt == XGEN_F32 ? 8 : 16; }
constexpr int kProdWarps = 6;
__host__ __device__ constexpr int tap_threads(int dt) { return (epi_warps(dt) + kProdWarps + 2) * 32; }
constexpr int kProdThreads = kProdWarps * 32;
constexpr int kMaxA = 6, kMaxB = 36;
constexpr int kTapSmemMax = 232448 - 4096;      // 227 KB less static shared memory
constexpr int kMaxFilterTile = 256;
constexpr int kStagePitch = 20;                 // words of a staged pixel's 16 sums: rows of 16-byte accesses in distinct banks
constexpr int kStageBytes = 32 * kStagePitch * 4;   // a warp's

struct TapParams {
    const void *x; void *y; const void *bias; const void *residual; const float *rq_scale;
    int *status;
    uint32_t wait_us;
    int hold;                                   // testing aid: arrivals that the stages of x wait for beyond their own
    int rq_zero, relu, pool;
    int n, h, w, ho, wo, c_in, c_out;
    int po, pw;                                 // stored extents
    int64_t npix;                               // product: rows of x
    int vh, straddle;                           // virtual rows per image; tiles may cross images
    uint32_t mg_vh, mg_pitch, mg_rows;          // division by these as a multiplication (div_by)
    int raster, pitch, rows, pixels, sub_px;    // staged tile: entries of a row, rows (of a parity), entries; of the second sub-tile
    int segs, nblk, nt, items, splits, per_split, stages, cut;
    int pl, pl_log, plane_pitch;
    int a_stages, a_bytes, b_slots, resident, b_bytes, tap_group;
    int b_off, tab_off, stage_off, sum_off;     // bytes into dynamic shared memory
    int tmem_cols, acc_bufs, staged;
    int tap_start[9];                           // first staged entry of a tap
    const uint8_t *wimg; int w_rows;            // the weight image (TapWeights)
    int tma, row_boxes, a_tx;                        // x comes by tensor copies; a copy per staged row
    int vec_x;                                  // 16-byte pieces of x can be copied as they are
    int vec_y, vec_r, y32;                      // 16-byte (32-byte) pieces of y / the residual can be moved whole
    uint32_t idesc;
};

// Elements of x per 16-byte plane entry (K of one matrix instruction = two planes), bf16 parts, bytes.
// `row_ch`: channels of a 128-byte row.
template <int DT> struct TapTraits;
template <> struct TapTraits<XGEN_F32> { static constexpr int cpp = 8, parts = 3, xb = 4, row_ch = 0; };
// The kernel instances use `taps` 9 or 1 and stride 1 or 2.  Stride 2 keeps four images of the tile, one per
// parity of row and column (even rows: even columns, odd columns; odd rows likewise), each with rows of 9
// and one row more than the tile, so that neighbouring output pixels read neighbouring entries there too.
template <> struct TapTraits<XGEN_F16_F32ACC> { static constexpr int cpp = 8, parts = 1, xb = 2, row_ch = 64; };
template <> struct TapTraits<XGEN_I8_I32> { static constexpr int cpp = 16, parts = 1, xb = 1, row_ch = 128; };

// ---- results -------------------------------------------------------------------
// W sums of adjacent channels of one pixel: bias, residual, activation, in fp32 (int32).
template <int DT, bool FUSED, int W>
__device__ __forceinline__ void tap_affine(const TapParams &P, const uint32_t *s_bias, uint32_t (&v)[W], int pixel,
                                           bool valid, int c0, int n0) {
#pragma unroll
    for (int q = 0; q < W / 4; ++q) {
        const uint4 b = *reinterpret_cast<const uint4 *>(s_bias + (c0 - n0) + 4 * q);
        const uint32_t bb[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
            v[4 * q + i] = DT == XGEN_I8_I32 ? v[4 * q + i] + bb[i]
                                             : __float_as_uint(__uint_as_float(v[4 * q + i]) + __uint_as_float(bb[i]));
    }
    if (FUSED && P.residual && valid) {
        const size_t off = (size_t)pixel * P.c_out + c0;
        if (DT == XGEN_F16_F32ACC) {
            const __half *r = static_cast<const __half *>(P.residual) + off;
            if (P.vec_r && c0 + W <= P.c_out) {
#pragma unroll
                for (int q = 0; q < W / 8; ++q) {
                    const uint4 a = __ldg(reinterpret_cast<const uint4 *>(r) + q);
                    const uint32_t aa[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&aa[i]));
                        v[8 * q + 2 * i] = __float_as_uint(__uint_as_float(v[8 * q + 2 * i]) + f.x);
                        v[8 * q + 2 * i + 1] = __float_as_uint(__uint_as_float(v[8 * q + 2 * i + 1]) + f.y);
                    }
                }
            } else {
#pragma unroll
                for (int i = 0; i < W; ++i)
                    if (c0 + i < P.c_out) v[i] = __float_as_uint(__uint_as_float(v[i]) + __half2float(r[i]));
            }
        } else {
            const uint32_t *r = static_cast<const uint32_t *>(P.residual) + off;
            uint32_t a[W];
            if (P.vec_r && c0 + W <= P.c_out) {
#pragma unroll
                for (int q = 0; q < W / 4; ++q) {
                    const uint4 t = __ldg(reinterpret_cast<const uint4 *>(r) + q);
                    a[4 * q] = t.x; a[4 * q + 1] = t.y; a[4 * q + 2] = t.z; a[4 * q + 3] = t.w;
                }
            } else {
#pragma unroll
                for (int i = 0; i < W; ++i) a[i] = c0 + i < P.c_out ? r[i] : 0u;
            }
#pragma unroll
            for (int i = 0; i < W; ++i)
                v[i] = DT == XGEN_I8_I32 ? v[i] + a[i] : __float_as_uint(__uint_as_float(v[i]) + __uint_as_float(a[i]));
        }
    }
    if (P.relu) {
#pragma unroll
        for (int i = 0; i < W; ++i) {
            if (DT == XGEN_I8_I32) v[i] = (uint32_t)max((int)v[i], 0);
            else {                                  // NaN stays NaN
                float f;
                asm("max.NaN.f32 %0, %1, 0f00000000;" : "=f"(f) : "f"(__uint_as_float(v[i])));
                v[i] = __float_as_uint(f);
            }
        }
    }
}

template <int DT> __device__ __forceinline__ uint32_t tap_max(uint32_t a, uint32_t b) {
    if (DT == XGEN_I8_I32) return (uint32_t)max((int)a, (int)b);
    float f;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(f) : "f"(__uint_as_float(a)), "f"(__uint_as_float(b)));
    return __float_as_uint(f);
}

// Re-quantisation of an int32 result: scaled, rounded, zero point added (saturating); then clamped to uint8.
__device__ __forceinline__ int tap_level(const TapParams &P, uint32_t v, float scale) {
    int r;
    asm("add.sat.s32 %0, %1, %2;" : "=r"(r) : "r"(__float2int_rn(__fmul_rn((float)(int)v, scale))), "r"(P.rq_zero));
    return r;
}
__device__ __forceinline__ uint32_t tap_code(const TapParams &P, uint32_t v, float scale) {
    return (uint32_t)max(min(tap_level(P, v, scale), 255), 0);
}
__device__ __forceinline__ uint32_t pack_codes(int a, int b, int c, int d) {
    uint32_t hi, r;
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, 0;" : "=r"(hi) : "r"(d), "r"(c));
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(b), "r"(a), "r"(hi));
    return r;
}
// Two fp32 additions (the packed instruction rounds each like the scalar one).
__device__ __forceinline__ void add2(uint32_t &a0, uint32_t &a1, uint32_t b0, uint32_t b1) {
    asm("{\n .reg .b64 a, b;\n mov.b64 a, {%0, %1};\n mov.b64 b, {%2, %3};\n add.rn.f32x2 a, a, b;\n mov.b64 {%0, %1}, a;\n}"
        : "+r"(a0), "+r"(a1) : "r"(b0), "r"(b1));
}

// (a0, a1) stays 0 while (v0, v1) is finite, and is NaN for good once it is not.
__device__ __forceinline__ void nan_of(uint32_t &a0, uint32_t &a1, uint32_t v0, uint32_t v1) {
    asm("{\n .reg .b64 a, v;\n mov.b64 a, {%0, %1};\n mov.b64 v, {%2, %3};\n fma.rn.f32x2 a, v, %4, a;\n mov.b64 {%0, %1}, a;\n}"
        : "+r"(a0), "+r"(a1) : "r"(v0), "r"(v1), "l"(0ull));
}

// Store W results of one pixel, converted; whole 16- or 32-byte pieces where the tensor allows it.
template <int DT, bool FUSED, int W>
__device__ __forceinline__ void tap_store(const TapParams &P, const float *s_scale, const uint32_t (&v)[W], int pixel,
                                          int c0, int n0) {
    const size_t off = (size_t)pixel * P.c_out + c0;
    const bool full = c0 + W <= P.c_out;
    if (FUSED && DT == XGEN_I8_I32 && P.rq_scale) {
        uint32_t code[W / 4];
#pragma unroll
        for (int q = 0; q < W / 4; ++q) {
            code[q] = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) code[q] |= tap_code(P, v[4 * q + i], s_scale[c0 - n0 + 4 * q + i]) << (8 * i);
        }
        uint8_t *y = static_cast<uint8_t *>(P.y) + off;
        if (full && P.vec_y) {
            if (W == 16) *reinterpret_cast<uint4 *>(y) = make_uint4(code[0], code[1], code[W / 4 - 2], code[W / 4 - 1]);
            else *reinterpret_cast<uint2 *>(y) = make_uint2(code[0], code[1]);
        } else {
#pragma unroll
            for (int i = 0; i < W; ++i) if (c0 + i < P.c_out) y[i] = (uint8_t)(code[i / 4] >> (8 * (i % 4)));
        }
        return;
    }
    constexpr int NW = DT == XGEN_F16_F32ACC ? W / 2 : W;
    uint32_t o[NW];
    if (DT == XGEN_F16_F32ACC) {
#pragma unroll
        for (int i = 0; i < NW; ++i) {
            const __half2 h = __floats2half2_rn(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
            o[i] = *reinterpret_cast<const uint32_t *>(&h);
        }
    } else {
#pragma unroll
        for (int i = 0; i < NW; ++i) o[i] = v[i];
    }
    if (full && P.vec_y) {
        uint32_t *y = reinterpret_cast<uint32_t *>(static_cast<char *>(P.y) + off * (DT == XGEN_F16_F32ACC ? 2 : 4));
        if (P.y32 && NW >= 8) {
#pragma unroll
            for (int q = 0; q < NW / 8; ++q)
                asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                             ::"l"(y + 8 * q), "r"(o[8 * q]), "r"(o[8 * q + 1]), "r"(o[8 * q + 2]), "r"(o[8 * q + 3]),
                               "r"(o[8 * q + 4]), "r"(o[8 * q + 5]), "r"(o[8 * q + 6]), "r"(o[8 * q + 7]) : "memory");
        } else {
#pragma unroll
            for (int q = 0; q < NW / 4; ++q)
                reinterpret_cast<uint4 *>(y)[q] = make_uint4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
        }
    } else if (DT == XGEN_F16_F32ACC) {
        unsigned short *y = static_cast<unsigned short *>(P.y) + off;
#pragma unroll
        for (int i = 0; i < W; ++i)
            if (c0 + i < P.c_out) y[i] = (unsigned short)(o[i / 2] >> (16 * (i % 2)));
    } else {
        uint32_t *y = static_cast<uint32_t *>(P.y) + off;
#pragma unroll
        for (int i = 0; i < W; ++i)
            if (c0 + i < P.c_out) y[i] = v[i];
    }
}

// One result, for tensors whose rows are not whole 16-byte pieces.
template <int DT, bool FUSED>
__device__ __forceinline__ uint32_t tap_affine1(const TapParams &P, uint32_t bias, uint32_t v, size_t off) {
    v = DT == XGEN_I8_I32 ? v + bias : __float_as_uint(__uint_as_float(v) + __uint_as_float(bias));
    if (FUSED && P.residual) {
        if (DT == XGEN_I8_I32) v += static_cast<const uint32_t *>(P.residual)[off];
        else if (DT == XGEN_F32) v = __float_as_uint(__uint_as_float(v) + static_cast<const float *>(P.residual)[off]);
        else v = __float_as_uint(__uint_as_float(v) + __half2float(static_cast<const __half *>(P.residual)[off]));
    }
    return P.relu ? tap_max<DT>(v, 0u) : v;
}
template <int DT, bool FUSED>
__device__ __forceinline__ void tap_store1(const TapParams &P, float scale, uint32_t v, size_t off) {
    if (FUSED && DT == XGEN_I8_I32 && P.rq_scale) static_cast<uint8_t *>(P.y)[off] = (uint8_t)tap_code(P, v, scale);
    else if (DT == XGEN_F16_F32ACC) static_cast<__half *>(P.y)[off] = __float2half_rn(__uint_as_float(v));
    else static_cast<uint32_t *>(P.y)[off] = v;
}

// A warp's 32 pixels x 16 channels, staged as rows of kStagePitch words: 16 sums, the pixel of the
// unpooled result (-1: none), where it is stored (pooled: the window whose first pixel it is).  Finish
// and store them so that neighbouring lanes hold neighbouring elements: where a residual is read (its
// 16-byte loads by lanes of different pixels touched 32 lines each, 11000 cycles for 128 x 128), and where
// rows of y are not whole 16-byte pieces.
template <int DT, bool FUSED>
__device__ __forceinline__ void tap_emit(const TapParams &P, const uint32_t *st, const uint32_t *s_bias, const float *s_scale,
                                         int c_base, int n0, int lane) {
    const bool pool = FUSED && P.pool;
    if constexpr (FUSED) if (P.vec_y && P.vec_r && !pool) {
        const int c = c_base + (lane & 3) * 4;
        if (c >= P.c_out) return;
        const uint4 b = *reinterpret_cast<const uint4 *>(s_bias + (c - n0));
        const float4 sc = *reinterpret_cast<const float4 *>(s_scale + (c - n0));
        const uint32_t *const row0 = st + (lane >> 2) * kStagePitch;
        uint4 res[4];
        int px[4];
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            px[it] = (int)row0[it * 8 * kStagePitch + 16];
            const size_t off = (size_t)max(px[it], 0) * P.c_out + c;
            if (DT == XGEN_F16_F32ACC) {
                const uint2 r = __ldg(reinterpret_cast<const uint2 *>(static_cast<const __half *>(P.residual) + off));
                const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&r.x)), g = __half22float2(*reinterpret_cast<const __half2 *>(&r.y));
                res[it] = make_uint4(__float_as_uint(f.x), __float_as_uint(f.y), __float_as_uint(g.x), __float_as_uint(g.y));
            } else res[it] = __ldg(reinterpret_cast<const uint4 *>(static_cast<const uint32_t *>(P.residual) + off));
        }
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            const uint4 a = *reinterpret_cast<const uint4 *>(row0 + it * 8 * kStagePitch + (lane & 3) * 4);
            uint32_t v[4] = {a.x, a.y, a.z, a.w};
            if (DT == XGEN_I8_I32) { v[0] += b.x + res[it].x; v[1] += b.y + res[it].y; v[2] += b.z + res[it].z; v[3] += b.w + res[it].w; }
            else {
                add2(v[0], v[1], b.x, b.y); add2(v[2], v[3], b.z, b.w);
                add2(v[0], v[1], res[it].x, res[it].y); add2(v[2], v[3], res[it].z, res[it].w);
            }
            if (P.relu) {
#pragma unroll
                for (int i = 0; i < 4; ++i) v[i] = tap_max<DT>(v[i], 0u);
            }
            if (px[it] < 0) continue;
            const size_t off = (size_t)px[it] * P.c_out + c;
            if (DT == XGEN_I8_I32 && P.rq_scale)
                *reinterpret_cast<uint32_t *>(static_cast<uint8_t *>(P.y) + off) =
                    pack_codes(tap_level(P, v[0], sc.x), tap_level(P, v[1], sc.y), tap_level(P, v[2], sc.z), tap_level(P, v[3], sc.w));
            else if (DT == XGEN_F16_F32ACC) {
                const __half2 f = __floats2half2_rn(__uint_as_float(v[0]), __uint_as_float(v[1])), g = __floats2half2_rn(__uint_as_float(v[2]), __uint_as_float(v[3]));
                *reinterpret_cast<uint2 *>(static_cast<__half *>(P.y) + off) = make_uint2(*reinterpret_cast<const uint32_t *>(&f), *reinterpret_cast<const uint32_t *>(&g));
            } else *reinterpret_cast<uint4 *>(static_cast<uint32_t *>(P.y) + off) = make_uint4(v[0], v[1], v[2], v[3]);
        }
        return;
    }
    const int c = c_base + (lane & 15);          // a lane keeps its channel, half-warps take a pixel each
    if (c >= P.c_out) return;
    const uint32_t bias = s_bias[c - n0];
    const float scale = FUSED ? s_scale[c - n0] : 0.0f;
    if (!pool && !(FUSED && P.residual)) {
#pragma unroll 4
        for (int it = 0; it < 16; ++it) {
            const uint32_t *const row = st + (2 * it + (lane >> 4)) * kStagePitch;
            const int px = (int)row[16];
            if (px >= 0) {
                const size_t off = (size_t)px * P.c_out + c;
                tap_store1<DT, FUSED>(P, scale, tap_affine1<DT, false>(P, bias, row[lane & 15], off), off);
            }
        }
        return;
    }
    if constexpr (FUSED) if (!pool) {
        // eight residuals asked for at a time: one by one, 24 images of 32 x 74 x 58 fp32 channels took
        // 52 us (25 now)
#pragma unroll 1
        for (int it = 0; it < 16; it += 8) {
            const uint32_t *const row0 = st + (2 * it + (lane >> 4)) * kStagePitch;
            int px[8];
            uint32_t res[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                px[i] = (int)row0[2 * i * kStagePitch + 16];
                const size_t off = (size_t)max(px[i], 0) * P.c_out + c;
                if (DT == XGEN_F16_F32ACC) res[i] = __ldg(static_cast<const unsigned short *>(P.residual) + off);
                else res[i] = __ldg(static_cast<const uint32_t *>(P.residual) + off);
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                uint32_t v = row0[2 * i * kStagePitch + (lane & 15)];
                if (DT == XGEN_I8_I32) v += bias + res[i];
                else {
                    const float r = DT == XGEN_F16_F32ACC ? __half2float(__ushort_as_half((unsigned short)res[i])) : __uint_as_float(res[i]);
                    v = __float_as_uint(__uint_as_float(v) + __uint_as_float(bias) + r);
                }
                if (P.relu) v = tap_max<DT>(v, 0u);
                if (px[i] >= 0) tap_store1<DT, FUSED>(P, scale, v, (size_t)px[i] * P.c_out + c);
            }
        }
        return;
    }
    if constexpr (FUSED) {
        // pooled: all sixteen residuals of a lane's four windows asked for before the first is used
        uint32_t res[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int jp = 2 * (i >> 2) + (lane >> 4), q = i & 3;
            const int px = (int)st[((jp >> 2) * 16 + (jp & 3) * 2 + (q & 1) + (q >> 1) * 8) * kStagePitch + 16];
            res[i] = 0u;
            if (P.residual) {
                const size_t off = (size_t)max(px, 0) * P.c_out + c;
                if (DT == XGEN_F16_F32ACC) res[i] = __float_as_uint(__half2float(__ushort_as_half(__ldg(static_cast<const unsigned short *>(P.residual) + off))));
                else res[i] = __ldg(static_cast<const uint32_t *>(P.residual) + off);
            }
        }
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            const int jp = 2 * it + (lane >> 4);
            const uint32_t *const row = st + ((jp >> 2) * 16 + (jp & 3) * 2) * kStagePitch;
            if ((int)row[16] < 0) continue;
            uint32_t best = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t v = row[((q & 1) + (q >> 1) * 8) * kStagePitch + (lane & 15)];
                if (DT == XGEN_I8_I32) v += bias + res[4 * it + q];
                else v = __float_as_uint(__uint_as_float(v) + __uint_as_float(bias) + __uint_as_float(res[4 * it + q]));
                if (P.relu) v = tap_max<DT>(v, 0u);
                best = q == 0 ? v : tap_max<DT>(best, v);
            }
            tap_store1<DT, FUSED>(P, scale, best, (size_t)(int)row[17] * P.c_out + c);
        }
    }
}

// 32 sums of one pixel, from channel c0 on, finished and stored by their own lane: 64 to 128 bytes in
// whole sectors.
template <int DT, bool FUSED>
__device__ __forceinline__ void tap_direct(const TapParams &P, const uint32_t *s_bias, const float *s_scale, uint32_t (&v)[32],
                                           int pix, int out, int c0, int n0) {
    if (FUSED && P.pool) {
        // The four lanes of a 2x2 window share its 32 channels out among them: each sends what the other
        // needs, 16 and then 8 words, and finishes 8 channels of the pooled pixel.
        const bool late = P.residual == nullptr;             // bias and activation commute with the maximum
        if (!late) {
#pragma unroll 1
            for (int g = 0; g < 4; ++g) {
                uint32_t w[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) w[i] = g == 0 ? v[i] : g == 1 ? v[8 + i] : g == 2 ? v[16 + i] : v[24 + i];
                if (pix >= 0 && c0 + 8 * g < P.c_out) tap_affine<DT, FUSED, 8>(P, s_bias, w, pix, true, c0 + 8 * g, n0);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    if (g == 0) v[i] = w[i]; else if (g == 1) v[8 + i] = w[i]; else if (g == 2) v[16 + i] = w[i]; else v[24 + i] = w[i];
                }
            }
        }
        const bool odd_x = threadIdx.x & 1, odd_y = threadIdx.x & 8;
        uint32_t w[8];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const uint32_t got = __shfl_xor_sync(0xFFFFFFFFu, odd_x ? v[i] : v[16 + i], 1);
            v[i] = tap_max<DT>(odd_x ? v[16 + i] : v[i], got);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t got = __shfl_xor_sync(0xFFFFFFFFu, odd_y ? v[i] : v[8 + i], 8);
            w[i] = tap_max<DT>(odd_y ? v[8 + i] : v[i], got);
        }
        const int c = c0 + (odd_x ? 16 : 0) + (odd_y ? 8 : 0);
        if (pix < 0 || c >= P.c_out) return;
        if (late) tap_affine<DT, FUSED, 8>(P, s_bias, w, pix, false, c, n0);
        tap_store<DT, FUSED, 8>(P, s_scale, w, out, c, n0);
        return;
    }
    if (pix < 0) return;
    if (c0 + 32 > P.c_out || !P.vec_y) {
#pragma unroll 1
        for (int g = 0; g < 4; ++g) {
            if (c0 + 8 * g >= P.c_out) break;
            uint32_t w[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) w[i] = g == 0 ? v[i] : g == 1 ? v[8 + i] : g == 2 ? v[16 + i] : v[24 + i];
            tap_affine<DT, FUSED, 8>(P, s_bias, w, pix, true, c0 + 8 * g, n0);
            tap_store<DT, FUSED, 8>(P, s_scale, w, pix, c0 + 8 * g, n0);
        }
        return;
    }
    const size_t off = (size_t)pix * P.c_out + c0;
    const uint32_t *const bias = s_bias + (c0 - n0);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const uint4 b = *reinterpret_cast<const uint4 *>(bias + 4 * q);
        if (DT == XGEN_I8_I32) { v[4 * q] += b.x; v[4 * q + 1] += b.y; v[4 * q + 2] += b.z; v[4 * q + 3] += b.w; }
        else { add2(v[4 * q], v[4 * q + 1], b.x, b.y); add2(v[4 * q + 2], v[4 * q + 3], b.z, b.w); }
    }
    if (FUSED && P.residual) {
        if (!P.vec_r) {
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = tap_affine1<DT, FUSED>(P, 0u, v[i], off + i);
        } else if (DT == XGEN_F16_F32ACC) {
            const uint4 *r = reinterpret_cast<const uint4 *>(static_cast<const __half *>(P.residual) + off);
            uint4 a[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) a[q] = __ldg(r + q);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t aa[4] = {a[q].x, a[q].y, a[q].z, a[q].w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&aa[i]));
                    add2(v[8 * q + 2 * i], v[8 * q + 2 * i + 1], __float_as_uint(f.x), __float_as_uint(f.y));
                }
            }
        } else {
            const uint4 *r = reinterpret_cast<const uint4 *>(static_cast<const uint32_t *>(P.residual) + off);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint4 a[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) a[q] = __ldg(r + 4 * h + q);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    uint32_t *const w = v + 16 * h + 4 * q;
                    if (DT == XGEN_I8_I32) { w[0] += a[q].x; w[1] += a[q].y; w[2] += a[q].z; w[3] += a[q].w; }
                    else { add2(w[0], w[1], a[q].x, a[q].y); add2(w[2], w[3], a[q].z, a[q].w); }
                }
            }
        }
    }
    if (P.relu) {
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = tap_max<DT>(v[i], 0u);
    }
    if (FUSED && DT == XGEN_I8_I32 && P.rq_scale) {
        uint8_t *const y = static_cast<uint8_t *>(P.y) + off;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t code[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 sc = *reinterpret_cast<const float4 *>(s_scale + (c0 - n0) + 16 * h + 4 * q);
                const uint32_t *const w = v + 16 * h + 4 * q;
                code[q] = pack_codes(tap_level(P, w[0], sc.x), tap_level(P, w[1], sc.y), tap_level(P, w[2], sc.z), tap_level(P, w[3], sc.w));
            }
            *reinterpret_cast<uint4 *>(y + 16 * h) = make_uint4(code[0], code[1], code[2], code[3]);
        }
        return;
    }
    constexpr int NW = DT == XGEN_F16_F32ACC ? 16 : 32;
    uint32_t *const y = reinterpret_cast<uint32_t *>(static_cast<char *>(P.y) + off * (DT == XGEN_F16_F32ACC ? 2 : 4));
    if (DT == XGEN_F16_F32ACC) {
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const __half2 h = __floats2half2_rn(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
            v[i] = *reinterpret_cast<const uint32_t *>(&h);
        }
    }
    if (P.y32) {
#pragma unroll
        for (int q = 0; q < NW / 8; ++q)
            asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                         ::"l"(y + 8 * q), "r"(v[8 * q]), "r"(v[8 * q + 1]), "r"(v[8 * q + 2]), "r"(v[8 * q + 3]),
                           "r"(v[8 * q + 4]), "r"(v[8 * q + 5]), "r"(v[8 * q + 6]), "r"(v[8 * q + 7]) : "memory");
    } else {
#pragma unroll
        for (int q = 0; q < NW / 4; ++q)
            reinterpret_cast<uint4 *>(y)[q] = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    }
}

// ---- operands ------------------------------------------------------------------
// fp32 -> three bf16 parts.  The first is clamped to the largest bf16 so that a finite value never
// becomes an infinity; the parts of an infinity or NaN hold a NaN, so that every sum they go into does.
__device__ __forceinline__ void split3(const float (&a)[8], uint4 &p0, uint4 &p1, uint4 &p2) {
    const float big = __uint_as_float(0x7F7F0000u);
    uint32_t o[3][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float x = a[2 * i], y = a[2 * i + 1];
        __nv_bfloat162 h = __floats2bfloat162_rn(fminf(fmaxf(x, -big), big), fminf(fmaxf(y, -big), big));
        o[0][i] = *reinterpret_cast<uint32_t *>(&h);
#pragma unroll
        for (int k = 1; k < 3; ++k) {
            x -= __uint_as_float(o[k - 1][i] << 16);
            y -= __uint_as_float(o[k - 1][i] & 0xFFFF0000u);
            h = __floats2bfloat162_rn(x, y);
            o[k][i] = *reinterpret_cast<uint32_t *>(&h);
        }
    }
    p0 = make_uint4(o[0][0], o[0][1], o[0][2], o[0][3]);
    p1 = make_uint4(o[1][0], o[1][1], o[1][2], o[1][3]);
    p2 = make_uint4(o[2][0], o[2][1], o[2][2], o[2][3]);
}

// 16 bytes from any address, bytes beyond `valid` zero: aligned words, shifted into place.  Only
// words that hold at least one wanted byte are read.
__device__ __forceinline__ uint4 gather16(const char *src, int valid) {
    if (valid <= 0) return make_uint4(0, 0, 0, 0);
    const uintptr_t a = reinterpret_cast<uintptr_t>(src);
    const uint32_t *w = reinterpret_cast<const uint32_t *>(a & ~(uintptr_t)3);
    const int lead = (int)(a & 3), nbytes = min(valid, 16), words = (lead + nbytes + 3) / 4;
    uint32_t in[5], o[4];
#pragma unroll
    for (int i = 0; i < 5; ++i) in[i] = i < words ? __ldg(w + i) : 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        o[i] = __funnelshift_r(in[i], in[i + 1], 8 * lead);
        const int left = nbytes - 4 * i;                       // wanted bytes of this word
        if (left < 4) o[i] = left <= 0 ? 0u : (o[i] & ((1u << (8 * left)) - 1u));
    }
    return make_uint4(o[0], o[1], o[2], o[3]);
}

__device__ __forceinline__ void sts128(uint32_t dst, const uint4 &v) {
    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(dst), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// n / d with the host's multiplier (0: a range for which none is exact).
__device__ __forceinline__ int div_by(int n, int d, uint32_t mg) { return mg ? (int)__umulhi((uint32_t)n, mg) : n / d; }

// Position of a block's work: item = (tile or pair of tiles, range of filters).  The second tile of the
// last pair may lie past the end: all of its pixels are invalid.
struct TapItem {
    int n0;                  // first filter
    int v0, ox0;             // 8-pixel columns: first virtual row, first column; raster: row and column of entry q0
    int q0;                  // raster: first output entry
};
template <int MT, bool PAIR> __device__ __forceinline__ TapItem tap_item(const TapParams &P, int item, int side) {
    TapItem t;
    int tile = item / P.nblk;
    t.n0 = (item - tile * P.nblk) * P.nt;
    if (PAIR) tile = 2 * tile + side;
    if (P.raster) {
        t.q0 = tile * 128 * MT;
        t.v0 = div_by(t.q0, P.pitch, P.mg_pitch);
        t.ox0 = t.q0 - t.v0 * P.pitch;
    } else {
        const int rt = tile / P.segs;
        t.q0 = 0;
        t.ox0 = (tile - rt * P.segs) * 8;
        t.v0 = rt * 16 * MT;
    }
    return t;
}

// Image and input row of staged row `i` (stride 2: i of the parity `odd`); outside the tensor for zeros.
struct TapRow { int img, y; };
template <int STRIDE> __device__ __forceinline__ TapRow tap_row(const TapParams &P, const TapItem &t, int i, int odd) {
    TapRow r;
    const int step = STRIDE == 1 ? i - 1 : i;                       // output rows from the tile's first
    if (P.straddle) {
        const int v = t.v0 + step;
        if (v < 0) return TapRow{0, -1};
        r.img = div_by(v, P.vh, P.mg_vh);
        r.y = v - r.img * P.vh;
    } else {
        r.img = div_by(t.v0, P.vh, P.mg_vh);
        r.y = t.v0 - r.img * P.vh + step;
    }
    if (STRIDE == 2) r.y = 2 * r.y - odd;
    return r;
}

// x's pixel of staged entry p, or -1 for zeros.
template <int STRIDE, int TAPS> __device__ __forceinline__ int tap_source(const TapParams &P, const TapItem &t, int p) {
    if (TAPS == 1) return (int64_t)t.v0 * 8 + p < P.npix ? t.v0 * 8 + p : -1;
    if (P.raster) p -= P.pitch - 1 - t.ox0;       // (all tiles keep their first output entry at the same place)
    if (p < 0) return -1;
    int i = div_by(p, P.pitch, P.mg_pitch), ix = p - i * P.pitch, odd = 0;
    if (STRIDE == 1) ix += (P.raster ? 0 : t.ox0) - 1;
    else {
        const int region = div_by(i, P.rows, P.mg_rows);
        i -= region * P.rows;
        odd = region >> 1;
        ix = 2 * (t.ox0 + ix) - (region & 1);
    }
    const TapRow r = tap_row<STRIDE>(P, t, i, odd);
    const bool in = r.img < P.n && (unsigned)r.y < (unsigned)P.h && (unsigned)ix < (unsigned)P.w;
    return in ? (r.img * P.h + r.y) * P.w + ix : -1;
}

// Output pixel `m` (0 .. 128 MT - 1) of a tile: of the unpooled result, and where it is stored; -1 if none.
struct TapPixel { int pix, out; };
template <int TAPS> __device__ __forceinline__ TapPixel tap_pixel(const TapParams &P, const TapItem &t, int m) {
    if (TAPS == 1) {
        const int p = (int64_t)t.v0 * 8 + m < P.npix ? t.v0 * 8 + m : -1;
        return TapPixel{p, p};
    }
    int v, ox;
    if (P.raster) {
        v = div_by(t.q0 + m, P.pitch, P.mg_pitch);
        ox = t.q0 + m - v * P.pitch;
    } else {
        v = t.v0 + (m >> 3);
        ox = t.ox0 + (m & 7);
    }
    const int img = div_by(v, P.vh, P.mg_vh), oy = v - img * P.vh;
    if (img >= P.n || oy >= P.ho || ox >= P.wo) return TapPixel{-1, -1};
    const int pix = (img * P.ho + oy) * P.wo + ox;
    return TapPixel{pix, P.pool ? (img * P.po + oy / 2) * P.pw + ox / 2 : pix};
}

// ---- sums that are not finite -----------------------------------------------------
// The matrix units multiply pruned weights too, as zeros, so an infinity or NaN of x reaches every
// filter there, and in fp32 the parts of an infinity do not add up to one.  Every such sum is infinite or
// NaN (an overflow of finite operands as well), and the layer's own value takes its place: the kept
// weights of the filter, in fp32, in the order of the image, where kept zeros are -0.  A lane goes through the
// weights of four adjacent filters from end to end, lanes side by side over their pixels.
__device__ __forceinline__ uint32_t half_of(const uint4 &a, int e) {
    const uint32_t w = e / 2 == 0 ? a.x : e / 2 == 1 ? a.y : e / 2 == 2 ? a.z : a.w;
    return w >> (16 * (e % 2)) & 0xFFFFu;
}
template <int DT, int STRIDE, int TAPS>
__device__ __noinline__ uint4 tap_anew(const TapParams &P, int pix, int oc) {
    constexpr int cpp = TapTraits<DT>::cpp, parts = TapTraits<DT>::parts;
    int img = 0, oy = 0, ox = 0;
    if (TAPS == 9) {
        const int row = pix / P.wo;
        ox = pix - row * P.wo;
        img = row / P.ho;
        oy = row - img * P.ho;
    }
    const size_t part = (size_t)P.w_rows * 16, step = part * parts;
    const uint8_t *w = P.wimg + (size_t)oc * 16;
    float sum[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 1
    for (int c = 0; c < P.c_in; c += cpp) {
#pragma unroll (DT == XGEN_F32 || TAPS == 1 ? 1 : 3)
        for (int t = 0; t < TAPS; ++t, w += step) {
            const uint4 z = make_uint4(0, 0, 0, 0);
            const int iy = TAPS == 9 ? oy * STRIDE + t / 3 - 1 : 0, ix = TAPS == 9 ? ox * STRIDE + t % 3 - 1 : 0;
            const bool in = TAPS == 1 || ((unsigned)iy < (unsigned)P.h && (unsigned)ix < (unsigned)P.w);
            const size_t at = (TAPS == 9 ? ((size_t)img * P.h + iy) * P.w + ix : (size_t)pix) * P.c_in + c;
            uint4 a[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) a[j] = __ldg(reinterpret_cast<const uint4 *>(w) + j);
            float x8[8];                          // zeros outside the image
            if (DT == XGEN_F32) {
#pragma unroll
                for (int e = 0; e < 8; ++e) x8[e] = in && c + e < P.c_in ? __ldg(static_cast<const float *>(P.x) + at + e) : 0.0f;
            } else {
                const unsigned short *const x = static_cast<const unsigned short *>(P.x) + at;
                if (P.vec_x) {
                    const uint4 q = in ? __ldg(reinterpret_cast<const uint4 *>(x)) : z;
#pragma unroll
                    for (int e = 0; e < 8; ++e) x8[e] = __half2float(__ushort_as_half((unsigned short)half_of(q, e)));
                } else {
#pragma unroll
                    for (int e = 0; e < 8; ++e) x8[e] = in && c + e < P.c_in ? __half2float(__ushort_as_half(__ldg(x + e))) : 0.0f;
                }
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                uint4 b1 = z, b2 = z;
                if (DT == XGEN_F32) {
                    b1 = __ldg(reinterpret_cast<const uint4 *>(w + part) + j);
                    b2 = __ldg(reinterpret_cast<const uint4 *>(w + 2 * part) + j);
                }
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const uint32_t bits = half_of(a[j], e);
                    const float wv = DT == XGEN_F32 ? __uint_as_float(bits << 16) + (__uint_as_float(half_of(b1, e) << 16) + __uint_as_float(half_of(b2, e) << 16))
                                                    : __half2float(__ushort_as_half((unsigned short)bits));      // (exact)
                    if (bits) sum[j] = fmaf(wv, x8[e], sum[j]);                 // (0: pruned)
                }
            }
        }
        const float all = sum[0] * sum[1] * sum[2] * sum[3];
        if (all != all && sum[0] != sum[0] && sum[1] != sum[1] && sum[2] != sum[2] && sum[3] != sum[3]) break;
    }
    return make_uint4(__float_as_uint(sum[0]), __float_as_uint(sum[1]), __float_as_uint(sum[2]), __float_as_uint(sum[3]));
}
template <int N> __device__ __forceinline__ bool all_finite(const uint32_t (&v)[N]) {
    uint32_t a0 = 0u, a1 = 0u, b0 = 0u, b1 = 0u;
#pragma unroll
    for (int i = 0; i < N; i += 4) {
        nan_of(a0, a1, v[i], v[i + 1]);
        nan_of(b0, b1, v[i + 2], v[i + 3]);
    }
    return __uint_as_float(a0) + __uint_as_float(a1) + (__uint_as_float(b0) + __uint_as_float(b1)) == 0.0f;
}
// All threads of a block, for what the block has stored: threads side by side over four filters each.
template <int DT, int STRIDE, int TAPS, int MT, bool PAIR>
__device__ __noinline__ void tap_repair(const TapParams &P) {
    // (the block's place anew: nothing need be kept for this until the end)
    const unsigned csize = (PAIR ? 2 : 1) * P.splits, crank = blockIdx.x % csize;
    const int side = PAIR ? (int)crank & 1 : 0, rank = (int)crank / (PAIR ? 2 : 1);
    const int item0 = (int)(blockIdx.x / csize), item_step = P.splits > 1 ? P.items : (int)(gridDim.x / csize);
    const int groups = P.nt / 4;
    const bool pool = TAPS == 9 && P.pool;
#pragma unroll 1
    for (int item = item0; item < P.items; item += item_step) {
        const TapItem t = tap_item<MT, PAIR>(P, item, side);
#pragma unroll 1
        for (int i = threadIdx.x; i < 128 * MT * groups; i += tap_threads(DT)) {
            const int m = i / groups, c = t.n0 + (i - m * groups) * 4;
            const TapPixel at = tap_pixel<TAPS>(P, t, m);
            if (at.pix < 0 || c >= P.c_out || (P.splits > 1 && m / 16 % P.splits != rank)) continue;
            if (pool && ((at.pix / P.wo % P.ho | at.pix % P.wo) & 1)) continue;              // (a window is its first pixel's)
            const size_t off = (size_t)at.out * P.c_out + c;
            bool odd[4], any = false;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                odd[j] = c + j < P.c_out &&
                         (DT == XGEN_F32 ? (static_cast<const volatile uint32_t *>(P.y)[off + j] & 0x7F800000u) == 0x7F800000u
                                         : (static_cast<const volatile unsigned short *>(P.y)[off + j] & 0x7C00u) == 0x7C00u);
                any |= odd[j];
            }
            if (!any) continue;
            uint32_t best[4] = {0u, 0u, 0u, 0u};
#pragma unroll 1
            for (int q = 0; q < (pool ? 4 : 1); ++q) {
                const int pix = at.pix + (q & 1) + (q >> 1) * P.wo;
                const uint4 s4 = tap_anew<DT, STRIDE, TAPS>(P, pix, c);
                const uint32_t s[4] = {s4.x, s4.y, s4.z, s4.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (!odd[j]) continue;
                    const uint32_t v = tap_affine1<DT, TAPS == 9>(P, P.bias ? static_cast<const uint32_t *>(P.bias)[c + j] : 0u, s[j],
                                                                  (size_t)pix * P.c_out + c + j);
                    best[j] = q == 0 ? v : tap_max<DT>(best[j], v);
                }
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (odd[j]) tap_store1<DT, TAPS == 9>(P, 0.0f, best[j], off + j);
        }
    }
}

template <int DT, int STRIDE, int TAPS, int MT, bool PAIR, bool CUT>
__global__ void __launch_bounds__(tap_threads(DT), 1)
tap_kernel(const __grid_constant__ TapParams P, const __grid_constant__ CUtensorMap wmap, const __grid_constant__ CUtensorMap xmap) {
    using T = TapTraits<DT>;
    constexpr int PARTS = T::parts;
    constexpr bool kF32 = DT == XGEN_F32, FUSED = TAPS == 9;
    constexpr int kEpiWarps = epi_warps(DT);
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    __shared__ int s_odd;                        // a sum has come out infinite or NaN
    __shared__ volatile int s_started;           // items whose x is being fetched
    __shared__ __align__(8) uint64_t s_bars[2 * kMaxA + 2 * kMaxB + 5];
    __shared__ __align__(16) uint32_t s_bias[kMaxFilterTile];
    __shared__ __align__(16) float s_scale[kMaxFilterTile];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t sbase = smem_u32(smem), bars = smem_u32(s_bars);
    auto a_full = [&](int s) { return bars + 8u * s; };
    auto a_empty = [&](int s) { return bars + 8u * (kMaxA + s); };
    auto b_full = [&](int s) { return bars + 8u * (2 * kMaxA + s); };
    auto b_empty = [&](int s) { return bars + 8u * (2 * kMaxA + kMaxB + s); };
    auto acc_full = [&](int s) { return bars + 8u * (2 * kMaxA + 2 * kMaxB + s); };
    auto acc_empty = [&](int s) { return bars + 8u * (2 * kMaxA + 2 * kMaxB + 2 + s); };
    const uint32_t all_done = bars + 8u * (2 * kMaxA + 2 * kMaxB + 4);
    // Nothing is steered by what a wait says: lanes of a warp and warps of a role may see it give up at different
    // places and would part, ahead of a barrier or an instruction that takes them all.  A launch that gave up goes
    // through all of its work, on whatever the buffers hold, and is reported.
    auto wait = [&](uint32_t bar, uint32_t parity) { mbar_wait<PAIR>(bar, parity, &s_abort, P.status, P.wait_us); };
    auto wait_warp = [&](uint32_t bar, uint32_t parity) { wait(bar, parity); __syncwarp(); };
    // Clusters: a pair of blocks (PAIR), or the blocks (pairs) that split an item's reduction.  The even
    // block of a pair holds the barriers that say "operands are there" and "sums have been read".
    const int csize = (PAIR ? 2 : 1) * P.splits;
    const int crank = csize > 1 ? (int)(blockIdx.x % (unsigned)csize) : 0;
    const int side = PAIR ? crank & 1 : 0, rank = PAIR ? crank >> 1 : crank;
    const uint16_t both = (uint16_t)(3u << (crank & ~1));
    auto lead = [&](uint32_t bar) { return PAIR ? cluster_addr(bar, (uint32_t)(crank & ~1)) : bar; };
    auto arrive_lead = [&](uint32_t bar) {
        if (PAIR) mbar_arrive_cluster(lead(bar));
        else mbar_arrive(bar);
    };

    asm volatile("griddepcontrol.launch_dependents;");
    if (tid == 0) {
        s_abort = 0; s_started = 0; s_odd = 0;
        for (int i = 0; i < P.a_stages; ++i) { mbar_init(a_full(i), (P.tma ? 1 : (PAIR ? 2 : 1) * kProdWarps) + P.hold); mbar_init(a_empty(i), 1); }
        for (int i = 0; i < P.b_slots; ++i) { mbar_init(b_full(i), 1); mbar_init(b_empty(i), 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(acc_full(i), 1); mbar_init(acc_empty(i), (PAIR ? 2 : 1) * kEpiWarps); }
        mbar_init(all_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_proxy();
    }
    if (warp == kEpiWarps + kProdWarps) tmem_alloc<PAIR>(smem_u32(&s_tmem), (uint32_t)P.tmem_cols);
    tc_fence_before();
    __syncthreads();
    if (csize > 1) cluster_meet();       // the other blocks run, their barriers stand
    tc_fence_after();
    const uint32_t tmem = s_tmem;

    // A block (pair) of an unsplit launch takes items its number, + number of blocks, ... (all of the
    // same filter range); a cluster of a split launch takes one item, each block a range of stages.
    const int item0 = (int)(blockIdx.x / (unsigned)csize);
    const int item_step = P.splits > 1 ? P.items : (int)(gridDim.x / (unsigned)csize);
    const int k0 = rank * P.per_split, k1 = min(P.stages, k0 + P.per_split);
    const int n0 = tap_item<MT, PAIR>(P, item0, side).n0;
    const int planes = (P.c_in + T::cpp * 2 - 1) / (T::cpp * 2) * 2;
    const uint32_t a_part = (uint32_t)P.pl * P.plane_pitch;       // fp32: bytes of one part of a stage

    if (warp >= kEpiWarps && warp < kEpiWarps + kProdWarps) {
        if (!kF32 && P.tma) {
            asm volatile("griddepcontrol.wait;" ::: "memory");
            if (warp == kEpiWarps) {
                // ---- x by tensor copies, zeros outside the image; the lanes share the copies of a stage
                // (rows one by one from one thread cost it 190 cycles each) ---------------------------------
                int s = 0;
                uint32_t ph = 1;
                const int per = TAPS == 1 || !P.row_boxes ? 1 : P.rows, boxes = (TAPS == 1 || STRIDE == 1 ? 1 : 4) * per;
                const int step = (P.row_boxes ? 1 : P.rows) * P.pitch * 128;
                for (int item = item0; item < P.items; item += item_step) {
                    const TapItem t = tap_item<MT, PAIR>(P, item, side);
                    if (lane == 0) s_started = s_started + 1;
                    for (int ks = k0; ks < k1; ++ks) {
                        wait_warp(a_empty(s), ph);
                        const uint32_t bar = lead(a_full(s));
                        const uint32_t dst = sbase + (uint32_t)(s * P.a_bytes) + (P.raster ? (uint32_t)(P.pitch - 1 - t.ox0) * 128u : 0u);
                        const int c = ks * T::row_ch;
                        if (side == 0 && lane == 0) mbar_expect_tx(a_full(s), (uint32_t)(P.a_tx * (PAIR ? 2 : 1)));
                        if (TAPS == 1) {
                            if (lane == 0) tensor_load4<PAIR>(dst, &xmap, c, t.v0 * 8, 0, 0, bar);
                        } else {
                            for (int b = lane; b < boxes; b += 32) {
                                const int region = STRIDE == 1 ? 0 : div_by(b, per, P.row_boxes ? P.mg_rows : 0u), i = b - region * per;
                                const int x0 = STRIDE == 1 ? (P.raster ? 0 : t.ox0) - 1 : 2 * t.ox0 - (region & 1);
                                const TapRow r = tap_row<STRIDE>(P, t, i, region >> 1);
                                tensor_load4<PAIR>(dst + (uint32_t)(b * step), &xmap, c, x0, r.y, r.img, bar);
                            }
                        }
                        __syncwarp();
                        if (++s == P.a_stages) { s = 0; ph ^= 1u; }
                    }
                }
            } else if (FUSED && P.residual && P.splits == 1) {
                // ---- the residual into L2, an item ahead of its use --------------------------
                const int pt = tid - (kEpiWarps + 1) * 32;
                const int row = min(P.nt, P.c_out - n0) * (DT == XGEN_F16_F32ACC ? 2 : 4), lines = (row + 127) / 128;
                auto fetch = [&](int item) {
                    if (item >= P.items) return;
                    const TapItem t = tap_item<MT, PAIR>(P, item, side);
                    for (int i = pt; i < 128 * MT * lines; i += kProdThreads - 32) {
                        const int m = i / lines, at = (i - m * lines) * 128;       // (always below `row`: of one filter it may be 2 bytes)
                        const int px = tap_pixel<TAPS>(P, t, m).pix;
                        if (px >= 0)
                            asm volatile("prefetch.global.L2 [%0];" ::"l"(static_cast<const char *>(P.residual) +
                                         ((size_t)px * P.c_out + n0) * (DT == XGEN_F16_F32ACC ? 2 : 4) + at));
                    }
                };
                fetch(item0);
                int done = 0;
                for (int item = item0; item < P.items; item += item_step, ++done) {
                    for (int it = 0; it < 100000 && s_started <= done; ++it) __nanosleep(100);     // (a pace, nothing depends on it)
                    fetch(item + item_step);
                }
            }
        } else {
            // ---- x through the producer warps ------------------------------------------------------
            const int pt = tid - kEpiWarps * 32;
            int s = 0;
            uint32_t ph = 1;
            bool par = false;
            const char *const x = static_cast<const char *>(P.x);
            const int total = kF32 ? P.pixels << P.pl_log : P.pixels * 8;
            for (int item = item0; item < P.items; item += item_step, par = !par) {
                const TapItem t = tap_item<MT, PAIR>(P, item, side);
                int *const pix = reinterpret_cast<int *>(smem + P.tab_off) + (par ? P.pixels : 0);
                for (int p = pt; p < P.pixels; p += kProdThreads) pix[p] = tap_source<STRIDE, TAPS>(P, t, p);
                asm volatile("bar.sync 1, %0;" ::"n"(kProdThreads) : "memory");
                if (item == item0) asm volatile("griddepcontrol.wait;" ::: "memory");
                for (int ks = k0; ks < k1; ++ks) {
                    wait_warp(a_empty(s), ph);
                    const uint32_t dst = sbase + (uint32_t)(s * P.a_bytes);
                    const int npl = min(P.pl, planes - ks * P.pl);
                    constexpr int U = kF32 ? 4 : 2;          // pieces of a thread in flight
                    for (int i0 = pt; i0 < total; i0 += U * kProdThreads) {
                        float f[kF32 ? U : 1][8];
                        uint4 g[kF32 ? 1 : U];
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            const int i = i0 + u * kProdThreads;
                            const int pl = kF32 ? i & (P.pl - 1) : i & 7, p = kF32 ? i >> P.pl_log : i >> 3;
                            const int c = (ks * P.pl + pl) * T::cpp;
                            const int px = i < total && pl < npl ? pix[p] : -1;
                            const char *src = x + ((size_t)(px < 0 ? 0 : px) * P.c_in + c) * T::xb;
                            const int left = px < 0 ? 0 : P.c_in - c;     // channels there are
                            if (kF32) {
                                float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
                                if (P.vec_x) {
                                    if (left > 0) lo = __ldg(reinterpret_cast<const float4 *>(src));
                                    if (left > 4) hi = __ldg(reinterpret_cast<const float4 *>(src) + 1);
                                } else {
                                    const float *q = reinterpret_cast<const float *>(src);
                                    if (left > 0) lo.x = __ldg(q);
                                    if (left > 1) lo.y = __ldg(q + 1);
                                    if (left > 2) lo.z = __ldg(q + 2);
                                    if (left > 3) lo.w = __ldg(q + 3);
                                    if (left > 4) hi.x = __ldg(q + 4);
                                    if (left > 5) hi.y = __ldg(q + 5);
                                    if (left > 6) hi.z = __ldg(q + 6);
                                    if (left > 7) hi.w = __ldg(q + 7);
                                }
                                float *const fu = f[kF32 ? u : 0];
                                fu[0] = lo.x; fu[1] = lo.y; fu[2] = lo.z; fu[3] = lo.w;
                                fu[4] = hi.x; fu[5] = hi.y; fu[6] = hi.z; fu[7] = hi.w;
                            } else {
                                g[kF32 ? 0 : u] = gather16(src, left * T::xb);
                            }
                        }
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            const int i = i0 + u * kProdThreads;
                            const int pl = kF32 ? i & (P.pl - 1) : i & 7, p = kF32 ? i >> P.pl_log : i >> 3;
                            if (i < total && pl < npl) {
                                if (kF32) {
                                    const uint32_t d = dst + (uint32_t)(pl * P.plane_pitch + p * 16);
                                    uint4 p0, p1, p2;
                                    split3(f[kF32 ? u : 0], p0, p1, p2);
                                    sts128(d, p0);
                                    sts128(d + a_part, p1);
                                    sts128(d + 2 * a_part, p2);
                                } else {
                                    sts128(dst + (uint32_t)(p * 128 + ((pl ^ (p & 7)) << 4)), g[kF32 ? 0 : u]);
                                }
                            }
                        }
                    }
                    fence_async_proxy();
                    __syncwarp();
                    if (lane == 0) arrive_lead(a_full(s));
                    if (++s == P.a_stages) { s = 0; ph ^= 1u; }
                }
            }
        }
    } else if (warp == kEpiWarps + kProdWarps) {
        // ---- matrix instructions: one thread, which also waits.  A wait that gives up is not looked at:
        // nothing per-thread may steer these loops, or every operand is moved to the uniform registers
        // anew; all later waits then return at once.  Three taps are unrolled and share a barrier, and
        // the next barrier is looked at before the instructions of this one are issued: in a rolled loop
        // with a wait of its own a tap costs 350 cycles, its four instructions of 128 x 128 x 16 take 256.
        // fp32 has instructions enough in a tap to roll the rest, and less code to fetch at the start of a
        // short launch. ------------------------------------------------------------------------------
        if (side == 0 && elect_one()) {
            const uint32_t b_rows = (uint32_t)P.nt / (PAIR ? 2 : 1);         // filters whose weights this block holds
            const uint32_t b_tap = PARTS * b_rows;                           // 16-byte units from here on
            const uint32_t b_plane = b_tap * (uint32_t)P.tap_group;
            const uint64_t a0 = kF32 ? operand_desc(sbase, (uint32_t)P.plane_pitch, (P.raster ? 8 : P.pitch) * 16)
                                     : operand_desc_swizzled(sbase, (P.raster ? 8 : P.pitch) * 128);
            const uint64_t b0 = operand_desc(sbase + P.b_off, b_plane * 16, 128);
            const uint32_t a_hi = (uint32_t)(a0 >> 32), b_hi = (uint32_t)(b0 >> 32), idesc = P.idesc;
            const uint32_t a_k = kF32 ? (uint32_t)P.plane_pitch * 2 / 16 : 2u, b_k = b_plane * 2, a_p = a_part / 16, b_p = b_rows;
            constexpr uint32_t a_px = kF32 ? 1 : 8;
            const uint32_t a_sub = (uint32_t)P.sub_px * a_px, a_step = (uint32_t)P.a_bytes / 16, b_step = (uint32_t)P.b_bytes / 16;
            int s = 0, b = 0, buf = 0, run = 0;                             // run: stages since the accumulator was empty (CUT)
            uint32_t pha = 0, phb = 0, phc = 1, as = (uint32_t)a0, bs = (uint32_t)b0;
            bool ready = mbar_try<PAIR>(b_full(0), 0);
            for (int item = item0; item < P.items; item += item_step) {
                for (int ks = k0; ks < k1; ++ks) {
                    if (kF32 || (CUT ? run == 0 : ks == k0)) wait(acc_empty(buf), phc);
                    wait(a_full(s), pha);
                    tc_fence_after();
                    const int kk_n = min(P.pl, planes - ks * P.pl) / 2;
                    const uint32_t d = tmem + (uint32_t)buf * (uint32_t)(MT * P.nt);
                    const uint32_t dc = d + 2u * P.nt;      // fp32: the small products (two buffers behind the two of the sums)
                    uint32_t bt = bs;
#pragma unroll (kF32 ? 1 : 3)
                    for (int t0 = 0; t0 < TAPS; t0 += 3) {
#pragma unroll
                    for (int t1 = 0; t1 < (TAPS == 1 ? 1 : 3); ++t1) {
                        const int tap = t0 + t1;
                        if ((P.tap_group == 1 || t1 == 0) && !ready)
                            mbar_wait_long<PAIR>(b_full(b), P.resident ? 0u : phb, &s_abort, P.status, P.wait_us);
                        const bool last = P.tap_group == 1 || t1 == 2;
                        if (last) {                         // (of its slot: look at the next one)
                            const bool wrap = b + 1 == P.b_slots;
                            ready = mbar_try<PAIR>(b_full(wrap ? 0 : b + 1), P.resident ? 0u : wrap ? phb ^ 1u : phb);
                        }
                        const uint32_t at = as + (uint32_t)P.tap_start[tap] * a_px;
#pragma unroll
                        for (int kk = 0; kk < (kF32 && TAPS == 9 ? 2 : 4); ++kk) {
                            if (kk < kk_n) {
                                const uint32_t ak = at + kk * a_k, bk = bt + kk * b_k;
                                const uint32_t first_s = tap > 0 || kk > 0 ? 1u : 0u;       // 0: the first of the stage
                                const uint32_t first_i = first_s | ((CUT ? run > 0 : ks > k0) ? 1u : 0u);     // 0: the first of the item (CUT: of its part)
                                if (kF32) {
                                    mma_f16<PAIR>(d, ak, a_hi, bk, b_hi, idesc, first_s);
                                    mma_f16<PAIR>(dc, ak, a_hi, bk + b_p, b_hi, idesc, first_s);
                                    mma_f16<PAIR>(dc, ak, a_hi, bk + 2 * b_p, b_hi, idesc, 1u);
                                    mma_f16<PAIR>(dc, ak + a_p, a_hi, bk, b_hi, idesc, 1u);
                                    mma_f16<PAIR>(dc, ak + a_p, a_hi, bk + b_p, b_hi, idesc, 1u);
                                    mma_f16<PAIR>(dc, ak + 2 * a_p, a_hi, bk, b_hi, idesc, 1u);
                                } else {
#pragma unroll
                                    for (int m = 0; m < MT; ++m) {
                                        if (DT == XGEN_I8_I32) mma_i8<PAIR>(d + m * P.nt, ak + m * a_sub, a_hi, bk, b_hi, idesc, first_i);
                                        else mma_f16<PAIR>(d + m * P.nt, ak + m * a_sub, a_hi, bk, b_hi, idesc, first_i);
                                    }
                                }
                            }
                        }
                        bt += b_tap;
                        if (last) {
                            if (!P.resident) tc_commit<PAIR>(b_empty(b), both);
                            bs += b_step;
                            if (++b == P.b_slots) { b = 0; phb ^= 1u; bs = (uint32_t)b0; }
                            bt = bs;
                        }
                    }
                    }
                    tc_commit<PAIR>(a_empty(s), both);
                    as += a_step;
                    if (++s == P.a_stages) { s = 0; pha ^= 1u; as = (uint32_t)a0; }
                    ++run;
                    if (kF32 || ks + 1 == k1 || (CUT && run == P.cut)) {
                        run = 0;
                        tc_commit<PAIR>(acc_full(buf), both);
                        if (++buf == P.acc_bufs) { buf = 0; phc ^= 1u; }
                    }
                }
            }
            tc_commit<PAIR>(all_done, both);
        }
        __syncwarp();
        for (int it = 0; it < 4000000 && !mbar_ready(all_done, 0); ++it) {}
    } else if (warp > kEpiWarps + kProdWarps) {
        // ---- weights ---------------------------------------------------------------
        if (elect_one()) {
            int b = 0, issued = 0;
            uint32_t ph = 1;
            for (int item = item0; item < P.items; item += item_step) {
                for (int ks = k0; ks < k1; ++ks) {
                    for (int tap = 0; tap < TAPS; tap += P.tap_group) {
                        if (issued >= P.b_slots) wait(b_empty(b), ph);
                        // one copy for a slot: pieces of 2 KB with a copy of their own cost 50 cycles
                        // of issue apiece and held the whole kernel to 5.5 TB/s of weights
                        if (side == 0) mbar_expect_tx(b_full(b), (uint32_t)P.b_bytes * (PAIR ? 2 : 1));
                        tensor_load4<PAIR>(sbase + P.b_off + (uint32_t)(b * P.b_bytes), &wmap, (n0 + side * P.nt / 2) * 2, 0, tap, ks * P.pl,
                                           lead(b_full(b)));
                        ++issued;
                        if (++b == P.b_slots) { b = 0; ph ^= 1u; }
                    }
                }
                if (P.resident) break;
            }
            // Nothing may land in shared memory after this block has gone (the wait for it may have given up).
            for (int q = max(0, issued - P.b_slots); q < issued && side == 0; ++q)
                for (int it = 0; it < 1000000 && !mbar_ready(b_full(q % P.b_slots), (uint32_t)(q / P.b_slots) & 1u); ++it) {}
        }
        __syncwarp();
    } else {
        // ---- epilogue ----------------------------------------------------------------
        asm volatile("griddepcontrol.wait;" ::: "memory");
        for (int i = tid; i < P.nt; i += kEpiWarps * 32) {
            const bool in = n0 + i < P.c_out;
            s_bias[i] = P.bias && in ? static_cast<const uint32_t *>(P.bias)[n0 + i] : 0u;
            s_scale[i] = FUSED && P.rq_scale && in ? P.rq_scale[n0 + i] : 0.0f;
        }
        asm volatile("bar.sync 2, %0;" ::"n"(kEpiWarps * 32) : "memory");
        // a warp's share: a quarter of the lanes, one of the tiles, every kGroups-th chunk of 32 filters
        constexpr int kGroups = kEpiWarps / 4 / MT;
        const int quarter = warp & 3, sub = (warp >> 2) % MT, group = (warp >> 2) / MT;
        const int chunks = P.nt / 32;
        const uint32_t lanes = (uint32_t)quarter << 21;
        const int m = quarter * 32 + lane;                       // pixel of the 128
        // Sums on their way out where they do not go straight from their lanes: the warp's 32 pixels x 16
        // filters, or (split) to the block of the cluster that adds up this pixel's, [source][pixel][filter].
        uint32_t *const st = reinterpret_cast<uint32_t *>(smem + P.stage_off + warp * kStageBytes);
        uint32_t *const st_own = st + lane * kStagePitch;
        uint32_t far = 0;
        if (P.splits > 1) {
            const int unit = sub * 8 + m / 16, adder = unit % P.splits, units = (8 * MT + P.splits - 1) / P.splits;
            far = cluster_addr(sbase + P.sum_off + (uint32_t)((rank * units + unit / P.splits) * 16 + m % 16) * (P.nt + 4) * 4,
                               (uint32_t)(PAIR ? 2 * adder + side : adder));
        }
        int buf = 0;
        uint32_t ph = 0;
        for (int item = item0; item < P.items; item += item_step) {
            const TapItem t = tap_item<MT, PAIR>(P, item, side);
            const TapPixel at = tap_pixel<TAPS>(P, t, sub * 128 + m);
            const int pix = at.pix, out = at.out;
            if (P.staged && P.splits == 1) { st_own[16] = (uint32_t)pix; st_own[17] = (uint32_t)out; }
            // 32 sums of this lane's pixel, from column c of the tile on
            auto finish = [&](uint32_t (&r)[32], int c) {
                if (P.splits > 1) {
#pragma unroll
                    for (int q = 0; q < 8; ++q) sts_cluster(far + (uint32_t)(c + 4 * q) * 4, r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]);
                    return;
                }
                if (n0 + c >= P.c_out) return;
                if (DT != XGEN_I8_I32 && !all_finite(r)) s_odd = 1;
                if (!P.staged) tap_direct<DT, FUSED>(P, s_bias, s_scale, r, pix, out, n0 + c, n0);
                else {
#pragma unroll 1
                    for (int h = 0; h < 2; ++h) {
                        __syncwarp();
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            *reinterpret_cast<uint4 *>(st_own + 4 * q) = make_uint4(r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]);
                        __syncwarp();
                        tap_emit<DT, FUSED>(P, st, s_bias, s_scale, n0 + c + 16 * h, n0, lane);
#pragma unroll
                        for (int i = 0; i < 16; ++i) r[i] = r[16 + i];
                    }
                    __syncwarp();
                }
            };
            auto release = [&]() {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) arrive_lead(acc_empty(buf));
                if (++buf == P.acc_bufs) { buf = 0; ph ^= 1u; }
            };
            if (kF32) {
                uint32_t sum[2][32];                 // chunks `group` and `group` + kGroups
#pragma unroll
                for (int i = 0; i < 64; ++i) sum[i / 32][i % 32] = 0u;
                for (int ks = k0; ks < k1; ++ks) {
                    wait_warp(acc_full(buf), ph);
                    tc_fence_after();
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const int q = group + h / 2 * kGroups;
                        if (q < chunks) {
                            const uint32_t ta = tmem + lanes + (uint32_t)(buf * P.nt + 32 * q + h % 2 * 16);
                            uint32_t a[16], b[16];
                            tmem_ld16(ta, a);
                            tmem_ld16(ta + 2 * P.nt, b);
                            tmem_wait_ld();
#pragma unroll
                            for (int i = 0; i < 16; i += 2) {
                                add2(a[i], a[i + 1], b[i], b[i + 1]);
                                add2(sum[h / 2][h % 2 * 16 + i], sum[h / 2][h % 2 * 16 + i + 1], a[i], a[i + 1]);
                            }
                        }
                    }
                    release();
                }
#pragma unroll 1
                for (int q = group; q < chunks; q += kGroups) {
                    finish(sum[0], 32 * q);
#pragma unroll
                    for (int i = 0; i < 32; ++i) sum[0][i] = sum[1][i];
                }
            } else if (CUT) {
                // the accumulator's sums go onto the item's, in columns behind the accumulators
                for (int ks = k0; ks < k1; ks += P.cut) {
                    wait_warp(acc_full(buf), ph);
                    tc_fence_after();
                    const uint32_t ta = tmem + lanes + (uint32_t)((buf * MT + sub) * P.nt), tt = tmem + lanes + (uint32_t)((P.acc_bufs * MT + sub) * P.nt);
                    const bool first = ks == k0, last = ks + P.cut >= k1;
#pragma unroll 1
                    for (int q = group; q < chunks; q += kGroups) {
                        uint32_t r[32];
                        tmem_ld16(ta + 32 * q, r);
                        tmem_ld16(ta + 32 * q + 16, r + 16);
                        tmem_wait_ld();
                        if (!first) {
#pragma unroll
                            for (int h = 0; h < 32; h += 16) {
                                uint32_t t16[16];
                                tmem_ld16(tt + 32 * q + h, t16);
                                tmem_wait_ld();
#pragma unroll
                                for (int i = 0; i < 16; i += 2) add2(r[h + i], r[h + i + 1], t16[i], t16[i + 1]);
                            }
                        }
                        if (last) finish(r, 32 * q);
                        else {
                            tmem_st16(tt + 32 * q, r);
                            tmem_st16(tt + 32 * q + 16, r + 16);
                            tmem_wait_st();
                        }
                    }
                    release();
                }
            } else {
                wait_warp(acc_full(buf), ph);
                tc_fence_after();
                const uint32_t ta = tmem + lanes + (uint32_t)((buf * MT + sub) * P.nt);
#pragma unroll 1
                for (int q = group; q < chunks; q += kGroups) {
                    uint32_t r[32];
                    tmem_ld16(ta + 32 * q, r);
                    tmem_ld16(ta + 32 * q + 16, r + 16);
                    tmem_wait_ld();
                    finish(r, 32 * q);
                }
                release();
            }
        }
    }

    // ---- split items: every block adds up its share of the pixels, in the order of the sources -------
    if (P.splits > 1) {
        __syncwarp();
        cluster_meet();
        constexpr int kAdders = (kEpiWarps + kProdWarps) * 32;
        if (tid < kAdders && !s_abort) {
            const TapItem t = tap_item<MT, PAIR>(P, item0, side);
            const int groups = P.nt / 8, pitch = (P.nt + 4) * 4;
            const bool pool = FUSED && P.pool;
            // units of two rows of eight pixels go round the blocks; a thread takes 8 channels of one (pooled) pixel
            const int units_all = (8 * MT + P.splits - 1) / P.splits, units = (8 * MT - rank + P.splits - 1) / P.splits;
            const int per_unit = (pool ? 4 : 16) * groups, source = units_all * 16 * pitch;
#pragma unroll 1
            for (int w = tid; w < units * per_unit; w += kAdders) {
                const int u = w / per_unit, wu = w - u * per_unit, row = wu / groups, g = wu - row * groups;
                const int c0 = n0 + 8 * g, in_unit = pool ? 2 * row : row;
                const TapPixel px = tap_pixel<TAPS>(P, t, 16 * (rank + u * P.splits) + in_unit);
                if (px.pix < 0 || c0 >= P.c_out) continue;
                uint32_t best[8];
#pragma unroll 1
                for (int q = 0; q < (pool ? 4 : 1); ++q) {
                    const unsigned char *own = smem + P.sum_off + (u * 16 + in_unit + (q & 1) + (q >> 1) * 8) * pitch + g * 32;
                    uint32_t v8[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) v8[i] = 0;
#pragma unroll 4
                    for (int r = 0; r < P.splits; ++r, own += source) {
                        const uint4 a = *reinterpret_cast<const uint4 *>(own), b = *reinterpret_cast<const uint4 *>(own + 16);
                        if (DT == XGEN_I8_I32) {
                            v8[0] += a.x; v8[1] += a.y; v8[2] += a.z; v8[3] += a.w; v8[4] += b.x; v8[5] += b.y; v8[6] += b.z; v8[7] += b.w;
                        } else {
                            add2(v8[0], v8[1], a.x, a.y); add2(v8[2], v8[3], a.z, a.w); add2(v8[4], v8[5], b.x, b.y); add2(v8[6], v8[7], b.z, b.w);
                        }
                    }
                    const int pix = px.pix + (q & 1) + (q >> 1) * P.wo;
                    if (DT != XGEN_I8_I32 && !all_finite(v8)) s_odd = 1;
                    tap_affine<DT, FUSED, 8>(P, s_bias, v8, pix, true, c0, n0);
#pragma unroll
                    for (int i = 0; i < 8; ++i) best[i] = q == 0 ? v8[i] : tap_max<DT>(best[i], v8[i]);
                }
                tap_store<DT, FUSED, 8>(P, s_scale, best, px.out, c0, n0);
            }
        }
    }
    __syncwarp();
    if (PAIR) cluster_meet();            // nobody leaves while the other may still use its memory
    tc_fence_before();
    __syncthreads();
    if (warp == kEpiWarps + kProdWarps) tmem_free<PAIR>(tmem, (uint32_t)P.tmem_cols);
    if (DT != XGEN_I8_I32 && s_odd) tap_repair<DT, STRIDE, TAPS, MT, PAIR>(P);
}

// ---- weight image ----------------------------------------------------------------
// A kept zero is stored as -0, a pruned one as +0 (tap_anew tells them apart; the sums do not).
template <int DT> __device__ __forceinline__ void put_weight(uint8_t *img, int taps, int rows, int oc, int ic, int tap, float w) {
    constexpr int cpp = TapTraits<DT>::cpp, parts = TapTraits<DT>::parts;
    uint8_t *const p = img + ((size_t)(ic / cpp * taps + tap) * parts * rows + oc) * 16;
    const int e = ic % cpp;
    if (DT == XGEN_I8_I32) reinterpret_cast<int8_t *>(p)[e] = (int8_t)(int)w;
    else if (DT == XGEN_F16_F32ACC) reinterpret_cast<__half *>(p)[e] = __float2half_rn(w == 0.0f ? -0.0f : w);      // exact: it was fp16
    else {
        const float big = __uint_as_float(0x7F7F0000u);
        if (!(fabsf(w) <= FLT_MAX)) {                        // once, or the parts would not add up to it
            reinterpret_cast<__nv_bfloat16 *>(p)[e] = __float2bfloat16_rn(w);
            return;
        }
        __nv_bfloat16 b = __float2bfloat16_rn(fminf(fmaxf(w, -big), big));
        if (__bfloat162float(b) == 0.0f) b = __float2bfloat16_rn(-0.0f);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            reinterpret_cast<__nv_bfloat16 *>(p + (size_t)k * rows * 16)[e] = b;
            w -= __bfloat162float(b);
            b = __float2bfloat16_rn(w);
        }
    }
}

// Kernels k0 to k0 + count - 1 of [c_out][c_in].
template <int DT>
__global__ void tap_expand_patterns(uint8_t *img, int c_in, int rows, int k0, int count, const int16_t *kpat, const uint4 *kw4,
                                    const uint16_t *masks) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, k = k0 + i;
    if (i >= count || kpat[i] < 0) return;
    const uint4 w = kw4[i];
    const unsigned mask = masks[kpat[i]];
    int n = 0;
    for (int t = 0; t < 9; ++t)
        if ((mask >> t) & 1) {
            put_weight<DT>(img, 9, rows, k / c_in, k % c_in, t, __uint_as_float(n == 0 ? w.x : n == 1 ? w.y : n == 2 ? w.z : w.w));
            ++n;
        }
}

template <int DT>
__global__ void tap_expand_dense(uint8_t *img, int c_in, int rows, int k0, int count, const void *dense, const uint8_t *row_keep,
                                 const uint8_t *col_keep, int br, int bc) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, k = k0 + i;
    if (i >= count) return;
    const int oc = k / c_in, ic = k % c_in;
    const size_t blk = (size_t)(oc / br) * ((c_in + bc - 1) / bc) + ic / bc;
    if (!row_keep[blk * br + oc % br] || !col_keep[blk * bc + ic % bc]) return;
    const float w = DT == XGEN_F32 ? static_cast<const float *>(dense)[i] : __half2float(static_cast<const __half *>(dense)[i]);
    put_weight<DT>(img, 1, rows, oc, ic, 0, w);
}

static int tap_cpp(xgen_dtype dt) { return dt == XGEN_I8_I32 ? 16 : 8; }
static int tap_parts(xgen_dtype dt) { return dt == XGEN_F32 ? 3 : 1; }

// Upload scratch: kPiece bytes a device, shared by all handles of the process, there while any handle is.  (Allocated
// and freed by every handle it cost 0.6 ms of the 2.2 that a 1000 x 1000 fp32 handle takes; kept by every handle
// it held a third of an fp32 image again.)  An upload holds `mu` until it has been waited for.
constexpr size_t kPiece = 1 << 20;
struct TapScratch {
    std::mutex mu;
    uint8_t *dev = nullptr;
    int users = 0;               // weight images there are
};
static TapScratch &tap_scratch(int device) {
    static TapScratch all[64];
    return all[device & 63];
}

// One upload into a new zeroed image.  Ends with `done`, or leaves nothing.
struct TapUpload {
    TapWeights &tw;
    TapScratch &sc;
    std::unique_lock<std::mutex> lock;
    uint8_t *scratch = nullptr, *own = nullptr;      // `own`: more than kPiece was asked for
    explicit TapUpload(TapWeights &w, int device) : tw(w), sc(tap_scratch(device)), lock(sc.mu) { tw.device = device; }
    ~TapUpload() {
        if (own) cudaFree(own);
        if (sc.users == 0 && sc.dev) { cudaFree(sc.dev); sc.dev = nullptr; }
    }
    xgen_status begin(xgen_dtype dt, int taps, int c_in, int c_out, size_t extra) {
        tw.dtype = dt; tw.taps = taps; tw.c_in = c_in; tw.c_out = c_out;
        tw.planes = (c_in + 2 * tap_cpp(dt) - 1) / (2 * tap_cpp(dt)) * 2;
        tw.rows = (c_out + 15) / 16 * 16;
        const size_t image = (size_t)tw.planes * taps * tap_parts(dt) * tw.rows * 16;
        tw.bytes = image + 16;                       // and the status word
        cudaError_t e = cudaMalloc(&tw.dev, tw.bytes);
        if (e == cudaSuccess && extra > kPiece) e = cudaMalloc(&own, extra);
        else if (e == cudaSuccess && !sc.dev) e = cudaMalloc(&sc.dev, kPiece);
        if (e == cudaSuccess) e = cudaMemsetAsync(tw.dev, 0, tw.bytes, 0);
        scratch = own ? own : sc.dev;
        if (e != cudaSuccess) return fail(e);
        tw.status = reinterpret_cast<int *>(tw.dev + image);
        return XGEN_OK;
    }
    xgen_status done(cudaError_t e) {
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(0);
        if (e != cudaSuccess) return fail(e);
        ++sc.users;
        return XGEN_OK;
    }
    xgen_status fail(cudaError_t e) {
        cudaGetLastError();
        if (tw.dev) cudaFree(tw.dev);
        tw = TapWeights();
        return e == cudaErrorMemoryAllocation ? XGEN_ERR_ALLOC : XGEN_ERR_CUDA;
    }
};

void tap_free(TapWeights &tw) {
    if (!tw.dev) return;
    TapScratch &sc = tap_scratch(tw.device);
    std::lock_guard<std::mutex> lock(sc.mu);
    cudaFree(tw.dev);
    if (--sc.users == 0 && sc.dev) { cudaFree(sc.dev); sc.dev = nullptr; }
    tw = TapWeights();
}

// Weights go up in pieces of the scratch.
xgen_status tap_upload_patterns(TapWeights &tw, xgen_dtype dt, int c_in, int c_out, const int16_t *kpat, const uint32_t *kw4,
                                const uint16_t *masks, int n_masks) {
    const size_t nk = (size_t)c_in * c_out, mb = ((size_t)n_masks * 2 + 15) / 16 * 16;
    const size_t piece = std::min(nk, (kPiece - mb) / 18 / 8 * 8);             // 16 bytes of weights and two of pattern each
    int device = 0;
    if (cudaGetDevice(&device) != cudaSuccess) return XGEN_ERR_CUDA;
    TapUpload up(tw, device);
    const xgen_status st = up.begin(dt, 9, c_in, c_out, mb + piece * 18);
    if (st != XGEN_OK) return st;
    uint8_t *const scratch = up.scratch;
    const uint16_t *mk = reinterpret_cast<const uint16_t *>(scratch);
    const uint4 *w = reinterpret_cast<const uint4 *>(scratch + mb);
    const int16_t *kp = reinterpret_cast<const int16_t *>(scratch + mb + piece * 16);
    cudaError_t e = cudaMemcpyAsync(scratch, masks, (size_t)n_masks * 2, cudaMemcpyHostToDevice, 0);
    for (size_t k0 = 0; k0 < nk && e == cudaSuccess; k0 += piece) {
        const size_t n = std::min(piece, nk - k0);
        e = cudaMemcpyAsync(scratch + mb, kw4 + k0 * 4, n * 16, cudaMemcpyHostToDevice, 0);
        if (e == cudaSuccess) e = cudaMemcpyAsync(scratch + mb + piece * 16, kpat + k0, n * 2, cudaMemcpyHostToDevice, 0);
        if (e != cudaSuccess) break;
        const unsigned blocks = (unsigned)((n + 255) / 256);
        if (dt == XGEN_F32) tap_expand_patterns<XGEN_F32><<<blocks, 256>>>(tw.dev, c_in, tw.rows, (int)k0, (int)n, kp, w, mk);
        else if (dt == XGEN_F16_F32ACC) tap_expand_patterns<XGEN_F16_F32ACC><<<blocks, 256>>>(tw.dev, c_in, tw.rows, (int)k0, (int)n, kp, w, mk);
        else tap_expand_patterns<XGEN_I8_I32><<<blocks, 256>>>(tw.dev, c_in, tw.rows, (int)k0, (int)n, kp, w, mk);
    }
    return up.done(e);
}

xgen_status tap_upload_dense(TapWeights &tw, xgen_dtype dt, int c_in, int c_out, const void *dense_w, const uint8_t *row_keep,
                             const uint8_t *col_keep, int br, int bc) {
    const size_t nk = (size_t)c_in * c_out, wb = dt == XGEN_F32 ? 4 : 2;
    const size_t blocks_of = (size_t)((c_out + br - 1) / br) * ((c_in + bc - 1) / bc);
    const size_t rb = blocks_of * br, cb = blocks_of * bc, fb = (rb + cb + 15) / 16 * 16;     // the keep flags, whole
    const size_t piece = std::min(nk, (std::max(kPiece, fb + kPiece / 4) - fb) / wb / 8 * 8);
    int device = 0;
    if (cudaGetDevice(&device) != cudaSuccess) return XGEN_ERR_CUDA;
    TapUpload up(tw, device);
    const xgen_status st = up.begin(dt, 1, c_in, c_out, fb + piece * wb);
    if (st != XGEN_OK) return st;
    uint8_t *const scratch = up.scratch;
    cudaError_t e = cudaMemcpyAsync(scratch, row_keep, rb, cudaMemcpyHostToDevice, 0);
    if (e == cudaSuccess) e = cudaMemcpyAsync(scratch + rb, col_keep, cb, cudaMemcpyHostToDevice, 0);
    for (size_t k0 = 0; k0 < nk && e == cudaSuccess; k0 += piece) {
        const size_t n = std::min(piece, nk - k0);
        e = cudaMemcpyAsync(scratch + fb, static_cast<const char *>(dense_w) + k0 * wb, n * wb, cudaMemcpyHostToDevice, 0);
        if (e != cudaSuccess) break;
        const unsigned blocks = (unsigned)((n + 255) / 256);
        if (dt == XGEN_F32) tap_expand_dense<XGEN_F32><<<blocks, 256>>>(tw.dev, c_in, tw.rows, (int)k0, (int)n, scratch + fb, scratch, scratch + rb, br, bc);
        else tap_expand_dense<XGEN_F16_F32ACC><<<blocks, 256>>>(tw.dev, c_in, tw.rows, (int)k0, (int)n, scratch + fb, scratch, scratch + rb, br, bc);
    }
    return up.done(e);
}

// ---- plans ---------------------------------------------------------------------
template <int DT, int TAPS> static const void *tap_kernel_dt(int stride, int mt, bool pair, bool cut) {
#define TAP_PICK_CUT(S, M, C) (pair ? (const void *)tap_kernel<DT, S, TAPS, M, true, C> : (const void *)tap_kernel<DT, S, TAPS, M, false, C>)
#define TAP_PICK(S, M) TAP_PICK_CUT(S, M, false)
    constexpr int M2 = DT == XGEN_F32 ? 1 : 2, S2 = TAPS == 1 ? 1 : 2;      // (what there is no instance of is never asked for)
    constexpr bool C = DT == XGEN_F16_F32ACC;
    if (cut) {
        if (stride == 1) return mt == 2 ? TAP_PICK_CUT(1, M2, C) : TAP_PICK_CUT(1, 1, C);
        return mt == 2 ? TAP_PICK_CUT(S2, M2, C) : TAP_PICK_CUT(S2, 1, C);
    }
    if (stride == 1) return mt == 2 ? TAP_PICK(1, M2) : TAP_PICK(1, 1);
    return mt == 2 ? TAP_PICK(S2, M2) : TAP_PICK(S2, 1);
#undef TAP_PICK
#undef TAP_PICK_CUT
}
static const void *tap_kernel_of(xgen_dtype dt, int stride, int taps, int mt, bool pair, bool cut) {
    if (taps == 1) return dt == XGEN_F32 ? tap_kernel_dt<XGEN_F32, 1>(1, mt, pair, cut) : tap_kernel_dt<XGEN_F16_F32ACC, 1>(1, mt, pair, cut);
    if (dt == XGEN_F32) return tap_kernel_dt<XGEN_F32, 9>(stride, mt, pair, cut);
    return dt == XGEN_F16_F32ACC ? tap_kernel_dt<XGEN_F16_F32ACC, 9>(stride, mt, pair, cut) : tap_kernel_dt<XGEN_I8_I32, 9>(stride, mt, pair, cut);
}

// Once per kernel and device: large shared memory, clusters of 16.
static cudaError_t tap_allow(const void *kern, int device) {
    static std::mutex mu;
    static std::vector<std::pair<const void *, int>> done;
    std::lock_guard<std::mutex> lock(mu);
    for (auto &d : done)
        if (d.first == kern && d.second == device) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kTapSmemMax);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) done.emplace_back(kern, device);
    return e;
}

// How many clusters of `size` blocks (one block per SM) the device holds at once.
static int tap_clusters(int size, int device, int sms) {
    static std::mutex mu;
    static int known[64][17];
    if (device < 0 || device >= 64) return sms / size;
    std::lock_guard<std::mutex> lock(mu);
    int &k = known[device][size];
    if (k) return k;
    const void *kern = tap_kernel_of(XGEN_F16_F32ACC, 1, 9, 1, false, false);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)size); cfg.blockDim = dim3(tap_threads(XGEN_F16_F32ACC)); cfg.dynamicSmemBytes = kTapSmemMax;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)size; at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = 1;
    int n = 0;
    if (tap_allow(kern, device) != cudaSuccess || cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
    k = n > 0 ? n : -1;
    return k;
}

int tap_block_threads(xgen_dtype dt) { return tap_threads(dt); }

bool tap_choose(const TapWeights &tw, const TapShape &s, int device, TapPlan &best) {
    static int sm_count[64];
    int sms = 148;
    if (device >= 0 && device < 64) {
        if (!sm_count[device]) cudaDeviceGetAttribute(&sm_count[device], cudaDevAttrMultiProcessorCount, device);
        if (sm_count[device]) sms = sm_count[device];
    }
    const xgen_dtype dt = tw.dtype;
    const int parts = tap_parts(dt), cpp = tap_cpp(dt), prod = dt == XGEN_F32 ? 6 : 1;
    const int xb = dt == XGEN_F32 ? 4 : dt == XGEN_F16_F32ACC ? 2 : 1, yb = dt == XGEN_F16_F32ACC ? 2 : 4;
    const int ho = (s.h - 1) / s.stride + 1, wo = (s.w - 1) / s.stride + 1;
    best = TapPlan();
    best.cycles = 1e30;
    const bool swizzled = dt != XGEN_F32, copied = swizzled && (size_t)tw.c_in * xb % 16 == 0;
    // Tiles: 8-pixel columns with every image rounded up to whole tiles (0), with one row of zeros between
    // images and tiles that cross them (1), or runs of the raster (2).
    for (int shape = 0; shape < 12; ++shape) {
        TapPlan p;
        p.pair = shape & 1;
        p.mt = 1 + (shape >> 1) % 2;
        const int form = (shape >> 1) / 2, mt = p.mt, ways = p.pair ? 2 : 1, R = 16 * mt;
        if (mt == 2 && dt == XGEN_F32) continue;
        p.raster = form == 2;
        p.straddle = form >= 1;
        int64_t tiles_all;
        if (tw.taps == 1) {
            if (form) continue;
            p.pitch = 8; p.rows = R; p.pixels = 8 * R; p.segs = 1; p.vh = 1;
            p.row_tiles = (s.h + R - 1) / R;
            tiles_all = p.row_tiles;
        } else if (p.raster) {
            if (s.stride != 1 || s.pool || s.w > 150) continue;
            p.vh = ho + 1;
            p.pitch = s.w + 1;
            p.rows = 3 + (128 * mt + p.pitch - 1) / p.pitch;
            p.pixels = p.rows * p.pitch + p.pitch - 1;
            p.segs = 1;
            tiles_all = ((int64_t)s.n * p.vh * p.pitch + 128 * mt - 1) / (128 * mt);
            p.row_tiles = (int)std::min<int64_t>(tiles_all, 0x7FFFFFFF);
        } else {
            const int whole = (ho + R - 1) / R * R, gap = ho + 1 + (s.pool && (ho + 1) % 2 ? 1 : 0);
            p.vh = p.straddle ? gap : whole;
            if (p.straddle && (int64_t)s.n * gap >= (int64_t)s.n * whole) continue;
            p.pitch = s.stride == 1 ? 10 : 9;
            p.rows = s.stride == 1 ? R + 2 : R + 1;
            p.pixels = p.rows * p.pitch * (s.stride == 1 ? 1 : 4);
            p.segs = (wo + 7) / 8;
            const int64_t rt = ((int64_t)s.n * p.vh + R - 1) / R;
            tiles_all = rt * p.segs;
            p.row_tiles = (int)std::min<int64_t>(rt, 0x7FFFFFFF);
        }
        if (tiles_all * ((tw.rows + 31) / 32) > 0x7FFFFFFF / 256) continue;
        if (p.pair && tiles_all == 1) continue;
        const int tiles = (int)((tiles_all + ways - 1) / ways), pixels = p.pixels;
        p.table_bytes = copied && tw.taps == 9 ? 0 : (pixels * 8 + 127) / 128 * 128;
        // fp32 keeps four accumulators of `nt` columns and 64 sums a thread; 512 columns hold all of the others'
        const int nt_top = dt == XGEN_F32 || !p.pair ? 128 : kMaxFilterTile;
        for (int nt_max = 32; nt_max <= nt_top; nt_max += 32) {
            p.nblk = (tw.c_out + nt_max - 1) / nt_max;
            p.nt = ((tw.c_out + p.nblk - 1) / p.nblk + 31) / 32 * 32;
            p.nblk = (tw.c_out + p.nt - 1) / p.nt;
            if (p.nt != nt_max) continue;
            p.items = tiles * p.nblk;
            for (int pl = 2; pl <= 8; pl *= 2) {
                if (swizzled && pl != 8) continue;                          // rows of 128 bytes
                if (!swizzled && pl > 2 && pl / 2 >= tw.planes) continue;
                if (!swizzled && tw.taps * pl / 2 > 18) continue;           // bounds the chain of the fp32 accumulator
                p.pl = swizzled ? std::min(8, tw.planes) : pl;
                p.stages = (tw.planes + pl - 1) / pl;
                // 16-byte accesses of 8 lanes (pl planes x 8 / pl pixels) fall into distinct banks
                p.plane_pitch = pixels * 16;
                while (p.plane_pitch % 128 != 128 / pl % 128) p.plane_pitch += 16;
                p.a_bytes = swizzled ? (pixels * 128 + 1023) / 1024 * 1024 : parts * pl * p.plane_pitch;
                if ((size_t)p.a_bytes > (size_t)kTapSmemMax) continue;
                for (int sp = 1; sp * ways <= 16 && sp <= p.stages; ++sp) {
                    p.per_split = (p.stages + sp - 1) / sp;
                    p.splits = (p.stages + p.per_split - 1) / p.per_split;
                    if (p.splits != sp) continue;
                    // fp16: 4 steps of 16 channels a tap and stage; a chain of more than 288 (512 channels in nine taps)
                    // is cut: every 144 steps where its sums and two accumulators fit tensor memory, every 288 with one
                    p.cut = 0;
                    if (dt == XGEN_F16_F32ACC && p.per_split * tw.taps * 4 > 288) {
                        if (2 * mt * p.nt > 512) continue;
                        p.cut = (3 * mt * p.nt <= 512 ? 144 : 288) / (tw.taps * 4);
                    }
                    int64_t waves;
                    if (sp == 1) {
                        const int units = p.pair ? std::max(0, tap_clusters(2, device, sms)) : sms;
                        if (units == 0) continue;
                        const int at_once = p.items <= units ? p.items : std::min(p.items, std::max(1, units / p.nblk) * p.nblk);
                        p.grid = at_once * ways;
                        waves = (p.items + at_once - 1) / at_once;
                    } else {
                        if (p.items * (int64_t)sp * ways > 4 * sms) continue;
                        const int cl = tap_clusters(sp * ways, device, sms);
                        if (cl <= 0) continue;
                        p.grid = p.items * sp * ways;
                        waves = (p.items + cl - 1) / cl;
                    }
                    const size_t tables = p.table_bytes + (sp > 1 ? (size_t)sp * ((8 * mt + sp - 1) / sp) * 16 * (p.nt + 4) * 4
                                                                  : s.staged ? (size_t)epi_warps(dt) * kStageBytes : 0);
                    const int64_t uses = (sp == 1 ? waves : 1) * p.per_split;      // stages one block goes through
                    // Shared memory: two tiles of x (more for a plain product, whose stages are short), the rest
                    // weights, by three taps if at least three such slots fit.
                    bool fits = false;
                    for (p.tap_group = tw.taps == 1 ? 1 : 3; p.tap_group >= 1 && !fits; p.tap_group -= 2) {
                        p.b_bytes = p.tap_group * p.pl * parts * p.nt * 16 / ways;
                        const int all_b = p.per_split * tw.taps / p.tap_group;
                        for (p.a_stages = (int)std::min<int64_t>(uses, tw.taps == 1 ? kMaxA : 2); p.a_stages >= 1; --p.a_stages) {
                            const size_t left_a = (size_t)p.a_stages * p.a_bytes + tables;
                            if (left_a >= (size_t)kTapSmemMax) continue;
                            const int room = (int)std::min<size_t>(kMaxB, ((size_t)kTapSmemMax - left_a) / p.b_bytes);
                            p.resident = all_b <= room;
                            p.b_slots = std::min(room, all_b);
                            if (p.b_slots >= std::min(all_b, 3) && p.a_stages >= std::min<int64_t>(2, uses)) { fits = true; break; }
                        }
                        if (fits) break;
                    }
                    if (!fits) continue;
                    p.smem = (size_t)p.a_stages * p.a_bytes + (size_t)p.b_slots * p.b_bytes + tables;
                    if (p.smem > (size_t)kTapSmemMax) continue;
                    p.acc_bufs = dt == XGEN_F32 || (p.cut ? 3 : 2) * mt * p.nt <= 512 ? 2 : 1;
                    const int cols = dt == XGEN_F32 ? 4 * p.nt : (p.acc_bufs + (p.cut ? 1 : 0)) * mt * p.nt;
                    for (p.tmem_cols = 32; p.tmem_cols < cols;) p.tmem_cols *= 2;
                    // Cycles of a stage: the matrix instructions (nt / 2 each; 46 to issue one and 90 for a tap), or
                    // what they and the copies move through shared memory at 128 bytes a cycle (128 rows of x,
                    // the block's filters), or what comes from L2.  A pair starts and ends later: 4000 cycles where it
                    // halves much (fp32: three parts of weights; stride 2: single taps in the slots), else 6000
                    // (256 -> 256 at 14x14, batch 32, fp16: 12.8 us as pairs, 11.7 without); the
                    // short stages of a product wait 300 cycles for its other block (1842 filters x 5421 rows,
                    // fp32: 77 us as pairs, 57 us without).
                    const double kk = (double)tw.planes / p.stages / 2, taps = tw.taps;
                    const double b_stage = taps * kk * 2 * parts * p.nt * 16.0 / ways, b_moved = p.resident && sp == 1 ? b_stage / waves : b_stage;
                    const double x_moved = (double)pixels * kk * 2 * cpp * xb, a_stage = (double)p.a_bytes * (swizzled ? 1 : 2);
                    const double per_tap = kk * mt * prod, instr = taps * per_tap;
                    const double mma = taps * std::max(per_tap * p.nt / 2.0, 90.0 + 46.0 * per_tap);
                    const double shared = (instr * (4096.0 + p.nt * 32.0 / ways) + b_moved + a_stage) / 128.0;
                    const double move = (x_moved + b_moved) / 40.0 + (copied && p.straddle ? 60.0 * p.rows * (s.stride == 1 ? 1 : 4) : 0.0) * 0.5;
                    const double stage = std::max(std::max(mma, shared), move) + 250.0 + 40.0 * taps / p.tap_group + (p.pair && tw.taps == 1 ? 300.0 : 0.0);
                    const double out = (double)mt * 128 * p.nt * yb / 24.0;
                    // (one accumulator that is cut waits for its sums to be added)
                    const double item = p.per_split * stage + (p.cut && p.acc_bufs == 1 ? (p.per_split - 1) / p.cut * 1500.0 : 0.0);
                    double c = 3500.0 + (p.pair ? dt == XGEN_F32 || s.stride == 2 ? 4000.0 : 6000.0 : 0.0);
                    if (sp == 1) c += waves * std::max(item, p.acc_bufs == 2 ? out : 0.0) + (p.acc_bufs == 2 ? out : waves * out);
                    else c += waves * (item + 3500.0 + 100.0 * sp + mt * 128.0 * p.nt * 4 / 64.0 + out / sp);
                    if (c < best.cycles * 0.999) { best = p; best.cycles = c; }
                }
            }
        }
    }
    if (best.cycles >= 1e30) return false;
    // [plane][tap][part][filter x 16 bytes], in units of 8 bytes; what lies beyond the image reads as zeros
    EncodeTiledFn encode = encode_tiled_fn();
    if (!encode) return false;
    const cuuint64_t dim[4] = {(cuuint64_t)tw.rows * 2, (cuuint64_t)parts, (cuuint64_t)tw.taps, (cuuint64_t)tw.planes};
    const cuuint64_t row = (cuuint64_t)tw.rows * 16;
    const cuuint64_t str[3] = {row, row * parts, row * parts * tw.taps};
    const cuuint32_t box[4] = {(cuuint32_t)(best.pair ? best.nt : best.nt * 2), (cuuint32_t)parts, (cuuint32_t)best.tap_group, (cuuint32_t)best.pl};
    const cuuint32_t one[4] = {1, 1, 1, 1};
    return encode(&best.wmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 4, tw.dev, dim, str, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The tensor map of x: boxes of 128 bytes of channels of the staged rows (one, or all of a tile).
static bool x_map(const TapWeights &tw, const TapShape &s, const TapPlan &p, const void *x, CUtensorMap &m) {
    EncodeTiledFn encode = encode_tiled_fn();
    if (!encode) return false;
    const cuuint64_t px = (cuuint64_t)tw.c_in * (tw.dtype == XGEN_I8_I32 ? 1 : 2);
    const cuuint64_t w = tw.taps == 1 ? (cuuint64_t)s.rows : (cuuint64_t)s.w, h = tw.taps == 1 ? 1 : (cuuint64_t)s.h;
    const cuuint64_t dim[4] = {(cuuint64_t)tw.c_in, w, h, (cuuint64_t)s.n};
    const cuuint64_t str[3] = {px, px * w, px * w * h};
    const cuuint32_t st = (cuuint32_t)s.stride;
    const cuuint32_t box[4] = {tw.dtype == XGEN_I8_I32 ? 128u : 64u, (cuuint32_t)(tw.taps == 1 ? p.pixels : p.pitch) * st,
                               (cuuint32_t)(tw.taps == 1 || p.straddle ? 1 : p.rows) * st, 1};
    const cuuint32_t step[4] = {1, st, st, 1};
    return encode(&m, tw.dtype == XGEN_I8_I32 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, const_cast<void *>(x), dim, str,
                  box, step, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

cudaError_t tap_launch(const TapWeights &tw, const TapShape &s, const TapPlan &p, const TapCall &c, cudaStream_t st) {
    CUtensorMap xm{};
    const xgen_dtype dt = tw.dtype;
    const int parts = tap_parts(dt), xb = dt == XGEN_F32 ? 4 : dt == XGEN_F16_F32ACC ? 2 : 1;
    const int yb = c.rq_scale ? 1 : dt == XGEN_F16_F32ACC ? 2 : 4, rb = dt == XGEN_F16_F32ACC ? 2 : 4;
    TapParams P{};
    P.x = c.x; P.y = c.y; P.bias = c.bias; P.residual = c.residual; P.rq_scale = c.rq_scale;
    P.status = c.status; P.wait_us = c.wait_us; P.hold = std::min(c.hold, 1000);       // (a barrier counts to 2^20)
    P.rq_zero = c.rq_zero; P.relu = c.relu ? 1 : 0; P.pool = c.pool;
    P.n = s.n; P.h = s.h; P.w = s.w;
    P.ho = (s.h - 1) / s.stride + 1; P.wo = (s.w - 1) / s.stride + 1;
    P.po = c.pool ? P.ho / 2 : P.ho; P.pw = c.pool ? P.wo / 2 : P.wo;
    P.npix = s.rows;
    P.c_in = tw.c_in; P.c_out = tw.c_out;
    P.vh = p.vh; P.straddle = p.straddle;
    P.segs = p.segs; P.nblk = p.nblk; P.nt = p.nt; P.items = p.items; P.splits = p.splits; P.per_split = p.per_split; P.stages = p.stages; P.cut = p.cut;
    P.pl = p.pl; P.pl_log = p.pl == 2 ? 1 : p.pl == 4 ? 2 : 3; P.plane_pitch = p.plane_pitch;
    P.a_stages = p.a_stages; P.b_slots = p.b_slots; P.resident = p.resident;
    P.b_bytes = p.b_bytes; P.tap_group = p.tap_group;
    P.a_bytes = p.a_bytes;
    P.b_off = p.a_stages * p.a_bytes;
    P.tab_off = P.b_off + p.b_slots * P.b_bytes;
    P.stage_off = P.sum_off = P.tab_off + p.table_bytes;       // (the one or the other)
    P.raster = p.raster; P.pitch = p.pitch; P.rows = p.rows; P.pixels = p.pixels; P.sub_px = p.raster ? 128 : 16 * p.pitch;
    {
        // exact for n < 2^32 / d: the largest n are the rows (raster entries) of all tiles
        auto magic = [](int64_t most, int d) { return d > 1 && (most + 1) * d < (1ll << 32) ? (uint32_t)((1ull << 32) / (uint64_t)d + 1) : 0u; };
        const int64_t last_tile = (int64_t)(p.items / p.nblk) * (p.pair ? 2 : 1) * p.mt;
        const int64_t rows_all = p.raster ? last_tile * 128 / p.pitch + 64 : (int64_t)(p.row_tiles + 2) * 16 * p.mt + 64;
        P.mg_pitch = magic(p.raster ? last_tile * 128 + 512 : p.pixels, p.pitch);
        P.mg_vh = magic(rows_all, p.vh);
        P.mg_rows = magic(p.pixels, p.rows);
    }
    P.row_boxes = p.straddle; P.a_tx = p.pixels * 128 - (p.raster ? (p.pitch - 1) * 128 : 0);
    P.wimg = tw.dev; P.w_rows = tw.rows;
    P.tmem_cols = p.tmem_cols; P.acc_bufs = p.acc_bufs; P.staged = s.staged;
    for (int t = 0; t < tw.taps; ++t) {
        const int dy = t / 3, dx = t % 3;
        if (tw.taps == 1) P.tap_start[t] = 0;
        else if (s.stride == 1) P.tap_start[t] = (p.raster ? p.pitch - 1 : 0) + dy * p.pitch + dx;
        else    // of the image of the tap's parities; the third row (column) is the second of the odd ones
            P.tap_start[t] = ((dy == 1 ? 0 : 2) + (dx == 1 ? 0 : 1)) * p.rows * p.pitch + (dy == 2 ? p.pitch : 0) + (dx == 2 ? 1 : 0);
    }
    auto aligned = [](const void *q, uintptr_t a) { return ((uintptr_t)q & (a - 1)) == 0; };
    P.vec_x = aligned(c.x, 16) && (size_t)tw.c_in * xb % 16 == 0;
    P.tma = dt != XGEN_F32 && P.vec_x && x_map(tw, s, p, c.x, xm);
    // a plan for tensor copies has no room for the table of pixels that gathering the rows takes
    if (!P.tma && p.table_bytes == 0) return cudaErrorInvalidValue;
    P.vec_y = aligned(c.y, 16) && (size_t)tw.c_out * yb % 16 == 0;
    P.y32 = aligned(c.y, 32) && (size_t)tw.c_out * yb % 32 == 0;
    P.vec_r = c.residual && aligned(c.residual, 16) && (size_t)tw.c_out * rb % 16 == 0;
    // D fp32 (int32), A fp16 / bf16 / u8, B fp16 / bf16 / s8, both K-major, 128 rows (256 of a pair)
    P.idesc = ((uint32_t)(p.nt >> 3) << 17) | ((p.pair ? 16u : 8u) << 24) |
              (dt == XGEN_I8_I32 ? (2u << 4) | (1u << 10) : (1u << 4) | (dt == XGEN_F32 ? (1u << 7) | (1u << 10) : 0u));
    const void *kern = tap_kernel_of(dt, s.stride, tw.taps, p.mt, p.pair, p.cut != 0);
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e == cudaSuccess) e = tap_allow(kern, device);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.grid); cfg.blockDim = dim3((unsigned)tap_threads(dt)); cfg.dynamicSmemBytes = p.smem; cfg.stream = st;
    cudaLaunchAttribute at[2];
    unsigned na = 0;
    if (c.overlap) {
        at[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[na++].val.programmaticStreamSerializationAllowed = 1;
    }
    const int cluster = (p.pair ? 2 : 1) * p.splits;
    if (cluster > 1) {
        at[na].id = cudaLaunchAttributeClusterDimension;
        at[na].val.clusterDim.x = (unsigned)cluster; at[na].val.clusterDim.y = at[na].val.clusterDim.z = 1;
        ++na;
    }
    cfg.attrs = at; cfg.numAttrs = na;
    void *args[3] = {&P, const_cast<CUtensorMap *>(&p.wmap), &xm};
    e = cudaLaunchKernelExC(&cfg, kern, args);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) count_launch();
    return e;
}

}  // namespace patconv
