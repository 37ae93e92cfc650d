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
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

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
constexpr int kMaxA = 6, kMaxB = 36, kMaxAcc = 4;
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
    int pl, plane_pitch;
    int a_stages, a_bytes, b_slots, resident, b_bytes, tap_group;
    int raw_slots, raw_px, raw_bytes, raw_pitch, row_log;    // x as it lies in memory: buffers, pixels and bytes of one, bytes of a pixel; pieces of a pixel (log2)
    int b_off, tab_off, raw_off, stage_off, sum_off;     // bytes into dynamic shared memory
    int tmem_cols, acc_bufs, staged;
    int tap_start[9];                           // first staged entry of a tap
    const uint8_t *wimg; int w_rows;            // the weight image (TapWeights)
    int row_boxes, a_tx;                             // a tensor copy of x per staged row; the bytes of a stage
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
// and store them so that neighbouring lanes hold neighbouring elements: where rows of y are not whole 16-byte pieces, and fp32
// with a residual (its sums are in registers, a pixel a lane; held in quads, as tap_quad has them, they cost every stage a choice of
// loads: 81 x 9x9, 91 -> 192 with residual 18.7 -> 19.2 us).
template <int DT, bool FUSED>
__device__ __forceinline__ void tap_emit(const TapParams &P, const uint32_t *st, const uint32_t *s_bias, const float *s_scale,
                                         int c_base, int n0, int lane) {
    const bool pool = FUSED && P.pool;
    if constexpr (FUSED && DT == XGEN_F32) if (P.vec_y && P.vec_r && !pool) {
        const int c = c_base + (lane & 3) * 4;
        if (c >= P.c_out) return;
        const uint4 b = *reinterpret_cast<const uint4 *>(s_bias + (c - n0));
        const uint32_t *const row0 = st + (lane >> 2) * kStagePitch;
        uint4 res[4];
        int px[4];
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            px[it] = (int)row0[it * 8 * kStagePitch + 16];
            const size_t off = (size_t)max(px[it], 0) * P.c_out + c;
            res[it] = __ldg(reinterpret_cast<const uint4 *>(static_cast<const uint32_t *>(P.residual) + off));
        }
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            const uint4 a = *reinterpret_cast<const uint4 *>(row0 + it * 8 * kStagePitch + (lane & 3) * 4);
            uint32_t v[4] = {a.x, a.y, a.z, a.w};
            add2(v[0], v[1], b.x, b.y); add2(v[2], v[3], b.z, b.w);
            add2(v[0], v[1], res[it].x, res[it].y); add2(v[2], v[3], res[it].z, res[it].w);
            if (P.relu) {
#pragma unroll
                for (int i = 0; i < 4; ++i) v[i] = tap_max<DT>(v[i], 0u);
            }
            if (px[it] < 0) continue;
            const size_t off = (size_t)px[it] * P.c_out + c;
            *reinterpret_cast<uint4 *>(static_cast<uint32_t *>(P.y) + off) = make_uint4(v[0], v[1], v[2], v[3]);
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
// whole sectors.  (A residual without a pool: tap_quad.)
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
            tap_affine<DT, false, 8>(P, s_bias, w, pix, true, c0 + 8 * g, n0);
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

// fp16 and int8 sums with a residual, in the layout of tmem_ld_quad: a lane holds two adjacent channels (of each of two blocks of
// eight) of four pixels, so that the four lanes of a quad hold 32 adjacent bytes of the residual and of y and nothing need pass
// through shared memory.  Pixels px[2 h + r]: row 16 h + 8 r + lane / 4 of the warp's 32; sum v[8 h + 4 i + 2 r + e]:
// channel c + 8 i + 2 (lane % 4) + e.  The residual is asked for before the sums are waited for.
// (32 lanes a pixel each touched 32 lines an access; by way of shared memory 256 x 64 int32 residuals took 7000 cycles:
// 64 images of 28x28x128 int8 20.9 us, 16.9 now.)
template <int DT> struct QuadRes { uint32_t v[DT == XGEN_F16_F32ACC ? 8 : 16]; };
template <int DT> __device__ __forceinline__ void quad_residual(const TapParams &P, QuadRes<DT> &res, const int (&px)[4], int c) {
    c += 2 * (threadIdx.x & 3);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const size_t off = (size_t)max(px[k], 0) * P.c_out;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const size_t at = off + min(c + 8 * i, P.c_out - 2);             // (c_out is even here)
            if constexpr (DT == XGEN_F16_F32ACC) res.v[2 * k + i] = __ldg(reinterpret_cast<const uint32_t *>(static_cast<const __half *>(P.residual) + at));
            else {
                const uint2 r = __ldg(reinterpret_cast<const uint2 *>(static_cast<const uint32_t *>(P.residual) + at));
                res.v[4 * k + 2 * i] = r.x;
                res.v[4 * k + 2 * i + 1] = r.y;
            }
        }
    }
}
template <int DT> __device__ __forceinline__ void tap_quad(const TapParams &P, const uint32_t *s_bias, const float *s_scale, const uint32_t *v,
                                                           const QuadRes<DT> &res, const int (&px)[4], int c, int n0) {
    const int q = threadIdx.x & 3;
    uint32_t codes[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int ci = c + 8 * i + 2 * q;
        const bool in = ci < P.c_out;
        const uint2 b = *reinterpret_cast<const uint2 *>(s_bias + (ci - n0));
        const float2 sc = *reinterpret_cast<const float2 *>(s_scale + (ci - n0));
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            uint32_t a0 = v[8 * (k / 2) + 4 * i + 2 * (k % 2)], a1 = v[8 * (k / 2) + 4 * i + 2 * (k % 2) + 1];
            if constexpr (DT == XGEN_I8_I32) { a0 += b.x + res.v[4 * k + 2 * i]; a1 += b.y + res.v[4 * k + 2 * i + 1]; }
            else {
                add2(a0, a1, b.x, b.y);
                const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&res.v[2 * k + i]));
                add2(a0, a1, __float_as_uint(f.x), __float_as_uint(f.y));
            }
            if (P.relu) { a0 = tap_max<DT>(a0, 0u); a1 = tap_max<DT>(a1, 0u); }
            if (DT == XGEN_I8_I32 && P.rq_scale) {
                codes[k] |= pack_codes(tap_level(P, a0, sc.x), tap_level(P, a1, sc.y), 0, 0) << (16 * i);
                continue;
            }
            if (px[k] < 0 || !in) continue;
            const size_t at = (size_t)px[k] * P.c_out + ci;
            if constexpr (DT == XGEN_F16_F32ACC) {
                const __half2 h = __floats2half2_rn(__uint_as_float(a0), __uint_as_float(a1));
                *reinterpret_cast<uint32_t *>(static_cast<__half *>(P.y) + at) = *reinterpret_cast<const uint32_t *>(&h);
            } else *reinterpret_cast<uint2 *>(static_cast<uint32_t *>(P.y) + at) = make_uint2(a0, a1);
        }
    }
    if (DT == XGEN_I8_I32 && P.rq_scale) {
        // lane q of a quad: the codes of channels c + 4 q to c + 4 q + 3, which two lanes hold
        const int from = (threadIdx.x & 28) + 2 * (q & 1), shift = 16 * (q >> 1);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t lo = __shfl_sync(0xFFFFFFFFu, codes[k], from) >> shift & 0xFFFFu, hi = __shfl_sync(0xFFFFFFFFu, codes[k], from + 1) >> shift;
            if (px[k] >= 0 && c + 4 * q < P.c_out)
                *reinterpret_cast<uint32_t *>(static_cast<uint8_t *>(P.y) + (size_t)px[k] * P.c_out + c + 4 * q) = lo | hi << 16;
        }
    }
}

// ---- operands ------------------------------------------------------------------
// fp32 -> three bf16 parts.  A finite value above the largest bf16 becomes an infinity; every sum that its parts or those
// of an infinity or NaN go into is infinite or NaN, and computed anew (tap_repair).
__device__ __forceinline__ void split3(const uint32_t (&a)[8], uint4 &p0, uint4 &p1, uint4 &p2) {
    uint32_t o[3][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float x = __uint_as_float(a[2 * i]), y = __uint_as_float(a[2 * i + 1]);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
            o[k][i] = *reinterpret_cast<const uint32_t *>(&h);
            x -= __uint_as_float(o[k][i] << 16);
            y -= __uint_as_float(o[k][i] & 0xFFFF0000u);
        }
    }
    p0 = make_uint4(o[0][0], o[0][1], o[0][2], o[0][3]);
    p1 = make_uint4(o[1][0], o[1][1], o[1][2], o[1][3]);
    p2 = make_uint4(o[2][0], o[2][1], o[2][2], o[2][3]);
}

// The 16 bytes that begin `lead` (0 to 15) bytes into o, which goes on in b.
__device__ __forceinline__ void shift16(uint32_t (&o)[4], const uint4 &b, int lead) {
    uint32_t in[7] = {o[0], o[1], o[2], o[3], b.x, b.y, b.z};
    uint32_t over = b.w;
    if (lead & 8) {
#pragma unroll
        for (int i = 0; i < 5; ++i) in[i] = in[i + 2];
        in[5] = over;
    }
    if (lead & 4) {
#pragma unroll
        for (int i = 0; i < 5; ++i) in[i] = in[i + 1];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) o[i] = __funnelshift_r(in[i], in[i + 1], 8 * (lead & 3));
}

__device__ __forceinline__ void sts128(uint32_t dst, const uint4 &v) {
    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(dst), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// n / d with the host's multiplier (0: a range for which none is exact).
// (The division is out of line: written out at every place it made up an eighth of a kernel's code.)
static __device__ __noinline__ int div_slow(int n, int d) { return n / d; }
__device__ __forceinline__ int div_by(int n, int d, uint32_t mg) { return mg ? (int)__umulhi((uint32_t)n, mg) : div_slow(n, d); }

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

template <int DT, int STRIDE, int TAPS, int MT, bool PAIR, bool CUT, bool FUSED, bool GATHER>
__global__ void __launch_bounds__(tap_threads(DT), 1)
tap_kernel(const __grid_constant__ TapParams P, const __grid_constant__ CUtensorMap wmap, const __grid_constant__ CUtensorMap xmap) {
    using T = TapTraits<DT>;
    constexpr int PARTS = T::parts;
    constexpr bool kF32 = DT == XGEN_F32;
    constexpr int kEpiWarps = epi_warps(DT);
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    __shared__ int s_odd;                        // a sum has come out infinite or NaN
    __shared__ volatile int s_started;           // items whose x is being fetched
    __shared__ __align__(8) uint64_t s_bars[2 * kMaxA + 2 * kMaxB + 2 * kMaxAcc + 2];
    __shared__ __align__(16) uint32_t s_bias[kMaxFilterTile];
    __shared__ __align__(16) float s_scale[kMaxFilterTile];

    const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;
    const uint32_t sbase = smem_u32(smem), bars = smem_u32(s_bars);
    auto a_full = [&](int s) { return bars + 8u * s; };
    auto a_empty = [&](int s) { return bars + 8u * (kMaxA + s); };
    auto b_full = [&](int s) { return bars + 8u * (2 * kMaxA + s); };
    auto b_empty = [&](int s) { return bars + 8u * (2 * kMaxA + kMaxB + s); };
    auto acc_full = [&](int s) { return bars + 8u * (2 * kMaxA + 2 * kMaxB + s); };
    auto acc_empty = [&](int s) { return bars + 8u * (2 * kMaxA + 2 * kMaxB + kMaxAcc + s); };
    const uint32_t all_done = bars + 8u * (2 * kMaxA + 2 * kMaxB + 2 * kMaxAcc), sums_there = all_done + 8u;
    // A role that fills buffers or issues ends where a wait of its gives up: it arms no barrier, copies nothing and hands no buffer
    // on any more.  So a barrier is armed again only when what it counted has come (an arrival where none is missing is a
    // fault), whatever the others are at; they wait for what this role owes them until their own waits give up, and end too.  The
    // lanes of a warp decide together: they may see a wait give up at different places.  What has been copied is waited for
    // before the block goes.  The epilogue, which arms nothing, goes through its work on whatever there is (its residual and sums
    // leave no registers for a way out: 64 images of 28x28x128 int8 with residual 17.0 us, 18.9 with one), and the launch is reported.
    auto wait = [&](uint32_t bar, uint32_t parity) { return mbar_wait<PAIR>(bar, parity, &s_abort, P.status, P.wait_us); };
    auto wait_warp = [&](uint32_t bar, uint32_t parity) { wait(bar, parity); __syncwarp(); };
    auto agreed = [&](uint32_t bar, uint32_t parity) { return __all_sync(0xFFFFFFFFu, wait(bar, parity)) != 0; };
    // Clusters: a pair of blocks (PAIR), or the blocks (pairs) that split an item's reduction.  The even
    // block of a pair holds the barriers that say "operands are there" and "sums have been read".
    const int csize = (PAIR ? 2 : 1) * P.splits;
    const int crank = csize > 1 ? (int)(blockIdx.x % (unsigned)csize) : 0;
    const int side = PAIR ? crank & 1 : 0, rank = PAIR ? crank >> 1 : crank;
    const uint16_t both = (uint16_t)(3u << (crank & ~1));
    // Copies that barriers first, first + 1, ... of `slots` in turn count, the last of `armed`, have come.  (Bounded, for what will not
    // come; the second block's copies are counted by the first's barriers: it waits for as long as one poll lasts.)
    auto drain = [&](uint32_t first, int slots, int armed) {
        for (int q = side == 0 ? max(0, armed - slots) : armed - 1; q < armed; ++q)
            for (int it = 0; it < 100000 && !mbar_ready(first + 8u * (uint32_t)(q % slots), (uint32_t)(q / slots) & 1u); ++it) {}
    };
    auto lead = [&](uint32_t bar) { return PAIR ? cluster_addr(bar, (uint32_t)(crank & ~1)) : bar; };
    auto arrive_lead = [&](uint32_t bar) {
        if (PAIR) mbar_arrive_cluster(lead(bar));
        else mbar_arrive(bar);
    };

    asm volatile("griddepcontrol.launch_dependents;");
    if (tid == 0) {
        s_abort = 0; s_started = 0; s_odd = 0;
        for (int i = 0; i < P.a_stages; ++i) { mbar_init(a_full(i), (GATHER ? (PAIR ? 2 : 1) * kProdWarps : 1) + P.hold); mbar_init(a_empty(i), 1); }
        for (int i = 0; i < P.b_slots; ++i) { mbar_init(b_full(i), 1); mbar_init(b_empty(i), 1); }
        for (int i = 0; i < P.acc_bufs; ++i) { mbar_init(acc_full(i), 1); mbar_init(acc_empty(i), (PAIR ? 2 : 1) * 4 * (kF32 ? min(P.nt / 32, 2) : MT * (P.nt / 32))); }
        mbar_init(all_done, 1);
        mbar_init(sums_there, 1);
        if (P.splits > 1) mbar_expect_tx(sums_there, (uint32_t)(P.splits * ((8 * MT - rank + P.splits - 1) / P.splits) * P.nt * 64));
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
        if constexpr (!GATHER) {
            asm volatile("griddepcontrol.wait;" ::: "memory");
            if (warp == kEpiWarps) {
                // ---- x by tensor copies, zeros outside the image; the lanes share the copies of a stage
                // (rows one by one from one thread cost it 190 cycles each) ---------------------------------
                int s = 0, armed = 0;
                uint32_t ph = 1;
                bool alive = true;
                const int per = TAPS == 1 || !P.row_boxes ? 1 : P.rows, boxes = (TAPS == 1 || STRIDE == 1 ? 1 : 4) * per;
                const int step = (P.row_boxes ? 1 : P.rows) * P.pitch * 128;
                for (int item = item0; item < P.items && alive; item += item_step) {
                    const TapItem t = tap_item<MT, PAIR>(P, item, side);
                    if (lane == 0) s_started = s_started + 1;
                    for (int ks = k0; ks < k1; ++ks) {
                        alive = agreed(a_empty(s), ph);
                        if (!alive) break;
                        ++armed;
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
                if (!alive) drain(a_full(0), P.a_stages, armed);
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
                    if (s_started <= done) break;
                    fetch(item + item_step);
                }
            }
        } else {
            // ---- x through the producer warps ------------------------------------------------------
            // Loads that were waited for where they are used held a stage to two trips to memory: 3300 cycles of 128 x 32
            // fp32, 8000 of 128 x 64 fp16 in odd rows, for 580 and 260 of matrix instructions.
            const int pt = tid - kEpiWarps * 32, own = pt >> 5;
            const char *const x = static_cast<const char *>(P.x);
            constexpr int kPiece = kF32 ? 32 : 16;       // bytes of a piece: a thread's, of one plane and pixel
            // a thread's pieces: always of the same plane of a stage, of every q_step-th pixel
            const int pl = pt & ((1 << P.row_log) - 1), q0 = pt >> P.row_log, q_step = kProdThreads >> P.row_log;
            const size_t row_bytes = (size_t)P.c_in * T::xb;
            auto table = [&](int tab) { return reinterpret_cast<int *>(smem + P.tab_off) + tab * P.pixels; };
            // Where the loads are, a batch (of all threads' pieces) or some stages ahead of their use, and the operands made.
            int item_f = item0, ks_f = k0, tab_f = 0;
            int row_f = 0;                                            // product: the item's first row
            int item = item0, ks = k0, s = 0;
            uint32_t ph = 1;
            auto begin = [&]() {                         // a new item: where its pixels come from, those of this warp
                const TapItem t = tap_item<MT, PAIR>(P, item_f, side);
                row_f = t.v0 * 8;
                if (TAPS == 9) {
                    int *const pix = table(tab_f);
                    const int g_log = 5 - P.row_log;
#pragma unroll 1
                    for (int i = lane;; i += 32) {
                        const int p = (i >> g_log) * q_step + (own << g_log) + (i & ((1 << g_log) - 1));
                        if (p >= P.pixels) break;
                        const int at = tap_source<STRIDE, TAPS>(P, t, p);
                        pix[p] = kF32 || at < 0 ? at : (int)((uint32_t)at * (uint32_t)row_bytes);      // fp16, int8: bytes from x on
                    }
                    __syncwarp();
                }
                if (item_f == item0) asm volatile("griddepcontrol.wait;" ::: "memory");
            };
            if constexpr (kF32) {
            // fp32: a batch is loaded into registers while the one before is split into its parts.  (Through shared
            // memory, like the rows below, it cost room for stages and weights and as many instructions again.)
            constexpr int U = 4;
            int q_f = 0, q = 0;                          // pixels of the stage that the batches before have taken
            auto load = [&](uint32_t (&v)[U][8]) {
                if (item_f >= P.items) return;
                if (ks_f == k0 && q_f == 0) begin();
                const int *const pix = table(tab_f);
                const int npl = min(P.pl, planes - ks_f * P.pl), c = (ks_f * P.pl + pl) * T::cpp, left = P.c_in - c;      // channels there are
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int qu = q_f + q0 + u * q_step;
                    const int px = qu >= P.pixels || pl >= npl ? -1 : TAPS == 9 ? pix[qu] : (int64_t)row_f + qu < P.npix ? row_f + qu : -1;
                    const float *const src = reinterpret_cast<const float *>(x + (size_t)max(px, 0) * row_bytes) + c;
                    const int n = px < 0 ? 0 : left;
                    if (P.vec_x) {
                        const uint4 z = make_uint4(0u, 0u, 0u, 0u);
                        const uint4 lo = n > 0 ? __ldg(reinterpret_cast<const uint4 *>(src)) : z, hi = n > 4 ? __ldg(reinterpret_cast<const uint4 *>(src) + 1) : z;
                        v[u][0] = lo.x; v[u][1] = lo.y; v[u][2] = lo.z; v[u][3] = lo.w;
                        v[u][4] = hi.x; v[u][5] = hi.y; v[u][6] = hi.z; v[u][7] = hi.w;
                    } else {
#pragma unroll
                        for (int e = 0; e < 8; ++e) v[u][e] = n > e ? __ldg(reinterpret_cast<const uint32_t *>(src) + e) : 0u;
                    }
                }
                q_f += U * q_step;
                if (q_f >= P.pixels) {
                    q_f = 0;
                    if (++ks_f == k1) { ks_f = k0; item_f += item_step; tab_f ^= 1; }
                }
            };
            auto make = [&](const uint32_t (&v)[U][8]) {
                if (q == 0 && !agreed(a_empty(s), ph)) {
                    item = P.items;
                    return;
                }
                const uint32_t dst = sbase + (uint32_t)(s * P.a_bytes + pl * P.plane_pitch);
                const bool some = pl < min(P.pl, planes - ks * P.pl);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int qu = q + q0 + u * q_step;
                    if (qu >= P.pixels || !some) continue;
                    uint4 p0, p1, p2;
                    split3(v[u], p0, p1, p2);
                    const uint32_t d = dst + (uint32_t)(qu * 16);
                    sts128(d, p0);
                    sts128(d + a_part, p1);
                    sts128(d + 2 * a_part, p2);
                }
                q += U * q_step;
                if (q < P.pixels) return;
                q = 0;
                fence_async_proxy();
                __syncwarp();
                if (lane == 0) arrive_lead(a_full(s));
                if (++s == P.a_stages) { s = 0; ph ^= 1u; }
                if (++ks == k1) { ks = k0; item += item_step; }
            };
            uint32_t v0[U][8], v1[U][8];
            load(v0);
#pragma unroll 1
            while (item < P.items) {
                load(v1);
                make(v0);
                if (item >= P.items) break;
                load(v0);
                make(v1);
            }
            } else {
            // fp16, int8: a stage's rows (or a part of them: raw_px, a multiple of q_step, where a stage's do not fit) are
            // copied as they lie in memory (the aligned 16-byte pieces that hold a wanted byte, zeros outside the image)
            // into one of raw_slots buffers, raw_slots - 1 of them ahead of their use, and shifted
            // into place from there.  A warp copies and shifts the same pixels, so warps need not meet.
            // Pieces are taken U at a time.  (The large tiles of stride 2 four: with two a stage waited for the latency of its
            // shared memory, 32 images of 28x28x503 -> 256 fp16 60.4 us, 57.4 now; four that all lie outside the image, as most do
            // of a tile over small images, are neither copied nor shifted.)
            constexpr int U = STRIDE == 2 ? 4 : 2;
            constexpr uint32_t kNone = 0xFFFFFFFFu;      // (bytes from x on: it has fewer than 2^31 elements)
            auto sources = [&](uint32_t (&px)[U], const int *pix, int first, int q, int end) {
                uint32_t all = kNone;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int qu = STRIDE == 2 ? q + u * q_step : min(q + u * q_step, end - 1);
                    if (STRIDE == 2 && qu >= end) px[u] = kNone;       // (its table entry may be another warp's, and not there yet)
                    else px[u] = TAPS == 9 ? (uint32_t)pix[qu] : (int64_t)first + qu < P.npix ? (uint32_t)(first + qu) * (uint32_t)row_bytes : kNone;
                    all &= px[u];
                }
                return STRIDE == 2 && all == kNone;
            };
            int slot_f = 0, slot = 0, tab = 0, row = 0;
            int part_f = 0, part = 0;                    // first pixel of the part
            const int ahead = P.raw_slots - 1;
#pragma unroll 1
            for (int turn = -ahead; item < P.items; ++turn) {
                if (item_f < P.items) {
                    if (ks_f == k0 && part_f == 0) begin();
                    const int *const pix = table(tab_f);
                    const int end = min(part_f + P.raw_px, P.pixels);
                    const int npl = min(P.pl, planes - ks_f * P.pl), want = min(npl * T::cpp, P.c_in - ks_f * P.pl * T::cpp) * T::xb;
                    uint32_t d = sbase + (uint32_t)(P.raw_off + slot_f * P.raw_bytes + q0 * P.raw_pitch + pl * kPiece);
                    const char *const at = x + (size_t)(ks_f * P.pl * T::cpp) * T::xb;
                    if (pl < npl) {
#pragma unroll 1
                        for (int q = part_f + q0; q < end; q += U * q_step, d += (uint32_t)(U * q_step * P.raw_pitch)) {
                            uint32_t px[U];
                            if (sources(px, pix, row_f, q, end)) continue;
#pragma unroll
                            for (int u = 0; u < U; ++u) {
                                if (q + u * q_step >= end) break;
                                const char *const src = at + (px[u] == kNone ? 0u : px[u]);
                                const int lead = P.vec_x ? 0 : (int)(reinterpret_cast<uintptr_t>(src) & 15);
                                const int left = px[u] == kNone ? 0 : lead + want - pl * kPiece;          // wanted bytes from this piece on
                                const char *const from = src - lead;
                                const uint32_t to = d + (uint32_t)(u * q_step * P.raw_pitch);
                                copy16(to, from + (left > 0 ? pl * kPiece : 0), left > 0 ? 16u : 0u);
                                if (!P.vec_x && pl == npl - 1) copy16(to + kPiece, from + (left > kPiece ? (pl + 1) * kPiece : 0), left > kPiece ? 16u : 0u);
                            }
                        }
                    }
                    if (++slot_f == P.raw_slots) slot_f = 0;
                    part_f = end;
                    if (part_f == P.pixels) {
                        part_f = 0;
                        if (++ks_f == k1) {
                            ks_f = k0;
                            item_f += item_step;
                            if (++tab_f == P.raw_slots) tab_f = 0;
                        }
                    }
                }
                copy_commit();
                if (turn < 0) continue;
                if (ahead == 0) copy_wait<0>();
                else if (ahead == 1) copy_wait<1>();
                else if (ahead == 2) copy_wait<2>();
                else copy_wait<3>();
                if (part != 0) __syncwarp();
                else if (!agreed(a_empty(s), ph)) break;
                const int end = min(part + P.raw_px, P.pixels);
                const unsigned char *const raw = smem + P.raw_off + slot * P.raw_bytes + pl * kPiece;
                const uint32_t dst = sbase + (uint32_t)(s * P.a_bytes);
                const int npl = min(P.pl, planes - ks * P.pl), left = P.c_in - (ks * P.pl + pl) * T::cpp;      // channels there are from this piece on
                if (TAPS == 1 && ks == k0) row = tap_item<MT, PAIR>(P, item, side).v0 * 8;
                if (pl < npl) {
                    const int *const pix = table(tab);
                    const uint32_t at15 = (uint32_t)reinterpret_cast<uintptr_t>(x) + (uint32_t)(ks * P.pl * T::cpp * T::xb);
#pragma unroll 1
                    for (int q = part + q0; q < end; q += U * q_step) {
                        uint32_t px[U], v[U][4];
                        if (sources(px, pix, row, q, end)) {
#pragma unroll
                            for (int u = 0; u < U; ++u) {
                                const int qu = q + u * q_step;
                                if (qu < end) sts128(dst + (uint32_t)(qu * 128 + ((pl ^ (qu & 7)) << 4)), make_uint4(0u, 0u, 0u, 0u));
                            }
                            continue;
                        }
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            const uint4 *const in = reinterpret_cast<const uint4 *>(raw + (min(q + u * q_step, end - 1) - (STRIDE == 2 ? part : 0)) * P.raw_pitch);
                            const uint4 a = in[0];
                            v[u][0] = a.x; v[u][1] = a.y; v[u][2] = a.z; v[u][3] = a.w;
                            if (!P.vec_x) shift16(v[u], in[1], (int)(at15 + px[u]) & 15);
                        }
                        if (!P.vec_x && left < T::cpp) {       // (0 or less: a plane that fills a pair up)
#pragma unroll
                            for (int u = 0; u < U; ++u)
#pragma unroll
                                for (int e = 0; e < 4; ++e) {
                                    const int bytes = left * T::xb - 4 * e;
                                    if (bytes < 4) v[u][e] = bytes <= 0 ? 0u : v[u][e] & ((1u << (8 * bytes)) - 1u);
                                }
                        }
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            const int qu = q + u * q_step;
                            if (qu < end) sts128(dst + (uint32_t)(qu * 128 + ((pl ^ (qu & 7)) << 4)), make_uint4(v[u][0], v[u][1], v[u][2], v[u][3]));
                        }
                    }
                }
                if (++slot == P.raw_slots) slot = 0;
                part = end;
                if (part < P.pixels) {
                    __syncwarp();                        // (the buffer is filled anew)
                    continue;
                }
                part = 0;
                fence_async_proxy();
                __syncwarp();
                if (lane == 0) arrive_lead(a_full(s));
                if (++s == P.a_stages) { s = 0; ph ^= 1u; }
                if (++ks == k1) {
                    ks = k0;
                    item += item_step;
                    if (++tab == P.raw_slots) tab = 0;
                }
            }
            copy_wait<0>();
            }
        }
    } else if (warp == kEpiWarps + kProdWarps) {
        // ---- matrix instructions: one thread, which also waits (and leaves where a wait gives up).  Three taps are unrolled and share a barrier, and
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
            bool ready = mbar_test<PAIR>(b_full(0), 0), look = true;           // look: weights may still be on their way
            // a tap's first entry is that of its row and that of its column of taps
            const uint32_t row0 = (uint32_t)P.tap_start[0] * a_px, row1 = TAPS == 1 ? 0u : (uint32_t)P.tap_start[3] * a_px, row2 = TAPS == 1 ? 0u : (uint32_t)P.tap_start[6] * a_px;
            const uint32_t col0 = 0u, col1 = TAPS == 1 ? 0u : (uint32_t)(P.tap_start[1] - P.tap_start[0]) * a_px, col2 = TAPS == 1 ? 0u : (uint32_t)(P.tap_start[2] - P.tap_start[0]) * a_px;
            for (int item = item0; item < P.items; item += item_step) {
                for (int ks = k0; ks < k1; ++ks) {
                    if ((kF32 || (CUT ? run == 0 : ks == k0)) && !wait(acc_empty(buf), phc)) goto gone;
                    if (!wait(a_full(s), pha)) goto gone;
                    tc_fence_after();
                    const int kk_n = min(P.pl, planes - ks * P.pl) / 2;
                    const uint32_t d = tmem + (uint32_t)buf * (uint32_t)(MT * P.nt);
                    const uint32_t dc = d + (uint32_t)(P.acc_bufs * P.nt);      // fp32: the small products (as many buffers, behind those of the sums)
                    uint32_t bt = bs;
#pragma unroll (kF32 ? 1 : 3)
                    for (int t0 = 0; t0 < TAPS; t0 += 3) {
                    const uint32_t row = as + (t0 == 0 ? row0 : t0 == 3 ? row1 : row2);
#pragma unroll
                    for (int t1 = 0; t1 < (TAPS == 1 ? 1 : 3); ++t1) {
                        const int tap = t0 + t1;
                        const bool last = P.tap_group == 1 || t1 == 2;
                        if (look) {
                            if ((P.tap_group == 1 || t1 == 0) && !ready) {
                                if (!mbar_wait_long<PAIR>(b_full(b), P.resident ? 0u : phb, &s_abort, P.status, P.wait_us)) goto gone;
                            }
                            if (last) {                     // (of its slot: look at the next one)
                                const bool wrap = b + 1 == P.b_slots;
                                ready = mbar_test<PAIR>(b_full(wrap ? 0 : b + 1), P.resident ? 0u : wrap ? phb ^ 1u : phb);
                            }
                        }
                        uint32_t ak = row + (t1 == 0 ? col0 : t1 == 1 ? col1 : col2), bk = bt;
                        uint32_t first_s = tap > 0 ? 1u : 0u;                               // 0: the first of the stage
                        uint32_t first_i = first_s | ((CUT ? run > 0 : ks > k0) ? 1u : 0u); // 0: the first of the item (CUT: of its part)
                        auto k_step = [&]() {
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
                            ak += a_k; bk += b_k; first_s = 1u; first_i = 1u;
                        };
                        if (kF32) {
#pragma unroll
                            for (int kk = 0; kk < (TAPS == 9 ? 2 : 4); ++kk)
                                if (kk < kk_n) k_step();
                        } else {
                            k_step();
                            if (kk_n > 1) {
                                k_step();
                                if (kk_n > 2) {
                                    k_step();
                                    if (kk_n > 3) k_step();
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
                if (P.resident) look = false;
            }
        gone:
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
                        if (issued >= P.b_slots && !wait(b_empty(b), ph)) goto last;
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
        last:
            // Nothing may land in shared memory after this block has gone (the wait for it may have given up).
            if (side == 0 || *(volatile int *)&s_abort) drain(b_full(0), P.b_slots, issued);
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
        // A warp's share: a quarter of the lanes, one of the tiles, every kGroups-th chunk of 32 filters, counted on
        // from item to item, so that all groups of warps have work where a tile has fewer chunks than there are groups
        // (a chunk takes one some 3000 cycles from the wait to the last store, most of it latency: one item after the
        // other held 117 x 66x66x16 -> 16, fp16, to 28.6 us).
        constexpr int kGroups = kEpiWarps / 4 / MT;
        const int quarter = warp & 3, sub = (warp >> 2) % MT, group = (warp >> 2) / MT;
        const int chunks = P.nt / 32;
        const uint32_t lanes = (uint32_t)quarter << 21;
        const int m = quarter * 32 + lane;                       // pixel of the 128
        // Sums on their way out where they do not go straight from their lanes: the warp's 32 pixels x 16 filters,
        uint32_t *const st = reinterpret_cast<uint32_t *>(smem + P.stage_off + warp * kStageBytes);
        uint32_t *const st_own = st + lane * kStagePitch;
        // or, where a reduction is split, into the buffers of operands that are done with, [unit of 16 pixels][chunk]
        // [pixel][128 bytes, 16-byte pieces swizzled by the pixel], from where a copy takes such a 2 KB piece to the
        // block of the cluster that adds the unit up, whose barrier counts the bytes.  (Stored there lane by lane, 16 bytes
        // apart by rows, 128 x 128 sums took 5200 cycles to leave and as long again till the cluster had met.)
        const int unit = sub * 8 + m / 16, units_all = (8 * MT + P.splits - 1) / P.splits;
        uint32_t far = 0, far_bar = 0;
        if (P.splits > 1) {
            const int adder = unit % P.splits;
            far = cluster_addr(sbase + P.sum_off + (uint32_t)((rank * units_all + unit / P.splits) * chunks) * 2048u, (uint32_t)(PAIR ? 2 * adder + side : adder));
            far_bar = cluster_addr(sums_there, (uint32_t)(PAIR ? 2 * adder + side : adder));
        }
        int buf = 0, next = group;                               // next: the group's next chunk, counted from this item's first
        uint32_t ph = 0;
        auto advance = [&]() {
            if (++buf == P.acc_bufs) { buf = 0; ph ^= 1u; }
        };
        // A group that leaves out items must not miss a whole turn of the accumulators, or it takes the end of one turn for that
        // of the next: with a buffer an item (fp16, int8) the items that a group leaves out are always the same buffers'; fp32, with a
        // buffer a stage, where an item has two at most.  (CUT: the chunks' sums wait in tensor memory for their group.)
        const bool turn = !CUT && (!kF32 || k1 - k0 <= 2);
        for (int item = item0; item < P.items; item += item_step, next = turn ? next - chunks : group) {
            if (next >= chunks) {
                for (int ks = kF32 || CUT ? k0 : k1 - 1; ks < k1; ks += CUT ? P.cut : 1) advance();
                continue;
            }
            const TapItem t = tap_item<MT, PAIR>(P, item, side);
            const TapPixel at = tap_pixel<TAPS>(P, t, sub * 128 + m);
            const int pix = at.pix, out = at.out;
            if (P.staged && P.splits == 1) { st_own[16] = (uint32_t)pix; st_own[17] = (uint32_t)out; }
            const bool quad = FUSED && !kF32 && P.residual && !P.pool && !P.staged && P.splits == 1;
            int px4[4];
            if (FUSED && !kF32) {
#pragma unroll
                for (int k = 0; k < 4; ++k) px4[k] = __shfl_sync(0xFFFFFFFFu, pix, 16 * (k / 2) + 8 * (k % 2) + lane / 4);
            }
            // 32 sums of this lane's pixel, from column c of the tile on
            auto finish = [&](uint32_t (&r)[32], int c) {
                if (P.splits > 1) {
                    const uint32_t piece = sbase + (uint32_t)(unit * chunks + c / 32) * 2048u;
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        sts128(piece + (uint32_t)((m & 15) * 128 + ((q ^ (m & 7)) << 4)), make_uint4(r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]));
                    fence_async_proxy();
                    __syncwarp();
                    if ((lane & 15) == 0) copy_cluster(far + (uint32_t)(c / 32) * 2048u, piece, 2048u, far_bar);
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
            // A chunk (fp32: all of the warp's) is in registers.
            auto release = [&]() {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) arrive_lead(acc_empty(buf));
            };
            if constexpr (kF32) {
                uint32_t sum[2][32];                 // chunks `next` and `next` + kGroups
#pragma unroll
                for (int i = 0; i < 64; ++i) sum[i / 32][i % 32] = 0u;
                for (int ks = k0; ks < k1; ++ks) {
                    wait_warp(acc_full(buf), ph);
                    tc_fence_after();
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const int q = next + h / 2 * kGroups;
                        if (q < chunks) {
                            const uint32_t ta = tmem + lanes + (uint32_t)(buf * P.nt + 32 * q + h % 2 * 16);
                            uint32_t a[16], b[16];
                            tmem_ld16(ta, a);
                            tmem_ld16(ta + P.acc_bufs * P.nt, b);
                            tmem_wait_ld();
#pragma unroll
                            for (int i = 0; i < 16; i += 2) {
                                add2(a[i], a[i + 1], b[i], b[i + 1]);
                                add2(sum[h / 2][h % 2 * 16 + i], sum[h / 2][h % 2 * 16 + i + 1], a[i], a[i + 1]);
                            }
                        }
                    }
                    release();
                    advance();
                }
#pragma unroll 1
                for (; next < chunks; next += kGroups) {
                    finish(sum[0], 32 * next);
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
                        if (last && !quad) finish(r, 32 * q);
                        else {
                            tmem_st16(tt + 32 * q, r);
                            tmem_st16(tt + 32 * q + 16, r + 16);
                            tmem_wait_st();
                        }
                        release();
                        if (last && quad) {          // (read again in the quad layout)
                            if (!all_finite(r)) s_odd = 1;
#pragma unroll 1
                            for (int c = n0 + 32 * q; c < min(n0 + 32 * q + 32, P.c_out); c += 16) {
                                QuadRes<DT> res;
                                quad_residual<DT>(P, res, px4, c);
                                uint32_t v[16];
                                tmem_ld_quad(tt + (uint32_t)(c - n0), v);
                                tmem_wait_ld();
                                tap_quad<DT>(P, s_bias, s_scale, v, res, px4, c, n0);
                            }
                        }
                    }
                    advance();
                }
            } else if (quad) {
                const uint32_t ta = tmem + lanes + (uint32_t)((buf * MT + sub) * P.nt);
                bool first = true;
#pragma unroll 1
                for (; next < chunks; next += kGroups) {
                    const int c = n0 + 32 * next;
                    QuadRes<DT> res0, res1;
                    quad_residual<DT>(P, res0, px4, c);
                    quad_residual<DT>(P, res1, px4, c + 16);
                    if (first) { wait_warp(acc_full(buf), ph); tc_fence_after(); first = false; }
                    uint32_t v[16];
                    tmem_ld_quad(ta + 32 * next, v);
                    tmem_wait_ld();
                    if (DT != XGEN_I8_I32 && !all_finite(v)) s_odd = 1;
                    if (c < P.c_out) tap_quad<DT>(P, s_bias, s_scale, v, res0, px4, c, n0);
                    tmem_ld_quad(ta + 32 * next + 16, v);
                    tmem_wait_ld();
                    release();
                    if (DT != XGEN_I8_I32 && !all_finite(v)) s_odd = 1;
                    if (c + 16 < P.c_out) tap_quad<DT>(P, s_bias, s_scale, v, res1, px4, c + 16, n0);
                }
                advance();
            } else {
                wait_warp(acc_full(buf), ph);
                tc_fence_after();
                const uint32_t ta = tmem + lanes + (uint32_t)((buf * MT + sub) * P.nt);
#pragma unroll 1
                for (; next < chunks; next += kGroups) {
                    uint32_t r[32];
                    tmem_ld16(ta + 32 * next, r);
                    tmem_ld16(ta + 32 * next + 16, r + 16);
                    tmem_wait_ld();
                    release();
                    finish(r, 32 * next);
                }
                advance();
            }
        }
    }

    // ---- split items: every block adds up its share of the pixels, in the order of the sources -------
    if (P.splits > 1) {
        constexpr int kAdders = (kEpiWarps + kProdWarps) * 32;
        __syncwarp();
        cluster_arrive();                // what this thread sends is on its way
        if (tid < kAdders) wait_warp(sums_there, 0);
        cluster_wait();
        // (only where a wait gave up is there still something to come: nothing may land in a block that has gone)
        for (int it = 0; it < 1000000 && !mbar_ready(sums_there, 0); ++it) {}
        __syncwarp();
        cluster_arrive();                // all that is sent here has come
        if (tid < kAdders && !s_abort) {
            const TapItem t = tap_item<MT, PAIR>(P, item0, side);
            const int groups = P.nt / 8, chunks = P.nt / 32;
            const bool pool = FUSED && P.pool;
            // units of two rows of eight pixels go round the blocks; a thread takes 8 channels of one (pooled) pixel
            const int units_all = (8 * MT + P.splits - 1) / P.splits, units = (8 * MT - rank + P.splits - 1) / P.splits;
            const int per_unit = (pool ? 4 : 16) * groups, source = units_all * chunks * 2048;
#pragma unroll 1
            for (int w = tid; w < units * per_unit; w += kAdders) {
                const int u = w / per_unit, wu = w - u * per_unit, row = wu / groups, g = wu - row * groups;
                const int c0 = n0 + 8 * g, in_unit = pool ? 2 * row : row;
                const TapPixel px = tap_pixel<TAPS>(P, t, 16 * (rank + u * P.splits) + in_unit);
                if (px.pix < 0 || c0 >= P.c_out) continue;
                uint32_t best[8];
#pragma unroll 1
                for (int q = 0; q < (pool ? 4 : 1); ++q) {
                    const int r16 = in_unit + (q & 1) + (q >> 1) * 8;             // pixel of the unit
                    const unsigned char *own = smem + P.sum_off + (u * chunks + g / 4) * 2048 + r16 * 128;
                    const int first = ((2 * (g & 3)) ^ (r16 & 7)) * 16, second = first ^ 16;
                    uint32_t v8[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) v8[i] = 0;
#pragma unroll 4
                    for (int r = 0; r < P.splits; ++r, own += source) {
                        const uint4 a = *reinterpret_cast<const uint4 *>(own + first), b = *reinterpret_cast<const uint4 *>(own + second);
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
    // nobody leaves while another may still use its memory, or while what it has sent is on its way
    if (P.splits > 1) cluster_wait();
    else if (PAIR) cluster_meet();
    tc_fence_before();
    __syncthreads();
    if (warp == kEpiWarps + kProdWarps) tmem_free<PAIR>(tmem, (uint32_t)P.tmem_cols);
    if (DT != XGEN_I8_I32 && s_odd) tap_repair<DT, STRIDE, TAPS, MT, PAIR>(P);
}

// ---- instances -------------------------------------------------------------------
// An instance carries the code of its own way only, the fused operators or not, x through the producer warps or by
// tensor copies: with all of it in one kernel an fp16 layer's code was 160 KB, which the instruction caches do not hold (a
// fifth of all stalls), and the first pass through it took a short launch several microseconds.
template <int DT, int STRIDE, int TAPS, int MT, bool PAIR, bool CUT> static const void *tap_pick(bool fused, bool gather) {
    constexpr bool F = TAPS == 9, G = DT == XGEN_F32;         // (what there is no instance of is never asked for)
    if (fused) return gather ? (const void *)tap_kernel<DT, STRIDE, TAPS, MT, PAIR, CUT, F, true> : (const void *)tap_kernel<DT, STRIDE, TAPS, MT, PAIR, CUT, F, G>;
    return gather ? (const void *)tap_kernel<DT, STRIDE, TAPS, MT, PAIR, CUT, false, true> : (const void *)tap_kernel<DT, STRIDE, TAPS, MT, PAIR, CUT, false, G>;
}
template <int DT, int STRIDE, int TAPS, bool CUT> static const void *tap_pick_tile(int mt, bool pair, bool fused, bool gather) {
    constexpr int M2 = DT == XGEN_F32 ? 1 : 2;
    if (mt == 2) return pair ? tap_pick<DT, STRIDE, TAPS, M2, true, CUT>(fused, gather) : tap_pick<DT, STRIDE, TAPS, M2, false, CUT>(fused, gather);
    return pair ? tap_pick<DT, STRIDE, TAPS, 1, true, CUT>(fused, gather) : tap_pick<DT, STRIDE, TAPS, 1, false, CUT>(fused, gather);
}
template <int DT, bool CUT> static const void *tap_pick_layer(int stride, int taps, int mt, bool pair, bool fused, bool gather) {
    if constexpr (DT != XGEN_I8_I32)
        if (taps == 1) return tap_pick_tile<DT, 1, 1, CUT>(mt, pair, fused, gather);
    return stride == 1 ? tap_pick_tile<DT, 1, 9, CUT>(mt, pair, fused, gather) : tap_pick_tile<DT, 2, 9, CUT>(mt, pair, fused, gather);
}

}  // namespace patconv
