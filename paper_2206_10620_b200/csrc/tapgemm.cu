// The matrix path's host side: the weight image, plans, launches (the kernels: tapgemm_kernel.cuh).
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstring>
#include <mutex>
#include <utility>
#include <vector>

#include "tapgemm_kernel.cuh"

namespace patconv {

// The instances (tapgemm_f32.cu and so on).
const void *tap_kernel_f32(int stride, int taps, int mt, bool pair, bool fused, bool gather);
const void *tap_kernel_f16(int stride, int taps, int mt, bool pair, bool fused, bool gather);
const void *tap_kernel_f16_cut(int stride, int taps, int mt, bool pair, bool fused, bool gather);
const void *tap_kernel_i8(int stride, int taps, int mt, bool pair, bool fused, bool gather);

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
// A pixel's planes of a stage, as a power of two.
static int row_log(int pl) { return pl <= 2 ? 1 : pl <= 4 ? 2 : 3; }

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
static const void *tap_kernel_of(xgen_dtype dt, int stride, int taps, int mt, bool pair, bool cut, bool fused, bool gather) {
    if (cut) return tap_kernel_f16_cut(stride, taps, mt, pair, fused, gather);
    return dt == XGEN_F32 ? tap_kernel_f32(stride, taps, mt, pair, fused, gather) : dt == XGEN_F16_F32ACC ? tap_kernel_f16(stride, taps, mt, pair, fused, gather)
                                                                                                       : tap_kernel_i8(stride, taps, mt, pair, fused, gather);
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
    const void *kern = tap_kernel_of(XGEN_F16_F32ACC, 1, 9, 1, false, false, false, false);
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
    const bool swizzled = dt != XGEN_F32, copied = swizzled && (size_t)tw.c_in * xb % 16 == 0 && !s.gather;
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
                    // (no plan whose instructions alone take as long as the best so far: 512 -> 512 at 14x14 fp32 is planned in 24 us, 57 without)
                    const double kk = (double)tw.planes / p.stages / 2, taps = tw.taps, per_tap = kk * mt * prod;
                    const double mma = taps * std::max(per_tap * p.nt / 2.0, 90.0 + 46.0 * per_tap);
                    if (3500.0 + (double)waves * p.per_split * mma >= best.cycles * 0.999) continue;
                    const size_t sums = sp > 1 ? (size_t)sp * ((8 * mt + sp - 1) / sp) * 64 * p.nt : s.staged ? (size_t)epi_warps(dt) * kStageBytes : 0;
                    const int64_t uses = (sp == 1 ? waves : 1) * p.per_split;      // stages one block goes through
                    // Shared memory: two tiles of x (more for a plain product, whose stages are short), the rest
                    // weights, by three taps if at least three such slots fit.  fp16 and int8 rows that the producer warps
                    // shift into place: up to two stages of them on their way (three of a product).  The tiles of stride 2 (612
                    // pixels) leave no room for those: quarters or eighths of a stage, or one tile of x, whatever
                    // is weighed best, so that there is a plan whatever else takes room.  (Without one 32 images of 56x56x67 -> 93
                    // fp16 took 176 us on the command stream, 40.6 now; 28x28x503 -> 256 1227, 57; int8 168, 20 and 1092, 33.)
                    size_t tables = sums;
                    const int raw_top = copied || dt == XGEN_F32 ? 0 : (int)std::min<int64_t>(uses, tw.taps == 1 ? 4 : 3);
                    const int two = (int)std::min<int64_t>(2, uses);
                    auto place = [&](int least_a) {
                        p.raw_pitch = p.pl * 16 + 16;
                        p.raw_bytes = p.raw_px * p.raw_pitch;
                        p.table_bytes = tw.taps == 1 || copied ? 0 : ((dt == XGEN_F32 ? 2 : p.raw_slots) * pixels * 4 + 127) / 128 * 128;
                        tables = sums + p.table_bytes + (size_t)p.raw_slots * p.raw_bytes;
                        for (p.tap_group = tw.taps == 1 ? 1 : 3; p.tap_group >= 1; p.tap_group -= 2) {
                            p.b_bytes = p.tap_group * p.pl * parts * p.nt * 16 / ways;
                            const int all_b = p.per_split * tw.taps / p.tap_group;
                            for (p.a_stages = (int)std::min<int64_t>(uses, tw.taps == 1 ? kMaxA : 2); p.a_stages >= least_a; --p.a_stages) {
                                const size_t left_a = (size_t)p.a_stages * p.a_bytes + tables;
                                if (left_a >= (size_t)kTapSmemMax) continue;
                                const int room = (int)std::min<size_t>(kMaxB, ((size_t)kTapSmemMax - left_a) / p.b_bytes);
                                p.resident = all_b <= room;
                                p.b_slots = std::min(room, all_b);
                                if (p.b_slots >= std::min(all_b, 3)) return true;
                            }
                        }
                        return false;
                    };
                    // What that makes of the time: the cost model, in cycles.
                    auto weigh = [&](bool large) {
                        // (the operands' buffers hold a block's own sums before they leave)
                        p.operands = std::max(p.a_stages * p.a_bytes + p.b_slots * p.b_bytes, sp > 1 ? 512 * mt * p.nt : 0);
                        p.smem = (size_t)p.operands + tables;
                        if (p.smem > (size_t)kTapSmemMax) return;
                        p.acc_bufs = p.cut ? (3 * mt * p.nt <= 512 ? 2 : 1) : (dt == XGEN_F32 ? 2 : 1) * 4 * mt * p.nt <= 512 ? 4 : dt == XGEN_F32 || 2 * mt * p.nt <= 512 ? 2 : 1;
                        const int cols = (dt == XGEN_F32 ? 2 * p.acc_bufs : p.acc_bufs + (p.cut ? 1 : 0)) * mt * p.nt;
                        for (p.tmem_cols = 32; p.tmem_cols < cols;) p.tmem_cols *= 2;
                        // Cycles of a stage: the matrix instructions (nt / 2 each; 46 to issue one and 90 for a tap), or
                        // what they and the copies move through shared memory at 128 bytes a cycle (128 rows of x,
                        // the block's filters), or what comes from L2.  A pair starts and ends later: 4000 cycles where it
                        // halves much (fp32: three parts of weights; stride 2: single taps in the slots), else 6000
                        // (256 -> 256 at 14x14, batch 32, fp16: 12.8 us as pairs, 11.7 without); the
                        // short stages of a product wait 300 cycles for its other block (1842 filters x 5421 rows,
                        // fp32: 77 us as pairs, 57 us without).
                        const double b_stage = taps * kk * 2 * parts * p.nt * 16.0 / ways, b_moved = p.resident && sp == 1 ? b_stage / waves : b_stage;
                        const double x_moved = (double)pixels * kk * 2 * cpp * xb, a_stage = (double)p.a_bytes * (swizzled ? 1 : 2);
                        const double instr = taps * per_tap;
                        const double shared = (instr * (4096.0 + p.nt * 32.0 / ways) + b_moved + a_stage) / 128.0;
                        const double move = (x_moved + b_moved) / 40.0 + (copied && p.straddle ? 60.0 * p.rows * (s.stride == 1 ? 1 : 4) : 0.0) * 0.5;
                        // cycles of the producer warps for a piece; no stage of x ahead
                        const double make = copied ? 0.0 : (double)pixels * kk * 2 * (swizzled ? 2.0 : 3.0) + (swizzled && p.raw_slots == 1 ? 1200.0 : 0.0);
                        const double ends = 250.0 + 40.0 * taps / p.tap_group + (p.pair && tw.taps == 1 ? 300.0 : 0.0);
                        const double out = (double)mt * 128 * p.nt * yb / 24.0;
                        // (one accumulator that is cut waits for its sums to be added)
                        const double cuts = p.cut && p.acc_bufs == 1 ? (p.per_split - 1) / p.cut * 1500.0 : 0.0;
                        const double item = p.per_split * (std::max(std::max(mma, shared), std::max(move, make)) + ends) + cuts;
                        double run = waves * std::max(item, sp == 1 && p.acc_bufs >= 2 ? out : 0.0), c = 3500.0 + (p.pair ? dt == XGEN_F32 || s.stride == 2 ? 4000.0 : 6000.0 : 0.0);
                        if (large) {                                   // (rows shifted into place at stride 2)
                            // The first stage is made before anything else happens; a piece takes the producer warps 2.2 cycles, one
                            // outside the image 0.8; x takes 1500 cycles to come, of which the parts ahead hide a share, and so
                            // does a slot of weights; one tile of x is only copied while the instructions read it; the blocks
                            // of a split begin anew in every wave.
                            const double full = std::min(1.0, 1.15 * s.n * s.h * s.w / ((double)tiles_all * pixels)), n_parts = (pixels + p.raw_px - 1) / p.raw_px;
                            const double pieces = (double)((int64_t)pixels << row_log(p.pl)) * (0.8 + 1.4 * full);
                            const double make = pieces + (n_parts > 1.0 ? n_parts * (300.0 + std::max(0.0, 1500.0 - (p.raw_slots - 1) * 0.6 * pieces / n_parts)) : p.raw_slots == 1 ? 1200.0 : 0.0);
                            const double slots = p.b_slots * p.tap_group;
                            const double busy = std::max(std::max(mma, p.resident ? 0.0 : (taps - slots) * 1500.0 / slots), std::max(shared, move));
                            auto block = [&](double n) { return p.a_stages >= two ? make + (n - 1) * std::max(busy, make) + busy : n * (make + std::max(0.0, busy - 0.3 * pieces)); };
                            run = sp == 1 ? std::max(block((double)uses), p.acc_bufs >= 2 ? waves * out : 0.0) + waves * (p.per_split * ends + cuts)
                                          : waves * (block(p.per_split) + p.per_split * ends + cuts) + (waves - 1) * 3500.0;
                        }
                        if (sp == 1) c += run + (p.acc_bufs >= 2 ? out : waves * out);
                        else c += run + waves * (2500.0 + 100.0 * sp + mt * 128.0 * p.nt * 4 / 64.0 + out / sp);
                        if (c < best.cycles * 0.999) { best = p; best.cycles = c; }
                    };
                    p.raw_px = pixels;
                    if (raw_top == 0 || s.stride == 1) {
                        bool fits = false;
                        for (p.raw_slots = raw_top; p.raw_slots >= std::min(raw_top, 1) && !(fits = place(two));) --p.raw_slots;
                        if (fits) weigh(false);
                    } else {
                        const int q_step = kProdThreads >> row_log(p.pl);             // pixels that the producer warps take at a time
                        for (int of : {1, 4, 8})
                            for (p.raw_slots = of == 1 ? raw_top : 4; p.raw_slots >= (of == 1 ? 1 : 2); --p.raw_slots) {
                                p.raw_px = of == 1 ? pixels : ((pixels + of - 1) / of + q_step - 1) / q_step * q_step;
                                if (place(two) || place(1)) weigh(true);
                            }
                    }
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
    P.pl = p.pl; P.plane_pitch = p.plane_pitch;
    P.a_stages = p.a_stages; P.b_slots = p.b_slots; P.resident = p.resident;
    P.b_bytes = p.b_bytes; P.tap_group = p.tap_group;
    P.a_bytes = p.a_bytes;
    P.b_off = p.a_stages * p.a_bytes;
    P.tab_off = p.operands;
    P.raw_off = P.tab_off + p.table_bytes;
    P.raw_slots = p.raw_slots; P.raw_px = p.raw_px; P.raw_bytes = p.raw_bytes; P.raw_pitch = p.raw_pitch;
    P.row_log = row_log(p.pl);
    P.stage_off = P.sum_off = P.raw_off + p.raw_slots * p.raw_bytes;       // (the one or the other)
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
    // a plan for tensor copies has no room for the rows that the producer warps read
    if (dt != XGEN_F32 && p.raw_slots == 0 && !(P.vec_x && x_map(tw, s, p, c.x, xm))) return cudaErrorNotSupported;
    P.vec_y = aligned(c.y, 16) && (size_t)tw.c_out * yb % 16 == 0;
    P.y32 = aligned(c.y, 32) && (size_t)tw.c_out * yb % 32 == 0;
    P.vec_r = c.residual && aligned(c.residual, 16) && (size_t)tw.c_out * rb % 16 == 0;
    // D fp32 (int32), A fp16 / bf16 / u8, B fp16 / bf16 / s8, both K-major, 128 rows (256 of a pair)
    P.idesc = ((uint32_t)(p.nt >> 3) << 17) | ((p.pair ? 16u : 8u) << 24) |
              (dt == XGEN_I8_I32 ? (2u << 4) | (1u << 10) : (1u << 4) | (dt == XGEN_F32 ? (1u << 7) | (1u << 10) : 0u));
    const void *kern = tap_kernel_of(dt, s.stride, tw.taps, p.mt, p.pair, p.cut != 0, c.residual || c.rq_scale || c.pool, dt == XGEN_F32 || p.raw_slots > 0);
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
