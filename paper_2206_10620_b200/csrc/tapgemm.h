// Host interface of the tensor-core kernel (tapgemm.cu): a 3x3 convolution as nine shifted matrix
// products over one staged tile, and a plain matrix product as the case of one tap.
#pragma once
#include <cstddef>
#include <cstdint>

#include <cuda.h>
#include <cuda_runtime.h>

#include "patconv.h"

namespace patconv {

// cuTensorMapEncodeTiled, or null where the driver has none (patconv.cu).
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled_fn();
// Whether a stream records a graph, in which nothing may be allocated (patconv.cu).
bool being_captured(cudaStream_t st);

// The layer's weights as the kernel reads them: pruned entries are zeros, fp32 weights are three
// bf16 parts whose sum is the weight.  Bytes [plane][tap][part][filter][16]: a plane is 16 bytes of
// input channels (8 fp16 / bf16, 16 int8); a tensor copy takes any range of filters and planes of a
// tap at once, so neither the filter tile nor the channels per stage is fixed here.
struct TapWeights {
    uint8_t *dev = nullptr;      // the image
    int device = -1;
    size_t bytes = 0;            // device memory: the image and the status word
    int *status = nullptr;       // behind the image: set by a kernel whose bounded wait ran out
    xgen_dtype dtype = XGEN_F32;
    int taps = 9, c_in = 0, c_out = 0;
    int planes = 0;              // a multiple of two (a matrix instruction takes two)
    int rows = 0;                // filters, rounded up to 16
};

// Geometry of a call.
struct TapShape {
    int n = 0, h = 0, w = 0;     // convolution input; product: n = 1, w = 8, h = rows / 8 rounded up
    int stride = 1;
    int64_t rows = 0;            // product: rows of x (0 for a convolution)
    bool pool = false;
    bool gather = false;         // rows of x are not whole aligned 16-byte pieces although their length is (its address is not)
    bool staged = false;         // results pass through shared memory: rows of y are not whole 16-byte pieces, or fp32 with a residual
};

// How the problem is cut up (tap_choose).
struct TapPlan {
    int mt = 1;                  // matrix-instruction tiles (128 pixels each) of a block's tile
    int pair = 0;                // two blocks of a cluster work as one: a tile each, the weights halved between them
    int nt = 0, nblk = 0;        // filters of a tile, tiles of filters
    int pl = 0, stages = 0;      // planes per stage, stages of the whole reduction
    int splits = 1, per_split = 0;   // blocks that share an item's reduction (one cluster), stages of each
    int cut = 0;                 // fp16: stages after which sums leave the matrix unit's accumulator (0: all of them)
    int vh = 0, straddle = 0, segs = 0, row_tiles = 0, items = 0, grid = 0;
    int raster = 0, pitch = 0, rows = 0, pixels = 0;     // staged tile: entries of a row, rows (of a parity), entries
    int a_stages = 0, a_bytes = 0, b_slots = 0, b_bytes = 0, tap_group = 1, resident = 0, operands = 0;   // (bytes of all of them)
    int plane_pitch = 0, table_bytes = 0;
    int raw_slots = 0, raw_px = 0, raw_bytes = 0, raw_pitch = 0;     // rows of x that the producer warps shift into place (none: tensor copies, or fp32)
    size_t smem = 0;
    int tmem_cols = 0, acc_bufs = 0;
    double cycles = 0;           // what the cost model expects
    CUtensorMap wmap;            // the weights of (planes of a stage, tap, parts, filters of a block) as one box
};

struct TapCall {
    const void *x; void *y; const void *bias; const void *residual; const float *rq_scale;
    int rq_zero, relu, pool;
    int *status; uint32_t wait_us;
    int hold;                    // testing aid: every stage of x waits for this many arrivals that never come
    bool overlap;                // programmatic stream serialisation
};

// Build the device weights; the device must be current.  Block-pruned matrix: dense_w [c_out][c_in]
// with the keep flags of include/blockgemm.h.
xgen_status tap_upload_dense(TapWeights &tw, xgen_dtype dt, int c_in, int c_out, const void *dense_w,
                             const uint8_t *row_keep, const uint8_t *col_keep, int br, int bc);
// Pattern-pruned convolution: kpat [c_out][c_in] pattern or -1, kw4 the four kept weights (fp32 bits).
xgen_status tap_upload_patterns(TapWeights &tw, xgen_dtype dt, int c_in, int c_out, const int16_t *kpat,
                                const uint32_t *kw4, const uint16_t *masks, int n_masks);
void tap_free(TapWeights &tw);

// Threads of a block.
int tap_block_threads(xgen_dtype dt);
// Pick a plan for the shape; false: this shape cannot run here.
bool tap_choose(const TapWeights &tw, const TapShape &s, int device, TapPlan &plan);
cudaError_t tap_launch(const TapWeights &tw, const TapShape &s, const TapPlan &plan, const TapCall &c, cudaStream_t st);

}  // namespace patconv
