// The matrix path's kernels for fp32 (tapgemm_kernel.cuh), compiled on their own.
#include "tapgemm_kernel.cuh"

namespace patconv {

const void *tap_kernel_f32(int stride, int taps, int mt, bool pair, bool fused, bool gather) {
    return tap_pick_layer<XGEN_F32, false>(stride, taps, mt, pair, fused, gather);
}

}  // namespace patconv
