// The matrix path's kernels for fp16 (tapgemm_kernel.cuh), compiled on their own.
#include "tapgemm_kernel.cuh"

namespace patconv {

const void *tap_kernel_f16(int stride, int taps, int mt, bool pair, bool fused, bool gather) {
    return tap_pick_layer<XGEN_F16_F32ACC, false>(stride, taps, mt, pair, fused, gather);
}

}  // namespace patconv
