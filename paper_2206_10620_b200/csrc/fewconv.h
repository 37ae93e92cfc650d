// Host interface of the kernel for layers of a few input channels (fewconv.cu).
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

#include "patconv.h"

namespace patconv {

// The layer's weights as the kernel reads them: fp32 [tap][input channel][filter], filters rounded up to 16,
// pruned ones +0, kept zeros -0.
struct FewWeights {
    float *dev = nullptr;
    xgen_dtype dtype = XGEN_F32;
    int c_in = 0, c_out = 0, rows = 0;
};

// Layers that the kernel takes.
constexpr bool few_channels(xgen_dtype dt, int c_in) { return c_in < (dt == XGEN_F32 ? 5 : 8); }

// Arguments as of tap_upload_patterns; the device must be current.
xgen_status few_upload(FewWeights &fw, xgen_dtype dt, int c_in, int c_out, const int16_t *kpat, const uint32_t *kw4,
                       const uint16_t *masks);
void few_free(FewWeights &fw);
cudaError_t few_launch(const FewWeights &fw, const void *x, int n, int h, int w, int stride, const void *bias, bool relu, void *y,
                       bool overlap, cudaStream_t st);

}  // namespace patconv
