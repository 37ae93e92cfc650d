// A stand-in for the CUDA runtime, linked with the library's own objects: device memory is host memory,
// launches are recorded and nothing runs.  The tests use it to see what the host code does when a call
// fails, and what it holds and launches; no device is needed.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <map>

static std::map<void *, size_t> live;
static long long live_bytes = 0;
static int fail_alloc = 0, fail_encode = 0, launches = 0, sms = 148;
static cudaError_t last = cudaSuccess;
static cudaError_t is(cudaError_t e) { if (e != cudaSuccess) last = e; return e; }
// grid, block, dynamic shared memory, cluster of the last launch
static long long launch[4];
// the current device, that of the last allocation; whether streams are being captured, and the driver has no tensor maps
static int device = 0, alloc_device = -1, capturing = 0, no_encode = 0;

extern "C" {
// The n-th allocation (encoding of a tensor map) from now on fails; 0: none does.
void fake_fail_alloc(int n) { fail_alloc = n; }
void fake_fail_encode(int n) { fail_encode = n; }
long long fake_live_bytes() { return live_bytes; }
int fake_launches() { return launches; }
long long fake_launch(int what) { return launch[what]; }
int fake_alloc_device() { return alloc_device; }
int fake_device() { return device; }
void fake_capture(int on) { capturing = on; }
void fake_no_encode(int on) { no_encode = on; }

cudaError_t cudaMalloc(void **p, size_t n) {
    if (fail_alloc && --fail_alloc == 0) return is(cudaErrorMemoryAllocation);
    alloc_device = device;
    *p = aligned_alloc(256, (n + 255) / 256 * 256);
    live[*p] = n;
    live_bytes += (long long)n;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    if (!p) return cudaSuccess;
    const auto it = live.find(p);
    if (it == live.end()) return is(cudaErrorInvalidValue);
    live_bytes -= (long long)it->second;
    live.erase(it);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemset(void *d, int v, size_t n) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }

cudaError_t cudaLaunchKernel(const void *, dim3 grid, dim3 block, void **, size_t smem, cudaStream_t) {
    ++launches;
    launch[0] = grid.x; launch[1] = block.x; launch[2] = (long long)smem; launch[3] = 1;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *k, void **a) {
    cudaLaunchKernel(k, c->gridDim, c->blockDim, a, c->dynamicSmemBytes, c->stream);
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) launch[3] = c->attrs[i].val.clusterDim.x;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *c) {
    *n = sms / (int)c->gridDim.x;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int, size_t smem) {
    *n = smem > 116224 ? 1 : 2;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = sms; return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { device = d; return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) {
    *s = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t)1; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *t, cudaEvent_t, cudaEvent_t) { *t = 0.0f; return cudaSuccess; }

static CUresult encode(CUtensorMap *m, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                       const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                       CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
    if (fail_encode && --fail_encode == 0) return CUDA_ERROR_INVALID_VALUE;
    memset(m, 0, sizeof(*m));
    return CUDA_SUCCESS;
}
cudaError_t cudaGetDriverEntryPoint(const char *, void **p, unsigned long long, cudaDriverEntryPointQueryResult *q) {
    *p = no_encode ? nullptr : (void *)encode;
    if (q) *q = no_encode ? cudaDriverEntryPointSymbolNotFound : cudaDriverEntryPointSuccess;
    return cudaSuccess;
}

// What nvcc's host code calls to make its kernels known, and around <<< >>>.
static dim3 pushed_grid, pushed_block;
static size_t pushed_smem;
void **__cudaRegisterFatBinary(void *) { static void *handle; return &handle; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, void *, void *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, void *) {
    pushed_grid = grid; pushed_block = block; pushed_smem = smem;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *stream) {
    *grid = pushed_grid; *block = pushed_block; *smem = pushed_smem;
    *(void **)stream = nullptr;
    return cudaSuccess;
}
}
