// A stand-in for the CUDA runtime: kernels do nothing, device memory is host memory, and an asynchronous copy is made when
// its stream is waited for.  For what the host side of the encoder does around its calls (test_encode_core.py).
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "entropack.h"

namespace {
struct Copy { void *to; const void *from; size_t n; };
std::vector<Copy> pending;
int host_allocs_left = 1 << 30;

void finish() {
    for (const Copy &c : pending) std::memcpy(c.to, c.from, c.n);
    pending.clear();
}
}  // namespace

extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) { std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *to, const void *from, size_t n, cudaMemcpyKind kind, cudaStream_t) {
    if (kind == cudaMemcpyDeviceToHost) pending.push_back({to, from, n});
    else std::memcpy(to, from, n);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { finish(); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { finish(); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) {
    if (host_allocs_left-- <= 0) return cudaErrorMemoryAllocation;
    *p = std::calloc(1, n);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaLaunchKernel(const void *, dim3, dim3, void **, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *, void **) { return cudaSuccess; }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, struct CUstream_st *) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaSuccess; }
void **__cudaRegisterFatBinary(void *) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
char __cudaInitModule(void **) { return 0; }
cudaError_t __cudaGetKernel(cudaKernel_t *, const void *) { return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void **, size_t, cudaStream_t) { return cudaSuccess; }
}

// argument: how many page-locked buffers there are; prints the status of an encode and the copies still under way after it
int main(int argc, char **argv) {
    host_allocs_left = std::atoi(argv[1]);
    ep_encode_opts o;
    ep_encode_opts_default(&o);
    void *ws = nullptr, *W = nullptr;
    const size_t need = ep_encode_device_workspace_bytes(16, 64, 4.0, &o);
    if (posix_memalign(&ws, 256, need) || posix_memalign(&W, 256, 16 * 64 * 4)) return 1;
    std::memset(ws, 0, need);
    std::memset(W, 0, 16 * 64 * 4);
    ep_blob *blob = nullptr;
    const int rc = ep_encode_device(static_cast<const float *>(W), 16, 64, 4.0, &o, ws, need, nullptr, &blob);
    std::printf("%d %zu\n", rc, pending.size());
    return 0;
}
