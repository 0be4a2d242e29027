// The wait for a table image that never comes, run by itself: the mbarrier is initialised and nothing ever completes its phase
// (test_gpu_decode.py).
#include "decode.cu"

#include <cstdio>

// warps 0 and 1 wait, warp 2 only meets the CTA's barrier
__global__ void wait_in_vain(uint32_t *seen) {
    extern __shared__ __align__(16) uint8_t smem[];
    const uint32_t lut = uint32_t(__cvta_generic_to_shared(smem)), bar = lut + kCtxBase + kCtxTablesBar;
    if (threadIdx.x == 0) mbar_init(bar, 1u);
    __syncthreads();
    if (threadIdx.x < 64u) {
        wait_for_tables({kTablesCopied, bar, 0u});
        seen[threadIdx.x] = 1u;              // a warp that went on
    }
    __syncthreads();
    if (threadIdx.x >= 64u) seen[threadIdx.x] = 2u;
}

int main() {
    uint32_t *seen = nullptr, host[96] = {};
    if (cudaMalloc(&seen, sizeof(host)) || cudaMemset(seen, 0, sizeof(host))) return 1;
    if (cudaFuncSetAttribute(wait_in_vain, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmemBytes))) return 1;
    wait_in_vain<<<1, 96, kSmemBytes>>>(seen);
    if (cudaMemcpy(host, seen, sizeof(host), cudaMemcpyDeviceToHost)) return 1;
    uint32_t on = 0, met = 0;
    for (int i = 0; i < 96; ++i) { on += host[i] == 1u; met += host[i] == 2u; }
    std::printf("%d %u %u\n", ep_last_device_status(nullptr), on, met);
    return cudaFree(seen) != cudaSuccess;
}
