// Searches by themselves, without a rate correction: does the device end them, or leave them to the host?  (test_gpu_encode.py)
#include <cstdio>
#include <cstdlib>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#define private public
#include "encode_gpu.cu"
#undef private

// arguments: a file of n R x C matrices, n, R, C, target bpp, b.  Prints 1 (ended) or 0 for each
int main(int, char **argv) {
    const uint32_t n = uint32_t(std::atoi(argv[2])), R = uint32_t(std::atoi(argv[3])), C = uint32_t(std::atoi(argv[4])), V = 256;
    const double bpp = std::atof(argv[5]);
    const int b = std::atoi(argv[6]);
    const size_t bytes = 4ull * R * C, need = carve(nullptr, R, C, V).bytes;
    std::vector<uint8_t> host(bytes);
    void *W = nullptr, *ws = nullptr;
    std::FILE *in = std::fopen(argv[1], "rb");
    if (!in || cudaMalloc(&W, bytes) || cudaMalloc(&ws, need)) return 1;
    for (uint32_t i = 0; i < n; ++i) {
        if (std::fread(host.data(), 1, bytes, in) != bytes || cudaMemcpy(W, host.data(), bytes, cudaMemcpyHostToDevice)) return 1;
        ep_encode_opts o;
        ep_encode_opts_default(&o);
        o.polish_steps = 0;
        DeviceBackend be(static_cast<const float *>(W), R, C, V, static_cast<uint8_t *>(ws), nullptr);
        const std::vector<uint32_t> rows = ep::sample_rows(R, C, o.sample_vectors);
        ep::SearchResult found;
        bool done = false;
        if (be.prepare(rows) || be.search({bpp, b, V, uint64_t(rows.size()) * (C / 8), rows.size()}, o, found, &done)) return 1;
        std::printf("%d\n", int(done));
    }
    std::fclose(in);
    return cudaFree(W) != cudaSuccess || cudaFree(ws) != cudaSuccess;
}
