// The host's part of a search on the device, run without one (fake_device.cpp): the passes do nothing but leave a state, and what the host takes
// from it is printed (test_encode_core.py).
#include <cstdio>
#include <cstdlib>
#include <ctime>

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

namespace {
uint32_t steps_left = 0, coded = 0, entries_made = 0;
}

extern "C" cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *kernel, void **args) {
    if (kernel == reinterpret_cast<const void *>(quantise_count_kernel)) {
        const CountParams &P = *static_cast<const CountParams *>(args[0]);
        SearchState &S = *P.state;
        if (P.mode == kPassSearch) S.left = steps_left;
        if (P.mode == kPassPolish) { S.polished = S.stop = 1; S.s_counted = 0.5f; S.code = coded; }
    }
    if (kernel == reinterpret_cast<const void *>(encode_entries_kernel)) ++entries_made;
    return cudaSuccess;
}

// arguments: the steps of the bisection that the passes leave undone; have they made the tile coder's entries?  Prints the call's status,
// whether the host takes its result, how often it has entries made for the tile coder then, and the milliseconds that the search kept its core
int main(int, char **argv) {
    steps_left = uint32_t(std::atoi(argv[1]));
    coded = uint32_t(std::atoi(argv[2]));
    const uint32_t R = 16, C = 64, V = 32;
    const size_t need = carve(nullptr, R, C, V).bytes;
    void *ws = nullptr, *W = nullptr;
    if (posix_memalign(&ws, 256, need) || posix_memalign(&W, 256, 4ull * R * C)) return 1;
    std::memset(ws, 0, need);
    std::memset(W, 0, 4ull * R * C);
    ep_encode_opts o;
    ep_encode_opts_default(&o);
    DeviceBackend be(static_cast<const float *>(W), R, C, V, static_cast<uint8_t *>(ws), nullptr);
    int rc = be.prepare(ep::sample_rows(R, C, o.sample_vectors));
    ep::SearchResult found;
    bool done = false;
    const std::clock_t since = std::clock();
    if (!rc) rc = be.search({4.0, 11, V, R * C / 8, R}, o, found, &done);
    const int busy = int(1000 * (std::clock() - since) / CLOCKS_PER_SEC);
    if (!rc && done) rc = be.begin_finish(found.s, 11, V, found.full);
    std::printf("%d %d %u %d\n", rc, int(done), entries_made, busy);
    return 0;
}
