// Host program around the Morton sort of the library (index.cu) and the CUDA runtime
// of fake_cuda_runtime.cpp (no CUDA runtime is linked): sorts the numbers of points
// given as arguments one after the other and prints, for each, the sort's result, the
// kernels counted, the kernels launched and the captures made so far. A first
// argument "refused": no capture can begin.
#include <cstdio>
#include <cstdlib>

#include "../paper_2007_07627_gb300/csrc/index.cu"

// fake_cuda_runtime.cpp
extern bool g_no_capture;
extern int g_launched, g_captures;

namespace fricp {
Counters &counters() {
    static Counters c{0, 0, 0};
    return c;
}
cudaError_t pool_alloc_bytes(void **p, size_t, cudaStream_t) {
    *p = reinterpret_cast<void *>((size_t)256);   // nothing is read or written
    return cudaSuccess;
}
}  // namespace fricp

int main(int argc, char **argv) {
    for (int k = 1; k < argc; ++k) {
        if (argv[k][0] == 'r') {
            g_no_capture = true;
            continue;
        }
        const int launched = g_launched;
        const int64_t counted = fricp::counters().launches;
        int *order = nullptr;
        const cudaError_t e = fricp::morton_order(nullptr, std::atoi(argv[k]), nullptr, nullptr, &order);
        std::printf("%d %d %d %d\n", (int)e, (int)(fricp::counters().launches - counted), g_launched - launched, g_captures);
    }
    return 0;
}
