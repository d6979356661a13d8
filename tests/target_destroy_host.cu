// Host program around the library's C entry points (api.cu) and the recorded CUDA
// runtime of fake_cuda_runtime.cpp, two devices (no CUDA runtime is linked): prints
// the calls fricp_target_destroy makes for the arguments "target's device, device of
// the thread's work stream, device current at the call" (-1: the thread has no work
// stream yet).
#include <cstdio>
#include <cstdlib>

#include "../paper_2007_07627_gb300/csrc/api.cu"

// fake_cuda_runtime.cpp
extern int g_current;
extern bool g_log;
int device_of(cudaStream_t s);

namespace fricp {
cudaError_t build_target(const float *, const float *, int64_t n, cudaStream_t s, TargetDev *t, int *) {
    t->n = n;
    return pool_alloc(&t->pts, sizeof(float4) * n, s);
}
cudaError_t target_nu_stats(TargetDev *, cudaStream_t) { return cudaSuccess; }
cudaError_t estimate_normals(const TargetDev *, int, const double *, float *, cudaStream_t, int *) { return cudaSuccess; }
cudaError_t build_fp16_storage(TargetDev *, cudaStream_t) { return cudaSuccess; }
cudaError_t prepare_source(const float *, int64_t, cudaStream_t, float4 *, float *, float *, int *, const float *, float4 *) {
    return cudaSuccess;
}
cudaError_t launch_closest(const TargetDev *, const float *, int64_t, const double *, int64_t *, double *, cudaStream_t) {
    return cudaSuccess;
}
cudaError_t launch_step(const StepArgs &, int, int, int, cudaStream_t, cudaEvent_t) { return cudaSuccess; }
cudaError_t launch_median(const double *, const double *, int, void *, double *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_after_init(PairState *, const double *, cudaStream_t) { return cudaSuccess; }
}  // namespace fricp

int main(int argc, char **argv) {
    const int target = std::atoi(argv[1]), stream = std::atoi(argv[2]), current = std::atoi(argv[3]);
    const float q[3] = {0.0f, 0.0f, 0.0f};
    fricp_target *t = nullptr;
    std::thread([&] {   // another thread's work stream
        g_current = target;
        if (fricp_target_create(q, nullptr, 1, 0, nullptr, &t) != FRICP_OK) std::abort();
    }).join();
    if (stream >= 0) {
        g_current = stream;
        work_stream();
    }
    g_current = current;
    g_log = true;
    if (fricp_target_destroy(t) != FRICP_OK) std::abort();
    std::printf("current %d\n", g_current);
    g_log = false;
    std::printf("work stream %d\n", device_of(work_stream()));
    return 0;
}
