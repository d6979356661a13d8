// Counting the kernels that a captured piece of work launches, for the launch
// counter behind fricp_counters.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

namespace fricp {
namespace host {

// Kernel nodes of a captured graph (what one replay launches).
inline int64_t graph_kernel_nodes(cudaGraph_t g) {
    size_t n = 0;
    if (cudaGraphGetNodes(g, nullptr, &n) != cudaSuccess || n == 0) return 0;
    std::vector<cudaGraphNode_t> nodes(n);
    if (cudaGraphGetNodes(g, nodes.data(), &n) != cudaSuccess) return 0;
    int64_t k = 0;
    for (size_t i = 0; i < n; ++i) {
        cudaGraphNodeType ty;
        if (cudaGraphNodeGetType(nodes[i], &ty) == cudaSuccess && ty == cudaGraphNodeTypeKernel) ++k;
    }
    return k;
}

// Kernels that `body` (returning a cudaError_t) launches on s, read off a capture
// that is not run; -1 if it cannot be captured. Leaves no error behind: the next
// call on this thread would take it for its own (a sort then does not run at all).
template <class Body>
int64_t captured_kernels(cudaStream_t s, Body body) {
    cudaGraph_t g = nullptr;
    int64_t k = -1;
    if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
        const cudaError_t eb = body();
        if (cudaStreamEndCapture(s, &g) == cudaSuccess && eb == cudaSuccess) k = graph_kernel_nodes(g);
    }
    if (g) cudaGraphDestroy(g);
    if (k < 0) cudaGetLastError();
    return k;
}

// Launches of a call on n elements where a larger n never takes fewer: the same
// number at two sizes is the number at every size between, so the sizes seen are
// kept as the ends of a few ranges.
class LaunchMemo {
  public:
    int64_t find(int64_t n) const {   // -1: not known
        for (const Range &r : r_)
            if (r.launches >= 0 && r.lo <= n && n <= r.hi) return r.launches;
        return -1;
    }
    void add(int64_t n, int64_t launches) {
        for (Range &r : r_) {
            if (r.launches == launches) {
                if (n < r.lo) r.lo = n;
                if (n > r.hi) r.hi = n;
                return;
            }
        }
        r_[next_] = Range{launches, n, n};   // the oldest makes room
        next_ = (next_ + 1) % kRanges;
    }

  private:
    static constexpr int kRanges = 4;
    struct Range {
        int64_t launches = -1, lo = 0, hi = 0;
    };
    Range r_[kRanges];
    int next_ = 0;
};

}  // namespace host
}  // namespace fricp
