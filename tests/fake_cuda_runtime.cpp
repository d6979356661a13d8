// A CUDA runtime for host programs that link none. A call succeeds and does nothing
// but keep track of
//   - the current device and each stream's; while g_log is set, which device was
//     waited for and on which device's stream an array was given back is printed;
//   - the kernels launched and those captured (a graph is the number of its kernels);
//   - the last error, which only a capture that cannot begin sets (g_no_capture).
#include <cstdio>
#include <cstdlib>
#include <driver_types.h>
#include <vector_types.h>

int g_current = 0;       // the device current in the process's threads, which take turns
bool g_log = false;
bool g_no_capture = false;
int g_launched = 0, g_captures = 0;
static int g_capturing = -1;   // kernels of the running capture
static cudaError_t g_error = cudaSuccess;
static int g_streams = 0, g_stream_device[64];
int device_of(cudaStream_t s) { return s ? g_stream_device[(size_t)s] : g_current; }   // NULL: the current device's

extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = g_current; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { g_current = d; return cudaSuccess; }
cudaError_t cudaStreamGetDevice(cudaStream_t s, int *d) { *d = device_of(s); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
    g_stream_device[++g_streams] = g_current;
    *s = (cudaStream_t)(size_t)g_streams;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
    if (g_log) std::printf("wait %d\n", g_current);
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void *, cudaStream_t s) {
    if (g_log) std::printf("free %d\n", device_of(s));
    return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t, cudaStream_t) { *p = std::malloc(n); return cudaSuccess; }
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t) { *p = std::malloc(n); return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *) { *p = (cudaMemPool_t)1; return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMemPoolGetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { *p = std::malloc(n); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 0.0f; return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaPeekAtLastError() { return g_error; }
cudaError_t cudaGetLastError() {
    const cudaError_t e = g_error;
    g_error = cudaSuccess;
    return e;
}
const char *cudaGetErrorString(cudaError_t) { return ""; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
    if (g_no_capture) return g_error = cudaErrorIllegalState;
    ++g_captures;
    g_capturing = 0;
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) {
    *g = (cudaGraph_t)(size_t)g_capturing;
    g_capturing = -1;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *, cudaGraph_t, unsigned long long) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphGetNodes(cudaGraph_t g, cudaGraphNode_t *, size_t *n) { *n = (size_t)g; return cudaSuccess; }
cudaError_t cudaGraphNodeGetType(cudaGraphNode_t, cudaGraphNodeType *t) { *t = cudaGraphNodeTypeKernel; return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int *n) { *n = 2; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrComputeCapabilityMajor ? 10
       : a == cudaDevAttrComputeCapabilityMinor ? 3 : a == cudaDevAttrWarpSize ? 32 : 1 << 16;
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) {
    *a = cudaFuncAttributes();
    a->ptxVersion = a->binaryVersion = 103;
    a->maxThreadsPerBlock = 1024;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
    *n = 2;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void **, size_t, cudaStream_t) {
    ++(g_capturing >= 0 ? g_capturing : g_launched);
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void *) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaSuccess; }
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void **__cudaRegisterFatBinary(void *) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
}
