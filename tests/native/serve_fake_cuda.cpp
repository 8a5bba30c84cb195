// A fake of the CUDA calls of csrc/ph0_serve.cu (serve_failure_check.cu): device
// memory is host memory, copies run at once, and every stream remembers the
// memory its work uses until it is waited for; a use of such memory on another
// stream is counted.
#include <atomic>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <vector>

#include <cuda_runtime.h>

namespace {
std::mutex g_mu;
struct Use {
    const char *p;
    size_t bytes;
    cudaStream_t s;
};
std::vector<Use> g_uses;
std::atomic<size_t> g_next{1};

void done(cudaStream_t s) {
    std::lock_guard<std::mutex> lk(g_mu);
    for (size_t i = 0; i < g_uses.size();)
        if (g_uses[i].s == s) g_uses.erase(g_uses.begin() + long(i));
        else ++i;
}
}  // namespace

std::atomic<int> g_overlaps{0};
std::atomic<bool> g_ready{false};  // whether recorded events have come to pass

void fake_use(const void *p, size_t bytes, cudaStream_t s) {
    std::lock_guard<std::mutex> lk(g_mu);
    const char *q = static_cast<const char *>(p);
    for (const Use &u : g_uses)
        if (u.s != s && q < u.p + u.bytes && u.p < q + bytes) ++g_overlaps;
    g_uses.push_back({q, bytes, s});
}

extern "C" {
// ---- what nvcc's host code registers ----
void **__cudaRegisterFatBinary(void *) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}

// ---- the CUDA calls ----
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) { return (*p = std::calloc(1, n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFree(void *p) { return std::free(p), cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { return std::free(p), cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
    return *s = reinterpret_cast<cudaStream_t>(g_next++), cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return done(s), cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { return *g = nullptr, cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) { return *x = nullptr, cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) {
    return *e = reinterpret_cast<cudaEvent_t>(g_next++), cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
// (the context makes each stream and then its event, so the handles follow each other)
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t e) {
    if (!g_ready) return cudaErrorNotReady;
    done(reinterpret_cast<cudaStream_t>(reinterpret_cast<size_t>(e) - 1));
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *to, const void *from, size_t n, cudaMemcpyKind kind, cudaStream_t s) {
    fake_use(kind == cudaMemcpyHostToDevice ? to : from, n, s);
    std::memcpy(to, from, n);
    return cudaSuccess;
}
}
