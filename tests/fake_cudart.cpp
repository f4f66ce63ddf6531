// A stand-in for the CUDA runtime with two devices and no kernels, linked with the library's
// objects so that their host code runs without a GPU.  Device memory is host memory.  It keeps
// which device is current, how much was enqueued on each and how much of that was waited for
// (device, stream or event), and which device owns each block of pool memory; counts blocks
// given back while their device was still at work (freeing pool memory does not wait), and
// device synchronisations during a capture, which fail and break the capture; and sums the
// bytes that cudaMalloc holds.
#include <cuda_runtime_api.h>
#include <stdlib.h>
#include <string.h>
#include <unistd.h>

#include <atomic>
#include <map>
#include <mutex>

namespace {
std::atomic<int> current{0}, early_frees{0}, launches{0}, captures{0}, broken_captures{0}, capture_ms{0};
std::atomic<long> enqueued[2], waited[2];
std::mutex mu;
std::map<void *, int> pool_blocks;
std::map<void *, size_t> held;
struct Event { int dev; long at; };
void wait_to(int dev, long at) {
    if (waited[dev] < at) waited[dev] = at;
}
thread_local cudaError_t last = cudaSuccess;  // kept until it is read, as the runtime does
cudaError_t give(void **p, size_t bytes) {  // (a device of 256 GB)
    *p = bytes < (size_t)1 << 38 ? calloc(1, bytes ? bytes : 1) : nullptr;
    return *p ? cudaSuccess : (last = cudaErrorMemoryAllocation);
}
cudaError_t handle(void *out) {
    *static_cast<void **>(out) = malloc(1);
    return cudaSuccess;
}
}  // namespace

extern "C" {
int fake_early_frees() { return early_frees; }
int fake_launches() { return launches; }
int fake_broken_captures() { return broken_captures; }
int fake_captures() { return captures; }
void fake_capture_elsewhere(int on) { captures += on ? 1 : -1; }  // another program's or thread's
void fake_capture_lasts(int ms) { capture_ms = ms; }
long long fake_held_bytes() {
    std::lock_guard<std::mutex> lk(mu);
    long long n = 0;
    for (auto &b : held) n += (long long)b.second;
    return n;
}
int fake_pool_blocks() { return (int)pool_blocks.size(); }

cudaError_t cudaGetDevice(int *d) { *d = current; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { current = d; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() {
    if (captures > 0) {
        ++broken_captures;
        return last = cudaErrorStreamCaptureUnsupported;
    }
    wait_to(current, enqueued[current]);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { wait_to(current, enqueued[current]); return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 4 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 227 * 1024 : 0;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
const char *cudaGetErrorName(cudaError_t) { return "fake"; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }

cudaError_t cudaMalloc(void **p, size_t n) {
    cudaError_t e = give(p, n);
    std::lock_guard<std::mutex> lk(mu);
    if (e == cudaSuccess) held[*p] = n;
    return e;
}
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t) { return give(p, n); }
cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t, cudaStream_t) {
    cudaError_t e = give(p, n);
    std::lock_guard<std::mutex> lk(mu);
    if (e == cudaSuccess) pool_blocks[*p] = current;
    return e;
}
cudaError_t cudaFree(void *p) {
    std::lock_guard<std::mutex> lk(mu);
    auto it = pool_blocks.find(p);
    if (it != pool_blocks.end()) {
        early_frees += waited[it->second] < enqueued[it->second];
        pool_blocks.erase(it);
    }
    held.erase(p);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t) {
    std::lock_guard<std::mutex> lk(mu);
    pool_blocks.erase(p);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *) { return handle(p); }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return give(p, n); }
cudaError_t cudaGetSymbolAddress(void **, const void *) { return cudaErrorNotSupported; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) {
    ++enqueued[current];
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) {
    ++enqueued[current];
    memset(d, v, n);
    return cudaSuccess;
}

static cudaError_t launched() {
    ++enqueued[current];
    ++launches;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *, void **) { return launched(); }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void **, size_t, cudaStream_t) { return launched(); }
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *) { *k = nullptr; return cudaSuccess; }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void *) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaSuccess; }
void **__cudaRegisterFatBinary(void *p) { return (void **)p; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) { memset(a, 0, sizeof *a); return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }

cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) {
    *s = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return handle(s); }
cudaError_t cudaStreamDestroy(cudaStream_t s) { free(s); return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
    ++captures;
    usleep(1000 * capture_ms);
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) {
    --captures;
    return handle(g);
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) { return handle(x); }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return launched(); }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { free(x); return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { free(g); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) {
    *e = reinterpret_cast<cudaEvent_t>(new Event{current, 0});
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete reinterpret_cast<Event *>(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) {
    *reinterpret_cast<Event *>(e) = Event{current, enqueued[current]};
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) {
    wait_to(reinterpret_cast<Event *>(e)->dev, reinterpret_cast<Event *>(e)->at);
    return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 0; return cudaSuccess; }
}
