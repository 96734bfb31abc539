// A CUDA runtime that runs nothing: it keeps, for every stream, which work of every other stream its next operation is
// ordered after (a vector clock), and can make one chosen call fail.  Linked in place of the real runtime, it shows on the
// CPU how the library's host code orders its streams, on the paths after an error too.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstring>
#include <map>

namespace {
typedef std::map<void *, long> Clock;                  // stream -> number of its operations
std::map<void *, Clock> streams, events;
long calls, fail_at;
cudaError_t last_error;
uintptr_t next_handle = 0x1000;
struct { dim3 grid, block; size_t smem; cudaStream_t stream; } pushed;

template <typename T> void make(T *out) { *out = reinterpret_cast<T>(next_handle); next_handle += 16; }

bool fails() {
    if (++calls != fail_at) return false;
    last_error = cudaErrorUnknown;
    return true;
}
cudaError_t work(cudaStream_t s) {
    if (fails()) return cudaErrorUnknown;
    ++streams[s][s];
    return cudaSuccess;
}
CUresult encode(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
    return CUDA_SUCCESS;
}
}  // namespace

extern "C" {
// ---- for the test
void fake_reset() { streams.clear(); events.clear(); }
void fake_fail_at(long k) { calls = 0; fail_at = k; last_error = cudaSuccess; }     // the k-th call from now on fails (0: none)
long fake_calls() { return calls; }
// streams with work that the next operation on `s` is not ordered after
int fake_unordered(void *s) {
    int n = 0;
    for (auto &t : streams) n += streams[s][t.first] < t.second[t.first];
    return n;
}

// ---- calls that enqueue
cudaError_t cudaLaunchKernel(const void *, dim3, dim3, void **, size_t, cudaStream_t s) { return work(s); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *, void **) { return work(c->stream); }
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t s) { return work(s); }
cudaError_t cudaMemcpy2DAsync(void *, size_t, const void *, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t s) { return work(s); }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t s) { return work(s); }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    if (fails()) return cudaErrorUnknown;
    events[e] = streams[s];
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    if (fails()) return cudaErrorUnknown;
    for (auto &t : events[e]) streams[s][t.first] = std::max(streams[s][t.first], t.second);
    return cudaSuccess;
}

// ---- everything else
cudaError_t cudaGetLastError() { cudaError_t e = last_error; last_error = cudaSuccess; return e; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
cudaError_t cudaDeviceGetStreamPriorityRange(int *lo, int *hi) { *lo = *hi = 0; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { make(s); return cudaSuccess; }
cudaError_t cudaStreamCreateWithPriority(cudaStream_t *s, unsigned, int) { make(s); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { streams.erase(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *c) { *c = cudaStreamCaptureStatusNone; return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { make(e); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { make(e); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetDriverEntryPoint(const char *, void **p, unsigned long long, cudaDriverEntryPointQueryResult *q) {
    *p = reinterpret_cast<void *>(&encode);
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *) { *p = reinterpret_cast<void *>(uintptr_t(1) << 40); return cudaSuccess; }

// ---- what compiled launches call
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t s) { pushed = {g, b, smem, s}; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *s) {
    *g = pushed.grid; *b = pushed.block; *smem = pushed.smem;
    *static_cast<cudaStream_t *>(s) = pushed.stream;
    return cudaSuccess;
}
char __cudaInitModule(void **) { return 0; }
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
}
