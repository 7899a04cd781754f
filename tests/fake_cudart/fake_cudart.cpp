// A CUDA runtime without a device, for tests of the library's host side: "device" memory is host memory under a
// settable limit, copies are copies, and a kernel launch is a line in a log.  Linked with the library's object
// files in place of the CUDA runtime (tests/fake_cudart/__init__.py).
#include <cuda_runtime_api.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <string>

namespace {

struct State {
    size_t limit = SIZE_MAX, live = 0;      // bytes that may be, and are, allocated
    int capturing = 0;                      // a stream capture is on: allocations and waits are errors
    int64_t mallocs = 0, frees = 0, uploads = 0, waits = 0;
    std::map<void *, size_t> blocks;
    std::map<const void *, std::string> names;   // kernel stub -> device name
    std::string log;
    cudaError_t last = cudaSuccess;
    dim3 grid, block;
    size_t smem = 0;
    cudaStream_t stream = nullptr;
};
State &st() { static State *s = new State(); return *s; }   // (registrations run before other static objects)

cudaError_t fail(cudaError_t e) { st().last = e; return e; }

cudaError_t launched(const void *f, dim3 g) {
    st().log += st().names.count(f) ? st().names[f] : std::string("?");
    st().log += " " + std::to_string(g.x) + "," + std::to_string(g.y) + "\n";
    return cudaSuccess;
}

}  // namespace

extern "C" {

// ---- the tests' side
void fake_set(uint64_t limit, int capturing) { st().limit = limit; st().capturing = capturing; }
void fake_counts(int64_t out[5]) {
    out[0] = st().mallocs; out[1] = st().frees; out[2] = st().uploads; out[3] = st().waits; out[4] = (int64_t)st().live;
}
const char *fake_log(void) { return st().log.c_str(); }
void fake_clear(void) { st().log.clear(); }

// ---- the runtime's side
cudaError_t cudaMalloc(void **p, size_t n) {
    *p = nullptr;
    if (st().capturing) return fail(cudaErrorStreamCaptureUnsupported);
    if (n > st().limit - (st().live < st().limit ? st().live : st().limit)) return fail(cudaErrorMemoryAllocation);
    if (posix_memalign(p, 256, n ? n : 1)) return fail(cudaErrorMemoryAllocation);
    st().blocks[*p] = n;
    st().live += n;
    ++st().mallocs;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    if (!p) return cudaSuccess;
    if (st().capturing) return fail(cudaErrorStreamCaptureUnsupported);
    if (!st().blocks.count(p)) return fail(cudaErrorInvalidValue);
    st().live -= st().blocks[p];
    st().blocks.erase(p);
    ++st().frees;
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); ++st().uploads; return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t) { return cudaMemcpy(d, s, n, k); }
cudaError_t cudaMemset(void *d, int v, size_t n) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { return cudaMemset(d, v, n); }
cudaError_t cudaStreamSynchronize(cudaStream_t) {
    if (st().capturing) return fail(cudaErrorStreamCaptureUnsupported);
    ++st().waits;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0;
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { const cudaError_t e = st().last; st().last = cudaSuccess; return e; }
const char *cudaGetErrorString(cudaError_t) { return "error of the fake runtime"; }
cudaError_t cudaGetSymbolAddress(void **p, const void *) { *p = nullptr; return fail(cudaErrorInvalidSymbol); }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
    *n = 2;
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 1.0f; return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) { return launched(f, c->gridDim); }

// ---- what the compiler's launch stubs call
void **__cudaRegisterFatBinary(void *) { static void *h = nullptr; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *f, char *, const char *name, int, void *, void *, void *, void *, int *) {
    st().names[f] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t s) {
    st().grid = g; st().block = b; st().smem = smem; st().stream = s;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *s) {
    *g = st().grid; *b = st().block; *smem = st().smem; *(cudaStream_t *)s = st().stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(const void **k, const void *f) { *k = f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(const void *k, dim3 g, dim3, void **, size_t, cudaStream_t) { return launched(k, g); }

}  // extern "C"
