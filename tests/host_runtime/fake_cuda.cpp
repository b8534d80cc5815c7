// A CUDA runtime without a device, for tests of the library's host code.
//
// The library's own objects are linked against the functions below instead of
// the CUDA runtime.  "Device" memory is host memory, so copies and fills do
// what they say; kernels do nothing; every call that touches a stream, memory
// or an event is appended to a log of JSON lines.  A freed block is handed out
// again to the next allocation of its size, so that address reuse, which on a
// device depends on the allocator, happens every time.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <cstdarg>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#define TEST_API extern "C" __attribute__((visibility("default")))

// One JSON line on what a launch of kernel `name` was given ("" for kernels no
// test asks about); step_arguments.cu, which knows the kernels' arguments.
std::string describe_launch(const std::string &name, void *const *args);

namespace {

struct State {
    std::string log;
    std::map<char *, size_t> live;
    std::map<size_t, std::vector<char *>> free_blocks;
    std::map<const void *, std::string> kernels;   // host stub -> mangled name
    std::map<void *, int> ids;                     // streams, events and graphs
    int next_id = 1;
    bool capturing = false;
    cudaStream_t capture_stream = nullptr;
    int captures = 0;
    int fail_box_x = 0, fail_box_y = 0, fail_encode_from = 0, encodes = 0;   // tensor maps that cannot be encoded
    size_t fail_malloc_bytes = 0;   // allocations of this size fail
    std::string fast, last_kernel;   // event times: short when the last kernel's name holds `fast`
    dim3 grid, block;
    size_t smem = 0;
    cudaStream_t stream = nullptr;
};

State &st() {
    static State s;
    return s;
}

void say(const char *fmt, ...) {
    char line[1024];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(line, sizeof(line), fmt, ap);
    va_end(ap);
    st().log += line;
    st().log += '\n';
}

template <class T>
int id_of(T handle) {
    auto it = st().ids.find((void *)handle);
    return it == st().ids.end() ? 0 : it->second;
}

template <class T>
void new_handle(T *out) {
    void *p = malloc(16);
    st().ids[p] = st().next_id++;
    *out = (T)p;
}

unsigned long long num(const void *p) { return (unsigned long long)(uintptr_t)p; }

bool on_hold(cudaStream_t s) { return st().capturing && s == st().capture_stream; }

void launched(const void *fn, void **args, cudaStream_t s, int attrs) {
    const std::string &name = st().kernels[fn];
    st().last_kernel = name;
    say("{\"op\": \"launch\", \"name\": \"%s\", \"stream\": %d, \"attrs\": %d}", name.c_str(), id_of(s), attrs);
    const std::string line = describe_launch(name, args);
    if (!line.empty()) st().log += line + '\n';
}

CUresult fake_encode(CUtensorMap *map, CUtensorMapDataType, cuuint32_t, void *base, const cuuint64_t *, const cuuint64_t *,
                     const cuuint32_t *box, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                     CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
    State &s = st();
    const bool match = s.fail_box_x == 0 || (box[0] == (cuuint32_t)s.fail_box_x && box[1] == (cuuint32_t)s.fail_box_y);
    if (s.fail_encode_from > 0 && match && ++s.encodes >= s.fail_encode_from) {
        say("{\"op\": \"encode_failed\", \"base\": %llu}", num(base));
        return CUDA_ERROR_INVALID_VALUE;
    }
    memset(map, 0, sizeof(*map));
    memcpy(map, box, 2 * sizeof(box[0]));   // the map remembers its box
    say("{\"op\": \"encode\", \"base\": %llu, \"box\": [%u, %u], \"map\": %llu}", num(base), box[0], box[1], num(map));
    return CUDA_SUCCESS;
}

}  // namespace

// ---- what the tests call
TEST_API const char *fake_log() { return st().log.c_str(); }
TEST_API void fake_clear() { st().log.clear(); }
TEST_API void *fake_malloc(size_t bytes) {
    void *p = nullptr;
    cudaMalloc(&p, bytes);
    return p;
}
TEST_API void fake_free(void *p) { cudaFree(p); }
TEST_API void *fake_stream() {
    cudaStream_t s;
    new_handle(&s);
    return (void *)s;
}
// From the nth on, encodings with this box fail (0 x 0: any box; n = 0: none).
TEST_API void fake_fail_encode(int box_x, int box_y, int nth) {
    st().fail_box_x = box_x;
    st().fail_box_y = box_y;
    st().fail_encode_from = nth;
    st().encodes = 0;
}
TEST_API void fake_fail_malloc(size_t bytes) { st().fail_malloc_bytes = bytes; }
TEST_API void fake_fast_kernel(const char *part) { st().fast = part; }

// ---- the runtime
extern "C" {

void **__cudaRegisterFatBinary(void *) {
    static void *h = nullptr;
    return &h;
}
char __cudaInitModule(void **) { return 1; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *,
                            int *) {
    st().kernels[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st *stream) {
    st().grid = grid;
    st().block = block;
    st().smem = smem;
    st().stream = stream;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *stream) {
    *grid = st().grid;
    *block = st().block;
    *smem = st().smem;
    *(cudaStream_t *)stream = st().stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *fn) {
    *k = (cudaKernel_t)fn;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **args, size_t, cudaStream_t s) {
    launched((const void *)k, args, s, 0);
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *fn, void **args) {
    launched(fn, args, c->stream, (int)c->numAttrs);
    return cudaSuccess;
}

cudaError_t cudaMalloc(void **p, size_t n) {
    State &s = st();
    if (n == s.fail_malloc_bytes && n > 0) return cudaErrorMemoryAllocation;
    auto &blocks = s.free_blocks[n];
    if (!blocks.empty()) {
        *p = blocks.back();
        blocks.pop_back();
    } else {
        *p = aligned_alloc(256, (n + 255) / 256 * 256);
    }
    memset(*p, 0xcd, n);
    s.live[(char *)*p] = n;
    say("{\"op\": \"malloc\", \"ptr\": %llu, \"bytes\": %zu}", num(*p), n);
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    State &s = st();
    auto it = s.live.find((char *)p);
    if (it == s.live.end()) return cudaErrorInvalidValue;
    s.free_blocks[it->second].push_back(it->first);
    say("{\"op\": \"free\", \"ptr\": %llu, \"bytes\": %zu}", num(p), it->second);
    s.live.erase(it);
    return cudaSuccess;
}
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t) { return cudaMalloc(p, n); }
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return cudaFree(p); }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) {
    *p = calloc(1, n);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) {
    free(p);
    return cudaSuccess;
}
cudaError_t cudaHostGetDevicePointer(void **d, void *h, unsigned) {
    *d = h;
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
    memset(a, 0, sizeof(*a));
    a->type = cudaMemoryTypeUnregistered;
    auto it = st().live.upper_bound((char *)p);
    if (it != st().live.begin()) {
        --it;
        if ((char *)p < it->first + it->second) {
            a->type = cudaMemoryTypeDevice;
            a->devicePointer = const_cast<void *>(p);
        }
    }
    return cudaSuccess;
}

cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t s) {
    say("{\"op\": \"memset\", \"dst\": %llu, \"bytes\": %zu, \"stream\": %d}", num(p), n, id_of(s));
    if (!on_hold(s)) memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *src, size_t n, cudaMemcpyKind kind, cudaStream_t s) {
    say("{\"op\": \"memcpy\", \"dst\": %llu, \"src\": %llu, \"bytes\": %zu, \"kind\": %d, \"stream\": %d}", num(d), num(src),
        n, (int)kind, id_of(s));
    if (!on_hold(s)) memmove(d, src, n);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *p, int v, size_t n) { return cudaMemsetAsync(p, v, n, nullptr); }
cudaError_t cudaMemcpy(void *d, const void *src, size_t n, cudaMemcpyKind kind) {
    return cudaMemcpyAsync(d, src, n, kind, nullptr);
}

cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
    new_handle(s);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    say("{\"op\": \"sync\", \"stream\": %d}", id_of(s));
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
    say("{\"op\": \"sync_device\"}");
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    say("{\"op\": \"wait\", \"stream\": %d, \"event\": %d}", id_of(s), id_of(e));
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) {
    new_handle(e);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t e, cudaStream_t s, unsigned) {
    say("{\"op\": \"record\", \"event\": %d, \"stream\": %d, \"capture\": %d}", id_of(e), id_of(s), on_hold(s));
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { return cudaEventRecordWithFlags(e, s, 0); }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
    const State &s = st();
    *ms = !s.fast.empty() && s.last_kernel.find(s.fast) != std::string::npos ? 0.5f : 1.0f;
    return cudaSuccess;
}

cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
    st().capturing = true;
    st().capture_stream = s;
    say("{\"op\": \"begin_capture\"}");
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) {
    st().capturing = false;
    new_handle(g);
    say("{\"op\": \"end_capture\"}");
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long) {
    new_handle(e);
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t s) {
    say("{\"op\": \"graph\", \"exec\": %d, \"stream\": %d}", id_of(e), id_of(s));
    return cudaSuccess;
}

cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorName(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "cudaErrorMemoryAllocation" : "error"; }
const char *cudaGetErrorString(cudaError_t e) { return cudaGetErrorName(e); }
cudaError_t cudaGetDevice(int *d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int *n) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 1;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) {
    memset(a, 0, sizeof(*a));
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int, size_t) {
    *n = 2;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
    *n = 2;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *) {
    *p = nullptr;
    return cudaErrorInvalidValue;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *name, void **fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q) {
    const bool known = strcmp(name, "cuTensorMapEncodeTiled") == 0;
    *fn = known ? (void *)fake_encode : nullptr;
    if (q) *q = known ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}

}  // extern "C"
