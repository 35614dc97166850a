// A CUDA runtime without a device, for host-side checks of libgsis on the CPU: the library's
// objects are linked with this file in place of libcudart.  Kernels are recorded and not run;
// device memory is host memory.  What it models is when the work that a call enqueues is
// complete, by the runtime's documented rules:
//
//  * everything given a stream completes when that stream (or an event recorded after it) is
//    waited for; streams made by the caller are not ordered after the default stream (they
//    are created non-blocking);
//  * cudaMemcpy from pageable memory returns once the source is staged, the arrival in device
//    memory is work of the default stream; cudaMemset is such work too;
//  * an asynchronous copy from pinned memory reads its source when it runs, not when it is
//    enqueued.
//
// Reported (fake_report, one line each):
//  unordered <name>   work on another stream while default-stream work is incomplete
//  rewritten          a pinned source that changed between a copy's enqueueing and its completion
//  null               a copy or clear of a null pointer
//  attribute <kernel> a kernel's attribute set to another value than before (the attribute
//                     belongs to the kernel, for every thread of the process)
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {

struct Op {
    long long seq;
    const void *src;                 // pinned source, or null
    std::vector<unsigned char> bytes;
};
struct Launch {
    std::string name;
    dim3 grid, block;
    size_t smem;
};
struct Event {
    cudaStream_t stream = nullptr;
    long long seq = 0;
};
struct State {
    std::map<cudaStream_t, std::vector<Op>> pending;
    std::map<const char *, size_t> pinned, device;
    std::map<std::pair<const void *, int>, int> attribute;
    std::map<const void *, std::string> names;
    std::vector<Launch> launches;
    std::vector<size_t> cleared;     // sizes of the device allocations cleared in full
    std::string report;
    cudaStream_t capturing = nullptr;
    long long seq = 0, mallocs_left = -1;
    dim3 grid, block;
    size_t smem = 0;
    cudaStream_t stream = nullptr;
};
State &S() {
    static State *s = new State;
    return *s;
}

void say(const std::string &line) { S().report += line + "\n"; }

void complete(cudaStream_t st, long long upto) {
    std::vector<Op> &v = S().pending[st];
    std::vector<Op> left;
    for (Op &o : v) {
        if (o.seq > upto) left.push_back(std::move(o));
        else if (o.src && std::memcmp(o.src, o.bytes.data(), o.bytes.size()) != 0) say("rewritten");
    }
    v.swap(left);
}

void enqueue(cudaStream_t st, const std::string &what, const void *src = nullptr, size_t n = 0) {
    State &s = S();
    if (s.capturing && st == s.capturing) return;
    if (st && !s.pending[nullptr].empty()) say("unordered " + what);
    Op o{++s.seq, nullptr, {}};
    if (src)
        for (auto &p : s.pinned)
            if ((const char *)src >= p.first && (const char *)src < p.first + p.second) {
                o.src = src;
                o.bytes.assign((const unsigned char *)src, (const unsigned char *)src + n);
            }
    s.pending[st].push_back(std::move(o));
}

void record(const void *fun, dim3 g, dim3 b, size_t smem, cudaStream_t st) {
    S().launches.push_back({S().names[fun], g, b, smem});
    enqueue(st, S().names[fun]);
}

// a null pointer among the buffers of a copy or clear
cudaError_t null_buffer() {
    say("null");
    return cudaErrorInvalidValue;
}

void note_clear(void *p, size_t n) {
    auto it = S().device.find((const char *)p);
    if (it != S().device.end() && n >= it->second) S().cleared.push_back(it->second);
}

}  // namespace

extern "C" {

// ---- the checks' side
const char *fake_report() { return S().report.c_str(); }
void fake_reset() {
    State &s = S();
    s.report.clear();
    s.launches.clear();
    s.attribute.clear();
    s.cleared.clear();
    s.mallocs_left = -1;
}
void fake_fail_malloc_after(long long n) { S().mallocs_left = n; }
size_t fake_device_bytes() {
    size_t n = 0;
    for (auto &p : S().device) n += p.second;
    return n;
}
int fake_launch_count() { return (int)S().launches.size(); }
const char *fake_launch(int k, int *grid, int *block) {
    const Launch &l = S().launches[k];
    *grid = (int)(l.grid.x * l.grid.y * l.grid.z);
    *block = (int)(l.block.x * l.block.y * l.block.z);
    return l.name.c_str();
}
int fake_cleared(size_t bytes) {
    int n = 0;
    for (size_t b : S().cleared) n += b == bytes;
    return n;
}

// ---- the runtime's side
void **__cudaRegisterFatBinary(void *) {
    static void *h;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *fun, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *,
                            int *) {
    S().names[fun] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t st) {
    S().grid = g;
    S().block = b;
    S().smem = smem;
    S().stream = st;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *st) {
    *g = S().grid;
    *b = S().block;
    *smem = S().smem;
    *(cudaStream_t *)st = S().stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *fun) {
    *k = (cudaKernel_t)fun;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void **, size_t smem, cudaStream_t st) {
    record((const void *)k, g, b, smem, st);
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *fun, void **) {
    record(fun, c->gridDim, c->blockDim, c->dynamicSmemBytes, c->stream);
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *fun, cudaFuncAttribute a, int value) {
    auto ins = S().attribute.insert({{fun, (int)a}, value});
    if (!ins.second && ins.first->second != value) say("attribute " + S().names[fun]);
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) {
    std::memset(a, 0, sizeof *a);
    a->numRegs = 64;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxRegistersPerMultiprocessor ? 65536 : 233472;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "error"; }

cudaError_t cudaMalloc(void **p, size_t n) {
    State &s = S();
    if (s.mallocs_left == 0) return cudaErrorMemoryAllocation;
    if (s.mallocs_left > 0) --s.mallocs_left;
    *p = std::calloc(1, n);
    s.device[(const char *)*p] = n;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    if (p && !S().device.erase((const char *)p)) say("freed twice");
    else std::free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) {
    *p = std::calloc(1, n);
    S().pinned[(const char *)*p] = n;
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) {
    S().pinned.erase((const char *)p);
    std::free(p);
    return cudaSuccess;
}

cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind k) {
    if (!d || !s) return null_buffer();
    complete(nullptr, S().seq);
    std::memcpy(d, s, n);
    if (k == cudaMemcpyHostToDevice) enqueue(nullptr, "copy");
    return cudaSuccess;
}
cudaError_t cudaMemcpy2D(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind k) {
    if (!d || !s) return null_buffer();
    complete(nullptr, S().seq);
    for (size_t r = 0; r < h; ++r) std::memcpy((char *)d + r * dp, (const char *)s + r * sp, w);
    if (k == cudaMemcpyHostToDevice) enqueue(nullptr, "copy");
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t st) {
    if (!d || !s) return null_buffer();
    enqueue(st, "copy", k == cudaMemcpyHostToDevice ? s : nullptr, n);
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind,
                              cudaStream_t st) {
    if (!d || !s) return null_buffer();
    enqueue(st, "copy");
    for (size_t r = 0; r < h; ++r) std::memcpy((char *)d + r * dp, (const char *)s + r * sp, w);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *p, int v, size_t n) {
    if (!p) return null_buffer();
    std::memset(p, v, n);
    note_clear(p, n);
    enqueue(nullptr, "clear");
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t st) {
    if (!p) return null_buffer();
    std::memset(p, v, n);
    note_clear(p, n);
    enqueue(st, "clear");
    return cudaSuccess;
}

cudaError_t cudaStreamCreateWithFlags(cudaStream_t *st, unsigned) {
    *st = (cudaStream_t)std::malloc(16);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t st) {
    S().pending.erase(st);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t st) {
    complete(st, S().seq);
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) {
    *e = (cudaEvent_t) new Event;
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
    delete (Event *)e;
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t st) {
    *(Event *)e = Event{st, S().seq};
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) {
    complete(((Event *)e)->stream, ((Event *)e)->seq);
    return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
    *ms = 0.0f;
    return cudaSuccess;
}

cudaError_t cudaStreamBeginCapture(cudaStream_t st, cudaStreamCaptureMode) {
    S().capturing = st;
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) {
    S().capturing = nullptr;
    *g = (cudaGraph_t)std::malloc(16);
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) {
    *x = (cudaGraphExec_t)std::malloc(16);
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
    std::free(g);
    return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) {
    std::free(x);
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t st) {
    enqueue(st, "graph");
    return cudaSuccess;
}

}  // extern "C"
