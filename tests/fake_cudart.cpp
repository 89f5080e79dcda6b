// A stand-in for the CUDA runtime that runs nothing: the host side of the library is linked against it so that its
// decisions (what is copied, launched, looked up and waited for, and what happens when a call fails) can be tested
// without a GPU.  "Device" memory is host memory; copies are done at once but count as in flight until their stream, or
// a stream that waits for an event behind them, has been synchronised; kernels are only noted by name.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <new>
#include <set>
#include <string>
#include <vector>

namespace {
struct Op {
    std::string what;
    bool done = false;
};
struct Stream {
    std::vector<size_t> ops;        // indices into g_ops, in order
};
struct Event {
    std::vector<size_t> behind;     // operations that an event stands for
};
struct Range {
    uintptr_t start;
    size_t size;
};
std::vector<Op> g_ops;
std::map<void*, Stream> g_streams;
std::map<void*, Event> g_events;
std::map<const void*, std::string>& names() {        // kernels register themselves before this file's globals exist
    static std::map<const void*, std::string> m;
    return m;
}
std::vector<Range> g_pinned;
std::string g_log, g_shapes;
int g_calls = 0, g_fail_at = 0, g_next_handle = 1;
int g_news = 0, g_new_fails_at = 0, g_quiet = 0;
struct Quiet {      // allocations of the stand-in itself neither count nor fail
    Quiet() { ++g_quiet; }
    ~Quiet() { --g_quiet; }
};
std::set<void*> g_device;

void note(const std::string& s) { g_log += s + "\n"; }
// One more call that may fail; true: it does.
bool fails() { return ++g_calls == g_fail_at; }
void enqueue(void* st, const std::string& what) {
    g_ops.push_back({what});
    g_streams[st].ops.push_back(g_ops.size() - 1);
}
std::string name_of(const void* fn) {
    auto it = names().find(fn);
    return it == names().end() ? "?" : it->second;
}
std::string at(const void* p) { return std::to_string((unsigned long long)(uintptr_t)p); }
}  // namespace

// Host allocations of the library: the k-th fails.
void* operator new(size_t n) {
    if (!g_quiet && ++g_news == g_new_fails_at) throw std::bad_alloc();
    void* p = malloc(n ? n : 1);
    if (!p) throw std::bad_alloc();
    return p;
}
void* operator new(size_t n, const std::nothrow_t&) noexcept {
    if (!g_quiet && ++g_news == g_new_fails_at) return nullptr;
    return malloc(n ? n : 1);
}
void operator delete(void* p) noexcept { free(p); }
void operator delete(void* p, size_t) noexcept { free(p); }
void operator delete(void* p, const std::nothrow_t&) noexcept { free(p); }

extern "C" {

// ---- control
void fake_fail_new(int at) {
    g_news = 0;
    g_new_fails_at = at;
}
int fake_news() { return g_news; }
void fake_reset(int fail_at) {
    Quiet quiet;
    g_ops.clear();
    g_streams.clear();
    g_events.clear();
    g_log.clear();
    g_shapes.clear();
    g_calls = 0;
    g_fail_at = fail_at;
}
int fake_calls() { return g_calls; }
const char* fake_log() { return g_log.c_str(); }
// "<kernel> <blocks> <threads> <dynamic shared memory>" of every launch by cudaLaunchKernel
const char* fake_shapes() { return g_shapes.c_str(); }
int fake_in_flight() {
    int k = 0;
    for (const Op& o : g_ops) k += !o.done;
    return k;
}
int fake_allocations() { return (int)g_device.size(); }
void fake_pin(const void* p, size_t size) {
    Quiet quiet;
    g_pinned.push_back({(uintptr_t)p, size});
}
void fake_unpin_all() { g_pinned.clear(); }

// ---- runtime
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "planted"; }
cudaError_t cudaDeviceSynchronize() {
    for (Op& o : g_ops) o.done = true;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 148 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 0;
    return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) {
    Quiet quiet;
    note("malloc " + std::to_string(n));
    if (fails()) return cudaErrorMemoryAllocation;
    *p = aligned_alloc(256, (n + 255) & ~size_t(255));
    memset(*p, 0, n);      // no kernel writes it: a status is that of a valid sequence
    g_device.insert(*p);
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    Quiet quiet;
    if (p) {
        note("free");
        if (!g_device.erase(p)) note("free of a foreign pointer");
        else free(p);
    }
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) {
    Quiet quiet;
    note("malloc_host " + std::to_string(n));
    if (fails()) return cudaErrorMemoryAllocation;
    return *p = malloc(n), cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) { return free(p), cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
    Quiet quiet;
    note("memcpy " + std::to_string(n));
    if (fails()) return cudaErrorUnknown;
    return memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind kind, cudaStream_t st) {
    Quiet quiet;
    note(std::string("copy ") + (kind == cudaMemcpyHostToDevice ? "h2d " : "d2h ") + at(s) + " " + std::to_string(n));
    if (fails()) return cudaErrorUnknown;
    enqueue(st, "copy");
    return memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) { return memset(d, v, n), cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { return memset(d, v, n), cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    if (fails()) return cudaErrorUnknown;
    return *s = (cudaStream_t)(uintptr_t)(0x1000 + g_next_handle++), cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
    if (fails()) return cudaErrorUnknown;
    return *e = (cudaEvent_t)(uintptr_t)(0x1000 + g_next_handle++), cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t st) {
    Quiet quiet;
    if (fails() || !e) return cudaErrorUnknown;
    g_events[e].behind = g_streams[st].ops;
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t st, cudaEvent_t e, unsigned) {
    Quiet quiet;
    if (fails() || !e) return cudaErrorUnknown;
    std::vector<size_t>& ops = g_streams[st].ops;
    for (size_t i : g_events[e].behind)
        if (std::find(ops.begin(), ops.end(), i) == ops.end()) ops.push_back(i);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t st) {
    Quiet quiet;
    note("sync");
    const bool bad = fails();       // reported, but the work is over all the same
    for (size_t i : g_streams[st].ops) g_ops[i].done = true;
    return bad ? cudaErrorUnknown : cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void* fn) {
    Quiet quiet;
    note("lookup " + name_of(fn));
    if (fails()) return cudaErrorUnknown;
    memset(a, 0, sizeof *a);
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* fn, cudaFuncAttribute, int) {
    Quiet quiet;
    note("lookup " + name_of(fn));
    return fails() ? cudaErrorUnknown : cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* nb, const void* fn, int threads, size_t smem) {
    Quiet quiet;
    note("lookup " + name_of(fn));
    if (fails()) return cudaErrorUnknown;
    const size_t regs = 64, by_smem = 233472 / (smem + 1024), by_regs = 65536 / (regs * threads);
    *nb = (int)std::min<size_t>(std::min<size_t>(by_smem, by_regs), 32);
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* nb, const void* fn, int threads, size_t smem, unsigned) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(nb, fn, threads, smem);
}
cudaError_t cudaLaunchKernel(const void* fn, dim3 grid, dim3 block, void**, size_t smem, cudaStream_t st) {
    Quiet quiet;
    note("launch " + name_of(fn));
    g_shapes += name_of(fn) + " " + std::to_string(grid.x) + " " + std::to_string(block.x) + " " + std::to_string(smem) + "\n";
    if (fails()) return cudaErrorUnknown;
    return enqueue(st, "launch"), cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* fn, void** args) {
    return cudaLaunchKernel(fn, c->gridDim, c->blockDim, args, c->dynamicSmemBytes, c->stream);
}
cudaError_t cudaGetSymbolAddress(void** p, const void* symbol) { return *p = (void*)symbol, cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    memset(a, 0, sizeof *a);
    for (const Range& r : g_pinned)
        if ((uintptr_t)p >= r.start && (uintptr_t)p < r.start + r.size) {
            a->type = cudaMemoryTypeHost;
            a->devicePointer = a->hostPointer = (void*)p;
        }
    return cudaSuccess;
}
static CUresult pointer_get_attributes(unsigned k, CUpointer_attribute* what, void** out, CUdeviceptr p) {
    const Range* in = nullptr;
    for (const Range& r : g_pinned)
        if (p >= r.start && p < r.start + r.size) in = &r;
    for (unsigned i = 0; i < k; ++i) switch (what[i]) {
            case CU_POINTER_ATTRIBUTE_MEMORY_TYPE: *(unsigned*)out[i] = in ? CU_MEMORYTYPE_HOST : 0; break;
            case CU_POINTER_ATTRIBUTE_DEVICE_POINTER: *(CUdeviceptr*)out[i] = in ? p : 0; break;
            case CU_POINTER_ATTRIBUTE_IS_MANAGED: *(unsigned*)out[i] = 0; break;
            case CU_POINTER_ATTRIBUTE_RANGE_START_ADDR: *(CUdeviceptr*)out[i] = in ? in->start : 0; break;
            case CU_POINTER_ATTRIBUTE_RANGE_SIZE: *(size_t*)out[i] = in ? in->size : 0; break;
            default: return CUDA_ERROR_INVALID_VALUE;
        }
    return CUDA_SUCCESS;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** fn, unsigned, unsigned long long, cudaDriverEntryPointQueryResult* r) {
    const bool known = !strcmp(name, "cuPointerGetAttributes");
    *fn = known ? (void*)pointer_get_attributes : nullptr;
    if (r) *r = known ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
    return known ? cudaSuccess : cudaErrorUnknown;
}

// ---- what the compiler's host code calls
static dim3 g_grid, g_block;
static size_t g_smem;
static void* g_stream;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t sm, void* st) {
    g_grid = g;
    g_block = b;
    g_smem = sm;
    g_stream = st;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* sm, void* st) {
    *g = g_grid;
    *b = g_block;
    *sm = g_smem;
    *(void**)st = g_stream;
    return cudaSuccess;
}
// every source file registers a module, and then its kernels with it
static std::map<void*, std::string>& modules() {
    static std::map<void*, std::string> m;
    return m;
}
void** __cudaRegisterFatBinary(void*) { return (void**)calloc(1, sizeof(void*)); }
const char* fake_modules() {
    static std::string all;
    all.clear();
    for (auto& m : modules()) all += m.second + "\n";
    return all.c_str();
}
void __cudaRegisterFatBinaryEnd(void**) {}
char __cudaInitModule(void**) { return 1; }
void __cudaUnregisterFatBinary(void** h) { free(h); }
void __cudaRegisterFunction(void** module, const char* host, char*, const char* name, int, void*, void*, void*, void*, int*) {
    modules()[module] += std::string(name) + " ";
    names()[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
}
