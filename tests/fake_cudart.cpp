// A CUDA runtime for host-side tests: the calls liblnr makes, on two pretended devices whose
// memory is host memory.  Kernels do not run; their launches are checked instead.  It follows
// the documented rules that the library's host code has to keep:
//  - a copy or fill of cudaMemcpy / cudaMemset from pageable memory is issued to the legacy
//    default stream and may still be in flight when the call returns, and non-blocking
//    streams do not wait for that stream (fk_get "unordered" counts work issued to one of them
//    meanwhile);
//  - a kernel's dynamic shared memory past 48 KiB needs the attribute set on the current device
//    (else the launch is refused and cudaGetLastError reports it once);
//  - a failed call's error stays for cudaGetLastError.
// fk_fail_alloc(k) fails the k-th allocation from now on; fk_refuse(name) refuses launches of
// the kernels whose name holds the text; fk_give_up(name, code) makes them store the code in the
// error word their parameters point to, as their bounded waits do when they run out.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <set>
#include <string>
#include <tuple>
#include <utility>
#include <vector>

namespace {

struct Alloc {
    size_t bytes;
    int device;  // -1: page-locked host memory
    uint64_t id;
};
struct Stream {
    bool blocking;
    bool capturing = false;
    std::set<uint64_t> deps;  // allocations the captured work uses
};
struct Graph {
    std::set<uint64_t> deps;
};

std::recursive_mutex mu;
std::map<uintptr_t, Alloc> allocs;
std::set<uint64_t> live;
std::map<const void*, std::string> names;
std::map<std::pair<int, const void*>, int> smem_attr;
std::map<std::string, long> counters;
uint64_t next_id = 1;
long fail_in = 0;
std::string refuse, give_up;
int give_up_code = 0;
bool pending_legacy = false;
thread_local int device = 0;
thread_local cudaError_t last = cudaSuccess;
thread_local struct { dim3 grid, block; size_t smem; cudaStream_t st; } call;

using Lock = std::lock_guard<std::recursive_mutex>;

cudaError_t set(cudaError_t e) {
    if (e != cudaSuccess) last = e;
    return e;
}

std::map<uintptr_t, Alloc>::iterator find(const void* p) {
    auto it = allocs.upper_bound((uintptr_t)p);
    if (it == allocs.begin()) return allocs.end();
    --it;
    return (uintptr_t)p < it->first + it->second.bytes ? it : allocs.end();
}

cudaError_t alloc(void** p, size_t n, int dev) {
    Lock l(mu);
    *p = nullptr;
    if (fail_in > 0 && --fail_in == 0) return set(cudaErrorMemoryAllocation);
    counters["allocs"]++;
    *p = calloc(n ? n : 1, 1);
    allocs[(uintptr_t)*p] = Alloc{n ? n : 1, dev, next_id};
    live.insert(next_id++);
    return cudaSuccess;
}

cudaError_t release(void* p) {
    Lock l(mu);
    if (!p) return cudaSuccess;
    auto it = allocs.find((uintptr_t)p);
    if (it == allocs.end()) return set(cudaErrorInvalidValue);
    live.erase(it->second.id);
    allocs.erase(it);
    free(p);
    return cudaSuccess;
}

Stream* of(cudaStream_t s) { return reinterpret_cast<Stream*>(s); }

// Work issued to stream s that reads or writes memory.
void issue(cudaStream_t s) {
    if (s && !of(s)->blocking && pending_legacy) counters["unordered"]++;
}

void use(cudaStream_t s, const void* p) {
    auto it = find(p);
    if (it != allocs.end() && s && of(s)->capturing) of(s)->deps.insert(it->second.id);
}

cudaError_t copy(void* d, const void* s, size_t n) {
    memcpy(d, s, n);
    return cudaSuccess;
}

CUresult encode(CUtensorMap* m, CUtensorMapDataType, cuuint32_t, void* addr, const cuuint64_t*, const cuuint64_t*,
                const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                CUtensorMapFloatOOBfill) {
    memset(m, 0, sizeof(*m));
    memcpy(m, &addr, sizeof(addr));
    return CUDA_SUCCESS;
}

}  // namespace

extern "C" {

long fk_get(const char* name) {
    Lock l(mu);
    return counters[name];
}
void fk_fail_alloc(long k) {
    Lock l(mu);
    fail_in = k;
}
void fk_refuse(const char* name) {
    Lock l(mu);
    refuse = name;
}
void fk_give_up(const char* name, int code) {
    Lock l(mu);
    give_up = name;
    give_up_code = code;
}

// ---- what nvcc's host code calls ----

void** __cudaRegisterFatBinary(void*) {
    static void* h;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    Lock l(mu);
    names[f] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t st) {
    call = {g, b, smem, st};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* st) {
    *g = call.grid;
    *b = call.block;
    *smem = call.smem;
    *static_cast<cudaStream_t*>(st) = call.st;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void** args, size_t smem, cudaStream_t st) {
    Lock l(mu);
    const void* f = reinterpret_cast<const void*>(k);
    const std::string& name = names[f];
    if (!g.x || !g.y || !g.z || !b.x) return set(cudaErrorInvalidConfiguration);
    auto at = smem_attr.find({device, f});
    if (smem > (at == smem_attr.end() ? 48u * 1024u : (size_t)at->second) ||
        (!refuse.empty() && name.find(refuse) != std::string::npos)) {
        counters["refused"]++;
        return set(cudaErrorInvalidValue);
    }
    counters["launches"]++;
    issue(st);
    const bool split = name.find("k_conv_split") != std::string::npos;
    if (split || name.find("k_conv_halo") != std::string::npos) {
        counters[split ? "conv_split" : "conv_halo"]++;
        const uint64_t* w = static_cast<const uint64_t*>(args[0]);  // one struct of more than 1024 bytes
        for (int i = 0; i < 128; ++i) {
            auto it = find(reinterpret_cast<const void*>(w[i]));
            if (it == allocs.end()) continue;
            use(st, reinterpret_cast<const void*>(w[i]));
            if (it->second.device >= 0 && it->second.device != device) counters["foreign"]++;
            if (it->second.bytes == sizeof(int) && !give_up.empty() && name.find(give_up) != std::string::npos)
                *reinterpret_cast<int*>(it->first) = give_up_code;
        }
    }
    return cudaSuccess;
}

// ---- runtime ----

cudaError_t cudaGetDeviceCount(int* n) {
    *n = 2;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
    device = d;
    return d < 2 ? cudaSuccess : set(cudaErrorInvalidDevice);
}
cudaError_t cudaGetDevice(int* d) {
    *d = device;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int d) {
    *v = a == cudaDevAttrMultiProcessorCount ? (d == 0 ? 152 : 76) : 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize(void) {
    Lock l(mu);
    pending_legacy = false;
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
    Lock l(mu);
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) smem_attr[{device, f}] = v;
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
    *f = reinterpret_cast<void*>(&encode);
    if (q) *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
    *n = 2;
    return cudaSuccess;
}

cudaError_t cudaMalloc(void** p, size_t n) { return alloc(p, n, device); }
cudaError_t cudaMallocHost(void** p, size_t n) { return alloc(p, n, -1); }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return alloc(p, n, -1); }
cudaError_t cudaFree(void* p) { return release(p); }
cudaError_t cudaFreeHost(void* p) { return release(p); }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { return alloc(p, 16u << 20, device); }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    Lock l(mu);
    auto it = find(p);
    a->type = it == allocs.end() ? cudaMemoryTypeUnregistered : it->second.device < 0 ? cudaMemoryTypeHost : cudaMemoryTypeDevice;
    return cudaSuccess;
}

cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) {
    Lock l(mu);
    if (k == cudaMemcpyHostToDevice && find(s) == allocs.end()) pending_legacy = true;
    if (k == cudaMemcpyDeviceToHost) pending_legacy = false;
    return copy(d, s, n);
}
cudaError_t cudaMemset(void* d, int v, size_t n) {
    Lock l(mu);
    pending_legacy = true;
    memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t st) {
    Lock l(mu);
    issue(st);
    use(st, d);
    use(st, s);
    return copy(d, s, n);
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) {
    Lock l(mu);
    issue(st);
    memset(d, v, n);
    return cudaSuccess;
}

cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned flags) {
    *s = reinterpret_cast<cudaStream_t>(new Stream{!(flags & cudaStreamNonBlocking)});
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
    delete of(s);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    Lock l(mu);
    if (!s || of(s)->blocking) pending_legacy = false;
    return cudaSuccess;
}
cudaError_t cudaStreamQuery(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* c) {
    *c = s && of(s)->capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
    Lock l(mu);
    of(s)->capturing = true;
    of(s)->deps.clear();
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) {
    Lock l(mu);
    of(s)->capturing = false;
    *g = reinterpret_cast<cudaGraph_t>(new Graph{of(s)->deps});
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long) {
    *e = reinterpret_cast<cudaGraphExec_t>(new Graph(*reinterpret_cast<Graph*>(g)));
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
    delete reinterpret_cast<Graph*>(g);
    return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) {
    delete reinterpret_cast<Graph*>(e);
    return cudaSuccess;
}
// "stale": a replay of work on memory that has been freed
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t st) {
    Lock l(mu);
    counters["graphs"]++;
    issue(st);
    for (uint64_t id : reinterpret_cast<Graph*>(e)->deps)
        if (!live.count(id)) {
            counters["stale"]++;
            break;
        }
    return cudaSuccess;
}

cudaError_t cudaEventCreate(cudaEvent_t* e) {
    *e = reinterpret_cast<cudaEvent_t>(new int);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
    delete reinterpret_cast<int*>(e);
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    *ms = 1.0f;
    return cudaSuccess;
}

}  // extern "C"
