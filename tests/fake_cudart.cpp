// A stand-in for the CUDA runtime, for tests of the library's host code on a machine without a GPU: linked
// with the library's objects in place of the real one.  "Device" memory is host memory; kernels do
// not run, their launches are recorded.  Of the selection the solve's loop sees what it needs: each
// one (or each replayed iteration) advances the mapped view after a set delay, with all signals
// active for a set number of iterations and none after them.
#include <cuda.h>

#include <atomic>
#include <chrono>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include "../paper_1302_5010_gb300/csrc/mpl_internal.cuh"

namespace {

struct Graph {
    bool iteration = false;
    mpl::Dev d{};
};

std::mutex mu;
std::map<const void*, std::string> names;  // kernels by host function
std::map<std::string, int> counts;         // calls by name of the runtime function or kernel
std::vector<std::string> log_;             // the same in order
std::map<std::string, mpl::Dev> devs;      // the Dev argument of each kernel's last launch
std::map<void*, size_t> live;              // device allocations
std::atomic<int> pending{0};
thread_local Graph* capture = nullptr;
int regs = 96, fail_malloc = 0, iterations = 1, delay_us = 0, view_on = 1;
unsigned flags = 0;
const void* train_part = nullptr;

void note(const char* what) {
    std::lock_guard<std::mutex> l(mu);
    ++counts[what];
    log_.push_back(what);
}

void advance(const mpl::Dev& d) {
    if (!view_on || !d.view) return;
    ++pending;
    auto work = [v = d.view, p = d.p] {
        if (delay_us) std::this_thread::sleep_for(std::chrono::microseconds(delay_us));
        const unsigned it = v->seq + 1u;
        v->act_next = (int)it < iterations ? p : 0;
        v->fin_n = 0;
        std::atomic_thread_fence(std::memory_order_release);
        *const_cast<volatile unsigned*>(&v->seq) = it;
        --pending;
    };
    if (delay_us) std::thread(work).detach();
    else work();
}

void drain() {
    while (pending.load()) std::this_thread::sleep_for(std::chrono::microseconds(20));
}

cudaError_t launch(const void* f, void** args) {
    const std::string& n = names.at(f);
    note(n.c_str());
    const bool fused = n.find("k_select") != std::string::npos && *static_cast<int*>(args[5]) != 0;
    const bool takes_dev = n.find("k_select") != std::string::npos || n.find("k_compact") != std::string::npos ||
                           n.find("k_corr_") != std::string::npos;
    if (takes_dev) {
        const mpl::Dev& d = *static_cast<const mpl::Dev*>(args[0]);
        {
            std::lock_guard<std::mutex> l(mu);
            devs[n] = d;
        }
        if (fused || n.find("k_compact") != std::string::npos) {
            if (capture) {
                capture->iteration = true;
                capture->d = d;
            } else {
                advance(d);
            }
        }
    }
    if (n.find("k_train_fwd_bwd") != std::string::npos) train_part = *static_cast<void**>(args[6]);
    return cudaSuccess;
}

CUresult fake_encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                     const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                     CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
    return CUDA_SUCCESS;
}
CUresult fake_context(CUcontext* c) {
    *c = reinterpret_cast<CUcontext>(&mu);
    return CUDA_SUCCESS;
}

template <typename T>
cudaError_t handle(T* out) {
    *out = reinterpret_cast<T>(std::malloc(1));
    return cudaSuccess;
}

}  // namespace

extern "C" {

// ---- what the tests set and read
void fake_set(int regs_, int fail_malloc_, int iterations_, int delay_us_, int view_on_, unsigned flags_) {
    drain();
    regs = regs_;
    fail_malloc = fail_malloc_;
    iterations = iterations_;
    delay_us = delay_us_;
    view_on = view_on_;
    flags = flags_;
    std::lock_guard<std::mutex> l(mu);
    counts.clear();
    log_.clear();
}
// Calls whose name contains `what`; the position of the last one in the log, or -1.
int fake_count(const char* what) {
    std::lock_guard<std::mutex> l(mu);
    int c = 0;
    for (auto& e : counts)
        if (e.first.find(what) != std::string::npos) c += e.second;
    return c;
}
int fake_last(const char* what) {
    std::lock_guard<std::mutex> l(mu);
    for (int i = (int)log_.size() - 1; i >= 0; --i)
        if (log_[i].find(what) != std::string::npos) return i;
    return -1;
}
int fake_live() { return (int)live.size(); }
int fake_train_part_null() { return train_part == nullptr; }
// bound_c, bound_f32, bound_q, bound_c32, bound_sub of the last launch of a kernel
int fake_bounds(const char* kernel, float* out) {
    for (auto& e : devs)
        if (e.first.find(kernel) != std::string::npos) {
            out[0] = e.second.bound_c;
            out[1] = e.second.bound_f32;
            out[2] = e.second.bound_q;
            out[3] = e.second.bound_c32;
            out[4] = e.second.bound_sub;
            return 1;
        }
    return 0;
}

// ---- kernels
void** __cudaRegisterFatBinary(void*) { return reinterpret_cast<void**>(&mu); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
static thread_local struct { dim3 g, b; size_t s; void* st; } conf;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, cudaStream_t st) {
    conf = {g, b, s, st};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
    *g = conf.g;
    *b = conf.b;
    *s = conf.s;
    *static_cast<void**>(st) = conf.st;
    return cudaSuccess;
}
cudaError_t CUDARTAPI __cudaGetKernel(cudaKernel_t* k, const void* f) {
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
    return cudaSuccess;
}
cudaError_t CUDARTAPI __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void** args, size_t, cudaStream_t) {
    return launch(k, args);
}
cudaError_t CUDARTAPI cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void* f, void** args) { return launch(f, args); }
cudaError_t CUDARTAPI cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
    std::memset(a, 0, sizeof(*a));
    a->numRegs = regs;
    return cudaSuccess;
}
cudaError_t CUDARTAPI cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t CUDARTAPI cudaGetSymbolAddress(void** p, const void*) {
    static char scratch[1 << 20];
    *p = scratch;
    return cudaSuccess;
}
cudaError_t CUDARTAPI cudaGetDriverEntryPointByVersion(const char* s, void** f, unsigned, unsigned long long,
                                                       cudaDriverEntryPointQueryResult* r) {
    *f = std::strstr(s, "TensorMap") ? reinterpret_cast<void*>(&fake_encode) : reinterpret_cast<void*>(&fake_context);
    if (r) *r = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}

// ---- device, errors
cudaError_t CUDARTAPI cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t CUDARTAPI cudaSetDevice(int) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaGetDeviceFlags(unsigned* f) { *f = flags; return cudaSuccess; }
cudaError_t CUDARTAPI cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t CUDARTAPI cudaDeviceGetStreamPriorityRange(int* a, int* b) { *a = *b = 0; return cudaSuccess; }
cudaError_t CUDARTAPI cudaDeviceSynchronize() { note("cudaDeviceSynchronize"); drain(); return cudaSuccess; }
cudaError_t CUDARTAPI cudaGetLastError() { return cudaSuccess; }
const char* CUDARTAPI cudaGetErrorString(cudaError_t) { return "error"; }

// ---- memory
cudaError_t CUDARTAPI cudaMalloc(void** p, size_t n) {
    *p = nullptr;
    if (fail_malloc && --fail_malloc == 0) return cudaErrorMemoryAllocation;
    *p = std::calloc(1, n ? n : 1);
    std::lock_guard<std::mutex> l(mu);
    live[*p] = n;
    return cudaSuccess;
}
cudaError_t CUDARTAPI cudaFree(void* p) {
    std::lock_guard<std::mutex> l(mu);
    live.erase(p);
    std::free(p);
    return cudaSuccess;
}
cudaError_t CUDARTAPI cudaMallocHost(void** p, size_t n) { *p = std::calloc(1, n); return cudaSuccess; }
cudaError_t CUDARTAPI cudaHostAlloc(void** p, size_t n, unsigned) { *p = std::calloc(1, n); return cudaSuccess; }
cudaError_t CUDARTAPI cudaFreeHost(void* p) { std::free(p); return cudaSuccess; }
cudaError_t CUDARTAPI cudaMemGetInfo(size_t* f, size_t* t) { *f = *t = (size_t)1 << 38; return cudaSuccess; }
cudaError_t CUDARTAPI cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t CUDARTAPI cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t CUDARTAPI cudaMemset(void* d, int v, size_t n) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t CUDARTAPI cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t CUDARTAPI cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) {
    std::memset(a, 0, sizeof(*a));
    a->type = cudaMemoryTypeDevice;
    return cudaSuccess;
}

// ---- streams, events, graphs
cudaError_t CUDARTAPI cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int) { return handle(s); }
cudaError_t CUDARTAPI cudaStreamDestroy(cudaStream_t s) { std::free(s); return cudaSuccess; }
cudaError_t CUDARTAPI cudaStreamQuery(cudaStream_t) {
    note("cudaStreamQuery");
    return pending.load() ? cudaErrorNotReady : cudaSuccess;
}
cudaError_t CUDARTAPI cudaStreamSynchronize(cudaStream_t) { note("cudaStreamSynchronize"); drain(); return cudaSuccess; }
cudaError_t CUDARTAPI cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaEventCreate(cudaEvent_t* e) { return handle(e); }
cudaError_t CUDARTAPI cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return handle(e); }
cudaError_t CUDARTAPI cudaEventDestroy(cudaEvent_t e) { std::free(e); return cudaSuccess; }
cudaError_t CUDARTAPI cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    note("cudaEventElapsedTime");
    *ms = 1.f;
    return cudaSuccess;
}
cudaError_t CUDARTAPI cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { capture = new Graph; return cudaSuccess; }
cudaError_t CUDARTAPI cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
    *g = reinterpret_cast<cudaGraph_t>(capture);
    capture = nullptr;
    return cudaSuccess;
}
cudaError_t CUDARTAPI cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long) {
    *e = reinterpret_cast<cudaGraphExec_t>(new Graph(*reinterpret_cast<Graph*>(g)));
    return cudaSuccess;
}
cudaError_t CUDARTAPI cudaGraphDestroy(cudaGraph_t g) { delete reinterpret_cast<Graph*>(g); return cudaSuccess; }
cudaError_t CUDARTAPI cudaGraphExecDestroy(cudaGraphExec_t g) { delete reinterpret_cast<Graph*>(g); return cudaSuccess; }
cudaError_t CUDARTAPI cudaGraphLaunch(cudaGraphExec_t g, cudaStream_t) {
    note("cudaGraphLaunch");
    Graph* q = reinterpret_cast<Graph*>(g);
    if (q->iteration) advance(q->d);
    return cudaSuccess;
}

}  // extern "C"
