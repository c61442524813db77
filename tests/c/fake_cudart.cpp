// A CUDA runtime without a GPU, for tests of the host code: "device" memory is zeroed host memory, copies
// are memcpy, kernel launches do nothing. A chosen cudaMalloc fails; bytes in use are counted; and a launch
// of a watched kernel with a null pointer among its arguments is noted. Linked with the library's own
// objects in place of the CUDA runtime, together with a hook that installs a hierarchy without kernels.
#include <cxxabi.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "../../paper_2403_04491_gb300/csrc/amg.h"
#include "../../paper_2403_04491_gb300/csrc/problem.h"
#include "../../paper_2403_04491_gb300/csrc/vcycle.h"

namespace {

struct Kernel {
    std::string name;                // demangled, up to the parameter list
    std::vector<bool> pointer;       // which parameters are pointers
};
std::map<const void*, Kernel> kernels;
std::map<void*, size_t> blocks;
size_t in_use = 0;
long countdown = 0;
std::vector<std::string> watched;
std::string null_launch;

Kernel parse(const char* mangled) {
    int status = 0;
    char* text = abi::__cxa_demangle(mangled, nullptr, nullptr, &status);
    Kernel k;
    std::string s = text ? text : mangled;
    std::free(text);
    int depth = 0;
    size_t open = std::string::npos;
    // the parameter list is the last top-level parenthesis ("(anonymous namespace)" comes before it)
    for (size_t i = s.size(); i-- > 0;) {
        if (s[i] == ')') ++depth;
        if (s[i] == '(' && --depth == 0) {
            open = i;
            break;
        }
    }
    if (open == std::string::npos) return k;
    k.name = s.substr(0, open);
    depth = 0;
    char last = 0;
    for (size_t i = open + 1; i < s.size(); ++i) {
        const char c = s[i];
        if (c == '(' || c == '<') ++depth;
        if (depth == 0 && (c == ',' || c == ')')) {
            k.pointer.push_back(last == '*');
            if (c == ')') break;
        }
        if (c == ')' || c == '>') --depth;
        if (c != ' ') last = c;
    }
    return k;
}

void launched(const void* fun, void** args) {
    const Kernel& k = kernels[fun];
    bool watch = false;
    for (const std::string& w : watched) watch |= k.name.find(w) != std::string::npos;
    for (size_t i = 0; watch && i < k.pointer.size(); ++i)
        if (k.pointer[i] && !*static_cast<void**>(args[i]) && null_launch.empty())
            null_launch = k.name + " argument " + std::to_string(i);
}

struct Config {
    dim3 grid, block;
    size_t shared;
    void* stream;
} config;

}  // namespace

extern "C" {

void fake_fail_at(long k) { countdown = k; }
long fake_pending() { return countdown; }
size_t fake_in_use() { return in_use; }
void fake_watch(const char* name) { watched.push_back(name); }
const char* fake_null_launch() { return null_launch.c_str(); }

// a hierarchy of one level, the identity, by the library's own hand-over from the host
int fake_identity_hierarchy(knp_problem* p, int inner_cg_max_it) {
    return knp::guarded([&] {
        const int64_t n = p->n_nodes;
        knp::HostHierarchy H;
        H.levels.resize(1);
        knp::HostLevel& L = H.levels[0];
        L.A.n_rows = L.A.n_cols = n;
        for (int64_t r = 0; r <= n; ++r) L.A.ptr.push_back(r);
        for (int64_t r = 0; r < n; ++r) L.A.col.push_back((int32_t)r);
        L.A.val.assign(4 * n, 1.0);
        L.dinv.assign(4 * n, 1.0);
        for (int f = 0; f < 4; ++f) {
            L.lmax[f] = 1.1;
            L.lmin[f] = 0.3;
        }
        H.nc = n;
        H.coarse_inv.assign(4 * n * n, 0.0);
        knp::amg_upload(p, H, 0, 2, 2);
        p->amg->inner_cg_max_it = inner_cg_max_it;
        p->amg->inner_cg_rtol = 1e-8;
    });
}

// ---- the runtime
void** __cudaRegisterFatBinary(void*) {
    static void* handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*,
                            int*) {
    kernels[host] = parse(name);
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, cudaStream_t st) {
    config = {g, b, s, st};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
    *g = config.grid;
    *b = config.block;
    *s = config.shared;
    *static_cast<void**>(st) = config.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* fun) {
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(fun));
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void** args, size_t, cudaStream_t) {
    launched(k, args);
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void* fun, void** args) {
    launched(fun, args);
    return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) {
    if (countdown > 0 && --countdown == 0) return cudaErrorMemoryAllocation;
    *p = std::calloc(n, 1);
    blocks[*p] = n;
    in_use += n;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    auto it = blocks.find(p);
    if (it == blocks.end()) return cudaErrorInvalidValue;
    in_use -= it->second;
    blocks.erase(it);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) {
    *p = std::calloc(n, 1);
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) { return cudaHostAlloc(p, n, 0); }
cudaError_t cudaFreeHost(void* p) {
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyToSymbolAsync(const void*, const void*, size_t, size_t, cudaMemcpyKind, cudaStream_t) {
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
    std::memset(d, v, n);
    return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "an error of the fake runtime"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceFlags(unsigned* f) {
    *f = 0;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamQuery(cudaStream_t) { return cudaSuccess; }
// not reached by the host code under test
cudaError_t cudaGetSymbolAddress(void**, const void*) { return cudaErrorNotSupported; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes*, const void*) { return cudaErrorNotSupported; }
cudaError_t cudaEventCreate(cudaEvent_t*) { return cudaErrorNotSupported; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t*, unsigned) { return cudaErrorNotSupported; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaErrorNotSupported; }
cudaError_t cudaEventElapsedTime(float*, cudaEvent_t, cudaEvent_t) { return cudaErrorNotSupported; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaErrorNotSupported; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t*, unsigned) { return cudaErrorNotSupported; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
}
