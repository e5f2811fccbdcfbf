// A CUDA runtime without a device, for CPU tests of the library's host code:
// the library's objects are linked against it instead of libcudart.  Memory is
// host memory and kernels do not run; calls are recorded, a launch is refused
// like the runtime refuses it (dynamic shared memory above the limit of that
// kernel on that device), and a test can make a named call fail.
#include <cuda_runtime_api.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <utility>
#include <vector>

struct CUgraph_st { std::vector<std::string> calls; };

namespace {

struct State {
    int dev = 0;
    cudaError_t last = cudaSuccess;
    std::map<std::pair<int, const void*>, int> limit;  // dynamic shared memory per device and kernel
    std::map<const void*, std::string> names;
    std::map<const void*, void*> symbols;
    std::vector<std::string> log;
    bool capturing = false;
    std::vector<std::string> captured;
    std::string fail_at;                               // call or kernel name that fails, once, ...
    int fail_after = 0;                                // ... after this many successes
    std::vector<int> table_items;                      // (instance, chunk) of the last threshold-table batch launch
    int table_chunk = 0;
    dim3 grid, block;
    size_t smem = 0;
    cudaStream_t stream = nullptr;
    std::string text;
};
State& S()
{
    static State s;
    return s;
}

cudaError_t ret(cudaError_t e)
{
    if (e != cudaSuccess) S().last = e;
    return e;
}
cudaError_t call(const char* name)
{
    State& s = S();
    if (!s.fail_at.empty() && std::string(name).find(s.fail_at) != std::string::npos && s.fail_after-- == 0) {
        s.fail_at.clear();
        return ret(cudaErrorUnknown);
    }
    return cudaSuccess;
}
void record(const std::string& what)
{
    State& s = S();
    (s.capturing ? s.captured : s.log).push_back(what);
}
cudaError_t launch(const void* f, dim3 grid, void** args, size_t smem, cudaStream_t st)
{
    State& s = S();
    const std::string& name = s.names[f];
    const auto lim = s.limit.find({s.dev, f});
    if (smem > (size_t)(lim == s.limit.end() ? 48 * 1024 : lim->second) || grid.x * grid.y * grid.z == 0)
        return ret(cudaErrorInvalidValue);
    const cudaError_t e = call(name.c_str());
    if (e != cudaSuccess) return e;
    if (name.find("sweep_batch_table_kernel") != std::string::npos) {
        // (RealStep, instances, items, number of items, chunk, counter)
        const int* items = *static_cast<const int**>(args[2]);
        s.table_items.assign(items, items + 2 * *static_cast<int*>(args[3]));
        s.table_chunk = *static_cast<int*>(args[4]);
    }
    record("launch " + name + " stream " + std::to_string((size_t)st) + " grid " + std::to_string(grid.x));
    return cudaSuccess;
}
void* symbol(const void* sym)
{
    void*& p = S().symbols[sym];
    if (!p) p = std::calloc(1, 1 << 23);
    return p;
}

}  // namespace

extern "C" {

// ---- the tests' side
void fake_reset()
{
    S().log.clear();
    S().fail_at.clear();
    S().last = cudaSuccess;
}
void fake_device(int dev) { S().dev = dev; }
void fake_fail(const char* name, int after)
{
    S().fail_at = name;
    S().fail_after = after;
}
const char* fake_log()
{
    State& s = S();
    s.text.clear();
    for (const auto& l : s.log) s.text += l + "\n";
    return s.text.c_str();
}
int fake_table_chunk() { return S().table_chunk; }
int fake_table_items(int* out, int n)
{
    const auto& t = S().table_items;
    for (int i = 0; i < n && i < (int)t.size(); ++i) out[i] = t[i];
    return (int)t.size() / 2;
}

// ---- registration and launches as nvcc's host code makes them
void** __cudaRegisterFatBinary(void*) { return reinterpret_cast<void**>(&S()); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*)
{
    S().names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st* st)
{
    State& s = S();
    s.grid = grid; s.block = block; s.smem = smem; s.stream = st;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* st)
{
    State& s = S();
    *grid = s.grid; *block = s.block; *smem = s.smem;
    *static_cast<cudaStream_t*>(st) = s.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f)
{
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void** args, size_t smem, cudaStream_t st)
{
    return launch(k, grid, args, smem, st);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args)
{
    return launch(f, c->gridDim, args, c->dynamicSmemBytes, c->stream);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v)
{
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) S().limit[{S().dev, f}] = v;
    return call("cudaFuncSetAttribute");
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int threads, size_t smem, unsigned)
{
    *n = (int)std::min<size_t>(2048 / threads, (227 << 10) / std::max<size_t>(smem, 1));
    return cudaSuccess;
}

// ---- device, memory
cudaError_t cudaGetDevice(int* d) { *d = S().dev; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = S().last; S().last = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : e == cudaErrorInvalidValue ? "invalid argument" : "failed by the test"; }
cudaError_t cudaMalloc(void** p, size_t n)
{
    const cudaError_t e = call("cudaMalloc");
    *p = e == cudaSuccess ? std::memset(std::aligned_alloc(256, (n + 255) / 256 * 256), 0, n) : nullptr;
    return e;
}
cudaError_t cudaFree(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    if (!S().capturing) std::memcpy(d, s, n);
    return call("cudaMemcpyAsync");
}
cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind, cudaStream_t)
{
    for (size_t i = 0; i < h; ++i) std::memcpy((char*)d + i * dp, (const char*)s + i * sp, w);
    return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t)
{
    if (!S().capturing) std::memset(d, v, n);
    return call("cudaMemsetAsync");
}
cudaError_t cudaGetSymbolAddress(void** p, const void* sym) { *p = symbol(sym); return cudaSuccess; }
cudaError_t cudaMemcpyToSymbolAsync(const void* sym, const void* s, size_t n, size_t off, cudaMemcpyKind, cudaStream_t)
{
    std::memcpy((char*)symbol(sym) + off, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyFromSymbolAsync(void* d, const void* sym, size_t n, size_t off, cudaMemcpyKind, cudaStream_t)
{
    std::memcpy(d, (char*)symbol(sym) + off, n);
    return cudaSuccess;
}

// ---- streams, events, graphs
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* st, unsigned)
{
    static size_t next = 0x5000;
    *st = reinterpret_cast<cudaStream_t>(next++);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t st)
{
    record("synchronize stream " + std::to_string((size_t)st));
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = static_cast<cudaEvent_t>(std::malloc(1)); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { std::free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t st)
{
    record("record " + std::to_string((size_t)e) + " stream " + std::to_string((size_t)st));
    return call("cudaEventRecord");
}
cudaError_t cudaStreamWaitEvent(cudaStream_t st, cudaEvent_t e, unsigned)
{
    record("wait " + std::to_string((size_t)e) + " stream " + std::to_string((size_t)st));
    return call("cudaStreamWaitEvent");
}
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.0f; return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s)
{
    *s = S().capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode)
{
    const cudaError_t e = call("cudaStreamBeginCapture");
    if (e != cudaSuccess) return e;
    S().capturing = true;
    S().captured.clear();
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g)
{
    S().capturing = false;
    *g = nullptr;
    const cudaError_t e = call("cudaStreamEndCapture");
    if (e == cudaSuccess) *g = new CUgraph_st{S().captured};
    return e;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t g, unsigned long long)
{
    *x = nullptr;
    const cudaError_t e = call("cudaGraphInstantiate");
    if (e == cudaSuccess) *x = reinterpret_cast<cudaGraphExec_t>(new CUgraph_st(*g));
    return e;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t)
{
    const cudaError_t e = call("cudaGraphLaunch");
    if (e == cudaSuccess)
        for (const auto& c : reinterpret_cast<CUgraph_st*>(x)->calls) S().log.push_back(c);
    return e;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { delete g; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { delete reinterpret_cast<CUgraph_st*>(x); return cudaSuccess; }

}  // extern "C"
