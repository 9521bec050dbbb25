// A stand-in for the CUDA runtime, for the library's host code on a machine
// without a GPU: it hands out addresses without memory, records what is
// launched, copied and waited for, and can fail a chosen call. No kernel runs.
// Device: 152 SMs, 129 MiB of L2.
#include "host_runtime.h"

#include <cuda.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>

std::vector<Work> g_work;
std::map<char*, size_t> g_device;
std::set<void*> g_other;
int g_fail_in = -1;
std::function<size_t(const std::string&)> g_arg_bytes = [](const std::string&) { return (size_t)0; };
std::function<double(const Launch&)> g_cost = [](const Launch&) { return 0.01; };

namespace {

// Filled before main by the objects' registration.
std::map<const void*, std::string>& names()
{
    static std::map<const void*, std::string> n;
    return n;
}
char* g_next = reinterpret_cast<char*>(0x7000000000ull);
std::vector<Work>* g_capture = nullptr;
double g_clock = 0.0;   // ms

bool failing() { return g_fail_in >= 0 && g_fail_in-- == 0; }

void add(Work w)
{
    if (g_capture) {
        g_capture->push_back(w);
        return;
    }
    if (w.kind == Work::kLaunch) g_clock += g_cost(w.launch);
    g_work.push_back(std::move(w));
}

void add_launch(const void* f, dim3 grid, dim3 block, void** args, cudaStream_t s, bool overlapped)
{
    Work w{Work::kLaunch};
    w.stream = s;
    w.launch.name = names().count(f) ? names()[f] : "?";
    w.launch.grid = grid;
    w.launch.block = block;
    w.launch.overlapped = overlapped;
    w.launch.arg.resize(g_arg_bytes(w.launch.name));
    if (!w.launch.arg.empty()) std::memcpy(w.launch.arg.data(), args[0], w.launch.arg.size());
    add(w);
}

struct Event {
    double time = 0.0;
};

}  // namespace

struct CUgraph_st {
    std::vector<Work> work;
};
struct CUgraphExec_st {
    std::vector<Work> work;
};

extern "C" {

void** __cudaRegisterFatBinary(void*)
{
    static void* h;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*)
{
    names()[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, struct CUstream_st*) { std::abort(); }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { std::abort(); }
cudaError_t __cudaGetKernel(cudaKernel_t*, const void*) { std::abort(); }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t) { std::abort(); }

cudaError_t cudaGetDevice(int* d)
{
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "injected"; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int)
{
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrL2CacheSize ? 129 << 20 : 0;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t)
{
    *n = 3;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*)
{
    *p = reinterpret_cast<void*>(0x6000000000ull);
    return cudaSuccess;
}
static CUresult address_range(CUdeviceptr* base, size_t* size, CUdeviceptr p)
{
    auto it = g_device.upper_bound(reinterpret_cast<char*>(p));
    if (it == g_device.begin()) return CUDA_ERROR_NOT_FOUND;
    --it;
    if (reinterpret_cast<char*>(p) >= it->first + it->second) return CUDA_ERROR_NOT_FOUND;
    *base = reinterpret_cast<CUdeviceptr>(it->first);
    *size = it->second;
    return CUDA_SUCCESS;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* found)
{
    const bool known = std::strcmp(name, "cuMemGetAddressRange") == 0;
    *f = known ? reinterpret_cast<void*>(address_range) : nullptr;
    if (found) *found = known ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p)
{
    std::memset(a, 0, sizeof(*a));
    char* c = static_cast<char*>(const_cast<void*>(p));
    auto it = g_device.upper_bound(c);
    if (it == g_device.begin()) return cudaErrorInvalidValue;
    --it;
    a->type = c < it->first + it->second ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
    return cudaSuccess;
}

cudaError_t cudaMalloc(void** p, size_t n)
{
    if (failing()) return cudaErrorMemoryAllocation;
    g_next += (n + 0xffffull) & ~0xffffull;
    *p = g_next;
    g_device[g_next] = n;
    g_next += (n + 0x1ffffull) & ~0xffffull;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p)
{
    if (p && !g_device.erase(static_cast<char*>(p))) std::printf("free of unknown memory\n");
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned)
{
    if (failing()) return cudaErrorMemoryAllocation;
    *p = std::calloc(n, 1);
    g_other.insert(*p);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p)
{
    if (!g_other.erase(p)) std::printf("free of unknown host memory\n");
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int, size_t, cudaStream_t s)
{
    if (failing()) return cudaErrorUnknown;
    Work w{Work::kMemset};
    w.stream = s;
    w.at = p;
    add(w);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void*, size_t n, cudaMemcpyKind k, cudaStream_t s)
{
    if (k == cudaMemcpyDeviceToHost) std::memset(d, 0, n);
    Work w{Work::kCopy};
    w.stream = s;
    w.at = d;
    add(w);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* p, size_t n, cudaMemcpyKind k) { return cudaMemcpyAsync(d, p, n, k, nullptr); }

cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned)
{
    if (failing()) return cudaErrorMemoryAllocation;
    *s = reinterpret_cast<cudaStream_t>(new int(0));
    g_other.insert(*s);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s)
{
    if (!g_other.erase(s)) std::printf("unknown stream destroyed\n");
    return cudaSuccess;   // the address stays its own
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned)
{
    Work w{Work::kWait};
    w.stream = s;
    w.at = e;
    add(w);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned)
{
    if (failing()) return cudaErrorMemoryAllocation;
    *e = reinterpret_cast<cudaEvent_t>(new Event());
    g_other.insert(*e);
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e)
{
    if (!g_other.erase(e)) std::printf("unknown event destroyed\n");
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s)
{
    Work w{Work::kRecord};
    w.stream = s;
    w.at = e;
    add(w);
    reinterpret_cast<Event*>(e)->time = g_clock;
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b)
{
    *ms = (float)(reinterpret_cast<Event*>(b)->time - reinterpret_cast<Event*>(a)->time);
    return cudaSuccess;
}

cudaError_t cudaLaunchKernel(const void* f, dim3 g, dim3 b, void** args, size_t, cudaStream_t s)
{
    add_launch(f, g, b, args, s, false);
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args)
{
    bool overlapped = false;
    for (unsigned i = 0; i < c->numAttrs; ++i)
        overlapped |= c->attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization;
    add_launch(f, c->gridDim, c->blockDim, args, c->stream, overlapped);
    return cudaSuccess;
}

cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode)
{
    g_capture = new std::vector<Work>();
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g)
{
    *g = new CUgraph_st{*g_capture};
    delete g_capture;
    g_capture = nullptr;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t g, unsigned long long)
{
    *x = new CUgraphExec_st{g->work};
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g)
{
    delete g;
    return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x)
{
    delete x;
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t s)
{
    for (Work w : x->work) {
        w.stream = s;
        w.replayed = true;
        add(w);
    }
    return cudaSuccess;
}

}  // extern "C"
