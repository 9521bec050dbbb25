// What tests/host_runtime.cpp, a stand-in for the CUDA runtime, records.
#pragma once

#include <cuda_runtime.h>

#include <functional>
#include <map>
#include <set>
#include <string>
#include <vector>

struct Launch {
    std::string name;
    dim3 grid, block;
    bool overlapped = false;
    std::vector<char> arg;   // the first kernel argument, where args_of knows its size
    template <class T>
    const T& as() const
    {
        return *reinterpret_cast<const T*>(arg.data());
    }
    bool is(const char* kernel) const { return name.find(kernel) != std::string::npos; }
};
// One entry of a stream's (or a graph's) work.
struct Work {
    enum Kind { kLaunch, kRecord, kWait, kMemset, kCopy } kind;
    cudaStream_t stream = nullptr;
    Launch launch;
    void* at = nullptr;   // event, or destination
    bool replayed = false;   // by a graph
};

extern std::vector<Work> g_work;
extern std::map<char*, size_t> g_device;    // live device allocations
extern std::set<void*> g_other;             // live host allocations, streams, events
extern int g_fail_in;                       // the call that this many fallible ones precede fails; -1: none
extern std::function<size_t(const std::string&)> g_arg_bytes;   // size of a kernel's first argument, 0: not kept
extern std::function<double(const Launch&)> g_cost;             // ms
