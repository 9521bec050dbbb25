// Arguments of the halo copy kernel (lbm_halo.cu).
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace lbm {

constexpr int kHaloMaxRuns = 18;   // slots with e_z = +1 (or -1) of the largest pair, D3Q27xD3Q27
constexpr int kHaloThreads = 256;

// A halo buffer is a list of runs, one plane of one slot each, contiguous both
// in the store and in the buffer: run k is the `plane` bytes at run[k] in the
// store and at k * plane in the buffer.
struct HaloSide {
    char* run[kHaloMaxRuns];
    char* buffer;
};
struct HaloArgs {
    HaloSide side[2];
    size_t plane;   // bytes of a run
    int pack;       // store -> buffer, else buffer -> store
};

// Kernel that copies `width` bytes (16, 4, 2 or 1) per thread and iteration;
// every run, the buffers and `plane` are multiples of width.
const void* halo_kernel(int width);

}  // namespace lbm
