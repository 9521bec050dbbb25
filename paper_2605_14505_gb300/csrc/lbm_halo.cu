// Halo pack and unpack of a z-slab: both buffers' slot planes in one launch.
//
// A buffer is one plane of every slot with e_z = +-1 (14 runs for D3Q27xD3Q19),
// so as one copy per run an exchange of two slabs is 112 copies a phase, bound
// by their launches (64 KB each at 128^2). 20 steps of a 128^3 FP32 lattice in
// two slabs: 9.34 ms with a copy per run and host waits between the slabs,
// 2.48 ms with these launches ordered by the slabs' streams (and the steps'
// own gains). Here grid.y is the run and grid.z the side; a run is a plain
// coalesced copy of the widest type that the alignment allows, four independent
// loads a thread before their stores.
#include <cuda_runtime.h>

#include "lbm_halo.cuh"

namespace lbm {

template <class V>
__global__ void __launch_bounds__(kHaloThreads) k_halo(const __grid_constant__ HaloArgs a)
{
    const HaloSide& s = a.side[blockIdx.z];
    V* store = reinterpret_cast<V*>(s.run[blockIdx.y]);
    V* buffer = reinterpret_cast<V*>(s.buffer + (size_t)blockIdx.y * a.plane);
    V* dst = a.pack ? buffer : store;
    const V* src = a.pack ? store : buffer;
    const size_t n = a.plane / sizeof(V);
    const size_t stride = (size_t)gridDim.x * kHaloThreads;
    size_t i = (size_t)blockIdx.x * kHaloThreads + threadIdx.x;
    for (; i + 3 * stride < n; i += 4 * stride) {
        const V v0 = src[i], v1 = src[i + stride], v2 = src[i + 2 * stride], v3 = src[i + 3 * stride];
        dst[i] = v0;
        dst[i + stride] = v1;
        dst[i + 2 * stride] = v2;
        dst[i + 3 * stride] = v3;
    }
    for (; i < n; i += stride) dst[i] = src[i];
}

const void* halo_kernel(int width)
{
    return width == 16  ? (const void*)k_halo<uint4>
           : width == 4 ? (const void*)k_halo<uint32_t>
           : width == 2 ? (const void*)k_halo<uint16_t>
                        : (const void*)k_halo<uint8_t>;
}

}  // namespace lbm
