// Programmatic dependent launch between the kernels of a time step.
//
// A launch_next() kernel may be placed on the SMs while the kernel before it
// in the stream drains: it sets up what needs no data and waits in
// pdl_wait() until that kernel has completed and its writes are visible. On
// short steps the launch latency between two dependent kernels is a good part
// of the step (boundary storage runs two kernels per forward and four per
// backward step). Every thread of such a kernel calls pdl_wait() before it
// touches what earlier kernels wrote, so a kernel's completion implies that of
// all kernels before it. (k_encode_march reads its weights before the wait, which
// the ordinary launch of the kernels of the scale allows: see ae_encode() in
// ae.cu.)
//
// A kernel that is placed early lives while kernels before it still write the
// fields: it may read those only through coherent loads (plain or at L2). The
// read-only path (__ldg, or a const __restrict__ pointer) asks for data that
// nobody writes while the kernel lives; it is for the coefficients, profiles,
// receiver and tap tables, observed data and stored snapshots of a call. Nor
// are fields __restrict__: a load through such a pointer may be moved above
// the wait.
#pragma once

#include <cuda_runtime.h>

namespace rtm {

__device__ __forceinline__ void pdl_wait() {
    // dependents may be placed from here on: they wait for this kernel anyway
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <class... Params, class... Args>
cudaError_t launch_dependent(bool early, void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem,
                             cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = early ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

// Blocks placed while others still hold their SMs are spread unevenly, which
// a grid of one or two plane-marching blocks per SM (those with dynamic shared
// memory) does not make up for: 104^3 in 182 blocks took 11.3 ms for a replayed
// 300-step shot each way against 8.4 placed afterwards, in 338 blocks 5.4
// against 5.6 (direct launches: 11.9 / 9.9 and 5.9 / 8.6)
template <class... Params, class... Args>
cudaError_t launch_next(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem,
                        cudaStream_t s, Args... args) {
    const bool early = smem == 0 || (long long)grid.x * grid.y * grid.z >= 2 * 152;
    return launch_dependent(early, kernel, grid, block, smem, s, args...);
}

}  // namespace rtm
