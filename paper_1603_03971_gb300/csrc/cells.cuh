// Walks over the cells of a grid by rows of x.
//
// Kernels that touch every cell once are bound by memory, but the x, y and z of
// a flat index are two or three 64-bit divisions, which took longer than the
// memory: 66 us for the image Laplacian of 192 x 170 x 149 cells. Here a row
// costs one 32-bit division, shared by its cells.
#pragma once

#include <cuda_runtime.h>

namespace rtm {

// f(x, y, z) for the cells of an nx x ny x nz grid, once each, over all
// threads of a 1-D grid of whole warps. A row takes 32 lanes, or fewer where it is
// shorter than a warp
template <class F>
__device__ __forceinline__ void for_cells(int nx, int ny, int nz, F&& f) {
    const int lanes = nx >= 32 ? 32 : nx >= 16 ? 16 : nx >= 8 ? 8 : 4;
    const long long rows = (long long)ny * nz;
    const long long step = (long long)gridDim.x * blockDim.x / lanes;
    const int x0 = threadIdx.x % lanes;
    for (long long r = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / lanes; r < rows; r += step) {
        int y, z;
        if (rows < (1LL << 31)) {
            z = (int)((unsigned)r / (unsigned)ny);
            y = (int)((unsigned)r - (unsigned)z * (unsigned)ny);
        } else {
            z = (int)(r / ny);
            y = (int)(r - (long long)z * ny);
        }
#pragma unroll 4
        for (int x = x0; x < nx; x += lanes) f(x, y, z);
    }
}

}  // namespace rtm
