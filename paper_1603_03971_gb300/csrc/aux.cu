// Small kernels around the stencil: model preparation, sponge profiles, the
// Ricker wavelet, source injection / receiver gather, adjoint injection,
// image and gradient finalisation, and the data misfit.

#include <math.h>

#include <algorithm>

#include "band.cuh"
#include "cells.cuh"
#include "pdl.cuh"
#include "rtm_internal.h"

namespace rtm {

namespace {

constexpr int kStatusInvalid = 1;  // == RTM_ERR_INVALID

__device__ __forceinline__ void flag(int* status, int code) {
    if (status) atomicCAS(status, 0, code);
}

// padded linear index of model coordinates (x, y, z), or -1 if outside the
// padded grid
__device__ __forceinline__ long long rec_index(const Geometry& G, const int32_t* rec, int j) {
    const int x = rec[3 * j + 0] + G.nb, y = rec[3 * j + 1] + G.nb, z = rec[3 * j + 2] + G.nb;
    if (x < 0 || x >= G.NX || y < 0 || y >= G.NY || z < 0 || z >= G.NZ) return -1;
    return ((long long)z * G.NY + y) * G.NX + x;
}


// Cerjan-type profile: exp(-(0.015 (nb - d))^2) within nb cells of a face
__device__ __forceinline__ float sponge_1d(int i, int n, int nb) {
    const int d = min(i, n - 1 - i);
    if (d >= nb) return 1.0f;
    const double s = 0.015 * (double)(nb - d);
    return (float)exp(-s * s);
}

__global__ void k_sponge(Geometry G, float* gx, float* gy, float* gz) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < G.NX) gx[i] = sponge_1d(i, G.NX, G.nb);
    if (i < G.NY) gy[i] = sponge_1d(i, G.NY, G.nb);
    if (i < G.NZ) gz[i] = sponge_1d(i, G.NZ, G.nb);
}

// Ricker: w(t) = (1 - 2 pi^2 f0^2 (t - t0)^2) exp(-pi^2 f0^2 (t - t0)^2), in double
__global__ void k_wavelet(int nt, double dt, double f0, double t0, float* w) {
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= nt) return;
    const double pf = 3.14159265358979323846 * f0 * ((double)n * dt - t0);
    const double a = pf * pf;
    w[n] = (float)((1.0 - 2.0 * a) * exp(-a));
}

// *bits = max(*bits, v) for a non-negative v of every thread of a block of at
// most 1024. Floats of one sign compare as unsigned. Same-address atomics are served
// one by one (one per warp of 19456: most of the 56 us of a 10 M cell model),
// so a block sends one, and only if it would change the value
__device__ __forceinline__ void block_max(float v, unsigned int* bits) {
    __shared__ float part[32];
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        v = threadIdx.x < blockDim.x >> 5 ? part[threadIdx.x] : 0.0f;
        for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
        if (threadIdx.x == 0 && __float_as_uint(v) > *reinterpret_cast<volatile unsigned int*>(bits))
            atomicMax(bits, __float_as_uint(v));
    }
}

// c = v^2 dt^2 on the padded grid (edge padding); max v^2 and validity over
// the model cells
__global__ void k_model_prep(Geometry G, const float* __restrict__ vel, int squared, float dt2,
                             float* __restrict__ c, unsigned int* vmax_bits, int* bad) {
    float local_max = 0.0f;
    int local_bad = 0;
    for_cells(G.NX, G.NY, G.NZ, [&](int x, int y, int z) {
        const int mx = min(max(x - G.nb, 0), G.nx - 1);
        const int my = min(max(y - G.nb, 0), G.ny - 1);
        const int mz = min(max(z - G.nb, 0), G.nz - 1);
        const float v = vel[((long long)mz * G.ny + my) * G.nx + mx];
        const float v2 = squared ? v : v * v;
        c[((long long)z * G.NY + y) * G.NX + x] = v2 * dt2;
        const bool interior = (x - G.nb == mx) && (y - G.nb == my) && (z - G.nb == mz);
        if (interior) {
            if (!(isfinite(v) && v > 0.0f)) local_bad = 1;
            else local_max = fmaxf(local_max, v2);
        }
    });
    if (local_bad) atomicOr(bad, 1);
    block_max(local_max, vmax_bits);
}

// the boundary band of the model region, gathered from a padded field or
// scattered into it by blocks first, first + 1, ... of a launch
__device__ __forceinline__ void copy_band(const Geometry& G, const BandCopy& B, long long n, int first) {
    const long long stride = (long long)(gridDim.x - first) * blockDim.x;
    for (long long b = (long long)(blockIdx.x - first) * blockDim.x + threadIdx.x; b < n; b += stride) {
        int mx, my, mz;
        if (n < (1LL << 31))
            band_cell_as<unsigned>((unsigned)b, G.nx, G.ny, G.nz, B.r, mx, my, mz);
        else
            band_cell(b, G.nx, G.ny, G.nz, B.r, mx, my, mz);
        const long long i =
            ((long long)(mz + G.nb) * G.NY + (my + G.nb)) * G.NX + (mx + G.nb);
        if (B.to_field)
            B.field[i] = B.band[b];
        else
            B.band[b] = B.field[i];
    }
}
__global__ void k_band_copy(Geometry G, BandCopy B, long long n) {
    pdl_wait();
    copy_band(G, B, n, 0);
}

__global__ void k_fwd_aux(Geometry G, const float* u_cur, float* u_prev,
                          const float* __restrict__ c, const float* gx, const float* gy,
                          const float* gz, const int32_t* __restrict__ rec, int nrec,
                          float* data_row, long long src, const float* w_n, float inv_dx3,
                          int* status, BandCopy B, long long nband) {
    pdl_wait();
    const int first = nrec / (int)blockDim.x + 1;  // blocks of the points
    if ((int)blockIdx.x >= first) return copy_band(G, B, nband, first);
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < nrec) {
        if (data_row) {
            const long long i = rec_index(G, rec, j);
            if (i < 0) flag(status, kStatusInvalid);
            data_row[j] = i >= 0 ? u_cur[i] : 0.0f;
        }
    } else if (j == nrec && w_n) {
        // the stencil computes g(...) - g^2 u_prev: lowering u_prev[s] by
        // c_s w / (dx^3 g_s^2) adds c_s w / dx^3 to u^{n+1}[s]
        const float g = sponge_at(G, gx, gy, gz, src);
        u_prev[src] -= c[src] * (*w_n) * inv_dx3 / (g * g);
    }
}

__global__ void k_bwd_aux(Geometry G, const float* mu_cur, float* mu_prev,
                          const float* __restrict__ c, const float* gx, const float* gy,
                          const float* gz, const int32_t* __restrict__ rec, int nrec,
                          const float* __restrict__ r_row, long long src, float* src_adj_slot,
                          float* grad_acc, const float* w_n, float inv_dx3, int* status,
                          BandCopy B, long long nband) {
    pdl_wait();
    const int first = nrec / (int)blockDim.x + 1;  // blocks of the points
    if ((int)blockIdx.x >= first) return copy_band(G, B, nband, first);
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < nrec) {
        if (r_row) {
            const long long i = rec_index(G, rec, j);
            if (i < 0) {
                flag(status, kStatusInvalid);
            } else {
                // lowering mu_prev[i] by c r / (dx^3 g) adds c g r / dx^3 to mu^m[i]
                const float g = sponge_at(G, gx, gy, gz, i);
                atomicAdd(&mu_prev[i], -c[i] * r_row[j] * inv_dx3 / g);
            }
        }
    } else if (j == nrec) {
        const float g = sponge_at(G, gx, gy, gz, src);
        const float m = mu_cur[src];
        if (src_adj_slot) *src_adj_slot = m / g;
        if (grad_acc && w_n) grad_acc[src] += m * (*w_n) * inv_dx3 / g;
    }
}

__global__ void k_image_finalize(Geometry G, const float* __restrict__ slab,
                                 float* __restrict__ image) {
    for_cells(G.nx, G.ny, G.nz, [&](int x, int y, int z) {
        const long long zy = (long long)z * G.ny + y;
        image[zy * G.nx + x] += slab[zy * G.NX + x + G.nb];
    });
}

// source illumination: illum[z][y][x] += u^2 of the model columns of a
// snapshot slab [nz][ny][NX]; 16-byte vectors along x when both rows allow
// first element of model row zy = z ny + y: in the slab, or in a padded field
__device__ __forceinline__ long long model_row(const Geometry& G, long long zy, int padded) {
    if (!padded) return zy * G.NX + G.nb;
    const long long z = zy / G.ny;
    return ((z + G.nb) * G.NY + (zy - z * G.ny) + G.nb) * G.NX + G.nb;
}

__global__ void k_illum_add(Geometry G, const float* slab, float* illum, int vec, int padded) {
    pdl_wait();
    const long long stride = (long long)gridDim.x * blockDim.x;
    if (vec) {
        const int nx4 = G.nx >> 2;
        const long long n4 = (long long)nx4 * G.ny * G.nz;
        for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
            const long long zy = i / nx4;
            const int x4 = (int)(i - zy * nx4);
            const float4 u =
                __ldcs(reinterpret_cast<const float4*>(slab + model_row(G, zy, padded)) + x4);
            float4* d = reinterpret_cast<float4*>(illum + zy * G.nx) + x4;
            float4 a = *d;
            a.x = fmaf(u.x, u.x, a.x);
            a.y = fmaf(u.y, u.y, a.y);
            a.z = fmaf(u.z, u.z, a.z);
            a.w = fmaf(u.w, u.w, a.w);
            *d = a;
        }
        return;
    }
    const long long n = (long long)G.nx * G.ny * G.nz;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const long long zy = i / G.nx;
        const int x = (int)(i % G.nx);
        const float u = slab[model_row(G, zy, padded) + x];
        illum[i] = fmaf(u, u, illum[i]);
    }
}

// largest value of a non-negative array (float bits compare as unsigned)
__global__ void k_max_nonneg(const float* __restrict__ a, long long n, unsigned int* bits) {
    float m = 0.f;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        m = fmaxf(m, a[i]);
    block_max(m, bits);
}

// out = image / (illum + eps_rel * max illum)
__global__ void k_image_normalize(const float* __restrict__ image, const float* __restrict__ illum,
                                  long long n, const unsigned int* max_bits, float eps_rel,
                                  float* __restrict__ out) {
    const float floor_ = eps_rel * __uint_as_float(*max_bits);
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        out[i] = image[i] / (illum[i] + floor_);
}

// out = -L image on the model grid, zero outside it; a[0] = 3 a0 / dx^2,
// a[k] = a_k / dx^2
__global__ void k_image_laplacian(const float* __restrict__ image, int nx, int ny, int nz,
                                  LapWeights w, float* __restrict__ out) {
    const long long sy = nx, sz = (long long)nx * ny;
    for_cells(nx, ny, nz, [&](int x, int y, int z) {
        const long long i = z * sz + y * sy + x;
        float acc = w.a[0] * image[i];
        for (int k = 1; k <= w.r; k++) {
            float s = 0.f;
            if (x + k < nx) s += image[i + k];
            if (x - k >= 0) s += image[i - k];
            if (y + k < ny) s += image[i + k * sy];
            if (y - k >= 0) s += image[i - k * sy];
            if (z + k < nz) s += image[i + k * sz];
            if (z - k >= 0) s += image[i - k * sz];
            acc = fmaf(w.a[k], s, acc);
        }
        out[i] = -acc;
    });
}

__device__ __forceinline__ void fold_range(int m, int n, int nb, int N, int& lo, int& hi) {
    lo = (m == 0) ? 0 : m + nb;
    hi = (m == n - 1) ? N - 1 : m + nb;
}

// grad_v2[model cell] = dt^2 * sum over the padded cells copied from that
// cell of dx^3 acc / c (the transpose of the edge padding), in float64. An inner
// cell has one padded cell, a face cell nb + 1, an edge cell (nb + 1)^2, a corner
// cell (nb + 1)^3 (2 nb + 1 along a side of a single model cell): one thread per
// model cell left the eight corner threads with 36 000 dependent sums at nb = 32
// (57 ms of a 75 ms gradient at 256^3). So a cell's padded cells decide who sums
// them: a thread (inner cells; z and y faces, where neighbouring threads read
// neighbouring columns), a warp (x faces, whose padded cells are a row, and
// edges) or a block (corners). The padded copies of a cell have its coefficient:
// their values are summed and divided once. Bound by the float64 units, which
// have about two lanes per SM and clock: 0.35 ms for the inner cells, 0.24 for
// the faces and edges, 0.03 for the corners at 256^3, nb = 32 (memory: 0.05).
// Sums and quotients as pairs of floats took 0.27 ms in all, but keep at most 48
// bits and a float's range
struct FoldBox {
    int x0, x1, y0, y1, z0, z1;
};
__device__ __forceinline__ FoldBox fold_box(const Geometry& G, int x, int y, int z) {
    FoldBox b;
    fold_range(x, G.nx, G.nb, G.NX, b.x0, b.x1);
    fold_range(y, G.ny, G.nb, G.NY, b.y0, b.y1);
    fold_range(z, G.nz, G.nb, G.NZ, b.z0, b.z1);
    return b;
}
enum FoldOwner { FOLD_CELL, FOLD_COLUMN, FOLD_WARP, FOLD_BLOCK };
__device__ __forceinline__ FoldOwner fold_owner(const FoldBox& b) {
    const bool x = b.x1 > b.x0, y = b.y1 > b.y0, z = b.z1 > b.z0;
    if (x && y && z) return FOLD_BLOCK;
    if (x || (y && z)) return FOLD_WARP;
    return y || z ? FOLD_COLUMN : FOLD_CELL;
}

// a / c in float64 by Newton's iteration: the float reciprocal, one step (48
// bits), and the quotient corrected by its remainder, so rounded once more. Half
// the float64 instructions of the operator: inner cells 0.78 -> 0.35 ms at 256^3
__device__ __forceinline__ double quotient(double a, float c) {
    if (!(c > 1e-30f && c < 1e30f)) return a / (double)c;
    const double d = c, x0 = 1.0f / c, x = fma(x0, fma(-d, x0, 1.0), x0), q = a * x;
    const bool finite = (__double2hiint(q) & 0x7ff00000) != 0x7ff00000;
    return finite ? fma(fma(-d, q, a), x, q) : q;
}
// sum of acc / c over padded cells whose coefficients are mostly c0
struct FoldSum {
    float c0;
    bool shared;          // c0 may divide a sum: 0 / 0 and x / 0 would differ
    double a = 0.0;       // values over c0
    double ratios = 0.0;  // quotients by other coefficients
    __device__ explicit FoldSum(float c) : c0(c), shared(c > 0.f && c < INFINITY) {}
    __device__ __forceinline__ void add(float v, float c) {
        if (shared && c == c0)
            a += (double)v;
        else
            ratios += quotient(v, c);
    }
    __device__ __forceinline__ double value() const {
        return shared ? quotient(a, c0) + ratios : ratios;
    }
};
__device__ __forceinline__ double warp_sum(double s) {
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}
struct FoldScale {
    double dx3, dt2;
};
__device__ __forceinline__ float fold_scaled(double s, const FoldScale& k) {
    return (float)(s * k.dx3 * k.dt2);
}

// inner cells, a row per block and pass
__global__ void k_grad_finalize(Geometry G, const float* __restrict__ acc,
                                const float* __restrict__ c, FoldScale scale,
                                float* __restrict__ grad) {
    const unsigned rows = (unsigned)G.ny * (unsigned)G.nz;
    for (unsigned row = blockIdx.x; row < rows; row += gridDim.x) {
        const int z = (int)(row / (unsigned)G.ny), y = (int)(row - (unsigned)z * G.ny);
        const long long p = ((long long)(z + G.nb) * G.NY + (y + G.nb)) * G.NX + G.nb;
        float* out = grad + (long long)row * G.nx;
        const bool yz_inner = fold_owner(fold_box(G, 1 < G.nx - 1 ? 1 : 0, y, z)) == FOLD_CELL;
        for (int x = threadIdx.x; x < G.nx; x += blockDim.x) {
            if (G.nb > 0 && (!yz_inner || x == 0 || x == G.nx - 1)) continue;
            out[x] = fold_scaled(quotient(__ldcs(acc + p + x), __ldcs(c + p + x)), scale);
        }
    }
}

// this thread's part of a box's sum: cells t, t + n, .. of `cells`, x fastest
template <class I>
__device__ __forceinline__ double fold_part(const Geometry& G, const FoldBox& b,
                                            const float* __restrict__ acc,
                                            const float* __restrict__ c, int t, int n, I cells) {
    const unsigned bx = b.x1 - b.x0 + 1, by = b.y1 - b.y0 + 1;
    auto at = [&](I k) {
        const I zy = k / bx, zz = zy / by;
        return ((long long)(b.z0 + zz) * G.NY + (b.y0 + (long long)(zy - zz * by))) * G.NX +
               (b.x0 + (long long)(k - zy * bx));
    };
    FoldSum s(c[at(0)]);
#pragma unroll 4
    for (I k = t; k < cells; k += n) {
        const long long p = at(k);
        s.add(acc[p], c[p]);
    }
    return s.value();
}
// a box's sum over `n` threads, thread `t` of them (a side of a single model
// cell is all in one box, so the counts may need 64 bits)
__device__ __forceinline__ double fold_sum(const Geometry& G, const FoldBox& b,
                                           const float* __restrict__ acc,
                                           const float* __restrict__ c, int t, int n) {
    const long long cells =
        (long long)(b.x1 - b.x0 + 1) * (b.y1 - b.y0 + 1) * (b.z1 - b.z0 + 1);
    return cells < (1LL << 31) ? fold_part<unsigned>(G, b, acc, c, t, n, (unsigned)cells)
                               : fold_part<unsigned long long>(G, b, acc, c, t, n, cells);
}

// a row of y- or z-face cells, a column of padded cells per thread
__device__ void fold_columns(const Geometry& G, int y, int z, const float* __restrict__ acc,
                             const float* __restrict__ c, const FoldScale& scale,
                             float* __restrict__ grad) {
    for (int x = threadIdx.x; x < G.nx; x += blockDim.x) {
        const FoldBox b = fold_box(G, x, y, z);
        if (fold_owner(b) != FOLD_COLUMN) continue;
        const bool along_y = b.y1 > b.y0;
        const int n = along_y ? b.y1 - b.y0 + 1 : b.z1 - b.z0 + 1;
        const long long step = along_y ? G.NX : (long long)G.NX * G.NY;
        long long p = ((long long)b.z0 * G.NY + b.y0) * G.NX + b.x0;
        FoldSum s(c[p]);
#pragma unroll 8
        for (int k = 0; k < n; k++, p += step) s.add(__ldcs(acc + p), __ldcs(c + p));
        grad[((long long)z * G.ny + y) * G.nx + x] = fold_scaled(s.value(), scale);
    }
}

__device__ void fold_warp(const Geometry& G, int x, int y, int z, const float* __restrict__ acc,
                          const float* __restrict__ c, const FoldScale& scale,
                          float* __restrict__ grad) {
    const FoldBox b = fold_box(G, x, y, z);
    if (fold_owner(b) != FOLD_WARP) return;  // the same for the whole warp
    const int lane = threadIdx.x & 31;
    const double s = warp_sum(fold_sum(G, b, acc, c, lane, 32));
    if (lane == 0) grad[((long long)z * G.ny + y) * G.nx + x] = fold_scaled(s, scale);
}

// the face and edge cells. blockIdx.y: 0 and 1 the x faces (a warp per cell),
// 2 and 3 the z faces, 4 and 5 the y faces (a row of cells per block), 6 the
// four edges along x (a warp per cell)
__global__ void k_grad_finalize_faces(Geometry G, const float* __restrict__ acc,
                                      const float* __restrict__ c, FoldScale scale,
                                      float* __restrict__ grad) {
    const int what = blockIdx.y, far_side = what & 1;
    const unsigned warp = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const unsigned nwarps = gridDim.x * (blockDim.x >> 5);
    if (what < 2) {
        if (far_side && G.nx == 1) return;
        const unsigned cells = (unsigned)G.ny * (unsigned)G.nz;
        for (unsigned f = warp; f < cells; f += nwarps) {
            const int z = (int)(f / (unsigned)G.ny), y = (int)(f - (unsigned)z * G.ny);
            fold_warp(G, far_side ? G.nx - 1 : 0, y, z, acc, c, scale, grad);
        }
    } else if (what < 4) {
        if (far_side && G.nz == 1) return;
        for (int y = blockIdx.x; y < G.ny; y += gridDim.x)
            fold_columns(G, y, far_side ? G.nz - 1 : 0, acc, c, scale, grad);
    } else if (what < 6) {
        if (far_side && G.ny == 1) return;
        for (int z = blockIdx.x; z < G.nz; z += gridDim.x)
            fold_columns(G, far_side ? G.ny - 1 : 0, z, acc, c, scale, grad);
    } else {
        for (unsigned f = warp; f < 4u * (unsigned)G.nx; f += nwarps) {
            const int e = (int)(f / (unsigned)G.nx), x = (int)(f - (unsigned)e * G.nx);
            if (x == 0 || x == G.nx - 1) continue;  // in the x faces
            if (((e & 1) && G.ny == 1) || ((e & 2) && G.nz == 1)) continue;
            fold_warp(G, x, e & 1 ? G.ny - 1 : 0, e & 2 ? G.nz - 1 : 0, acc, c, scale, grad);
        }
    }
}

// the corner cells, one per block
__global__ void __launch_bounds__(1024) k_grad_finalize_corners(Geometry G,
                                                                const float* __restrict__ acc,
                                                                const float* __restrict__ c,
                                                                FoldScale scale,
                                                                float* __restrict__ grad) {
    __shared__ double part[32];
    const int e = blockIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (((e & 1) && G.nx == 1) || ((e & 2) && G.ny == 1) || ((e & 4) && G.nz == 1)) return;
    const int x = e & 1 ? G.nx - 1 : 0, y = e & 2 ? G.ny - 1 : 0, z = e & 4 ? G.nz - 1 : 0;
    const FoldBox b = fold_box(G, x, y, z);
    double s = warp_sum(fold_sum(G, b, acc, c, threadIdx.x, blockDim.x));
    if (lane == 0) part[wid] = s;
    __syncthreads();
    if (wid == 0) {
        s = warp_sum(part[lane]);
        if (lane == 0) grad[((long long)z * G.ny + y) * G.nx + x] = fold_scaled(s, scale);
    }
}

__global__ void k_misfit(const float* __restrict__ d, const float* __restrict__ obs, long long n,
                         float* resid, double* J) {
    double local = 0.0;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const float r = d[i] - obs[i];
        if (resid) resid[i] = r;
        local += 0.5 * (double)r * (double)r;
    }
    for (int o = 16; o > 0; o >>= 1) local += __shfl_xor_sync(0xffffffffu, local, o);
    __shared__ double warp_sum[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) warp_sum[wid] = local;
    __syncthreads();
    if (wid == 0) {
        double v = lane < (int)(blockDim.x >> 5) ? warp_sum[lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) atomicAdd(J, v);
    }
}

// any non-finite value among n floats sets the status word to
// RTM_ERR_NUMERIC (6); 16-byte loads when the base is aligned
__global__ void k_finite_scan(const float* __restrict__ f, long long n, int vec, int* status) {
    bool bad = false;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (vec) {
        const long long n4 = n / 4;
        const float4* f4 = reinterpret_cast<const float4*>(f);
        for (long long i = t; i < n4; i += stride) {
            const float4 v = __ldcs(f4 + i);
            bad |= !isfinite(v.x) || !isfinite(v.y) || !isfinite(v.z) || !isfinite(v.w);
        }
        for (long long i = 4 * n4 + t; i < n; i += stride) bad |= !isfinite(f[i]);
    } else {
        for (long long i = t; i < n; i += stride) bad |= !isfinite(__ldcs(f + i));
    }
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) flag(status, 6);
}

// decimated storage, coding: keep every other sample of the model region
// on each axis, coarse[kz][ky][kx] = u[nb + 2 kz][nb + 2 ky][nb + 2 kx] of a
// padded field; coarse sides are (n + 1) / 2. A block walks coarse rows
// (ky, kz), its threads along x
__global__ void k_decimate(Geometry G, const float* u, float* coarse, int cx, int cy, int cz) {
    pdl_wait();
    for (int row = blockIdx.x; row < cy * cz; row += gridDim.x) {
        const int ky = row % cy, kz = row / cy;
        const float* src = u + ((long long)(G.nb + 2 * kz) * G.NY + (G.nb + 2 * ky)) * G.NX + G.nb;
        float* dst = coarse + (long long)row * cx;
        for (int kx = threadIdx.x; kx < cx; kx += blockDim.x) dst[kx] = __ldcs(src + 2 * kx);
    }
}

// per axis: fine sample j from coarse samples i0 and i0 + 1 with weight w1 on
// the second: an even sample is a kept one; an odd sample is the mean of its
// two neighbours, or a copy of the left one past the last kept sample
__device__ __forceinline__ void lin_axis(int j, int nc, int& i0, float& w1) {
    i0 = j >> 1;
    w1 = ((j & 1) && i0 + 1 < nc) ? 0.5f : 0.0f;
}

// decimated storage, decoding: linear interpolation along each axis back to
// the model region of a snapshot slab [nz][ny][NX] (columns nb .. nb + nx);
// the weights (1, 1/2) are exact. One warp per output row (y, z): each lane
// interpolates one kept column along y and z from the four coarse rows
// (coalesced loads), takes its right neighbour's value by a shuffle, and
// writes the even output sample (the kept column) and the odd one (the mean
// of the two, or a copy past the last kept column)
__global__ void k_upsample(Geometry G, const float* __restrict__ coarse, int cx, int cy, int cz,
                           float* slab) {
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    // rows start 16-byte aligned (NX % 4 == 0): output pairs are 8-byte
    // aligned when the model's first column is even
    const bool pairs = (G.nb % 2) == 0;
    for (long long row = warp; row < (long long)G.ny * G.nz; row += nwarps) {
        const int y = (int)(row % G.ny), z = (int)(row / G.ny);
        int y0, z0;
        float wy, wz;
        lin_axis(y, cy, y0, wy);
        lin_axis(z, cz, z0, wz);
        const int y1 = wy > 0.f ? y0 + 1 : y0, z1 = wz > 0.f ? z0 + 1 : z0;
        const float* r00 = coarse + ((long long)z0 * cy + y0) * cx;
        const float* r01 = coarse + ((long long)z0 * cy + y1) * cx;
        const float* r10 = coarse + ((long long)z1 * cy + y0) * cx;
        const float* r11 = coarse + ((long long)z1 * cy + y1) * cx;
        float* out = slab + row * G.NX + G.nb;
        auto kept = [&](int k) {  // kept column k interpolated along y, then z
            const float a0 = (1.f - wy) * __ldg(r00 + k) + wy * __ldg(r01 + k);
            const float a1 = (1.f - wy) * __ldg(r10 + k) + wy * __ldg(r11 + k);
            return (1.f - wz) * a0 + wz * a1;
        };
        // four groups of 32 kept columns at a time: their loads are in flight together
        constexpr int U = 4;
        for (int base = 0; base < cx; base += 32 * U) {
            float bk[U + 1];
#pragma unroll
            for (int u = 0; u < U; u++) {
                const int k = base + 32 * u + lane;
                bk[u] = k < cx ? kept(k) : 0.f;
            }
            const int kl = base + 32 * U;  // the column after the last group, for lane 31
            bk[U] = (lane == 31 && kl < cx) ? kept(kl) : 0.f;
#pragma unroll
            for (int u = 0; u < U; u++) {
                const int k = base + 32 * u + lane;
                // the next kept column: lane + 1's, or for lane 31 the next
                // group's first (lane 0), or the extra column after the last group
                const float right = __shfl_down_sync(0xffffffffu, bk[u], 1);
                const float head = __shfl_sync(0xffffffffu, u + 1 < U ? bk[u + 1] : 0.f, 0);
                const float bn = lane < 31 ? right : (u + 1 < U ? head : bk[U]);
                if (k < cx) {
                    const float odd = k + 1 < cx ? 0.5f * bk[u] + 0.5f * bn : bk[u];
                    if (pairs && 2 * k + 1 < G.nx) {  // whole lines per warp
                        __stcs(reinterpret_cast<float2*>(out + 2 * k), make_float2(bk[u], odd));
                    } else {
                        __stcs(out + 2 * k, bk[u]);
                        if (2 * k + 1 < G.nx) __stcs(out + 2 * k + 1, odd);
                    }
                }
            }
        }
    }
}

int grid_for(long long n, int block) {
    long long g = (n + block - 1) / block;
    if (g > 152 * 16) g = 152 * 16;
    if (g < 1) g = 1;
    return (int)g;
}

}  // namespace

cudaError_t launch_sponge(const Geometry& G, float* gx, float* gy, float* gz, cudaStream_t s) {
    const int n = max(G.NX, max(G.NY, G.NZ));
    k_sponge<<<(n + 255) / 256, 256, 0, s>>>(G, gx, gy, gz);
    return cudaGetLastError();
}

cudaError_t launch_wavelet(int nt, double dt, double f0, double t0, float* w, cudaStream_t s) {
    k_wavelet<<<(nt + 255) / 256, 256, 0, s>>>(nt, dt, f0, t0, w);
    return cudaGetLastError();
}

cudaError_t launch_model_prep(const Geometry& G, const float* vel, int squared, double dt,
                              float* c, unsigned int* vmax_bits, int* bad, cudaStream_t s) {
    const long long N = (long long)G.NX * G.NY * G.NZ;
    k_model_prep<<<grid_for(N, 256), 256, 0, s>>>(G, vel, squared, (float)(dt * dt), c,
                                                  vmax_bits, bad);
    return cudaGetLastError();
}

// Boundary storage copies the band beside the points: as a launch of its own
// (3-5 us at 150 x 131 x 117) it stood between two dependent kernels of every step
cudaError_t launch_fwd_aux(const Geometry& G, const float* u_cur, float* u_prev, const float* c,
                           const float* gx, const float* gy, const float* gz,
                           const int32_t* rec, int nrec, float* data_row, long long src,
                           const float* w_n, float inv_dx3, int* status, cudaStream_t s,
                           const BandCopy& band) {
    const long long nb = band.band ? band_cells(G.nx, G.ny, G.nz, band.r) : 0;
    return launch_next(k_fwd_aux, nrec / 256 + 1 + (nb ? grid_for(nb, 256) : 0), 256, 0, s, G, u_cur,
                       u_prev, c, gx, gy, gz, rec, nrec, data_row, src, w_n, inv_dx3, status, band, nb);
}

cudaError_t launch_bwd_aux(const Geometry& G, const float* mu_cur, float* mu_prev,
                           const float* c, const float* gx, const float* gy, const float* gz,
                           const int32_t* rec, int nrec, const float* r_row, long long src,
                           float* src_adj_slot, float* grad_acc, const float* w_n,
                           float inv_dx3, int* status, cudaStream_t s, const BandCopy& band) {
    const long long nb = band.band ? band_cells(G.nx, G.ny, G.nz, band.r) : 0;
    return launch_next(k_bwd_aux, nrec / 256 + 1 + (nb ? grid_for(nb, 256) : 0), 256, 0, s, G, mu_cur,
                       mu_prev, c, gx, gy, gz, rec, nrec, r_row, src, src_adj_slot, grad_acc, w_n,
                       inv_dx3, status, band, nb);
}

cudaError_t launch_image_finalize(const Geometry& G, const float* slab, float* image,
                                  cudaStream_t s) {
    const long long n = (long long)G.nx * G.ny * G.nz;
    k_image_finalize<<<grid_for(n, 256), 256, 0, s>>>(G, slab, image);
    return cudaGetLastError();
}

cudaError_t launch_band_copy(const Geometry& G, const BandCopy& band, cudaStream_t s) {
    const long long n = band_cells(G.nx, G.ny, G.nz, band.r);
    return launch_next(k_band_copy, grid_for(n, 256), 256, 0, s, G, band, n);
}

cudaError_t launch_illum_add(const Geometry& G, const float* slab, float* illum, int padded,
                             cudaStream_t s) {
    const long long n = (long long)G.nx * G.ny * G.nz;
    // slab and padded rows start 16-byte aligned (NX % 4 == 0); the model
    // columns do when nb % 4 == 0, the illumination rows when nx % 4 == 0
    const int vec = (G.nb % 4 == 0) && (G.nx % 4 == 0) &&
                    (reinterpret_cast<uintptr_t>(illum) % 16 == 0) &&
                    (reinterpret_cast<uintptr_t>(slab) % 16 == 0);
    return launch_next(k_illum_add, grid_for(vec ? n / 4 : n, 256), 256, 0, s, G, slab, illum, vec,
                       padded);
}

cudaError_t launch_image_normalize(const float* image, const float* illum, long long n,
                                   unsigned int* max_bits, float eps_rel, float* out,
                                   cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(max_bits, 0, sizeof(unsigned int), s);
    if (e != cudaSuccess) return e;
    k_max_nonneg<<<grid_for(n, 256), 256, 0, s>>>(illum, n, max_bits);
    k_image_normalize<<<grid_for(n, 256), 256, 0, s>>>(image, illum, n, max_bits, eps_rel, out);
    return cudaGetLastError();
}

cudaError_t launch_image_laplacian(const float* image, int nx, int ny, int nz,
                                   const LapWeights& w, float* out, cudaStream_t s) {
    const long long n = (long long)nx * ny * nz;
    k_image_laplacian<<<grid_for(n, 256), 256, 0, s>>>(image, nx, ny, nz, w, out);
    return cudaGetLastError();
}

cudaError_t launch_grad_finalize(const Geometry& G, const float* acc, const float* c,
                                 double dx3, double dt2, float* grad_v2, cudaStream_t s) {
    const FoldScale scale{dx3, dt2};
    const long long rows = (long long)G.ny * G.nz;
    k_grad_finalize<<<grid_for(rows, 1), 256, 0, s>>>(G, acc, c, scale, grad_v2);
    if (G.nb > 0) {
        const dim3 grid(grid_for(std::max(rows / 8, (long long)std::max(G.ny, G.nz)), 1), 7);
        k_grad_finalize_faces<<<grid, 256, 0, s>>>(G, acc, c, scale, grad_v2);
        k_grad_finalize_corners<<<8, 1024, 0, s>>>(G, acc, c, scale, grad_v2);
    }
    return cudaGetLastError();
}

cudaError_t launch_finite_scan(const float* f, long long n, int* status, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int vec = reinterpret_cast<uintptr_t>(f) % 16 == 0;
    k_finite_scan<<<grid_for(vec ? n / 4 + 1 : n, 256), 256, 0, s>>>(f, n, vec, status);
    return cudaGetLastError();
}

// rows of a row-walking kernel: 16 resident blocks per SM on 152 SMs at most
static int row_blocks(long long rows) { return (int)(rows < 152 * 16 ? rows : 152 * 16); }

cudaError_t launch_decimate(const Geometry& G, const float* u, float* coarse, cudaStream_t s) {
    const int cx = (G.nx + 1) / 2, cy = (G.ny + 1) / 2, cz = (G.nz + 1) / 2;
    const int tb = cx > 128 ? 256 : 128;
    return launch_next(k_decimate, row_blocks((long long)cy * cz), tb, 0, s, G, u, coarse, cx, cy, cz);
}

cudaError_t launch_upsample(const Geometry& G, const float* coarse, float* slab, cudaStream_t s) {
    const int cx = (G.nx + 1) / 2, cy = (G.ny + 1) / 2, cz = (G.nz + 1) / 2;
    // a warp per row: 256-thread blocks, eight resident per SM
    const long long rows = (long long)G.ny * G.nz;
    const int blocks = (int)std::min<long long>((rows + 7) / 8, 152 * 8);
    return launch_next(k_upsample, blocks, 256, 0, s, G, coarse, cx, cy, cz, slab);
}

cudaError_t launch_misfit(const float* d, const float* obs, long long n, float* resid, double* J,
                          cudaStream_t s) {
    k_misfit<<<grid_for(n, 256), 256, 0, s>>>(d, obs, n, resid, J);
    return cudaGetLastError();
}

}  // namespace rtm
