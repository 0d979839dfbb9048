// Training layers of the snapshot codec whose operands are plain 16-byte
// gathers: forward E2 and D1, their data gradients, and every weight and bias
// gradient.
//
// One 128-thread CTA computes a 128 x N tile on the tensor cores, as in
// tc_gemm.cuh, with nothing in its slab loop that waits for global memory:
//  - Weights are packed once per step into the shared-memory image of each
//    slab's B operand (k_pack_weights), so B is a contiguous cp.async. Reading
//    the float32 parameters in every slab (for D1's gradient 512 of them 4 KB
//    apart) stalled each of the 64 slabs of a tile.
//  - The weight gradients contract over voxels, and activations are stored
//    [voxel][channel]: both operands are MN-major for that product, so a
//    voxel's channels are copied as they lie and the transposition is the
//    instruction descriptor's. Writing the transposed slab element by element
//    took 32-48 two-byte stores per thread and slab.
//  - E2's data gradient runs one launch row per output parity: a parity reaches
//    1, 2, 4 or 8 of the 27 taps, the tile of all parities gathered all 27.
//  - The rank-8 gradients of the patch convolutions and their biases are one
//    product: rows [ga1 | g1 | ga3], columns [x patch | gy patch | 1].
// Every accumulator still sums its taps in the order of the general engine.
//
// us per 192^3 sample, before -> now: E2 99 -> 68, D1 109 -> 73, D1's data
// gradient 219 -> 145, E2's 175 -> 64, weight gradients of E2 241 -> 68,
// of D1 218 -> 82, of E1 and D2 with the biases 387 -> 118. A sample's
// activations are 57 MB each: 8 us per pass over one at the HBM copy rate.

#include <cuda_bf16.h>
#include <stdint.h>

#include <algorithm>

#include "ae_internal.h"
#include "ae_train.h"
#include "tc_gemm.cuh"

namespace rtm {
namespace ae {

namespace {

struct Pos {
    int x, y, z, ok;
};
// voxel v of an nx x ny x nz grid (below 2^31 voxels: the codec's volumes have
// at most 2^34)
__device__ __forceinline__ Pos position_of(unsigned v, const Dims3& d) {
    Pos p;
    const unsigned total = (unsigned)d.nx * (unsigned)d.ny * (unsigned)d.nz;
    const unsigned t = v / (unsigned)d.nx;
    p.x = (int)(v - t * (unsigned)d.nx);
    p.z = (int)(t / (unsigned)d.ny);
    p.y = (int)(t - (unsigned)p.z * (unsigned)d.ny);
    p.ok = v < total;
    return p;
}
__device__ __forceinline__ bool inside(int x, int y, int z, const Dims3& d) {
    return x >= 0 && x < d.nx && y >= 0 && y < d.ny && z >= 0 && z < d.nz;
}
__device__ __forceinline__ long long at(int x, int y, int z, const Dims3& d) {
    return ((long long)z * d.ny + y) * d.nx + x;
}

__device__ __forceinline__ void copy16(uint8_t* dst, const void* src, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(tc::smem_u32(dst)), "l"(src),
                 "r"(valid ? 16 : 0)
                 : "memory");
}
// 16-byte chunk `g` of row r of a K-major slab (8 k values of one row)
__device__ __forceinline__ uint8_t* kmaj(uint8_t* slab, int r, int g) {
    return slab + (r >> 3) * 512 + g * 128 + (r & 7) * 16;
}
// 16-byte chunk `g` (8 rows) at k of an MN-major slab: the same core matrices
// with rows and k exchanged
__device__ __forceinline__ uint8_t* mnmaj(uint8_t* slab, int g, int k) {
    return slab + g * 512 + (k >> 3) * 128 + (k & 7) * 16;
}
// a packed B slab of n rows
__device__ __forceinline__ void copy_packed(uint8_t* sB, const uint4* slab, int n, int tid) {
    if (tid < 4 * n) copy16(sB + 16 * tid, slab + tid, true);
}

// transposed conv (kernel 4, stride 2, padding 1): parity q, tap index tau
// -> input offset t and kernel index k
__device__ __forceinline__ void convt(int q, int tau, int& t, int& k) {
    if (q == 0) {
        t = tau ? -1 : 0;
        k = tau ? 3 : 1;
    } else {
        t = tau ? 0 : 1;
        k = tau ? 2 : 0;
    }
}

__device__ __forceinline__ void store_row(bf16* dst, const float* f, int n) {
    for (int j = 0; j < n; j += 8) *reinterpret_cast<uint4*>(dst + j) = tc::pack8(f + j);
}
// f *= LeakyReLU'(activation) of 32 channels
__device__ __forceinline__ void mask_row(const bf16* act, float* f) {
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const uint4 u = reinterpret_cast<const uint4*>(act)[j];
        const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const float2 t = __bfloat1622float2(h[e]);
            f[8 * j + 2 * e] *= t.x > 0.f ? 1.0f : kSlope;
            f[8 * j + 2 * e + 1] *= t.y > 0.f ? 1.0f : kSlope;
        }
    }
}
__device__ __forceinline__ float leaky_relu(float a) { return a > 0.f ? a : kSlope * a; }

// ---- packed weights: slab images, in 16-byte chunks -------------------------
constexpr int kE2Slab = 64, kD1Slab = 128, kD1dSlab = 64, kE2dSlab = 128;  // chunks per slab
constexpr int kE2At = 0;                         // 27 taps
constexpr int kD1At = kE2At + 27 * kE2Slab;      // 8 parities x 4 slabs of two taps
constexpr int kD1dAt = kD1At + 32 * kD1Slab;     // 64 taps
constexpr int kE2dAt = kD1dAt + 64 * kD1dSlab;   // 14 slabs of two taps over 8 parities
constexpr int kPackedChunks = kE2dAt + 14 * kE2dSlab;
static_assert(kPackedChunks * 16 == kAePackedBytes, "packed weights");

// E2's data gradient at output parity q (bits z, y, x; 1: odd): an even
// coordinate is reached by kernel index 1, an odd one by 0 (from the next
// latent voxel) and 2
__device__ __forceinline__ int e2d_taps(int q) { return 1 << __popc(q); }
__device__ __forceinline__ int e2d_first_slab(int q) {  // slabs of the parities before q
    constexpr int before[8] = {0, 1, 2, 3, 5, 6, 8, 10};
    return before[q];
}
// tap i of parity q: kernel indices and latent offsets per axis
__device__ __forceinline__ void e2d_tap(int q, int i, int& kz, int& ky, int& kx, int& dz, int& dy,
                                        int& dx) {
    int bit = __popc(q);
    auto axis = [&](int odd, int& k, int& d) {
        if (!odd) {
            k = 1;
            d = 0;
            return;
        }
        const int b = (i >> --bit) & 1;
        k = b ? 2 : 0;
        d = b ? 0 : 1;
    };
    axis((q >> 2) & 1, kz, dz);
    axis((q >> 1) & 1, ky, dy);
    axis(q & 1, kx, dx);
}

__global__ void k_pack_weights(const float* __restrict__ P, uint4* __restrict__ out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= kPackedChunks) return;
    // chunk c of a slab: row n and k0 .. k0 + 7 of a K-major image
    auto place = [](int i, int& n, int& k0) {
        n = (i >> 5) * 8 + (i & 7);
        k0 = ((i >> 3) & 3) * 8;
    };
    float w[8];
    int n, k0;
    if (c < kD1At) {
        const int tap = c / kE2Slab;
        place(c % kE2Slab, n, k0);
        for (int e = 0; e < 8; e++) w[e] = P[kOW2 + n * 864 + tap * 32 + k0 + e];
    } else if (c < kD1dAt) {
        const int slab = (c - kD1At) / kD1Slab, q = slab >> 2;
        place((c - kD1At) % kD1Slab, n, k0);
        const int tau = 2 * (slab & 3) + (k0 >> 4);
        int t, kz, ky, kx;
        convt(q >> 2, tau >> 2, t, kz);
        convt((q >> 1) & 1, (tau >> 1) & 1, t, ky);
        convt(q & 1, tau & 1, t, kx);
        for (int e = 0; e < 8; e++)
            w[e] = P[kOW3 + n * 1024 + ((kz * 4 + ky) * 4 + kx) * 16 + (k0 & 15) + e];
    } else if (c < kE2dAt) {
        const int tap = (c - kD1dAt) / kD1dSlab;
        place((c - kD1dAt) % kD1dSlab, n, k0);
        for (int e = 0; e < 8; e++) w[e] = P[kOW3 + (k0 + e) * 1024 + tap * 16 + n];
    } else {
        const int slab = (c - kE2dAt) / kE2dSlab;
        place((c - kE2dAt) % kE2dSlab, n, k0);
        int q = 7;
        while (e2d_first_slab(q) > slab) q--;
        const int i = 2 * (slab - e2d_first_slab(q)) + (k0 >> 4);
        int kz, ky, kx, dz, dy, dx;
        e2d_tap(q, i, kz, ky, kx, dz, dy, dx);
        for (int e = 0; e < 8; e++)
            w[e] = i < e2d_taps(q)
                       ? P[kOW2 + ((k0 & 15) + e) * 864 + ((kz * 3 + ky) * 3 + kx) * 32 + n]
                       : 0.f;
    }
    out[c] = tc::pack8(w);
}

// ---- layers -------------------------------------------------------------------
struct LayerArgs {
    const bf16* in;    // gathered activation or gradient
    const bf16* act;   // activation whose LeakyReLU' masks the output, or NULL
    bf16* out;
    const uint4* W;    // packed weights
    const float* P;
    Dims3 h, l;        // half- and quarter-resolution grids
};

struct TE2 {  // h1 -> latent
    using Args = LayerArgs;
    static constexpr int N = 16;
    static constexpr bool kMN = false;
    __device__ static void range(const Args&, int& c0, int& c1) {
        c0 = 0;
        c1 = 27;
    }
    __device__ static Pos position(const Args& a, int tid) {
        return position_of(blockIdx.x * 128u + tid, a.l);
    }
    __device__ static void load(const Args& a, const Pos& p, int tap, uint8_t* sA, uint8_t* sB,
                                int tid) {
        const int kz = tap / 9, ky = (tap / 3) % 3, kx = tap % 3;
        const int x = 2 * p.x + kx - 1, y = 2 * p.y + ky - 1, z = 2 * p.z + kz - 1;
        const bool ok = p.ok && inside(x, y, z, a.h);
        const bf16* src = ok ? a.in + at(x, y, z, a.h) * 32 : a.in;
#pragma unroll
        for (int j = 0; j < 4; j++) copy16(kmaj(sA, tid, j), src + 8 * j, ok);
        copy_packed(sB, a.W + kE2At + tap * kE2Slab, N, tid);
    }
    __device__ static void epilogue(const Args& a, const Pos& p, int, const float* acc) {
        if (!p.ok) return;
        float f[16];
#pragma unroll
        for (int o = 0; o < 16; o++) f[o] = acc[o] + a.P[kOB2 + o];
        store_row(a.out + at(p.x, p.y, p.z, a.l) * 16, f, 16);
    }
};

struct TD1 {  // latent -> g1, output parity blockIdx.y
    using Args = LayerArgs;
    static constexpr int N = 32;
    static constexpr bool kMN = false;
    __device__ static void range(const Args&, int& c0, int& c1) {
        c0 = 0;
        c1 = 4;
    }
    __device__ static Pos position(const Args& a, int tid) {
        return position_of(blockIdx.x * 128u + tid, a.l);
    }
    __device__ static void load(const Args& a, const Pos& p, int ch, uint8_t* sA, uint8_t* sB,
                                int tid) {
        const int q = blockIdx.y;
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int tau = 2 * ch + h;
            int tz, ty, tx, k;
            convt(q >> 2, tau >> 2, tz, k);
            convt((q >> 1) & 1, (tau >> 1) & 1, ty, k);
            convt(q & 1, tau & 1, tx, k);
            const int x = p.x + tx, y = p.y + ty, z = p.z + tz;
            const bool ok = p.ok && inside(x, y, z, a.l);
            const bf16* src = ok ? a.in + at(x, y, z, a.l) * 16 : a.in;
            copy16(kmaj(sA, tid, 2 * h), src, ok);
            copy16(kmaj(sA, tid, 2 * h + 1), src + 8, ok);
        }
        copy_packed(sB, a.W + kD1At + (4 * q + ch) * kD1Slab, N, tid);
    }
    __device__ static void epilogue(const Args& a, const Pos& p, int, const float* acc) {
        if (!p.ok) return;
        const int q = blockIdx.y;
        float f[32];
#pragma unroll
        for (int c = 0; c < 32; c++) f[c] = leaky_relu(acc[c] + a.P[kOB3 + c]);
        store_row(a.out + at(2 * p.x + (q & 1), 2 * p.y + ((q >> 1) & 1), 2 * p.z + (q >> 2), a.h) * 32,
                  f, 32);
    }
};

struct TD1d {  // ga3 -> glat: dlat[j] = sum_k W3[.,k,.]^T ga3[2j + k - 1]
    using Args = LayerArgs;
    static constexpr int N = 16;
    static constexpr bool kMN = false;
    __device__ static void range(const Args&, int& c0, int& c1) {
        c0 = 0;
        c1 = 64;
    }
    __device__ static Pos position(const Args& a, int tid) {
        return position_of(blockIdx.x * 128u + tid, a.l);
    }
    __device__ static void load(const Args& a, const Pos& p, int tap, uint8_t* sA, uint8_t* sB,
                                int tid) {
        const int x = 2 * p.x + (tap & 3) - 1, y = 2 * p.y + ((tap >> 2) & 3) - 1,
                  z = 2 * p.z + (tap >> 4) - 1;
        const bool ok = p.ok && inside(x, y, z, a.h);
        const bf16* src = ok ? a.in + at(x, y, z, a.h) * 32 : a.in;
#pragma unroll
        for (int j = 0; j < 4; j++) copy16(kmaj(sA, tid, j), src + 8 * j, ok);
        copy_packed(sB, a.W + kD1dAt + tap * kD1dSlab, N, tid);
    }
    __device__ static void epilogue(const Args& a, const Pos& p, int, const float* acc) {
        if (p.ok) store_row(a.out + at(p.x, p.y, p.z, a.l) * 16, acc, 16);
    }
};

struct TE2d {  // glat -> ga1 at output parity blockIdx.y: (sum of W2^T glat) * leaky'(a1)
    using Args = LayerArgs;
    static constexpr int N = 32;
    static constexpr bool kMN = false;
    __device__ static void range(const Args&, int& c0, int& c1) {
        c0 = 0;
        c1 = (e2d_taps(blockIdx.y) + 1) / 2;
    }
    __device__ static Pos position(const Args& a, int tid) {
        return position_of(blockIdx.x * 128u + tid, a.l);
    }
    __device__ static void load(const Args& a, const Pos& p, int ch, uint8_t* sA, uint8_t* sB,
                                int tid) {
        const int q = blockIdx.y;
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int i = 2 * ch + h;
            int kz, ky, kx, dz, dy, dx;
            e2d_tap(q, i, kz, ky, kx, dz, dy, dx);
            const int x = p.x + dx, y = p.y + dy, z = p.z + dz;
            const bool ok = p.ok && i < e2d_taps(q) && inside(x, y, z, a.l);
            const bf16* src = ok ? a.in + at(x, y, z, a.l) * 16 : a.in;
            copy16(kmaj(sA, tid, 2 * h), src, ok);
            copy16(kmaj(sA, tid, 2 * h + 1), src + 8, ok);
        }
        copy_packed(sB, a.W + kE2dAt + (e2d_first_slab(q) + ch) * kE2dSlab, N, tid);
    }
    __device__ static void epilogue(const Args& a, const Pos& p, int, const float* acc) {
        if (!p.ok) return;
        const int q = blockIdx.y;
        const long long v =
            at(2 * p.x + (q & 1), 2 * p.y + ((q >> 1) & 1), 2 * p.z + (q >> 2), a.h);
        float f[32];
#pragma unroll
        for (int c = 0; c < 32; c++) f[c] = acc[c];
        mask_row(a.act + v * 32, f);
        store_row(a.out + v * 32, f, 32);
    }
};

// ---- weight gradients: contractions over voxels, MN-major operands ------------
struct WeightArgs {
    const bf16 *a, *b;  // row and column operands
    const bf16 *c;      // (patch gradients) third row operand
    const bf16* gy;     // (patch gradients) output gradients, full resolution
    Vol in;             // (patch gradients) the snapshot
    const float* inv_sigma;
    float* grad;
    Dims3 h, l;
    int slabs, per_cta;  // slabs of 32 voxels, and how many a CTA takes
};
__device__ __forceinline__ void slab_range(const WeightArgs& a, int cta, int& c0, int& c1) {
    c0 = cta * a.per_cta;
    c1 = min(a.slabs, c0 + a.per_cta);
    if (c1 < c0) c1 = c0;
}

struct TE2w {  // dW2[o][tap][i] += sum_v glat[v][o] h1[2v + tap - 1][i]; blockIdx.x: four taps
    using Args = WeightArgs;
    static constexpr int N = 16;
    static constexpr bool kMN = true;
    __device__ static void range(const Args& a, int& c0, int& c1) { slab_range(a, blockIdx.y, c0, c1); }
    __device__ static Pos position(const Args&, int) { return Pos{0, 0, 0, 1}; }
    __device__ static void load(const Args& a, const Pos&, int ch, uint8_t* sA, uint8_t* sB, int tid) {
        const int vv = tid & 31, tt = tid >> 5, tap = blockIdx.x * 4 + tt;
        const Pos p = position_of(ch * 32u + vv, a.l);
        const int kz = tap / 9, ky = (tap / 3) % 3, kx = tap % 3;
        const int x = 2 * p.x + kx - 1, y = 2 * p.y + ky - 1, z = 2 * p.z + kz - 1;
        const bool ok = p.ok && tap < 27 && inside(x, y, z, a.h);
        const bf16* src = ok ? a.a + at(x, y, z, a.h) * 32 : a.a;
#pragma unroll
        for (int j = 0; j < 4; j++) copy16(mnmaj(sA, 4 * tt + j, vv), src + 8 * j, ok);
        if (tid < 64)  // columns: two chunks of 8 output channels
            copy16(mnmaj(sB, tt, vv), a.b + (p.ok ? at(p.x, p.y, p.z, a.l) * 16 + 8 * tt : 0), p.ok);
    }
    __device__ static void epilogue(const Args& a, const Pos&, int row, const float* acc) {
        const int r = blockIdx.x * 128 + row;  // tap * 32 + i
        if (r >= 27 * 32) return;
        for (int o = 0; o < 16; o++) atomicAdd(&a.grad[kOW2 + o * 864 + r], acc[o]);
    }
};

struct TD1w {  // dW3[o][k][i] += sum_j ga3[2j + q][o] lat[j + t][i], parity q = blockIdx.x
    using Args = WeightArgs;
    static constexpr int N = 32;
    static constexpr bool kMN = true;
    __device__ static void range(const Args& a, int& c0, int& c1) { slab_range(a, blockIdx.y, c0, c1); }
    __device__ static Pos position(const Args&, int) { return Pos{0, 0, 0, 1}; }
    __device__ static void load(const Args& a, const Pos&, int ch, uint8_t* sA, uint8_t* sB, int tid) {
        const int q = blockIdx.x, vv = tid & 31;
        const Pos p = position_of(ch * 32u + vv, a.l);
#pragma unroll
        for (int rep = 0; rep < 2; rep++) {
            const int tau = (tid >> 5) + 4 * rep;  // rows tau * 16 + i
            int tz, ty, tx, k;
            convt(q >> 2, tau >> 2, tz, k);
            convt((q >> 1) & 1, (tau >> 1) & 1, ty, k);
            convt(q & 1, tau & 1, tx, k);
            const int x = p.x + tx, y = p.y + ty, z = p.z + tz;
            const bool ok = p.ok && inside(x, y, z, a.l);
            const bf16* src = ok ? a.a + at(x, y, z, a.l) * 16 : a.a;
            copy16(mnmaj(sA, 2 * tau, vv), src, ok);
            copy16(mnmaj(sA, 2 * tau + 1, vv), src + 8, ok);
        }
        const int j = tid >> 5;  // columns: four chunks of 8 output channels
        const long long o =
            p.ok ? at(2 * p.x + (q & 1), 2 * p.y + ((q >> 1) & 1), 2 * p.z + (q >> 2), a.h) : 0;
        copy16(mnmaj(sB, j, vv), a.b + o * 32 + 8 * j, p.ok);
    }
    __device__ static void epilogue(const Args& a, const Pos&, int row, const float* acc) {
        const int q = blockIdx.x, tau = row >> 4, i = row & 15;
        int t, kz, ky, kx;
        convt(q >> 2, tau >> 2, t, kz);
        convt((q >> 1) & 1, (tau >> 1) & 1, t, ky);
        convt(q & 1, tau & 1, t, kx);
        const int ktap = (kz * 4 + ky) * 4 + kx;
        for (int o = 0; o < 32; o++) atomicAdd(&a.grad[kOW3 + o * 1024 + ktap * 16 + i], acc[o]);
    }
};

// dW1[c][d] += sum_v ga1[v][c] xq[2v + d], dW4[d][i] += sum_v gy[2v + d] g1[v][i],
// db1 += sum ga1, db3 += sum ga3: rows [ga1 | g1 | ga3 | -] of 32 channels,
// columns [xq patch | gy patch | 1 | -] of 8
struct TPatch {
    using Args = WeightArgs;
    static constexpr int N = 32;
    static constexpr bool kMN = true;
    __device__ static void range(const Args& a, int& c0, int& c1) { slab_range(a, blockIdx.x, c0, c1); }
    __device__ static Pos position(const Args&, int) { return Pos{0, 0, 0, 1}; }
    __device__ static void load(const Args& a, const Pos&, int ch, uint8_t* sA, uint8_t* sB, int tid) {
        const int vv = tid & 31, part = tid >> 5;
        const unsigned v = ch * 32u + vv;
        const Pos p = position_of(v, a.h);
        if (part < 3) {
            const bf16* src = (part == 0 ? a.a : part == 1 ? a.b : a.c) + (p.ok ? (long long)v * 32 : 0);
#pragma unroll
            for (int j = 0; j < 4; j++) copy16(mnmaj(sA, 4 * part + j, vv), src + 8 * j, p.ok);
        } else {
#pragma unroll
            for (int j = 0; j < 4; j++) copy16(mnmaj(sA, 12 + j, vv), a.a, false);  // zeros
        }
        uint4 w = make_uint4(0, 0, 0, 0);
        if (part == 0 && p.ok) {  // the voxel's patch of normalised inputs
            const float s = *a.inv_sigma;
            const float* src = a.in.p + 2LL * p.z * a.in.sz + 2LL * p.y * a.in.sy + 2 * p.x;
            float f[8];
#pragma unroll
            for (int d = 0; d < 8; d++)
                f[d] = src[(d >> 2) * a.in.sz + ((d >> 1) & 1) * a.in.sy + (d & 1)] * s;
            w = tc::pack8(f);
        } else if (part == 1 && p.ok) {  // its patch of output gradients: pairs along x
            const long long NX = 2 * a.h.nx, NY = 2 * a.h.ny;
            const bf16* src = a.gy + ((2LL * p.z) * NY + 2 * p.y) * NX + 2 * p.x;
            w.x = *reinterpret_cast<const uint32_t*>(src);
            w.y = *reinterpret_cast<const uint32_t*>(src + NX);
            w.z = *reinterpret_cast<const uint32_t*>(src + NY * NX);
            w.w = *reinterpret_cast<const uint32_t*>(src + NY * NX + NX);
        } else if (part == 2) {
            w.x = 0x3F80;  // bf16 1.0 in the first of the eight columns
        }
        *reinterpret_cast<uint4*>(mnmaj(sB, part, vv)) = w;
    }
    __device__ static void epilogue(const Args& a, const Pos&, int row, const float* acc) {
        const int c = row & 31, part = row >> 5;
        if (part == 0) {
            for (int d = 0; d < 8; d++) atomicAdd(&a.grad[kOW1 + c * 8 + d], acc[d]);
            atomicAdd(&a.grad[kOB1 + c], acc[16]);
        } else if (part == 1) {
            for (int d = 0; d < 8; d++) atomicAdd(&a.grad[kOW4 + d * 32 + c], acc[8 + d]);
        } else if (part == 2) {
            atomicAdd(&a.grad[kOB3 + c], acc[16]);
        }
    }
};

// ---- engine: the pipeline of k_tc_gemm_async ----------------------------------
constexpr int kS = 4, kAhead = 2;  // stages; slabs loaded ahead of the one multiplied

template <class Op>
__global__ void __launch_bounds__(128) k_tc_train(const __grid_constant__ typename Op::Args args,
                                                  int* status) {
    constexpr int N = Op::N;
    __shared__ __align__(1024) uint8_t smem[kS][tc::kStageBytes];
    __shared__ __align__(8) uint64_t bars[kS];
    __shared__ uint32_t tmem_slot;
    const int tid = threadIdx.x, warp = tid >> 5;
    int c0, c1;
    Op::range(args, c0, c1);
    const int nch = c1 - c0;
    const Pos pos = Op::position(args, tid);

    if (tid == 0) {
        for (int s = 0; s < kS; s++) tc::mbar_init(&bars[s], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tc::tmem_alloc(&tmem_slot, tc::kTmemCols);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = tmem_slot;
    // MN-major A and B: transpose bits 15 and 16
    constexpr uint32_t idesc = tc::idesc_bf16(tc::kRows, N) | (Op::kMN ? (3u << 15) : 0u);

    for (int c = 0; c < kAhead; c++) {
        if (c < nch) Op::load(args, pos, c0 + c, smem[c], smem[c] + tc::kABytes, tid);
        tc::cp_async_commit();
    }
    bool ok = true;
    int issued = 0;
    for (int i = 0; i < nch && ok; i++) {
        const int j = i + kAhead;
        if (j < nch) {
            // slab j takes the stage of slab j - kS, multiplied two iterations ago
            if (j >= kS) ok = tc::mbar_wait(&bars[j % kS], (uint32_t)(((j - kS) / kS) & 1));
            ok = __syncthreads_and(ok);
            if (!ok) break;
            Op::load(args, pos, c0 + j, smem[j % kS], smem[j % kS] + tc::kABytes, tid);
        }
        tc::cp_async_commit();
        tc::cp_async_wait<kAhead>();
        tc::fence_proxy_async();
        __syncthreads();
        if (tid == 0) {
            tc::tc_fence_after();
            const uint32_t a0 = tc::smem_u32(smem[i % kS]), b0 = a0 + tc::kABytes;
#pragma unroll
            for (int s = 0; s < tc::kBK / 16; s++)
                tc::mma_bf16(tmem, tc::sdesc(a0 + 256 * s, 128, 512),
                             tc::sdesc(b0 + 256 * s, 128, 512), idesc, (i > 0 || s > 0) ? 1u : 0u);
            tc::mma_commit(&bars[i % kS]);
        }
        issued = i + 1;
    }
    tc::cp_async_wait<0>();
    if (issued > 0) {
        const int last = issued - 1;
        const bool done = tc::mbar_wait(&bars[last % kS], (uint32_t)((last / kS) & 1));
        ok = ok && done;
    }
    ok = __syncthreads_and(ok);
    tc::tc_fence_after();
    if (ok && nch > 0) {
        float acc[N];
        const uint32_t t = tmem + ((uint32_t)(warp * 32) << 16);
        tc::tmem_ld16(t, acc);
        if constexpr (N == 32) tc::tmem_ld16(t + 16, acc + 16);
        Op::epilogue(args, pos, tid, acc);
    } else if (!ok && tid == 0 && status) {
        atomicCAS(status, 0, tc::kErrTimeout);
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, tc::kTmemCols);
}

// db2 += sum_v glat[v]
__global__ void k_latent_bias(const bf16* __restrict__ glat, long long nl, float* grad) {
    const int ch = threadIdx.x & 15;
    float s = 0.f;
    for (long long v = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 4; v < nl;
         v += ((long long)gridDim.x * blockDim.x) >> 4)
        s += __bfloat162float(glat[v * 16 + ch]);
    __shared__ float part[256];
    part[threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.x < 16) {
        for (int w = 1; w < 16; w++) s += part[16 * w + threadIdx.x];
        atomicAdd(&grad[kOB2 + threadIdx.x], s);
    }
}

template <class Op>
cudaError_t run(const typename Op::Args& a, dim3 grid, int* status, cudaStream_t s) {
    k_tc_train<Op><<<grid, 128, 0, s>>>(a, status);
    return cudaGetLastError();
}

unsigned tiles_of(const Dims3& d) { return (unsigned)(((long long)d.nx * d.ny * d.nz + 127) / 128); }

// slabs of a contraction over the voxels of d, split over about `ctas` CTAs
void split(WeightArgs& w, const Dims3& d, int ctas, unsigned& rows) {
    w.slabs = (int)(((long long)d.nx * d.ny * d.nz + 31) / 32);
    w.per_cta = std::max(8, (w.slabs + ctas - 1) / ctas);
    rows = (unsigned)((w.slabs + w.per_cta - 1) / w.per_cta);
}

}  // namespace

}  // namespace ae

using namespace ae;

cudaError_t ae_pack_weights(const float* P, void* packed, cudaStream_t s) {
    k_pack_weights<<<(kPackedChunks + 255) / 256, 256, 0, s>>>(P, reinterpret_cast<uint4*>(packed));
    return cudaGetLastError();
}

cudaError_t ae_train_e2(const float* P, const void* W, const bf16* h1, bf16* lat, Dims3 h, Dims3 l,
                        int* status, cudaStream_t s) {
    const LayerArgs a{h1, nullptr, lat, reinterpret_cast<const uint4*>(W), P, h, l};
    return run<TE2>(a, dim3(tiles_of(l)), status, s);
}
cudaError_t ae_train_d1(const float* P, const void* W, const bf16* lat, bf16* g1, Dims3 h, Dims3 l,
                        int* status, cudaStream_t s) {
    const LayerArgs a{lat, nullptr, g1, reinterpret_cast<const uint4*>(W), P, h, l};
    return run<TD1>(a, dim3(tiles_of(l), 8), status, s);
}
cudaError_t ae_train_d1_grad(const void* W, const bf16* ga3, bf16* glat, Dims3 h, Dims3 l, int* status,
                             cudaStream_t s) {
    const LayerArgs a{ga3, nullptr, glat, reinterpret_cast<const uint4*>(W), nullptr, h, l};
    return run<TD1d>(a, dim3(tiles_of(l)), status, s);
}
cudaError_t ae_train_e2_grad(const void* W, const bf16* glat, const bf16* h1, bf16* ga1, Dims3 h,
                             Dims3 l, int* status, cudaStream_t s) {
    const LayerArgs a{glat, h1, ga1, reinterpret_cast<const uint4*>(W), nullptr, h, l};
    return run<TE2d>(a, dim3(tiles_of(l), 8), status, s);
}

cudaError_t ae_train_d1_weights(const bf16* lat, const bf16* ga3, float* grad, Dims3 h, Dims3 l,
                                int* status, cudaStream_t s) {
    WeightArgs w{};
    w.a = lat;
    w.b = ga3;
    w.grad = grad;
    w.h = h;
    w.l = l;
    unsigned rows;
    split(w, l, 152, rows);
    return run<TD1w>(w, dim3(8, rows), status, s);
}
cudaError_t ae_train_e2_weights(const bf16* h1, const bf16* glat, float* grad, Dims3 h, Dims3 l,
                                int* status, cudaStream_t s) {
    WeightArgs w{};
    w.a = h1;
    w.b = glat;
    w.grad = grad;
    w.h = h;
    w.l = l;
    unsigned rows;
    split(w, l, 152, rows);
    cudaError_t e = run<TE2w>(w, dim3(7, rows), status, s);
    if (e != cudaSuccess) return e;
    const long long nl = (long long)l.nx * l.ny * l.nz;
    k_latent_bias<<<(unsigned)std::min<long long>((nl + 255) / 256, 152), 256, 0, s>>>(glat, nl, grad);
    return cudaGetLastError();
}
cudaError_t ae_train_patch_weights(const Vol& in, const float* inv_sigma, const bf16* ga1,
                                   const bf16* gy, const bf16* g1, const bf16* ga3, float* grad,
                                   Dims3 h, Dims3 l, int* status, cudaStream_t s) {
    WeightArgs w{};
    w.a = ga1;
    w.b = g1;
    w.c = ga3;
    w.gy = gy;
    w.in = in;
    w.inv_sigma = inv_sigma;
    w.grad = grad;
    w.h = h;
    w.l = l;
    unsigned rows;
    split(w, h, 152 * 5, rows);
    return run<TPatch>(w, dim3(rows), status, s);
}

}  // namespace rtm
