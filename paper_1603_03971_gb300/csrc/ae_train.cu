// Training layers of the snapshot codec whose operands are plain 16-byte
// gathers: forward E2 and D1, their data gradients, and every weight and bias
// gradient.
//
// A CTA computes a 128 x N tile on the tensor cores: four warps copy operand
// slabs into a ring, a fifth multiplies (k_tc_train).
//  - Weights are packed once per step into the shared-memory image of each
//    slab's B operand (k_pack_weights), so B is a contiguous cp.async. Reading
//    the float32 parameters in every slab (for D1's gradient 512 of them 4 KB
//    apart) stalled each of the 64 slabs of a tile.
//  - Four lanes copy one 64-byte row of a gather, through L1: of the rows that
//    one tap reads, the next tap along x reads half again.
//  - The weight gradients contract over voxels, and activations are stored
//    [voxel][channel]: both operands are MN-major for that product, so a
//    voxel's channels are copied as they lie and the transposition is the
//    instruction descriptor's. Writing the transposed slab element by element
//    took 32-48 two-byte stores per thread and slab. Every CTA adds its sums
//    to the same few hundred gradients, about 60 ns per CTA, so there are few
//    (the patch gradients: 1456 CTAs 143 us, 304 CTAs 71 us).
//  - E2's data gradient runs one launch row per output parity: a parity reaches
//    1, 2, 4 or 8 of the 27 taps, the tile of all parities gathered all 27.
//  - The rank-8 gradients of the patch convolutions and their biases are one
//    product: rows [ga1 | g1 | ga3], columns [x patch | gy patch | 1].
// Every accumulator sums its taps in the order of the general engine.
//
// us per 192^3 sample, general engine -> one role for copies and products ->
// now: E2 99 -> 68 -> 48, D1 109 -> 73 -> 56, D1's data gradient 219 -> 145 ->
// 103, E2's 175 -> 64 -> 54, weight gradients of E2 241 -> 68 -> 56, of D1
// 218 -> 82 -> 47, of E1 and D2 with the biases 387 -> 118 -> 81. A sample's
// activations are 57 MB each: 8 us per pass over one at the HBM copy rate.
// What is left: a CTA's copies are issued slab by slab, about 0.8 us each with
// their index arithmetic (L2 is 12-20 % busy), and tiles of two to four slabs
// spend most of their time in start-up and epilogue.

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
__device__ __forceinline__ int at(int x, int y, int z, const Dims3& d) {
    return (z * d.ny + y) * d.nx + x;
}
// where the taps of a voxel lie in grid g: the index of the first (it may be
// outside) and, four bits per axis, which of the next offsets are inside
struct Tap0 {
    int lin;
    unsigned in;
};
__device__ __forceinline__ Tap0 tap0(const Pos& p, int scale, int org, const Dims3& g) {
    const int x = scale * p.x + org, y = scale * p.y + org, z = scale * p.z + org;
    auto axis = [](int c, int n) {
        unsigned b = 0;
#pragma unroll
        for (int k = 0; k < 4; k++) b |= (unsigned)((unsigned)(c + k) < (unsigned)n) << k;
        return b;
    };
    Tap0 t;
    t.lin = (int)(((unsigned)z * (unsigned)g.ny + (unsigned)y) * (unsigned)g.nx + (unsigned)x);
    t.in = p.ok ? axis(x, g.nx) | axis(y, g.ny) << 4 | axis(z, g.nz) << 8 : 0u;
    return t;
}
__device__ __forceinline__ bool tap_in(unsigned in, int kx, int ky, int kz) {
    return (in >> kx) & (in >> (4 + ky)) & (in >> (8 + kz)) & 1u;
}

// 16 bytes through L1 (gathered rows: the next taps of the tile read them again)
__device__ __forceinline__ void copy16(uint8_t* dst, const void* src, bool valid) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(tc::smem_u32(dst)), "l"(src),
                 "r"(valid ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void copy4(uint8_t* dst, const void* src, bool valid) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(tc::smem_u32(dst)), "l"(src),
                 "r"(valid ? 4 : 0)
                 : "memory");
}
// 16 bytes past L1 (read once)
__device__ __forceinline__ void stream16(uint8_t* dst, const void* src, bool valid) {
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
// Four lanes take the chunks of one row, so a warp's copy reads 8 rows of 64
// bytes (or 16 of 32) and not 16 bytes of each of 32 rows, which are 32 cache
// lines. A thread's rows: (tid >> 2) + 32 i
struct Rows {
    Tap0 t[4];
};
__device__ __forceinline__ Rows rows_of(const Dims3& l, int scale, int org, const Dims3& g, int tid) {
    Rows R;
#pragma unroll
    for (int i = 0; i < 4; i++)
        R.t[i] = tap0(position_of(blockIdx.x * 128u + (tid >> 2) + 32 * i, l), scale, org, g);
    return R;
}
// chunk tid & 3 of the thread's rows: 8 of the C channels, from e on, at tap
// (kx, ky, kz); zeros unless `on`
template <int C>
__device__ __forceinline__ void copy_rows(uint8_t* sA, const bf16* in, const Rows& R, const Dims3& g,
                                          int kx, int ky, int kz, bool on, int e, int tid) {
    const int off = at(kx, ky, kz, g);
    uint8_t* dst = kmaj(sA, tid >> 2, tid & 3);
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const bool ok = on && tap_in(R.t[i].in, kx, ky, kz);
        copy16(dst + 2048 * i, in + (ok ? (long long)(R.t[i].lin + off) * C + e : 0), ok);
    }
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
__device__ __forceinline__ void mask_row(const uint4* act, float* f) {
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(act + j);
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const float2 t = __bfloat1622float2(h[e]);
            f[8 * j + 2 * e] *= t.x > 0.f ? 1.0f : kSlope;
            f[8 * j + 2 * e + 1] *= t.y > 0.f ? 1.0f : kSlope;
        }
    }
}
// rows of 32 channels between a lane's registers and voxels v (negative: none)
// of its warp, four lanes per row on the memory side; buf: 2 KB of the warp
__device__ __forceinline__ uint4* row_chunk(uint8_t* buf, int r, int j) {
    return reinterpret_cast<uint4*>(buf + (r * 4 + (j ^ ((r >> 1) & 3))) * 16);
}
__device__ __forceinline__ void store_rows(uint8_t* buf, bf16* out, int v, const float* f) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < 4; j++) *row_chunk(buf, lane, j) = tc::pack8(f + 8 * j);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const int r = (lane >> 2) + 8 * i, vr = __shfl_sync(0xffffffffu, v, r);
        if (vr >= 0)
            *reinterpret_cast<uint4*>(out + (long long)vr * 32 + 8 * (lane & 3)) =
                *row_chunk(buf, r, lane & 3);
    }
}
__device__ __forceinline__ void load_rows(uint8_t* buf, const bf16* in, int v, uint4* u) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const int r = (lane >> 2) + 8 * i, vr = __shfl_sync(0xffffffffu, v, r);
        if (vr >= 0)
            *row_chunk(buf, r, lane & 3) =
                *reinterpret_cast<const uint4*>(in + (long long)vr * 32 + 8 * (lane & 3));
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 4; j++) u[j] = *row_chunk(buf, lane, j);
    __syncwarp();
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
    using Where = Rows;
    __device__ static void init(uint8_t*, int) {}
    static constexpr int kS = 6;
    static constexpr int N = 16;
    static constexpr bool kMN = false;
    static constexpr int kTurn = 1 << 30;  // one accumulator
    __device__ static void range(const Args&, int& c0, int& c1) {
        c0 = 0;
        c1 = 27;
    }
    __device__ static Where where(const Args& a, int tid) { return rows_of(a.l, 2, -1, a.h, tid); }
    __device__ static void load(const Args& a, const Where& R, int tap, uint8_t* sA, uint8_t* sB,
                                int tid) {
        copy_rows<32>(sA, a.in, R, a.h, tap % 3, (tap / 3) % 3, tap / 9, true, 8 * (tid & 3), tid);
        copy_packed(sB, a.W + kE2At + tap * kE2Slab, N, tid);
    }
    __device__ static void epilogue(const Args& a, int row, uint8_t*, const float* acc) {
        const Pos p = position_of(blockIdx.x * 128u + row, a.l);
        if (!p.ok) return;
        float f[16];
#pragma unroll
        for (int o = 0; o < 16; o++) f[o] = acc[o] + a.P[kOB2 + o];
        store_row(a.out + (long long)(blockIdx.x * 128u + row) * 16, f, 16);
    }
};

struct TD1 {  // latent -> g1, output parity blockIdx.y
    using Args = LayerArgs;
    using Where = Rows;
    __device__ static void init(uint8_t*, int) {}
    static constexpr int kS = 2;
    static constexpr int N = 32;
    static constexpr bool kMN = false;
    static constexpr int kTurn = 1 << 30;  // one accumulator
    __device__ static void range(const Args&, int& c0, int& c1) {
        c0 = 0;
        c1 = 4;
    }
    __device__ static Where where(const Args& a, int tid) { return rows_of(a.l, 1, -1, a.l, tid); }
    __device__ static void load(const Args& a, const Where& R, int ch, uint8_t* sA, uint8_t* sB,
                                int tid) {
        const int q = blockIdx.y, tau = 2 * ch + ((tid >> 1) & 1);
        int tz, ty, tx, k;
        convt(q >> 2, tau >> 2, tz, k);
        convt((q >> 1) & 1, (tau >> 1) & 1, ty, k);
        convt(q & 1, tau & 1, tx, k);
        copy_rows<16>(sA, a.in, R, a.l, tx + 1, ty + 1, tz + 1, true, 8 * (tid & 1), tid);
        copy_packed(sB, a.W + kD1At + (4 * q + ch) * kD1Slab, N, tid);
    }
    __device__ static void epilogue(const Args& a, int row, uint8_t* buf, const float* acc) {
        const Pos p = position_of(blockIdx.x * 128u + row, a.l);
        const int q = blockIdx.y;
        float f[32];
#pragma unroll
        for (int c = 0; c < 32; c++) f[c] = leaky_relu(acc[c] + a.P[kOB3 + c]);
        store_rows(buf, a.out,
                   p.ok ? at(2 * p.x + (q & 1), 2 * p.y + ((q >> 1) & 1), 2 * p.z + (q >> 2), a.h) : -1,
                   f);
    }
};

struct TD1d {  // ga3 -> glat: dlat[j] = sum_k W3[.,k,.]^T ga3[2j + k - 1]
    using Args = LayerArgs;
    using Where = Rows;
    __device__ static void init(uint8_t*, int) {}
    static constexpr int kS = 6;
    static constexpr int N = 16;
    static constexpr bool kMN = false;
    static constexpr int kTurn = 1 << 30;  // one accumulator
    __device__ static void range(const Args&, int& c0, int& c1) {
        c0 = 0;
        c1 = 64;
    }
    __device__ static Where where(const Args& a, int tid) { return rows_of(a.l, 2, -1, a.h, tid); }
    __device__ static void load(const Args& a, const Where& R, int tap, uint8_t* sA, uint8_t* sB,
                                int tid) {
        copy_rows<32>(sA, a.in, R, a.h, tap & 3, (tap >> 2) & 3, tap >> 4, true, 8 * (tid & 3), tid);
        copy_packed(sB, a.W + kD1dAt + tap * kD1dSlab, N, tid);
    }
    __device__ static void epilogue(const Args& a, int row, uint8_t*, const float* acc) {
        const Pos p = position_of(blockIdx.x * 128u + row, a.l);
        if (p.ok) store_row(a.out + (long long)(blockIdx.x * 128u + row) * 16, acc, 16);
    }
};

struct TE2d {  // glat -> ga1 at output parity blockIdx.y: (sum of W2^T glat) * leaky'(a1)
    using Args = LayerArgs;
    using Where = Rows;
    __device__ static void init(uint8_t*, int) {}
    static constexpr int kS = 2;
    static constexpr int N = 32;
    static constexpr bool kMN = false;
    static constexpr int kTurn = 1 << 30;  // one accumulator
    __device__ static void range(const Args&, int& c0, int& c1) {
        c0 = 0;
        c1 = (e2d_taps(blockIdx.y) + 1) / 2;
    }
    __device__ static Where where(const Args& a, int tid) { return rows_of(a.l, 1, 0, a.l, tid); }
    __device__ static void load(const Args& a, const Where& R, int ch, uint8_t* sA, uint8_t* sB,
                                int tid) {
        const int q = blockIdx.y, i = 2 * ch + ((tid >> 1) & 1);
        int kz, ky, kx, dz, dy, dx;
        e2d_tap(q, i, kz, ky, kx, dz, dy, dx);
        copy_rows<16>(sA, a.in, R, a.l, dx, dy, dz, i < e2d_taps(q), 8 * (tid & 1), tid);
        copy_packed(sB, a.W + kE2dAt + (e2d_first_slab(q) + ch) * kE2dSlab, N, tid);
    }
    __device__ static void epilogue(const Args& a, int row, uint8_t* buf, const float* acc) {
        const Pos p = position_of(blockIdx.x * 128u + row, a.l);
        const int q = blockIdx.y;
        const int v =
            p.ok ? at(2 * p.x + (q & 1), 2 * p.y + ((q >> 1) & 1), 2 * p.z + (q >> 2), a.h) : -1;
        uint4 act[4];
        load_rows(buf, a.act, v, act);
        float f[32];
#pragma unroll
        for (int c = 0; c < 32; c++) f[c] = acc[c];
        mask_row(act, f);
        store_rows(buf, a.out, v, f);
    }
};

// ---- weight gradients: contractions over voxels, MN-major operands ------------
struct WeightArgs {
    const bf16 *a, *b;  // row and column operands
    const bf16 *c;      // (patch gradients) third row operand
    const bf16* gy;     // (patch gradients) output gradients, full resolution
    const bf16* xq;     // (patch gradients) normalised inputs, 8 per voxel
    float* grad;
    Dims3 h, l;
    int slabs, per_cta;  // slabs of 32 voxels, and how many a CTA takes
};
__device__ __forceinline__ void slab_range(const WeightArgs& a, int cta, int& c0, int& c1) {
    c0 = cta * a.per_cta;
    c1 = min(a.slabs, c0 + a.per_cta);
    if (c1 < c0) c1 = c0;
}

// a warp's 32 voxels of a slab, one per lane, handed to the lanes that copy
// their chunks
struct NoRows {};
__device__ __forceinline__ Tap0 from_lane(const Tap0& t, int lane) {
    return Tap0{__shfl_sync(0xffffffffu, t.lin, lane), __shfl_sync(0xffffffffu, t.in, lane)};
}
__device__ __forceinline__ unsigned voxels(const Dims3& d) {
    return (unsigned)d.nx * (unsigned)d.ny * (unsigned)d.nz;
}

struct TE2w {  // dW2[o][tap][i] += sum_v glat[v][o] h1[2v + tap - 1][i]; blockIdx.x: four taps
    using Args = WeightArgs;
    using Where = NoRows;
    __device__ static void init(uint8_t*, int) {}
    static constexpr int kS = 6;
    static constexpr int N = 16;
    static constexpr bool kMN = true;
    static constexpr int kTurn = 4;
    __device__ static void range(const Args& a, int& c0, int& c1) { slab_range(a, blockIdx.y, c0, c1); }
    __device__ static Where where(const Args&, int) { return Where{}; }
    __device__ static void load(const Args& a, const Where&, int ch, uint8_t* sA, uint8_t* sB, int tid) {
        const int lane = tid & 31, tt = tid >> 5, tap = blockIdx.x * 4 + tt, j = lane & 3;
        const Tap0 t = tap0(position_of(ch * 32u + lane, a.l), 2, -1, a.h);
        const int kz = tap / 9, ky = (tap / 3) % 3, kx = tap % 3, off = at(kx, ky, kz, a.h);
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int vv = (lane >> 2) + 8 * i;
            const Tap0 u = from_lane(t, vv);
            const bool ok = tap < 27 && tap_in(u.in, kx, ky, kz);
            copy16(mnmaj(sA, 4 * tt + j, vv), a.a + (ok ? (long long)(u.lin + off) * 32 + 8 * j : 0), ok);
        }
        if (tid < 64) {  // columns: two chunks of 8 output channels
            const unsigned v = ch * 32u + (tid >> 1);
            const bool ok = v < voxels(a.l);
            copy16(mnmaj(sB, tid & 1, tid >> 1), a.b + (ok ? (long long)v * 16 + 8 * (tid & 1) : 0), ok);
        }
    }
    __device__ static void epilogue(const Args& a, int row, uint8_t*, const float* acc) {
        const int r = blockIdx.x * 128 + row;  // tap * 32 + i
        if (r >= 27 * 32) return;
        for (int o = 0; o < 16; o++) atomicAdd(&a.grad[kOW2 + o * 864 + r], acc[o]);
    }
};

struct TD1w {  // dW3[o][k][i] += sum_j ga3[2j + q][o] lat[j + t][i], parity q = blockIdx.x
    using Args = WeightArgs;
    using Where = NoRows;
    __device__ static void init(uint8_t*, int) {}
    static constexpr int kS = 6;
    static constexpr int N = 32;
    static constexpr bool kMN = true;
    static constexpr int kTurn = 4;
    __device__ static void range(const Args& a, int& c0, int& c1) { slab_range(a, blockIdx.y, c0, c1); }
    __device__ static Where where(const Args&, int) { return Where{}; }
    __device__ static void load(const Args& a, const Where&, int ch, uint8_t* sA, uint8_t* sB, int tid) {
        const int q = blockIdx.x, lane = tid & 31, warp = tid >> 5;
        const Pos p = position_of(ch * 32u + lane, a.l);
        const Tap0 t = tap0(p, 1, -1, a.l);
#pragma unroll
        for (int half = 0; half < 2; half++) {
            const int vv = (lane >> 1) + 16 * half;
            const Tap0 u = from_lane(t, vv);
#pragma unroll
            for (int rep = 0; rep < 2; rep++) {
                const int tau = warp + 4 * rep;  // rows tau * 16 + i
                int tz, ty, tx, k;
                convt(q >> 2, tau >> 2, tz, k);
                convt((q >> 1) & 1, (tau >> 1) & 1, ty, k);
                convt(q & 1, tau & 1, tx, k);
                const bool ok = tap_in(u.in, tx + 1, ty + 1, tz + 1);
                copy16(mnmaj(sA, 2 * tau + (lane & 1), vv),
                       a.a + (ok ? (long long)(u.lin + at(tx + 1, ty + 1, tz + 1, a.l)) * 16 +
                                       8 * (lane & 1)
                                 : 0),
                       ok);
            }
        }
        // columns: four chunks of 8 output channels, 8 voxels per warp
        const int v =
            p.ok ? at(2 * p.x + (q & 1), 2 * p.y + ((q >> 1) & 1), 2 * p.z + (q >> 2), a.h) : -1;
        const int vr = __shfl_sync(0xffffffffu, v, tid >> 2);
        copy16(mnmaj(sB, tid & 3, tid >> 2), a.b + (vr >= 0 ? (long long)vr * 32 + 8 * (tid & 3) : 0),
               vr >= 0);
    }
    __device__ static void epilogue(const Args& a, int row, uint8_t*, const float* acc) {
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
    using Where = NoRows;
    static constexpr int kS = 10;
    static constexpr int N = 32;
    static constexpr bool kMN = true;
    static constexpr int kTurn = 1;
    __device__ static void range(const Args& a, int& c0, int& c1) { slab_range(a, blockIdx.x, c0, c1); }
    __device__ static Where where(const Args&, int) { return Where{}; }
    __device__ static void load(const Args& a, const Where&, int ch, uint8_t* sA, uint8_t* sB, int tid) {
        const int lane = tid & 31, part = tid >> 5;
        const bf16* rows = part == 0 ? a.a : part == 1 ? a.b : a.c;
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int vv = (lane >> 2) + 8 * i, j = lane & 3;
            const unsigned v = ch * 32u + vv;
            const bool ok = part < 3 && v < voxels(a.h);  // (the fourth part: zeros)
            stream16(mnmaj(sA, 4 * part + j, vv), rows + (ok ? (long long)v * 32 + 8 * j : 0), ok);
        }
        const unsigned v = ch * 32u + lane;
        uint8_t* dst = mnmaj(sB, part, lane);
        if (part == 0) {  // the voxel's patch of normalised inputs
            const bool ok = v < voxels(a.h);
            stream16(dst, a.xq + (ok ? (long long)v * 8 : 0), ok);
        } else if (part == 1) {  // its patch of output gradients: pairs along x
            const Pos p = position_of(v, a.h);
            const long long NX = 2 * a.h.nx, NY = 2 * a.h.ny;
            const bf16* src = a.gy + (p.ok ? ((2LL * p.z) * NY + 2 * p.y) * NX + 2 * p.x : 0);
#pragma unroll
            for (int d = 0; d < 4; d++)
                copy4(dst + 4 * d, src + (p.ok ? (d >> 1) * NY * NX + (d & 1) * NX : 0), p.ok);
        }
    }
    // columns 16-23: bf16 1.0 in the first; 24-31: zeros
    __device__ static void init(uint8_t* sB, int tid) {
        if (tid >= 64)
            *reinterpret_cast<uint4*>(mnmaj(sB, tid >> 5, tid & 31)) =
                make_uint4((tid >> 5) == 2 ? 0x3F80u : 0u, 0u, 0u, 0u);
    }
    __device__ static void epilogue(const Args& a, int row, uint8_t*, const float* acc) {
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

// ---- engine -------------------------------------------------------------------
// Warps 0-3 copy slabs into a ring, each as soon as its stage is free, and
// leave the arrival at the slab's barrier to their copies; warp 4 waits for a
// slab, makes it visible to the tensor cores and multiplies. A proxy fence in
// the threads that copy would wait for all of their copies in flight, and with
// it every slab for the memory's full latency, however deep the ring.
// Op::kS: stages of 10 KB; two for the products of few slabs (six CTAs per SM),
// 6 to 10 for the long ones (104 against 127 us with two for D1's gradient).
//
// The weight gradients' contractions are as long as the volume, and the tensor
// cores truncate what they add to an accumulator: over the 180 steps of a CTA
// at 192^3 the gradients of W1, W4, b1 and b3 lost 4-8 times what float32 sums
// of the lanes had lost. So two accumulators take turns, Op::kTurn steps each, and
// warps 5-8 add the finished one to sums in registers, rounded to nearest,
// while the next is filled. Relative L2 error against float64 sums of the same
// operands, lanes / one accumulator / turns: W1 3.8e-7 / 3.0e-6 / 2.5e-7, W4
// 3.7e-7 / 2.3e-6 / 2.6e-7, W2 5.9e-7 / 1.3e-6 / 1.4e-7, W3 9.3e-7 / 2.9e-6 /
// 1.4e-7 at 192^3; at 64^3 W1 1.2e-7 / 5.4e-7 / 1.2e-7, W3 1.7e-7 / 5.8e-7 / 9e-8.
// The patch products, whose lanes had summed single voxels, take a turn per step
// (72 -> 81 us), the others four steps, which cost them 1-2 us
template <class Op>
constexpr int train_smem() {
    return Op::kS * tc::kStageBytes + 1024;
}
template <class Op>
constexpr int train_threads() {
    return Op::kMN ? 288 : 160;
}

template <class Op>
__global__ void __launch_bounds__(train_threads<Op>()) k_tc_train(
    const __grid_constant__ typename Op::Args args, int* status) {
    constexpr int N = Op::N, kS = Op::kS;
    constexpr int kCols = Op::kMN ? 2 * tc::kTmemCols : tc::kTmemCols;
    constexpr int kSteps = tc::kBK / 16, kTurn = Op::kTurn;
    extern __shared__ uint8_t raw[];
    uint8_t(*smem)[tc::kStageBytes] = reinterpret_cast<uint8_t(*)[tc::kStageBytes]>(
        (reinterpret_cast<uintptr_t>(raw) + 1023) & ~static_cast<uintptr_t>(1023));
    __shared__ __align__(8) uint64_t full[kS], empty[kS], done;
    __shared__ __align__(8) uint64_t acc_full[2], acc_free[2];  // kMN: an accumulator's turns
    __shared__ uint32_t tmem_slot;
    const int tid = threadIdx.x, warp = tid >> 5;
    int c0, c1;
    Op::range(args, c0, c1);
    const int nch = c1 - c0;

    if (tid == 0) {
        for (int s = 0; s < kS; s++) {
            tc::mbar_init(&full[s], 128);
            tc::mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; b++) {
            tc::mbar_init(&acc_full[b], 1);
            tc::mbar_init(&acc_free[b], 128);
        }
        tc::mbar_init(&done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tc::tmem_alloc(&tmem_slot, kCols);
    if (warp < 4) {
        for (int s = 0; s < kS; s++) Op::init(smem[s] + tc::kABytes, tid);
        tc::fence_proxy_async();
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = tmem_slot;

    bool ok = true;
    float sum[N];
#pragma unroll
    for (int n = 0; n < N; n++) sum[n] = 0.f;
    if (warp == 4) {
        if (tid == 128 && nch > 0) {
            // MN-major A and B: transpose bits 15 and 16
            constexpr uint32_t idesc = tc::idesc_bf16(tc::kRows, N) | (Op::kMN ? (3u << 15) : 0u);
            for (int i = 0; i < nch && ok; i++) {
                ok = tc::mbar_wait(&full[i % kS], (uint32_t)((i / kS) & 1));
                if (!ok) break;
                tc::fence_proxy_async();
                tc::tc_fence_after();
                const uint32_t a0 = tc::smem_u32(smem[i % kS]), b0 = a0 + tc::kABytes;
#pragma unroll
                for (int s = 0; s < kSteps; s++) {
                    const int step = kSteps * i + s, turn = step / kTurn, b = turn & 1;
                    const bool first = step % kTurn == 0;
                    if (first && turn >= 2) {
                        ok = tc::mbar_wait(&acc_free[b], (uint32_t)((turn / 2 - 1) & 1));
                        if (!ok) break;
                        tc::tc_fence_after();
                    }
                    tc::mma_bf16(tmem + b * tc::kTmemCols, tc::sdesc(a0 + 256 * s, 128, 512),
                                 tc::sdesc(b0 + 256 * s, 128, 512), idesc, first ? 0u : 1u);
                    if (Op::kMN && (step % kTurn == kTurn - 1 || step == kSteps * nch - 1))
                        tc::mma_commit(&acc_full[b]);
                }
                if (ok) tc::mma_commit(&empty[i % kS]);
            }
            tc::mma_commit(&done);
        }
        __syncwarp();
    } else if (warp < 4) {
        const typename Op::Where where = Op::where(args, tid);
        for (int j = 0; j < nch; j++) {
            if (j >= kS) ok = tc::mbar_wait(&empty[j % kS], (uint32_t)((j / kS - 1) & 1));
            if (!ok) break;
            Op::load(args, where, c0 + j, smem[j % kS], smem[j % kS] + tc::kABytes, tid);
            asm volatile("cp.async.mbarrier.arrive.noinc.shared.b64 [%0];" ::"r"(
                             tc::smem_u32(&full[j % kS]))
                         : "memory");
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else if constexpr (Op::kMN) {
        for (int turn = 0; turn * kTurn < kSteps * nch; turn++) {
            const int b = turn & 1;
            ok = tc::mbar_wait(&acc_full[b], (uint32_t)((turn / 2) & 1));
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc::tc_fence_after();
            float acc[N];
            const uint32_t t = tmem + b * tc::kTmemCols + ((uint32_t)((warp & 3) * 32) << 16);
            tc::tmem_ld16(t, acc);
            if constexpr (N == 32) tc::tmem_ld16(t + 16, acc + 16);
            tc::tc_fence_before();
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(&acc_free[b]))
                         : "memory");
#pragma unroll
            for (int n = 0; n < N; n++) sum[n] += acc[n];
        }
    }
    // the products are done with the stages and the accumulators
    if (nch > 0 && tid <= 128) ok = tc::mbar_wait(&done, 0) && ok;
    ok = __syncthreads_and(ok);
    tc::tc_fence_after();
    if (ok && nch > 0) {
        if constexpr (Op::kMN) {
            if (warp > 4) Op::epilogue(args, (warp & 3) * 32 + (tid & 31), nullptr, sum);
        } else if (warp < 4) {
            float acc[N];
            const uint32_t t = tmem + ((uint32_t)(warp * 32) << 16);
            tc::tmem_ld16(t, acc);
            if constexpr (N == 32) tc::tmem_ld16(t + 16, acc + 16);
            Op::epilogue(args, tid, smem[0] + 2048 * warp, acc);
        }
    } else if (!ok && tid == 0 && status) {
        atomicCAS(status, 0, tc::kErrTimeout);
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, kCols);
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
    const cudaError_t e = cudaFuncSetAttribute(
        k_tc_train<Op>, cudaFuncAttributeMaxDynamicSharedMemorySize, train_smem<Op>());
    if (e != cudaSuccess) return e;
    k_tc_train<Op><<<grid, train_threads<Op>(), train_smem<Op>(), s>>>(a, status);
    return cudaGetLastError();
}

unsigned tiles_of(const Dims3& d) { return (unsigned)(((long long)d.nx * d.ny * d.nz + 127) / 128); }

// slabs of a contraction over the voxels of d, split over about `ctas` CTAs
void split(WeightArgs& w, const Dims3& d, int ctas, unsigned& rows) {
    w.slabs = (int)(((long long)d.nx * d.ny * d.nz + 31) / 32);
    w.per_cta = std::max(16, (w.slabs + ctas - 1) / ctas);
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
    split(w, l, 57, rows);
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
    split(w, l, 65, rows);
    cudaError_t e = run<TE2w>(w, dim3(7, rows), status, s);
    if (e != cudaSuccess) return e;
    const long long nl = (long long)l.nx * l.ny * l.nz;
    k_latent_bias<<<(unsigned)std::min<long long>((nl + 255) / 256, 152), 256, 0, s>>>(glat, nl, grad);
    return cudaGetLastError();
}
cudaError_t ae_train_patch_weights(const bf16* xq, const bf16* ga1, const bf16* gy, const bf16* g1,
                                   const bf16* ga3, float* grad, Dims3 h, Dims3 l, int* status,
                                   cudaStream_t s) {
    WeightArgs w{};
    w.a = ga1;
    w.b = g1;
    w.c = ga3;
    w.gy = gy;
    w.xq = xq;
    w.grad = grad;
    w.h = h;
    w.l = l;
    unsigned rows;
    split(w, h, 304, rows);
    return run<TPatch>(w, dim3(rows), status, s);
}

}  // namespace rtm
