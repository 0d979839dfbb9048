// The star Laplacian of ROWS neighbouring rows of four points, from a plane in
// shared memory and a register queue along z, on packed point pairs.
//
// With two rows per thread the rows y - r .. y + r + 1 serve both: half the
// y-neighbour reads per point. Every cell's sums run in the order of the
// one-row form: at radius 8 even and odd offsets in two chains, added last.
#pragma once

#include "packed_f32x2.cuh"
#include "stencil_common.cuh"

namespace rtm {

// S: this thread's first point of the plane (row stride SW); q[h][t .. t + 2R]:
// its column along z in row h; a: the weights
template <int R, int ROWS, int QN>
__device__ __forceinline__ void star_rows(const float* S, const int SW, const F4 (&q)[ROWS][QN],
                                          const int t, const float* a, F4 (&lap)[ROWS]) {
    static_assert(ROWS == 1 || ROWS == 2, "one or two rows per thread");
    float v[ROWS][4 + 2 * R];
    uint64_t L[ROWS][2], Lo[ROWS][2];
    const uint64_t a0 = f32x2::pack(a[0], a[0]);
#pragma unroll
    for (int h = 0; h < ROWS; h++) {
#pragma unroll
        for (int g = 0; g < R / 4; g++) {
            const F4 l = lds4(S + h * SW - R + 4 * g), r = lds4(S + h * SW + 4 + 4 * g);
#pragma unroll
            for (int i = 0; i < 4; i++) {
                v[h][4 * g + i] = l.v[i];
                v[h][R + 4 + 4 * g + i] = r.v[i];
            }
        }
        const F4& qc = q[h][R + t];
#pragma unroll
        for (int i = 0; i < 4; i++) v[h][R + i] = qc.v[i];
#pragma unroll
        for (int j = 0; j < 2; j++) {
            L[h][j] = f32x2::mul(a0, f32x2::pack(qc.v[2 * j], qc.v[2 * j + 1]));
            Lo[h][j] = 0;  // the bit pattern of two +0.0f
        }
    }
    // two rows: rows 1 - k and k, read for one row at offset k - 1, serve the
    // other at offset k
    F4 below = q[0][R + t], above = q[ROWS - 1][R + t];
#pragma unroll
    for (int k = 1; k <= R; k++) {
        const F4 lo = lds4(S - k * SW), hi = lds4(S + (k + ROWS - 1) * SW);
        const uint64_t ak = f32x2::pack(a[k], a[k]);
#pragma unroll
        for (int h = 0; h < ROWS; h++) {
            const F4& ylo = h == 0 ? lo : below;
            const F4& yhi = h == ROWS - 1 ? hi : above;
            const F4 &zm = q[h][R + t - k], &zp = q[h][R + t + k];
            const float* w = v[h];
#pragma unroll
            for (int j = 0; j < 2; j++) {
                const int i = 2 * j;
                // at odd offsets the pairs straddle register pairs: two scalar
                // sums cost less than moving them together
                const uint64_t px =
                    (k & 1) ? f32x2::pack(w[R + i - k] + w[R + i + k],
                                          w[R + i + 1 - k] + w[R + i + 1 + k])
                            : f32x2::add(f32x2::pack(w[R + i - k], w[R + i + 1 - k]),
                                         f32x2::pack(w[R + i + k], w[R + i + 1 + k]));
                const uint64_t py = f32x2::add(f32x2::pack(ylo.v[i], ylo.v[i + 1]),
                                               f32x2::pack(yhi.v[i], yhi.v[i + 1]));
                const uint64_t pz = f32x2::add(f32x2::pack(zm.v[i], zm.v[i + 1]),
                                               f32x2::pack(zp.v[i], zp.v[i + 1]));
                const uint64_t s = f32x2::add(f32x2::add(px, py), pz);
                if (R == 8 && (k & 1))
                    Lo[h][j] = f32x2::fma(ak, s, Lo[h][j]);
                else
                    L[h][j] = f32x2::fma(ak, s, L[h][j]);
            }
        }
        below = lo;
        above = hi;
    }
#pragma unroll
    for (int h = 0; h < ROWS; h++)
#pragma unroll
        for (int j = 0; j < 2; j++)
            f32x2::unpack(R == 8 ? f32x2::add(L[h][j], Lo[h][j]) : L[h][j], lap[h].v[2 * j],
                          lap[h].v[2 * j + 1]);
}

}  // namespace rtm
