// The radius-8 stencil step with two rows per thread (16-row tiles).
//
// The plane march of stencil_tma.cu is bound at radius 8 by shared memory, not
// by HBM: per point its 8-row tiles read 23 floats from it (16 y neighbours,
// 4 floats of x neighbours, three operands) and the copies write 6.75 into it
// (a 64 x 8 tile brings an 80 x 24 plane), 119 wavefronts of 128 points where
// the HBM rate allows 96 clocks. Here a thread owns 4 x points of two
// neighbouring rows: rows y - 8 .. y + 9 serve both, 8 y-neighbour floats per
// point instead of 16, and a 64 x 16 tile brings 2.5 floats of plane per point
// instead of 3.75. That is 82 wavefronts. The z queue of both rows takes 144
// registers, so two blocks of 128 threads run per SM: the loads of a plane
// are independent, so eight warps keep the shared-memory pipe busy.
//
// Microseconds per launch for a 512^3 model in 576^3, automatic slabs (8-row
// tiles of one row per thread -> here, and of the measured HBM copy rate):
// forward 663 -> 536 (69 -> 85 %), forward + snapshot 687 -> 584 (78 -> 91 %),
// backward + imaging 760 -> 728 (91 -> 95 %); a 300^3 model in 364^3: 206 -> 164,
// 209 -> 180, 225 -> 199. 32 x 32 tiles (2.25 floats of plane per point) took
// 537 / 624 / 800 at 576^3 without a sponge, where these take 534 / 592 / 780:
// their narrower rows cost more than the smaller halo gains. The queue moves
// every second plane; every plane (8 fewer registers) was the same within 1 %.
//
// The rings, barriers and epilogues are those of the split-ring instances of
// stencil_tma.cu, and every cell sees their operations in their order, so the
// results are the same bits.

#include <cuda.h>
#include <string.h>

#include "../../include/rtm.h"
#include "pdl.cuh"
#include "rtm_internal.h"
#include "star_rows.cuh"
#include "stencil_common.cuh"
#include "tma_encode.h"
#include "wait_clock.cuh"

namespace rtm {

namespace {

constexpr int R = 8;
constexpr int BX = 16, BY = 8;           // threads
constexpr int TX = 4 * BX, TY = 2 * BY;  // tile
constexpr int SW = TX + 2 * R, SH = TY + 2 * R;
constexpr int UPLANE = SW * SH, APLANE = TX * TY;  // floats
constexpr int G = 2;                     // planes per queue move

template <int MODE>
__host__ __device__ constexpr bool two_aux() {
    return MODE == MODE_BWD_IMAGE || MODE == MODE_BWD_GRAD;
}
template <int MODE>
struct Cfg {
    // planes loaded ahead; a third helps where a step stores two fields (576^3:
    // 614 -> 592 us per forward + snapshot launch), not elsewhere
    static constexpr int P = (MODE == MODE_FWD_SNAP || MODE == MODE_FWD_LU) ? 3 : 2;
    static constexpr int NS = P + 1;                         // ring slots
    static constexpr int NA = (two_aux<MODE>() ? 4 : 2) + 1;  // operand tiles, queue head last
    static constexpr int SMEM = NS * (UPLANE + NA * APLANE) * 4;
    static_assert(2 * (SMEM + 1024 + 256) <= 228 * 1024, "rings do not fit two blocks");
};

struct RowMaps {
    CUtensorMap u, prev, c, e1, e2, uh;
};

__device__ __forceinline__ uint32_t sptr(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void expect(uint64_t* b, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(sptr(b)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool poll(uint64_t* b, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(sptr(b)), "r"(parity)
        : "memory");
    return done != 0;
}
// bounded wait; false if it ran out (the block's abort flag is raised) or the
// block aborted meanwhile
__device__ __forceinline__ bool wait_slot(uint64_t* b, uint32_t parity, int* abort_flag) {
    if (poll(b, parity)) return true;
    const unsigned long long t0 = wait_now();
    for (long long i = 0;; i++) {
        if (poll(b, parity)) return true;
        if (*reinterpret_cast<volatile int*>(abort_flag)) return false;
        if (wait_expired(i, t0)) break;
    }
    *reinterpret_cast<volatile int*>(abort_flag) = 1;
    return false;
}
__device__ __forceinline__ void copy3(float* dst, const CUtensorMap* map, int x, int y, int z,
                                      uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%2, %3, %4}], [%5];" ::"r"(sptr(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(sptr(bar))
        : "memory");
}

// STALL: the instance that takes a test-armed stall (rtm_set_test_stall)
template <int MODE, bool STALL = false>
__global__ void __launch_bounds__(BX* BY, 2)
    k_stencil_rows(const __grid_constant__ StepArgs A, const __grid_constant__ RowMaps M,
                   int* status, int stall) {
    using C = Cfg<MODE>;
    extern __shared__ __align__(128) float dsm[];
    float* uring = dsm;
    float* aring = dsm + C::NS * UPLANE;
    __shared__ __align__(8) uint64_t bar[C::NS];
    __shared__ int abort_flag;

    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * BX + tx;
    const int x0 = A.xorg + blockIdx.x * TX, y0 = A.yorg + blockIdx.y * TY;
    const int x = x0 + 4 * tx, y = y0 + 2 * ty;
    const int zb = A.zorg + blockIdx.z * A.zchunk;
    const int ze = min(A.zend, zb + A.zchunk);
    const int xend_v = (A.xend + 3) & ~3;  // a vector across the region's x end is computed whole
    const bool xin = x < A.NX && x < xend_v;
    bool own[2];
    bool ym[2];
#pragma unroll
    for (int h = 0; h < 2; h++) {
        own[h] = xin && y + h < A.NY && y + h < A.yend;
        ym[h] = y + h >= A.nb && y + h < A.nb + A.ny;
    }
    const bool xm = x + 3 >= A.nb && x < A.nb + A.nx;
    const size_t plane = (size_t)A.NX * (size_t)A.NY;
    const size_t col = (size_t)y * A.NX + x;
    const size_t slab_col = (size_t)(y - A.nb) * A.NX + x;  // wraps for y < nb, unused there
    const size_t slab_plane = (size_t)A.ny * A.NX;

    if (tid == 0) {
        for (int s = 0; s < C::NS; s++)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sptr(&bar[s])));
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    pdl_wait();

    int issued = zb;  // thread 0: planes [zb, issued) are on their way
    auto issue = [&](int p) {
        issued = p + 1;
        const int slot = (p - zb) % C::NS;
        float* base = aring + slot * C::NA * APLANE;
        uint32_t extra = 0;
        if constexpr (STALL) {
            // 16 bytes that never arrive, for one of the last planes of block 0: no
            // later copy takes its slot and completes the stuck phase's successor
            if (p == ze - 1 - stall && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0)
                extra = 16;
        }
        expect(&bar[slot], (UPLANE + C::NA * APLANE) * 4 + extra);
        copy3(uring + slot * UPLANE, &M.u, x0 - R, y0 - R, p, &bar[slot]);
        copy3(base + (C::NA - 1) * APLANE, &M.uh, x0, y0, p + R, &bar[slot]);
        copy3(base, &M.prev, x0, y0, p, &bar[slot]);
        copy3(base + APLANE, &M.c, x0, y0, p, &bar[slot]);
        if constexpr (MODE == MODE_BWD_IMAGE) {
            if (A.snap_padded)
                copy3(base + 2 * APLANE, &M.e1, x0, y0, p, &bar[slot]);
            else
                copy3(base + 2 * APLANE, &M.e1, x0, y0 - A.nb, p - A.nb, &bar[slot]);
            copy3(base + 3 * APLANE, &M.e2, x0, y0 - A.nb, p - A.nb, &bar[slot]);
        } else if constexpr (MODE == MODE_BWD_GRAD) {
            copy3(base + 2 * APLANE, &M.e1, x0, y0, p, &bar[slot]);
            copy3(base + 3 * APLANE, &M.e2, x0, y0, p, &bar[slot]);
        }
    };
    if (tid == 0)
        for (int p = zb; p < zb + C::P && p < ze; p++) issue(p);

    F4 gxy[2];
#pragma unroll
    for (int h = 0; h < 2; h++) {
        gxy[h] = zero4();
        if (own[h]) {
            const float gyv = A.gy[y + h];
#pragma unroll
            for (int i = 0; i < 4; i++) gxy[h].v[i] = A.gx[x + i] * gyv;
        }
    }
    // queue: plane z0 + t of a group reads entries t .. t + 2r
    F4 q[2][2 * R + G];
#pragma unroll
    for (int h = 0; h < 2; h++) {
#pragma unroll
        for (int i = 0; i < 2 * R; i++) {
            const int zz = zb - R + i;
            q[h][i] = own[h] && zz >= 0 && zz < A.NZ
                          ? ld_l2(A.u_cur + (size_t)zz * plane + col + (size_t)h * A.NX)
                          : zero4();
        }
#pragma unroll
        for (int i = 2 * R; i < 2 * R + G; i++) q[h][i] = zero4();
    }

    const int aux_off = 2 * ty * TX + 4 * tx;
    float ssq = 0.f;
    int slot = 0;
    uint32_t phase = 0;
    for (int z0 = zb; z0 < ze; z0 += G) {
#pragma unroll
        for (int t = 0; t < G; t++) {
            const int z = z0 + t;
            if (z >= ze) break;  // the same for every thread of the block
            if (tid == 0 && z + C::P < ze && !abort_flag) issue(z + C::P);
            const bool ok = !*reinterpret_cast<volatile int*>(&abort_flag) &&
                            wait_slot(&bar[slot], phase, &abort_flag);
            const float* aux = aring + slot * C::NA * APLANE + aux_off;
            // this thread's first row in the centre plane
            const float* S = uring + slot * UPLANE + (R + 2 * ty) * SW + R + 4 * tx;
#pragma unroll
            for (int h = 0; h < 2; h++) q[h][2 * R + t] = lds4(aux + (C::NA - 1) * APLANE + h * TX);
            if (own[0] && ok) {
                F4 lap[2];
                star_rows<R, 2>(S, SW, q, t, A.a, lap);
                const float gzv = A.gz[z];
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    if (!own[h]) break;
                    const F4 up = lds4(aux + h * TX);
                    const F4 cc = lds4(aux + APLANE + h * TX);
                    const F4& qc = q[h][R + t];
                    F4 out;
                    if constexpr (MODE == MODE_REV) {
#pragma unroll
                        for (int i = 0; i < 4; i++) {
                            out.v[i] = fmaf(cc.v[i], lap[h].v[i], 2.0f * qc.v[i]) - up.v[i];
                            // cells outside the model keep their value
                            const int mx = x + i - A.nb;
                            if (mx < 0 || mx >= A.nx || !ym[h]) out.v[i] = up.v[i];
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < 4; i++) {
                            const float g = gxy[h].v[i] * gzv;
                            out.v[i] = g * fmaf(cc.v[i], lap[h].v[i], 2.0f * qc.v[i]) -
                                       (g * g) * up.v[i];
                        }
                    }
                    const size_t o = (size_t)z * plane + col + (size_t)h * A.NX;
                    st_stream(A.u_prev + o, out);
                    const bool inm = xm && ym[h] && z >= A.nb && z < A.nb + A.nz;
                    const size_t so =
                        (size_t)(z - A.nb) * slab_plane + slab_col + (size_t)h * A.NX;
                    if constexpr (MODE == MODE_FWD_SUMSQ) {
                        if (inm) {
#pragma unroll
                            for (int i = 0; i < 4; i++)
                                if (x + i >= A.nb && x + i < A.nb + A.nx)
                                    ssq = fmaf(out.v[i], out.v[i], ssq);
                        }
                    } else if constexpr (MODE == MODE_FWD_SNAP) {
                        if (inm) st_stream(A.snap + so, out);
                    } else if constexpr (MODE == MODE_FWD_LU) {
                        st_stream(A.snap + o, lap[h]);
                    } else if constexpr (two_aux<MODE>()) {
                        if (MODE == MODE_BWD_GRAD || inm) {
                            const F4 sv = lds4(aux + 2 * APLANE + h * TX);
                            F4 acc = lds4(aux + 3 * APLANE + h * TX);
#pragma unroll
                            for (int i = 0; i < 4; i++) acc.v[i] = fmaf(sv.v[i], out.v[i], acc.v[i]);
                            st_stream(A.acc + (MODE == MODE_BWD_GRAD ? o : so), acc);
                        }
                    }
                }
            }
            __syncthreads();  // every thread is done with the slot: it may be refilled
            if (++slot == C::NS) slot = 0, phase ^= 1;
        }
#pragma unroll
        for (int h = 0; h < 2; h++)
#pragma unroll
            for (int i = 0; i < 2 * R; i++) q[h][i] = q[h][i + G];
    }
    if constexpr (MODE == MODE_FWD_SUMSQ) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ssq += __shfl_xor_sync(0xffffffffu, ssq, o);
        if ((tid & 31) == 0 && ssq != 0.f) atomicAdd(A.sumsq, (double)ssq);
    }
    // after an abort the newest copy into each slot may still be in flight:
    // wait for it, bounded, before the block leaves its shared memory
    if (tid == 0 && abort_flag) {
        for (int p = max(zb, issued - C::NS); p < issued; p++) {
            const unsigned long long t0 = wait_now();
            uint64_t* b = &bar[(p - zb) % C::NS];
            for (long long i = 0; !poll(b, ((p - zb) / C::NS) & 1) && !wait_expired(i, t0); i++) {
            }
        }
        if (status) atomicCAS(status, 0, RTM_ERR_TIMEOUT);
    }
}

template <int MODE>
cudaError_t launch_t(const StepArgs& a, int* status, cudaStream_t s) {
    constexpr int smem = Cfg<MODE>::SMEM;
    cudaError_t e = cudaFuncSetAttribute(k_stencil_rows<MODE>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    RowMaps M;
    memset(&M, 0, sizeof M);
    if ((e = tma_map3(&M.u, a.u_cur, a.NX, a.NY, a.NZ, SW, SH)) != cudaSuccess ||
        (e = tma_map3(&M.uh, a.u_cur, a.NX, a.NY, a.NZ, TX, TY)) != cudaSuccess ||
        (e = tma_map3(&M.prev, a.u_prev, a.NX, a.NY, a.NZ, TX, TY)) != cudaSuccess ||
        (e = tma_map3(&M.c, a.c, a.NX, a.NY, a.NZ, TX, TY)) != cudaSuccess)
        return e;
    if (two_aux<MODE>()) {
        const bool padded = MODE == MODE_BWD_GRAD || a.snap_padded;
        if ((e = tma_map3(&M.e1, a.snap, a.NX, padded ? a.NY : a.ny, padded ? a.NZ : a.nz, TX, TY)) !=
            cudaSuccess)
            return e;
        const bool full = MODE == MODE_BWD_GRAD;
        if ((e = tma_map3(&M.e2, a.acc, a.NX, full ? a.NY : a.ny, full ? a.NZ : a.nz, TX, TY)) !=
            cudaSuccess)
            return e;
    }
    if (a.xorg % 4 || a.xend <= a.xorg || a.yend <= a.yorg || a.zend <= a.zorg || a.zchunk < 1)
        return cudaErrorInvalidValue;
    const dim3 grid((a.xend - a.xorg + TX - 1) / TX, (a.yend - a.yorg + TY - 1) / TY,
                    (a.zend - a.zorg + a.zchunk - 1) / a.zchunk);
    if constexpr (MODE == MODE_FWD) {
        const int stall = take_test_stall(RTM_STALL_ROWS);
        if (stall >= 0) {
            e = cudaFuncSetAttribute(k_stencil_rows<MODE, true>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            if (e != cudaSuccess) return e;
            return launch_next(k_stencil_rows<MODE, true>, grid, dim3(BX, BY), smem, s, a, M, status,
                               stall < Cfg<MODE>::NS ? stall : Cfg<MODE>::NS - 1);
        }
    }
    return launch_next(k_stencil_rows<MODE>, grid, dim3(BX, BY), smem, s, a, M, status, -1);
}

// encoded maps of this thread, by every encoding argument: a shot launches its
// steps thousands of times on the same few buffers
struct MapKey {
    const float* base;
    int nx, ny, nz, bx, by;
    bool operator==(const MapKey& o) const {
        return base == o.base && nx == o.nx && ny == o.ny && nz == o.nz && bx == o.bx && by == o.by;
    }
};
constexpr int kMaps = 64;
struct MapCache {
    MapKey key[kMaps];
    CUtensorMap map[kMaps];
    int used = 0, next = 0;
};
thread_local MapCache t_maps;

}  // namespace

cudaError_t tma_map3(CUtensorMap* m, const float* base, int nx, int ny, int nz, int bx, int by) {
    const MapKey k{base, nx, ny, nz, bx, by};
    MapCache& c = t_maps;
    for (int i = 0; i < c.used; i++)
        if (c.key[i] == k) {
            *m = c.map[i];
            return cudaSuccess;
        }
    EncodeTiledFn f = tma_encoder();
    if (!f) return cudaErrorNotSupported;
    if (((uintptr_t)base % 16) || (nx % 4)) return cudaErrorInvalidValue;
    const cuuint64_t dims[3] = {(cuuint64_t)nx, (cuuint64_t)ny, (cuuint64_t)nz};
    const cuuint64_t strides[2] = {(cuuint64_t)nx * 4, (cuuint64_t)nx * ny * 4};
    const cuuint32_t box[3] = {(cuuint32_t)bx, (cuuint32_t)by, 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    const CUresult r = f(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(base), dims,
                         strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                         CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
    const int slot = c.used < kMaps ? c.used++ : c.next;
    if (c.used == kMaps) c.next = (slot + 1) % kMaps;
    c.key[slot] = k;
    c.map[slot] = *m;
    return cudaSuccess;
}

cudaError_t launch_stencil_rows(int mode, const StepArgs& a, int* status, cudaStream_t s) {
    switch (mode) {
        case MODE_FWD: return launch_t<MODE_FWD>(a, status, s);
        case MODE_FWD_SNAP: return launch_t<MODE_FWD_SNAP>(a, status, s);
        case MODE_BWD_IMAGE: return launch_t<MODE_BWD_IMAGE>(a, status, s);
        case MODE_FWD_LU: return launch_t<MODE_FWD_LU>(a, status, s);
        case MODE_BWD_GRAD: return launch_t<MODE_BWD_GRAD>(a, status, s);
        case MODE_REV: return launch_t<MODE_REV>(a, status, s);
        case MODE_FWD_SUMSQ: return launch_t<MODE_FWD_SUMSQ>(a, status, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace rtm
