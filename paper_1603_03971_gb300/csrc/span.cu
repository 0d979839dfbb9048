// Many time steps in one cooperative launch, for grids that the L2 cache
// holds.
//
// On such grids a step is bound by latencies, not by bytes: at 104^3 padded,
// radius 4, the receiver kernel and the plane-marching stencil take 10 us (21
// before they were dependent launches), and HBM would need 2.7 us. Here the padded
// grid is cut into one brick per SM, each block keeps its brick for every step of the span, and blocks meet at a
// grid barrier between steps. The brick's u^n with its halo arrives as one
// bulk tensor copy, so a step pays one copy latency; its u^{n-1}, c, snapshot
// and image, which no other block writes, and the receivers' terms are
// fetched while the barrier is under way. Each thread then owns 4 x points by
// PZ planes: its z column is read once into registers (PZ + 2r vectors,
// nothing is shifted), its x and y neighbours come from shared memory.
// The source, the receivers, the snapshots and the image are handled by the
// owners of the cells inside the step (data and boundary band are gathered
// one step later, from a complete field), so a step has one barrier in either
// direction.
//
// Microseconds per step of a 60-step shot that keeps every snapshot, forward /
// backward + imaging, against the launch-per-step kernels (8-row tiles, receiver
// kernel included) and against these before they were dependent launches:
//   40 x 36 x 32, r = 4:      3.8 / 4.3      8.9 / 8.8      21 / 20
//   64 x 60 x 56, r = 4:      4.0 / 4.7      9.9 / 8.8      21 / 20
//   104^3, r = 4:             7.5 / 9.3      10.5 / 9.8     21 / 21
//   128 x 122 x 112, r = 4:   9.9 / 12.2     11.8 / 11.4    21 / 21
//   104^3, r = 8 (forward):   11.9           11.8           27
//   104^3, r = 4, off grid:   12.2 / 14.7    26 / 25        34 / 33   (1024 receivers)
// A brick has to fit one SM's shared memory, which is also where a launch per
// step has caught up. A span takes every SM: shots of several host threads run
// one after another (ms per 100-step shot with 1 / 4 / 8 threads, spans against
// launches: 40 x 36 x 32 0.87 / 0.28 / 0.24 and 1.77 / 0.58 / 0.39; 104^3 1.68 /
// 1.58 / 1.57 and 2.05 / 1.06 / 1.15). A call cannot see the others, so whoever
// runs four such shots or more at a time names a variant (rtm_set_tuning).
// Off the grid a receiver is up to 8^3 taps and its neighbours share bricks:
// taken by the bricks that they reach, 1024 receivers made a backward step 39
// us (3969: 120). So the blocks share the receivers out evenly and the data go
// through one of two padded fields, a step ahead (3969: 20).
// What is left at 104^3: about 4 us of shared-memory reads and instructions,
// the rest barrier, copy and store latency (3.1 us on the smallest grid).
//
// Every cell sees the operations of the plane-marching kernels in their
// order, so both paths give the same bits, except where receivers meet: those of
// one cell, and off the grid the taps of neighbours, are summed before they are
// scaled and added to the field, where the launches add each to the field by
// itself. There the results differ by roundings, and in either path by the order
// of the atomic sums (three terms or more).

#include <string.h>

#include <algorithm>

#include "../../include/rtm.h"
#include "band.cuh"
#include "packed_f32x2.cuh"
#include "span.h"
#include "stencil_common.cuh"
#include "tma_encode.h"
#include "wait_clock.cuh"

namespace rtm {

namespace {

// planes per thread: a column of 4 shares its z neighbours' loads; grids that
// leave a block few columns spread them over four times the threads
constexpr int kColumn = 4;
constexpr int kTapCap = 32;                              // tap tables of a block kept in shared memory
constexpr unsigned long long kBarrierNs = 20000000000ull;  // bound of a grid barrier: 20 s (SpanArgs)
constexpr int kSmemMax = 227 * 1024;

// threads of a block: what the registers of one block per SM allow (128, 168
// or 255 each; a warp count that is a multiple of the four SM partitions)
template <int R, bool BWD, int PZ>
__host__ __device__ constexpr int span_threads() {
    return PZ == 1 || R == 4 ? 512 : 384;
}

static_assert(sizeof(rtm_point_taps) * kTapCap <= 4 * kSpanListCap, "tap tables share the list's room");

struct SpanMaps {
    CUtensorMap u[2];
};

__device__ __forceinline__ uint32_t su32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void load_box(float* dst, const CUtensorMap* map, int x, int y, int z,
                                         uint32_t bytes, uint64_t* bar) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(bar)),
                 "r"(bytes)
                 : "memory");
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%2, %3, %4}], [%5];" ::"r"(su32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(su32(bar))
        : "memory");
}
// bounded wait for a box, whose copy follows thread 0's bounded wait for the
// other blocks. One that runs out ends the span at the next grid barrier
__device__ __forceinline__ bool poll_box(uint64_t* bar, uint32_t parity, const SpanArgs& A) {
    const uint32_t a = su32(bar);
    if (mbar_try_wait_sleep(a, parity, 20000)) return true;
    const unsigned long long t0 = wait_now();
    while (!mbar_try_wait_sleep(a, parity, 20000))
        if (wait_now() - t0 > A.limit_ns + kWaitNs) return false;
    return true;
}

__device__ __forceinline__ void wait_box(uint64_t* bar, uint32_t parity, const SpanArgs& A) {
    if (poll_box(bar, parity, A)) return;
    atomicExch(&A.ctrl->abort, 1);
    if (A.status) atomicCAS(A.status, 0, RTM_ERR_TIMEOUT);
    if (threadIdx.x == 0) poll_box(bar, parity, A);  // the copy should land before the block leaves
}

// thread 0's half of the grid barrier between two steps, split so that what
// does not depend on other blocks runs between the halves. The block has met
// at a block barrier before the arrival, so its writes come first
__device__ __forceinline__ void grid_arrive(SpanCtrl* ctrl) {
    __threadfence();
    atomicAdd(&ctrl->count, 1u);
}
// false if the wait ran out or another block gave up; otherwise this thread
// may issue copies of what the other blocks wrote before they arrived
__device__ __forceinline__ bool grid_wait(const SpanArgs& A, unsigned int target) {
    SpanCtrl* const ctrl = A.ctrl;
    unsigned long long t0 = 0;
    bool ok = *reinterpret_cast<volatile int*>(&ctrl->abort) == 0;
    for (long long i = 0; ok; i++) {
        unsigned int v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&ctrl->count) : "memory");
        if ((int)(v - target) >= 0) break;
        if ((i & 63) == 63) {
            const unsigned long long t = wait_now();
            if (t0 == 0) t0 = t;
            if (*reinterpret_cast<volatile int*>(&ctrl->abort) || t - t0 > A.limit_ns) {
                atomicExch(&ctrl->abort, 1);
                if (A.status) atomicCAS(A.status, 0, RTM_ERR_TIMEOUT);
                ok = false;
            }
        }
    }
    // the other blocks wrote through the generic proxy, the copies read
    // through the asynchronous one
    asm volatile("fence.proxy.async.global;" ::: "memory");
    return ok;
}

__device__ __forceinline__ int taps_of(const rtm_point_taps& P) {
    const bool ok = P.nx >= 1 && P.nx <= 8 && P.ny >= 1 && P.ny <= 8 && P.nz >= 1 && P.nz <= 8;
    return ok ? P.nx * P.ny * P.nz : 0;
}
// f(x, y, z, weight) for the taps of P, over the lanes of a warp: a lane takes
// (x, y) columns of the box, whose z taps are independent
template <class F>
__device__ __forceinline__ void for_taps(const rtm_point_taps& P, int lane, F&& f) {
    if (taps_of(P) == 0) return;
    const int nx = P.nx, nxy = nx * P.ny, nz = P.nz;
    for (int p = lane; p < nxy; p += 32) {
        const int b = p / nx, a = p - b * nx;
        const float w = P.wx[a] * P.wy[b];
#pragma unroll
        for (int c = 0; c < 8; c++)
            if (c < nz) f(P.i0 + a, P.j0 + b, P.k0 + c, w * P.wz[c]);
    }
}

// an entry without taps, or with taps outside the padded grid
__device__ __forceinline__ bool taps_outside(const rtm_point_taps& P, const SpanArgs& A) {
    return taps_of(P) == 0 || P.i0 < 0 || P.i0 > A.NX - P.nx || P.j0 < 0 || P.j0 > A.NY - P.ny ||
           P.k0 < 0 || P.k0 > A.NZ - P.nz;
}

template <bool OFF>
__device__ __forceinline__ bool rec_outside(const SpanArgs& A, int j) {
    if constexpr (OFF) {
        return taps_outside(A.taps[1 + j], A);
    } else {
        const int x = A.rec[3 * j] + A.nb, y = A.rec[3 * j + 1] + A.nb, z = A.rec[3 * j + 2] + A.nb;
        return x < 0 || x >= A.NX || y < 0 || y >= A.NY || z < 0 || z >= A.NZ;
    }
}

// BWD: receiver propagation; OFF: the source and receivers come from a tap table
template <int R, bool BWD, int PZ, bool OFF>
__global__ void __launch_bounds__(span_threads<R, BWD, PZ>(), 1)
    k_span(const __grid_constant__ SpanArgs A, const __grid_constant__ SpanMaps M) {
    extern __shared__ __align__(128) float dsm[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ int s_ok, s_count, s_zlo, s_zhi;
    __shared__ rtm_point_taps s_src;  // OFF: the source
    const SpanPlan& P = A.P;
    const int tid = threadIdx.x, T = blockDim.x;
    const int SW = 4 * P.bxv + 2 * R, SH = P.by + 2 * R, SD = P.bz + 2 * R;
    const int box = SW * SH * SD;
    const int bx = 4 * P.bxv, cells = bx * P.by * P.bz;
    float* inj = dsm + ((box + 31) & ~31);                 // BWD: receiver data by cell of the brick
    // BWD: receivers that reach the brick; OFF: tap tables of the receivers
    // that this block gathers or scatters (every gridDim.x-th)
    int* list = reinterpret_cast<int*>(inj + (BWD ? cells : 0));
    rtm_point_taps* tables = reinterpret_cast<rtm_point_taps*>(list);
    const bool scatter = OFF && BWD && A.scatter[0] != nullptr;
    const int my_recs = (A.nrec - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    const size_t plane = (size_t)A.NX * A.NY;
    const int ix = blockIdx.x % P.nbx, iyz = blockIdx.x / P.nbx;
    const int x0 = ix * bx, y0 = iyz % P.nby * P.by, z0 = iyz / P.nby * P.bz;  // the brick

    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&bar)));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_count = 0;
        s_zlo = A.NZ;
        s_zhi = -1;
        if (OFF && !BWD) s_src = A.taps[0];
        s_ok = *reinterpret_cast<volatile int*>(&A.ctrl->abort) == 0;
    }
    __syncthreads();
    if (!*reinterpret_cast<volatile int*>(&s_ok)) return;  // an earlier span gave up

    // out-of-range receivers and broken tap entries, once per span
    if (BWD ? A.rdata != nullptr : A.data != nullptr) {
        for (int j = blockIdx.x * T + tid; j < A.nrec; j += gridDim.x * T)
            if (rec_outside<OFF>(A, j)) atomicCAS(A.status, 0, RTM_ERR_INVALID);
    }
    if (!BWD && OFF && blockIdx.x == 0 && tid == 0 && taps_outside(A.taps[0], A))
        atomicCAS(A.status, 0, RTM_ERR_INVALID);

    // BWD: the receivers that reach the brick; over kSpanListCap of them every
    // step scans all receivers instead
    int nlist = 0;
    if constexpr (BWD) {
        for (int i = tid; i < cells; i += T) inj[i] = 0.f;
        if (scatter) {
            // the planes that any receiver's taps reach
            int lo = A.NZ, hi = -1;
            for (int j = tid; j < A.nrec; j += T) {
                const rtm_point_taps& t = A.taps[1 + j];
                if (taps_outside(t, A) && taps_of(t) == 0) continue;
                lo = min(lo, max(t.k0, 0));
                hi = max(hi, min(t.k0 + t.nz, A.NZ) - 1);
            }
            atomicMin(&s_zlo, lo);
            atomicMax(&s_zhi, hi);
        } else if (A.rdata) {
            for (int j = tid; j < A.nrec; j += T) {
                bool hit;
                if constexpr (OFF) {
                    const rtm_point_taps& t = A.taps[1 + j];
                    hit = taps_of(t) > 0 && t.i0 < x0 + bx && t.i0 > x0 - t.nx &&
                          t.j0 < y0 + P.by && t.j0 > y0 - t.ny && t.k0 < z0 + P.bz &&
                          t.k0 > z0 - t.nz;
                } else {
                    const int x = A.rec[3 * j] + A.nb, y = A.rec[3 * j + 1] + A.nb,
                              z = A.rec[3 * j + 2] + A.nb;
                    hit = x >= x0 && x < x0 + bx && y >= y0 && y < y0 + P.by && z >= z0 &&
                          z < z0 + P.bz && x < A.NX && y < A.NY && z < A.NZ;
                }
                if (hit) {
                    const int k = atomicAdd(&s_count, 1);
                    if (k < kSpanListCap) list[k] = j;
                }
            }
        }
        __syncthreads();
        nlist = s_count;
    }
    if constexpr (OFF) {
        if (!BWD || scatter)
            for (int k = tid; k < min(my_recs, kTapCap); k += T)
                tables[k] = A.taps[1 + blockIdx.x + k * gridDim.x];
        __syncthreads();
    }
    // receiver blockIdx.x + k gridDim.x
    auto table = [&](int k) -> const rtm_point_taps& {
        return k < kTapCap ? tables[k] : A.taps[1 + blockIdx.x + k * gridDim.x];
    };
    // OFF: many receivers' taps meet in few bricks, so all blocks take a share
    // of them and add the data of step m into a padded field, which the cells'
    // owners read (and clear) one barrier later
    auto scatter_taps = [&](int m, float* field) {
        const float* row = A.rdata + (size_t)(m - 1) * A.nrec;
        for (int k = tid >> 5; k < my_recs; k += T >> 5) {
            const float r = row[blockIdx.x + k * gridDim.x];
            for_taps(table(k), tid & 31, [&](int x, int y, int z, float w) {
                if (x >= 0 && x < A.NX && y >= 0 && y < A.NY && z >= 0 && z < A.NZ)
                    atomicAdd(field + (size_t)z * plane + (size_t)y * A.NX + x, w * r);
            });
        }
    };
    // the data of step m at the brick's receivers, summed per cell (times the
    // tap weights). They need no other block's work, so they are formed while
    // the grid barrier is under way
    auto inject = [&](int m) {
        if (nlist == 0) return;
        const bool all = nlist > kSpanListCap;
        const int count = all ? A.nrec : nlist;
        const float* row = A.rdata + (size_t)(m - 1) * A.nrec;
        auto put = [&](int x, int y, int z, float r) {
            if (x < x0 || x >= x0 + bx || y < y0 || y >= y0 + P.by || z < z0 || z >= z0 + P.bz) return;
            atomicAdd(&inj[((z - z0) * P.by + (y - y0)) * bx + (x - x0)], r);
        };
        if constexpr (OFF) {
            for (int e = tid >> 5; e < count; e += T >> 5) {
                const int j = all ? e : list[e];
                const float r = row[j];
                for_taps(A.taps[1 + j], tid & 31,
                         [&](int x, int y, int z, float w) { put(x, y, z, w * r); });
            }
        } else {
            for (int e = tid; e < count; e += T) {
                const int j = all ? e : list[e];
                put(A.rec[3 * j] + A.nb, A.rec[3 * j + 1] + A.nb, A.rec[3 * j + 2] + A.nb, row[j]);
            }
        }
        __syncthreads();
    };
    if constexpr (BWD) inject(A.first);

    const int srz = (int)(A.src / (long long)plane), srr = (int)(A.src % (long long)plane);
    const int sry = srr / A.NX, srx = srr % A.NX;
    const int items = P.bxv * P.by * (P.bz / PZ);
    const size_t slab_plane = (size_t)A.ny * A.NX;

    // forward: this thread's first receiver, if any, and its cell (-1: outside)
    const int j0 = blockIdx.x * T + tid;
    long long cell0 = -1;
    if constexpr (!BWD && !OFF) {
        if (A.data && j0 < A.nrec && !rec_outside<OFF>(A, j0))
            cell0 = (long long)(A.rec[3 * j0 + 2] + A.nb) * (long long)plane +
                    (long long)(A.rec[3 * j0 + 1] + A.nb) * A.NX + (A.rec[3 * j0] + A.nb);
    }

    for (int i = 0; i < A.nsteps; i++) {
        const float* cur = A.f[1 - (i & 1)];
        float* prev = A.f[i & 1];
        const int n = BWD ? A.first - i : A.first + i;
        const int k = BWD ? n : n + 1;  // the state this step writes
        const bool snap_now = A.snap && k % A.every == 0;
        float* snap = snap_now ? A.snap + (long long)(k / A.div - A.off) * A.snap_stride : nullptr;
        const float w = BWD ? 0.f : __ldg(A.wav + n);
        // the first items' operands are fetched before the wait for the other
        // blocks: nobody else writes them
        bool here = false;  // this thread has waited for the box
        float d0 = 0.f;     // u^n at its first receiver
        auto wait_here = [&]() {
            if (here) return;
            here = true;
            if (tid == 0) {
                // (a stalled wait: a step more than the others can get to without block 0)
                const unsigned int more = i == A.stall && blockIdx.x == 0 ? 1u : 0u;
                if (i > 0 && !grid_wait(A, A.base + gridDim.x * ((unsigned int)i + more))) {
                    s_ok = 0;  // no copy: the arrival alone completes the phase
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(&bar)) : "memory");
                } else {
                    load_box(dsm, &M.u[1 - (i & 1)], x0 - R, y0 - R, z0 - R, (uint32_t)box * 4, &bar);
                }
            }
            wait_box(&bar, i & 1, A);
            if constexpr (!BWD && !OFF) {
                if (cell0 >= 0) d0 = __ldcg(cur + cell0);
            }
        };
        for (int it = tid; it < items; it += T) {
            const int tx = it % P.bxv, rr = it / P.bxv;
            const int ty = rr % P.by, zg = rr / P.by;
            const int x = x0 + 4 * tx, y = y0 + ty, z = z0 + PZ * zg;
            if (x >= A.NX || y >= A.NY || z >= A.NZ) continue;
            const size_t o = (size_t)z * plane + (size_t)y * A.NX + x;
            const bool ym = y >= A.nb && y < A.nb + A.ny;
            const bool xm = x + 3 >= A.nb && x < A.nb + A.nx;
            const size_t so = (size_t)(z - A.nb) * slab_plane + (size_t)(y - A.nb) * A.NX + x;
            const float* pu = prev + o;
            const float* pc = A.c + o;
            auto in_model = [&](int p) {
                return xm && ym && z + p >= A.nb && z + p < A.nb + A.nz;
            };
            const bool src_here = y == sry && srx >= x && srx < x + 4;
            // pointwise operands: planes p and p + 1 are in registers or on their way
            F4 up[2], cc[2], sv[2], av[2];
            auto fetch = [&](int p) {
                const int h = p & 1;
                const bool in = z + p < A.NZ;
                up[h] = in ? ld_l2(pu + p * plane) : zero4();
                cc[h] = in ? ld_keep(pc + p * plane) : zero4();
                if constexpr (BWD) {
                    if (snap && (A.grad ? in : in_model(p))) {
                        const size_t at = A.grad ? o + p * plane : so + p * slab_plane;
                        sv[h] = ld_l2(snap + at);
                        av[h] = ld_l2(A.acc + at);
                    }
                }
            };
            fetch(0);
            if constexpr (PZ > 1) fetch(1);
            F4 gxy;
            {
                const float gyv = __ldg(A.gy + y);
                const F4 gxv = ld_keep(A.gx + x);
#pragma unroll
                for (int v = 0; v < 4; v++) gxy.v[v] = gxv.v[v] * gyv;
            }
            wait_here();
            bool hit = nlist > 0;  // receivers' data may lie in these cells
            float* given = BWD ? &inj[(PZ * zg * P.by + ty) * bx + 4 * tx] : nullptr;
            if constexpr (OFF && BWD) {
                if (scatter && z <= s_zhi && z + PZ > s_zlo) {
                    hit = true;
                    float* src = A.scatter[i & 1] + o;
#pragma unroll
                    for (int p = 0; p < PZ; p++)
                        if (z + p < A.NZ)
                            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                             su32(given + p * P.by * bx)),
                                         "l"(src + p * plane)
                                         : "memory");
                    asm volatile("cp.async.commit_group;" ::: "memory");
                }
            }
            // the z column of the vector: planes z - R .. z + PZ - 1 + R
            const float* colp = dsm + (PZ * zg * SH + R + ty) * SW + R + 4 * tx;
            F4 zc[PZ + 2 * R];
#pragma unroll
            for (int p = 0; p < PZ + 2 * R; p++) zc[p] = lds4(colp + p * SH * SW);
#pragma unroll
            for (int p = 0; p < PZ; p++) {
                if (z + p >= A.NZ) break;
                const float* S = colp + (p + R) * SH * SW;
                float v[4 + 2 * R];
#pragma unroll
                for (int h = 0; h < R / 4; h++) {
                    const F4 l = lds4(S - R + 4 * h), r = lds4(S + 4 + 4 * h);
#pragma unroll
                    for (int e = 0; e < 4; e++) {
                        v[4 * h + e] = l.v[e];
                        v[R + 4 + 4 * h + e] = r.v[e];
                    }
                }
                const F4& qc = zc[p + R];
#pragma unroll
                for (int e = 0; e < 4; e++) v[R + e] = qc.v[e];
                const float gzv = __ldg(A.gz + z + p);
                uint64_t L[2], Lo[2];
                const uint64_t a0 = f32x2::pack(A.a[0], A.a[0]);
#pragma unroll
                for (int j = 0; j < 2; j++) {
                    L[j] = f32x2::mul(a0, f32x2::pack(qc.v[2 * j], qc.v[2 * j + 1]));
                    Lo[j] = 0;
                }
#pragma unroll
                for (int d = 1; d <= R; d++) {
                    const F4 ym_ = lds4(S - d * SW), yp_ = lds4(S + d * SW);
                    const F4 &zm = zc[p + R - d], &zp = zc[p + R + d];
                    const uint64_t ak = f32x2::pack(A.a[d], A.a[d]);
#pragma unroll
                    for (int j = 0; j < 2; j++) {
                        const int e = 2 * j;
                        // at odd offsets the pairs straddle register pairs: two scalar
                        // sums cost less than moving them together
                        const uint64_t px =
                            (d & 1) ? f32x2::pack(v[R + e - d] + v[R + e + d],
                                                  v[R + e + 1 - d] + v[R + e + 1 + d])
                                    : f32x2::add(f32x2::pack(v[R + e - d], v[R + e + 1 - d]),
                                                 f32x2::pack(v[R + e + d], v[R + e + 1 + d]));
                        const uint64_t py = f32x2::add(f32x2::pack(ym_.v[e], ym_.v[e + 1]),
                                                       f32x2::pack(yp_.v[e], yp_.v[e + 1]));
                        const uint64_t pz = f32x2::add(f32x2::pack(zm.v[e], zm.v[e + 1]),
                                                       f32x2::pack(zp.v[e], zp.v[e + 1]));
                        const uint64_t sum = f32x2::add(f32x2::add(px, py), pz);
                        if (R == 8 && (d & 1))
                            Lo[j] = f32x2::fma(ak, sum, Lo[j]);
                        else
                            L[j] = f32x2::fma(ak, sum, L[j]);
                    }
                }
                F4 lap;
#pragma unroll
                for (int j = 0; j < 2; j++)
                    f32x2::unpack(R == 8 ? f32x2::add(L[j], Lo[j]) : L[j], lap.v[2 * j],
                                  lap.v[2 * j + 1]);
                if constexpr (!BWD) {
                    // the source: lower u^{n-1} by c w / (dx^3 g^2)
                    if constexpr (OFF) {
                        const rtm_point_taps& t = s_src;
                        const int dz = z + p - t.k0, dy = y - t.j0;
                        if (dz >= 0 && dz < t.nz && dy >= 0 && dy < t.ny && taps_of(t) > 0) {
#pragma unroll
                            for (int e = 0; e < 4; e++) {
                                const int dx = x + e - t.i0;
                                if (dx >= 0 && dx < t.nx) {
                                    const float wt = t.wx[dx] * t.wy[dy] * t.wz[dz];
                                    const float g = gxy.v[e] * gzv;
                                    up[p & 1].v[e] -= cc[p & 1].v[e] * (wt * w) * A.inv_dx3 / (g * g);
                                }
                            }
                        }
                    } else if (src_here && z + p == srz) {
#pragma unroll
                        for (int e = 0; e < 4; e++)
                            if (x + e == srx) {
                                const float g = gxy.v[e] * gzv;
                                up[p & 1].v[e] -= cc[p & 1].v[e] * w * A.inv_dx3 / (g * g);
                            }
                    }
                } else if (hit) {
                    if (OFF && p == 0) asm volatile("cp.async.wait_group 0;" ::: "memory");
                    float4* ip = reinterpret_cast<float4*>(given + p * P.by * bx);
                    const float4 t = *ip;
                    if (t.x != 0.f || t.y != 0.f || t.z != 0.f || t.w != 0.f) {
                        // lower u^{m+1} by c r / (dx^3 g): the step adds c g r / dx^3
                        const float r[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
                        for (int e = 0; e < 4; e++)
                            if (r[e] != 0.f)
                                up[p & 1].v[e] +=
                                    -cc[p & 1].v[e] * r[e] * A.inv_dx3 / (gxy.v[e] * gzv);
                        if (OFF && scatter)
                            st_plain4(A.scatter[i & 1] + o + p * plane, zero4());
                        else
                            *ip = make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                }
                F4 out;
#pragma unroll
                for (int e = 0; e < 4; e++) {
                    const float g = gxy.v[e] * gzv;
                    out.v[e] = g * fmaf(cc[p & 1].v[e], lap.v[e], 2.0f * qc.v[e]) -
                               (g * g) * up[p & 1].v[e];
                }
                F4 s_now, a_now;
                if constexpr (BWD) {
                    s_now = sv[p & 1];
                    a_now = av[p & 1];
                }
                if (p + 2 < PZ) fetch(p + 2);
                st_plain4(prev + o + p * plane, out);
                if constexpr (BWD) {
                    if (A.grad) {
                        if (src_here && n < A.nt && z + p == srz) {
                            // the source term of the gradient
#pragma unroll
                            for (int e = 0; e < 4; e++)
                                if (x + e == srx)
                                    a_now.v[e] += qc.v[e] * A.wav[n] * A.inv_dx3 /
                                                  (gxy.v[e] * gzv);
                        }
                        F4 acc;
#pragma unroll
                        for (int e = 0; e < 4; e++)
                            acc.v[e] = fmaf(out.v[e], s_now.v[e], a_now.v[e]);
                        st_plain4(A.acc + o + p * plane, acc);
                    } else if (snap && in_model(p)) {
                        F4 acc;
#pragma unroll
                        for (int e = 0; e < 4; e++)
                            acc.v[e] = fmaf(s_now.v[e], out.v[e], a_now.v[e]);
                        st_plain4(A.acc + so + p * slab_plane, acc);
                        if (A.illum) {
                            float* ill = A.illum +
                                         ((size_t)(z + p - A.nb) * A.ny + (y - A.nb)) * A.nx;
#pragma unroll
                            for (int e = 0; e < 4; e++) {
                                const int mx = x + e - A.nb;
                                if (mx >= 0 && mx < A.nx)
                                    ill[mx] = fmaf(s_now.v[e], s_now.v[e], ill[mx]);
                            }
                        }
                    }
                } else {
                    if (snap) {
                        if (A.grad)
                            st_plain4(snap + o + p * plane, lap);
                        else if (in_model(p))
                            st_plain4(snap + so + p * slab_plane, out);
                    }
                }
            }
        }
        wait_here();  // a thread without cells
        const bool ok = *reinterpret_cast<volatile int*>(&s_ok) != 0;
        if (!ok) return;  // the same in every thread: set before the phase completed
        if constexpr (!BWD) {
            // gather d[n-1] = u^n at the receivers
            if (A.band && n >= 1 && n <= A.band_last) {
                // the model region's boundary band of u^n
                float* band = A.band + (long long)(n - 1) * A.band_stride;
                for (long long e = j0; e < A.band_stride; e += gridDim.x * T) {
                    int mx, my, mz;
                    band_cell_as<unsigned>((unsigned)e, A.nx, A.ny, A.nz, R, mx, my, mz);
                    band[e] = __ldcg(cur + (size_t)(mz + A.nb) * plane +
                                     (size_t)(my + A.nb) * A.NX + (mx + A.nb));
                }
            }
            if (A.data && n >= 1) {
                float* row = A.data + (size_t)(n - 1) * A.nrec;
                if constexpr (OFF) {
                    const int lane = tid & 31;
                    for (int k = tid >> 5; k < my_recs; k += T >> 5) {
                        // a lane's columns of the box, their z taps in flight together
                        const rtm_point_taps& t = table(k);
                        const int n0 = t.nx, nxy = taps_of(t) ? t.nx * t.ny : 0;
                        float sum = 0.f;
#pragma unroll 2
                        for (int q = lane; q < nxy; q += 32) {
                            const int tb = q / n0, ta = q - tb * n0;
                            const int x = t.i0 + ta, y = t.j0 + tb;
                            const bool in = x >= 0 && x < A.NX && y >= 0 && y < A.NY;
                            const float* src =
                                cur + (long long)t.k0 * (long long)plane + (long long)y * A.NX + x;
                            float u[8];
#pragma unroll
                            for (int c = 0; c < 8; c++)
                                u[c] = in && c < t.nz && t.k0 + c >= 0 && t.k0 + c < A.NZ
                                           ? __ldcg(src + c * plane)
                                           : 0.f;
                            const float wxy = t.wx[ta] * t.wy[tb];
#pragma unroll
                            for (int c = 0; c < 8; c++)
                                if (c < t.nz) sum += wxy * t.wz[c] * u[c];
                        }
                        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                        if (lane == 0) row[blockIdx.x + k * gridDim.x] = sum;
                    }
                } else {
                    if (j0 < A.nrec) row[j0] = d0;
                    for (int j = j0 + gridDim.x * T; j < A.nrec; j += gridDim.x * T) {
                        const int x = A.rec[3 * j] + A.nb, y = A.rec[3 * j + 1] + A.nb,
                                  z = A.rec[3 * j + 2] + A.nb;
                        row[j] = rec_outside<OFF>(A, j)
                                     ? 0.f
                                     : __ldcg(cur + (size_t)z * plane + (size_t)y * A.NX + x);
                    }
                }
            }
        } else {
            if (A.src_adj && n < A.nt && blockIdx.x == 0 && tid == 0)
                A.src_adj[n] = __ldcg(cur + A.src) / (A.gx[srx] * A.gy[sry] * A.gz[srz]);
        }
        if constexpr (OFF && BWD) {
            if (scatter && i + 1 < A.nsteps) scatter_taps(n - 1, A.scatter[(i + 1) & 1]);
        }
        if (i + 1 < A.nsteps) {
            __syncthreads();  // the box, the receiver terms and the block's writes are done with
            if (tid == 0) grid_arrive(A.ctrl);
            if constexpr (BWD) inject(n - 1);
        }
    }
}

// the data of a span's first step, as scatter_taps does for the others
__global__ void k_scatter_first(const __grid_constant__ SpanArgs A) {
    const int j = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (j >= A.nrec) return;
    const float r = A.rdata[(size_t)(A.first - 1) * A.nrec + j];
    for_taps(A.taps[1 + j], threadIdx.x & 31, [&](int x, int y, int z, float w) {
        if (x >= 0 && x < A.NX && y >= 0 && y < A.NY && z >= 0 && z < A.NZ)
            atomicAdd(A.scatter[0] + ((size_t)z * A.NY + y) * A.NX + x, w * r);
    });
}

cudaError_t encode_box(CUtensorMap* m, const float* base, const SpanArgs& a, int R) {
    EncodeTiledFn f = tma_encoder();
    if (!f) return cudaErrorNotSupported;
    const cuuint64_t dims[3] = {(cuuint64_t)a.NX, (cuuint64_t)a.NY, (cuuint64_t)a.NZ};
    const cuuint64_t strides[2] = {(cuuint64_t)a.NX * 4, (cuuint64_t)a.NX * a.NY * 4};
    const cuuint32_t b[3] = {(cuuint32_t)(4 * a.P.bxv + 2 * R), (cuuint32_t)(a.P.by + 2 * R),
                             (cuuint32_t)(a.P.bz + 2 * R)};
    const cuuint32_t estr[3] = {1, 1, 1};
    const CUresult r = f(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(base), dims,
                         strides, b, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <int R, bool BWD, int PZ, bool OFF>
cudaError_t launch_span_t(const SpanArgs& a, cudaStream_t s) {
    const auto kernel = k_span<R, BWD, PZ, OFF>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kSmemMax - 1024);
    if (e != cudaSuccess) return e;
    if (OFF && BWD && a.scatter[0] && a.nrec > 0) {
        const size_t bytes = sizeof(float) * a.NX * a.NY * a.NZ;
        for (int i = 0; i < 2; i++)
            if ((e = cudaMemsetAsync(a.scatter[i], 0, bytes, s)) != cudaSuccess) return e;
        k_scatter_first<<<(a.nrec + 7) / 8, 256, 0, s>>>(a);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    SpanMaps M;
    memset(&M, 0, sizeof M);
    for (int i = 0; i < 2; i++)
        if ((e = encode_box(&M.u[i], a.f[i], a, R)) != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.P.nbricks);
    // off the grid the block's warps share its receivers too: a small brick's
    // cells alone would leave them to one or two warps
    cfg.blockDim = dim3(OFF ? span_threads<R, BWD, PZ>() : a.P.threads);
    cfg.dynamicSmemBytes = a.P.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, a, M);
}

template <int R, bool BWD>
cudaError_t launch_span_r(const SpanArgs& a, cudaStream_t s) {
    if (a.taps)
        return a.P.pz == 1 ? launch_span_t<R, BWD, 1, true>(a, s)
                           : launch_span_t<R, BWD, kColumn, true>(a, s);
    return a.P.pz == 1 ? launch_span_t<R, BWD, 1, false>(a, s)
                       : launch_span_t<R, BWD, kColumn, false>(a, s);
}

template <class F>
F driver_entry(const char* name, unsigned int version) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    return cudaGetDriverEntryPointByVersion(name, &p, version, cudaEnableDefault, &q) == cudaSuccess &&
                   q == cudaDriverEntryPointSuccess
               ? reinterpret_cast<F>(p)
               : nullptr;
}

}  // namespace

// Blocks of a span wait for one another, so all of them have to be resident: a
// stream of a green context runs on that context's SMs only
int span_sms(cudaStream_t stream) {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    // (the second version of the call, with the green context)
    static const auto contexts_of =
        driver_entry<CUresult (*)(CUstream, CUcontext*, CUgreenCtx*)>("cuStreamGetCtx", 12050);
    static const auto resource_of =
        driver_entry<CUresult (*)(CUgreenCtx, CUdevResource*, CUdevResourceType)>(
            "cuGreenCtxGetDevResource", 12040);
    if (!contexts_of || !resource_of) return n;  // a driver without green contexts
    CUcontext ctx = nullptr;
    CUgreenCtx green = nullptr;
    // fails for the per-thread default stream of a green context
    if (contexts_of(stream, &ctx, &green) != CUDA_SUCCESS) return 0;
    if (green) {
        CUdevResource r;
        memset(&r, 0, sizeof r);
        if (resource_of(green, &r, CU_DEV_RESOURCE_TYPE_SM) != CUDA_SUCCESS) return 0;
        n = std::min(n, (int)r.sm.smCount);
    }
    return n;
}

// wavefronts per 8 lanes of a 16-byte shared-memory load whose lanes run over
// rows of bxv vectors in a box of row stride bxv + R / 2 vectors (1: no conflict)
static double conflicts(int bxv, int R) {
    const int stride = bxv + R / 2;
    int total = 0;
    for (int g = 0; g < bxv; g++) {  // the pattern repeats after bxv groups of 8
        int hits[8] = {0}, most = 0;
        for (int l = 0; l < 8; l++) {
            const int t = 8 * g + l;
            most = std::max(most, ++hits[(t / bxv * stride + t % bxv) % 8]);
        }
        total += most;
    }
    return (double)total / bxv;
}

SpanPlan span_plan(int R, int NX, int NY, int NZ, int backward, int sms) {
    SpanPlan best;
    const long long N = (long long)NX * NY * NZ;
    // a brick's box has to fit the shared memory of one SM
    if (!tma_available() || sms < 1 || N > (long long)sms * (kSmemMax / 4)) return best;
    struct Key {
        int r, nx, ny, nz, b, sms;
    };
    static thread_local Key key[8];
    static thread_local SpanPlan val[8];
    static thread_local int used = 0, next = 0;
    for (int i = 0; i < used; i++)
        if (key[i].r == R && key[i].nx == NX && key[i].ny == NY && key[i].nz == NZ &&
            key[i].b == backward && key[i].sms == sms)
            return val[i];
    double best_cost = 1e30;
    for (int pz = 1; pz <= kColumn; pz += kColumn - 1) {
        const int T = pz == 1 || R == 4 ? 512 : 384;
        int last_x = 0;
        for (int kx = 1; kx <= 64; kx++) {
            const int bxv = (NX / 4 + kx - 1) / kx;
            if (bxv == last_x || 4 * bxv + 2 * R > 256) continue;
            last_x = bxv;
            const int nbx = (NX / 4 + bxv - 1) / bxv;
            const double conflict = conflicts(bxv, R);
            int last_y = 0;
            for (int ky = 1; ky <= 64; ky++) {
                const int by = (NY + ky - 1) / ky;
                if (by == last_y || by + 2 * R > 256) continue;
                last_y = by;
                const int nby = (NY + by - 1) / by;
                if (nbx * nby > sms) break;
                int last_z = 0;
                for (int kz = 1; kz <= 64; kz++) {
                    const int bz = ((NZ + kz - 1) / kz + pz - 1) / pz * pz;
                    if (bz == last_z || bz + 2 * R > 256) continue;
                    last_z = bz;
                    const int nbricks = nbx * nby * ((NZ + bz - 1) / bz);
                    if (nbricks > sms) break;  // one brick per SM
                    const long long box = (long long)(4 * bxv + 2 * R) * (by + 2 * R) * (bz + 2 * R);
                    const long long smem = (box + 31) / 32 * 128 +
                                           (backward ? 16LL * bxv * by * bz + 4 * kSpanListCap
                                                     : (long long)sizeof(rtm_point_taps) * kTapCap) +
                                           128;
                    if (smem > kSmemMax - 1024) continue;
                    const int items = bxv * by * (bz / pz);
                    const int rounds = (items + T - 1) / T;
                    // clocks per brick: the copy; the items' shared-memory
                    // wavefronts or instructions behind one item's latency
                    const double copy = 1200 + box * 4.0 / 40.0;
                    const double warps = (items + 31) / 32;
                    const double loads = pz == 1 ? 4 * R + 1 + R / 2 : 4 * (2 * R + R / 2) + 4 + 2 * R;
                    const double math = rounds * (pz == 1 ? 1000.0 : 2500.0) +
                                        warps * std::max(loads * 4 * conflict,
                                                         (pz == 1 ? 350.0 : 1000.0) * R / 4 / 3);
                    const double cost = copy + math;
                    if (cost < best_cost) {
                        best_cost = cost;
                        best = SpanPlan{1, pz, bxv, by, bz, nbx, nby, nbricks,
                                        std::min(T, (items + 31) / 32 * 32), (int)smem};
                    }
                }
            }
        }
    }
    const int slot = used < 8 ? used++ : (next = (next + 1) % 8);
    key[slot] = Key{R, NX, NY, NZ, backward, sms};
    val[slot] = best;
    return best;
}

cudaError_t launch_span(SpanArgs a, cudaStream_t s) {
    if (!a.P.ok || a.nsteps < 1) return cudaErrorInvalidValue;
    a.stall = -1;
    a.limit_ns = kBarrierNs;
    if (a.nsteps > 1) {
        const int stall = take_test_stall(RTM_STALL_SPAN);
        if (stall >= 0) {
            a.stall = std::max(1, a.nsteps - 1 - stall);
            a.limit_ns = kWaitNs;
        }
    }
    if (a.radius == 4) return a.backward ? launch_span_r<4, true>(a, s) : launch_span_r<4, false>(a, s);
    if (a.radius == 8) return a.backward ? launch_span_r<8, true>(a, s) : launch_span_r<8, false>(a, s);
    return cudaErrorInvalidValue;
}

}  // namespace rtm
