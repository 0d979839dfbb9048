// A span: consecutive time steps of one recursion in a single cooperative
// launch (span.cu), for padded grids small enough that a step's fields stay
// in the L2 cache.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "rtm_internal.h"

namespace rtm {

// words of a span launch in the workspace's status block; zero before the
// first span of a call, `count` runs on over the spans of that call
struct SpanCtrl {
    unsigned int count;  // arrivals at the grid barrier
    int abort;           // a bounded wait ran out: every block leaves
};
constexpr size_t kSpanCtrlOffset = 64;  // bytes into the status block

// tiling of a padded grid into bricks, one block (and SM) per brick
struct SpanPlan {
    int ok = 0;
    int pz = 0;                       // planes per thread
    int bxv = 0, by = 0, bz = 0;      // brick: bxv vectors of 4 x points, rows, planes (pz | bz)
    int nbx = 0, nby = 0, nbricks = 0;
    int threads = 0, smem = 0;
};

// receivers of a brick that its block keeps in shared memory in a backward span;
// over them every step looks at all receivers
constexpr int kSpanListCap = 2048;

struct SpanArgs {
    SpanPlan P;
    const float *c, *gx, *gy, *gz, *wav;
    float* f[2];         // step i reads f[1 - (i & 1)] as u^n, f[i & 1] holds u^{n-1} -> u^{n+1}
    int NX, NY, NZ, nb, nx, ny, nz;
    int radius, backward, grad;
    int first, nsteps;   // forward: steps n = first, first + 1, ..; backward: m = first, first - 1, ..
    int nt;
    // source and receivers: point receivers or a tap table
    const int32_t* rec;
    const rtm_point_taps* taps;
    int nrec;
    long long src;
    float inv_dx3;
    float* data;         // forward: d[n-1] = u^n at the receivers (n >= 1), or NULL
    const float* rdata;  // backward: rows injected at the receivers
    float* scatter[2];   // backward, tap table: padded fields of scratch, or NULL
    float* src_adj;      // backward: trace at the source, or NULL
    // snapshot of state k (k = n + 1 forward, m backward): written or imaged
    // with where k % every == 0, at snap + (k / div - off) * stride; NULL: none
    float* snap;
    long long snap_stride;
    int every, div, off;
    float* acc;          // backward: image slab or gradient accumulator
    float* illum;        // backward: source illumination on the model grid, or NULL
    // forward: boundary band of the states 1 .. band_last (band_stride cells
    // each, gathered by the step that reads the state), or NULL
    float* band;
    long long band_stride;
    int band_last;
    float a[kMaxRadius + 1];
    SpanCtrl* ctrl;
    unsigned int base;   // ctrl->count before this launch
    int stall;           // step whose wait for the other blocks a test lets run out, or -1
    unsigned long long limit_ns;  // bound of that wait in every step
    int* status;
};

// SMs that work of this stream runs on (0: unknown, no spans)
int span_sms(cudaStream_t stream);
// the tiling for a padded grid over `sms` SMs, or ok = 0 where the plain launches are used
SpanPlan span_plan(int radius, int NX, int NY, int NZ, int backward, int sms);
// barriers of a launch: what ctrl->count grows by is P.nbricks * (nsteps - 1)
cudaError_t launch_span(SpanArgs a, cudaStream_t s);

}  // namespace rtm
