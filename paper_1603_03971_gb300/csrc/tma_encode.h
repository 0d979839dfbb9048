// The driver's tensor-map encoder (cuTensorMapEncodeTiled), looked up once
// through the runtime's driver entry-point query so that librtm does not link
// libcuda directly. NULL when the driver does not provide it.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

namespace rtm {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn tma_encoder();
// map of a dense float32 [nz][ny][nx] array with boxes of by rows of bx, kept
// per thread by its arguments
cudaError_t tma_map3(CUtensorMap* m, const float* base, int nx, int ny, int nz, int bx, int by);

}  // namespace rtm
