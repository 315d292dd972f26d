// cuTensorMapEncodeTiled through the runtime's driver entry point (the library does not link against the driver).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

namespace bcnn {

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                  const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled_fn();          // nullptr where the driver has none

}  // namespace bcnn
