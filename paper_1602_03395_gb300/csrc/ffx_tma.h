// The driver's tile-map encoder (cuTensorMapEncodeTiled), found through the
// runtime's driver entry point (no link against the driver library).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <cstring>

namespace ffx {

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// NULL if the driver does not offer it
inline EncodeTiledFn encode_tiled() {
  static const EncodeTiledFn fn = []() -> EncodeTiledFn {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    return reinterpret_cast<EncodeTiledFn>(p);
  }();
  return fn;
}

// Encode a tile map (no interleave, unit element strides, zeros past the ends);
// false if the driver cannot.  The encoder needs the device's context current
// on the calling thread, which a thread's first CUDA call alone makes so (an
// autograd worker's may be this one): on failure the device is set and the
// encoding tried once more.
inline bool make_tile_map(CUtensorMap* map, CUtensorMapDataType type, unsigned rank, const void* base,
                          const cuuint64_t* dims, const cuuint64_t* strides, const cuuint32_t* box,
                          CUtensorMapSwizzle swizzle) {
  std::memset(map, 0, sizeof(*map));
  const EncodeTiledFn enc = encode_tiled();
  if (!enc) return false;
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  for (int attempt = 0; attempt < 2; ++attempt) {
    if (enc(map, type, rank, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS)
      return true;
    int dev = 0;
    if (attempt || cudaGetDevice(&dev) != cudaSuccess || cudaSetDevice(dev) != cudaSuccess) break;
  }
  std::memset(map, 0, sizeof(*map));
  return false;
}

}  // namespace ffx
