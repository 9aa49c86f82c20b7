// What code that is compiled for the host as well needs of the grid.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#include "dms_common.cuh"
#define DMS_HD __host__ __device__ __forceinline__
#else
#define DMS_HD inline
namespace dms {
struct Grid {  // as in dms_common.cuh, which needs the CUDA headers
  int64_t nx, ny, nz, n;
  int64_t sxy;
};
}  // namespace dms
#endif

namespace dms {

// a load of what no one writes meanwhile
template <class T>
DMS_HD T ro(const T* p) {
#ifdef __CUDA_ARCH__
  return __ldg(p);
#else
  return *p;
#endif
}

}  // namespace dms
