// The grid and what code shared with the host tests needs.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define DMS_HD __host__ __device__ __forceinline__
#else
#define DMS_HD inline
#endif

namespace dms {

struct Grid {
  int64_t nx, ny, nz, n;
  int64_t sxy;  // nx*ny
};

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
