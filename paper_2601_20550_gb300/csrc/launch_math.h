// Index arithmetic of the kernels and their launches that has no place for 32 bits, in plain
// C++ so that the host tests compile and run the same code.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define HEOM_HD __host__ __device__ __forceinline__
#else
#define HEOM_HD inline
#endif

namespace heom {

// First element of d x d matrix n of a state.  A branch may hold more than 2^31 elements
// (d = 64, 646646 ADOs: 42 GB).
HEOM_HD int64_t ado_offset(int64_t n, int d) { return n * ((int64_t)d * d); }

}  // namespace heom
