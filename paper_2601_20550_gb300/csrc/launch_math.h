// Arithmetic of the kernels' indexes and of their launches, in plain C++ so that the host
// tests compile and run the same code.
#pragma once

#include <algorithm>
#include <cstdint>
#include <map>
#include <utility>
#include <vector>

#ifdef __CUDACC__
#define HEOM_HD __host__ __device__ __forceinline__
#else
#define HEOM_HD inline
#endif

namespace heom {

// First element of d x d matrix n of a state.  A branch may hold more than 2^31 elements
// (d = 64, 646646 ADOs: 42 GB).
HEOM_HD int64_t ado_offset(int64_t n, int d) { return n * ((int64_t)d * d); }

// Launch shapes (threads per block, blocks) kept per (kernel kind, elements).
using Shape = std::pair<int, int>;
using ShapeMap = std::map<std::pair<int, int64_t>, Shape>;

// The kept shape, if it is one of this kernel's: kernels of one kind (a launch for all steps,
// a launch per stage) record theirs under the same key.  nullptr: none.
inline const Shape *kept_shape(const ShapeMap &kept, int kind, int64_t total, const Shape &dflt,
                               const std::vector<Shape> &candidates) {
  const auto it = kept.find({kind, total});
  if (it == kept.end()) return nullptr;
  const bool ours = it->second == dflt || std::find(candidates.begin(), candidates.end(), it->second) != candidates.end();
  return ours ? &it->second : nullptr;
}

}  // namespace heom
