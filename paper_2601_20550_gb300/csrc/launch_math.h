// Arithmetic of the kernels' indexes and of their launches, in plain C++ so that the host
// tests compile and run the same code.
#pragma once

#include <algorithm>
#include <cstdint>
#include <map>
#include <stdexcept>
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

// Blocks of a launch along x.
constexpr int64_t kMaxBlocks = 0x7fffffff;

inline unsigned grid_blocks(int64_t blocks) {
  if (blocks < 0 || blocks > kMaxBlocks) throw std::invalid_argument("too many work items for one launch");
  return (unsigned)blocks;
}

// Items that one launch takes of the rest, at per_item blocks each.
inline int64_t launch_share(int64_t rest, int per_item) { return std::min(rest, kMaxBlocks / per_item); }

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
