// Host-side rules that need neither CUDA nor a GPU (plain C++, tested by themselves).
#pragma once

#include <cstddef>
#include <cstdint>

namespace fastav {

// [at, at + bytes) lies inside the range of `size` bytes that starts at `start`.
inline bool inside_range(uintptr_t at, size_t bytes, uintptr_t start, size_t size) {
  return at >= start && bytes <= size && at - start <= size - bytes;
}

}  // namespace fastav
