// What a call allocates when it cannot have all it would like to: host code
// without CUDA, the allocations themselves are arguments.
#pragma once
#include <cstddef>
#include <cstdint>

namespace mtp {

// Memory that a call needs (`must` tries to allocate it), with memory it could
// do without already taken: where it does not fit beside that, `drop` gives the
// other memory back (false: there is none) and it is tried once more.
template <class Must, class Drop>
bool allocate_dropping(Must must, Drop drop) {
  if (must()) return true;
  return drop() && must();
}

}  // namespace mtp
