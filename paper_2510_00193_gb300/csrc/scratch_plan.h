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

// Scratch of the split kernels (levels with component groups): the moments of
// `parts` shares of every atom's neighbours and the adjoints, with the atoms
// rounded up to whole tiles of 8; then, for the straight-line contraction, the
// values and adjoints of `graphs` graphs for whole blocks of 128 threads.
inline size_t split_scratch_bytes(int comps, int64_t n, int parts, size_t entry, int graphs) {
  return entry * ((size_t)comps * (size_t)((n + 7) / 8 * 8) * (size_t)(parts + 1) +
                  2 * (size_t)graphs * (size_t)((n + 127) / 128 * 128));
}

// How the split kernels run in the memory there is: fits(bytes) says whether
// (and sees to it that) the scratch has that size.  First without the graph
// values (the tile program contracts without them), then with one share.
struct SplitPlan {
  bool ok;       // false: not even the smallest fits
  int parts;
  bool graphs;
};
template <class Fits>
SplitPlan plan_split_scratch(int comps, int64_t n, int parts, size_t entry, int graphs, Fits fits) {
  if (graphs > 0 && fits(split_scratch_bytes(comps, n, parts, entry, graphs))) return {true, parts, true};
  if (fits(split_scratch_bytes(comps, n, parts, entry, 0))) return {true, parts, false};
  if (parts > 1 && fits(split_scratch_bytes(comps, n, 1, entry, 0))) return {true, 1, false};
  return {false, 0, false};
}

}  // namespace mtp
