// A workspace whose size is a choice: the largest of several sizes that the allocator grants (host logic
// only, no CUDA types, so it also builds in a plain C++ test).
#pragma once

#include <cstddef>

namespace qf {

// Tries sizes[0 .. count) in turn (largest first) with alloc(size) while it fails with `oom`; any other result
// ends the search.  *taken: the size granted, 0 if none.  Returns the last result.
template <class Error, class Alloc>
Error alloc_largest(const size_t* sizes, int count, Error oom, Alloc alloc, size_t* taken) {
  *taken = 0;
  Error e = oom;
  for (int i = 0; i < count && e == oom; ++i) {
    if (i > 0 && sizes[i] >= sizes[i - 1]) continue;  // no smaller than what was refused
    e = alloc(sizes[i]);
    if (e != oom) *taken = sizes[i];
  }
  return e;
}

}  // namespace qf
