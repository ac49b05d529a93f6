// Host-only check of alloc_largest: the largest size that a fake allocator of limited memory grants, other
// errors passed on at once, and sizes no smaller than a refused one not tried again.  Exit status 0 on success.
#include <cstdio>

#include "../../paper_2606_04186_gb300/csrc/alloc_largest.h"

#define CHECK(c)                                         \
  do {                                                   \
    if (!(c)) {                                          \
      std::fprintf(stderr, "failed: %s (line %d)\n", #c, __LINE__); \
      return 1;                                          \
    }                                                    \
  } while (0)

enum Err { kOk, kOom, kOther };

int main() {
  const size_t sizes[3] = {700, 24, 20}, same[3] = {24, 24, 20};
  size_t got = 1;
  int calls = 0;
  auto with = [&](size_t room) {
    calls = 0;
    return [&calls, room](size_t n) {
      ++calls;
      return n <= room ? kOk : kOom;
    };
  };
  CHECK(qf::alloc_largest(sizes, 3, kOom, with(1000), &got) == kOk && got == 700 && calls == 1);
  CHECK(qf::alloc_largest(sizes, 3, kOom, with(699), &got) == kOk && got == 24 && calls == 2);
  CHECK(qf::alloc_largest(sizes, 3, kOom, with(20), &got) == kOk && got == 20 && calls == 3);
  CHECK(qf::alloc_largest(sizes, 3, kOom, with(19), &got) == kOom && got == 0 && calls == 3);
  CHECK(qf::alloc_largest(same, 3, kOom, with(20), &got) == kOk && got == 20 && calls == 2);
  calls = 0;
  CHECK(qf::alloc_largest(sizes, 3, kOom, [&](size_t) { ++calls; return kOther; }, &got) == kOther && calls == 1);
  std::puts("ok");
  return 0;
}
