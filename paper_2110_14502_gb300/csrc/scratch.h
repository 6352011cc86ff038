// A grow-only scratch buffer, part of which its user can do without.
#pragma once

#include <cstddef>

namespace tn {

struct Scratch {
  void* p = nullptr;
  size_t bytes = 0;
  size_t refused = 0;  // a size that could not be had (0: none) ..
  int passed = 0;      // .. and the calls that have not asked for it since
};

// At least `need` bytes, and `want` (>= need) if they can be had; false: not even
// `need`, the buffer is then empty.  A buffer that holds `need` is kept when `want`
// cannot be had, and that size is asked for again only by every 64th call: a failed
// allocation, and giving up a buffer that recorded launches point to, cost far more
// than the wider buffer gains.  alloc(size) returns null on failure, release(p)
// waits for the device, replacing() is called before a buffer is released.
template <class Alloc, class Release, class Replacing>
bool reserve(Scratch& s, size_t need, size_t want, Alloc&& alloc, Release&& release, Replacing&& replacing) {
  if (s.bytes >= want) return true;
  const bool enough = s.bytes >= need;
  if (enough && s.refused && want >= s.refused && ++s.passed < 64) return true;
  auto take = [&](void* p, size_t bytes) {
    s.p = p;
    s.bytes = bytes;
    s.refused = 0;
    s.passed = 0;
  };
  auto drop = [&] {
    if (!s.p) return;
    replacing();
    release(s.p);
    s.p = nullptr;
    s.bytes = 0;
  };
  if (!enough) drop();
  if (void* p = alloc(want)) {
    drop();
    take(p, want);
    return true;
  }
  if (!enough) {
    void* p = want > need ? alloc(need) : nullptr;
    if (!p) return false;
    take(p, need);
  }
  s.refused = want;
  s.passed = 0;
  return true;
}

}  // namespace tn
