// A buffer that its user can do without.
#pragma once

#include <cstddef>

namespace fs {

// Mem::alloc(bytes) returns nullptr when it has none (and reports nothing),
// Mem::free(p) gives back what alloc returned.
template <class Mem>
struct OptionalBuf {
  void* p = nullptr;
  size_t bytes = 0;
  bool declined = false;  // the last request was refused: none is made until retry()
  // At least `want` bytes. A refusal leaves the buffer as it is, smaller or none.
  bool ensure(size_t want) {
    if (want <= bytes) return true;
    if (declined) return false;
    void* q = Mem::alloc(want);
    if (!q) {
      declined = true;
      return false;
    }
    release();
    p = q;
    bytes = want;
    return true;
  }
  void retry() { declined = false; }
  void release() {
    if (p) Mem::free(p);
    p = nullptr;
    bytes = 0;
  }
};

}  // namespace fs
