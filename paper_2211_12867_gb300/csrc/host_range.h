// Which host memory a kernel may write over the link.
#pragma once
#include <cstddef>
#include <cstdint>

// A piece of page-locked memory: [start, start + bytes), at the same addresses
// on the device or not.
struct PinnedPiece {
  uintptr_t start = 0;
  size_t bytes = 0;
  bool same_address = false;
};

// True if page-locked pieces cover [p, p + bytes) without a gap and the device
// sees all of them at their host addresses.  piece(q, &out) finds the piece
// that holds q, if any: looking at both ends alone would take two registered
// pieces with pageable memory between them for one.
template <typename Find>
bool pinned_throughout(uintptr_t p, size_t bytes, Find piece) {
  const uintptr_t end = p + bytes;
  while (p < end) {
    PinnedPiece q;
    if (!piece(p, &q) || !q.same_address || q.start > p || q.start + q.bytes <= p) return false;
    p = q.start + q.bytes;
  }
  return true;
}
