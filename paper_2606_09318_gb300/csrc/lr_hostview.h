// lr_hostview.h -- host buffers that kernels may read and write where they are.
#pragma once
#include <cstddef>

namespace lr {

// A piece of pinned memory around an address: what the device calls the
// address, and the bytes from there to the end of the allocation or
// registration.
struct PinnedPiece {
  void *device;
  size_t left;
};

// What the device calls `bytes` bytes from p on, if all of them are pinned and
// follow each other there too; null otherwise.  ask(q, piece) says whether q
// is pinned.  Every piece is asked for: two registrations may have pages
// between them that are not.
template <class Ask>
void *pinned_view(const void *p, size_t bytes, Ask &&ask) {
  const char *const from = static_cast<const char *>(p);
  char *first = nullptr;
  for (size_t at = 0; at < bytes;) {
    PinnedPiece piece;
    if (!ask(from + at, piece) || !piece.device || piece.left == 0) return nullptr;
    if (at == 0) first = static_cast<char *>(piece.device);
    if (static_cast<char *>(piece.device) != first + at) return nullptr;
    at = piece.left < bytes - at ? at + piece.left : bytes;
  }
  return first;
}

}  // namespace lr
