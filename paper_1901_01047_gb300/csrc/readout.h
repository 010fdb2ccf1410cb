// readout.h -- device buffers that a read-out makes at its first call and keeps.
#pragma once
#include <cstddef>
#include <initializer_list>

namespace dca {

struct ReadoutPiece {
  void** dst;
  size_t bytes;
};

// One allocation cut into 256-byte aligned pieces, and whether what is filled in
// once is there.  A call that fails on the way leaves no pointer that a later
// call would take for a complete set: that one starts where this one failed.
struct ReadoutBuffers {
  char* base = nullptr;
  bool ready = false;

  // alloc(bytes) -> void* (null: no memory), fill() -> int (0: done).
  // Returns 0, the code of fill(), or no_memory.
  template <typename Alloc, typename Fill>
  int prepare(std::initializer_list<ReadoutPiece> pieces, int no_memory, Alloc alloc, Fill fill) {
    if (ready) return 0;
    auto up = [](size_t b) { return (b + 255) / 256 * 256; };
    if (!base) {
      size_t total = 0;
      for (const ReadoutPiece& p : pieces) total += up(p.bytes);
      base = static_cast<char*>(alloc(total));
      if (!base) return no_memory;
      size_t off = 0;
      for (const ReadoutPiece& p : pieces) {
        *p.dst = base + off;
        off += up(p.bytes);
      }
    }
    const int rc = fill();
    ready = rc == 0;
    return rc;
  }
};

}  // namespace dca
