// Bookkeeping of the staging arena: which bytes of the pinned host buffer may be written.
// (Plain C++, without CUDA, so that it can be tested on a host.)
#pragma once
#include <stddef.h>

namespace gbs {

// Each call stages from the arena's start, one region behind the other.  The copies out of
// it are asynchronous, and a call may end with some of them still queued (a sampler step's
// conditioning): those bytes are not written again before the stream has been waited for.
struct StageArena {
  size_t cap = 0, off = 0;
  size_t open = 0;                  // [open, off): queued by this call since the last wait
  size_t held_lo = 0, held_hi = 0;  // [held_lo, held_hi): queued by an earlier call and not waited for

  static size_t align(size_t x) { return (x + 255) / 256 * 256; }
  // A new call begins.  True: wait first (waited(), then begin() again).
  bool begin() {
    if (open < off) {
      if (held_lo < held_hi) return true;  // two calls' leftovers: no need to keep track of both
      held_lo = open;
      held_hi = off;
    }
    off = open = 0;
    return false;
  }
  size_t next() const { return align(off); }
  bool fits(size_t bytes) const { return next() + bytes <= cap; }
  // Whether the next `bytes` may be written at once; otherwise wait first.
  bool clear(size_t bytes) const { return held_lo >= held_hi || next() + bytes <= held_lo || next() >= held_hi; }
  // Takes the next `bytes`: their offset.
  size_t take(size_t bytes) {
    const size_t at = next();
    off = at + bytes;
    return at;
  }
  // Everything queued so far is done.
  void waited() {
    held_lo = held_hi = 0;
    open = off;
  }
};

}  // namespace gbs
