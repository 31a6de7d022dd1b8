// Which of a context's optional scratch is taken (host only).
#pragma once

#include <cstddef>

namespace rec {

// Scratch that only saves time, in the order in which it is given up: the
// coefficient cache of the FP64 form first, then the compact velocity copy (a
// tenth of its size, and what the march gains most from).
enum ScratchLevel { kScratchLeast = 0, kScratchCopy = 1, kScratchAll = 2 };

// Up to 256 MB is taken without asking; more only where it is at most an eighth
// of the free memory.  copy, cache: bytes of the two parts.
inline int scratch_level(size_t copy, size_t cache, size_t free_bytes) {
  const size_t small = (size_t)256 << 20;
  auto fits = [&](size_t bytes) { return bytes <= small || bytes <= free_bytes / 8; };
  if (!fits(copy)) return kScratchLeast;
  return fits(copy + cache) ? kScratchAll : kScratchCopy;
}

}  // namespace rec
