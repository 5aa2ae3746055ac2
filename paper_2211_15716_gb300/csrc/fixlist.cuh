// The list of points that the kernels of the emulated FP64 cell leave to the
// fix-up launch (tma.cu: k_fixup_f64): layout and the entries a warp stages.
#pragma once

#include <cstddef>

namespace igg {
namespace {

// A tile set's fix-up buffer (layout in igg_internal.h): the entries, then
// the entry count and a block counter.
struct FixEntry {
  long long p;    // index of the first of 32 consecutive points of a row
  unsigned bits;  // bit l: point p + l left to the fix-up
  unsigned pad;
};
// Entries a consumer warp stages in shared memory before it reserves their
// slots in the list with one atomic (a warp waits for each atomic's return:
// with 16 entries twenty steps of 2x2x2 x 256x128x128, modes up to 8 about 0,
// took 11.91 ms, with 32, as many as one store of the warp appends, 11.87; ten
// steps of 2x2x2 x 512x256x256, smooth, 10.35 and 10.33).
constexpr unsigned kFixPend = 32;
struct FixList {
  FixEntry *e;
  unsigned *count, *done;
  unsigned long long *totals;  // segments and points fixed up since the buffer was made
};
__device__ __forceinline__ FixList fix_list(void *fix, size_t cap) {
  FixEntry *e = reinterpret_cast<FixEntry *>(fix);
  unsigned *c = reinterpret_cast<unsigned *>(e + cap);
  return {e, c, c + 1, reinterpret_cast<unsigned long long *>(c + 2)};
}

}  // namespace
}  // namespace igg
