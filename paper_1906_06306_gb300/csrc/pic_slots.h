// The walk of a thread block over its share of a species' particle slots.
// Plain C++ apart from the qualifiers, so that the arithmetic at the upper end
// of the slot range can be checked on the host.
#pragma once

#ifdef __CUDACC__
#define PIC_HD __host__ __device__ __forceinline__
#else
#define PIC_HD inline
#endif

namespace pic {

// A particle slot.  Counts are below 2^31, but the last batch of a share runs
// up to a block's threads past its end: signed 32-bit indexes wrapped there.
typedef unsigned slot_t;

// The slots [a, b), taken in batches that begin at base, at or below a.
struct SlotWalk {
  slot_t a, b, base;
  PIC_HD bool more() const { return base < b; }
  PIC_HD void next(slot_t threads) { base += threads; }
  PIC_HD slot_t slot(slot_t thread) const { return base + thread; }
  PIC_HD bool mine(slot_t p) const { return p >= a && p < b; }
};

// Batches that begin at a; with `line`, on the 128-byte line of a where that
// takes no batch more; with `quad`, on the aligned quad of a (where any do).
PIC_HD SlotWalk slot_walk(slot_t a, slot_t b, slot_t threads, bool line, bool quad) {
  SlotWalk w = {a, b, a};
  if (quad && a < b) w.base = a & ~3u;
  if (line && a < b && (b - a - 1) / threads == (b - (a & ~31u) - 1) / threads) w.base = a & ~31u;
  return w;
}

}  // namespace pic
