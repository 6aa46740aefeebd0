// Sizes of the fused kernel's work items and CTAs from a context's size (host code, plain C++).
#pragma once

namespace mpmrom {

// The fused kernel takes up to kItem particles per work item, kItem / CH per thread, in CTAs of CH threads,
// 768 threads per SM.  3D: grid blocks of 4^3 cells at 8 particles per cell, 512 = 256 x 2.
constexpr int kItem = 512;
constexpr int kItemMin = 128;         // smallest bound of a work item (small contexts)

struct ItemRule {
  int cap;       // particles per work item at most
  bool narrow;   // 2D: CTAs of 128 threads
};

// 2D blocks of 8^2 cells at 4 per cell hold about 256 particles.  In CTAs of 128 threads twice as many items
// are in flight per SM (an item's phases are separated by barriers and dependent loads): 1.04 M particles in
// 16 bodies 68.8 -> 54.9 us a step, 212,000 22.7 -> 21.0.  That needs items enough: a block then takes two
// passes of 128 threads where one of 256 would do, and below about 768 particles per SM the wide CTAs are one
// wave anyway (one body of 75,000 particles 12.5 us a step in wide CTAs, 15.8 in narrow ones; 100,000 12.6 and
// 16.4; 115,000 16.3 and 17.1).  From 135,000 on 152 SMs the narrow ones were the faster in every shape
// measured: one body of 134,689 particles 18.2 -> 17.4, of 144,400 17.4 -> 16.8, 16 of 140,494 18.7 -> 17.4.
inline ItemRule item_rule(int dim, long long P, int n_sm) {
  ItemRule r{kItem, dim == 2 && P > 896ll * n_sm};
  // An item's latency, not its work, sets the time of a small context, so blocks are split over several items
  // there; but only while all items are resident at once (3 wide CTAs per SM), since one more wave costs what the
  // split gains.  With half a full block per item that holds while the halves fill no more than 7/8 of the places
  // (the rest is for blocks at the bodies' surfaces).
  const long long half = dim == 2 ? 128 : 256, places = 3ll * n_sm;
  if (8 * P > 7 * places * half) return r;
  if (dim == 2) {
    // Up to 128 particles per SM one item per block; past it 3/4 of a full block, so that one of a few particles
    // more than 256 is cut in two and not in three: one body of 9,680 particles 11.2 -> 10.9 us a step (bound 512
    // -> 256), five of 28,125 12.9 -> 11.5, one of 50,176 12.8 -> 12.2.
    r.cap = P > 128ll * n_sm ? 192 : 256;
  } else {
    // About two items per SM: 12,240 plastic particles 33 -> 24 us a step (bound 512 -> 128), 36,000 41 -> 24,
    // 84,915 48.8 -> 37.4.  Past the line above the same bound cost up to 14 %: 123,750 particles 26.2 -> 29.5,
    // 139,536 plastic ones 52.2 -> 60.5.
    const long long cap = ((P + 2ll * n_sm - 1) / (2ll * n_sm) + 31) / 32 * 32;
    r.cap = (int)(cap < kItemMin ? kItemMin : cap > kItem ? kItem : cap);
  }
  return r;
}

}  // namespace mpmrom
