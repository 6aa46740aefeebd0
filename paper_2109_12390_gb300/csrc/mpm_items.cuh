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
  // work items small enough that every SM has about two (an item's latency, not its work, sets the
  // time of a small context): 84,915 plastic particles in 3D, 20 steps with the state's load and read,
  // 1104 us with items of 512, 896 with 288 (two full halves of a 4^3-cell block; 1.2x more with 192)
  // together with the rotations that the return mapping hands on
  const long long two = (P + 2ll * n_sm - 1) / (2ll * n_sm);
  const long long cap = (two + 31) / 32 * 32;
  r.cap = (int)(cap < kItemMin ? kItemMin : cap > kItem ? kItem : cap);
  return r;
}

}  // namespace mpmrom
