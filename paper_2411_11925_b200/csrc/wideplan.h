// How the wide chain kernel (widechain.cuh) cuts up a chain.  Host arithmetic only.
#pragma once

namespace csd {

constexpr int kWcRows = 256;              // rows of a slot

// Groups of W / 128 CTA pairs that a device holds at a time, of `pairs` pairs.
inline int wide_groups(int pairs, int W) { return pairs / (W / 128); }

// Row blocks (an even number) and slots of R token rows; the form of the kernel (halves 1: two slots a group, 2: one slot with
// twice the epilogue warps); slots of a launch (a part of the rows where not all of a launch's CTAs would find an SM), its CTAs.
struct WideCut { int nb, slots, part, ctas, halves; };
// most: groups that the device holds at a time, at least 1.
inline WideCut wide_cut(int most, int W, int R, int cfg, int halves) {
  WideCut c{};
  const int nb = cfg ? (R + 63) / 64 : (R + 127) / 128, group = 2 * (W / 128), gs = 2 / halves;
  c.nb = nb + (nb & 1); c.slots = c.nb / 2; c.halves = halves;
  const int groups = (c.slots + gs - 1) / gs, parts = (groups + most - 1) / most;
  c.part = ((c.slots + parts - 1) / parts + gs - 1) / gs * gs;
  c.ctas = ((c.part < c.slots ? c.part : c.slots) + gs - 1) / gs * group;
  return c;
}

}  // namespace csd
