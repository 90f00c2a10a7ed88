// How the wide chain kernel (widechain.cuh) cuts up a chain.  Host arithmetic only.
#pragma once

namespace csd {

constexpr int kWcRows = 256;              // rows of a slot

// Whether the wide chain kernel is the faster one for a head of L blocks and so many head rows.  Time over that of the layer kernels, chain
// alone | round of two equal heads, with guidance, 20 steps (100 steps: 0.05 to 0.1 less):
//   few rows, where a second slot is nearly empty      258: 2 x 768 1.02 | 0.84, 4 x 1024 0.97 | 0.85, 4 x 1280 0.91 | 1.00, 8 x 1536 0.99 | 1.21,
//                                                      8 x 2048 1.00 | 1.25 (100 steps 1.00 and 1.02); 514: 0.90 | 0.95, 0.78 | 0.95.  Taken all the
//                                                      same: beside a narrower head in this kernel it is the better one (272 rows of 6 x 1024 and
//                                                      12 x 1536, 100 steps, ms a round: 26.8; the target in layer kernels 31.4, both 29.4)
//   one block, where a step is mostly its projections  512: 1 x 768 1.30 | 0.81, 1 x 1024 1.23 | 0.91; 1024: 1.12 | 0.72, 1.00 | 0.78; 384 of 1 x 1280 1.04 | 0.89
//   many rows, whose tiles fill the GPU in waves       2560: 4 x 1280 0.79 | 0.81, 4 x 1536 0.86 | 0.86, 4 x 1792 0.90 | 0.83, 4 x 2048 0.92 | 0.98;
//                                                      3400: 1.01 | 0.94, 1.03 | 1.02, 1.03 | 1.03, 1.02 | 1.04; 4608: 4 x 768 0.86 | 0.89, 4 x 1024 0.98 | 0.97
// Beyond the last line a step's products alone are up to 1 GB, for no gain.
inline bool wide_pays(int L, int W, int rows) {
  if (rows <= kWcRows || rows > 4608) return false;
  return (L > 1 || rows * W >= 1 << 19) && rows * W <= 4750000;
}

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
