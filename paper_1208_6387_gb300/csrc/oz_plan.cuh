// The MMAs of one 64-wide block of a sliced FP64 product (oz.cuh).  Plain C++: checked on the host (tests/host/oz_plan.cpp).
#pragma once

namespace fetirp {

constexpr int OZ_S = 7, OZ_BITS = 9;
constexpr int OZ_COLS = 64;   // rows of B of a CTA: accumulator columns of a level

// The digit pairs (i, j) of A and B go by their level i + j into the OZ_S accumulators of 64 columns.  A slice i meets several
// consecutive B slices in one MMA, and MMAs of a block accumulate into the same columns.  Such MMAs are only sure to
// execute in the order of issue when they have the same accumulator and the same shape, so the levels form two groups, each
// one accumulator with one shape: 0 .. 3 (N = 256) and 4 .. 6 (N = 192).  Every A slice of a group multiplies as many B
// slices as the group has levels, the B slices -OZ_PAD .. -1 being zeros: 11 MMAs and 2368 columns a block, where shapes
// that shrink with i (on two halves of 32 columns, 14 MMAs) issue 1792 whose order nothing states.  The apply of oz.cu's
// comment took 1114 us with those; 1570 us with these in a loop whose every step cost the issuing thread some 1100 cycles
// of address arithmetic and counters, and 966 us with the loop unrolled and the counters gone.
// In a group i descends, so that the B slices are needed, and in the second group given up, from 0 on: the next block's are
// loaded into their place meanwhile.
constexpr int OZ_LOW = 4, OZ_PAD = 3;
constexpr int OZ_MMAS = OZ_LOW + OZ_S;

struct OzMma {
  int a, b;      // A slice, first B slice
  int n, col;    // columns of the MMA (64 per B slice), first accumulator column
  bool first;    // the first of its accumulator in a block: it overwrites
  int new_b;     // B slice that no earlier MMA of the block reads (-1: none)
};

// MMA q of a block, in order of issue
constexpr OzMma oz_mma(int q) {
  const bool low = q < OZ_LOW;
  const int i = low ? OZ_LOW - 1 - q : OZ_MMAS - 1 - q;
  const int l0 = low ? 0 : OZ_LOW, l1 = low ? OZ_LOW : OZ_S, top = l1 - 1 - i;
  return OzMma{i, l0 - i, OZ_COLS * (l1 - l0), OZ_COLS * l0, top == 0, low || top >= OZ_LOW ? top : -1};
}

// Place of A slice i in the order of first use (3, 2, 1, 0, 6, 5, 4).  The A slices of a block sit in OZ_RING slots, each until
// the second group's MMA of its slice; the first four are held meanwhile, the others pass through.  A block's first four
// take the slots that the block before gives up first, those of its passing slices: slot = place, with its halves
// exchanged in every other block.  use: how often the slot was used before.
constexpr int OZ_RING = 8;
constexpr int oz_place(int i) { return i < OZ_LOW ? OZ_LOW - 1 - i : OZ_LOW + OZ_S - 1 - i; }
constexpr int oz_slot(int block, int place) { return place ^ ((block & 1) * OZ_LOW); }
constexpr int oz_use(int block, int i) { return oz_place(i) == OZ_LOW - 1 ? block >> 1 : block; }   // seven places of eight

// Copies of a block in the order in which the block before gives up their places: A slice a, or B slice b.  B slices 0 to 3
// follow the A slice whose slot the same MMA gave up, so that waiting for it is enough for them as well.
struct OzLoad {
  int a, b;   // one of them, the other is -1
};
constexpr int OZ_LOADS = 2 * OZ_S;
constexpr OzLoad oz_load(int o) {
  if (o < OZ_LOW) return OzLoad{OZ_LOW - 1 - o, -1};
  if (o >= OZ_LOADS - OZ_LOW) return OzLoad{-1, o - (OZ_LOADS - OZ_S)};
  return (o - OZ_LOW) % 2 ? OzLoad{OZ_S - 1 - (o - OZ_LOW) / 2, -1} : OzLoad{-1, (o - OZ_LOW) / 2};
}

}  // namespace fetirp
