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

// Beside the digits a tile holds the magnitudes |x| 2^-E in bf16 as a slice of its own, OZ_MAG: one more MMA a block adds
// sum |a||b| of every output over all blocks (what it is for: oz.cuh).
constexpr int OZ_MAG = OZ_S, OZ_SLICES = OZ_S + 1;
constexpr int OZ_MMAS = OZ_LOW + OZ_S + 1;

struct OzMma {
  int a, b;      // A slice, first B slice
  int n, col;    // columns of the MMA (64 per B slice), first accumulator column
  bool first;    // the first of its accumulator in a block: it overwrites
  bool whole;    // of an accumulator that is kept from block to block
  int new_b;     // B slice that no earlier MMA of the block reads (-1: none)
};

// A slices in order of issue: 3, 2, 1, 0 (levels 0 .. 3), then 6, 5, 4, the magnitudes, 3, 2, 1, 0 (levels 4 .. 6)
constexpr int oz_mma_slice(int q) {
  return q < OZ_LOW ? OZ_LOW - 1 - q : q < OZ_S ? OZ_S + OZ_LOW - 1 - q : q == OZ_S ? OZ_MAG : OZ_MMAS - 1 - q;
}
constexpr OzMma oz_mma(int q) {
  const bool low = q < OZ_LOW;
  const int i = oz_mma_slice(q);
  if (i == OZ_MAG) return OzMma{OZ_MAG, OZ_MAG, OZ_COLS, OZ_COLS * OZ_S, false, true, OZ_MAG};
  const int l0 = low ? 0 : OZ_LOW, l1 = low ? OZ_LOW : OZ_S, top = l1 - 1 - i;
  return OzMma{i, l0 - i, OZ_COLS * (l1 - l0), OZ_COLS * l0, top == 0, false, low || top >= OZ_LOW ? top : -1};
}

// Place of an A slice in the order of first use (3, 2, 1, 0, 6, 5, 4, magnitudes).  The A slices of a block sit in OZ_RING
// slots, each until its last MMA of the block (the second group's, the magnitudes'); the first four are held meanwhile, the
// others pass through.  A block's first four take the slots that the block before gives up first, those of its
// passing slices: slot = place, with its halves exchanged in every other block.
constexpr int OZ_RING = OZ_SLICES;
constexpr int oz_place(int i) { return i < OZ_LOW ? OZ_LOW - 1 - i : i < OZ_S ? OZ_LOW + OZ_S - 1 - i : OZ_MAG; }
constexpr int oz_slot(int block, int place) { return place ^ ((block & 1) * OZ_LOW); }

// Copies of a block in the order in which the block before gives up their places: A slice a, or B slice b.  A B slice
// follows the A slice whose slot the same MMA gave up, so that waiting for it is enough for both.
struct OzLoad {
  int a, b;   // one of them, the other is -1
};
constexpr int OZ_LOADS = 2 * OZ_SLICES;
constexpr OzLoad oz_load(int o) {
  constexpr int B = 16;
  constexpr int order[OZ_LOADS] = {3, 2, 1, B + 0, 0, B + OZ_MAG, 6, B + 1, 5, B + 2, 4, B + 3, OZ_MAG, B + 4, B + 5, B + 6};
  return order[o] < B ? OzLoad{order[o], -1} : OzLoad{-1, order[o] - B};
}

}  // namespace fetirp
