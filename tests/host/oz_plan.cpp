// The MMAs and copies of a sliced FP64 product (csrc/oz_plan.cuh).  MMAs: every digit pair of the levels 0 .. OZ_S - 1 and the
// pair of magnitude slices exactly once and no other, nothing but zero slices read outside B, and two MMAs that accumulate into a common column have the
// same accumulator and the same shape (what makes their order certain).  Copies: played through for several blocks, a
// slot or slice is overwritten only after an MMA that the copying thread has waited for, later than its last reader; every
// MMA finds the slices of its own block; and a slot is used once a block, which the waits' parities count.
#include <cstdio>

#include "oz_plan.cuh"

using namespace fetirp;

int main() {
  int bad = 0, cols = 0;
  int times[OZ_SLICES][OZ_SLICES] = {};
  for (int q = 0; q < OZ_MMAS; ++q) {
    const OzMma x = oz_mma(q);
    cols += x.n;
    bad += x.n % OZ_COLS != 0 || x.n < OZ_COLS || x.n > 256 || x.col < 0 || x.col + x.n > 512;
    bad += x.b < -OZ_PAD || x.b + x.n / OZ_COLS > (x.whole ? OZ_SLICES : OZ_S) || x.whole != (x.a == OZ_MAG);
    for (int s = 0; s < x.n / OZ_COLS; ++s) {
      const int j = x.b + s, level = x.col / OZ_COLS + s;
      if (j < 0) continue;
      bad += x.whole ? level != OZ_S : x.a + j != level;
      ++times[x.a][j];
    }
    bool overlaps = false;
    for (int p = 0; p < q; ++p) {
      const OzMma y = oz_mma(p);
      const bool common = x.col < y.col + y.n && y.col < x.col + x.n;
      overlaps = overlaps || common;
      bad += common && (x.col != y.col || x.n != y.n);
    }
    bad += (x.first || x.whole) == overlaps;   // overwrites exactly when nothing of this block is there yet
  }
  for (int i = 0; i < OZ_SLICES; ++i)
    for (int j = 0; j < OZ_SLICES; ++j) bad += times[i][j] != (i + j < OZ_S || (i == OZ_MAG && j == OZ_MAG));

  // time of MMA q of block c: c * OZ_MMAS + q.  The copying thread knows the MMAs up to `known` to be complete.
  const int blocks = 7;
  int known = -1;
  int a_block[OZ_RING], a_slice[OZ_RING], a_uses[OZ_RING] = {}, a_free[OZ_RING], b_block[OZ_SLICES], b_free[OZ_SLICES];
  for (int s = 0; s < OZ_RING; ++s) a_block[s] = a_slice[s] = a_free[s] = -1;
  for (int j = 0; j < OZ_SLICES; ++j) b_block[j] = b_free[j] = -1;
  for (int c = 0; c < blocks; ++c) {
    for (int o = 0; o < OZ_LOADS; ++o) {
      const OzLoad L = oz_load(o);
      if (L.a >= 0) {
        const int s = oz_slot(c, oz_place(L.a));
        bad += L.b >= 0 || s < 0 || s >= OZ_RING || a_uses[s] != c;
        if (a_uses[s] > 0 && a_free[s] > known) known = a_free[s];   // the wait for the slot's last use
        bad += a_free[s] > known;
        ++a_uses[s];
        a_block[s] = c;
        a_slice[s] = L.a;
      } else {
        bad += b_free[L.b] > known;
        b_block[L.b] = c;
      }
    }
    for (int q = 0; q < OZ_MMAS; ++q) {
      const OzMma x = oz_mma(q);
      const int s = oz_slot(c, oz_place(x.a));
      bad += a_block[s] != c || a_slice[s] != x.a;
      if (q >= OZ_LOW) a_free[s] = c * OZ_MMAS + q;   // the commit that gives up the slot
      else a_free[s] = 1 << 30;                       // held
      for (int k = 0; k < x.n / OZ_COLS; ++k) {
        const int j = x.b + k;
        if (j < 0) continue;
        bad += b_block[j] != c;
        b_free[j] = c * OZ_MMAS + q;
      }
    }
    for (int s = 0; s < OZ_RING; ++s) bad += a_free[s] == 1 << 30;
  }
  // a B slice is waited for by the first MMA that reads it
  int waited[OZ_SLICES] = {};
  for (int q = 0; q < OZ_MMAS; ++q) {
    const OzMma x = oz_mma(q);
    if (x.new_b >= 0) bad += waited[x.new_b]++;
    for (int j = x.b < 0 ? 0 : x.b; j < x.b + x.n / OZ_COLS; ++j) bad += !waited[j];
  }
  for (int j = 0; j < OZ_SLICES; ++j) bad += !waited[j];
  std::printf("%d MMAs, %d columns, %d faults\n", OZ_MMAS, cols, bad);
  if (bad) return 1;
  std::printf("ok\n");
  return 0;
}
