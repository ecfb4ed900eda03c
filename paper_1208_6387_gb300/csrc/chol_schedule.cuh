// Order of the launches of a right-looking tile Cholesky on a stream and, for the trailing updates that the next column
// does not wait for, a side stream.  Plain C++: the order is checked on the host (tests/host/chol_schedule.cpp).
#pragma once

namespace fetirp {

// col_rows[col_off[k] .. col_off[k + 1]): the rows I > k of the nonzero tiles of column k; pairs [pair_off[k],
// pair_off[k + 1]): the tiles (I, J) that step k updates, those of J = the column's first row first.  The updates beyond
// the next column go to the side stream from split_pairs of them on (0: never), so that the chain of diagonal tiles and panels
// goes on beside them; every tile still receives its updates in the order of k.
//   ops.tile(k), ops.panel(k), ops.update(k, first_pair, count, on_side)
//   ops.fork(): the side stream waits for the stream's work so far; ops.mark(): a mark on the side stream
//   ops.join(): the stream waits for the last mark
template <class Ops>
void chol_schedule(int nt, const int* col_off, const int* col_rows, const int* pair_off, int split_pairs, Ops& ops) {
  bool pending = false;   // the side stream holds updates that the stream has not waited for
  for (int k = 0; k < nt; ++k) {
    ops.tile(k);
    const int nr = col_off[k + 1] - col_off[k];
    if (nr > 0) ops.panel(k);
    const int p0 = pair_off[k], np = pair_off[k + 1] - p0;
    const int next = nr > 0 && col_rows[col_off[k]] == k + 1 ? nr : 0;   // pairs of column k + 1
    const bool split = split_pairs > 0 && np - next >= split_pairs;
    if (split) ops.fork();
    // Every earlier update is waited for here, by an empty column too: its step touches no tile, but the next column's may
    // be among those that the side stream still updates.
    if (pending) ops.join();
    pending = split;
    const int here = split ? next : np;
    if (here > 0) ops.update(k, p0, here, false);
    if (split) {
      ops.update(k, p0 + next, np - next, true);
      ops.mark();
    }
  }
  if (pending) ops.join();
}

}  // namespace fetirp
