// The launch order of the tile Cholesky (csrc/chol_schedule.cuh) on two streams: whichever of the two runs ahead, every
// tile is read and written in the order of the single-stream algorithm.  Vector clocks over the two streams; an access to
// a tile must have every earlier conflicting access among its predecessors.
#include <cstdint>
#include <cstdio>
#include <random>
#include <utility>
#include <vector>

#include "chol_schedule.cuh"

struct Plan {
  int nt;
  std::vector<int> col_rows, col_off, pair_off;
  std::vector<std::pair<int, int>> pairs;
  // symbolic factorisation of the lower tile pattern nz (row-major nt x nt)
  Plan(int n, std::vector<uint8_t> nz) : nt(n), col_off(n + 1), pair_off(n + 1) {
    for (int k = 0; k < nt; ++k) {
      col_off[k] = (int)col_rows.size();
      pair_off[k] = (int)pairs.size();
      std::vector<int> rows;
      for (int i = k + 1; i < nt; ++i)
        if (nz[i * nt + k]) rows.push_back(i);
      col_rows.insert(col_rows.end(), rows.begin(), rows.end());
      for (int first = 1; first >= 0; --first)   // the first row's column, then the others
        for (int i : rows)
          for (int j : rows)
            if (j <= i && (j == rows[0]) == (first == 1)) {
              pairs.emplace_back(i, j);
              nz[i * nt + j] = 1;
            }
    }
    col_off[nt] = (int)col_rows.size();
    pair_off[nt] = (int)pairs.size();
  }
};

struct Order {
  const Plan& P;
  int clock[2][2] = {};      // clock[a][b]: how many operations of stream b are known to precede stream a's next one
  int mark_clock[2] = {};
  std::vector<int> wr[2], rd[2];   // last write / read of a tile by stream b (1 + operation index; 0 none)
  std::vector<int> step;     // last step whose update a tile has received, or nt once it is factorised
  long long bad = 0;
  int side_updates = 0;
  explicit Order(const Plan& p) : P(p), step(p.nt * p.nt, -1) {
    for (int b = 0; b < 2; ++b) {
      wr[b].assign(P.nt * P.nt, 0);
      rd[b].assign(P.nt * P.nt, 0);
    }
  }
  void access(int a, int i, int j, bool write) {
    const int t = i * P.nt + j, b = 1 - a;
    bad += wr[b][t] > clock[a][b];
    if (write) bad += rd[b][t] > clock[a][b];
    (write ? wr : rd)[a][t] = clock[a][a] + 1;
  }
  void tile(int k) {
    access(0, k, k, true);
    ++clock[0][0];
  }
  void panel(int k) {
    access(0, k, k, false);
    for (int e = P.col_off[k]; e < P.col_off[k + 1]; ++e) access(0, P.col_rows[e], k, true);
    ++clock[0][0];
  }
  void update(int k, int p0, int count, bool side) {
    for (int e = p0; e < p0 + count; ++e) {
      const int i = P.pairs[e].first, j = P.pairs[e].second;
      access(side, i, k, false);
      access(side, j, k, false);
      access(side, i, j, true);
      bad += step[i * P.nt + j] >= k;   // once a step, in the order of the steps
      step[i * P.nt + j] = k;
    }
    ++clock[side][side];
    side_updates += side;
  }
  void fork() {
    for (int b = 0; b < 2; ++b) clock[1][b] = clock[0][b] > clock[1][b] ? clock[0][b] : clock[1][b];
  }
  void mark() {
    mark_clock[0] = clock[1][0];
    mark_clock[1] = clock[1][1];
  }
  void join() {
    for (int b = 0; b < 2; ++b) clock[0][b] = mark_clock[b] > clock[0][b] ? mark_clock[b] : clock[0][b];
  }
  void finish() {   // the factor is read on the stream
    for (int i = 0; i < P.nt; ++i)
      for (int j = 0; j <= i; ++j) access(0, i, j, true);
  }
};

static long long check(int nt, const std::vector<uint8_t>& nz, int split, int* side) {
  const Plan P(nt, nz);
  Order O(P);
  fetirp::chol_schedule(nt, P.col_off.data(), P.col_rows.data(), P.pair_off.data(), split, O);
  O.finish();
  *side += O.side_updates;
  std::vector<int> last(nt * nt, -1);
  for (int k = 0; k < nt; ++k)
    for (int e = P.pair_off[k]; e < P.pair_off[k + 1]; ++e) last[P.pairs[e].first * nt + P.pairs[e].second] = k;
  return O.bad + (last != O.step);   // every update was made
}

int main() {
  long long bad = 0;
  int side = 0, plans = 0;
  auto run = [&](int nt, const std::vector<uint8_t>& nz) {
    for (int split : {0, 1, 5, 76}) bad += check(nt, nz, split, &side), ++plans;
  };
  // dense; a band with an arrow (interior planes, then the boundary), without and with one or two decoupled tile columns
  for (int nt : {1, 2, 13, 30}) run(nt, std::vector<uint8_t>(nt * nt, 1));
  for (int band : {1, 3, 6})
    for (int hole = -1; hole < 24; ++hole)
      for (int holes = 1; holes <= 2; ++holes) {
        const int nt = 40, arrow = 24;
        std::vector<uint8_t> nz(nt * nt, 0);
        for (int i = 0; i < nt; ++i)
          for (int j = 0; j <= i; ++j) {
            const bool cut = hole >= 0 && ((i >= hole && i < hole + holes) || (j >= hole && j < hole + holes));
            nz[i * nt + j] = i == j || ((i - j <= band || i >= arrow) && !cut);
          }
        run(nt, nz);
      }
  std::mt19937 rng(1);
  for (int t = 0; t < 200; ++t) {   // random patterns, a third of the columns empty below the diagonal
    const int nt = 5 + (int)(rng() % 36);
    const unsigned density = 1 + rng() % 9;
    std::vector<uint8_t> nz(nt * nt, 0), empty(nt);
    for (auto& e : empty) e = rng() % 3 == 0;
    for (int i = 0; i < nt; ++i)
      for (int j = 0; j < i; ++j) nz[i * nt + j] = !empty[i] && !empty[j] && rng() % 10 < density;
    run(nt, nz);
  }
  std::printf("%d plans, %d updates on the side stream, %lld accesses out of order\n", plans, side, bad);
  if (bad || !side) return 1;
  std::printf("ok\n");
  return 0;
}
