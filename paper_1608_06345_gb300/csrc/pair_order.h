// The two-step kernel's grid, and its waits as rules on row numbers, so that
// both can be checked on the host.
//
// Two groups of warps (A) do the first step of the band's even and odd rows t
// = 0 .. rows + 5, two groups (B) the second step of the even and odd rows q =
// 0 .. rows - 1, and B's row q pulls A's rows q .. q + 6.  Each row has an
// arrival of every warp of its group, A's on stored[t mod 8] once the row is
// in the ring, B's on pulled[q mod 8] once it has been read.  A barrier's
// phase n / 8 is complete when row n's arrivals are in, and a wait for row n
// tests that phase's parity, so it is right only while the barrier cannot be a
// whole phase further on: row n + 8 must need something that the waiting warp
// does only after the wait.  That holds for every wait below:
//   - A on pulled[t - 8]: the next phase is pulled[t], which needs this warp's
//     own row t stored;
//   - A on stored[t - 3], t < 8: the next phase is stored[t + 5], which needs
//     pulled[t - 3], hence row t stored;
//   - B on stored[q + 6]: the next phase is stored[q + 14], which needs
//     pulled[q + 6], of this warp's group and after row q;
//   - B on stored[q + 5]: the next phase is stored[q + 13], which needs
//     pulled[q + 5] of the other group, hence stored[q + 10] and so pulled[q +
//     2], of this warp's group and after row q.
// A wait of B's first rows for A's earlier rows would not be right: A's row 8
// needs only the even group's pull of row 0, so stored[0] can be a phase ahead
// of a warp of the odd group that has not looked yet.  Nor is it needed, since
// each group of A arrives row after row: rows q + 5 and q + 6 stored means
// that all earlier ones are.
#pragma once

namespace lbm {

constexpr int kPairBars = 8;  // barriers of each kind

// A may store row t once B has pulled row pair_a_pulled(t) (the rows that it
// replaces in the ring were last read there) and, where no such row exists,
// once A's row pair_a_stored(t) is stored (the band's first rows replace only
// rows that nobody pulls, but must not overtake the other group's); below 0:
// no such wait
constexpr int pair_a_pulled(int t) { return t - kPairBars; }
constexpr int pair_a_stored(int t) { return t < kPairBars ? t - 3 : -1; }

// B may pull row q once A's rows pair_b_begin(q) .. pair_b_end(q) are stored
constexpr int pair_b_begin(int q) { return q + 5; }
constexpr int pair_b_end(int q) { return q + 6; }

constexpr int kPairTries = 1 << 20;   // of a wait, about a microsecond each
constexpr int kPairW = 128;           // A's columns
constexpr int kPairOut = kPairW - 6;  // columns a strip can hold

// The grid of the two-step kernel: strips of width columns by bands of rows.
// share is that of the iterations which full strips without a band's 7 extra
// iterations would need; 0 where there is no grid.
struct PairGrid {
  int strips, bands, width;
  double share;
};

// One block fits an SM, and a block's time is that of its rows + 7 iterations,
// so take the number of bands with the fewest iterations over all waves.  (512
// candidates of two divisions each take a few microseconds of the host's time,
// half of a small step's, so an instance does this once, when it is made.)
inline PairGrid pair_grid(int nx, int ny, int sms) {
  PairGrid g;
  g.strips = (nx + kPairOut - 1) / kPairOut;
  g.width = (nx + g.strips - 1) / g.strips;
  g.bands = 1;
  long long best = -1;
  for (int nb = 1; nb <= ny && nb <= 512; ++nb) {
    const long long waves = ((long long)g.strips * nb + sms - 1) / sms;
    const long long cost = waves * ((ny + nb - 1) / nb + 7);
    if (best < 0 || cost < best) {
      best = cost;
      g.bands = nb;
    }
  }
  g.share = (double)((long long)nx * ny) / ((double)kPairOut * sms * (double)best);
  return g;
}

}  // namespace lbm
