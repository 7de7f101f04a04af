// unit_rows.h -- rows of the units of work that a D2Q9 step is cut into.
// Host code.
#pragma once

namespace mlsw {

// Rows of a unit. A unit costs its rows plus about five rows of warm-up. On
// a lattice that leaves each warp a scheduler of its own (4 per SM) with at
// most 3 rows, a row takes the latency of one warp whatever the others do:
// units are as flat as that allows (three layers, us a step: 256^2 with 1, 2,
// 3, 4 rows 8.3, 7.8, 7.5, 8.5). Larger lattices run as one wave of the warps
// that fit (slots), which also spreads them evenly over the SMs: 512^2 with
// 2, 3, 4 rows 15.9, 12.4, 14.2; 1024^2 with 8, 11, 13 rows 33.3, 28.7, 32.5;
// 2048^2 with 32, 43, 51 rows 101, 89, 104 (before image pairs had one store,
// which took 8 % off each: 26.6 and 80.9 now). Units taller than 64 rows would
// put neighbouring units further apart in time than the L2 keeps the rows
// they share; then several waves.
//
// One and two layers gain less from warps that share a scheduler (k of them
// take per_row[k - 1] times one's time for a row): there a wave of the warps
// that fit is for more than four rows a unit, and below that the height is the
// cheapest by that model. One layer, 448^2: 8.1 us a step with 1 row (the
// wave), 5.0 with 3; 25 x 1870 5.1 and 4.4 with 2; two layers, 320^2: 7.3 with
// 1, 5.8 with 2; 25 x 1870 8.2 and 6.0 with 2.
//
// heavy: rows of more than 3 us (four layers with tau != 1, five with many terms a
// cell, see step_dear): these run as one wave from three rows a unit on (four layers,
// tau = 0.8, 256^2: 15.1 us a step with 3 rows, 13.3 with 2; five layers, far
// pairs: 20.1 and 18.8).
inline int march_rows(int n, bool heavy, int ny, int strips, int num_sms, int slots) {
  if (slots < 1) slots = 1;
  const long total = (long)ny * strips, flat = (total + 4L * num_sms - 1) / (4L * num_sms);
  if (n <= 2 && total <= 4L * slots) {
    constexpr double per_row[2][5] = {{1.0, 1.12, 1.33, 1.51, 1.95}, {1.0, 1.25, 1.66, 1.95, 2.4}};
    double best = 0.0;
    int best_rows = 0;
    for (int rows = 1; rows <= 8; ++rows) {
      const long units = (long)strips * ((ny + rows - 1) / rows);
      const long k = (units + 4L * num_sms - 1) / (4L * num_sms);
      if (units > slots || k > 5) continue;
      const double cost = (rows + 5) * per_row[n > 1][k - 1];
      if (best_rows == 0 || cost < best) {
        best = cost;
        best_rows = rows;
      }
    }
    if (best_rows > 0) return best_rows;
  }
  if (flat <= (heavy ? 2 : 3)) return (int)flat;
  for (long wave = 1;; ++wave) {
    const long chunks = (long)slots * wave / strips;
    if (chunks < 1) continue;
    const long rows = (ny + chunks - 1) / chunks;
    if (rows <= 64) return (int)rows;
  }
}

// Whether the march of an n-layer lattice takes one column a lane (26 columns a
// strip) instead of a pair (56). Per row and warp that is the shorter chain
// with half the registers and ring, so more warps; per column it is more
// instructions. It pays, from four layers on, where
//   * both forms have one strip: 25 x 1870, us a step with pairs and with single
//     columns, four layers 12.6 and 9.9 (tau = 1, near pairs), 15.6 and 12.5 (far
//     pairs), 18.1 and 11.5 (tau = 0.8), five 15.3 and 11.3, 20.9 and 16.0, 26.8 and
//     15.1; 26 x 30000, five layers, tau = 0.8, 270 and 153;
//   * pairs leave a third of their strips empty (57 to 78 columns) and give a
//     scheduler two rows or more: 57 x 800, four layers, 14.4 and 12.4 (far
//     pairs); above four rows a scheduler only in the general mode, whose
//     pairs hold four to six warps an SM (57 x 10000, five layers 171 and 118,
//     but four layers with near pairs, 78 x 2500, 18.2 and 19.7);
//   * pairs have two to three rows a scheduler and every cell many terms (dear:
//     tau != 1, far pairs, a substrate or the exponential potential): 256^2, five
//     layers, 20.2 and 18.2 (far pairs), 20.4 and 18.7 (tau = 0.8); without them,
//     four layers, 10.1 and 10.6.
// Fewer rows a scheduler go to pairs (130^2: 10.4 and 13.8).
inline bool march_solo(int n, bool general, bool dear, int nx, int ny, int num_sms) {
  if (n < 4) return false;
  const long pairs = (nx + 55) / 56, solo = (nx + 25) / 26, total = pairs * ny, s = 4L * num_sms;
  if (solo == 1) return true;
  if (total <= 2 * s) return false;
  if (2 * solo <= 3 * pairs && (general || total <= 4 * s)) return true;
  return dear && solo <= 2 * pairs && total <= 3 * s;
}

// Rows of a unit with one column a lane: the cheapest by rows plus warm-up (five
// rows, in the general mode one and a half) times what a row takes with k warps
// on a scheduler; beyond 16 rows one wave of the warps that fit, as for pairs.
// 25 x 1870, four layers, tau = 1, with 1, 2, 3, 4 rows: 15.2, 12.5, 13.9, 14.4 us.
inline int solo_rows(bool general, int ny, int strips, int num_sms, int slots) {
  constexpr double per_row[2][6] = {{1.0, 1.17, 1.38, 1.7, 2.1, 2.5}, {1.0, 1.06, 1.27, 1.6, 2.0, 2.4}};
  double best = 0.0;
  int best_rows = 0;
  for (int rows = 1; rows <= 16; ++rows) {
    const long units = (long)strips * (((long)ny + rows - 1) / rows);
    const long k = (units + 4L * num_sms - 1) / (4L * num_sms);
    if (units > slots || k > 6) continue;
    const double cost = (rows + (general ? 1.5 : 5.0)) * per_row[general][k - 1];
    if (best_rows == 0 || cost < best) {
      best = cost;
      best_rows = rows;
    }
  }
  return best_rows > 0 ? best_rows : march_rows(4, true, ny, strips, num_sms, slots);
}

// Batches whose units are cut to equal duration. What a row counts (us), by layers
// and mode (StepMode; four and five layers of the general one with one column a
// lane): about what it takes a warp alone where that is slow, and more where it is
// quick, because warps that share an SM with slow kinds wait with them. (Alone,
// from the slope between 4 and 16 rows a unit: general 0.9 to 4.4, tau = 1 with far
// pairs 0.7 to 3.4, fast 0.47, 0.62, 0.84, 1.08, 1.3, a substrate 1.0 more. With these
// 60 random batches step in 0.995 of the time on average, but five in up to 1.6.)
inline double batch_weight(int n, int mode, bool substrate) {
  constexpr double w[3][5] = {{0.75, 1.3, 2.1, 2.9, 3.9}, {0.6, 1.0, 1.45, 2.45, 3.5}, {0.5, 0.85, 1.3, 1.8, 2.2}};
  return w[mode][n - 1] * (substrate ? 2.0 : 1.0);
}

// Rows of a unit that lasts about t (us): rows and about five of warm-up, at
// most 64 rows.
inline int batch_rows(double weight, double t) {
  double r = t / weight - 5.0;
  r = r < 1.0 ? 1.0 : (r > 64.0 ? 64.0 : r);
  return (int)(r + 0.5);
}

// The height of nominal 8-row units where that is a choice: half.
inline int half_rows(int rows) { return (rows + 1) / 2; }

// What a step takes (us) in units of at most `longest` us, `work` us in all: in one
// wave the longest unit, stretched by the warps beside it; in several the work at
// the rate of full schedulers and the longest unit at the end. Coefficients that
// choose best over 15 batches of 6 to 60 lattices (1 to 5 layers, all modes, sides
// 16 to 320) stepped with 28 durations each: 3 % from the best duration on average
// (time at the end of the last wave counted twice as dear, and warps beside one
// another: 19 %).
inline double batch_cost(double units, double work, double longest, int num_sms, int slots) {
  if (units <= slots) return 1.4 * longest;
  return 0.35 * work / (4.0 * num_sms) + 1.5 * longest;
}

}  // namespace mlsw
