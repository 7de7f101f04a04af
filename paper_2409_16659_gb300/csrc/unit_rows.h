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
inline int march_rows(int n, int ny, int strips, int num_sms, int slots) {
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
  if (flat <= 3) return (int)flat;
  for (long wave = 1;; ++wave) {
    const long chunks = (long)slots * wave / strips;
    if (chunks < 1) continue;
    const long rows = (ny + chunks - 1) / chunks;
    if (rows <= 64) return (int)rows;
  }
}

}  // namespace mlsw
