// Split of a far field by pairs of triangles (bem_pairs.cu) into tasks, and the partial sums that it takes.  Host only,
// no CUDA types.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdint>

namespace pbfb {

constexpr int PAIR_TILE = 32;  // triangles per tile: one per lane

struct PairSplit {
  int nT, tpg, G, K, nsub, ntask;  // tiles, tiles per group, groups, step parts, point shares, tasks
  size_t rows;                     // rows of partial sums, a float64 value per quadrature point each
};

// Tasks to aim at: 32 a SM (float64); 128 a SM (float-float), ten waves of the resident warps or so, which keeps the
// last one short (Laplace + Yukawa, 8000 triangles: one tile per group 3.99 + 5.77 ms, two 4.09 + 5.79; 15,680: two
// 15.1 + 21.9, three 15.7 + 22.7), or 8 ff_bps with a tuned ff_blocks_per_sm.  Past 16 of those the partial rows grow
// and the time does not (K operator, GB300, ff_bps 16, 24, 64: 12,500 triangles 9.66, 9.65, 9.65 ms; 15,680 15.11,
// 15.10, 15.11; 20,480 25.97, 25.63, 25.74): 16 is the most, and what pair_rows_max counts holds for every tuning.
constexpr int PAIR_FF_BPS = 16;
inline int pair_want(bool f64, int ff_bps) {
  return 152 * (f64 ? 32 : 8 * (ff_bps > 0 ? std::min(ff_bps, PAIR_FF_BPS) : PAIR_FF_BPS));
}

// G groups of tpg tiles, K parts of the 32 steps, and nsub shares of a triangle's points (3: a packed pair per lane;
// 1: all six).  tpg is rounded down: a group has one tile until there are twice as many tiles as the sqrt(2 want)
// groups that give `want` tasks, so that a surface just below that (393 tiles, float-float) has four times the tasks
// aimed at, and one just below three times as many 9/4 of them.  That is the better side: more tasks cost partial rows,
// fewer an uneven last wave (8000 triangles, 250 tiles, above; rounding up would take two tiles a group there).  Below
// some thousand tasks the chip is not full, and the steps are cut into parts and (float-float) the points into shares,
// which cost 12 % more operations but a third of the serial work of a lane.  GB300, one call of a K operator, us,
// (nsub, K), before the pair loop was unrolled -- float-float, 320 triangles (10 tiles): (1, 8) 75, (3, 4) 72, (3, 8)
// 76; 980 (31): (1, 2) 145, (3, 4) 139; 1280 (40): (1, 2) 192, (3, 2) 192; 2000 (63): (1, 2) 373, (3, 1) 371; 2880 (90):
// (1, 2) 683, (3, 1) 719; 3920 (123): (1, 1) 1209, (3, 1) 1266.  The float64 pipe is one unit per SM, so only the
// balance counts: 1620 triangles (51), Yukawa: K = 1 3694, 4 3097, 8 2817.
inline PairSplit pair_split(int nt, int want, bool f64) {
  PairSplit S;
  S.nT = std::max(1, (nt + PAIR_TILE - 1) / PAIR_TILE);
  S.nsub = 1;
  S.K = 1;
  const int G = std::max(1, std::min((int)std::sqrt(2.0 * want), S.nT));
  S.tpg = S.nT / G;
  S.G = (S.nT + S.tpg - 1) / S.tpg;
  auto tasks = [&] { return (int64_t)S.G * (S.G + 1) / 2 * S.K * S.nsub; };
  if (S.tpg == 1) {
    if (!f64 && tasks() <= 2048) S.nsub = 3;
    while (tasks() * 2 <= (f64 ? 24000 : 8192) && S.K < (f64 ? 8 : 4)) S.K *= 2;
  }
  S.ntask = (int)tasks();
  S.rows = S.nsub == 1 ? (size_t)S.K * (S.G + 1) : (size_t)S.K * S.G * (1 + S.nsub);
  return S;
}

// the rows of the larger of the two forms, at any tuning
inline size_t pair_rows_max(int nt) {
  return std::max(pair_split(nt, pair_want(true, 0), true).rows, pair_split(nt, pair_want(false, 0), false).rows);
}

}  // namespace pbfb
