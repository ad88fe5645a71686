// lbm_tile_plan.cu -- when a lattice takes several steps a launch (lbm_tile.cuh), and with
// which tiles: the cheapest of all cuts into at most two tiles an SM by a cost model, if
// that is cheaper than the single-step (FP32: two-step) kernels by more than the
// model's error.
//
// Microseconds, fitted on GB300 (152 SMs, complete model, diagnostics off):
//   a launch 1.25; a step of a tile L + m n c, n its nodes in that step, m tiles an SM:
//   FP64 storage L = 1.35, c = 1/220; FP32 and FP16 L = 0.7, c = 1/650 (e.g. 64^2 FP64 in
//   8 x 4 tiles, 2 / 3 / 4 / 6 steps: 4.3, 5.8, 7.5, 11.8 a launch; FP32 4.2 and 5.7
//   for 4 and 6 steps; 512^2 FP32 in 64 x 27 tiles 7.7, 11.6 and 15.4 for 2, 3 and 4)
//   a single step of the other kernels 2.2 + nodes / 33e3 (FP64 storage: 2.45, 4.5, 6.5
//   and 10.0 at 64^2, 256^2, 384^2 and 512^2) or 2.3 + nodes / 100e3 (FP32, FP16: 2.4,
//   3.2, 4.8 and 12.2 at 64^2, 256^2, 512^2 and 1024^2).
// So the line lies near 150^2 nodes for FP64 storage (64^2: 2.45 -> 1.9 us a step, 256^2
// stays at 4.5 against 4.8 in tiles) and near 600^2 for FP32 (512^2 4.8 -> 3.8,
// 768^2 7.6 against 8.3); for FP16 between 390^2 and 550^2, by the waves of its single steps. Walls cost the single steps another launch (about 2 us), which the
// tiles do not need, so lattices with walls take tiles up to a higher line.
#include "lbm_tile.h"

namespace olbm {

namespace {

struct Cost {
  double L, c, per_node;
};

Cost cost_of(int prec) {
  return prec == 0 || prec == 3 ? Cost{1.35, 1.0 / 220.0, 1.0 / 33e3} : Cost{0.7, 1.0 / 650.0, 1.0 / 100e3};
}

}  // namespace

TilesPlan tile_plan(const Geometry& g, int prec, double theta, double tau, int sms, bool walls) {
  TilesPlan best;
  const bool f64 = prec == 0 || prec == 3;
  if (f64 && !fx::make_coefs(theta, tau).on) return best;  // the tiles take the fixed-point collision
  const Cost k = cost_of(prec);
  const int elem = prec == 1 ? 4 : (prec == 2 ? 2 : 8);
  double single = (f64 ? 2.2 : 2.3) + (double)g.nx * g.ny * k.per_node;
  // FP16's single steps take one row a CTA on these lattices and at most 3.35 while those are one wave of the three
  // resident an SM, whatever the nodes (us a step in tiles / single: 391 x 383 3.8 / 3.6, 378 x 413
  // 3.8 / 3.3, 450^2 3.8 / 3.5, 2042 x 106 4.3 / 3.5, 400^2 3.25 / 3.4; 512^2, two waves, 3.95 / 4.6).
  const long long strips = (g.nx + stream_tile_width(2) - 1) / stream_tile_width(2);
  if (prec == 2 && strips * g.ny <= (long long)stream_ctas_per_sm(2) * sms) single = std::min(single, 3.35);
  double least = (prec == 2 ? 0.85 : 0.95) * (single + (walls ? 2.0 : 0.0));
  if (1.25 / 8 + k.L + (double)g.nx * g.ny * k.c / sms > least) return best;  // no cut can be cheaper
  for (int a = 1; a <= std::min(g.nx, 2 * sms); ++a) {
    const int tx = (g.nx + a - 1) / a;
    if ((g.nx + tx - 1) / tx != a) continue;  // the same tiles as a smaller cut
    for (int b = 1; b <= std::min(g.ny, 2 * sms / a); ++b) {
      const int ty = (g.ny + b - 1) / b;
      if ((g.ny + ty - 1) / ty != b) continue;
      const int m = (a * b + sms - 1) / sms;
      // no number of steps makes this cut cheaper than the best so far
      if (1.25 / kTileStepsMax + k.L + (double)m * ((double)tx * ty) * k.c > least) continue;
      double work = 0.0;  // of the steps so far, last first (the region grows towards the first)
      for (int s = 1; s <= kTileStepsMax; ++s) {
        const int grow = 2 * (s - 1);
        if ((a > 1 && tx + grow > g.nx) || (b > 1 && ty + grow > g.ny)) break;  // a tile would meet itself
        const long long n = tile_nodes(g, tx, ty, s);
        if (tile_smem(g, tx, ty, s, elem) * m > kTileSmemMax) break;
        const double step = k.L + (double)m * (double)n * k.c;
        work += step;
        const double t = (1.25 + work) / s;
        if (step > least && t > least) break;  // and every further step costs as much
        if (s >= 2 && t < least) least = t, best.tx = tx, best.ty = ty, best.steps = s;
      }
    }
  }
  return best;
}

}  // namespace olbm
