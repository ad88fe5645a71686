// Host check of the small-lattice tiles' index arithmetic (lbm_tile.h): for every lattice
// width NX0 .. NX1 (step STRIDE) of NY rows that tile_plan gives a plan, the rows and
// columns that the kernel forms from a linear index in the regions of every step of a launch, against
// integer division, for the full tile and the ragged last ones. Prints the widths looked at,
// those with a plan, the largest region (in columns), the number of wrong indices, and of every eighth plan
// those that are dearer than the cheapest of all cuts by the cost model.
// Usage: tile_check PREC WALLS SMS NY NX0 NX1 STRIDE
#include <algorithm>
#include <cstdio>
#include <cstdlib>

#include "lbm_tile_plan.cu"

// (lbm_reduce.cu's, which needs a device)
namespace olbm {
int stream_tile_width(int prec) { return prec == 1 ? 256 : 512; }
int stream_ctas_per_sm(int) { return 3; }
}  // namespace olbm
using namespace olbm;

// Microseconds a step of a plan by the cost model, and the least of all cuts and step counts.
static double cost(const Geometry& g, int prec, int sms, int tx, int ty, int steps) {
  const Cost k = cost_of(prec);
  const int a = (g.nx + tx - 1) / tx, b = (g.ny + ty - 1) / ty, m = (a * b + sms - 1) / sms;
  double work = 1.25;
  for (int s = 1; s <= steps; ++s) work += k.L + (double)m * (double)tile_nodes(g, tx, ty, s) * k.c;
  return work / steps;
}
static double least_cost(const Geometry& g, int prec, int sms) {
  const int elem = prec == 1 ? 4 : (prec == 2 ? 2 : 8);
  double least = 1e9;
  for (int a = 1; a <= std::min(g.nx, 2 * sms); ++a)
    for (int b = 1; b <= std::min(g.ny, 2 * sms / a); ++b) {
      const int tx = (g.nx + a - 1) / a, ty = (g.ny + b - 1) / b;
      const int ca = (g.nx + tx - 1) / tx, cb = (g.ny + ty - 1) / ty, m = (ca * cb + sms - 1) / sms;
      for (int s = 2; s <= kTileStepsMax; ++s) {
        if ((ca > 1 && tx + 2 * (s - 1) > g.nx) || (cb > 1 && ty + 2 * (s - 1) > g.ny)) break;
        if (tile_smem(g, tx, ty, s, elem) * m > kTileSmemMax) break;
        least = std::min(least, cost(g, prec, sms, tx, ty, s));
      }
    }
  return least;
}

int main(int, char** v) {
  const int prec = atoi(v[1]), walls = atoi(v[2]), sms = atoi(v[3]), ny = atoi(v[4]);
  const bool f64 = prec == 0 || prec == 3;
  long long widths = 0, planned = 0, largest = 0, wrong = 0, dear = 0;
  for (int nx = atoi(v[5]); nx <= atoi(v[6]); nx += atoi(v[7])) {
    ++widths;
    const Geometry g{nx, ny, nx, (long long)nx * ny};
    const TilesPlan p = tile_plan(g, prec, 1.0 / 3.0, 0.8, sms, walls != 0);
    if (!p.on()) continue;
    ++planned;
    if (planned % 8 == 1 && cost(g, prec, sms, p.tx, p.ty, p.steps) > least_cost(g, prec, sms) * (1 + 1e-12)) ++dear;
    const bool wrapx = p.tx >= nx, wrapy = p.ty >= ny;
    const int lastx = nx - (nx - 1) / p.tx * p.tx, lasty = ny - (ny - 1) / p.ty * p.ty;
    for (int ring = 0; ring < p.steps; ++ring)
      for (int e = 0; e < 4; ++e) {  // full and ragged tiles
        const int w = (e & 1 ? lastx : std::min(p.tx, nx)) + (wrapx ? 0 : 2 * ring);
        const int h = (e & 2 ? lasty : std::min(p.ty, ny)) + (wrapy ? 0 : 2 * ring);
        const int cols = f64 ? w : (w + 1) / 2;  // nodes, or node pairs
        largest = std::max<long long>(largest, w);
        const unsigned inv = tile_row_inv(cols);
        for (int idx = 0; idx < cols * h; ++idx) wrong += tile_row(idx, inv) != idx / cols;
      }
  }
  printf("%lld %lld %lld %lld %lld\n", widths, planned, largest, wrong, dear);
  return 0;
}
