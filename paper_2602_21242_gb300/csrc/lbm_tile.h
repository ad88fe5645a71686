// lbm_tile.h -- host side of the several-steps-a-launch tiles (lbm_tile.cuh).
#pragma once

#include <algorithm>

#include "lbm_launch.h"

namespace olbm {

// Tiles of tx x ty output nodes (tx >= nx, ty >= ny: the whole dimension, wrapping
// around), up to `steps` steps a launch; steps < 2: the path is not used.
struct TilesPlan {
  int tx = 0, ty = 0, steps = 0;
  bool on() const { return steps >= 2; }
};

constexpr int kTileSmemMax = 200 * 1024;  // two tiles' nodes of the first step; leaves room for static shared memory

constexpr int kTileStepsMax = 32;

// Nodes of the first of `steps` steps, and the shared memory of a CTA (two buffers of
// nine values a node).
inline long long tile_nodes(const Geometry& g, int tx, int ty, int steps) {
  const int w = tx >= g.nx ? g.nx : tx + 2 * (steps - 1), h = ty >= g.ny ? g.ny : ty + 2 * (steps - 1);
  return (long long)w * h;
}
inline long long tile_smem(const Geometry& g, int tx, int ty, int steps, int elem) {
  return steps < 2 ? 0 : 18LL * elem * tile_nodes(g, tx, ty, steps);
}

TilesPlan tile_plan(const Geometry& g, int prec, double theta, double tau, int sms, bool walls);

cudaError_t launch_tile_f64(const StepArgs& a, const TilesPlan& p, int steps, cudaStream_t st);
cudaError_t launch_tile_f32(const StepArgs& a, const TilesPlan& p, int steps, cudaStream_t st);
cudaError_t launch_tile_f16(const StepArgs& a, const TilesPlan& p, int steps, cudaStream_t st);
cudaError_t launch_tile_f64df(const StepArgs& a, const TilesPlan& p, int steps, cudaStream_t st);

}  // namespace olbm
