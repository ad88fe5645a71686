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

// Row of index idx in a region of `cols` columns, idx / cols by a multiplication (the reciprocal
// once a step): inv = 2^28 / cols rounded up, by e < cols / 2^28 of a column too much, so the
// quotient is exact while idx * cols < 2^28. Both are at most a region's nodes.
__host__ __device__ inline unsigned tile_row_inv(int cols) {
  return ((1u << 28) + (unsigned)cols - 1u) / (unsigned)cols;
}
__host__ __device__ inline int tile_row(int idx, unsigned inv) {
  return (int)(((unsigned long long)(unsigned)idx * inv) >> 28);
}
constexpr long long kTileNodesMax = kTileSmemMax / (18 * 2);  // of the smallest storage type
static_assert(kTileNodesMax * kTileNodesMax < (1LL << 28), "tile_row is exact for every region that fits");

TilesPlan tile_plan(const Geometry& g, int prec, double theta, double tau, int sms, bool walls);

cudaError_t launch_tile_f64(const StepArgs& a, const TilesPlan& p, int steps, cudaStream_t st);
cudaError_t launch_tile_f32(const StepArgs& a, const TilesPlan& p, int steps, cudaStream_t st);
cudaError_t launch_tile_f16(const StepArgs& a, const TilesPlan& p, int steps, cudaStream_t st);
cudaError_t launch_tile_f64df(const StepArgs& a, const TilesPlan& p, int steps, cudaStream_t st);

}  // namespace olbm
