// lbm_tile.cuh -- several steps of Eq. 1 per launch on small lattices, each CTA
// advancing a tile (and the halo that its later steps need) in shared memory.
//
// What bounds a small lattice is not arithmetic or memory but the chain of dependent
// launches: a 64 x 64 FP64 step is one warp's worth of work on a fraction of the SMs and
// takes a few microseconds however many SMs there are. A CTA that owns tx x ty output
// nodes of step t + k computes step t + s on the tile grown by k - 1 - s nodes on every
// side, from the stored state (s = 0) or from shared memory, so k steps cost one
// launch and no communication between CTAs; the price is the grown rings, computed by
// every tile that needs them. A tile that spans a whole dimension of the lattice wraps
// around in it and needs no ring there (one-row and one-column lattices). Between the
// steps values are rounded to the storage type as a store would, and every node collides
// as in the single-step kernels, so the results are theirs bit for bit (FP32 and FP16:
// those of the node-pair kernels). Walls and the diagnostics of the first step are
// handled in the same pass.
//
// tile_plan (lbm_tile_plan.cu) chooses tile and steps by a cost model and says
// where the line to the single-step kernels lies.
#pragma once

#include "lbm_kernels.cuh"
#include "lbm_tile.h"

namespace olbm {

constexpr int kTileThreads = 512;  // at most; launched with the nodes of a region, rounded up to warps

__host__ __device__ constexpr int opposite_of(int i) {
  // Fig. 1a numbering: 1 <-> 3, 2 <-> 4, 5 <-> 7, 6 <-> 8
  return i == 0 ? 0 : (i < 5 ? ((i + 1) & 3) + 1 : ((i - 3) & 3) + 5);
}

// The nodes of one CTA: local (lx, ly) in [0, W) x [0, H) is the lattice node
// (x0 + lx, y0 + ly), taken periodically.
struct TileBox {
  int W, H;        // nodes of the first step
  int x0, y0;      // lattice position of local (0, 0), within one period
  int hx, hy;      // ring of the first step around the output nodes (0 where the tile wraps)
  int w, h;        // output nodes
};

__device__ __forceinline__ float tile_ld(const float* p) { return *p; }
__device__ __forceinline__ float tile_ld(const __half* p) { return __half2float(*p); }

// FP64 storage: the floating-point collision of a node outside the fixed-point range.
template <int MODEL, int PREC, typename CT>
__device__ __noinline__ void tile_float(double* f, const Coef<CT>& c, NodeMoments<CT>* m) {
  if constexpr (PREC == 3) {
    double r[9];
    df64 d[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) r[i] = f[i];
    split_node(r, d);
    collide_df<MODEL>(d, c, [&](const NodeMoments<df64>& x) { *m = x; },
                      [&](int i, df64 v) {
                        f[i] = kDfJoin == 2 ? join_f64_int(v) : (kDfJoin == 1 ? join_f64_fp64pipe(v) : join_f64(v));
                      });
  } else {
    double r[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) r[i] = f[i];
    collide<MODEL, false, double>(r, c, [&](const NodeMoments<double>& x) { *m = x; });
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = r[i];
  }
}

template <int MODEL, int PREC, bool DIAG>
__global__ void __launch_bounds__(kTileThreads)
    tile_steps_kernel(const typename Form<PREC>::S* src, typename Form<PREC>::S* dst, Geometry g,
                      Coef<typename std::conditional<kHasFixed<typename Form<PREC>::T>, typename Form<PREC>::T, f32x2>::type> c,
                      int steps, int tx, int ty, const unsigned char* __restrict__ walls,
                      double* __restrict__ partials) {
  using S = typename Form<PREC>::S;
  constexpr bool kF64 = kHasFixed<typename Form<PREC>::T>;
  using CT = typename std::conditional<kF64, typename Form<PREC>::T, f32x2>::type;
  extern __shared__ __align__(128) unsigned char smem[];
  const bool wrapx = tx >= g.nx, wrapy = ty >= g.ny;
  TileBox b;
  b.hx = wrapx ? 0 : steps - 1, b.hy = wrapy ? 0 : steps - 1;
  const int ox = blockIdx.x * tx, oy = blockIdx.y * ty;
  b.w = min(tx, g.nx - ox), b.h = min(ty, g.ny - oy);
  b.W = b.w + 2 * b.hx, b.H = b.h + 2 * b.hy;
  b.x0 = ox - b.hx, b.y0 = oy - b.hy;
  const int area = b.W * b.H;
  S* cur = reinterpret_cast<S*>(smem);
  S* nxt = cur + 9 * area;
  DiagAcc<CT> acc;
  FixedDiagAcc facc;
  pdl_wait();
  pdl_launch_dependents();
  for (int s = 0; s < steps; ++s) {
    const bool first = s == 0, last = s == steps - 1;
    const int mx = wrapx ? 0 : s, my = wrapy ? 0 : s;  // ring already consumed
    const int w = b.W - 2 * mx, h = b.H - 2 * my;
    const int cols = kF64 ? w : (w + 1) / 2;           // nodes, or node pairs, of a row
    const unsigned inv = tile_row_inv(cols);
    for (int idx = threadIdx.x; idx < cols * h; idx += blockDim.x) {
      const int row = tile_row(idx, inv), col = idx - row * cols;
      const int lx = mx + (kF64 ? col : 2 * col), ly = my + row;
      int gx = b.x0 + lx, gy = b.y0 + ly;
      gx = gx < 0 ? gx + g.nx : (gx >= g.nx ? gx - g.nx : gx);
      gy = gy < 0 ? gy + g.ny : (gy >= g.ny ? gy - g.ny : gy);
      const bool two = !kF64 && lx + 1 < b.W - mx;       // the pair's second node is part of the region
      const int gx2 = gx + 1 >= g.nx ? 0 : gx + 1;
      // f_i pulled at x - c_i: element offsets of columns x - 1 .. x + 2 and rows y - 1 .. y + 1
      const S* base;
      long long plane;
      long long rw[3];
      int cl[4];
      if (first) {
        base = src, plane = g.plane;
        rw[0] = (long long)(gy == 0 ? g.ny - 1 : gy - 1) * g.pitch;
        rw[1] = (long long)gy * g.pitch;
        rw[2] = (long long)(gy == g.ny - 1 ? 0 : gy + 1) * g.pitch;
        cl[0] = gx == 0 ? g.nx - 1 : gx - 1, cl[1] = gx, cl[2] = gx2, cl[3] = gx2 + 1 >= g.nx ? 0 : gx2 + 1;
      } else {
        base = cur, plane = area;
        const int ym = wrapy && ly == 0 ? b.H - 1 : ly - 1, yp = wrapy && ly == b.H - 1 ? 0 : ly + 1;
        rw[0] = ym * b.W, rw[1] = ly * b.W, rw[2] = yp * b.W;
        cl[0] = wrapx && lx == 0 ? b.W - 1 : lx - 1, cl[1] = lx;
        cl[2] = wrapx && lx == b.W - 1 ? 0 : lx + 1;
        cl[3] = wrapx && cl[2] == b.W - 1 ? 0 : cl[2] + 1;
      }
      S* out = last ? dst + (long long)gy * g.pitch + gx : nxt + ly * b.W + lx;
      const long long oplane = last ? g.plane : area;
      const bool owned = lx >= b.hx && lx < b.hx + b.w && ly >= b.hy && ly < b.hy + b.h;
      if constexpr (kF64) {
        double f[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i] = base[i * plane + rw[1 - cy_of(i)] + cl[1 - cx_of(i)]];
        const bool wall = walls != nullptr && walls[(long long)gy * g.nx + gx] != 0;
        auto store = [&](int i, double v) { out[i * oplane] = v; };
        double e[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) e[i] = f[i];
        const bool ok = collide_fixed<MODEL>(
            e, c.fixed,
            [&](const FixedMoments& m) {
              if constexpr (DIAG) {
                if (first && owned) facc.add(m);
              }
            },
            [](double (&)[9]) {}, store);
        if (!ok) {
          double t[9];
          NodeMoments<CT> m;
#pragma unroll
          for (int i = 0; i < 9; ++i) t[i] = f[i];
          tile_float<MODEL, PREC, CT>(t, c, &m);
          if constexpr (DIAG) {
            if (first && owned) acc.add(m);
          }
#pragma unroll
          for (int i = 0; i < 9; ++i) store(i, t[i]);
        }
        if (wall) {
#pragma unroll
          for (int i = 0; i < 9; ++i) store(i, f[opposite_of(i)]);
        }
      } else {
        const int second = two ? 1 : 0;  // (a lone node fills both lanes)
        f32x2 f[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          const S* p = base + i * plane + rw[1 - cy_of(i)];
          f[i] = f32x2(make_float2(tile_ld(p + cl[1 - cx_of(i)]),
                                   tile_ld(p + cl[1 - cx_of(i) + second])));
        }
        f32x2 e[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) e[i] = f[i];
        collide<MODEL, true, f32x2>(e, c, [&](NodeMoments<f32x2> m) {
          if constexpr (DIAG) {
            if (first) {
              const bool owned2 = two && lx + 1 >= b.hx && lx + 1 < b.hx + b.w && ly >= b.hy && ly < b.hy + b.h;
              if (!owned) m.m0.v.x = m.jx.v.x = m.jy.v.x = m.ux.v.x = m.uy.v.x = 0.0f;
              if (!owned2) m.m0.v.y = m.jx.v.y = m.jy.v.y = m.ux.v.y = m.uy.v.y = 0.0f;
              acc.add(m);
            }
          }
        });
        S* out2 = last ? dst + (long long)gy * g.pitch + gx2 : out + 1;
        if (walls != nullptr) {
          if (walls[(long long)gy * g.nx + gx] != 0) {
#pragma unroll
            for (int i = 0; i < 9; ++i) e[i].v.x = f[opposite_of(i)].v.x;
          }
          if (walls[(long long)gy * g.nx + gx2] != 0) {
#pragma unroll
            for (int i = 0; i < 9; ++i) e[i].v.y = f[opposite_of(i)].v.y;
          }
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          st_t(out + i * oplane, e[i].v.x);
          if (two) st_t(out2 + i * oplane, e[i].v.y);
        }
      }
    }
    if (last) break;
    __syncthreads();
    S* const t = cur;
    cur = nxt, nxt = t;
  }
  if constexpr (DIAG) {
    __syncthreads();
    block_diag_acc(acc, partials + (long long)(blockIdx.y * gridDim.x + blockIdx.x) * 5, kF64 ? &facc : nullptr);
  }
}

// One thread a node (node pair) of the first step's region, whole warps.
inline unsigned tile_threads(const Geometry& g, int tx, int ty, int steps, int nodes_per_thread) {
  const long long n = (tile_nodes(g, tx, ty, steps) + nodes_per_thread - 1) / nodes_per_thread;
  return (unsigned)std::min<long long>(kTileThreads, (n + 31) / 32 * 32);
}

// ------------------------------------------------------------------ launcher
template <int PREC> struct LaunchTile {
  using S = typename Form<PREC>::S;
  static constexpr bool kF64 = kHasFixed<typename Form<PREC>::T>;
  using CT = typename std::conditional<kF64, typename Form<PREC>::T, f32x2>::type;

  template <int MODEL, bool DIAG> static cudaError_t run(const StepArgs& a, const TilesPlan& p, int steps, cudaStream_t st) {
    auto kernel = tile_steps_kernel<MODEL, PREC, DIAG>;
    constexpr int kMaxDev = 64;
    static bool ready[kMaxDev] = {false};  // once per device: opt in to the large shared-memory carve-out
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDev) return cudaErrorInvalidDevice;
    if (!ready[dev]) {
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTileSmemMax);
      if (e != cudaSuccess) return e;
      ready[dev] = true;
    }
    const dim3 grid((a.g.nx + p.tx - 1) / p.tx, (a.g.ny + p.ty - 1) / p.ty);
    if (a.parts_used) *a.parts_used = (long long)grid.x * grid.y;
    const Coef<CT> c = make_coef<CT>(a.theta, a.tau, a.rho_ref);
    if constexpr (kF64) {
      if (!c.fixed.on) return cudaErrorInvalidValue;
    }
    return launch_step_kernel(kernel, grid, dim3(tile_threads(a.g, p.tx, p.ty, steps, kF64 ? 1 : 2)),
                              (size_t)tile_smem(a.g, p.tx, p.ty, steps, (int)sizeof(S)),
                              st, (const S*)a.src, (S*)a.dst, a.g, c, steps, p.tx, p.ty, a.wall_mask, a.partials);
  }

  template <int MODEL> static cudaError_t run_m(const StepArgs& a, const TilesPlan& p, int steps, cudaStream_t st) {
    return a.diag ? run<MODEL, true>(a, p, steps, st) : run<MODEL, false>(a, p, steps, st);
  }

  static cudaError_t steps(const StepArgs& a, const TilesPlan& p, int steps, cudaStream_t st) {
    switch (a.model) {
      case 0: return run_m<0>(a, p, steps, st);
      case 1: return run_m<1>(a, p, steps, st);
      case 2: return run_m<2>(a, p, steps, st);
      case 3: return run_m<3>(a, p, steps, st);
      case 4: return run_m<4>(a, p, steps, st);
      case 5: return run_m<5>(a, p, steps, st);
      default: return cudaErrorInvalidValue;
    }
  }
};

}  // namespace olbm

#define OLBM_DEFINE_TILE(PREC, SUFFIX)                                                                      \
  namespace olbm {                                                                                          \
  cudaError_t launch_tile_##SUFFIX(const StepArgs& a, const TilesPlan& p, int steps, cudaStream_t st) {      \
    return LaunchTile<PREC>::steps(a, p, steps, st);                                                        \
  }                                                                                                         \
  }
