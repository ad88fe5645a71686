// lbm_reduce.cu -- final, fixed-order reduction of the per-block diagnostics
// partials written by the step and diagnostics kernels, and the shared grid
// shape of the node-parallel kernels.
#include "lbm_kernels.cuh"

namespace olbm {

long long node_blocks(const Geometry& g) {
  const dim3 gr = grid_of(g);
  return (long long)gr.x * gr.y;
}

long long diag_blocks(const Geometry& g) {
  const dim3 gr = diag_grid(g);
  return (long long)gr.x * gr.y;
}

long long step_blocks(const Geometry& g, const LaunchCfg& k, int prec) {
  const dim3 gr = step_grid(g, k, prec);
  const long long one = (long long)gr.x * gr.y;
  if (!step2_applies(prec, g, k)) return one;
  const dim3 g2 = step2_grid(g, k, prec);
  return std::max(one, (long long)g2.x * g2.y);  // kind 2 also launches single steps
}

int stream_tile_width(int prec) { return stream_width(prec); }

int step2_tile_width(int prec) { return stream2_width(prec); }

bool uses_step2(int prec, const Geometry& g, const LaunchCfg& k) { return step2_applies(prec, g, k); }

long long step2_blocks(const Geometry& g, const LaunchCfg& k, int prec) {
  const dim3 gr = step2_grid(g, k, prec);
  return (long long)gr.x * gr.y;
}

// The ring fits three times in an SM's shared memory for both shifted forms;
// FP16 is compiled for three CTAs (registers), FP32 (160 threads) fits them.
#ifndef OLBM_STREAM_CTAS
#define OLBM_STREAM_CTAS 3
#endif
int stream_ctas_per_sm(int) { return OLBM_STREAM_CTAS; }

// Fixed-order final sums of the block partials, one block a diagnosed step: out[0..4] as in
// lbm_diagnostics (mass gets rho_ref for every finite node), out[5] = t of the last step;
// non-finite nodes of every step are added to *sticky.
//
// A sum alone is a launch, two events and a stream wait for the host and breaks the chain of
// programmatically launched steps; on small lattices that was most of a diagnosed step
// (64^2, diagnostics every step: FP32 10.9 -> 3.8 us, FP64 10.9 -> 5.3).
// 128 threads: the butterfly of every warp goes through the FP64 pipe of one SM, which holds it longer
// than more threads save at any number of partials (a call of one diagnosed step with its sum, us, by
// threads 128 / 256 / 512: 64^2 FP32 8.3 / 10.3 / 12.4, 1024^2 FP16 20.6 / 20.6 / 23.6).
constexpr int kFinalThreads = 128;
__global__ void __launch_bounds__(kFinalThreads) finalize_kernel(FinalJobs jobs, double rho_ref, long long nodes,
                                                                 double* __restrict__ out,
                                                                 unsigned long long* __restrict__ sticky) {
  const double* __restrict__ partials = jobs.partials[blockIdx.x];
  const int nparts = jobs.nparts[blockIdx.x];
  double v[kNDiag] = {0.0, 0.0, 0.0, 0.0, 0.0};
  for (int j = threadIdx.x; j < nparts; j += kFinalThreads)
#pragma unroll
    for (int k = 0; k < kNDiag; ++k) v[k] += partials[(long long)j * kNDiag + k];
  double tot[kNDiag];
  block_sum<kNDiag, kFinalThreads>(v, tot);
  if (threadIdx.x == 0) {
    const double bad = tot[4];
    if (blockIdx.x + 1 == gridDim.x) {
      out[0] = tot[0] + rho_ref * (double)(nodes - (long long)bad);
      out[1] = tot[1];
      out[2] = tot[2];
      out[3] = tot[3];
      out[4] = bad;
      out[5] = (double)jobs.t[blockIdx.x];
    }
    if (bad > 0.0 && sticky != nullptr) atomicAdd(sticky, (unsigned long long)bad);
  }
}

cudaError_t launch_finalize(const FinalJobs& jobs, double rho_ref, long long nodes, double* out,
                            unsigned long long* sticky, cudaStream_t st) {
  finalize_kernel<<<jobs.count, kFinalThreads, 0, st>>>(jobs, rho_ref, nodes, out, sticky);
  return cudaGetLastError();
}

}  // namespace olbm
