// Several time steps of a small box in one launch (FP32 storage, D3Q19 or
// D3Q15, Nx even): the work-list step's jobs without the list.
//
// A box of up to a few tiles per resident block spends most of a step on
// launching it and on the launch's ragged end: 32^3, 48^3 and 64^3 took 10.3,
// 10.3 and 16.4 us per work-list launch, the jobs themselves about 6.  Here
// every block owns tiles (tile jobs of lbm_worklist.cuh, positions b, b + grid,
// ...) and takes them through `nsteps` steps: the fused jobs of its tiles, then
// their psi jobs, with two counters per tile that say how many steps of each
// job are done.  A psi job waits for the fused jobs of its neighbourhood in
// this step, a fused job of a later step for the psi jobs of its neighbourhood
// in the step before: nothing else needs an order.
//  - What a fused job reads (psi and f* within one node) comes from psi jobs it
//    has waited for and from the fused jobs those have waited for.
//  - What it overwrites (the f of the step before) was read within one node by
//    fused jobs of blocks whose psi jobs it has waited for; the psi a psi job
//    overwrites was read by fused jobs of the step before the fused jobs it has
//    waited for.
//  - The launch is cooperative, so every block is resident, and a block waits
//    only for jobs that come earlier in every block's own order: the earliest
//    unfinished phase of any block can always go on.
// Waits are bounded (KParams::spin_limit, once per block: after a wait that gave
// up, kErrTimeout is set and the block goes on without waiting).
// Populations and psi written in this launch are read with plain loads after an
// acquire, or through L2.  The arithmetic is that of the two-pass kernels.
#include <algorithm>

#include "lbm_device.cuh"
#include "lbm_internal.h"
#include "lbm_pair.cuh"
#include "lbm_pair15.cuh"
#include "lbm_worklist.cuh"

namespace lbm {
namespace {

constexpr int kBlocks = 7;  // resident blocks per SM the registers are set for
// Tiles per block up to which a box is stepped here: per step, this kernel /
// the list, 32^3 4.9 / 9.3 us, 48^3 7.2 / 12.1, 64^3 10.2 / 18.9, 80^3 18.1 / 26.6,
// 96^3 34.4 / 38.7, 104^3 (4.1 tiles per block) 47.0 / 45.9, 112^3 (5.2) 59.3 / 53.1;
// D3Q15 64^3 9.1 / 16.4, 96^3 29.1 / 35.0, 104^3 38.8 / 41.1, 112^3 50.4 / 47.5.  (At 6, 7
// and 8 blocks per SM 64^3 takes 13.0, 10.2 and 11.3 us, 80^3 20.5, 18.1 and 19.5, 96^3
// 33.6, 34.5 and 34.6.  At 7, 72 registers, the D3Q19 kernels spill 84 to 136 bytes,
// the D3Q15 ones 48 to 60.)
constexpr int max_tiles(int q) { return q == 15 ? 5 : 4; }

struct StepBuffers {
  float *g[2], *psi[2];  // [0]: the state the launch starts from
};

template <int OP, int EOS, bool DF, int Q>
__global__ void __launch_bounds__(NTH, kBlocks)
    steps_kernel(const StepBuffers B, const KParams P, const TileMap G, int nsteps, int *__restrict__ fused_done,
                 int *__restrict__ psi_done, int stamp, unsigned *__restrict__ err) {
  const int lane = threadIdx.x, tid = threadIdx.y * TXP + lane, nf = P.nz * G.T;
  unsigned e = 0;
  // This block alone counts its tiles: anything but stamp - 1 means that the counters are not those this launch was
  // made for (a launch captured in a graph and replayed), and nothing would be waited for.
  if (__ldcg(fused_done + blockIdx.x) != stamp - 1) {
    if (tid == 0) atomicOr(err, kErrTimeout);
    return;
  }
  for (int s = 0; s < nsteps; ++s) {
    const float *g_in = B.g[s & 1], *psi_in = B.psi[s & 1];
    float *g_out = B.g[(s & 1) ^ 1], *psi_out = B.psi[(s & 1) ^ 1];
#pragma unroll 1
    for (int j = blockIdx.x; j < nf; j += gridDim.x) {
      int z = j / G.T, t = j - z * G.T;
      asm volatile("" : "+r"(z), "+r"(t));  // keep the row offsets out of the registers across jobs
      if (s > 0 && !wait_for_jobs(G, true, P, psi_done, 0, nf, z, t, lane, stamp + s - 1 + P.wait_bias,
                                  e & kErrTimeout ? 0 : P.spin_limit))
        e |= kErrTimeout;
      __syncwarp();
      int x, y;
      if (tile_node(G, true, P, t, tid, x, y)) {
        if constexpr (Q == 15)
          fused_pair15_at<float, true, true, false, PlainLoad, PlainLoad>(g_in, g_out, psi_in, P, x, y, z);
        else
          fused_pair_at<float, OP, true, true, false, PlainLoad, PlainLoad>(g_in, g_out, psi_in, P, x, y, z, Rates<V2>(P));
      }
      __syncthreads();
      if (tid == 0) counter_release_add(fused_done + LBM_IDX(j, nf), 1);
    }
#pragma unroll 1
    for (int j = blockIdx.x; j < nf; j += gridDim.x) {
      int z = j / G.T, t = j - z * G.T;
      asm volatile("" : "+r"(z), "+r"(t));
      if (!wait_for_jobs(G, true, P, fused_done, 0, nf, z, t, lane, stamp + s + P.wait_bias,
                         e & kErrTimeout ? 0 : P.spin_limit))
        e |= kErrTimeout;
      __syncwarp();
      int x, y;
      if (tile_node(G, true, P, t, tid, x, y)) {
        if constexpr (Q == 15)
          psi_pair15_at_l2<float, EOS, DF, true, false>(g_out, psi_out, P, x, y, z, e);
        else
          psi_pair_at_l2<float, EOS, DF, true, false>(g_out, psi_out, P, x, y, z, e);
      }
      __syncthreads();
      if (tid == 0) counter_release_add(psi_done + LBM_IDX(j, nf), 1);
    }
  }
  if (e) atomicOr(err, e);
}

using Kernel = void (*)(const StepBuffers, const KParams, const TileMap, int, int *, int *, int, unsigned *);

template <int OP, int Q>
Kernel kernel_by_eos(int eos, bool df) {
  switch (eos) {
    case kEosCS: return df ? steps_kernel<OP, kEosCS, true, Q> : steps_kernel<OP, kEosCS, false, Q>;
    case kEosExp: return steps_kernel<OP, kEosExp, false, Q>;  // (its FP32 arithmetic is the same either way)
    default: return steps_kernel<OP, kEosNone, false, Q>;
  }
}

Kernel kernel_of(const KParams &P, int op, bool df) {
  if (P.q == 15) return kernel_by_eos<kNonOrth, 15>(P.eos, df);
  return op == kNonOrth ? kernel_by_eos<kNonOrth, 19>(P.eos, df) : kernel_by_eos<kOrth, 19>(P.eos, df);
}

}  // namespace

// Thread blocks of the launch, as even a share of the tiles as fits the device; 0: not a box for this kernel.
cudaError_t steps_grid(const KParams &P, int precision, int *grid) {
  *grid = 0;
  if (precision != kF32 || P.px != P.nx || P.px % 2 != 0) return cudaSuccess;
  const TileMap G = tile_map(P);
  int dev = 0, sms = 0, coop = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (e != cudaSuccess) return e;
  const long long nf = (long long)P.nz * G.T, most = (long long)kBlocks * sms;
  if (!coop || !G.lin || nf > most * max_tiles(P.q)) return cudaSuccess;
  const long long share = (nf + most - 1) / most;
  *grid = (int)((nf + share - 1) / share);
  return cudaSuccess;
}

size_t steps_counters(const KParams &P) { return 2 * (size_t)P.nz * tile_map(P).T; }

cudaError_t launch_steps(const KParams &P, int op, bool df, void *g_in, void *g_out, void *psi_in, void *psi_out,
                         int grid, int *counters, int nsteps, int stamp, unsigned *err, cudaStream_t s) {
  StepBuffers B{{(float *)g_in, (float *)g_out}, {(float *)psi_in, (float *)psi_out}};
  KParams Pc = P;
  TileMap G = tile_map(P);
  int *fused_done = counters, *psi_done = counters + (size_t)P.nz * G.T;
  void *args[] = {(void *)&B, (void *)&Pc, (void *)&G, (void *)&nsteps, (void *)&fused_done, (void *)&psi_done,
                  (void *)&stamp, (void *)&err};
  return cudaLaunchCooperativeKernel((const void *)kernel_of(P, op, df), dim3(grid), dim3(TXP, kRows), args, 0, s);
}

}  // namespace lbm
