// Two-pass kernels for the FP32-arithmetic forms with two x-adjacent nodes per
// thread (rows of even length, KParams::px).
//
// A thread owns the pair (x, x+1), x even.  Populations that arrive along
// e_x = 0 come from an aligned pair (x, x+1) of the source row: one 64-bit
// load (FP32 storage) or 32-bit load (FP16 storage).  Those with e_x = +1 come
// from (x-1, x) and those with e_x = -1 from (x+1, x+2), read as two scalars.
// The psi neighbourhood is read the same way: the nine rows of the stencil as
// aligned pairs plus x-1 and x+2 where a direction moves in x.  All arithmetic
// of the two nodes runs on packed FP32 pairs (V2): per node it is the
// arithmetic of the one-node kernels in lbm_kernels.cu, and a packed
// instruction issues the work of two nodes.
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "lbm_device.cuh"
#include "lbm_internal.h"
#include "lbm_pair.cuh"
#include "lbm_pair15.cuh"
#include "lbm_q15.cuh"

namespace lbm {
namespace {

// R4: a block's 128 pairs as 32 of each of four rows (every block full: rows4).
template <bool R4 = false>
__device__ __forceinline__ bool pair_of_thread(const KParams &P, PairX &px, int &y, int &z) {
  if (R4) {
    const unsigned q = blockIdx.x * 32, w = (unsigned)P.px / 2, by = P.pair_m ? __umulhi(q, P.pair_m) : q / w;
    y = (int)(4 * by + threadIdx.x / 32);
    z = blockIdx.z;
    px = pair_x(P, 2 * (int)(q - by * w + threadIdx.x % 32));
    return true;
  }
  const unsigned p = blockIdx.x * blockDim.x + threadIdx.x, W = (unsigned)P.px / 2;
  y = (int)(P.pair_m ? __umulhi(p, P.pair_m) : p / W);
  z = blockIdx.z;
  px = pair_x(P, 2 * (int)(p - y * W));
  return y < P.ny;
}

// Twelve blocks an SM (40 registers): 256^3 FP32 217 -> 201 us against 48 registers
// (the loads in flight need the warps; 205 with plain loads), FP16 183 -> 180.
// ODD: rows padded for an odd Nx, set for FP16 storage only (FP32 sums round alike
// either way), with eight blocks (the scalar sums spill 68 bytes at twelve).
template <typename S, int EOS, bool DF, bool ODD>
__global__ void __launch_bounds__(128, ODD ? 8 : 12) psi_pair_kernel(const S *g, float *__restrict__ psi,
                                                       const KParams P, unsigned *__restrict__ err) {
  chain_wait();
  PairX px;
  int y, z;
  if (!pair_of_thread(P, px, y, z)) return;
  const Nbhd nb(px.x, y, z, P);
  const V2 drho = pull_drho<S, PlainLoad, ODD>(g, (unsigned)P.np, P, nb, px);
  unsigned e = 0;
  store_pair_psi<true>(psi, P, px.x, (unsigned)nb.self, psi_pair<EOS, DF>(pad_lane<true>(drho, P, px.x), P, e));
  if (e) atomicOr(err, e);
}

// Six blocks of 128 an SM (80 registers) for even boxes: FP16 256^3 fused 263 -> 258
// us, FP32 192^3 orthogonal 164 -> 161; odd boxes, whose nodes collide in scalar code,
// would spill, five there (96 registers).
template <typename S, int OP, bool SIGMA, bool ODD, bool R4 = false>
__global__ void __launch_bounds__(128, ODD ? 5 : 6) fused_pair_kernel(const S *g_in, S *__restrict__ g_out,
                                                         const float *psi, const KParams P) {
  chain_wait();
  PairX px;
  int y, z;
  if (!pair_of_thread<R4>(P, px, y, z)) return;
  const Nbhd nb(px.x, y, z, P);
  V2 f[19];
  pull_pair<S, PlainLoad, ODD>(g_in, (unsigned)P.np, nb, px, f);
  V2 p[19];
  gather_psi_pair<PlainLoad>(psi, nb, px, p);
  if constexpr (ODD)
    force_collide_lanes<S, OP, SIGMA, 19>(f, p, P);
  else
    force_collide_pair<OP, SIGMA>(f, p, P, Rates<V2>(P), OP);
  store_pair_f<S, ODD>(g_out, P, px.x, (unsigned)nb.self, f);
}

// ------------------------------------------------------------------ D3Q15
// The same two-node scheme for the D3Q15 variant (lbm_pair15.cuh).

template <typename S, int EOS, bool DF, bool ODD>
__global__ void __launch_bounds__(128, ODD ? 8 : 12) psi_pair15_kernel(const S *g, float *__restrict__ psi,
                                                         const KParams P, unsigned *__restrict__ err) {
  chain_wait();
  PairX px;
  int y, z;
  if (!pair_of_thread(P, px, y, z)) return;
  const Nbhd nb(px.x, y, z, P);
  V2 f[q15::kQ];
  pull_pair15<S, PlainLoad, ODD>(g, (unsigned)P.np, nb, px, f);
  V2 drho;
  if constexpr (ODD)
    drho = drho_lanes<S, q15::kQ>(f);
  else
    drho = q15::drho(f);
  unsigned e = 0;
  store_pair_psi<true>(psi, P, px.x, (unsigned)nb.self, psi_pair<EOS, DF>(pad_lane<true>(drho, P, px.x), P, e));
  if (e) atomicOr(err, e);
}

template <typename S, bool SIGMA, bool ODD>
__global__ void __launch_bounds__(128) fused_pair15_kernel(const S *g_in, S *__restrict__ g_out,
                                                           const float *psi, const KParams P) {
  chain_wait();
  PairX px;
  int y, z;
  if (!pair_of_thread(P, px, y, z)) return;
  if constexpr (ODD) {
    const Nbhd nb(px.x, y, z, P);
    V2 f[q15::kQ], p[q15::kQ];
    pull_pair15<S, PlainLoad, true>(g_in, (unsigned)P.np, nb, px, f);
    gather_psi_pair15<PlainLoad>(psi, nb, px, p);
    force_collide_lanes<S, kNonOrth, SIGMA, q15::kQ>(f, p, P);
    store_pair15_f<S, ODD>(g_out, P, px.x, (unsigned)nb.self, f);
  } else {
    fused_pair15_at<S, SIGMA, false, ODD, PlainLoad, PlainLoad>(g_in, g_out, psi, P, px.x, y, z);
  }
}

dim3 pair_grid(const KParams &P) { return plane_grid(P.px / 2 * P.ny, P.nz); }

template <typename S, bool DF, bool ODD>
cudaError_t psi_pair_dispatch(const KParams &P, const void *g, void *psi, unsigned *err, const Launch &L) {
  const dim3 grid = pair_grid(P), block(kThreads);
  auto run = [&](auto kernel) {
    return launch_chained(P.n >= kChainPairs, kernel, grid, block, L.stream, (const S *)g, (float *)psi, P, err);
  };
  if (P.q == 15) {
    switch (P.eos) {
      case kEosCS: return run(psi_pair15_kernel<S, kEosCS, DF, ODD>);
      case kEosExp: return run(psi_pair15_kernel<S, kEosExp, DF, ODD>);
      default: return run(psi_pair15_kernel<S, kEosNone, false, false>);
    }
  }
  switch (P.eos) {
    case kEosCS: return run(psi_pair_kernel<S, kEosCS, DF, ODD>);
    case kEosExp: return run(psi_pair_kernel<S, kEosExp, DF, ODD>);
    default: return run(psi_pair_kernel<S, kEosNone, false, false>);
  }
}

// Rows that fill blocks of 32 pairs x 4 rows.  The orthogonal FP16 fused pass, bound
// by its issue slots, runs better on those (the rows of a block share psi in L1):
// steps of 128^3 61.2 -> 61.0 us, 64 x 200 x 200 74.1 -> 73.5, 192^3 194.0 -> 191.4, 256^3
// 449 -> 444, 320^3 876 -> 863 (64^3 12.1 / 12.2).  The non-orthogonal one does not (256^3
// fused 263 -> 264), FP32 loses (375 -> 401), and the psi pass too (201 -> 208).
bool rows4(const KParams &P) { return P.px % 64 == 0 && P.ny % 4 == 0; }

template <typename S, bool ODD>
cudaError_t fused_pair_dispatch(const KParams &P, int op, bool sigma, const void *g_in, void *g_out,
                                const void *psi, const Launch &L) {
  const dim3 grid = pair_grid(P), block(kThreads);
  const S *gi = (const S *)g_in;
  S *go = (S *)g_out;
  const float *pp = (const float *)psi;
  auto run = [&](auto kernel) { return launch_chained(P.n >= kChainPairs, kernel, grid, block, L.stream, gi, go, pp, P); };
  if (P.q == 15) return sigma ? run(fused_pair15_kernel<S, true, ODD>) : run(fused_pair15_kernel<S, false, ODD>);
  if (op == kNonOrth)
    return sigma ? run(fused_pair_kernel<S, kNonOrth, true, ODD>) : run(fused_pair_kernel<S, kNonOrth, false, ODD>);
  if constexpr (!ODD && std::is_same<S, __half>::value)
    if (rows4(P))
      return sigma ? run(fused_pair_kernel<S, kOrth, true, ODD, true>) : run(fused_pair_kernel<S, kOrth, false, ODD, true>);
  return sigma ? run(fused_pair_kernel<S, kOrth, true, ODD>) : run(fused_pair_kernel<S, kOrth, false, ODD>);
}

// Batched boxes, two-pass step, psi pass: work item w = (box, tile_x | tile_y
// << 16, z0, z1) is a TXP x TY tile of pairs (2 TXP x TY nodes) of one box
// through planes [z0, z1).  The fused pass (batch_flat_fused_kernel) reads
// level in = cur ^ parity (populations and psi) and writes the populations of
// level in ^ 1; this pass then evaluates psi of level in ^ 1, so after a step
// psi of the current level is always valid.  (A flat grid of one plane per
// block, as for the fused pass, measured 2 % slower here.)
// ODD: some box has padded rows (in code of their own: 32 even boxes, FP32, stepped in
// 482 us with the pads' stores compiled in, 400 without).
template <typename S, int EOS, int TXP, int TY, bool ODD>
__global__ void __launch_bounds__(TXP *TY) batch_psi_kernel(const BatchBox *__restrict__ boxes,
                                                            const int4 *__restrict__ items, int nitems, int parity,
                                                            unsigned *__restrict__ err) {
  __shared__ BatchBox bb;
  const int tid = threadIdx.y * TXP + threadIdx.x;
  unsigned e = 0;
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    const int4 w = items[it];
    __syncthreads();  // every thread is done with the previous item's descriptor
    {
      const int *src = (const int *)(boxes + w.x);
      int *dst = (int *)&bb;
      for (int k = tid; k < (int)(sizeof(BatchBox) / sizeof(int)); k += TXP * TY) dst[k] = src[k];
    }
    __syncthreads();
    const KParams &P = bb.P;
    const int in = bb.cur ^ parity;
    const int x = (w.y & 0xffff) * (2 * TXP) + 2 * threadIdx.x, y = (w.y >> 16) * TY + threadIdx.y;
    if (x >= P.nx || y >= P.ny) continue;
    const PairX px{x, x == 0 ? P.nx - 1 : x - 1, x + 2 >= P.nx ? x + 2 - P.nx : x + 2};
    const S *g = (const S *)bb.g[in ^ 1];
    float *psi = bb.psi[in ^ 1];
    for (int z = w.z; z < w.w; ++z) {
      const Nbhd nb(x, y, z, P, ODD ? P.px : P.nx);
      const V2 drho = pull_drho<S, PairIO<S>, ODD>(g, (unsigned)(ODD ? P.np : P.n), P, nb, px);
      store_pair_psi<ODD>(psi, P, x, (unsigned)nb.self, psi_pair<EOS, false>(pad_lane<ODD>(drho, P, x), P, e));
    }
  }
  if (e) atomicOr(err, e);
}

// Threads per SM the flat fused kernel's registers are set for: 640 (at most 102 registers a thread; both
// operators fit without spilling, the orthogonal one took 108 unbounded; 80 registers spilled and was slower).
constexpr int kFlatFusedThreadsPerSM = 640;

// The fused pass of a batch as a flat grid, one launch per operator: block b
// is one plane of one 2 TXP x TY tile of one box, block_box[offset + b] names
// the box, whose first block is its descriptor's qbase; planes are numbered
// box by box, tiles x-fastest within a plane.  One node pair per thread and no
// loop, as in fused_pair_kernel: a persistent kernel looping over the planes of
// an item held 128 registers (16 warps per SM) and reached 0.86 of the copy
// bandwidth, this one holds 96 (5 blocks of 128 threads) and 0.94.
template <typename S, int OP, int TXP, int TY, bool ODD>
__global__ void __launch_bounds__(TXP *TY, kFlatFusedThreadsPerSM / (TXP * TY)) batch_flat_fused_kernel(const BatchBox *__restrict__ boxes,
                                                                   const int *__restrict__ block_box, int offset,
                                                                   int parity) {
  const int gb = offset + (int)blockIdx.x;
  const int slot = __ldg(block_box + gb);
  const BatchBox &bb = boxes[slot];  // read where used (cached; a copy to shared memory measured the same)
  const KParams &P = bb.P;
  const int ntx = (P.nx + 2 * TXP - 1) / (2 * TXP), nty = (P.ny + TY - 1) / TY, T = ntx * nty;
  const int local = gb - bb.qbase, z = local / T, t = local - z * T;
  const int x = (t % ntx) * (2 * TXP) + 2 * threadIdx.x, y = (t / ntx) * TY + threadIdx.y;
  if (x >= P.nx || y >= P.ny || z >= P.nz) return;
  const int in = bb.cur ^ parity;
  fused_pair_at<S, OP, true, false, ODD>((const S *)bb.g[in], (S *)bb.g[in ^ 1], bb.psi[in], P, x, y, z, Rates<V2>(P));
}

// The fused and psi kernels of one step for a storage type and tile shape;
// with query set, per_sm receives their resident blocks per SM instead.
template <typename S, int TXP, int TY, bool ODD>
cudaError_t batch_pair_shape(int eos, const BatchBox *boxes, const int4 *items, int nitems, const int *block_box,
                             const int fused_blocks[2], int parity, int sms, int per_sm[2], bool query, unsigned *err,
                             cudaStream_t s) {
  using K = void (*)(const BatchBox *, const int4 *, int, int, unsigned *);
  K kpsi;
  switch (eos) {
    case kEosCS: kpsi = batch_psi_kernel<S, kEosCS, TXP, TY, ODD>; break;
    case kEosExp: kpsi = batch_psi_kernel<S, kEosExp, TXP, TY, ODD>; break;
    default: kpsi = batch_psi_kernel<S, kEosNone, TXP, TY, ODD>; break;
  }
  if (query) {
    per_sm[0] = 0;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm[1], kpsi, TXP * TY, 0);
  }
  // fused pass: the flat launches (non-orthogonal boxes' blocks first in block_box, then the orthogonal ones)
  if (fused_blocks[0] > 0)
    batch_flat_fused_kernel<S, kNonOrth, TXP, TY, ODD><<<fused_blocks[0], dim3(TXP, TY), 0, s>>>(boxes, block_box, 0, parity);
  if (fused_blocks[1] > 0)
    batch_flat_fused_kernel<S, kOrth, TXP, TY, ODD><<<fused_blocks[1], dim3(TXP, TY), 0, s>>>(boxes, block_box, fused_blocks[0],
                                                                                       parity);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int grid = std::max(1, std::min(sms * std::max(per_sm[1], 1), nitems));
  kpsi<<<grid, dim3(TXP, TY), 0, s>>>(boxes, items, nitems, parity, err);
  return cudaGetLastError();
}

template <typename S, bool ODD>
cudaError_t batch_pair_tile(int tile, int eos, const BatchBox *boxes, const int4 *items, int nitems,
                            const int *block_box, const int fused_blocks[2], int parity, int sms, int per_sm[2],
                            bool query, unsigned *err, cudaStream_t s) {
  switch (tile) {
    case kTile32x4:
      return batch_pair_shape<S, 16, 4, ODD>(eos, boxes, items, nitems, block_box, fused_blocks, parity, sms, per_sm, query,
                                        err, s);
    case kTile64x4:
      return batch_pair_shape<S, 32, 4, ODD>(eos, boxes, items, nitems, block_box, fused_blocks, parity, sms, per_sm, query,
                                        err, s);
    default:
      return batch_pair_shape<S, 16, 8, ODD>(eos, boxes, items, nitems, block_box, fused_blocks, parity, sms, per_sm, query,
                                        err, s);
  }
}

cudaError_t batch_pair_dispatch(int precision, int tile, int eos, bool odd, const BatchBox *boxes, const int4 *items,
                                int nitems, const int *block_box, const int fused_blocks[2], int parity, int sms,
                                int per_sm[2], bool query, unsigned *err, cudaStream_t s) {
  if (precision != kF32 && precision != kF16) return cudaErrorInvalidValue;
  auto launch = precision == kF32 ? (odd ? batch_pair_tile<float, true> : batch_pair_tile<float, false>)
                                  : (odd ? batch_pair_tile<__half, true> : batch_pair_tile<__half, false>);
  return launch(tile, eos, boxes, items, nitems, block_box, fused_blocks, parity, sms, per_sm, query, err, s);
}

}  // namespace

bool pair_supported(const KParams &P, int precision) { return precision != kF64 && P.px % 2 == 0; }

cudaError_t batch_pair_occupancy(int precision, int eos, int tile, bool odd, int per_sm[2]) {
  const int none[2] = {0, 0};
  return batch_pair_dispatch(precision, tile, eos, odd, nullptr, nullptr, 0, nullptr, none, 0, 0, per_sm, true, nullptr,
                             0);
}

cudaError_t launch_batch_pair(int precision, int eos, int tile, bool odd, const BatchBox *boxes, const int4 *items,
                              int nitems, const int *block_box, const int fused_blocks[2], int parity, int sms,
                              const int per_sm[2], unsigned *err, cudaStream_t s) {
  int ps[2] = {per_sm[0], per_sm[1]};
  return batch_pair_dispatch(precision, tile, eos, odd, boxes, items, nitems, block_box, fused_blocks, parity, sms, ps,
                             false, err, s);
}

cudaError_t launch_psi_pair(const KParams &P, int precision, const void *g, void *psi, unsigned *err,
                            const Launch &L, bool df) {
  auto launch = df ? psi_pair_dispatch<float, true, false> : psi_pair_dispatch<float, false, false>;
  if (precision == kF16)
    launch = P.px != P.nx ? (df ? psi_pair_dispatch<__half, true, true> : psi_pair_dispatch<__half, false, true>)
                          : (df ? psi_pair_dispatch<__half, true, false> : psi_pair_dispatch<__half, false, false>);
  return launch(P, g, psi, err, L);
}

cudaError_t launch_fused_pair(const KParams &P, int precision, int op, bool sigma, const void *g_in, void *g_out,
                              const void *psi, const Launch &L) {
  const bool odd = P.px != P.nx;
  auto launch = precision == kF32 ? (odd ? fused_pair_dispatch<float, true> : fused_pair_dispatch<float, false>)
                                  : (odd ? fused_pair_dispatch<__half, true> : fused_pair_dispatch<__half, false>);
  return launch(P, op, sigma, g_in, g_out, psi, L);
}

}  // namespace lbm
