// Single-pass time step on an ordered work list (FP32-arithmetic forms, D3Q19 and
// D3Q15, Nx even; batches of D3Q19 boxes with any Nx): one persistent launch per
// step runs both passes of the two-pass step as interleaved work.
//
// Work item k is a pair of tile jobs (128 node pairs of one plane that follow
// each other in row order, one per thread; see tile_map):
//   fused job (z, tile): the fused pass (Eqs. 4-6 and 15, pull streaming of
//     Eq. 5): reads f(t) and psi(t), writes f*(t); then counts itself done;
//   psi job (z', tile'): the psi pass of the next step: rho(t+1) from the
//     pulled f*(t) (Eq. 6), the EOS, psi(t+1).  It needs the fused jobs of
//     planes z'-1..z'+1 on its rows and the rows next to them (periodic) and
//     pulls their output through L2, where it still is.
// The host builds the list (and checks it): fused jobs plane by plane; each
// psi job in the first free item at least psi_lag items (3/8 or 5/8 of a wave of
// the grid; batches: half a wave) after the last fused job it reads: by the time
// a block reaches the psi job those fused jobs are normally finished, so the
// wait is one poll, while writer and reader stay close enough for the
// populations to be still in L2 (a whole wave waits less but re-reads about twice
// as much from DRAM, and is slower; a quarter waits more).
//
// Block b starts with item b; from then on it claims the next unclaimed item
// (one atomic fetch per item, issued when an item starts and read when it
// ends), so blocks take items in list order whatever their speed.  (With the
// static order b, b + grid, ..., blocks drifted up to five items apart within
// a wave, and the psi jobs of the fast ones waited on the slow ones: 0.556
// against 0.528 ms per 256^3 step, with 64 x 4 tiles.)  Claims are in increasing order
// and the launch is cooperative (every block resident): a block holding an
// unfinished fused job is busy with an earlier item, so the psi job of the
// lowest unfinished item waits only on fused jobs that are finished or
// running, and progress needs no timing assumption.  Waits are bounded all
// the same (KParams::spin_limit; a wait that gives up sets kErrTimeout and
// the launch still ends).
//
// What this buys over two launches: the psi jobs' FP64 EOS runs on the same
// SMs while the fused jobs stream HBM, and the populations they pull come from
// L2 (writer and reader are about two planes plus the lag apart):
// DRAM traffic per node is f(t) read and f*(t) written once plus psi read and
// written once (2 x 19 x s + 8 bytes) against 3 x 19 x s + 8.  The
// arithmetic and its order are those of the two-pass kernels, so the results
// are equal bit for bit.
//
// Counters: done[z * T + tile] counts the launches in which fused job
// (z, tile) has finished (one release increment after a block barrier), so a
// psi job of launch `stamp` waits for done >= stamp and nothing is ever reset.
// done[nz * T + 16] counts the item claims: exactly nitems per launch (one
// for every item a block runs; the one made during a block's last item names
// no item), so launch `stamp` claims numbers (stamp - 1) * nitems onwards,
// modulo 2^32.
#include <cuda_fp16.h>

#include <algorithm>
#include <vector>

#include "lbm_device.cuh"
#include "lbm_internal.h"
#include "lbm_pair.cuh"
#include "lbm_pair15.cuh"
#include "lbm_worklist.cuh"

namespace lbm {
namespace {

// Resident blocks per SM the register budgets are set for.  The fused jobs wait
// for memory most of the time, so a block more is worth some spilled registers,
// up to a point; taking the force from psi before the populations are pulled
// (FORCE_FIRST) is what lets a thread live on 80 or fewer.  Steps at 6, 7 and 8
// blocks: 256^3 FP32 non-orthogonal 508, 523 and 583 us, orthogonal 526, 538 and 603,
// D3Q15 436 (6 and 7) and 429; 192^3 218, 223 and 249, 224, 228 and 258, 187 and 185;
// FP16 storage at 6 and 7 256^3 485 and 455, 192^3 208 and 195.  Batches take 6 (848
// against 842 us for 64 boxes at 7, with 180 bytes spilled).
constexpr int kBatchBlocks = 6;
// FP16 batches with odd boxes collide those node by node (force_collide_lanes): 372 bytes spilled at 6 blocks.
constexpr int kOddHalfBatchBlocks = 5;
template <typename S> __host__ __device__ constexpr int min_blocks(int q) {
  return q == 15 ? 8 : std::is_same<S, __half>::value ? 7 : 6;
}
// The psi jobs convert to and from FP64 with the conversion instructions, not
// the integer path of the psi pass kernel (the same results): this kernel is
// not bound by the FP64 unit, and the integer work cost 1 % (FP32 storage) and
// 3 % (FP16) of a 256^3 step on GB300.
constexpr bool kIntCvt = false;

// The item claim number c of this launch names: gridDim.x + c.  Every launch
// makes exactly nitems claims, so c < nitems; a claim outside that range
// (claim counter and launch count out of step) ends the block's loop and is
// reported as a timeout: the list could not be followed.
__device__ __forceinline__ int next_item(unsigned c, int nitems, unsigned &e) {
  if (c >= (unsigned)nitems) {
    e |= kErrTimeout;
    return nitems;
  }
  return (int)gridDim.x + (int)c;
}

// item: x = fused plane (or -1), y = its tile, z = psi plane (or -1), w = its tile.
// Q: 19 (both operators) or 15 (the D3Q15 non-orthogonal variant).  LIN: TileMap::lin.
// The Eq. 16 term is compiled in (a zero coefficient switches it off).
template <typename S, int OP, bool LIN, int EOS, bool DF, int Q>
__global__ void __launch_bounds__(NTH, min_blocks<S>(Q))
    queue_kernel(const S *__restrict__ g_in, S *__restrict__ g_out, const float *__restrict__ psi_in,
                 float *__restrict__ psi_out, const KParams P, const TileMap G, const int4 *__restrict__ items,
                 int nitems, int *__restrict__ done, int stamp, unsigned *__restrict__ err) {
  const int lane = threadIdx.x, row = threadIdx.y;
  unsigned e = 0;
  // the claimed next item, by item parity: thread 0 writes slot i & 1 before item i's barrier and the block
  // reads it after that barrier; the slot is written again two items later, after every thread has passed
  // item i + 1's barrier
  __shared__ int s_next[2];
  unsigned *claims = (unsigned *)(done + P.nz * G.T + 16);
  const unsigned base = (unsigned)(stamp - 1) * (unsigned)nitems;
  int k = blockIdx.x;
  int par = 0;
#pragma unroll 1
  while (k < nitems) {
    unsigned claim = 0;
    if (lane == 0 && row == 0) claim = atomicAdd(claims, 1u);  // the next item: gridDim.x + claim - base
    const int4 it = __ldg(items + k);
    if (it.x >= 0) {
      int z = it.x, t = it.y;
      asm volatile("" : "+r"(z), "+r"(t));  // keep the row offsets out of the registers across items
      int x, y;
      if (tile_node(G, LIN, P, t, row * TXP + lane, x, y)) {
        if constexpr (Q == 15)
          fused_pair15_at<S, true, true, false>(g_in, g_out, psi_in, P, x, y, z);
        else
          fused_pair_at<S, OP, true, true, false>(g_in, g_out, psi_in, P, x, y, z, Rates<V2>(P));
      }
      if (lane == 0 && row == 0) s_next[par] = next_item(claim - base, nitems, e);
      __syncthreads();
      if (lane == 0 && row == 0) counter_release_add(done + LBM_IDX(z * G.T + t, P.nz * G.T), 1);
    } else {
      if (lane == 0 && row == 0) s_next[par] = next_item(claim - base, nitems, e);
      __syncthreads();
    }
    const int kn = s_next[par];
    par ^= 1;
    if (it.z >= 0) {
      int z = it.z, t = it.w;
      asm volatile("" : "+r"(z), "+r"(t));
      if (!wait_for_jobs(G, LIN, P, done, 0, P.nz * G.T, z, t, lane, stamp + P.wait_bias, P.spin_limit))
        e |= kErrTimeout;
      int x, y;
      if (tile_node(G, LIN, P, t, row * TXP + lane, x, y)) {
        if constexpr (Q == 15)
          psi_pair15_at_l2<S, EOS, DF, kIntCvt, false>(g_out, psi_out, P, x, y, z, e);
        else
          psi_pair_at_l2<S, EOS, DF, kIntCvt, false>(g_out, psi_out, P, x, y, z, e);
      }
    }
    k = kn;
  }
  if (e) atomicOr(err, e);
}

template <typename S, int OP, bool LIN, int EOS, bool DF, int Q>
cudaError_t launch_kernel(const KParams &P, const void *g_in, void *g_out, const void *psi_in, void *psi_out,
                          const QueueState &q, int stamp, unsigned *err, cudaStream_t s) {
  auto kern = queue_kernel<S, OP, LIN, EOS, DF, Q>;
  const S *gi = (const S *)g_in;
  S *go = (S *)g_out;
  const float *pi = (const float *)psi_in;
  float *po = (float *)psi_out;
  KParams Pc = P;
  TileMap G = tile_map(P);
  const int4 *items = q.items;
  int nitems = q.nitems, *done = q.done;
  void *args[] = {(void *)&gi,    (void *)&go,     (void *)&pi,   (void *)&po,    (void *)&Pc,   (void *)&G,
                  (void *)&items, (void *)&nitems, (void *)&done, (void *)&stamp, (void *)&err};
  return cudaLaunchCooperativeKernel((const void *)kern, dim3(q.grid), dim3(TXP, kRows), args, 0, s);
}

template <typename S, int OP, bool LIN, int Q = 19>
cudaError_t by_eos(const KParams &P, bool df, const void *g_in, void *g_out, const void *psi_in, void *psi_out,
                   const QueueState &q, int stamp, unsigned *err, cudaStream_t s) {
  switch (P.eos) {
    case kEosCS:
      return df ? launch_kernel<S, OP, LIN, kEosCS, true, Q>(P, g_in, g_out, psi_in, psi_out, q, stamp, err, s)
                : launch_kernel<S, OP, LIN, kEosCS, false, Q>(P, g_in, g_out, psi_in, psi_out, q, stamp, err, s);
    case kEosExp:
      return df ? launch_kernel<S, OP, LIN, kEosExp, true, Q>(P, g_in, g_out, psi_in, psi_out, q, stamp, err, s)
                : launch_kernel<S, OP, LIN, kEosExp, false, Q>(P, g_in, g_out, psi_in, psi_out, q, stamp, err, s);
    default:
      return launch_kernel<S, OP, LIN, kEosNone, false, Q>(P, g_in, g_out, psi_in, psi_out, q, stamp, err, s);
  }
}

template <typename S>
cudaError_t by_op(const KParams &P, int op, bool lin, bool df, const void *g_in, void *g_out, const void *psi_in,
                  void *psi_out, const QueueState &q, int stamp, unsigned *err, cudaStream_t s) {
  if (P.q == 15)
    return lin ? by_eos<S, kNonOrth, true, 15>(P, df, g_in, g_out, psi_in, psi_out, q, stamp, err, s)
                 : by_eos<S, kNonOrth, false, 15>(P, df, g_in, g_out, psi_in, psi_out, q, stamp, err, s);
  if (op == kNonOrth)
    return lin ? by_eos<S, kNonOrth, true>(P, df, g_in, g_out, psi_in, psi_out, q, stamp, err, s)
                 : by_eos<S, kNonOrth, false>(P, df, g_in, g_out, psi_in, psi_out, q, stamp, err, s);
  return lin ? by_eos<S, kOrth, true>(P, df, g_in, g_out, psi_in, psi_out, q, stamp, err, s)
               : by_eos<S, kOrth, false>(P, df, g_in, g_out, psi_in, psi_out, q, stamp, err, s);
}

// Resident blocks per SM of the kernels a context launches: what the launch
// bounds promise for every instantiation of the storage type and lattice, so that
// a cooperative launch of that many fits whichever one runs; fewer where the
// device gives one of those looked at fewer (shared memory set aside by a tool).
template <typename S>
cudaError_t occupancy_of(int q, int *per_sm) {
  using K = void (*)(const S *, S *, const float *, float *, const KParams, const TileMap, const int4 *, int, int *, int,
                     unsigned *);
  const K k19[] = {queue_kernel<S, kNonOrth, true, kEosCS, false, 19>, queue_kernel<S, kOrth, true, kEosCS, false, 19>,
                   queue_kernel<S, kNonOrth, false, kEosCS, true, 19>, queue_kernel<S, kOrth, false, kEosExp, false, 19>};
  const K k15[] = {queue_kernel<S, kNonOrth, true, kEosCS, false, 15>, queue_kernel<S, kNonOrth, false, kEosExp, true, 15>};
  int m = 1 << 30;
  for (int i = 0; i < (q == 15 ? 2 : 4); ++i) {
    const K k = q == 15 ? k15[i] : k19[i];
    int v = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k, NTH, 0);
    if (e != cudaSuccess) return e;
    m = std::min(m, v);
  }
  *per_sm = std::min(m, min_blocks<S>(q));
  return cudaSuccess;
}

// ------------------------------------------------------------------ batches
// The same work list over many boxes.  Every job carries its box, whose
// descriptor (parameters, buffers, operator, level, tile width) the block
// copies to shared memory one item ahead (asynchronous copies, double
// buffered), so it is there when the item starts; a fused job of box B
// reads level in = B.cur ^ parity and writes in ^ 1, the psi job evaluates psi
// of level in ^ 1.  Both operators and the Eq. 16 term (zero coefficient when
// off) are compiled in.
// Copy box descriptors to shared memory with asynchronous 16-byte copies (one
// commit group per call), so that the next item's descriptors arrive while the
// current item runs.
__device__ __forceinline__ void prefetch_boxes(BatchBox *dst, const BatchBox *__restrict__ boxes, int4 it, int tid,
                                               int nthreads = NTH) {
  constexpr int chunks = (int)(sizeof(BatchBox) / 16);
  static_assert(sizeof(BatchBox) % 16 == 0, "descriptor copies move 16-byte pieces");
  for (int side = 0; side < 2; ++side) {
    const int box = side ? it.z : it.x;
    if (box < 0) continue;
    const char *src = (const char *)(boxes + box);
    char *d = (char *)(dst + side);
    for (int c = tid; c < chunks; c += nthreads) {
      const unsigned sa = (unsigned)__cvta_generic_to_shared(d + 16 * c);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(src + 16 * c) : "memory");
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// ODD: some box has an odd Nx (rows padded to an even length, KParams::px).
template <typename S, int EOS, bool ODD>
__global__ void __launch_bounds__(NTH, one_node_rounding<S, ODD>() ? kOddHalfBatchBlocks : kBatchBlocks)
    batch_queue_kernel(const BatchBox *__restrict__ boxes, const int4 *__restrict__ items, int nitems, int parity,
                       int *__restrict__ done, int ndone, unsigned *__restrict__ err) {
  __shared__ BatchBox bb[2][2];  // [item parity][fused job's box, psi job's box]
  const int tid = threadIdx.y * TXP + threadIdx.x;
  unsigned e = 0;
  // block b starts with item b, then claims the next unclaimed item (one atomic fetch per item, issued
  // when an item starts); warp 0 reads the claimed item and copies its descriptors during the psi job
  __shared__ int s_next;
  __shared__ int4 s_it;
  unsigned *claims = (unsigned *)(done + ndone + 16);  // cleared with the counters before every launch
  int k = blockIdx.x;
  int4 it = k < nitems ? __ldg(items + k) : make_int4(-1, -1, -1, -1);
  prefetch_boxes(bb[0], boxes, it, tid);
#pragma unroll 1
  for (int i = 0; k < nitems; ++i) {
    unsigned claim = 0;
    if (tid == 0) claim = atomicAdd(claims, 1u);  // the next item: gridDim.x + claim
    asm volatile("cp.async.wait_group 0;" ::: "memory");  // this item's descriptors have arrived
    __syncthreads();
    if (it.x >= 0) {
      const BatchBox &B = bb[i & 1][0];
      const KParams &P = B.P;
      int z = (int)((unsigned)it.y & 0xffffu), t = (int)((unsigned)it.y >> 16);
      asm volatile("" : "+r"(z), "+r"(t));
      const int in = B.cur ^ parity;
      int x, y;
      if (tile_node(B.map, B.map.lin, P, t, tid, x, y)) {
        const S *gi = (const S *)B.g[in];
        S *go = (S *)B.g[in ^ 1];
        if (B.op == kNonOrth)
          fused_pair_at<S, kNonOrth, true, false, ODD>(gi, go, B.psi[in], P, x, y, z, Rates<V2>(P));
        else
          fused_pair_at<S, kOrth, true, false, ODD>(gi, go, B.psi[in], P, x, y, z, Rates<V2>(P));
      }
      __syncthreads();
      if (tid == 0) counter_release_add(done + LBM_IDX(B.qbase + z * B.map.T + t, ndone), 1);
    }
    if (threadIdx.y == 0) {  // the next item and its descriptors (buffer (i + 1) & 1 was item i - 1's)
      const int kn = (int)min((unsigned)gridDim.x + __shfl_sync(0xffffffffu, claim, 0), (unsigned)nitems);
      const int4 nx = kn < nitems ? __ldg(items + kn) : make_int4(-1, -1, -1, -1);
      prefetch_boxes(bb[(i + 1) & 1], boxes, nx, threadIdx.x, TXP);
      if (threadIdx.x == 0) {
        s_next = kn;
        s_it = nx;
      }
    }
    if (it.z >= 0) {
      const BatchBox &B = bb[i & 1][1];
      const KParams &P = B.P;
      int z = (int)((unsigned)it.w & 0xffffu), t = (int)((unsigned)it.w >> 16);
      asm volatile("" : "+r"(z), "+r"(t));
      // counters are cleared before every launch
      if (!wait_for_jobs(B.map, B.map.lin, P, done, B.qbase, ndone, z, t, threadIdx.x, 1 + P.wait_bias, P.spin_limit))
        e |= kErrTimeout;
      const int in = B.cur ^ parity;
      int x, y;
      if (tile_node(B.map, B.map.lin, P, t, tid, x, y))
        psi_pair_at_l2<S, EOS, false, kIntCvt, ODD>((const S *)B.g[in ^ 1], B.psi[in ^ 1], P, x, y, z, e);
    }
    __syncthreads();  // s_next and s_it are written; rewritten only after the next item's first barrier
    k = s_next;
    it = s_it;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");  // no copy outlives the block
  if (e) atomicOr(err, e);
}

template <typename S, int EOS, bool ODD>
cudaError_t batch_launch(const BatchBox *boxes, const int4 *items, int nitems, int parity, int grid, int *done,
                         int ndone, unsigned *err, cudaStream_t s, int *per_sm) {
  auto kern = batch_queue_kernel<S, EOS, ODD>;
  if (per_sm) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, kern, NTH, 0);
  void *args[] = {(void *)&boxes, (void *)&items, (void *)&nitems, (void *)&parity,
                  (void *)&done,  (void *)&ndone, (void *)&err};
  return cudaLaunchCooperativeKernel((const void *)kern, dim3(grid), dim3(TXP, kRows), args, 0, s);
}

template <typename S, bool ODD>
cudaError_t batch_by_eos(int eos, const BatchBox *boxes, const int4 *items, int nitems, int parity, int grid,
                         int *done, int ndone, unsigned *err, cudaStream_t s, int *per_sm) {
  switch (eos) {
    case kEosCS: return batch_launch<S, kEosCS, ODD>(boxes, items, nitems, parity, grid, done, ndone, err, s, per_sm);
    case kEosExp: return batch_launch<S, kEosExp, ODD>(boxes, items, nitems, parity, grid, done, ndone, err, s, per_sm);
    default: return batch_launch<S, kEosNone, ODD>(boxes, items, nitems, parity, grid, done, ndone, err, s, per_sm);
  }
}

// The psi jobs in order of the last fused job they read (stable).
std::vector<long long> by_ready(const std::vector<long long> &ready) {
  std::vector<long long> start(ready.size() + 1, 0), order(ready.size());
  for (long long r : ready) ++start[r + 1];
  for (size_t k = 1; k < start.size(); ++k) start[k] += start[k - 1];
  for (size_t p = 0; p < ready.size(); ++p) order[start[ready[p]]++] = (long long)p;
  return order;
}

// Items between a psi job and the last fused job it reads: 3/8 of a wave of the
// grid where a plane is large (the populations leave L2 sooner), 5/8 where it
// is small (more of the list hangs on each plane).  FP32 non-orthogonal steps at 1/4,
// 3/8, 1/2, 5/8 and 3/4: 128^3 (64 tiles a plane) 89.8, 84.4, 77.4, 72.8 and 71.7 us,
// 160^3 (100) 167, 152, 136, 133 and 133, 192^3 (144) 267, 225, 218.5, 218 and 219,
// 224^3 (196) 428, 364, 353, 355 and 359, 240^3 (225) 525, 432, 423, 425 and 430,
// 256^3 537, 508, 511, 518 and 527, 320^3 (400) 1120, 1001, 1002, 1012 and 1024, 512^3
// 4.51, 4.38, 4.40, 4.43 and 4.46 ms; orthogonal and D3Q15 boxes alike (D3Q15 240^3
// 489, 377, 360, 360 and 361).
long long psi_lag(int grid, int tiles_per_plane) {
  return std::max(1LL, (long long)grid * (tiles_per_plane < 240 ? 5 : 3) / 8);
}

// Psi jobs go to the first free item at least `lag` items after the last of
// the fused jobs they read (ready[]); fused job j sits in item j.  Checks the
// result as the single-box list does.
bool place_psi_jobs(std::vector<int4> &out, const std::vector<long long> &ready, const std::vector<int2> &job,
                    long long nf, long long lag) {
  const std::vector<long long> order = by_ready(ready);
  long long next = 0;
  for (long long p : order) {
    const long long k = std::max(next, ready[p] + lag);
    while ((long long)out.size() <= k) out.push_back(make_int4(-1, -1, -1, -1));
    out[k].z = job[p].x;
    out[k].w = job[p].y;
    next = k + 1;
  }
  return (long long)out.size() < (1LL << 31);
}

}  // namespace

// 128 consecutive pairs of the plane leave no lane idle and start on a sector
// wherever the row does, whatever Nx is; 64 x 4 tiles leave lanes idle where Nx
// is no multiple of 64 or Ny of 4 (80 x 80: 38 %, 200 x 180: 22 %), and tiles
// narrowed to 16 nodes start off a 32-byte sector in most rows.  They are also
// the faster ones where 64 x 4 fits: per step, 64 x 4 (with the better lag) /
// consecutive, 80^3 34.3 / 26.3 us, 128^3 73.9 / 72.8, 160^3 148 / 133, 192^3 225 /
// 218, 200 x 180 x 256 (orthogonal) 354 / 295, 256^3 535 / 508, 320^3 1028 / 1001,
// 512^3 4.49 / 4.38 ms; a batch of six boxes of edges 62 to 140 314 / 257 us (16-
// and 32-node tiles: 301).  A psi job then waits for whole rows around its
// tile; past 512 nodes a row that is more tiles than a warp has lanes to poll
// with, and the 64 x 4 tiles take over.
TileMap tile_map(const KParams &P) {
  TileMap G{};
  G.W = P.px / 2;
  G.M = G.W * P.ny;
  G.ntx = (P.nx + 2 * TXP - 1) / (2 * TXP);
  G.nty = (P.ny + kRows - 1) / kRows;
  const long long rows = NTH / G.W + 4;  // rows a psi job of a tile of consecutive pairs reads, at most
  if (P.px % 2 == 0 && (rows * G.W + NTH - 1) / NTH + 2 <= kMaxLin && (long long)G.M * G.W < (1LL << 32)) {
    G.lin = 1;
    G.T = (G.M + NTH - 1) / NTH;
    G.m = (unsigned)(((1ull << 32) + G.W - 1) / G.W);
  } else {
    G.T = G.ntx * G.nty;
  }
  return G;
}

// For every tile, the last of the tiles a psi job of it reads in a plane.
static std::vector<int> last_tiles(const TileMap &G) {
  std::vector<int> last((size_t)G.T, 0);
  for (int t = 0; t < G.T; ++t)
    for (int lane = 0; lane < 32; ++lane) {
      int dz, tile;
      if (dep_of_lane(G, G.lin != 0, t, lane, dz, tile)) last[t] = std::max(last[t], tile);
    }
  return last;
}
// Position (z T + tile) of the last fused job that psi job (z, t) reads: in
// plane z + 1, or in the last plane where the box wraps.
static long long last_read(const TileMap &G, const std::vector<int> &last, int nz, int z, int t) {
  return (long long)(z == 0 || z == nz - 1 ? nz - 1 : z + 1) * G.T + last[t];
}

bool queue_supported(const KParams &P, int precision) { return precision != kF64 && P.nx % 2 == 0; }

// Thread blocks of the launch: all that are resident, but no more than there are fused jobs (blocks without one only
// cost their launch and a longer list: FP16 32^3 10.3 -> 9.3 us a step, D3Q15 10.3 -> 8.8).
cudaError_t queue_grid(const KParams &P, int precision, int *grid) {
  int per_sm = 0, dev = 0, sms = 0;
  cudaError_t e = precision == kF32 ? occupancy_of<float>(P.q, &per_sm) : occupancy_of<__half>(P.q, &per_sm);
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  *grid = (int)std::min<long long>((long long)per_sm * sms, (long long)P.nz * tile_map(P).T);
  return cudaSuccess;
}

size_t queue_counters(const KParams &P) { return (size_t)P.nz * tile_map(P).T + 32; }  // + the claim counter

bool queue_items(const KParams &P, int grid, std::vector<int4> &out) {
  const TileMap G = tile_map(P);
  const long long nf = (long long)P.nz * G.T;
  if (P.nz < 3 || grid < 1 || nf >= (1LL << 30)) return false;
  // fused job j = (j / T, j % T); psi job (z, t) is ready after the last of the
  // fused jobs it reads and goes to the first free item >= ready + lag
  const long long lag = psi_lag(grid, G.T);
  const std::vector<int> last = last_tiles(G);
  std::vector<long long> ready((size_t)nf);
  for (long long p = 0; p < nf; ++p) {
    ready[p] = last_read(G, last, P.nz, (int)(p / G.T), (int)(p % G.T));
  }
  const std::vector<long long> order = by_ready(ready);
  out.assign((size_t)nf, make_int4(-1, -1, -1, -1));
  for (long long j = 0; j < nf; ++j) out[j] = make_int4((int)(j / G.T), (int)(j % G.T), -1, -1);
  long long next = 0;  // first item that may still take a psi job
  for (long long p : order) {
    const long long k = std::max(next, ready[p] + lag);
    while ((long long)out.size() <= k) out.push_back(make_int4(-1, -1, -1, -1));
    out[k].z = (int)(p / G.T);
    out[k].w = (int)(p % G.T);
    next = k + 1;
  }
  if ((long long)out.size() >= (1LL << 31)) return false;
  // check: every job once; each psi job in an item after the fused jobs it reads
  std::vector<char> fseen((size_t)nf, 0), pseen((size_t)nf, 0);
  for (size_t k = 0; k < out.size(); ++k) {
    const int4 it = out[k];
    if (it.x >= 0) {
      const long long j = (long long)it.x * G.T + it.y;
      if (j != (long long)k || fseen[j]) return false;
      fseen[j] = 1;
    }
    if (it.z >= 0) {
      if (it.z >= P.nz || it.w < 0 || it.w >= G.T) return false;
      const long long p = (long long)it.z * G.T + it.w;
      if (pseen[p] || ready[p] >= (long long)k) return false;
      pseen[p] = 1;
    }
  }
  for (long long p = 0; p < nf; ++p)
    if (!fseen[p] || !pseen[p]) return false;
  return true;
}

cudaError_t launch_queue(const KParams &P, int precision, int op, bool df, const void *g_in, void *g_out,
                         const void *psi_in, void *psi_out, const QueueState &q, int stamp, unsigned *err,
                         cudaStream_t s) {
  if (!queue_supported(P, precision)) return cudaErrorInvalidValue;
  const bool lin = tile_map(P).lin != 0;
  if (precision == kF32) return by_op<float>(P, op, lin, df, g_in, g_out, psi_in, psi_out, q, stamp, err, s);
  return by_op<__half>(P, op, lin, df, g_in, g_out, psi_in, psi_out, q, stamp, err, s);
}

bool batch_queue_items(const std::vector<const KParams *> &boxes, int grid, std::vector<int4> &out,
                       std::vector<int> &base, long long *ncounters) {
  // fused jobs box by box, plane by plane: global fused position = item index
  std::vector<long long> first(boxes.size() + 1, 0);
  base.assign(boxes.size(), 0);
  for (size_t b = 0; b < boxes.size(); ++b) {
    const KParams &P = *boxes[b];
    const TileMap G = tile_map(P);
    if (P.nz < 3 || P.px % 2 != 0 || P.nz > 0xffff || G.T > 0xffff || grid < 1) return false;
    first[b + 1] = first[b] + (long long)P.nz * G.T;
    if (first[b + 1] >= (1LL << 30)) return false;
    base[b] = (int)first[b];
  }
  const long long nf = first.back();
  *ncounters = nf;
  out.assign((size_t)nf, make_int4(-1, -1, -1, -1));
  std::vector<long long> ready((size_t)nf);
  std::vector<int2> job((size_t)nf);  // (box, z | tile << 16) of psi job p (same numbering as fused job p)
  for (size_t b = 0; b < boxes.size(); ++b) {
    const KParams &P = *boxes[b];
    const TileMap G = tile_map(P);
    const std::vector<int> last = last_tiles(G);
    for (int z = 0; z < P.nz; ++z)
      for (int t = 0; t < G.T; ++t) {
        const long long j = first[b] + (long long)z * G.T + t;
        const int zt = (int)((unsigned)z | ((unsigned)t << 16));
        out[j] = make_int4((int)b, zt, -1, -1);
        job[j] = make_int2((int)b, zt);
        ready[j] = first[b] + last_read(G, last, P.nz, z, t);
      }
  }
  if (!place_psi_jobs(out, ready, job, nf, std::max(1, grid / 2))) return false;
  // check: every job once, each psi job in an item after the fused jobs it reads
  std::vector<char> fseen((size_t)nf, 0), pseen((size_t)nf, 0);
  for (size_t k = 0; k < out.size(); ++k) {
    const int4 it = out[k];
    for (int side = 0; side < 2; ++side) {
      const int b = side ? it.z : it.x;
      if (b < 0) continue;
      if (b >= (int)boxes.size()) return false;
      const unsigned zt = (unsigned)(side ? it.w : it.y);
      const int z = (int)(zt & 0xffffu), t = (int)(zt >> 16);
      const TileMap G = tile_map(*boxes[b]);
      if (z >= boxes[b]->nz || t >= G.T) return false;
      const long long j = first[b] + (long long)z * G.T + t;
      if (!side) {
        if (j != (long long)k || fseen[j]) return false;
        fseen[j] = 1;
      } else {
        if (pseen[j] || ready[j] >= (long long)k) return false;
        pseen[j] = 1;
      }
    }
  }
  for (long long p = 0; p < nf; ++p)
    if (!fseen[p] || !pseen[p]) return false;
  return true;
}

cudaError_t batch_queue_grid(int precision, int eos, bool odd, int *grid) {
  int per_sm = 0, dev = 0, sms = 0;
  auto query = precision == kF32 ? (odd ? batch_by_eos<float, true> : batch_by_eos<float, false>)
                                 : (odd ? batch_by_eos<__half, true> : batch_by_eos<__half, false>);
  cudaError_t e = query(eos, nullptr, nullptr, 0, 0, 0, nullptr, 0, nullptr, 0, &per_sm);
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  *grid = per_sm * sms;
  return cudaSuccess;
}

cudaError_t launch_batch_queue(int precision, int eos, bool odd, const BatchBox *boxes, const int4 *items, int nitems,
                               int parity, int grid, int *done, int ndone, unsigned *err, cudaStream_t s) {
  if (precision != kF32 && precision != kF16) return cudaErrorInvalidValue;
  auto launch = precision == kF32 ? (odd ? batch_by_eos<float, true> : batch_by_eos<float, false>)
                                  : (odd ? batch_by_eos<__half, true> : batch_by_eos<__half, false>);
  return launch(eos, boxes, items, nitems, parity, grid, done, ndone, err, s, nullptr);
}

}  // namespace lbm
