// Tiles, neighbourhoods and waits of the work-list kernels (lbm_queue.cu,
// lbm_steps.cu).
#pragma once

#include "lbm_device.cuh"
#include "lbm_internal.h"
#include "lbm_pair.cuh"

namespace lbm {

constexpr int TXP = 32;          // pair columns of a tile: 64 nodes
constexpr int kRows = 4;         // rows of a tile (one warp each)
constexpr int NTH = TXP * kRows;

// The pair of thread tid in tile t of a plane: true if there is one.
__device__ __forceinline__ bool tile_node(const TileMap &G, bool lin, const KParams &P, int t, int tid, int &x,
                                          int &y) {
  if (lin) {
    const unsigned p = (unsigned)t * NTH + tid;
    y = (int)__umulhi(p, G.m);
    x = 2 * ((int)p - y * G.W);
    return (int)p < G.M;
  }
  const int ty = t / G.ntx;
  x = (t - ty * G.ntx) * 2 * TXP + 2 * (tid & (TXP - 1));
  y = ty * kRows + tid / TXP;
  return x < P.nx && y < P.ny;
}

// The tiles a psi job of tile t reads in planes z - 1, z, z + 1: lane's share
// (dz, tile), false if it has none.  64 x 4 tiles: the 3 x 3 around it.  lin: all
// tiles of the rows from one before its first to one after its last (a pair at
// the end of a row reads the row's other end), at most kMaxLin of them, which
// follow each other modulo T.
constexpr int kMaxLin = 10;
__host__ __device__ __forceinline__ bool dep_of_lane(const TileMap &G, bool lin, int t, int lane, int &dz,
                                                               int &tile) {
  if (lin) {
    const int a = t * NTH, b = a + NTH < G.M ? a + NTH - 1 : G.M - 1;
    const int ya = (int)(((unsigned long long)(unsigned)a * G.m) >> 32);
    const int yb = (int)(((unsigned long long)(unsigned)b * G.m) >> 32);
    int s = (ya - 1) * G.W, e = (yb + 2) * G.W - 1;
    const bool all = e - s + 1 + NTH >= G.M;  // the range meets itself
    if (s < 0) s += G.M;
    if (e >= G.M) e -= G.M;
    const int first = all ? 0 : s / NTH;
    int cnt = all ? G.T : e / NTH - first + 1;
    if (cnt <= 0) cnt += G.T;
    dz = lane / kMaxLin - 1;
    const int j = lane % kMaxLin;
    tile = first + j;
    if (tile >= G.T) tile -= G.T;
    return dz <= 1 && j < cnt;
  }
  const int ty = t / G.ntx, tx = t - ty * G.ntx;
  int xx = tx + lane % 3 - 1, yy = ty + (lane / 3) % 3 - 1;
  xx = xx < 0 ? xx + G.ntx : (xx >= G.ntx ? xx - G.ntx : xx);
  yy = yy < 0 ? yy + G.nty : (yy >= G.nty ? yy - G.nty : yy);
  dz = lane / 9 - 1;
  tile = yy * G.ntx + xx;
  return lane < 27;
}

// Polls, by the lanes that have one, the counters of the jobs of tile t's
// neighbourhood (dep_of_lane) until each shows `target`; false (on every lane)
// if one gave up after `limit` polls.
__device__ __forceinline__ bool wait_for_jobs(const TileMap &G, bool lin, const KParams &P, const int *__restrict__ done,
                                              int base, int count, int z, int t, int lane, int target, int limit) {
  bool ok = true;
  int dz, tile;
  if (dep_of_lane(G, lin, t, lane, dz, tile)) {
    int zz = z + dz;
    zz = zz < 0 ? zz + P.nz : (zz >= P.nz ? zz - P.nz : zz);
    const int *c = done + LBM_IDX(base + zz * G.T + tile, count);
    for (int n = 0; (int)((unsigned)counter_acquire(c) - (unsigned)target) < 0; ++n) {  // (counts may wrap)
      if (n >= limit) {
        ok = false;
        break;
      }
      __nanosleep(32);
    }
  }
  return __all_sync(0xffffffffu, ok);
}

}  // namespace lbm
