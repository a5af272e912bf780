// Internal interface between the C ABI (lbm_api.cu) and the kernels
// (lbm_kernels.cu).  Not installed; not part of the public ABI.
#pragma once

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

namespace lbm {

enum Precision { kF64 = 0, kF32 = 1, kF16 = 2 };
enum Operator { kOrth = 0, kNonOrth = 1, kNonOrthQ15 = 2 };
enum EosKind { kEosCS = 0, kEosExp = 1, kEosNone = 2 };

// Error bits the kernels set in the device error word.
enum : unsigned { kErrEosDomain = 1u, kErrNonFinite = 2u, kErrTimeout = 4u };

// Everything a kernel needs about the box and the physics, passed by value.
struct KParams {
  int nx, ny, nz;
  int n;             // nx * ny * nz (< 2^31)
  // The stored arrays (populations, psi): px is the length of an x row in them,
  // np = px * ny * nz the distance from one direction to the next.  px = nx but
  // for an odd nx in the FP32-arithmetic forms, whose two-node kernels want rows
  // that start on a pair: there px = nx + 1 and the last element of a row repeats
  // its first (the periodic neighbour of node nx - 1), kept by whoever writes
  // node 0.  Arrays of the public interface (rho, u, f) have rows of nx.
  int px, np;
  // ceil(2^32 / nx), ceil(2^32 / (px / 2)): a plane's node or pair p lies in row (p m) >> 32; 0 (planes too large
  // for that): divide
  unsigned row_m, pair_m;
  int q;             // lattice: 19 (D3Q19, both operators) or 15 (D3Q15 non-orthogonal)
  double G;          // interaction strength, Eq. 15
  double half_force; // -G/2 times the diagonal (D3Q15: corner) weight of Eq. 15, 1/12 (1/24)
  double rho_ref;    // reference density of the deviation storage
  // relaxation rates (see lbm_rates in lbm.h)
  double s_e, s_nu, s_q, s_pi, s_eps, s_m;
  // Eq. 16 coefficient: the extra S_4 is sigma_coef * |sum_a w_a psi(x+e_a) e_a|^2
  // (= 6 sigma |F|^2 / (psi^2 (1/s_e - 1/2)) with F = -G psi sum(...)).
  double sigma_coef;
  // equation of state
  int eos;
  double a, b, RT;   // Carnahan-Starling (Eq. 58), RT = R * T
  double psi0, rho0; // exponential pseudopotential
  double exp_k;      // -rho0 log2(e)
  double b4;         // b / 4
  double two_over_G; // 2 / G
  // (2/G) (RT num - (a rho + 1/3) den) = q0 + q1 rho + q2 rho^2 + q3 rho^3 + q4 rho^4,
  // num = 1 + eta + eta^2 - eta^3, den = (1 - eta)^3, eta = b rho / 4 (Eq. 58)
  double q0, q1, q2, q3, q4;
  float f_rho_max;   // 4 / b: the packing limit eta < 1
  // FP32 copies for the reduced-precision kernels (no conversions on device)
  float fG, frho_ref, fs_e, fs_nu, fs_q, fs_pi, fs_eps, fs_m, fsigma_coef, fb4;
  // density-dependent shear viscosity: nu(rho) = nu_v + (rho - rho_v) nu_slope,
  // clamped to [nu_lo, nu_hi]; s_nu(rho) = 1 / (3 nu + 1/2).  Off unless varnu.
  int varnu;
  double nu_v, rho_v_nu, nu_slope, nu_lo, nu_hi;
  float fnu_v, frho_v_nu, fnu_slope, fnu_lo, fnu_hi;
  // the radicand coefficients and rho_ref as unevaluated sums of two floats
  // (hi + lo), for the compensated-FP32 evaluation of the EOS
  float qh[5], ql[5], rr_h, rr_l;
  // the same radicand as a quintic in d = rho - rho_ref: sum_k c[k] d^k
  double c[6];
  // bounded device-side waits (single-pass kernels): polls before a wait gives
  // up and sets kErrTimeout; wait_bias is added to every cross-block wait
  // target (0; 1 makes the targets unreachable, a host-side fault injection)
  int spin_limit;
  int wait_bias;
};

// ceil(2^32 / d) if (v m) >> 32 is v / d for every v < count, else 0.
inline unsigned row_multiplier(long long d, long long count) {
  return d >= 2 && count * d < (1LL << 32) ? (unsigned)(((1ull << 32) + d - 1) / d) : 0u;
}

// KParams::px of a box: rows of an odd nx get one element more where the
// two-node kernels run, unless that leaves the index range (19 np < 2^32) or a
// plane has more tiles, of 128 pairs or 64 x 4 nodes, than the 16 bits a batch's
// work list has for one (65535: 16.7 10^6 nodes): the one-node kernels step those.
inline int stored_row(int precision, const int grid[3]) {
  const long long plane = (long long)(grid[0] + 1) * grid[1];
  const long long tiles = std::max((plane / 2 + 127) / 128, (grid[0] + 63LL) / 64 * ((grid[1] + 3LL) / 4));
  return precision != kF64 && grid[0] % 2 != 0 && 19 * plane * grid[2] < (1LL << 32) && tiles <= 0xffff ? grid[0] + 1
                                                                                                         : grid[0];
}

constexpr int kDefaultSpinLimit = 1 << 22;

// An NVTX range around a scope (a kernel launch, a graph launch): visible in
// profilers that trace NVTX; a cheap no-op otherwise.
struct NvtxRange {
  explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange &) = delete;
  NvtxRange &operator=(const NvtxRange &) = delete;
};

// Layout of the scratch buffer.
constexpr int kReduceBlocks = 1024;
constexpr size_t kScratchErrOffset = 0;      // unsigned error word
constexpr size_t kScratchPartialOffset = 256;  // kReduceBlocks x 5 doubles
constexpr size_t kScratchResultOffset = kScratchPartialOffset + sizeof(double) * 5 * kReduceBlocks;
constexpr size_t kScratchBytes = kScratchResultOffset + 256;

// Droplets handed to the density-field kernel in chunks.
constexpr int kDropletChunk = 64;
struct DropletChunk {
  int count;
  double cx[kDropletChunk], cy[kDropletChunk], cz[kDropletChunk], r[kDropletChunk];
};

struct Launch {
  cudaStream_t stream;
};

// Threads per block of the per-node and per-pair kernels.  A block takes as many
// consecutive nodes (pairs) of a plane in row order: blocks of 32 x 4 nodes left
// lanes idle where Nx is no multiple of 32 (pairs: 64), which the kernels bound
// by the FP64 unit pay in full (72^3 FP64 step 242 -> 187 us, 72^3
// FP16 20.9 -> 13.4, 65^3 FP32 18.9 -> 14.8).
constexpr int kThreads = 128;
inline dim3 plane_grid(int per_plane, int nz, int threads = kThreads) {
  return dim3((unsigned)((per_plane + threads - 1) / threads), 1, (unsigned)nz);
}

// Launch of a kernel of the two-pass step that may start while its predecessor
// in the stream is ending (programmatic stream serialization): its blocks take
// the places the last ones leave and wait in chain_wait (lbm_device.cuh) until
// the predecessor has completed, so only the launch itself overlaps.  Blocks that
// come in this way fill one SM after the other, so a grid that would not fill the
// device has to start by itself.  Two-pass steps not chained / chained: FP16 16^3 8.2 / 5.1 us,
// 32^3 8.2 / 7.2, 40^3 10.3 / 10.4, 48^3 12.3 / 8.4, 64^3 16.4 / 11.9, 96^3 30.8 / 25.8, 128^3
// 63.5 / 58.7, 256^3 434 / 429; FP32 32^3 8.2 / 7.7, 40^3 10.3 / 10.3, 48^3 12.3 / 9.3, 65^3 18.5
// / 16.9, 127^3 87.8 / 83.8; FP64, a third as many warps resident, 24^3 14.4 / 24.2, 32^3
// 19.5 / 25.0, 40^3 28.7 / 27.8, 48^3 38.9 / 36.5, 64^3 76.0 / 71.8, 128^3 510 / 505.  So from
// 2^15 nodes the two-node kernels, from 2^18 the FP64 ones.
constexpr int kChainPairs = 1 << 15, kChainFP64 = 1 << 18;  // nodes
template <typename... P, typename... A>
cudaError_t launch_chained(bool chain, void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t s, A... args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = chain ? 1 : 0;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = chain ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, (P)args...);
}

// Fill the FP32 copies of KParams from its doubles (call after any change).
inline void refresh_float_params(KParams &P) {
  P.fG = (float)P.G;
  P.frho_ref = (float)P.rho_ref;
  P.fs_e = (float)P.s_e;
  P.fs_nu = (float)P.s_nu;
  P.fs_q = (float)P.s_q;
  P.fs_pi = (float)P.s_pi;
  P.fs_eps = (float)P.s_eps;
  P.fs_m = (float)P.s_m;
  P.fsigma_coef = (float)P.sigma_coef;
  P.fb4 = (float)P.b4;
  const double q[5] = {P.q0, P.q1, P.q2, P.q3, P.q4};
  for (int k = 0; k < 5; ++k) {
    P.qh[k] = (float)q[k];
    P.ql[k] = (float)(q[k] - (double)P.qh[k]);
  }
  P.fnu_v = (float)P.nu_v;
  P.frho_v_nu = (float)P.rho_v_nu;
  P.fnu_slope = (float)P.nu_slope;
  P.fnu_lo = (float)P.nu_lo;
  P.fnu_hi = (float)P.nu_hi;
  P.rr_h = (float)P.rho_ref;
  P.rr_l = (float)(P.rho_ref - (double)P.rr_h);
  // X(rho) = sum_{m=1..5} q[m-1] rho^m with rho = rho_ref + d:
  // c[k] = sum_{m >= max(k, 1)} q[m-1] binom(m, k) rho_ref^(m-k)
  static const double binom[6][6] = {{1, 0, 0, 0, 0, 0},  {1, 1, 0, 0, 0, 0},   {1, 2, 1, 0, 0, 0},
                                     {1, 3, 3, 1, 0, 0},  {1, 4, 6, 4, 1, 0},   {1, 5, 10, 10, 5, 1}};
  for (int k = 0; k <= 5; ++k) {
    double acc = 0.0;
    for (int m = k > 1 ? k : 1; m <= 5; ++m) {
      double rp = 1.0;
      for (int j = 0; j < m - k; ++j) rp *= P.rho_ref;
      acc += q[m - 1] * binom[m][k] * rp;
    }
    P.c[k] = acc;
  }
}

// Coefficients of the collision (Eq. 4, 11, 13, 14, 16), one set per operator.
// The relaxed moments enter the inverse transform with constant factors (1/4,
// 1/6, 1/12, ...); with those multiplied into the rates on the host, a moment is
// relaxed and scaled by the same instructions.  s is a rate, a = 1 - s, c = 1 - s/2.
enum Coeff {
  // shear rate: a/12, a/4, s/8, c/4, a/36 (D3Q15: s/16, c/8 and a/8 for the last three)
  kN5 = 0, kN7, kNb1, kNb2, kON,
  // odd moments
  kQ2,        // a_q                    (non-orthogonal and D3Q15)
  kQa,        // a_q / 2; orthogonal: a_q / 40
  kQb1, kQb2, // s_q / 12, c_q / 12; orthogonal over 60, D3Q15 over 24
  // energy; non-orthogonal and D3Q15: of moment 4 (relax4); orthogonal: of e over 2394
  kE1, kE2, kE3, kE4, kE5,
  // fourth-order moments over 4 (D3Q15: over 8); orthogonal: pi_xx over 72
  kP1, kP2, kP3, kP4, kP5,
  // orthogonal only: eps over 252, (1 - s_m) / 8
  kO1, kO2, kO3, kO4, kO5, kO6, kOm,
  kForce,  // F_i = force psi(x) S_i
  kCoeffs
};

struct Coeffs64 {
  double k[kCoeffs];
};

// force and sig: -G and the Eq. 16 coefficient (KParams::sigma_coef) for the
// sums of Eq. 15 in units of the diagonal (corner) weight, 1/12 (1/24).
inline Coeffs64 coeffs64(const KParams &P, int op) {
  Coeffs64 c64;
  double *k = c64.k;
  const double se = P.s_e, sn = P.s_nu, sq = P.s_q, sp = P.s_pi, sx = P.s_eps, sm = P.s_m;
  const double units = P.q == 15 ? 24.0 : 12.0, sig = P.sigma_coef / (units * units);
  const double ce = 1 - 0.5 * se, cn = 1 - 0.5 * sn, cq = 1 - 0.5 * sq, cp = 1 - 0.5 * sp, cx = 1 - 0.5 * sx;
  for (int i = 0; i < kCoeffs; ++i) k[i] = 0.0;
  k[kForce] = -P.G / units;
  k[kN5] = (1 - sn) / 12;
  k[kN7] = (1 - sn) / 4;
  k[kNb1] = sn / 8;
  k[kNb2] = cn / 4;
  k[kON] = (1 - sn) / 36;
  k[kQ2] = 1 - sq;
  if (op == kOrth) {
    k[kQa] = (1 - sq) / 40;
    k[kQb1] = sq / 60;
    k[kQb2] = cq / 60;
    // e = 19 (A + 2 B) - 30 drho, A and B the axis and diagonal sums of f
    k[kE1] = (1 - se) * 19 / 2394;
    k[kE2] = (-30 * (1 - se) - 11 * se) / 2394;
    k[kE3] = 19 * se / 2394;
    k[kE4] = 38 * ce / 2394;
    k[kE5] = 19 * ce * sig / 2394;
    // eps = 12 drho - 16 A - 11 B
    k[kO1] = -16 * (1 - sx) / 252;
    k[kO2] = -11 * (1 - sx) / 252;
    k[kO3] = (12 * (1 - sx) + 3 * sx) / 252;
    k[kO4] = -5.5 * sx / 252;
    k[kO5] = -11 * cx / 252;
    k[kO6] = -16 * cx * sig / 252;
    // pi_xx over 72 (a, s/2, c) and pi_ww over 24 (three times those)
    k[kP1] = (1 - sp) / 72;
    k[kP2] = 0.5 * sp / 72;
    k[kP3] = cp / 72;
    k[kOm] = (1 - sm) / 8;
  } else {
    k[kQa] = (1 - sq) / 2;
    k[kQb1] = sq / 12;
    k[kQb2] = cq / 12;
    k[kE1] = se;
    k[kE4] = 2 * ce / se;
    k[kE5] = ce * sig / se;
    if (op == kNonOrth) {
      k[kP1] = sp;
      k[kP4] = cp / (6 * sp);  // F . u
    } else {             // D3Q15: corner moments over 8
      k[kON] = (1 - sn) / 8;
      k[kNb1] = sn / 16;
      k[kNb2] = cn / 8;
      k[kQb1] = sq / 24;
      k[kQb2] = cq / 24;
      k[kP1] = sp;
      k[kP4] = cp / (18 * sp);
    }
  }
  return c64;
}

// x-y tile shapes of the single-pass kernel.
enum Tile { kTile32x4 = 0, kTile32x8 = 1, kTile64x4 = 2 };

// Single-pass step (FP32 and FP16-storage forms): reads populations g_in and
// psi(t) from psi_in, writes populations g_out and psi(t+1) to psi_out.  zc is
// the number of z planes each CTA marches through.
cudaError_t launch_onepass(const KParams &P, int precision, int op, bool sigma, int tile, int zc, const void *g_in,
                           void *g_out, const void *psi_in, void *psi_out, unsigned *err, cudaStream_t s);

// Which node pairs of a plane a work-list tile job covers: 128 consecutive
// pairs of the plane in row order (lin), or 64 x 4 nodes.
struct TileMap {
  int lin;
  int T;         // tiles per plane
  int W, M;      // pairs per row and per plane
  int ntx, nty;  // 64 x 4 tiles along x and y
  unsigned m;    // lin: ceil(2^32 / W), so that v / W is (v m) >> 32 for every pair v of a plane
};
TileMap tile_map(const KParams &P);

// One box of a batch as the batched kernel sees it (copied to shared memory
// per work item).  g[k] / psi[k]: the two time levels; cur: which level holds
// the state at the batch's parity 0.
struct alignas(16) BatchBox {  // 16-byte aligned: copied to shared memory in 16-byte pieces
  KParams P;
  void *g[2];
  float *psi[2];
  int op;
  int cur;
  int qbase;  // first completion counter of this box in the batch work list, or (two-pass step) its first
              // block of the flat fused grid
  TileMap map;  // its tiles there
};

// Persistent single-pass launch over the work items (box, tx | ty << 16, z0, z1)
// of many boxes; grid = number of thread blocks.  FP32 arithmetic forms only.
// The batch's two-pass step on the pair kernels (every box's rows of even length, KParams::px):
// the fused pass, then the psi pass of the new level, for one parity.  The
// fused pass is a flat grid per operator, one block per plane of a tile of the
// chosen shape: block_box holds the box of every block, the non-orthogonal
// boxes' fused_blocks[0] blocks first, then the orthogonal boxes'
// fused_blocks[1]; a box's blocks are consecutive from its descriptor's qbase,
// plane by plane, tiles x-fastest.  The psi pass is a persistent grid of
// sms x per_sm[1] blocks over the items (at most one per item), per_sm as
// batch_pair_occupancy gives it (resident blocks per SM; [0] is unused).
// odd: some box has rows padded for an odd Nx.
cudaError_t batch_pair_occupancy(int precision, int eos, int tile, bool odd, int per_sm[2]);
cudaError_t launch_batch_pair(int precision, int eos, int tile, bool odd, const BatchBox *boxes, const int4 *items,
                              int nitems, const int *block_box, const int fused_blocks[2], int parity, int sms,
                              const int per_sm[2], unsigned *err, cudaStream_t s);
cudaError_t launch_batch_onepass(int precision, int eos, int tile, const BatchBox *boxes, const int4 *items,
                                 int nitems, int parity, int grid, unsigned *err, cudaStream_t s);
// Block shape of a tile choice: returns threads per block, sets bx, by.
int onepass_tile_shape(int tile, int *bx, int *by);

// Single-pass step whose data movement runs on bulk asynchronous copies
// (FP32 storage, 32x8 tiles, nx % 4 == 0 and nx >= 40).
bool onepass_tma_supported(const KParams &P, int precision);
cudaError_t launch_onepass_tma(const KParams &P, int precision, int op, bool sigma, int zc, const void *g_in,
                               void *g_out, const void *psi_in, void *psi_out, unsigned *err, cudaStream_t s);

// Two-pass kernels of the FP32-arithmetic forms with two x-adjacent nodes per
// thread (rows of even length), in packed FP32 arithmetic where Nx is even.
bool pair_supported(const KParams &P, int precision);
cudaError_t launch_psi_pair(const KParams &P, int precision, const void *g, void *psi, unsigned *err,
                            const Launch &L, bool df);
cudaError_t launch_fused_pair(const KParams &P, int precision, int op, bool sigma, const void *g_in, void *g_out,
                              const void *psi, const Launch &L);

// Single-pass step with psi evaluated on chip by producer warps and the
// collision run by consumer warps (FP32 arithmetic, Nx even); no psi array.
bool onchip_supported(const KParams &P, int precision);
cudaError_t launch_onchip(const KParams &P, int precision, int op, bool sigma, bool df, const void *g_in, void *g_out,
                          unsigned *err, cudaStream_t s);

// Single-pass step in which psi of the next step trails the fused pass by one
// plane in one cooperative launch (FP32 arithmetic, Nx even).  flags: an int
// per (tile, plane), lagged_flag_count(P) of them, zero before the first
// launch; stamp: a number larger than in every earlier launch on these flags.
bool lagged_supported(const KParams &P, int precision);
size_t lagged_flag_count(const KParams &P);
cudaError_t launch_lagged(const KParams &P, int precision, int op, bool sigma, bool df, const void *g_in, void *g_out,
                          const void *psi_in, void *psi_out, int *flags, int stamp, unsigned *err, cudaStream_t s);

// Single-pass step on an ordered work list (FP32 arithmetic, D3Q19 or D3Q15, Nx even):
// items of a fused tile job and a lagging psi tile job, one cooperative launch
// of `grid` blocks (queue_grid) working through the list queue_items builds
// (and checks: false if it cannot).  The device side: the item table, a
// completion counter per fused job and the blocks' item-claim counter
// (queue_counters ints, zero before the first launch).
struct QueueState {
  const int4 *items;
  int nitems;
  int grid;
  int *done;
};
bool queue_supported(const KParams &P, int precision);
cudaError_t queue_grid(const KParams &P, int precision, int *grid);
size_t queue_counters(const KParams &P);
bool queue_items(const KParams &P, int grid, std::vector<int4> &out);
// stamp: 1 + the number of earlier launches on these counters.
cudaError_t launch_queue(const KParams &P, int precision, int op, bool df, const void *g_in, void *g_out,
                         const void *psi_in, void *psi_out, const QueueState &q, int stamp, unsigned *err,
                         cudaStream_t s);

// Up to nsteps steps of a small box in one launch (FP32 storage, even Nx; the
// work-list jobs, each block keeping its tiles).  steps_grid gives the grid, 0
// for a box that is too large or not of that form.  counters: steps_counters
// ints, zero before the first launch; stamp: 1 + the steps launched on them.
// The state and psi after nsteps steps are in g_in / psi_in (nsteps even) or
// g_out / psi_out (odd).
cudaError_t steps_grid(const KParams &P, int precision, int *grid);
size_t steps_counters(const KParams &P);
cudaError_t launch_steps(const KParams &P, int op, bool df, void *g_in, void *g_out, void *psi_in, void *psi_out,
                         int grid, int *counters, int nsteps, int stamp, unsigned *err, cudaStream_t s);

// The work-list step over a batch (every box D3Q19, rows of even length): one
// cooperative launch per step; items hold a fused tile job and a psi tile job
// of any boxes (x / z: box index or -1, y / w: z | tile << 16).  The list is
// built for the boxes in the given order; base[k] receives box k's first
// completion counter, *ncounters their total.  Counters must be zero when a
// launch starts (the step graph clears them).
bool batch_queue_items(const std::vector<const KParams *> &boxes, int grid, std::vector<int4> &out,
                       std::vector<int> &base, long long *ncounters);
// odd: some box has rows padded for an odd Nx.
cudaError_t batch_queue_grid(int precision, int eos, bool odd, int *grid);
cudaError_t launch_batch_queue(int precision, int eos, bool odd, const BatchBox *boxes, const int4 *items, int nitems,
                               int parity, int grid, int *done, int ndone, unsigned *err, cudaStream_t s);

// Debug build (-DLBM_BOUNDS_CHECK): OR of the bounds-error words of every
// translation unit, each cleared (synchronous); 0 in the normal build.
namespace dbg {
unsigned take_all();
}

size_t storage_bytes(int precision);  // bytes per stored population
size_t psi_elem_bytes(int precision);

// One time step is launch_psi followed by launch_fused (buffers swapped by the caller).
// df: evaluate the EOS radicand in compensated FP32 pairs (FP32 / FP16 forms)
cudaError_t launch_psi(const KParams &P, int precision, const void *g, void *psi,
                       unsigned *err, const Launch &L, bool df = false);
cudaError_t launch_fused(const KParams &P, int precision, int op, bool sigma,
                         const void *g_in, void *g_out, const void *psi, const Launch &L);

cudaError_t launch_moments(const KParams &P, int precision, const void *g, const void *psi,
                           double *rho, double *u, const Launch &L);
cudaError_t launch_diag(const KParams &P, int precision, const void *g, const void *psi,
                        double *partials, double *result, const Launch &L);

// max |u - u_prev| over the box into *out (atomic max; *out must start at 0), u_prev := u.
cudaError_t launch_max_du(const KParams &P, int precision, const void *g, const void *psi, float *u_prev,
                          double *out, const Launch &L);
cudaError_t launch_rho_droplets(const KParams &P, double *rho, const DropletChunk &chunk,
                                double W, double rho_l, double rho_v, bool first, const Launch &L);
cudaError_t launch_rho_slab(const KParams &P, double *rho, int axis, double lo, double hi,
                            double W, double rho_l, double rho_v, const Launch &L);
cudaError_t launch_state_from_rho(const KParams &P, int precision, const double *rho, void *g,
                                  const Launch &L);
cudaError_t launch_get_populations(const KParams &P, int precision, const void *g, double *out,
                                   int a_lo, int a_hi, const Launch &L);
cudaError_t launch_set_populations(const KParams &P, int precision, const double *f, void *g,
                                   int a_lo, int a_hi, const Launch &L);

}  // namespace lbm
