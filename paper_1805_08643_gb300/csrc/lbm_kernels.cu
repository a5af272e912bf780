// Kernels of the pseudopotential MRT step and their launchers, for the D3Q19
// lattice of the paper (both operators) and its D3Q15 non-orthogonal variant
// (lbm_q15.cuh); the lattice is a template parameter Q of the one-node kernels.
//
// State layout: the stored buffer g holds, per direction a (SoA, a*N + i),
// the deviation of the post-collision population f*_a(x, t-1) from
// w_a rho_ref.  The post-streaming population of time t is pulled:
// f_a(x, t) = g_a(x - e_a) (Eq. 5).  One step is
//   psi pass:   rho(x,t) = sum_a f_a(x,t) -> psi(x)               (Eq. 6, EOS)
//   fused pass: pull f, F from psi (Eq. 15), u (Eq. 6), collide in moment
//               space (Eq. 4), store f*(x, t) at x into the other buffer.
#include <cuda_fp16.h>

#include <algorithm>

#include "lbm_collide64.cuh"
#include "lbm_device.cuh"
#include "lbm_internal.h"
#include "lbm_q15.cuh"

namespace lbm {

size_t storage_bytes(int precision) {
  return precision == kF64 ? 8 : (precision == kF32 ? 4 : 2);
}
size_t psi_elem_bytes(int precision) { return precision == kF64 ? 8 : 4; }

namespace {

template <int P> struct Types;
template <> struct Types<kF64> { using S = double; using T = double; using Psi = double; };
template <> struct Types<kF32> { using S = float; using T = float; using Psi = float; };
template <> struct Types<kF16> { using S = __half; using T = float; using Psi = float; };

// Lattice-dependent pieces of the one-node kernels.
template <int Q> struct Lat;
template <> struct Lat<19> {
  static __device__ __forceinline__ int src(const Nbhd &nb, int a) { return nb.src(a); }
  static __device__ __forceinline__ int dst(const Nbhd &nb, int a) { return nb.dst(a); }
  static __device__ __forceinline__ double w(int a) { return lattice_w(a); }
  template <typename S> static __device__ __forceinline__ typename Storage<S>::Compute decode(S v, int a) {
    return Storage<S>::decode(v, a);
  }
  template <typename S> static __device__ __forceinline__ typename Storage<S>::Compute load(const S *p, int a) {
    return Storage<S>::load(p, a);
  }
  template <typename S, typename T> static __device__ __forceinline__ void store(S *p, int a, T v) {
    Storage<S>::store(p, a, v);
  }
  template <typename T> static __device__ __forceinline__ void gradient(const T *p, T &Sx, T &Sy, T &Sz) {
    psi_gradient<T>(p, Sx, Sy, Sz);
  }
};
template <> struct Lat<15> {
  static __device__ __forceinline__ int src(const Nbhd &nb, int a) { return q15::src(nb, a); }
  static __device__ __forceinline__ int dst(const Nbhd &nb, int a) { return q15::dst(nb, a); }
  static __device__ __forceinline__ double w(int a) { return q15::w(a); }
  template <typename S> static __device__ __forceinline__ typename Storage<S>::Compute decode(S v, int a) {
    return q15::Storage<S>::decode(v, a);
  }
  template <typename S> static __device__ __forceinline__ typename Storage<S>::Compute load(const S *p, int a) {
    return q15::Storage<S>::load(p, a);
  }
  template <typename S, typename T> static __device__ __forceinline__ void store(S *p, int a, T v) {
    q15::Storage<S>::store(p, a, v);
  }
  template <typename T> static __device__ __forceinline__ void gradient(const T *p, T &Sx, T &Sy, T &Sz) {
    q15::psi_gradient<T>(p, Sx, Sy, Sz);
  }
};

// RO: through the read-only path (not in chained kernels: chain_wait).
template <int Q, bool RO, typename S, typename T>
__device__ __forceinline__ void pull_q(const S *g, int n, const Nbhd &nb, T f[Q]) {
#pragma unroll
  for (int a = 0; a < Q; ++a) {
    const S *p = g + (size_t)a * n + Lat<Q>::src(nb, a);
    f[a] = RO ? (T)Lat<Q>::load(p, a) : (T)Lat<Q>::template decode<S>(*p, a);
  }
}

// Stores one node's population of direction a, and its copy at the end of a padded row.
template <int Q, typename S, typename T>
__device__ __forceinline__ void store_node(S *__restrict__ g, int a, const KParams &P, const Nbhd &nb, T v) {
  S *at = g + (size_t)a * P.np + nb.self;
  Lat<Q>::store(at, a, v);
  if (sizeof(S) < sizeof(double) && P.px != P.nx && nb.x == 0) Lat<Q>::store(at + P.nx, a, v);
}

__device__ __forceinline__ bool node_of_thread(const KParams &P, int &x, int &y, int &z) {
  const unsigned p = blockIdx.x * blockDim.x + threadIdx.x;
  y = (int)(P.row_m ? __umulhi(p, P.row_m) : p / (unsigned)P.nx);
  x = (int)p - y * P.nx;
  z = blockIdx.z;
  return y < P.ny;
}

// ------------------------------------------------------------------ psi pass
template <int PREC, int EOS, bool DF, int Q>
__global__ void __launch_bounds__(256) psi_kernel(const typename Types<PREC>::S *g,
                                                  typename Types<PREC>::Psi *__restrict__ psi,
                                                  const KParams P, unsigned *__restrict__ err) {
  chain_wait();
  using S = typename Types<PREC>::S;
  using T = typename Types<PREC>::T;
  int x, y, z;
  if (!node_of_thread(P, x, y, z)) return;
  const Nbhd nb(x, y, z, P);
  T f[Q];
  pull_q<Q, false, S, T>(g, P.np, nb, f);
  T drho;
  if constexpr (PREC == kF64) {
    drho = sum64(f);
  } else if constexpr (Q == 15) {
    drho = q15::drho(f);
  } else {
    // sum in the order of the forward chain: rest + axis pairs + diagonal pairs
    const T sax = (f[1] + f[2]) + (f[3] + f[4]) + (f[5] + f[6]);
    const T sdg = ((f[7] + f[8]) + (f[9] + f[10])) + ((f[11] + f[12]) + (f[13] + f[14])) +
                  ((f[15] + f[16]) + (f[17] + f[18]));
    drho = f[0] + sax + sdg;
  }
  unsigned e = 0;
  if constexpr (PREC == kF64) {
    const double rho = P.rho_ref + drho;
    psi[nb.self] = eos_psi<EOS, double>(rho, narrow_f64(rho), P, e);
  } else {
    psi[nb.self] = DF ? eos_psi_f2<EOS>(drho, P, e) : eos_psi_d<EOS>(drho, P, e);
  }
  if (e) atomicOr(err, e);
}

// ------------------------------------------------------------------ fused pass
template <int PREC, int OP, bool SIGMA, int Q>
__global__ void __launch_bounds__(256) fused_kernel(const typename Types<PREC>::S *g_in,
                                                    typename Types<PREC>::S *__restrict__ g_out,
                                                    const typename Types<PREC>::Psi *psi,
                                                    const KParams P, const Coeffs64 C) {
  chain_wait();
  using S = typename Types<PREC>::S;
  using T = typename Types<PREC>::T;
  int x, y, z;
  if (!node_of_thread(P, x, y, z)) return;
  const Nbhd nb(x, y, z, P);
  T f[Q];
  pull_q<Q, false, S, T>(g_in, P.np, nb, f);
  // interaction force, Eq. 15
  T p[Q];
#pragma unroll
  for (int a = 1; a < Q; ++a) p[a] = (T)psi[Lat<Q>::dst(nb, a)];
  p[0] = (T)psi[nb.self];
  T Sx, Sy, Sz;
  auto out = [&](int a, T v) { Lat<Q>::store(g_out + (size_t)a * P.np + nb.self, a, v); };
  if constexpr (PREC == kF64) {
    psi_sums64(p, Sx, Sy, Sz);
    const double k = C.k[kForce] * p[0], S2 = SIGMA ? Sx * Sx + Sy * Sy + Sz * Sz : 0.0;
    collide64<OP>(f, P.rho_ref, k * Sx, k * Sy, k * Sz, S2, P, C, out);
    return;
  }
  Lat<Q>::gradient(p, Sx, Sy, Sz);
  const T k = -Phys<T>::G(P) * p[0];
  const T Fx = k * Sx, Fy = k * Sy, Fz = k * Sz;
  // Eq. 16: 6 sigma |F|^2 / (psi^2 (1/s_e - 1/2)) = sigma_coef |S|^2
  const T dS4 = SIGMA ? Phys<T>::sigma_coef(P) * (Sx * Sx + Sy * Sy + Sz * Sz) : T(0);
  const Rates<T> r(P);
  if constexpr (Q == 15)
    q15::collide<T>(f, Phys<T>::rho_ref(P), Fx, Fy, Fz, dS4, r);
  else if (OP == kNonOrth)
    collide_nonorth<T>(f, Phys<T>::rho_ref(P), Fx, Fy, Fz, dS4, r);
  else
    collide_orth<T>(f, Phys<T>::rho_ref(P), Fx, Fy, Fz, dS4, r);
#pragma unroll
  for (int a = 0; a < Q; ++a) out(a, f[a]);
}

// ------------------------------------------------------------------ observables
// rho and u (Eq. 6) of the current state, in FP64 whatever the storage.
//
// GB300 issues two FP64 instructions per SM and clock, so these kernels are
// bound by the FP64 unit unless almost all of the work runs elsewhere: with
// every conversion, sum and division in FP64 (149 instructions per node) the
// fields of a 256^3 FP32 box took 5.11 ms, against 0.28 ms for their bytes;
// they take 0.99 ms now (FP16 storage: 5.89 -> 0.98, FP64 at 128^3: 0.50 -> 0.31).
// Both forms below share the pair differences among the sums and take one
// reciprocal for the three velocities (0.82 ms without their remainders, which
// round each like a division).  The FP32-arithmetic forms also take their sums
// on the FP32 units, exactly (split_scale), which leaves 36 FP64 instructions
// per node.

__device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float mad(float a, float b, float c) { return fmaf(a, b, c); }

// sum_a v_a e_a (axis entries times axw) and, with R, r = sum_a v_a.
template <int Q, bool R, typename T>
__device__ __forceinline__ void moment_sums(const T v[Q], T axw, T &r, T &x, T &y, T &z) {
  const T d12 = v[1] - v[2], d34 = v[3] - v[4], d56 = v[5] - v[6];
  const T d78 = v[7] - v[8], d910 = v[9] - v[10], d1112 = v[11] - v[12], d1314 = v[13] - v[14];
  if (R) {
    r = v[0] + ((v[1] + v[2]) + (v[3] + v[4]) + (v[5] + v[6])) +
        ((v[7] + v[8]) + (v[9] + v[10]) + (v[11] + v[12]) + (v[13] + v[14]));
    if constexpr (Q == 19) r = r + ((v[15] + v[16]) + (v[17] + v[18]));
  }
  if constexpr (Q == 19) {
    const T d1516 = v[15] - v[16], d1718 = v[17] - v[18];
    x = mad(axw, d12, (d78 + d910) + (d1112 + d1314));
    y = mad(axw, d34, (d78 - d910) + (d1516 + d1718));
    z = mad(axw, d56, (d1112 - d1314) + (d1516 - d1718));
  } else {
    const T ab = d78 + d910, cd = d1112 - d1314;
    x = mad(axw, d12, ab + cd);
    y = mad(axw, d34, ab - cd);
    z = mad(axw, d56, (d78 - d910) + (d1112 + d1314));
  }
}

// Constants that split FP32 values v (all |v| < 2^(e+1), e the exponent of the
// largest) into v = h + l + t: adding and subtracting 1.5 * 2^(e+5) leaves h, a
// multiple of 2^(e-18); the same with 1.5 * 2^(e-15) splits the (exact)
// remainder into l, a multiple of 2^(e-38), and t, |t| <= 2^(e-39).  Sums of up
// to 32 times the largest value are then exact in FP32 over the h and over the
// l (24 bits hold them), and the FP32 sum of the t is good to 2^(e-54) at
// worst: closer than an FP64 sum of the v, whose every addition may round at
// 2^(e-53) and above.  (The error-free extraction of Rump, Ogita and Oishi's
// accurate summation.)  Not ok: infinities, NaN and ranges where the constants
// or the t would leave the normal numbers; those nodes sum in FP64.
struct SplitScale {
  float m1, m2;
  bool ok;
};
__device__ __forceinline__ SplitScale split_scale(unsigned max_abs_bits) {
  constexpr unsigned lo = (127u - 60u) << 23, hi = (127u + 60u) << 23;
  const unsigned ef = max_abs_bits & 0x7f800000u;
  SplitScale s;
  s.ok = max_abs_bits == 0u || (ef >= lo && ef <= hi);
  const unsigned e = s.ok ? max(ef, lo) : lo;
  s.m1 = __uint_as_float((e + (5u << 23)) | 0x400000u);
  s.m2 = __uint_as_float((e - (15u << 23)) | 0x400000u);
  return s;
}

// moment_sums of FP32 values through that split, assembled in FP64.  s is the scale of
// v[1..]: v[0] enters r alone and is added there, so that a large one leaves x, y
// and z their last places.
template <int Q, bool R>
__device__ __forceinline__ void moment_sums_split(float v[Q], float axw, const SplitScale &s, double &r, double &x,
                                                  double &y, double &z) {
  float h[3][4];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    float w[Q];
    const float m = k == 0 ? s.m1 : s.m2;
    w[0] = 0.f;
#pragma unroll
    for (int a = 1; a < Q; ++a) {
      w[a] = k == 2 ? v[a] : __fsub_rn(__fadd_rn(v[a], m), m);
      v[a] = __fsub_rn(v[a], w[a]);
    }
    moment_sums<Q, R, float>(w, axw, h[k][0], h[k][1], h[k][2], h[k][3]);
  }
  auto join = [&](int q) { return widen_f32(h[0][q]) + (widen_f32(h[1][q]) + widen_f32(h[2][q])); };
  if (R) r = widen_f32(v[0]) + join(0);
  x = join(1);
  y = join(2);
  z = join(3);
}

// Of v[1..].
template <int Q>
__device__ __forceinline__ unsigned max_abs_bits(const float v[Q]) {
  unsigned m = 0;
#pragma unroll
  for (int a = 1; a < Q; ++a) m = max(m, __float_as_uint(v[a]) & 0x7fffffffu);
  return m;
}

template <int PREC, int Q>
__device__ __forceinline__ void node_moments(const typename Types<PREC>::S *__restrict__ g,
                                             const typename Types<PREC>::Psi *__restrict__ psi,
                                             const KParams &P, const Nbhd &nb, double &rho,
                                             double &rux, double &ruy, double &ruz) {
  using S = typename Types<PREC>::S;
  using T = typename Types<PREC>::T;
  // the sums of Eq. 15 with the diagonal (corner) weight taken out: axis entries weigh 2 (8) times as much
  constexpr float axw = Q == 19 ? 2.0f : 8.0f;
  T f[Q], p[Q];
  pull_q<Q, true, S, T>(g, P.np, nb, f);
#pragma unroll
  for (int a = 1; a < Q; ++a) p[a] = psi[Lat<Q>::dst(nb, a)];
  p[0] = psi[nb.self];
  double drho, jx, jy, jz, sx, sy, sz, p0, unused;
  if constexpr (PREC == kF64) {
    moment_sums<Q, true, double>(f, 1.0, drho, jx, jy, jz);
    moment_sums<Q, false, double>(p, (double)axw, unused, sx, sy, sz);
    p0 = p[0];
  } else {
    const SplitScale cf = split_scale(max_abs_bits<Q>(f)), cp = split_scale(max_abs_bits<Q>(p));
    p0 = widen_f32(p[0]);
    if (cf.ok && cp.ok) {
      moment_sums_split<Q, true>(f, 1.0f, cf, drho, jx, jy, jz);
      moment_sums_split<Q, false>(p, axw, cp, unused, sx, sy, sz);
    } else {
      double d[Q];
#pragma unroll
      for (int a = 0; a < Q; ++a) d[a] = (double)f[a];
      moment_sums<Q, true, double>(d, 1.0, drho, jx, jy, jz);
#pragma unroll
      for (int a = 0; a < Q; ++a) d[a] = (double)p[a];
      moment_sums<Q, false, double>(d, (double)axw, unused, sx, sy, sz);
    }
  }
  const double k = P.half_force * p0;  // half the force: F / 2 = k (sx, sy, sz)
  rho = P.rho_ref + drho;
  rux = jx + k * sx;
  ruy = jy + k * sy;
  ruz = jz + k * sz;
}

template <int PREC, int Q>
__global__ void moments_kernel(const typename Types<PREC>::S *__restrict__ g,
                               const typename Types<PREC>::Psi *__restrict__ psi, const KParams P,
                               double *__restrict__ rho_out, double *__restrict__ u_out) {
  int x, y, z;
  if (!node_of_thread(P, x, y, z)) return;
  const Nbhd nb(x, y, z, P);
  double rho, rux, ruy, ruz;
  node_moments<PREC, Q>(g, psi, P, nb, rho, rux, ruy, ruz);
  const int i = x + P.nx * (y + P.ny * z);
  if (rho_out) rho_out[i] = rho;
  if (u_out) {
    const double inv = recip(rho);
    u_out[i] = quotient(rux, rho, inv);
    u_out[(size_t)P.n + i] = quotient(ruy, rho, inv);
    u_out[2 * (size_t)P.n + i] = quotient(ruz, rho, inv);
  }
}

// Block-partial FP64 sums of (rho, rho u) and max |u|, grid-stride over nodes,
// then one block folds the partials in a fixed order (deterministic).
template <int PREC, int Q>
__global__ void __launch_bounds__(256) diag_partial_kernel(const typename Types<PREC>::S *__restrict__ g,
                                                           const typename Types<PREC>::Psi *__restrict__ psi,
                                                           const KParams P, double *__restrict__ partials) {
  // sums of rho and rho u; of the fastest node |u|^2 (to compare by), |rho u|^2 and rho
  double acc[7] = {0, 0, 0, 0, 0, 0, 1};
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P.n; i += gridDim.x * blockDim.x) {
    const int x = i % P.nx, yz = i / P.nx, y = yz % P.ny, z = yz / P.ny;
    const Nbhd nb(x, y, z, P);
    double rho, rux, ruy, ruz;
    node_moments<PREC, Q>(g, psi, P, nb, rho, rux, ruy, ruz);
    acc[0] += rho;
    acc[1] += rux;
    acc[2] += ruy;
    acc[3] += ruz;
    const double inv = recip(rho);
    const double j2 = rux * rux + ruy * ruy + ruz * ruz;
    double u2 = j2 * inv * inv;
    if (__double2hiint(rho) < 0) u2 = -u2;  // a negative density never holds the maximum
    if (u2 > acc[4] || u2 != u2) acc[4] = u2, acc[5] = j2, acc[6] = rho;
  }
  __shared__ double red[7][256];
#pragma unroll
  for (int k = 0; k < 7; ++k) red[k][threadIdx.x] = acc[k];
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
#pragma unroll
      for (int k = 0; k < 4; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + s];
      const double a = red[4][threadIdx.x], b = red[4][threadIdx.x + s];
      if (b > a || b != b)
#pragma unroll
        for (int k = 4; k < 7; ++k) red[k][threadIdx.x] = red[k][threadIdx.x + s];
    }
    __syncthreads();
  }
  if (threadIdx.x < 4) partials[blockIdx.x * 5 + threadIdx.x] = red[threadIdx.x][0];
  if (threadIdx.x == 0) partials[blockIdx.x * 5 + 4] = sqrt(red[5][0]) / red[6][0];
}

// max over nodes of |u(x) - u_prev(x)| (Eq. 6 velocity, FP64), folded into
// *out with an atomic max on the bit pattern (non-negative doubles order like
// their bits); u_prev is overwritten with u in FP32.
template <int PREC, int Q>
__global__ void __launch_bounds__(256) max_du_kernel(const typename Types<PREC>::S *__restrict__ g,
                                                     const typename Types<PREC>::Psi *__restrict__ psi,
                                                     const KParams P, float *__restrict__ u_prev,
                                                     unsigned long long *__restrict__ out) {
  double m = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P.n; i += gridDim.x * blockDim.x) {
    const int x = i % P.nx, yz = i / P.nx, y = yz % P.ny, z = yz / P.ny;
    const Nbhd nb(x, y, z, P);
    double rho, rux, ruy, ruz;
    node_moments<PREC, Q>(g, psi, P, nb, rho, rux, ruy, ruz);
    const double inv = recip(rho);
    const double u[3] = {quotient(rux, rho, inv), quotient(ruy, rho, inv), quotient(ruz, rho, inv)};
    double d2 = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double d = u[k] - widen_f32(u_prev[(size_t)k * P.n + i]);
      d2 += d * d;
      u_prev[(size_t)k * P.n + i] = narrow_f64(u[k]);
    }
    m = (d2 > m || d2 != d2) ? d2 : m;
  }
  __shared__ double red[256];
  red[threadIdx.x] = m;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      const double a = red[threadIdx.x], b = red[threadIdx.x + s];
      red[threadIdx.x] = (b > a || b != b) ? b : a;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) atomicMax(out, (unsigned long long)__double_as_longlong(sqrt(red[0])));
}

// One block: each thread folds every 256th partial, then a tree.  (One thread
// folding the 1024 partials in a row took 0.37 ms, most of a diag of a small box.)
__global__ void __launch_bounds__(256) diag_final_kernel(const double *__restrict__ partials, int nblocks,
                                                         double *__restrict__ result) {
  __shared__ double red[5][256];
  double acc[5] = {0, 0, 0, 0, 0};
  for (int b = threadIdx.x; b < nblocks; b += 256) {
    for (int k = 0; k < 4; ++k) acc[k] += partials[b * 5 + k];
    const double u = partials[b * 5 + 4];
    acc[4] = (u > acc[4] || u != u) ? u : acc[4];
  }
  for (int k = 0; k < 5; ++k) red[k][threadIdx.x] = acc[k];
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      for (int k = 0; k < 4; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + s];
      const double a = red[4][threadIdx.x], b = red[4][threadIdx.x + s];
      red[4][threadIdx.x] = (b > a || b != b) ? b : a;
    }
    __syncthreads();
  }
  if (threadIdx.x < 5) result[threadIdx.x] = red[threadIdx.x][0];
}

// ------------------------------------------------------------------ initial state
__device__ __forceinline__ double min_image(double d, int n) {
  d = fabs(d);
  return fmin(d, (double)n - d);
}

// Eq. 59 for each droplet of the chunk; several droplets combine by maximum.
__global__ void rho_droplets_kernel(double *__restrict__ rho, const KParams P, const DropletChunk C,
                                    double W, double rho_l, double rho_v, int first) {
  int x, y, z;
  if (!node_of_thread(P, x, y, z)) return;
  const int i = x + P.nx * (y + P.ny * z);
  double best = first ? -1e300 : rho[i];
  for (int k = 0; k < C.count; ++k) {
    const double dx = min_image(x - C.cx[k], P.nx), dy = min_image(y - C.cy[k], P.ny);
    const double dz = min_image(z - C.cz[k], P.nz);
    const double r = sqrt(dx * dx + dy * dy + dz * dz);
    const double v = 0.5 * (rho_l + rho_v) - 0.5 * (rho_l - rho_v) * tanh(2.0 * (r - C.r[k]) / W);
    best = fmax(best, v);
  }
  rho[i] = best;
}

// Liquid slab between planes lo and hi across one axis (Sec. IV D).
__global__ void rho_slab_kernel(double *__restrict__ rho, const KParams P, int axis, double lo,
                                double hi, double W, double rho_l, double rho_v) {
  int x, y, z;
  if (!node_of_thread(P, x, y, z)) return;
  const double c = axis == 0 ? x : (axis == 1 ? y : z);
  rho[x + P.nx * (y + P.ny * z)] =
      rho_v + 0.5 * (rho_l - rho_v) * (tanh(2.0 * (c - lo) / W) - tanh(2.0 * (c - hi) / W));
}

// f_a(x, 0) = w_a rho0(x): store g_a(y) = w_a (rho0(y + e_a) - rho_ref).
template <int PREC, int Q>
__global__ void state_from_rho_kernel(const double *__restrict__ rho, typename Types<PREC>::S *__restrict__ g,
                                      const KParams P) {
  using S = typename Types<PREC>::S;
  int x, y, z;
  if (!node_of_thread(P, x, y, z)) return;
  const Nbhd nb(x, y, z, P), pub(x, y, z, P, PREC == kF64 ? P.px : P.nx);
#pragma unroll
  for (int a = 0; a < Q; ++a) {
    const double v = Lat<Q>::w(a) * (rho[Lat<Q>::dst(pub, a)] - P.rho_ref);
    store_node<Q>(g, a, P, nb, (typename Types<PREC>::T)v);
  }
}

// out[(a - a_lo) N + i] = f_a(x_i, t) for a in [a_lo, a_hi).
template <int PREC, int Q>
__global__ void get_populations_kernel(const typename Types<PREC>::S *__restrict__ g, double *__restrict__ out,
                                       const KParams P, int a_lo, int a_hi) {
  using S = typename Types<PREC>::S;
  int x, y, z;
  if (!node_of_thread(P, x, y, z)) return;
  const Nbhd nb(x, y, z, P);
  const int i = PREC == kF64 ? nb.self : x + P.nx * (y + P.ny * z);
#pragma unroll
  for (int a = 0; a < Q; ++a)
    if (a >= a_lo && a < a_hi)
      out[(size_t)(a - a_lo) * P.n + i] =
          Lat<Q>::w(a) * P.rho_ref + (double)Lat<Q>::load(g + (size_t)a * P.np + Lat<Q>::src(nb, a), a);
}

// Reverse of the above: g_a(y) = f_a(y + e_a) - w_a rho_ref.
template <int PREC, int Q>
__global__ void set_populations_kernel(const double *__restrict__ f, typename Types<PREC>::S *__restrict__ g,
                                       const KParams P, int a_lo, int a_hi) {
  using S = typename Types<PREC>::S;
  int x, y, z;
  if (!node_of_thread(P, x, y, z)) return;
  const Nbhd nb(x, y, z, P), pub(x, y, z, P, PREC == kF64 ? P.px : P.nx);
#pragma unroll
  for (int a = 0; a < Q; ++a)
    if (a >= a_lo && a < a_hi) {
      const double v = f[(size_t)(a - a_lo) * P.n + Lat<Q>::dst(pub, a)] - Lat<Q>::w(a) * P.rho_ref;
      store_node<Q>(g, a, P, nb, (typename Types<PREC>::T)v);
    }
}

dim3 node_grid(const KParams &P, int threads = kThreads) { return plane_grid(P.nx * P.ny, P.nz, threads); }

// Nodes from which the kernels of a precision are chained (launch_chained).
template <int PREC> bool chained(const KParams &P) { return P.n >= (PREC == kF64 ? kChainFP64 : kChainPairs); }

template <int PREC, bool DF, int Q>
cudaError_t psi_dispatch(const KParams &P, const void *g, void *psi, unsigned *err, const Launch &L) {
  using S = typename Types<PREC>::S;
  using Psi = typename Types<PREC>::Psi;
  auto run = [&](auto kernel) {
    return launch_chained(chained<PREC>(P), kernel, node_grid(P), dim3(kThreads), L.stream, (const S *)g, (Psi *)psi, P,
                          err);
  };
  switch (P.eos) {
    case kEosCS: return run(psi_kernel<PREC, kEosCS, DF, Q>);
    case kEosExp: return run(psi_kernel<PREC, kEosExp, DF, Q>);
    default: return run(psi_kernel<PREC, kEosNone, DF, Q>);
  }
}

template <int PREC, int OP, int Q>
cudaError_t fused_dispatch(const KParams &P, bool sigma, const void *g_in, void *g_out, const void *psi,
                           const Launch &L) {
  using S = typename Types<PREC>::S;
  using Psi = typename Types<PREC>::Psi;
  // FP64: blocks of one warp.  Every warp holds the SM's FP64 unit for the same time, so the last round is
  // shortest when warps are dealt out singly: 32^3 steps 20.5 -> 18.5 us (blocks of four warps leave 8 on some
  // SMs, single ones 7), no difference from 64^3 on.
  constexpr int threads = PREC == kF64 ? 32 : kThreads;
  const Coeffs64 C = coeffs64(P, Q == 15 ? kNonOrthQ15 : OP);
  auto kernel = sigma ? fused_kernel<PREC, OP, true, Q> : fused_kernel<PREC, OP, false, Q>;
  return launch_chained(chained<PREC>(P), kernel, node_grid(P, threads), dim3(threads), L.stream, (const S *)g_in,
                        (S *)g_out, (const Psi *)psi, P, C);
}

}  // namespace

cudaError_t launch_psi(const KParams &P, int precision, const void *g, void *psi, unsigned *err,
                       const Launch &L, bool df) {
  if (P.q == 15) {
    if (pair_supported(P, precision)) return launch_psi_pair(P, precision, g, psi, err, L, df);
    switch (precision) {
      case kF64: return psi_dispatch<kF64, false, 15>(P, g, psi, err, L);
      case kF32:
        return df ? psi_dispatch<kF32, true, 15>(P, g, psi, err, L) : psi_dispatch<kF32, false, 15>(P, g, psi, err, L);
      default:
        return df ? psi_dispatch<kF16, true, 15>(P, g, psi, err, L) : psi_dispatch<kF16, false, 15>(P, g, psi, err, L);
    }
  }
  switch (precision) {
    case kF64: return psi_dispatch<kF64, false, 19>(P, g, psi, err, L);
    case kF32:
      if (pair_supported(P, precision)) return launch_psi_pair(P, precision, g, psi, err, L, df);
      return df ? psi_dispatch<kF32, true, 19>(P, g, psi, err, L) : psi_dispatch<kF32, false, 19>(P, g, psi, err, L);
    default:
      if (pair_supported(P, precision)) return launch_psi_pair(P, precision, g, psi, err, L, df);
      return df ? psi_dispatch<kF16, true, 19>(P, g, psi, err, L) : psi_dispatch<kF16, false, 19>(P, g, psi, err, L);
  }
}

cudaError_t launch_fused(const KParams &P, int precision, int op, bool sigma, const void *g_in, void *g_out,
                         const void *psi, const Launch &L) {
  if (P.q == 15) {
    if (pair_supported(P, precision)) return launch_fused_pair(P, precision, op, sigma, g_in, g_out, psi, L);
    switch (precision) {
      case kF64: return fused_dispatch<kF64, kNonOrth, 15>(P, sigma, g_in, g_out, psi, L);
      case kF32: return fused_dispatch<kF32, kNonOrth, 15>(P, sigma, g_in, g_out, psi, L);
      default: return fused_dispatch<kF16, kNonOrth, 15>(P, sigma, g_in, g_out, psi, L);
    }
  }
  if (pair_supported(P, precision)) return launch_fused_pair(P, precision, op, sigma, g_in, g_out, psi, L);
  if (op == kNonOrth) {
    switch (precision) {
      case kF64: return fused_dispatch<kF64, kNonOrth, 19>(P, sigma, g_in, g_out, psi, L);
      case kF32: return fused_dispatch<kF32, kNonOrth, 19>(P, sigma, g_in, g_out, psi, L);
      default: return fused_dispatch<kF16, kNonOrth, 19>(P, sigma, g_in, g_out, psi, L);
    }
  }
  switch (precision) {
    case kF64: return fused_dispatch<kF64, kOrth, 19>(P, sigma, g_in, g_out, psi, L);
    case kF32: return fused_dispatch<kF32, kOrth, 19>(P, sigma, g_in, g_out, psi, L);
    default: return fused_dispatch<kF16, kOrth, 19>(P, sigma, g_in, g_out, psi, L);
  }
}

// CALL with PR = the precision and QQ = the lattice, both compile-time constants.
#define LBM_PREC_SWITCH_Q(precision, QV, CALL)                     \
  switch (precision) {                                             \
    case kF64: { constexpr int PR = kF64, QQ = QV; CALL; } break; \
    case kF32: { constexpr int PR = kF32, QQ = QV; CALL; } break; \
    default: { constexpr int PR = kF16, QQ = QV; CALL; } break;   \
  }
#define LBM_PREC_SWITCH(precision, CALL)                         \
  if (P.q == 15) {                                               \
    LBM_PREC_SWITCH_Q(precision, 15, CALL)                       \
  } else {                                                       \
    LBM_PREC_SWITCH_Q(precision, 19, CALL)                       \
  }

cudaError_t launch_moments(const KParams &P, int precision, const void *g, const void *psi, double *rho,
                           double *u, const Launch &L) {
  const dim3 grid = node_grid(P), block(kThreads);
  LBM_PREC_SWITCH(precision, (moments_kernel<PR, QQ><<<grid, block, 0, L.stream>>>(
                                 (const typename Types<PR>::S *)g, (const typename Types<PR>::Psi *)psi, P, rho, u)));
  return cudaGetLastError();
}

cudaError_t launch_diag(const KParams &P, int precision, const void *g, const void *psi, double *partials,
                        double *result, const Launch &L) {
  LBM_PREC_SWITCH(precision, (diag_partial_kernel<PR, QQ><<<kReduceBlocks, 256, 0, L.stream>>>(
                                 (const typename Types<PR>::S *)g, (const typename Types<PR>::Psi *)psi, P, partials)));
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  diag_final_kernel<<<1, 256, 0, L.stream>>>(partials, kReduceBlocks, result);
  return cudaGetLastError();
}

cudaError_t launch_max_du(const KParams &P, int precision, const void *g, const void *psi, float *u_prev,
                          double *out, const Launch &L) {
  const int blocks = (int)std::min<long long>(4 * 152, ((long long)P.n + 255) / 256);
  LBM_PREC_SWITCH(precision, (max_du_kernel<PR, QQ><<<blocks, 256, 0, L.stream>>>(
                                 (const typename Types<PR>::S *)g, (const typename Types<PR>::Psi *)psi, P, u_prev,
                                 (unsigned long long *)out)));
  return cudaGetLastError();
}

cudaError_t launch_rho_droplets(const KParams &P, double *rho, const DropletChunk &chunk, double W,
                                double rho_l, double rho_v, bool first, const Launch &L) {
  rho_droplets_kernel<<<node_grid(P), kThreads, 0, L.stream>>>(rho, P, chunk, W, rho_l, rho_v,
                                                                           first ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_rho_slab(const KParams &P, double *rho, int axis, double lo, double hi, double W,
                            double rho_l, double rho_v, const Launch &L) {
  rho_slab_kernel<<<node_grid(P), kThreads, 0, L.stream>>>(rho, P, axis, lo, hi, W, rho_l, rho_v);
  return cudaGetLastError();
}

cudaError_t launch_state_from_rho(const KParams &P, int precision, const double *rho, void *g, const Launch &L) {
  const dim3 grid = node_grid(P), block(kThreads);
  LBM_PREC_SWITCH(precision, (state_from_rho_kernel<PR, QQ><<<grid, block, 0, L.stream>>>(
                                 rho, (typename Types<PR>::S *)g, P)));
  return cudaGetLastError();
}

cudaError_t launch_get_populations(const KParams &P, int precision, const void *g, double *out, int a_lo,
                                   int a_hi, const Launch &L) {
  const dim3 grid = node_grid(P), block(kThreads);
  LBM_PREC_SWITCH(precision, (get_populations_kernel<PR, QQ><<<grid, block, 0, L.stream>>>(
                                 (const typename Types<PR>::S *)g, out, P, a_lo, a_hi)));
  return cudaGetLastError();
}

cudaError_t launch_set_populations(const KParams &P, int precision, const double *f, void *g, int a_lo,
                                   int a_hi, const Launch &L) {
  const dim3 grid = node_grid(P), block(kThreads);
  LBM_PREC_SWITCH(precision, (set_populations_kernel<PR, QQ><<<grid, block, 0, L.stream>>>(
                                 f, (typename Types<PR>::S *)g, P, a_lo, a_hi)));
  return cudaGetLastError();
}

}  // namespace lbm
