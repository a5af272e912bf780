// The collisions of the FP64 kernels, both D3Q19 operators and the D3Q15
// variant, written for few FP64 instructions: the FP64 unit (two instructions
// per SM and clock) is all that bounds these kernels.  The reduced-precision
// kernels keep the moment-by-moment forms of lbm_device.cuh and lbm_q15.cuh:
// they are bound by memory and registers, and holding F, u and B through the
// inverse transform costs more registers than the instructions are worth there
// (the FP32 work list spilled 90 bytes a thread and went from 527 to 598 us
// per 256^3 step).
//
// Every moment relaxes as m* = m - s (m - m_eq) + (1 - s/2) S (Eq. 4).  Here:
//  - m* = a m + s m_eq + c S with a = 1 - s, c = 1 - s/2, the inverse
//    transform's constant factors (1/4, 1/6, ...) multiplied into a, s and c on
//    the host (coeffs64), but for the even moments that carry the density (relax4);
//  - rho u_i u_j and F_i u_j + F_j u_i relax with the same rate, so s rho u_i u_j
//    + c (F_i u_j + F_j u_i) = u_i B_j + u_j B_i, B_i = s rho u_i / 2 + c F_i;
//  - the third-order moments of a pair of diagonals (corners) relax with one
//    rate: the differences d78, d910, ... relax themselves, no moments are formed;
//  - 2 x + y is written fma(2, x, y) (2 * x + y compiles to two additions), and
//    the reciprocal takes three instructions (recip).
//  - the linear parts (the forward and inverse chains, the sums of Eq. 15) run on
//    the integer units, as sums of 64-bit fixed-point numbers: see Fixed.
// FP64 instructions per node of the fused pass, with the force: 104 non-orthogonal
// (255 moment by moment, 214 with these formulas in FP64 throughout), 92 orthogonal
// (304, 259), 88 on D3Q15.  Fused pass at 128^3, FP64 throughout -> as it is: 855 ->
// 434, 1018 -> 401 and 725 -> 352 us; bound by the FP64 unit (the FP64 instructions
// alone take 347 us; at 64^3 its pipe is busy 76 % of the time, the integer one 49 %).
// More resident warps (96 registers) and larger blocks are within 2 % of it.  Errors
// of a step's populations against extended precision (droplets and slabs, with and
// without noise, T/Tc 0.70 to 0.85, a = 0.25): 0.63 - 0.93 (non-orthogonal), 0.72 - 0.90
// (orthogonal) and 0.56 - 0.76 (D3Q15) of what FP64 throughout has.
#pragma once

#include <type_traits>

#include "lbm_device.cuh"
#include "lbm_internal.h"

namespace lbm {

// The coefficients that follow the shear rate (kN5 ...), of the box or of the
// node (density-dependent viscosity).
struct Shear64 {
  double n5, n7, b1, b2, nx;
};
template <int Q>
__device__ __forceinline__ Shear64 shear64(const KParams &P, const Coeffs64 &C, double rho) {
  if (!P.varnu) return Shear64{C.k[kN5], C.k[kN7], C.k[kNb1], C.k[kNb2], C.k[kON]};
  const double s = shear_rate(Rates<double>(P), rho), a = 1.0 - s;
  if (Q == 15) return Shear64{a * (1.0 / 12.0), a * 0.25, s * 0.0625, 0.125 - s * 0.0625, a * 0.125};
  return Shear64{a * (1.0 / 12.0), a * 0.25, s * 0.125, 0.25 - s * 0.125, a * (1.0 / 36.0)};
}

// ------------------------------------------------------------------ linear parts
// A chain of additions and small integer factors over values of one node, in the
// numbers of a scale c: doubles (InDouble), or 64-bit fixed-point ones (InFixed).
// An FP64 addition takes 16 cycles of an SM's FP64 unit for a warp (19 as it runs),
// a 64-bit integer one a single cycle of the integer units, and the conversions
// about 6 and 12.
//
// InFixed<S>: v 2^(1075 + S - E) for the largest exponent field E of the values the
// chain starts from, so those have at most 53 + S bits; S is the largest for which
// the chain's sums of factors, 2^(10 - S) at most, cannot leave 64 bits whatever
// the values.  Sums are exact.  A value is cut off S bits below the last place of
// the largest one, and a result is rounded once (to nearest, ties to even), where
// an FP64 sum rounds each partial result: what is lost is less than a last place of
// the largest value over 2^S for each value cut, and values within a factor 2^S of the
// largest lose nothing.  What a chain starts from is chosen accordingly (of the inverse
// chains everything but drho, which only the rest population takes).
struct Fixed {
  long long v;
};
__device__ __forceinline__ Fixed operator+(Fixed a, Fixed b) { return {a.v + b.v}; }
__device__ __forceinline__ Fixed operator-(Fixed a, Fixed b) { return {a.v - b.v}; }
template <int K> __device__ __forceinline__ Fixed times(Fixed a) { return {a.v * K}; }
template <int K> __device__ __forceinline__ double times(double a) { return (double)K * a; }

struct InDouble {
  using Value = double;
  __device__ __forceinline__ double in(double v) const { return v; }
  __device__ __forceinline__ double out(double v) const { return v; }
  __device__ __forceinline__ double out_half(double v) const { return 0.5 * v; }
  template <int K> __device__ __forceinline__ double out_over(double v) const { return v * (1.0 / (1 << K)); }
  __device__ __forceinline__ double out_twice(double v) const { return 2.0 * v; }
  static __device__ __forceinline__ double half(double v) { return 0.5 * v; }
};
template <int S> struct InFixed {
  using Value = Fixed;
  int E;
  __device__ __forceinline__ Fixed in(double v) const {
    const int hi = __double2hiint(v);
    const unsigned d = (unsigned)(E - ((hi >> 20) & 0x7ff));  // a zero is shifted out
    unsigned long long m = ((unsigned long long)(((unsigned)hi & 0xfffffu) | 0x100000u) << 32 | (unsigned)__double2loint(v)) << S;
    m >>= min(d, 63u);
    const long long s = (long long)(hi >> 31);
    return {((long long)m ^ s) - s};
  }
  __device__ __forceinline__ double out(Fixed x) const { return back(x, E); }
  __device__ __forceinline__ double out_half(Fixed x) const { return back(x, E - 1); }
  template <int K> __device__ __forceinline__ double out_over(Fixed x) const { return back(x, E - K); }  // over 2^K
  __device__ __forceinline__ double out_twice(Fixed x) const { return back(x, E + 1); }
  static __device__ __forceinline__ Fixed half(Fixed x) { return {x.v >> 1}; }
  static __device__ __forceinline__ double back(Fixed x, int E) {
    const long long s = x.v >> 63;
    const unsigned long long u = (unsigned long long)((x.v ^ s) - s);
    const int lz = __clzll((long long)u);
    const unsigned long long n = u << (lz & 63), m = n >> 11;  // 53 bits, the top one at 2^(E + 11 - S - lz)
    const unsigned rest = ((unsigned)n & 0x7ffu) + ((unsigned)m & 1u) + 0x3ffu;
    const unsigned long long r = m + (rest >> 11);  // a carry out of the fraction moves into the exponent
    const unsigned hi = (unsigned)(r >> 32) + ((unsigned)(E + 10 - S - lz) << 20);
    return u == 0 ? 0.0 : __hiloint2double((int)(hi | ((unsigned)s & 0x80000000u)), (int)(unsigned)r);
  }
};

// E for the values from index I on; -1 where Fixed is not for them (infinities, NaN, nothing but very small values).
template <int I = 0, int N>
__device__ __forceinline__ int top_exponent(const double (&v)[N]) {
  unsigned m = 0;
#pragma unroll
  for (int k = I; k < N; ++k) m = max(m, (unsigned)__double2hiint(v[k]) & 0x7fffffffu);
  const int e = (int)(m >> 20);
  if (m == 0) return 128;
  return e >= 128 && e < 2000 ? e : -1;
}

// The sums of Eq. 15 in units of the diagonal (D3Q15: corner) weight, where
// the axes weigh 2 (8).  p[a] = psi(x + e_a).
template <int Q, typename C>
__device__ __forceinline__ void psi_sums_l(const double p[Q], const C &c, double &Sx, double &Sy, double &Sz) {
  using L = typename C::Value;
  constexpr int axw = Q == 19 ? 2 : 8;
  L q[Q];
#pragma unroll
  for (int a = 1; a < Q; ++a) q[a] = c.in(p[a]);
  const L d78 = q[7] - q[8], d910 = q[9] - q[10], d1112 = q[11] - q[12], d1314 = q[13] - q[14];
  if constexpr (Q == 19) {
    const L d1516 = q[15] - q[16], d1718 = q[17] - q[18];
    Sx = c.out(times<axw>(q[1] - q[2]) + ((d78 + d910) + (d1112 + d1314)));
    Sy = c.out(times<axw>(q[3] - q[4]) + ((d78 - d910) + (d1516 + d1718)));
    Sz = c.out(times<axw>(q[5] - q[6]) + ((d1112 - d1314) + (d1516 - d1718)));
  } else {
    const L ab = d78 + d910, cd = d1112 - d1314;
    Sx = c.out(times<axw>(q[1] - q[2]) + (ab + cd));
    Sy = c.out(times<axw>(q[3] - q[4]) + (ab - cd));
    Sz = c.out(times<axw>(q[5] - q[6]) + ((d78 - d910) + (d1112 + d1314)));
  }
}
template <int Q>
__device__ __forceinline__ void psi_sums64(const double (&p)[Q], double &Sx, double &Sy, double &Sz) {
  const int E = top_exponent(p);
  if (E >= 0)
    psi_sums_l<Q>(p, InFixed<Q == 19 ? 6 : 5>{E}, Sx, Sy, Sz);  // factors up to 12, 24
  else
    psi_sums_l<Q>(p, InDouble{}, Sx, Sy, Sz);
}

// Sum of a node's populations.  The psi pass is bound by the FP64 unit as well: with
// this sum, and its rounding to FP32 and its tests on integers, it does 18 FP64
// instructions a node instead of 38, 128^3 153 -> 80 us (49 us of memory traffic).
template <int Q>
__device__ __forceinline__ double sum64(const double (&f)[Q]) {
  auto sum = [&](const auto &c) {
    auto t = c.in(f[0]);
#pragma unroll
    for (int a = 1; a < Q; ++a) t = t + c.in(f[a]);
    return c.out(t);
  };
  const int E = top_exponent(f);
  return E >= 0 ? sum(InFixed<5>{E}) : sum(InDouble{});
}

// What the nonlinear parts need of a node's collision.
struct Node64 {
  double rho, Fx, Fy, Fz, S2;
  double rux, ruy, ruz, ux, uy, uz, qxx, qyy, qzz, Fux, Fuy, Fuz;
  // j: momenta of the populations; Eq. 6
  __device__ __forceinline__ Node64(double rho_, double jx, double jy, double jz, double Fx_, double Fy_, double Fz_,
                                    double S2_)
      : rho(rho_), Fx(Fx_), Fy(Fy_), Fz(Fz_), S2(S2_) {
    const double inv_rho = recip(rho);
    rux = jx + 0.5 * Fx, ruy = jy + 0.5 * Fy, ruz = jz + 0.5 * Fz;
    ux = rux * inv_rho, uy = ruy * inv_rho, uz = ruz * inv_rho;
    qxx = rux * ux, qyy = ruy * uy, qzz = ruz * uz;  // rho u_i^2
    Fux = Fx * ux, Fuy = Fy * uy, Fuz = Fz * uz;
  }
};

// The even moments that carry the density, m4 and the fourth-order ones, of the
// raw-monomial bases (the non-orthogonal operator and D3Q15): m + s d with the small d =
// m_eq + (c / s) S - m.  (As a m + s m_eq + c S, whose terms all round at the size of m,
// rest populations were up to a fifth further off than FP64 sums'.)  m4, the density's
// part of m_eq and m subtracted first, which leaves one rounding at its size:
__device__ __forceinline__ double relax4(double m, double drho, double usq, double Fu, double S2, const Coeffs64 &C) {
  const double d = (drho - m) + fma(C.k[kE5], S2, fma(C.k[kE4], Fu, usq));
  return fma(C.k[kE1], d, m);
}

// ------------------------------------------------------------------ non-orthogonal operator
// f* = M^-1 m* (App. A) from drho - m4*, e4 = m4* / 6, e5 = m5* / 12, e6 = m6* / 4,
// p_k = m_k* / 4 (16, 17, 18, 7, 8, 9), twice the odd parts of the axes, and the
// odd parts of the diagonals.
template <typename Sc, typename Out>
__device__ __forceinline__ void inverse_nonorth_l(const double (&v)[19], const Sc &c, Out &&out) {
  using L = typename Sc::Value;
  const L e4 = c.in(v[1]), e5 = c.in(v[2]), e6 = c.in(v[3]);
  const L p16 = c.in(v[4]), p17 = c.in(v[5]), p18 = c.in(v[6]);
  const L a = p16 + p17;
  out(0, fma(4.0, c.out(a + p18), v[0]));  // v[0] in the sums would set their cut
  auto axis = [&](int k, const L &even2, double odd2) {  // both twice their value
    const L o = c.in(odd2);
    out(k, c.out_half(even2 + o));
    out(k + 1, c.out_half(even2 - o));
  };
  const L e45 = e4 - e5;
  axis(1, times<2>(e4 + times<2>(e5)) - times<4>(a), v[10]);
  axis(3, times<2>(e45 + e6) - times<4>(p16 + p18), v[11]);
  axis(5, times<2>(e45 - e6) - times<4>(p17 + p18), v[12]);
  auto diagonal = [&](int k, const L &p, double shear, double odd1, double odd2) {
    const L s = c.in(shear), o1 = c.in(odd1), o2 = c.in(odd2), ev = p + s, ew = p - s;
    out(k, c.out(ev + o1));
    out(k + 1, c.out(ev - o1));
    out(k + 2, c.out(ew + o2));
    out(k + 3, c.out(ew - o2));
  };
  diagonal(7, p16, v[7], v[13], v[14]);
  diagonal(11, p17, v[8], v[15], v[16]);
  diagonal(15, p18, v[9], v[17], v[18]);
}

// Forward chains of Eq. 12 (deviation form, m - rho_ref M w), equilibria Eq. 13,
// forcing Eq. 14, the Eq. 16 term from S2 (the squared sum of Eq. 15).  f_ holds the
// deviations f_a - w_a rho_ref; out(a, f*_a) takes the results (deviations again).
template <typename Sc, typename Out>
__device__ __forceinline__ void collide_nonorth_l(const double (&f_)[19], const Sc &c, double rho_ref, double Fx,
                                                  double Fy, double Fz, double S2, const KParams &P, const Coeffs64 &C,
                                                  Out &&out) {
  using L = typename Sc::Value;
  L f[19];
#pragma unroll
  for (int a = 0; a < 19; ++a) f[a] = c.in(f_[a]);
  const L s12 = f[1] + f[2], d12 = f[1] - f[2];
  const L s34 = f[3] + f[4], d34 = f[3] - f[4];
  const L s56 = f[5] + f[6], d56 = f[5] - f[6];
  const L s78 = f[7] + f[8], d78 = f[7] - f[8];
  const L s910 = f[9] + f[10], d910 = f[9] - f[10];
  const L s1112 = f[11] + f[12], d1112 = f[11] - f[12];
  const L s1314 = f[13] + f[14], d1314 = f[13] - f[14];
  const L s1516 = f[15] + f[16], d1516 = f[15] - f[16];
  const L s1718 = f[17] + f[18], d1718 = f[17] - f[18];
  const L l16 = s78 + s910, l17 = s1112 + s1314, l18 = s1516 + s1718;
  const L lx = (d78 + d910) + (d1112 + d1314);    // m11 + m13
  const L ly = (d78 - d910) + (d1516 + d1718);    // m10 + m15
  const L lz = (d1112 - d1314) + (d1516 - d1718);  // m12 + m14
  const L syz = s34 + s56, sax = s12 + syz, sxx = l16 + l17, sdg = sxx + l18;
  const double drho = c.out(f[0] + sax + sdg);
  const double Dx = c.out(lx), Dy = c.out(ly), Dz = c.out(lz);
  const double jx = c.out(d12 + lx), jy = c.out(d34 + ly), jz = c.out(d56 + lz);
  const Node64 N(rho_ref + drho, jx, jy, jz, Fx, Fy, Fz, S2);
  const double usq = N.qxx + N.qyy + N.qzz, Fu = N.Fux + N.Fuy + N.Fuz;
  double v[19];
  // relaxed moments (Eq. 4 with Eqs. 11, 13, 14, 16), scaled as the inverse takes them
  const double m4 = relax4(c.out(sax + times<2>(sdg)), drho, usq, Fu, S2, C);
  v[0] = drho - m4;
  v[1] = (1.0 / 6.0) * m4;
  // Eq. 13's phi + (rho - rho_ref)/9 and third-axis parts, over 4: m16 takes the sum over the axes less the z part, ...
  // (the three share the density's part of m_eq: subtracting it from each m first rounds a little less, 0.60 - 0.82 of
  // FP64 throughout against 0.63 - 0.93, for 514 instead of 506 us at 128^3)
  const double c4 = fma(1.0 / 36.0, drho, fma(C.k[kP4], Fu, (1.0 / 24.0) * usq));
  auto relax_p = [&](double m, double q, double Fq) {
    return fma(C.k[kP1], fma(-C.k[kP4], Fq, fma(-1.0 / 12.0, q, c4)) - m, m);
  };
  v[4] = relax_p(c.template out_over<2>(l16), N.qzz, N.Fuz);
  v[5] = relax_p(c.template out_over<2>(l17), N.qyy, N.Fuy);
  v[6] = relax_p(c.template out_over<2>(l18), N.qxx, N.Fux);
  const Shear64 n = shear64<19>(P, C, N.rho);
  const double Bx = n.b1 * N.rux + n.b2 * Fx, By = n.b1 * N.ruy + n.b2 * Fy, Bz = n.b1 * N.ruz + n.b2 * Fz;
  const double Gx = N.ux * Bx, Gy = N.uy * By, Gz = N.uz * Bz;
  v[2] = fma(-2.0 / 3.0, fma(-2.0, Gx, Gy + Gz), n.n5 * c.out(times<2>(s12 - l18) + (sxx - syz)));
  v[3] = fma(2.0, Gy - Gz, n.n7 * c.out((s34 - s56) + (l16 - l17)));
  v[7] = n.n7 * c.out(s78 - s910) + N.ux * By + N.uy * Bx;
  v[8] = n.n7 * c.out(s1112 - s1314) + N.ux * Bz + N.uz * Bx;
  v[9] = n.n7 * c.out(s1516 - s1718) + N.uy * Bz + N.uz * By;
  // odd parts: b_i carries Eq. 13/14's rho u_i / 3 and F_i / 3 of the third-order moments; 2 kQa = 1 - s_q
  const double bx = C.k[kQb1] * N.rux + C.k[kQb2] * Fx, by = C.k[kQb1] * N.ruy + C.k[kQb2] * Fy;
  const double bz = C.k[kQb1] * N.ruz + C.k[kQb2] * Fz, qa = C.k[kQa], q2 = -C.k[kQ2];
  v[10] = fma(-8.0, bx, fma(q2, Dx, jx + Fx));
  v[11] = fma(-8.0, by, fma(q2, Dy, jy + Fy));
  v[12] = fma(-8.0, bz, fma(q2, Dz, jz + Fz));
  v[13] = qa * c.out(d78) + (bx + by);
  v[14] = qa * c.out(d910) + (bx - by);
  v[15] = qa * c.out(d1112) + (bx + bz);
  v[16] = qa * c.out(d1314) + (bx - bz);
  v[17] = qa * c.out(d1516) + (by + bz);
  v[18] = qa * c.out(d1718) + (by - bz);
  const int E = std::is_same<Sc, InDouble>::value ? -1 : top_exponent<1>(v);
  if (E >= 0)
    inverse_nonorth_l(v, InFixed<6>{E}, out);
  else
    inverse_nonorth_l(v, InDouble{}, out);
}

// ------------------------------------------------------------------ orthogonal operator
// d'Humieres et al. D3Q19 basis at the Eq. 2 ordering: m = M_o f, m_eq = M_o f_eq,
// S = M_o G (Guo), f* = M_o^T diag(1/|row|^2) m*.  The Eq. 16 term enters as
// dS4 * (0, 19, -16, 0, ...), its image in this basis.
// v: n_k = m_k* / |row k|^2 for k = 0, 1, 2, 9, 10, 11, a third of 12, 16, 17, 18, 13,
// 15, 14 (xy, xz, yz), then j*/10 and q*/40 of x, y, z.
template <typename Sc, typename Out>
__device__ __forceinline__ void inverse_orth_l(const double (&v)[19], const Sc &c, Out &&out) {
  using L = typename Sc::Value;
  const L n0 = c.in(v[0]), n1 = c.in(v[1]), n2 = c.in(v[2]);
  out(0, c.out_twice((c.half(n0) - times<15>(n1)) + times<6>(n2)));
  const L Ca = (n0 - times<11>(n1)) - times<4>(n2), Cd = (n0 + times<8>(n1)) + n2;
  const L n9 = c.in(v[3]), n10 = c.in(v[4]), n11 = c.in(v[5]), n12 = c.in(v[6]);
  // axis parts of the stresses: x gets 2 q9, y and z -q9 +- w11
  const L q9 = n9 - times<2>(n10), w11 = n11 - times<6>(n12), r9 = n9 + n10, r11 = n11 + times<3>(n12);
  const L gx = c.in(v[13]), gy = c.in(v[14]), gz = c.in(v[15]), hx = c.in(v[16]), hy = c.in(v[17]), hz = c.in(v[18]);
  auto pair = [&](int k, const L &even, const L &odd) {
    out(k, c.out(even + odd));
    out(k + 1, c.out(even - odd));
  };
  pair(1, Ca + times<2>(q9), gx - times<4>(hx));
  pair(3, (Ca - q9) + w11, gy - times<4>(hy));
  pair(5, (Ca - q9) - w11, gz - times<4>(hz));
  const L X = gx + hx, Y = gy + hy, Z = gz + hz, Cr = Cd + r9;
  const L n16 = c.in(v[7]), n17 = c.in(v[8]), n18 = c.in(v[9]);
  {  // xy diagonals 7..10: signs of (p_xy, m_x, m_y) are (+,+,-), (+,-,+), (-,+,+), (-,-,-)
    const L e = Cr + r11, s = c.in(v[10]);
    pair(7, e + s, (X + Y) + (n16 - n17));
    pair(9, e - s, (X - Y) + (n16 + n17));
  }
  {  // xz diagonals 11..14: signs of (p_xz, m_x, m_z) are (+,-,+), (+,+,-), (-,-,-), (-,+,+)
    const L e = Cr - r11, s = c.in(v[11]);
    pair(11, e + s, (X + Z) + (n18 - n16));
    pair(13, e - s, (X - Z) - (n16 + n18));
  }
  {  // yz diagonals 15..18: signs of (p_yz, m_y, m_z) are (+,+,-), (+,-,+), (-,+,+), (-,-,-)
    const L e = Cd - times<2>(r9), s = c.in(v[12]);
    pair(15, e + s, (Y + Z) + (n17 - n18));
    pair(17, e - s, (Y - Z) + (n17 + n18));
  }
}

template <typename Sc, typename Out>
__device__ __forceinline__ void collide_orth_l(const double (&f_)[19], const Sc &c, double rho_ref, double Fx,
                                               double Fy, double Fz, double S2, const KParams &P, const Coeffs64 &C,
                                               Out &&out) {
  using L = typename Sc::Value;
  L f[19];
#pragma unroll
  for (int a = 0; a < 19; ++a) f[a] = c.in(f_[a]);
  const L s12 = f[1] + f[2], d12 = f[1] - f[2];
  const L s34 = f[3] + f[4], d34 = f[3] - f[4];
  const L s56 = f[5] + f[6], d56 = f[5] - f[6];
  const L s78 = f[7] + f[8], d78 = f[7] - f[8];
  const L s910 = f[9] + f[10], d910 = f[9] - f[10];
  const L s1112 = f[11] + f[12], d1112 = f[11] - f[12];
  const L s1314 = f[13] + f[14], d1314 = f[13] - f[14];
  const L s1516 = f[15] + f[16], d1516 = f[15] - f[16];
  const L s1718 = f[17] + f[18], d1718 = f[17] - f[18];
  const L sxy = s78 + s910, sxz = s1112 + s1314, syz = s1516 + s1718;
  const L sp = s34 + s56, sm = s34 - s56, lA = s12 + sp, sxyz = sxy + sxz, lB = sxyz + syz;
  // diagonal parts of the momenta, plane by plane
  const L x1 = d78 + d910, y1 = d78 - d910, x2 = d1112 + d1314, z1 = d1112 - d1314, y2 = d1516 + d1718, z2 = d1516 - d1718;
  const L dx = x1 + x2, dy = y1 + y2, dz = z1 + z2;
  const double drho = c.out(f[0] + lA + lB), A = c.out(lA), B = c.out(lB);
  const double jx = c.out(d12 + dx), jy = c.out(d34 + dy), jz = c.out(d56 + dz);
  const Node64 N(rho_ref + drho, jx, jy, jz, Fx, Fy, Fz, S2);
  const double qp = N.qyy + N.qzz, usq = N.qxx + qp, Fp = N.Fuy + N.Fuz, Fu = N.Fux + Fp;
  double v[19];
  v[0] = (1.0 / 19.0) * drho;
  v[1] = C.k[kE1] * fma(2.0, B, A) + C.k[kE2] * drho + C.k[kE3] * usq + C.k[kE4] * Fu + C.k[kE5] * S2;
  v[2] = C.k[kO1] * A + C.k[kO2] * B + C.k[kO3] * drho + C.k[kO4] * usq + C.k[kO5] * Fu + C.k[kO6] * S2;
  const Shear64 n = shear64<19>(P, C, N.rho);
  const double Bx = n.b1 * N.rux + n.b2 * Fx, By = n.b1 * N.ruy + n.b2 * Fy, Bz = n.b1 * N.ruz + n.b2 * Fz;
  const double Gx = N.ux * Bx, Gy = N.uy * By, Gz = N.uz * Bz;
  const L a9 = sp - times<2>(s12), b9 = sxyz - times<2>(syz), b11 = sxy - sxz;
  v[3] = fma(-2.0 / 9.0, fma(-2.0, Gx, Gy + Gz), n.nx * c.out(b9 - a9));
  v[4] = C.k[kP1] * c.out(b9 + times<2>(a9)) + C.k[kP2] * fma(-2.0, N.qxx, qp) + C.k[kP3] * fma(-2.0, N.Fux, Fp);
  v[5] = n.n5 * c.out(sm + b11) + (2.0 / 3.0) * (Gy - Gz);
  v[6] = C.k[kP1] * c.out(b11 - times<2>(sm)) + C.k[kP2] * (N.qzz - N.qyy) + C.k[kP3] * (N.Fuz - N.Fuy);
  v[7] = C.k[kOm] * c.out(x1 - x2);
  v[8] = C.k[kOm] * c.out(y2 - y1);
  v[9] = C.k[kOm] * c.out(z1 - z2);
  v[10] = n.n7 * c.out(s78 - s910) + N.ux * By + N.uy * Bx;
  v[11] = n.n7 * c.out(s1112 - s1314) + N.ux * Bz + N.uz * Bx;
  v[12] = n.n7 * c.out(s1516 - s1718) + N.uy * Bz + N.uz * By;
  v[13] = 0.1 * (jx + Fx);
  v[14] = 0.1 * (jy + Fy);
  v[15] = 0.1 * (jz + Fz);
  v[16] = C.k[kQa] * c.out(dx - times<4>(d12)) - (C.k[kQb1] * N.rux + C.k[kQb2] * Fx);
  v[17] = C.k[kQa] * c.out(dy - times<4>(d34)) - (C.k[kQb1] * N.ruy + C.k[kQb2] * Fy);
  v[18] = C.k[kQa] * c.out(dz - times<4>(d56)) - (C.k[kQb1] * N.ruz + C.k[kQb2] * Fz);
  const int E = std::is_same<Sc, InDouble>::value ? -1 : top_exponent(v);
  if (E >= 0)
    inverse_orth_l(v, InFixed<5>{E}, out);
  else
    inverse_orth_l(v, InDouble{}, out);
}

// ------------------------------------------------------------------ D3Q15
// The basis and readings of lbm_q15.cuh; the four odd corner moments relax with one
// rate, so the corner differences relax themselves.  v: drho - m4*, m4* / 6, -m5* / 12,
// m6* / 4, m_k* / 8 (14, 7, 8, 9), twice the odd parts of the axes, the odd parts of
// the corner pairs.
template <typename Sc, typename Out>
__device__ __forceinline__ void inverse_q15_l(const double (&v)[15], const Sc &c, Out &&out) {
  using L = typename Sc::Value;
  const L e4 = c.in(v[1]), e5 = c.in(v[2]), e6 = c.in(v[3]), p14 = c.in(v[4]);
  out(0, fma(16.0, v[4], v[0]));
  auto axis = [&](int k, const L &even, double odd2) {
    const L e = times<2>(even), o = c.in(odd2);
    out(k, c.out_half(e + o));
    out(k + 1, c.out_half(e - o));
  };
  const L c4 = e4 - times<4>(p14), c45 = c4 + e5;
  axis(1, c4 - times<2>(e5), v[8]);
  axis(3, c45 + e6, v[9]);
  axis(5, c45 - e6, v[10]);
  const L p7 = c.in(v[5]), p8 = c.in(v[6]), p9 = c.in(v[7]);
  const L q1 = p14 + p7, q2 = p8 + p9, q3 = p14 - p7, q4 = p8 - p9;
  auto corner = [&](int k, const L &even, double odd) {
    const L o = c.in(odd);
    out(k, c.out(even + o));
    out(k + 1, c.out(even - o));
  };
  corner(7, q1 + q2, v[11]);
  corner(9, q1 - q2, v[12]);
  corner(11, q3 + q4, v[13]);
  corner(13, q3 - q4, v[14]);
}

template <typename Sc, typename Out>
__device__ __forceinline__ void collide_q15_l(const double (&f_)[15], const Sc &c, double rho_ref, double Fx,
                                              double Fy, double Fz, double S2, const KParams &P, const Coeffs64 &C,
                                              Out &&out) {
  using L = typename Sc::Value;
  L f[15];
#pragma unroll
  for (int a = 0; a < 15; ++a) f[a] = c.in(f_[a]);
  const L s12 = f[1] + f[2], d12 = f[1] - f[2];
  const L s34 = f[3] + f[4], d34 = f[3] - f[4];
  const L s56 = f[5] + f[6], d56 = f[5] - f[6];
  // corner pairs -> even (count, e_x e_y, e_x e_z, e_y e_z) moments by two butterfly stages; corner parts of e_x, ...
  const L s78 = f[7] + f[8], d78 = f[7] - f[8];
  const L s910 = f[9] + f[10], d910 = f[9] - f[10];
  const L s1112 = f[11] + f[12], d1112 = f[11] - f[12];
  const L s1314 = f[13] + f[14], d1314 = f[13] - f[14];
  const L u1 = s78 + s910, u2 = s1112 + s1314, v1 = s78 - s910, v2 = s1112 - s1314, l14 = u1 + u2;
  const L U1 = d78 + d910, U2 = d1112 - d1314;
  const L lx = U1 + U2, ly = U1 - U2, lz = (d78 - d910) + (d1112 + d1314);
  const L syz = s34 + s56, sax = s12 + syz;
  const double drho = c.out(f[0] + sax + l14);
  const double Dx = c.out(lx), Dy = c.out(ly), Dz = c.out(lz);
  const double jx = c.out(d12 + lx), jy = c.out(d34 + ly), jz = c.out(d56 + lz);
  const Node64 N(rho_ref + drho, jx, jy, jz, Fx, Fy, Fz, S2);
  const double usq = N.qxx + N.qyy + N.qzz, Fu = N.Fux + N.Fuy + N.Fuz;
  double v[15];
  const double m4 = relax4(c.out(sax + times<3>(l14)), drho, usq, Fu, S2, C);
  v[0] = drho - m4;
  v[1] = (1.0 / 6.0) * m4;
  const double p14 = c.template out_over<3>(l14);
  v[4] = fma(C.k[kP1], fma(1.0 / 72.0, drho, -p14) + fma(C.k[kP4], Fu, (1.0 / 144.0) * usq), p14);
  const Shear64 n = shear64<15>(P, C, N.rho);
  const double Bx = n.b1 * N.rux + n.b2 * Fx, By = n.b1 * N.ruy + n.b2 * Fy, Bz = n.b1 * N.ruz + n.b2 * Fz;
  const double Gx = N.ux * Bx, Gy = N.uy * By, Gz = N.uz * Bz;
  v[2] = fma(4.0 / 3.0, fma(-2.0, Gx, Gy + Gz), n.n5 * c.out(syz - times<2>(s12)));
  v[3] = fma(4.0, Gy - Gz, n.n7 * c.out(s34 - s56));
  v[5] = n.nx * c.out(u1 - u2) + N.ux * By + N.uy * Bx;
  v[6] = n.nx * c.out(v1 + v2) + N.ux * Bz + N.uz * Bx;
  v[7] = n.nx * c.out(v1 - v2) + N.uy * Bz + N.uz * By;
  const double bx = C.k[kQb1] * N.rux + C.k[kQb2] * Fx, by = C.k[kQb1] * N.ruy + C.k[kQb2] * Fy;
  const double bz = C.k[kQb1] * N.ruz + C.k[kQb2] * Fz, qa = C.k[kQa], q2 = -C.k[kQ2], bp = bx + by, bm = bx - by;
  v[8] = fma(-8.0, bx, fma(q2, Dx, jx + Fx));
  v[9] = fma(-8.0, by, fma(q2, Dy, jy + Fy));
  v[10] = fma(-8.0, bz, fma(q2, Dz, jz + Fz));
  v[11] = qa * c.out(d78) + (bp + bz);
  v[12] = qa * c.out(d910) + (bp - bz);
  v[13] = qa * c.out(d1112) + (bm + bz);
  v[14] = qa * c.out(d1314) - (bm - bz);
  const int E = std::is_same<Sc, InDouble>::value ? -1 : top_exponent<1>(v);
  if (E >= 0)
    inverse_q15_l(v, InFixed<6>{E}, out);
  else
    inverse_q15_l(v, InDouble{}, out);
}

// Collision of a node of operator OP: linear parts in fixed point where the populations allow it.
template <int OP, int N, typename Out>
__device__ __forceinline__ void collide64(const double (&f)[N], double rho_ref, double Fx, double Fy, double Fz, double S2,
                                          const KParams &P, const Coeffs64 &C, Out &&out) {
  auto run = [&](const auto &scale) {
    if constexpr (N == 15)
      collide_q15_l(f, scale, rho_ref, Fx, Fy, Fz, S2, P, C, out);
    else if constexpr (OP == kNonOrth)
      collide_nonorth_l(f, scale, rho_ref, Fx, Fy, Fz, S2, P, C, out);
    else
      collide_orth_l(f, scale, rho_ref, Fx, Fy, Fz, S2, P, C, out);
  };
  const int E = top_exponent(f);
  if (E >= 0)
    run(InFixed<5>{E});  // factors up to 32
  else
    run(InDouble{});
}

}  // namespace lbm
