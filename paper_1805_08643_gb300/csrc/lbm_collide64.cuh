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
//    the host (coeffs64);
//  - rho u_i u_j and F_i u_j + F_j u_i relax with the same rate, so s rho u_i u_j
//    + c (F_i u_j + F_j u_i) = u_i B_j + u_j B_i, B_i = s rho u_i / 2 + c F_i;
//  - the third-order moments of a pair of diagonals (corners) relax with one
//    rate: the differences d78, d910, ... relax themselves, no moments are formed;
//  - 2 x + y is written fma(2, x, y) (2 * x + y compiles to two additions), and
//    the reciprocal takes three instructions (recip).
// FP64 instructions per node of the fused pass, with the force: 214
// non-orthogonal (255 moment by moment), 259 orthogonal; at 128^3 the pass takes
// 852 us (1014) and 1027 us (1235), D3Q15 725 us (808), 0.84 of the unit's rate.
#pragma once

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

// The sums of Eq. 15 in units of the diagonal (D3Q15: corner) weight, where
// the axes weigh 2 (8).  p[a] = psi(x + e_a).
template <int Q>
__device__ __forceinline__ void psi_sums64(const double p[Q], double &Sx, double &Sy, double &Sz) {
  constexpr double axw = Q == 19 ? 2.0 : 8.0;
  const double d78 = p[7] - p[8], d910 = p[9] - p[10], d1112 = p[11] - p[12], d1314 = p[13] - p[14];
  if constexpr (Q == 19) {
    const double d1516 = p[15] - p[16], d1718 = p[17] - p[18];
    Sx = fma(axw, p[1] - p[2], (d78 + d910) + (d1112 + d1314));
    Sy = fma(axw, p[3] - p[4], (d78 - d910) + (d1516 + d1718));
    Sz = fma(axw, p[5] - p[6], (d1112 - d1314) + (d1516 - d1718));
  } else {
    const double ab = d78 + d910, cd = d1112 - d1314;
    Sx = fma(axw, p[1] - p[2], ab + cd);
    Sy = fma(axw, p[3] - p[4], ab - cd);
    Sz = fma(axw, p[5] - p[6], (d78 - d910) + (d1112 + d1314));
  }
}

// Non-orthogonal operator: forward chains of Eq. 12, equilibria Eq. 13,
// forcing Eq. 14, the Eq. 16 term from S2 (the squared sum of Eq. 15), inverse
// chains of App. A.  f holds the deviations f_a - w_a rho_ref; out(a, f*_a)
// takes the results (deviations again).
template <typename Out>
__device__ __forceinline__ void collide_nonorth64(const double f[19], double rho_ref, double Fx, double Fy, double Fz,
                                                  double S2, const KParams &P, const Coeffs64 &C, Out &&out) {
  // opposite-pair sums and differences
  const double s12 = f[1] + f[2], d12 = f[1] - f[2];
  const double s34 = f[3] + f[4], d34 = f[3] - f[4];
  const double s56 = f[5] + f[6], d56 = f[5] - f[6];
  const double s78 = f[7] + f[8], d78 = f[7] - f[8];
  const double s910 = f[9] + f[10], d910 = f[9] - f[10];
  const double s1112 = f[11] + f[12], d1112 = f[11] - f[12];
  const double s1314 = f[13] + f[14], d1314 = f[13] - f[14];
  const double s1516 = f[15] + f[16], d1516 = f[15] - f[16];
  const double s1718 = f[17] + f[18], d1718 = f[17] - f[18];
  // m = M f (Eq. 12), in deviation form (m - rho_ref M w)
  const double m16 = s78 + s910, m17 = s1112 + s1314, m18 = s1516 + s1718;
  const double m7 = s78 - s910, m8 = s1112 - s1314, m9 = s1516 - s1718;
  const double Dx = (d78 + d910) + (d1112 + d1314);  // m11 + m13
  const double Dy = (d78 - d910) + (d1516 + d1718);  // m10 + m15
  const double Dz = (d1112 - d1314) + (d1516 - d1718);  // m12 + m14
  const double syz = s34 + s56, sax = s12 + syz;
  const double sxx = m16 + m17, sdg = sxx + m18;
  const double drho = f[0] + sax + sdg;
  const double m4 = fma(2.0, sdg, sax);
  const double m5 = fma(2.0, s12 - m18, sxx - syz);
  const double m6 = (s34 - s56) + (m16 - m17);
  // macroscopic quantities, Eq. 6
  const double rho = rho_ref + drho;
  const double inv_rho = recip(rho);
  const double rux = (d12 + Dx) + 0.5 * Fx, ruy = (d34 + Dy) + 0.5 * Fy, ruz = (d56 + Dz) + 0.5 * Fz;
  const double ox = d12 + C.k[kQs] * Dx, oy = d34 + C.k[kQs] * Dy, oz = d56 + C.k[kQs] * Dz;
  const double ux = rux * inv_rho, uy = ruy * inv_rho, uz = ruz * inv_rho;
  const double qxx = rux * ux, qyy = ruy * uy, qzz = ruz * uz;  // rho u_i^2
  const double usq = qxx + qyy + qzz;
  const double Fux = Fx * ux, Fuy = Fy * uy, Fuz = Fz * uz;
  const double Fu = Fux + Fuy + Fuz;
  // relaxed moments (Eq. 4 with Eqs. 11, 13, 14, 16), scaled: e4 = m4* / 6, e5 = m5* / 12, e6 = m6* / 4,
  // p_k = m_k* / 4
  const double e4 = C.k[kE1] * m4 + C.k[kE2] * (drho + usq) + C.k[kE4] * Fu + C.k[kE5] * S2;
  // Eq. 13's phi + (rho - rho_ref)/9 and third-axis parts: m16 takes the sum over the axes less the z part, ...
  const double c4 = C.k[kP2] * drho + C.k[kP3] * usq + C.k[kP4] * Fu;
  const double p16 = C.k[kP1] * m16 + (c4 - (C.k[kP5] * qzz + C.k[kP4] * Fuz));
  const double p17 = C.k[kP1] * m17 + (c4 - (C.k[kP5] * qyy + C.k[kP4] * Fuy));
  const double p18 = C.k[kP1] * m18 + (c4 - (C.k[kP5] * qxx + C.k[kP4] * Fux));
  out(0, (drho - 6.0 * e4) + 4.0 * ((p16 + p17) + p18));
  const Shear64 n = shear64<19>(P, C, rho);
  const double Bx = n.b1 * rux + n.b2 * Fx, By = n.b1 * ruy + n.b2 * Fy, Bz = n.b1 * ruz + n.b2 * Fz;
  const double Gx = ux * Bx, Gy = uy * By, Gz = uz * Bz;
  const double e5 = fma(-2.0 / 3.0, fma(-2.0, Gx, Gy + Gz), n.n5 * m5);
  const double e6 = fma(2.0, Gy - Gz, n.n7 * m6);
  // f* = M^-1 m* (App. A); odd parts: b_i carries Eq. 13/14's rho u_i / 3 and F_i / 3 of the third-order moments
  const double bx = C.k[kQb1] * rux + C.k[kQb2] * Fx, by = C.k[kQb1] * ruy + C.k[kQb2] * Fy;
  const double bz = C.k[kQb1] * ruz + C.k[kQb2] * Fz;
  const double h = 0.5;
  const double e45 = e4 - e5;
  {
    const double even = fma(-2.0, p16 + p17, fma(2.0, e5, e4)), odd = (ox + Fx) - 8.0 * bx;
    out(1, even + h * odd);
    out(2, even - h * odd);
  }
  {
    const double even = fma(-2.0, p16 + p18, e45 + e6), odd = (oy + Fy) - 8.0 * by;
    out(3, even + h * odd);
    out(4, even - h * odd);
  }
  {
    const double even = fma(-2.0, p17 + p18, e45 - e6), odd = (oz + Fz) - 8.0 * bz;
    out(5, even + h * odd);
    out(6, even - h * odd);
  }
  {
    const double p7 = n.n7 * m7 + ux * By + uy * Bx;
    const double ev = p16 + p7, od = C.k[kQa] * d78 + (bx + by), ew = p16 - p7, oe = C.k[kQa] * d910 + (bx - by);
    out(7, ev + od);
    out(8, ev - od);
    out(9, ew + oe);
    out(10, ew - oe);
  }
  {
    const double p8 = n.n7 * m8 + ux * Bz + uz * Bx;
    const double ev = p17 + p8, od = C.k[kQa] * d1112 + (bx + bz), ew = p17 - p8, oe = C.k[kQa] * d1314 + (bx - bz);
    out(11, ev + od);
    out(12, ev - od);
    out(13, ew + oe);
    out(14, ew - oe);
  }
  {
    const double p9 = n.n7 * m9 + uy * Bz + uz * By;
    const double ev = p18 + p9, od = C.k[kQa] * d1516 + (by + bz), ew = p18 - p9, oe = C.k[kQa] * d1718 + (by - bz);
    out(15, ev + od);
    out(16, ev - od);
    out(17, ew + oe);
    out(18, ew - oe);
  }
}

// Orthogonal operator (d'Humieres et al. D3Q19 basis at the Eq. 2 ordering):
// m = M_o f, m_eq = M_o f_eq, S = M_o G (Guo), f* = M_o^T diag(1/|row|^2) m*.
// The Eq. 16 term enters as dS4 * (0, 19, -16, 0, ...), its image in this basis.
template <typename Out>
__device__ __forceinline__ void collide_orth64(const double f[19], double rho_ref, double Fx, double Fy, double Fz,
                                                  double S2, const KParams &P, const Coeffs64 &C, Out &&out) {
  const double s12 = f[1] + f[2], d12 = f[1] - f[2];
  const double s34 = f[3] + f[4], d34 = f[3] - f[4];
  const double s56 = f[5] + f[6], d56 = f[5] - f[6];
  const double s78 = f[7] + f[8], d78 = f[7] - f[8];
  const double s910 = f[9] + f[10], d910 = f[9] - f[10];
  const double s1112 = f[11] + f[12], d1112 = f[11] - f[12];
  const double s1314 = f[13] + f[14], d1314 = f[13] - f[14];
  const double s1516 = f[15] + f[16], d1516 = f[15] - f[16];
  const double s1718 = f[17] + f[18], d1718 = f[17] - f[18];
  const double sxy = s78 + s910, sxz = s1112 + s1314, syz = s1516 + s1718;
  const double sp = s34 + s56, sm = s34 - s56;
  const double A = s12 + sp, sxyz = sxy + sxz, B = sxyz + syz;
  const double drho = f[0] + A + B;
  // diagonal parts of the momenta, plane by plane
  const double x1 = d78 + d910, y1 = d78 - d910;
  const double x2 = d1112 + d1314, z1 = d1112 - d1314;
  const double y2 = d1516 + d1718, z2 = d1516 - d1718;
  const double dx = x1 + x2, dy = y1 + y2, dz = z1 + z2;
  const double jx = d12 + dx, jy = d34 + dy, jz = d56 + dz;
  // macroscopic quantities, Eq. 6
  const double rho = rho_ref + drho;
  const double inv_rho = recip(rho);
  const double rux = jx + 0.5 * Fx, ruy = jy + 0.5 * Fy, ruz = jz + 0.5 * Fz;
  const double ux = rux * inv_rho, uy = ruy * inv_rho, uz = ruz * inv_rho;
  const double qxx = rux * ux, qyy = ruy * uy, qzz = ruz * uz;
  const double qp = qyy + qzz, usq = qxx + qp;
  const double Fux = Fx * ux, Fuy = Fy * uy, Fuz = Fz * uz;
  const double Fp = Fuy + Fuz, Fu = Fux + Fp;
  // relaxed moments over the squared row norms: n_k = m_k* / |row k|^2 (the numbers are the rows')
  const double n0 = 1.0 / 19.0 * drho;
  const double n1 = C.k[kE1] * fma(2.0, B, A) + C.k[kE2] * drho + C.k[kE3] * usq + C.k[kE4] * Fu + C.k[kE5] * S2;
  const double n2 = C.k[kO1] * A + C.k[kO2] * B + C.k[kO3] * drho + C.k[kO4] * usq + C.k[kO5] * Fu + C.k[kO6] * S2;
  out(0, (n0 - 30.0 * n1) + 12.0 * n2);
  const double Ca = (n0 - 11.0 * n1) - 4.0 * n2;
  const double Cd = (n0 + 8.0 * n1) + n2;
  const Shear64 n = shear64<19>(P, C, rho);
  const double Bx = n.b1 * rux + n.b2 * Fx, By = n.b1 * ruy + n.b2 * Fy, Bz = n.b1 * ruz + n.b2 * Fz;
  const double Gx = ux * Bx, Gy = uy * By, Gz = uz * Bz;
  const double a9 = fma(-2.0, s12, sp), b9 = fma(-2.0, syz, sxyz), b11 = sxy - sxz;
  const double n9 = fma(-2.0 / 9.0, fma(-2.0, Gx, Gy + Gz), n.nx * (b9 - a9));
  const double n11 = n.n5 * (sm + b11) + 2.0 / 3.0 * (Gy - Gz);
  const double n10 = C.k[kP1] * fma(2.0, a9, b9) + C.k[kP2] * fma(-2.0, qxx, qp) + C.k[kP3] * fma(-2.0, Fux, Fp);
  const double n12 = C.k[kP1] * fma(-2.0, sm, b11) + C.k[kP2] * (qzz - qyy) + C.k[kP3] * (Fuz - Fuy);  // a third of it
  const double q9 = fma(-2.0, n10, n9), w11 = n11 - 6.0 * n12;  // axis parts of the stresses: x gets 2 q9, y and z -q9 +- w11
  const double r9 = n9 + n10, r11 = n11 + 3.0 * n12;
  const double n16 = C.k[kOm] * (x1 - x2), n17 = C.k[kOm] * (y2 - y1), n18 = C.k[kOm] * (z1 - z2);
  // odd parts of an axis: j* / 10 and q* / 40; xo, yo, zo on the axis, X, Y, Z on the diagonals
  const double gx = 0.1 * (jx + Fx), gy = 0.1 * (jy + Fy), gz = 0.1 * (jz + Fz);
  const double hx = C.k[kQa] * (dx - 4.0 * d12) - (C.k[kQb1] * rux + C.k[kQb2] * Fx);
  const double hy = C.k[kQa] * (dy - 4.0 * d34) - (C.k[kQb1] * ruy + C.k[kQb2] * Fy);
  const double hz = C.k[kQa] * (dz - 4.0 * d56) - (C.k[kQb1] * ruz + C.k[kQb2] * Fz);
  const double xo = gx - 4.0 * hx, yo = gy - 4.0 * hy, zo = gz - 4.0 * hz;
  const double X = gx + hx, Y = gy + hy, Z = gz + hz;
  {
    const double cx = fma(2.0, q9, Ca), cy = (Ca - q9) + w11, cz = (Ca - q9) - w11;
    out(1, cx + xo);
    out(2, cx - xo);
    out(3, cy + yo);
    out(4, cy - yo);
    out(5, cz + zo);
    out(6, cz - zo);
  }
  const double Cr = Cd + r9;
  // xy diagonals 7..10: signs of (p_xy, m_x, m_y) are (+,+,-), (+,-,+), (-,+,+), (-,-,-)
  {
    const double E = Cr + r11, n13 = n.n7 * (s78 - s910) + ux * By + uy * Bx;
    const double ev = E + n13, od = (X + Y) + (n16 - n17), ew = E - n13, oe = (X - Y) + (n16 + n17);
    out(7, ev + od);
    out(8, ev - od);
    out(9, ew + oe);
    out(10, ew - oe);
  }
  // xz diagonals 11..14: signs of (p_xz, m_x, m_z) are (+,-,+), (+,+,-), (-,-,-), (-,+,+)
  {
    const double E = Cr - r11, n15 = n.n7 * (s1112 - s1314) + ux * Bz + uz * Bx;
    const double ev = E + n15, od = (X + Z) + (n18 - n16), ew = E - n15, oe = (X - Z) - (n16 + n18);
    out(11, ev + od);
    out(12, ev - od);
    out(13, ew + oe);
    out(14, ew - oe);
  }
  // yz diagonals 15..18: signs of (p_yz, m_y, m_z) are (+,+,-), (+,-,+), (-,+,+), (-,-,-)
  {
    const double E = fma(-2.0, r9, Cd), n14 = n.n7 * (s1516 - s1718) + uy * Bz + uz * By;
    const double ev = E + n14, od = (Y + Z) + (n17 - n18), ew = E - n14, oe = (Y - Z) + (n17 + n18);
    out(15, ev + od);
    out(16, ev - od);
    out(17, ew + oe);
    out(18, ew - oe);
  }
}

// D3Q15 (the basis and readings of lbm_q15.cuh); the four odd corner moments
// relax with one rate, so the corner differences relax themselves.
template <typename Out>
__device__ __forceinline__ void collide_q15_64(const double f[15], double rho_ref, double Fx, double Fy, double Fz,
                                                  double S2, const KParams &P, const Coeffs64 &C, Out &&out) {
  // axis pairs
  const double s12 = f[1] + f[2], d12 = f[1] - f[2];
  const double s34 = f[3] + f[4], d34 = f[3] - f[4];
  const double s56 = f[5] + f[6], d56 = f[5] - f[6];
  // corner pairs -> even (count, e_x e_y, e_x e_z, e_y e_z) moments by two
  // butterfly stages; corner parts of e_x, e_y, e_z
  const double s78 = f[7] + f[8], d78 = f[7] - f[8];
  const double s910 = f[9] + f[10], d910 = f[9] - f[10];
  const double s1112 = f[11] + f[12], d1112 = f[11] - f[12];
  const double s1314 = f[13] + f[14], d1314 = f[13] - f[14];
  const double u1 = s78 + s910, u2 = s1112 + s1314, v1 = s78 - s910, v2 = s1112 - s1314;
  const double m14 = u1 + u2, m7 = u1 - u2, m8 = v1 + v2, m9 = v1 - v2;
  const double U1 = d78 + d910, U2 = d1112 - d1314;
  const double Dx = U1 + U2, Dy = U1 - U2, Dz = (d78 - d910) + (d1112 + d1314);
  const double syz = s34 + s56, sax = s12 + syz;
  const double drho = f[0] + sax + m14;
  const double m4 = sax + 3.0 * m14;
  const double m5 = fma(-2.0, s12, syz);  // negated, and e5 below
  const double m6 = s34 - s56;
  // macroscopic quantities, Eq. 6
  const double rho = rho_ref + drho;
  const double inv_rho = recip(rho);
  const double rux = (d12 + Dx) + 0.5 * Fx, ruy = (d34 + Dy) + 0.5 * Fy, ruz = (d56 + Dz) + 0.5 * Fz;
  const double ux = rux * inv_rho, uy = ruy * inv_rho, uz = ruz * inv_rho;
  const double usq = rux * ux + ruy * uy + ruz * uz;  // rho |u|^2
  const double Fu = Fx * ux + Fy * uy + Fz * uz;
  // relaxed moments, scaled: e4 = m4* / 6, e5 = -m5* / 12, e6 = m6* / 4, p_k = m_k* / 8
  const double e4 = C.k[kE1] * m4 + C.k[kE2] * (drho + usq) + C.k[kE4] * Fu + C.k[kE5] * S2;
  const double p14 = C.k[kP1] * m14 + C.k[kP2] * drho + C.k[kP3] * usq + C.k[kP4] * Fu;
  out(0, (drho - 6.0 * e4) + 16.0 * p14);
  const Shear64 n = shear64<15>(P, C, rho);
  const double Bx = n.b1 * rux + n.b2 * Fx, By = n.b1 * ruy + n.b2 * Fy, Bz = n.b1 * ruz + n.b2 * Fz;
  const double Gx = ux * Bx, Gy = uy * By, Gz = uz * Bz;
  const double e5 = fma(4.0 / 3.0, fma(-2.0, Gx, Gy + Gz), n.n5 * m5);
  const double e6 = n.n7 * m6 + 4.0 * (Gy - Gz);
  const double p7 = n.nx * m7 + ux * By + uy * Bx;
  const double p8 = n.nx * m8 + ux * Bz + uz * Bx;
  const double p9 = n.nx * m9 + uy * Bz + uz * By;
  // f* = M^-1 m*
  const double bx = C.k[kQb1] * rux + C.k[kQb2] * Fx, by = C.k[kQb1] * ruy + C.k[kQb2] * Fy;
  const double bz = C.k[kQb1] * ruz + C.k[kQb2] * Fz;
  const double h = 0.5;
  const double c4 = e4 - 4.0 * p14, c45 = c4 + e5;
  {
    const double even = fma(-2.0, e5, c4), odd = ((d12 + Fx) + C.k[kQs] * Dx) - 8.0 * bx;
    out(1, even + h * odd);
    out(2, even - h * odd);
  }
  {
    const double even = c45 + e6, odd = ((d34 + Fy) + C.k[kQs] * Dy) - 8.0 * by;
    out(3, even + h * odd);
    out(4, even - h * odd);
  }
  {
    const double even = c45 - e6, odd = ((d56 + Fz) + C.k[kQs] * Dz) - 8.0 * bz;
    out(5, even + h * odd);
    out(6, even - h * odd);
  }
  const double q1 = p14 + p7, q2 = p8 + p9, q3 = p14 - p7, q4 = p8 - p9;
  const double bp = bx + by, bm = bx - by;
  {
    const double ev = q1 + q2, od = C.k[kQa] * d78 + (bp + bz), ew = q1 - q2, oe = C.k[kQa] * d910 + (bp - bz);
    out(7, ev + od);
    out(8, ev - od);
    out(9, ew + oe);
    out(10, ew - oe);
  }
  {
    const double ev = q3 + q4, od = C.k[kQa] * d1112 + (bm + bz), ew = q3 - q4, oe = C.k[kQa] * d1314 - (bm - bz);
    out(11, ev + od);
    out(12, ev - od);
    out(13, ew + oe);
    out(14, ew - oe);
  }
}

}  // namespace lbm
