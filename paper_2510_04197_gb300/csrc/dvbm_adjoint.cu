// dvbm_adjoint.cu -- hand-written discrete adjoint of the FP64 time step.
//
// For the map X^{n+1} = Phi(X^n; mu, Pr, gamma) of Eq. finalDiscretePDE (FP64
// storage, periodic domain) the kernels compute lambda^n = (dPhi/dX^n)^T
// lambda^{n+1} and the per-cell contributions to dL/d(mu, Pr, gamma):
//
//  * local (collision) part: with a1 = 1 - dt/tau1 and the combined Grad
//    coefficients C (dvbm_device.cuh), X^{n+1}_k = a1 X_k + W_k sum C H_k - adv_k,
//      lambda^n_i = a1 lambda_i + sum_j mbar_j dm_j/dX_i,
//    where (abar1, Cbar) = (sum_k lambda_k X_k, sum_k lambda_k W_k H_k) are
//    pulled back through the coefficient function by the reverse pass
//    collision_coeffs_rev (the forward statements in reverse order), giving
//    the moment adjoints mbar and the parameter adjoints;
//  * advection part, written as a gather: the flux difference of cell c',
//    F(c') = D_c' + sigma_c' - sigma_{c'-1} (v > 0) or
//    D_{c'+1} - sigma_{c'+1} + sigma_c' (v < 0), with D_k = X_k - X_{k-1} and
//    sigma_k = minmod3(hb D_k, (D_k + D_{k+1})/4, hb D_{k+1}); its adjoint
//    needs X and lambda at c-2 .. c+2 only.  The minmod branch of each slope
//    gives the partial derivatives (hb, 0), (1/4, 1/4), (0, hb) or (0, 0).
//    As in the forward kernel the linear combinations run in block floating
//    point on the integer pipe.
#include <algorithm>

#include "dvbm_device.cuh"
#include "dvbm_cellmom.cuh"
#include "dvbm_internal.h"

namespace dvbm {

// ---------------------------------------------------------------- reverse pass
struct ParamBar { double dt_mu, Pr, gm1, epsf; };

// Reverse of collision_coeffs<PRC> for the outputs C (f, g) and a1.
template <int PRC>
__device__ __forceinline__ double collision_coeffs_rev(const Moments& m, const Phys& P, const Coeffs& Cb,
                                                       double a1b, Moments& mb, ParamBar& pb) {
  // ---- forward recomputation of the intermediates
  const double rho = m.m00;
  const double irho = 1.0 / rho;
  const double ux = m.m10 * irho, uy = m.m01 * irho;
  const double Et = fma(0.5, m.m20 + m.m02, m.g00 * P.inv_c2);
  const double q = fma(ux, ux, uy * uy);
  const double w = fma(-0.5, q, Et * irho);
  const double theta = P.gm1 * w;
  const double s = theta - 1.0;
  const double p = rho * P.c2 * theta;
  double k1, k2;
  if (PRC <= 0) { k1 = P.dt_mu * p; k2 = k1 * P.Pr; }
  else          { k2 = P.dt_mu * p; k1 = k2 * P.Pr; }
  const double s1 = k1 - k2;
  const EqF e = eq_f(rho, ux, uy, s);
  const double reps = rho * P.epsf * theta;
  double Dxx = 0, Dxy = 0, Dyy = 0, kap = 0, Px = 0, Py = 0, Tx = 0;
  double d20 = 0, d11 = 0, d02 = 0, d30 = 0, d21 = 0, d12 = 0, d03 = 0, d40 = 0, d31 = 0, d13 = 0, d04 = 0;
  double dg10 = 0, dg01 = 0;
  if (PRC != 0) {
    Dxx = (m.m20 - rho) - e.a20;
    Dxy = m.m11 - e.a11;
    Dyy = (m.m02 - rho) - e.a02;
    if (PRC < 0) {
      kap = 0.25 * (Dxx + Dyy);
      Px = Dxx - kap; Py = Dyy - kap;
      d30 = (fma(-3.0, m.m10, m.m30) - e.a30) - 3.0 * ux * Px;
      d21 = ((m.m21 - m.m01) - e.a21) - fma(2.0 * ux, Dxy, uy * Px);
      d12 = ((m.m12 - m.m10) - e.a12) - fma(2.0 * uy, Dxy, ux * Py);
      d03 = (fma(-3.0, m.m01, m.m03) - e.a03) - 3.0 * uy * Py;
      dg10 = m.g10 * P.inv_c2 - reps * ux;
      dg01 = m.g01 * P.inv_c2 - reps * uy;
    } else {
      Tx = 0.5 * (Dxx - Dyy);
      d20 = Tx; d11 = Dxy; d02 = -Tx;
      d30 = 3.0 * ux * Tx;
      d21 = fma(uy, Tx, 2.0 * ux * Dxy);
      d12 = fma(-ux, Tx, 2.0 * uy * Dxy);
      d03 = -3.0 * uy * Tx;
      d40 = -6.0 * Tx; d31 = -3.0 * Dxy; d13 = -3.0 * Dxy; d04 = 6.0 * Tx;
    }
  }
  const double kg = k1 * P.c2, sg = s1 * P.c2;
  const double KR = kg * reps;

  // ---- reverse
  double uxb = 0, uyb = 0, sb = 0, rhob = 0, thetab = 0, k1b = 0, k2b = 0, s1b = 0, repsb = 0;
  // g outputs
  double KRb = Cb.g00 + Cb.g10 * ux + Cb.g01 * uy + Cb.g20 * fma(ux, ux, s) + Cb.g11 * ux * uy + Cb.g02 * fma(uy, uy, s);
  double sgb = Cb.g10 * dg10 + Cb.g01 * dg01;
  const double dg10b = Cb.g10 * sg, dg01b = Cb.g01 * sg;
  uxb += KR * (Cb.g10 + 2.0 * ux * Cb.g20 + uy * Cb.g11);
  uyb += KR * (Cb.g01 + 2.0 * uy * Cb.g02 + ux * Cb.g11);
  sb += KR * (Cb.g20 + Cb.g02);
  const double kgb = KRb * reps;
  repsb += KRb * kg;
  k1b += kgb * P.c2;
  s1b += sgb * P.c2;
  // f outputs: C.fab = k1 a_ab + s1 d_ab
  double a00b = Cb.f00 * k1, a10b = Cb.f10 * k1, a01b = Cb.f01 * k1, a20b = Cb.f20 * k1, a11b = Cb.f11 * k1,
         a02b = Cb.f02 * k1, a30b = Cb.f30 * k1, a21b = Cb.f21 * k1, a12b = Cb.f12 * k1, a03b = Cb.f03 * k1,
         a40b = Cb.f40 * k1, a31b = Cb.f31 * k1, a22b = Cb.f22 * k1, a13b = Cb.f13 * k1, a04b = Cb.f04 * k1;
  k1b += Cb.f00 * e.a00 + Cb.f10 * e.a10 + Cb.f01 * e.a01 + Cb.f20 * e.a20 + Cb.f11 * e.a11 + Cb.f02 * e.a02 +
         Cb.f30 * e.a30 + Cb.f21 * e.a21 + Cb.f12 * e.a12 + Cb.f03 * e.a03 + Cb.f40 * e.a40 + Cb.f31 * e.a31 +
         Cb.f22 * e.a22 + Cb.f13 * e.a13 + Cb.f04 * e.a04;
  s1b += Cb.f20 * d20 + Cb.f11 * d11 + Cb.f02 * d02 + Cb.f30 * d30 + Cb.f21 * d21 + Cb.f12 * d12 + Cb.f03 * d03 +
         Cb.f40 * d40 + Cb.f31 * d31 + Cb.f13 * d13 + Cb.f04 * d04;
  const double d20b = Cb.f20 * s1, d11b = Cb.f11 * s1, d02b = Cb.f02 * s1, d30b = Cb.f30 * s1, d21b = Cb.f21 * s1,
               d12b = Cb.f12 * s1, d03b = Cb.f03 * s1, d40b = Cb.f40 * s1, d31b = Cb.f31 * s1, d13b = Cb.f13 * s1,
               d04b = Cb.f04 * s1;
  if (PRC != 0) {
    double Dxxb = 0, Dxyb = 0, Dyyb = 0;
    if (PRC < 0) {
      // dg10 = g10 inv_c2 - reps ux ; dg01 = g01 inv_c2 - reps uy
      mb.g10 += dg10b * P.inv_c2;
      mb.g01 += dg01b * P.inv_c2;
      repsb -= dg10b * ux + dg01b * uy;
      uxb -= dg10b * reps;
      uyb -= dg01b * reps;
      double Pxb = 0, Pyb = 0;
      // d03 = m03 - 3 m01 - a03 - 3 uy Py
      mb.m03 += d03b; mb.m01 -= 3.0 * d03b; a03b -= d03b; uyb -= 3.0 * d03b * Py; Pyb -= 3.0 * d03b * uy;
      // d12 = m12 - m10 - a12 - 2 uy Dxy - ux Py
      mb.m12 += d12b; mb.m10 -= d12b; a12b -= d12b; uyb -= 2.0 * d12b * Dxy; Dxyb -= 2.0 * d12b * uy;
      uxb -= d12b * Py; Pyb -= d12b * ux;
      // d21 = m21 - m01 - a21 - 2 ux Dxy - uy Px
      mb.m21 += d21b; mb.m01 -= d21b; a21b -= d21b; uxb -= 2.0 * d21b * Dxy; Dxyb -= 2.0 * d21b * ux;
      uyb -= d21b * Px; Pxb -= d21b * uy;
      // d30 = m30 - 3 m10 - a30 - 3 ux Px
      mb.m30 += d30b; mb.m10 -= 3.0 * d30b; a30b -= d30b; uxb -= 3.0 * d30b * Px; Pxb -= 3.0 * d30b * ux;
      // Px = Dxx - kap, Py = Dyy - kap, kap = (Dxx + Dyy)/4
      const double kapb = -(Pxb + Pyb);
      Dxxb += Pxb + 0.25 * kapb;
      Dyyb += Pyb + 0.25 * kapb;
    } else {
      const double Txb = d20b - d02b + 3.0 * ux * d30b + uy * d21b - ux * d12b - 3.0 * uy * d03b - 6.0 * d40b + 6.0 * d04b;
      Dxyb += d11b + 2.0 * ux * d21b + 2.0 * uy * d12b - 3.0 * d31b - 3.0 * d13b;
      uxb += 3.0 * Tx * d30b + 2.0 * Dxy * d21b - Tx * d12b;
      uyb += Tx * d21b + 2.0 * Dxy * d12b - 3.0 * Tx * d03b;
      Dxxb += 0.5 * Txb;
      Dyyb -= 0.5 * Txb;
    }
    // Dxx = m20 - rho - a20 ; Dxy = m11 - a11 ; Dyy = m02 - rho - a02
    mb.m20 += Dxxb; rhob -= Dxxb; a20b -= Dxxb;
    mb.m11 += Dxyb; a11b -= Dxyb;
    mb.m02 += Dyyb; rhob -= Dyyb; a02b -= Dyyb;
  }
  // reps = rho epsf theta
  rhob += repsb * P.epsf * theta;
  pb.epsf += repsb * rho * theta;
  thetab += repsb * rho * P.epsf;
  // eq_f reverse (statements in reverse order)
  double rsb = 0;
  a20b += a22b * fma(uy, uy, s); uyb += a22b * e.a20 * 2.0 * uy; sb += a22b * e.a20;
  a03b += a13b * ux; uxb += a13b * e.a03;
  a30b += a31b * uy; uyb += a31b * e.a30;
  a03b += a04b * uy; uyb += a04b * e.a03; sb += 3.0 * a04b * e.a02; a02b += 3.0 * s * a04b;
  a30b += a40b * ux; uxb += a40b * e.a30; sb += 3.0 * a40b * e.a20; a20b += 3.0 * s * a40b;
  a02b += a12b * ux; uxb += a12b * e.a02;
  a20b += a21b * uy; uyb += a21b * e.a20;
  a02b += a03b * uy; uyb += a03b * e.a02; sb += 2.0 * a03b * e.a01; a01b += 2.0 * s * a03b;
  a20b += a30b * ux; uxb += a30b * e.a20; sb += 2.0 * a30b * e.a10; a10b += 2.0 * s * a30b;
  a01b += a02b * uy; uyb += a02b * e.a01; rsb += a02b;
  a10b += a11b * uy; uyb += a11b * e.a10;
  a10b += a20b * ux; uxb += a20b * e.a10; rsb += a20b;
  rhob += a01b * uy; uyb += a01b * rho;
  rhob += a10b * ux; uxb += a10b * rho;
  rhob += a00b;
  rhob += rsb * s; sb += rsb * rho;
  // a1 = 1 - k1 ; s1 = k1 - k2
  k1b += s1b - a1b;
  k2b -= s1b;
  double pbar;
  if (PRC <= 0) {  // k1 = dt_mu p ; k2 = k1 Pr
    k1b += k2b * P.Pr; pb.Pr += k2b * k1;
    pb.dt_mu += k1b * p; pbar = k1b * P.dt_mu;
  } else {         // k2 = dt_mu p ; k1 = k2 Pr
    k2b += k1b * P.Pr; pb.Pr += k1b * k2;
    pb.dt_mu += k2b * p; pbar = k2b * P.dt_mu;
  }
  // p = rho c2 theta
  rhob += pbar * P.c2 * theta;
  thetab += pbar * rho * P.c2;
  // s = theta - 1
  thetab += sb;
  // theta = gm1 w, w = Et irho - q/2
  pb.gm1 += thetab * w;
  const double wb = thetab * P.gm1;
  const double Etb = wb * irho;
  double irhob = wb * Et;
  const double qb = -0.5 * wb;
  uxb += 2.0 * ux * qb;
  uyb += 2.0 * uy * qb;
  mb.m20 += 0.5 * Etb; mb.m02 += 0.5 * Etb; mb.g00 += Etb * P.inv_c2;
  mb.m10 += uxb * irho; irhob += uxb * m.m10;
  mb.m01 += uyb * irho; irhob += uyb * m.m01;
  rhob -= irhob * irho * irho;
  mb.m00 += rhob;
  return 1.0 - k1;  // a1 of the forward step
}

// Reverse of the (rho, T) read-out of the moments (macro_from_moments): given
// dL/drho and dL/dT, accumulate the moment adjoints and dL/d(gamma - 1).
__device__ __forceinline__ void macro_rev(const Moments& m, const Phys& P, double T_ref, double rhob_in, double Tb,
                                          Moments& mb, ParamBar& pb) {
  const double rho = m.m00;
  const double irho = 1.0 / rho;
  const double ux = m.m10 * irho, uy = m.m01 * irho;
  const double Et = fma(0.5, m.m20 + m.m02, m.g00 * P.inv_c2);
  const double w = fma(-0.5, fma(ux, ux, uy * uy), Et * irho);
  const double thetab = Tb * T_ref;
  pb.gm1 += thetab * w;
  const double wb = thetab * P.gm1;
  const double Etb = wb * irho;
  double irhob = wb * Et;
  const double qb = -0.5 * wb;
  const double uxb = 2.0 * ux * qb, uyb = 2.0 * uy * qb;
  mb.m20 += 0.5 * Etb; mb.m02 += 0.5 * Etb; mb.g00 += Etb * P.inv_c2;
  mb.m10 += uxb * irho; irhob += uxb * m.m10;
  mb.m01 += uyb * irho; irhob += uyb * m.m01;
  mb.m00 += rhob_in - irhob * irho * irho;
}

// Reverse of equilibrium_coeffs (initial conditions): from Cbar to the
// adjoints of rho, u (units of c), theta and epsf.
__device__ __forceinline__ void equilibrium_rev(double rho, double ux, double uy, double theta, const Phys& P,
                                                const Coeffs& Cb, double& rhob, double& uxb, double& uyb,
                                                double& thetab, double& epsfb) {
  const double s = theta - 1.0;
  const EqF e = eq_f(rho, ux, uy, s);
  const double reps = rho * P.epsf * theta * P.c2;
  double sb = 0;
  const double repsb = Cb.g00 + Cb.g10 * ux + Cb.g01 * uy + Cb.g20 * fma(ux, ux, s) + Cb.g11 * ux * uy +
                       Cb.g02 * fma(uy, uy, s);
  uxb = reps * (Cb.g10 + 2.0 * ux * Cb.g20 + uy * Cb.g11);
  uyb = reps * (Cb.g01 + 2.0 * uy * Cb.g02 + ux * Cb.g11);
  sb += reps * (Cb.g20 + Cb.g02);
  rhob = repsb * P.epsf * theta * P.c2;
  epsfb = repsb * rho * theta * P.c2;
  thetab = repsb * rho * P.epsf * P.c2;
  double a00b = Cb.f00, a10b = Cb.f10, a01b = Cb.f01, a20b = Cb.f20, a11b = Cb.f11, a02b = Cb.f02, a30b = Cb.f30,
         a21b = Cb.f21, a12b = Cb.f12, a03b = Cb.f03, a40b = Cb.f40, a31b = Cb.f31, a22b = Cb.f22, a13b = Cb.f13,
         a04b = Cb.f04;
  double rsb = 0;
  a20b += a22b * fma(uy, uy, s); uyb += a22b * e.a20 * 2.0 * uy; sb += a22b * e.a20;
  a03b += a13b * ux; uxb += a13b * e.a03;
  a30b += a31b * uy; uyb += a31b * e.a30;
  a03b += a04b * uy; uyb += a04b * e.a03; sb += 3.0 * a04b * e.a02; a02b += 3.0 * s * a04b;
  a30b += a40b * ux; uxb += a40b * e.a30; sb += 3.0 * a40b * e.a20; a20b += 3.0 * s * a40b;
  a02b += a12b * ux; uxb += a12b * e.a02;
  a20b += a21b * uy; uyb += a21b * e.a20;
  a02b += a03b * uy; uyb += a03b * e.a02; sb += 2.0 * a03b * e.a01; a01b += 2.0 * s * a03b;
  a20b += a30b * ux; uxb += a30b * e.a20; sb += 2.0 * a30b * e.a10; a10b += 2.0 * s * a30b;
  a01b += a02b * uy; uyb += a02b * e.a01; rsb += a02b;
  a10b += a11b * uy; uyb += a11b * e.a10;
  a10b += a20b * ux; uxb += a20b * e.a10; rsb += a20b;
  rhob += a01b * uy; uyb += a01b * rho;
  rhob += a10b * ux; uxb += a10b * rho;
  rhob += a00b;
  rhob += rsb * s; sb += rsb * rho;
  thetab += sb;
}

// ------------------------------------------------------- projections / moments
// kh(k, n) 2^63 for every node (no per-node scaling: the projection sums over
// nodes at one scale); |kh| < 0.54
__host__ __device__ constexpr long long c0fix(int k, int n) { return (long long)(kh(k, n) * 9223372036854775808.0); }

// Cbar_ab = sum over the node's populations of lambda W W He_a He_b /(a! b!):
// accumulate the contribution of x-node p (lf, lg: the 5 f and g values).
template <int p>
__device__ __forceinline__ void accumulate_projection(Coeffs& Cb, const double (&lf)[5], const double (&lg)[5]) {
  double hb[5];  // hbar^b_p = sum_q lambda_pq kh(q, b)
  {
    const double sA = lf[1] + lf[2], dA = lf[1] - lf[2], sB = lf[3] + lf[4], dB = lf[3] - lf[4];
    hb[0] = fma(kh(3, 0), sB, fma(kh(1, 0), sA, kh(0, 0) * lf[0]));
    hb[1] = fma(kh(3, 1), dB, kh(1, 1) * dA);
    hb[2] = fma(kh(3, 2), sB, fma(kh(1, 2), sA, kh(0, 2) * lf[0]));
    hb[3] = fma(kh(3, 3), dB, kh(1, 3) * dA);
    hb[4] = fma(kh(3, 4), sB, fma(kh(1, 4), sA, kh(0, 4) * lf[0]));
  }
  Cb.f00 = fma(kh(p, 0), hb[0], Cb.f00);
  Cb.f01 = fma(kh(p, 0), hb[1], Cb.f01);
  Cb.f02 = fma(kh(p, 0), hb[2], Cb.f02);
  Cb.f03 = fma(kh(p, 0), hb[3], Cb.f03);
  Cb.f04 = fma(kh(p, 0), hb[4], Cb.f04);
  Cb.f20 = fma(kh(p, 2), hb[0], Cb.f20);
  Cb.f21 = fma(kh(p, 2), hb[1], Cb.f21);
  Cb.f22 = fma(kh(p, 2), hb[2], Cb.f22);
  Cb.f40 = fma(kh(p, 4), hb[0], Cb.f40);
  if (p != 0) {
    Cb.f10 = fma(kh(p, 1), hb[0], Cb.f10);
    Cb.f11 = fma(kh(p, 1), hb[1], Cb.f11);
    Cb.f12 = fma(kh(p, 1), hb[2], Cb.f12);
    Cb.f13 = fma(kh(p, 1), hb[3], Cb.f13);
    Cb.f30 = fma(kh(p, 3), hb[0], Cb.f30);
    Cb.f31 = fma(kh(p, 3), hb[1], Cb.f31);
  }
  double gb[3];
  {
    const double sA = lg[1] + lg[2], dA = lg[1] - lg[2], sB = lg[3] + lg[4], dB = lg[3] - lg[4];
    gb[0] = fma(kh(3, 0), sB, fma(kh(1, 0), sA, kh(0, 0) * lg[0]));
    gb[1] = fma(kh(3, 1), dB, kh(1, 1) * dA);
    gb[2] = fma(kh(3, 2), sB, fma(kh(1, 2), sA, kh(0, 2) * lg[0]));
  }
  Cb.g00 = fma(kh(p, 0), gb[0], Cb.g00);
  Cb.g01 = fma(kh(p, 0), gb[1], Cb.g01);
  Cb.g02 = fma(kh(p, 0), gb[2], Cb.g02);
  Cb.g20 = fma(kh(p, 2), gb[0], Cb.g20);
  if (p != 0) {
    Cb.g10 = fma(kh(p, 1), gb[0], Cb.g10);
    Cb.g11 = fma(kh(p, 1), gb[1], Cb.g11);
  }
}

// The same projection in block fixed point on the integer pipe (the adjoint
// of the fixed-point expansion of the forward step): lambda of the cell at a
// shared exponent per f / g (60-bit), node constants kh 2^63, products as
// high words; the partial sums of all five x-nodes share one scale, so that
// cbar accumulates across nodes without renormalisation.  Value of cbar_ab:
// cb 2^(E - 1080).  cb: this thread's 21 accumulators in shared memory (f
// fields 0..14 in Coeffs order, g fields 15..20, stride 256).
template <int p>
__device__ __forceinline__ void accumulate_projection_fix(long long* __restrict__ cb, const double (&lf)[5],
                                                          const double (&lg)[5], int Ef, int Eg) {
  long long hb[5];
  {
    const long long l0 = to_block_fixed(lf[0], Ef), l1 = to_block_fixed(lf[1], Ef), l2 = to_block_fixed(lf[2], Ef),
                    l3 = to_block_fixed(lf[3], Ef), l4 = to_block_fixed(lf[4], Ef);
    const long long sA = l1 + l2, dA = l1 - l2, sB = l3 + l4, dB = l3 - l4;
    hb[0] = mhk(l0, c0fix(0, 0)) + mhk(sA, c0fix(1, 0)) + mhk(sB, c0fix(3, 0));
    hb[1] = mhk(dA, c0fix(1, 1)) + mhk(dB, c0fix(3, 1));
    hb[2] = mhk(l0, c0fix(0, 2)) + mhk(sA, c0fix(1, 2)) + mhk(sB, c0fix(3, 2));
    hb[3] = mhk(dA, c0fix(1, 3)) + mhk(dB, c0fix(3, 3));
    hb[4] = mhk(l0, c0fix(0, 4)) + mhk(sA, c0fix(1, 4)) + mhk(sB, c0fix(3, 4));
  }
  // field order f00, f10, f01, f20, f11, f02, f30, f21, f12, f03, f40, f31, f22, f13, f04
  cb[0 * 256] += mhk(hb[0], c0fix(p, 0));
  cb[2 * 256] += mhk(hb[1], c0fix(p, 0));
  cb[5 * 256] += mhk(hb[2], c0fix(p, 0));
  cb[9 * 256] += mhk(hb[3], c0fix(p, 0));
  cb[14 * 256] += mhk(hb[4], c0fix(p, 0));
  cb[3 * 256] += mhk(hb[0], c0fix(p, 2));
  cb[7 * 256] += mhk(hb[1], c0fix(p, 2));
  cb[12 * 256] += mhk(hb[2], c0fix(p, 2));
  cb[10 * 256] += mhk(hb[0], c0fix(p, 4));
  if (p != 0) {
    cb[1 * 256] += mhk(hb[0], c0fix(p, 1));
    cb[4 * 256] += mhk(hb[1], c0fix(p, 1));
    cb[8 * 256] += mhk(hb[2], c0fix(p, 1));
    cb[13 * 256] += mhk(hb[3], c0fix(p, 1));
    cb[6 * 256] += mhk(hb[0], c0fix(p, 3));
    cb[11 * 256] += mhk(hb[1], c0fix(p, 3));
  }
  long long gb[3];
  {
    const long long l0 = to_block_fixed(lg[0], Eg), l1 = to_block_fixed(lg[1], Eg), l2 = to_block_fixed(lg[2], Eg),
                    l3 = to_block_fixed(lg[3], Eg), l4 = to_block_fixed(lg[4], Eg);
    const long long sA = l1 + l2, dA = l1 - l2, sB = l3 + l4, dB = l3 - l4;
    gb[0] = mhk(l0, c0fix(0, 0)) + mhk(sA, c0fix(1, 0)) + mhk(sB, c0fix(3, 0));
    gb[1] = mhk(dA, c0fix(1, 1)) + mhk(dB, c0fix(3, 1));
    gb[2] = mhk(l0, c0fix(0, 2)) + mhk(sA, c0fix(1, 2)) + mhk(sB, c0fix(3, 2));
  }
  // g order g00, g10, g01, g20, g11, g02
  cb[15 * 256] += mhk(gb[0], c0fix(p, 0));
  cb[17 * 256] += mhk(gb[1], c0fix(p, 0));
  cb[20 * 256] += mhk(gb[2], c0fix(p, 0));
  cb[18 * 256] += mhk(gb[0], c0fix(p, 2));
  if (p != 0) {
    cb[16 * 256] += mhk(gb[0], c0fix(p, 1));
    cb[19 * 256] += mhk(gb[1], c0fix(p, 1));
  }
}

// sum_j mbar_j dm_j/dX for the populations (p, q) of one x-node:
// f: sum_{a+b<=3} mbar_ab xi_p^a xi_q^b ; g: gbar00 + gbar10 xi_p + gbar01 xi_q
template <int p>
__device__ __forceinline__ void moment_pullback(const Moments& mb, double (&pf)[5], double (&pg)[5]) {
  constexpr double x = xi_of(p);
  const double b0 = fma(x * x * x, mb.m30, fma(x * x, mb.m20, fma(x, mb.m10, mb.m00)));
  const double b1 = fma(x * x, mb.m21, fma(x, mb.m11, mb.m01));
  const double b2 = fma(x, mb.m12, mb.m02);
  const double b3 = mb.m03;
  const double g0 = fma(x, mb.g10, mb.g00);
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    const double y = xi_of(q);
    pf[q] = fma(y * y * y, b3, fma(y * y, b2, fma(y, b1, b0)));
    pg[q] = fma(y, mb.g01, g0);
  }
}

// ------------------------------------------------------------ advection adjoint
// minmod branch of sigma(Da, Db) with block-fixed integers: 0 zero, 1 hb Da,
// 2 (Da + Db)/4, 3 hb Db.  Ties resolve in the order hb Da, (Da+Db)/4, hb Db.
__device__ __forceinline__ int slope_branch(long long Da, long long Db, long long ra, long long rb) {
  if ((Da ^ Db) < 0) return 0;
  const long long y = (Da + Db) >> 2;
  if (Da >= 0) {
    if (ra <= y && ra <= rb) return 1;
    return y <= rb ? 2 : 3;
  }
  if (ra >= y && ra >= rb) return 1;
  return y >= rb ? 2 : 3;
}
// partial derivatives (first, second argument) times an integer sbar
__device__ __forceinline__ long long slope_d1(int br, long long sbar, long long Hq) {
  return br == 1 ? __mul64hi(sbar << 2, Hq) : (br == 2 ? (sbar >> 2) : 0ll);
}
__device__ __forceinline__ long long slope_d2(int br, long long sbar, long long Hq) {
  return br == 3 ? __mul64hi(sbar << 2, Hq) : (br == 2 ? (sbar >> 2) : 0ll);
}

// lambda values at block exponent with 6 fraction-guard bits less than the
// forward conversion (headroom for the sums below)
__device__ __forceinline__ long long to_block_fixed6(double v, int E) { return to_block_fixed(v, E) >> 1; }

// Adjoint of the flux difference of one population along one axis, gathered
// at cell c: returns sum_{c'} lambda(c') dF(c')/dX(c) (multiply by -k outside).
__device__ __forceinline__ double advection_adjoint(const double* __restrict__ X, const double* __restrict__ L,
                                                    long long stride, long long Hq, int sgn) {
  double xv[5], lv[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    xv[k] = __ldg(X + (k - 2) * stride);
    lv[k] = __ldg(L + (k - 2) * stride);
  }
  const int EX = max(max(max(bexp(xv[0]), bexp(xv[1])), max(bexp(xv[2]), bexp(xv[3]))), bexp(xv[4]));
  long long xi[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) xi[k] = to_block_fixed(xv[k], EX);
  // differences D_{c-1} .. D_{c+2} (index 0..3) and slope branches of
  // sigma_{c-1} (D_{c-1}, D_c), sigma_c (D_c, D_{c+1}), sigma_{c+1} (D_{c+1}, D_{c+2})
  long long D[4], r[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    D[k] = xi[k + 1] - xi[k];
    r[k] = __mul64hi(D[k] << 2, Hq);
  }
  const int bm = slope_branch(D[0], D[1], r[0], r[1]);
  const int b0 = slope_branch(D[1], D[2], r[1], r[2]);
  const int bp = slope_branch(D[2], D[3], r[2], r[3]);
  const int EL = max(max(max(bexp(lv[0]), bexp(lv[1])), max(bexp(lv[2]), bexp(lv[3]))), bexp(lv[4]));
  long long l[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) l[k] = to_block_fixed6(lv[k], EL);
  long long Xb;
  if (sgn > 0) {
    // sbar_k = l_k - l_{k+1}; Dbar_c = l_c + d1(sigma_c) sbar_c + d2(sigma_{c-1}) sbar_{c-1}
    const long long sbm = l[1] - l[2], sb0 = l[2] - l[3], sbp = l[3] - l[4];
    const long long Dc = l[2] + slope_d1(b0, sb0, Hq) + slope_d2(bm, sbm, Hq);
    const long long Dc1 = l[3] + slope_d1(bp, sbp, Hq) + slope_d2(b0, sb0, Hq);
    Xb = Dc - Dc1;
  } else {
    // sbar_k = l_k - l_{k-1}; Dbar_k = l_{k-1} + d1(sigma_k) sbar_k + d2(sigma_{k-1}) sbar_{k-1}
    const long long sbm = l[1] - l[0], sb0 = l[2] - l[1], sbp = l[3] - l[2];
    const long long Dc = l[1] + slope_d1(b0, sb0, Hq) + slope_d2(bm, sbm, Hq);
    const long long Dc1 = l[2] + slope_d1(bp, sbp, Hq) + slope_d2(b0, sb0, Hq);
    Xb = Dc - Dc1;
  }
  // value at exponent EL: Xb 2^(EL - 1081)
  if (EL < 64) return 0.0;
  return ll_to_double_scaled(Xb, EL - 1081);
}

// Rational-beta variant (beta = lp/lq): every partial derivative times 4 lq is
// a small integer (2 lp for beta/2, lq for 1/4), so the adjoint combinations
// are exact integer arithmetic without high multiplies.  Returns 4 lq times
// sum_{c'} lambda(c') dF(c')/dX(c).  lambda enters with a 50-bit significand.
__device__ __forceinline__ int slope_branch_rat(long long Da, long long Db, long long lp2, long long lq) {
  if ((Da ^ Db) < 0) return 0;
  const long long ra = lp2 * Da, rb = lp2 * Db, y = lq * (Da + Db);
  if (Da >= 0) {
    if (ra <= y && ra <= rb) return 1;
    return y <= rb ? 2 : 3;
  }
  if (ra >= y && ra >= rb) return 1;
  return y >= rb ? 2 : 3;
}

// lambda part of the rational-beta advection adjoint, given the minmod branch
// codes bm, b0, bp of the slopes sigma_{c-1}, sigma_c, sigma_{c+1} along the
// stride.  Returns 4 lq sum_{c'} lambda(c') dF(c')/dX(c).
__device__ __forceinline__ double adjoint_combine_rat(const double* __restrict__ L, long long stride, int bm, int b0,
                                                      int bp, int lp, int lq, int sgn) {
  double lv[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) lv[k] = __ldg(L + (k - 2) * stride);
  const long long lp2 = 2 * lp, q = lq, q4 = 4 * lq;
  const int EL = max(max(max(bexp(lv[0]), bexp(lv[1])), max(bexp(lv[2]), bexp(lv[3]))), bexp(lv[4]));
  long long l[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) l[k] = to_block_fixed(lv[k], EL) >> 10;
  auto d1 = [&](int br, long long sb) { return br == 1 ? lp2 * sb : (br == 2 ? q * sb : 0ll); };
  auto d2 = [&](int br, long long sb) { return br == 3 ? lp2 * sb : (br == 2 ? q * sb : 0ll); };
  long long Xb;
  if (sgn > 0) {
    const long long sbm = l[1] - l[2], sb0 = l[2] - l[3], sbp = l[3] - l[4];
    Xb = (q4 * l[2] + d1(b0, sb0) + d2(bm, sbm)) - (q4 * l[3] + d1(bp, sbp) + d2(b0, sb0));
  } else {
    const long long sbm = l[1] - l[0], sb0 = l[2] - l[1], sbp = l[3] - l[2];
    Xb = (q4 * l[1] + d1(b0, sb0) + d2(bm, sbm)) - (q4 * l[2] + d1(bp, sbp) + d2(b0, sb0));
  }
  if (EL < 64) return 0.0;
  return ll_to_double_scaled(Xb, EL - 1072);  // lambda was scaled by 2^(1072 - EL)
}

__device__ __forceinline__ double advection_adjoint_rat(const double* __restrict__ X, const double* __restrict__ L,
                                                        long long stride, int lp, int lq, int sgn) {
  double xv[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) xv[k] = __ldg(X + (k - 2) * stride);
  const int EX = max(max(max(bexp(xv[0]), bexp(xv[1])), max(bexp(xv[2]), bexp(xv[3]))), bexp(xv[4]));
  const long long lp2 = 2 * lp, q = lq;
  long long D[4];
  {
    long long xi[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) xi[k] = to_block_fixed52(xv[k], EX);
#pragma unroll
    for (int k = 0; k < 4; ++k) D[k] = xi[k + 1] - xi[k];
  }
  const int bm = slope_branch_rat(D[0], D[1], lp2, q);
  const int b0 = slope_branch_rat(D[1], D[2], lp2, q);
  const int bp = slope_branch_rat(D[2], D[3], lp2, q);
  return adjoint_combine_rat(L, stride, bm, b0, bp, lp, lq, sgn);
}

// ------------------------------------------------- the coded adjoint step over tiles
// One adjoint step in one launch, with the branch codes of the recomputed forward
// step, in the forward step's two phases (k_step_tile): first one population per
// warp over a 32 x R tile, then one cell per thread.  512^2: 0.47 ms for the two
// kernels it replaces (one thread per cell and population in the advection, 64-bit
// high products in the projection) -> 0.36 ms.  Bound by the FP64 pipe (53 % busy, 436
// instructions a cell, about half of them the reverse pass over the collision
// coefficients) and by latency at 15 warps an SM.  100^2, all latency, with 4-row
// tiles and the parts of a cell on several threads: 110 -> 75 us a step with the
// recompute.

// a code's multipliers 4 lq d(sigma)/d(first argument), /d(second), as a byte table
// indexed by the code (lp and lq are coprime and lq <= 64, so 2 lp <= 254 fits)
__device__ __forceinline__ unsigned code_factor(unsigned table, unsigned code) {
  return __byte_perm(table, 0u, (code & 3u) | 0x4440u);
}

// What a warp reads of one population: the adjoint state at its lane's column in
// stream rows -1 .. R + 1, one cell of the x-halo, the branch codes of its
// column in rows -1 .. R (packed: x bits of rows 0 .., y bits of rows -1 ..)
// and, lanes 0 .. 2 R - 1, of the cells before and behind row lane % R.
template <int R>
struct AdjointLoad {
  double v[R + 3], h;
  unsigned char code[R + 2], edge;
};
struct CodePlane {
  const unsigned char *own, *lo, *hi;  // [Ny][Nx]; the rows below y = 0 and above y = Ny - 1
  int Nx, Ny;
  __device__ __forceinline__ const unsigned char* row(int y) const {
    return y < 0 ? lo : y >= Ny ? hi : own + (long long)y * Nx;
  }
};
template <int R>
__device__ __forceinline__ void adjoint_load(AdjointLoad<R>& L, const double* __restrict__ plane, long long PT,
                                             const CodePlane& C, int x0, int y0, const AdvTile& T) {
  const int i = min(T.lane, T.W - 1);
  const int cx = T.fx ? T.W - 1 - i : i;
  const long long sy = T.fy ? -PT : PT;
  const double* row0 = plane + (T.fy ? (T.H - 1) * PT : 0);
#pragma unroll
  for (int j = -1; j <= R + 1; ++j) L.v[j + 1] = __ldg(at(row0 + min(j, T.H + 1) * sy, (unsigned)cx * 8u));
  const int hr = min(T.lane % R, T.H - 1), hc = T.lane / R;  // stream columns -1, W, W + 1 (or 0)
  const int h = hc == 0 ? -1 : hc > 2 ? 0 : T.W - 1 + hc;
  L.h = __ldg(row0 + hr * sy + (T.fx ? T.W - 1 - h : h));
#pragma unroll
  for (int j = -1; j <= R; ++j) {
    const int y = y0 + (T.fy ? T.H - 1 - min(j, T.H) : min(j, T.H));
    L.code[j + 1] = __ldg(C.row(y) + x0 + cx);
  }
  const int he = T.lane < R ? -1 : T.W;
  int xe = x0 + (T.fx ? T.W - 1 - he : he);
  xe = xe < 0 ? C.Nx - 1 : xe >= C.Nx ? 0 : xe;
  L.edge = __ldg(C.own + (long long)(y0 + (T.fy ? T.H - 1 - hr : hr)) * C.Nx + xe);
}

// The transpose of advect_tile, gathered: with sb_i = l_i - l_{i+1} along the
// stream and the slopes' partial derivatives d1, d2,
//     Dbar_i = l_i + d1(sigma_i) sb_i + d2(sigma_{i-1}) sb_{i-1},
// cell i gets k (Dbar_i - Dbar_{i+1}), subtracted from its adjoint.  Writes the
// sums over both axes as integers in units of 2^(E - 1076), returns E.  Walked
// against an axis, the codes' arguments are swapped (tables t1, t2).
template <int R, bool MX, bool MY, class Next>
__device__ __forceinline__ int adjoint_walk(const AdjointLoad<R>& L, const Next& next, long long* out, long long PT,
                                            const AdvTile& T, const Phys& P, long long kx, long long ky, long long* xs) {
  const int lane = T.lane;
  const bool in = lane < T.W;
  const unsigned lx = in ? (unsigned)(T.fx ? T.W - 1 - lane : lane) : 0u;
  const long long sy = T.fy ? -PT : PT;
  constexpr int J0 = MY ? -1 : 0, J1 = MY ? R + 1 : R - 1;
  unsigned key = 0;
#pragma unroll
  for (int j = J0; j <= J1; ++j) key = max(key, ((unsigned)__double2hiint(L.v[j + 1]) + 0x100000u) & 0x7fffffffu);
  if (MX) key = max(key, ((unsigned)__double2hiint(L.h) + 0x100000u) & 0x7fffffffu);
  key = __reduce_max_sync(0xffffffffu, key);
  const int E = (int)(key >> 20) - 1;
  const BlockScale B(E, P.advn + 3);
  __syncwarp();
#pragma unroll
  for (int j = J0; j <= J1; ++j) xs[(j + 1) * kAdvPitch + lane + 1] = block_fix(L.v[j + 1], B);
  const int hr = lane % R, hc = lane / R;
  if (MX) {
    __syncwarp();
    if (hc < 3 && hr < T.H) xs[(hr + 1) * kAdvPitch + (hc == 0 ? 0 : T.W + hc)] = block_fix(L.h, B);
  }
  unsigned xb = 0, yb = 0;  // codes of rows 0 .. R - 1 (x), -1 .. R (y), two bits each
#pragma unroll
  for (int j = 0; j < R; ++j) xb |= (unsigned)(L.code[j + 1] & 3) << (2 * j);
#pragma unroll
  for (int j = -1; j <= R; ++j) yb |= (unsigned)(L.code[j + 1] >> 2) << (2 * (j + 1));
  const unsigned edge = L.edge & 3u;
  next();
  __syncwarp();
  const unsigned q4 = 4u * (unsigned)P.lq;
  const unsigned f1 = (2u * (unsigned)P.lp) << 8 | (unsigned)P.lq << 16, f3 = (2u * (unsigned)P.lp) << 24 | (unsigned)P.lq << 16;
  const unsigned x1 = T.fx ? f3 : f1, x2 = T.fx ? f1 : f3, y1 = T.fy ? f3 : f1, y2 = T.fy ? f1 : f3;
  if (MX) {
    // Dbar of column W, one row per lane, kept in column W + 1
    const unsigned last = __shfl_sync(0xffffffffu, xb, T.W - 1);  // codes of column W - 1
    const unsigned be = __shfl_sync(0xffffffffu, edge, R + lane % R);
    if (lane < T.H) {
      long long* r = xs + (lane + 1) * kAdvPitch + T.W;  // column W - 1
      const long long a = r[0] - r[1], b = r[1] - r[2];
      r[2] = mad_small(r[1], q4, mad_small(b, code_factor(x1, be), mad_small(a, code_factor(x2, last >> (2 * lane)), 0)));
    }
    __syncwarp();
  }
  const Limbs KX(kx), KY(ky);
  const long long* own = xs + kAdvPitch + lane + 1;  // (row 0, this column)
  long long c = own[0], sb = 0, dy = 0;
  if (MY) {
    const long long n = own[kAdvPitch], sm = own[-kAdvPitch] - c;
    sb = c - n;
    dy = mad_small(c, q4, mad_small(sb, code_factor(y1, yb >> 2), mad_small(sm, code_factor(y2, yb), 0)));
    yb >>= 2;
  }
  long long* orow = out + (T.fy ? (T.H - 1) * PT : 0);
#pragma unroll 1
  for (int j = 0; j < T.H; ++j) {
    LimbAcc w;
    if (MX) {
      const unsigned b0 = xb & 3u;
      unsigned bm = __shfl_up_sync(0xffffffffu, b0, 1);
      const unsigned e0 = __shfl_sync(0xffffffffu, edge, j);
      if (lane == 0) bm = e0;
      const long long s0 = c - own[1], sm = own[-1] - c;
      const long long d = mad_small(c, q4, mad_small(s0, code_factor(x1, b0), mad_small(sm, code_factor(x2, bm), 0)));
      long long dn = __shfl_down_sync(0xffffffffu, d, 1);
      const long long de = xs[(j + 1) * kAdvPitch + T.W + 2];
      if (lane == T.W - 1) dn = de;
      const Limbs f(d - dn);
      w.mac(f.h, f.l, KX.h, KX.l);
      xb >>= 2;
    }
    const long long n = own[kAdvPitch];
    if (MY) {
      const long long s1 = n - own[2 * kAdvPitch];
      const long long d = mad_small(n, q4, mad_small(s1, code_factor(y1, yb >> 2), mad_small(sb, code_factor(y2, yb), 0)));
      const Limbs f(dy - d);
      w.mac(f.h, f.l, KY.h, KY.l);
      dy = d;
      sb = s1;
      yb >>= 2;
    }
    if (in) *at(orow, lx * 8) = w.floor();
    c = n;
    own += kAdvPitch;
    orow += sy;
  }
  return E;
}

// node constants W_k He_n(xi_k)/n! 2^61 without a node's own scale: the projection
// sums over nodes
constexpr long long kK0[3][5] = {
    {1229782938247303441ll, 0ll, -614891469123651721ll, 0ll, 153722867280912930ll},
    {512072212271327456ll, 694178496992351028ll, 214487165913345387ll, -134471359870578684ll, -99195015452660690ll},
    {25957823211867799ll, 74160722541717783ll, 92958568648480473ll, 63806373539842544ll, 22333581812204225ll}};
template <int cls, int n>
__device__ __forceinline__ void k0mac(LimbAcc& s, const Limbs& x) {
  s.mac(x.h, x.l, limb_hi(kK0[cls][n]), limb_lo(kK0[cls][n]));
}

// The projection Cbar_ab = sum lambda W W He_a He_b / (a! b!) of one family in block
// fixed point (the transpose of the forward expansion): N = 4 (f) or 2 (g), 58-bit
// values at the block exponent E; also a1b += sum lambda X.  cb: fields in Coeffs order.
template <int N>
__device__ __forceinline__ void project(const double* __restrict__ lam, const double* __restrict__ X, unsigned off,
                                        long long PL, double (&cb)[N == 4 ? 15 : 6], double& a1b) {
  double v[25];
  unsigned key = 0;
#pragma unroll
  for (int i = 0; i < 25; ++i) {
    v[i] = __ldg(at(lam + i * PL, off));
    key = max(key, ((unsigned)__double2hiint(v[i]) + 0x100000u) & 0x7fffffffu);
  }
  const int E = (int)(key >> 20) - 1;
  const BlockScale B(E, 2);
  long long c[N + 1], s[2][N + 1], d[2][N + 1];  // y-projections: centre node, sums and differences of the node pairs
#pragma unroll
  for (int p = 0; p < 5; ++p) {
    long long h[N + 1];
#pragma unroll
    for (int q = 0; q < 5; ++q) a1b = fma(v[5 * p + q], __ldg(at(X + (5 * p + q) * PL, off)), a1b);
    const long long l0 = block_fix(v[5 * p], B), l1 = block_fix(v[5 * p + 1], B),
                    l2 = block_fix(v[5 * p + 2], B), l3 = block_fix(v[5 * p + 3], B),
                    l4 = block_fix(v[5 * p + 4], B);
    const Limbs z(l0), sA(l1 + l2), dA(l1 - l2), sB(l3 + l4), dB(l3 - l4);
    LimbAcc a0, a1, a2;
    k0mac<0, 0>(a0, z); k0mac<1, 0>(a0, sA); k0mac<2, 0>(a0, sB);
    k0mac<1, 1>(a1, dA); k0mac<2, 1>(a1, dB);
    k0mac<0, 2>(a2, z); k0mac<1, 2>(a2, sA); k0mac<2, 2>(a2, sB);
    h[0] = a0.value8(); h[1] = a1.value8(); h[2] = a2.value8();
    if constexpr (N == 4) {
      LimbAcc a3, a4;
      k0mac<1, 3>(a3, dA); k0mac<2, 3>(a3, dB);
      k0mac<0, 4>(a4, z); k0mac<1, 4>(a4, sA); k0mac<2, 4>(a4, sB);
      h[3] = a3.value8(); h[4] = a4.value8();
    }
#pragma unroll
    for (int b = 0; b <= N; ++b) {
      if (p == 0) c[b] = h[b];
      else if (p & 1) s[p >> 1][b] = h[b];
      else {
        const long long t = s[(p >> 1) - 1][b];
        s[(p >> 1) - 1][b] = t + h[b];
        d[(p >> 1) - 1][b] = t - h[b];
      }
    }
  }
  const int sc = E - 1080;
#define DVBM_EVEN(a, b)                                                                         \
  [&] {                                                                                         \
    LimbAcc t;                                                                                  \
    k0mac<0, a>(t, Limbs(c[b])); k0mac<1, a>(t, Limbs(s[0][b])); k0mac<2, a>(t, Limbs(s[1][b])); \
    return fix_to_double(t.value8(), sc);                                                 \
  }()
#define DVBM_ODD(a, b)                                                \
  [&] {                                                               \
    LimbAcc t;                                                        \
    k0mac<1, a>(t, Limbs(d[0][b])); k0mac<2, a>(t, Limbs(d[1][b]));   \
    return fix_to_double(t.value8(), sc);                       \
  }()
  if constexpr (N == 4) {
    // f00, f10, f01, f20, f11, f02, f30, f21, f12, f03, f40, f31, f22, f13, f04
    cb[0] = DVBM_EVEN(0, 0); cb[1] = DVBM_ODD(1, 0); cb[2] = DVBM_EVEN(0, 1); cb[3] = DVBM_EVEN(2, 0);
    cb[4] = DVBM_ODD(1, 1); cb[5] = DVBM_EVEN(0, 2); cb[6] = DVBM_ODD(3, 0); cb[7] = DVBM_EVEN(2, 1);
    cb[8] = DVBM_ODD(1, 2); cb[9] = DVBM_EVEN(0, 3); cb[10] = DVBM_EVEN(4, 0); cb[11] = DVBM_ODD(3, 1);
    cb[12] = DVBM_EVEN(2, 2); cb[13] = DVBM_ODD(1, 3); cb[14] = DVBM_EVEN(0, 4);
  } else {
    // g00, g10, g01, g20, g11, g02
    cb[0] = DVBM_EVEN(0, 0); cb[1] = DVBM_ODD(1, 0); cb[2] = DVBM_EVEN(0, 1);
    cb[3] = DVBM_EVEN(2, 0); cb[4] = DVBM_ODD(1, 1); cb[5] = DVBM_EVEN(0, 2);
  }
#undef DVBM_EVEN
#undef DVBM_ODD
}

// (XA / XB)^n 2^61
constexpr long long kR61[4] = {0, 1094117591372063814ll, 519156464237355984ll, 246338635339406942ll};
template <int n>
__device__ __forceinline__ void rmac(LimbAcc& s, long long x) {
  const Limbs l(x);
  s.mac(l.h, l.l, limb_hi(kR61[n]), limb_lo(kR61[n]));
}
// the moment adjoints of one family as 58-bit integers times XB^(a + b) at one
// exponent: polynomials in xi / XB, whose outer nodes are +-1
template <int N>
__device__ __forceinline__ int scale_moments(const double (&m)[N], long long (&Q)[N]) {
  unsigned key = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) key = max(key, abs_key(m[i]));
  const BlockScale B((int)(key >> 20), 2);
#pragma unroll
  for (int i = 0; i < N; ++i) Q[i] = block_fix(m[i], B);
  return max(B.E, 128);  // as in fields_to_smem
}

// BAND: a band of a slab-decomposed grid, whose code rows beyond its edges are glo
// and ghi ([NPOP][Nx]; NULL: the codes wrap).  moms: the moments of X, or NULL.
// partial[4 blk + k]: the block's sums of the parameter adjoints (dt_mu, Pr, gm1,
// epsf).
// R: tile height, as in k_step_tile; with R < 8 a cell has 8 / R threads: the first
// projects f and forms the moment adjoints, the second projects g, all share the
// populations.
template <int R, int PRC>
__global__ void __launch_bounds__(256, R == 8 ? 2 : 1) k_adjoint_tile(const double* __restrict__ X,
                                                         const double* __restrict__ Lin,
                                                         double* Lout, double* __restrict__ partial,
                                                         const unsigned char* __restrict__ codes,
                                                         const double* __restrict__ moms,
                                                         const unsigned char* __restrict__ glo,
                                                         const unsigned char* __restrict__ ghi, Geom G, Phys P) {
  __shared__ long long s_xs[8 * (R + 3) * kAdvPitch];
  __shared__ int s_exp[NPOP];
  const int x0 = blockIdx.x * 32, y0 = blockIdx.y * R;
  const long long PL = G.plane, PT = G.pitch, cplane = (long long)G.Nx * G.Ny;
  const double* ltile = Lin + cell_index(G, y0, x0);
  const double* xtile = X + cell_index(G, y0, x0);
  double* otile = Lout + cell_index(G, y0, x0);
  {
    const int w = __shfl_sync(0xffffffffu, (int)threadIdx.y, 0);
    const int c0 = 25 * (w >> 2), p = 1 + (w & 3);
    AdvTile T;
    T.W = min(32, G.Nx - x0);
    T.H = min(R, G.Ny - y0);
    T.lane = threadIdx.x;
    long long* xs = s_xs + w * ((R + 3) * kAdvPitch);
    auto tile = [&](int pp, int q) {
      AdvTile t = T;
      t.fx = Lat25::backward(pp);
      t.fy = Lat25::backward(q);
      return t;
    };
    AdjointLoad<R> V;
    auto load = [&](int pp, int q) {
      const int c = c0 + 5 * pp + q;
      CodePlane C;
      C.own = codes + c * cplane;
      C.Nx = G.Nx;
      C.Ny = G.Ny;
      C.lo = glo ? glo + (long long)c * G.Nx : C.own + (cplane - G.Nx);
      C.hi = ghi ? ghi + (long long)c * G.Nx : C.own;
      adjoint_load<R>(V, ltile + c * PL, PT, C, x0, y0, tile(pp, q));
    };
    auto out = [&](int c) { return (long long*)(otile + c * PL); };
    load(p, 0);
    int E = adjoint_walk<R, true, false>(V, [&] { load(p, 1); }, out(c0 + 5 * p), PT, tile(p, 0), P, P.kxq[p], 0, xs);
    if (T.lane == 0) s_exp[c0 + 5 * p] = E;
#pragma unroll 1
    for (int q = 1; q < 5; ++q) {
      const int c = c0 + 5 * p + q;
      E = adjoint_walk<R, true, true>(V, [&] { load(q < 4 ? p : 0, q < 4 ? q + 1 : p); }, out(c), PT, tile(p, q), P,
                                      P.kxq[p], P.kyq[q], xs);
      if (T.lane == 0) s_exp[c] = E;
    }
    E = adjoint_walk<R, false, true>(V, [] {}, out(c0 + p), PT, tile(0, p), P, 0, P.kyq[p], xs);
    if (T.lane == 0) s_exp[c0 + p] = E;
    if (p == 1) {
      if (T.lane == 0) s_exp[c0] = 0;
      if (T.lane < T.W)
        for (int j = 0; j < T.H; ++j) ((long long*)otile)[c0 * PL + j * PT + T.lane] = 0;
    }
  }
  __syncthreads();
  constexpr int NG = 8 / R;
  const int row = threadIdx.y % R, group = threadIdx.y / R;
  // threads beyond a ragged tile work on its last cell again and write nothing:
  // uniform control flow keeps the planes' addresses in uniform registers
  const bool active = x0 + (int)threadIdx.x < G.Nx && y0 + row < G.Ny;
  const int x = min(x0 + (int)threadIdx.x, G.Nx - 1), y = min(y0 + row, G.Ny - 1);
  const unsigned off = ((y - y0) * (unsigned)PT + (x - x0)) * 8u;
  ParamBar pb = {0, 0, 0, 0};
  // the moment adjoints of the collision (from the projections cb, cg and sum lambda X)
  // as fixed-point polynomials: f at exponent Ef, g at Eg
  double a1;
  long long F[10], H[3];
  int Ef, Eg;
  auto pull_back = [&](const double (&cb)[15], const double (&cg)[6], double a1b) {
    Coeffs Cb = {};
    Cb.f00 = cb[0]; Cb.f10 = cb[1]; Cb.f01 = cb[2]; Cb.f20 = cb[3]; Cb.f11 = cb[4]; Cb.f02 = cb[5];
    Cb.f30 = cb[6]; Cb.f21 = cb[7]; Cb.f12 = cb[8]; Cb.f03 = cb[9]; Cb.f40 = cb[10]; Cb.f31 = cb[11];
    Cb.f22 = cb[12]; Cb.f13 = cb[13]; Cb.f04 = cb[14];
    Cb.g00 = cg[0]; Cb.g10 = cg[1]; Cb.g01 = cg[2]; Cb.g20 = cg[3]; Cb.g11 = cg[4]; Cb.g02 = cg[5];
    Moments m;
    if (moms) {
      const long long ci = (long long)y * G.Nx + x;
      m.m00 = moms[0 * cplane + ci]; m.m10 = moms[1 * cplane + ci]; m.m01 = moms[2 * cplane + ci];
      m.m20 = moms[3 * cplane + ci]; m.m11 = moms[4 * cplane + ci]; m.m02 = moms[5 * cplane + ci];
      m.m30 = moms[6 * cplane + ci]; m.m21 = moms[7 * cplane + ci]; m.m12 = moms[8 * cplane + ci];
      m.m03 = moms[9 * cplane + ci]; m.g00 = moms[10 * cplane + ci]; m.g10 = moms[11 * cplane + ci];
      m.g01 = moms[12 * cplane + ci];
    } else {
      m = moments_fix<double>(xtile, off, PL);
    }
    Moments mb = {};
    a1 = collision_coeffs_rev<PRC>(m, P, Cb, a1b, mb, pb);
    // the pullback sum_j mbar_j dm_j/dX of population (p, q) is the polynomial
    // sum mbar_ab xi_p^a xi_q^b, in fixed point with the flux sum taken off
    const double mf[10] = {mb.m00, XB * mb.m10, XB * mb.m01, (XB * XB) * mb.m20, (XB * XB) * mb.m11, (XB * XB) * mb.m02,
                           (XB * XB * XB) * mb.m30, (XB * XB * XB) * mb.m21, (XB * XB * XB) * mb.m12,
                           (XB * XB * XB) * mb.m03};
    const double mg[3] = {mb.g00, XB * mb.g10, XB * mb.g01};
    Ef = scale_moments(mf, F);
    Eg = scale_moments(mg, H);
  };
  if constexpr (NG == 1) {
    double cb[15], cg[6], a1b = 0.0;
    project<4>(ltile, xtile, off, PL, cb, a1b);
    project<2>(ltile + 25 * PL, xtile + 25 * PL, off, PL, cg, a1b);
    pull_back(cb, cg, a1b);
  } else {
    __shared__ double s_g[7][32 * R], s_a1[32 * R];
    __shared__ long long s_p[13][32 * R];
    __shared__ int s_e[2][32 * R];
    const int cell = row * 32 + threadIdx.x;
    double cb[15], cg[6], a1b = 0.0;
    if (group == 0) project<4>(ltile, xtile, off, PL, cb, a1b);
    if (group == 1) {
      project<2>(ltile + 25 * PL, xtile + 25 * PL, off, PL, cg, a1b);
#pragma unroll
      for (int k = 0; k < 6; ++k) s_g[k][cell] = cg[k];
      s_g[6][cell] = a1b;
    }
    __syncthreads();
    if (group == 0) {
#pragma unroll
      for (int k = 0; k < 6; ++k) cg[k] = s_g[k][cell];
      pull_back(cb, cg, a1b + s_g[6][cell]);
#pragma unroll
      for (int k = 0; k < 10; ++k) s_p[k][cell] = F[k];
#pragma unroll
      for (int k = 0; k < 3; ++k) s_p[10 + k][cell] = H[k];
      s_a1[cell] = a1;
      s_e[0][cell] = Ef;
      s_e[1][cell] = Eg;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 10; ++k) F[k] = s_p[k][cell];
#pragma unroll
    for (int k = 0; k < 3; ++k) H[k] = s_p[10 + k][cell];
    a1 = s_a1[cell];
    Ef = s_e[0][cell];
    Eg = s_e[1][cell];
  }
  {
    // even and odd parts in x of the inner node pair
    LimbAcc t0, u0, t1, u1, u2, v0;
    rmac<2>(t0, F[3]);
    rmac<1>(u0, F[1]); rmac<3>(u0, F[6]);
    rmac<2>(t1, F[7]);
    rmac<1>(u1, F[4]);
    rmac<1>(u2, F[8]);
    rmac<1>(v0, H[1]);
    const long long eA0 = F[0] + t0.value8(), oA0 = u0.value8(), eA1 = F[2] + t1.value8(), oA1 = u1.value8(),
                    oA2 = u2.value8(), gA = v0.value8();
#pragma unroll 1
    for (int p0 = 0; p0 < 5; p0 += NG > 2 ? NG / 2 : 1) {
      const int p = NG > 2 ? p0 + (group >> 1) : p0;  // as in k_step_tile
      if (NG > 2 && p >= 5) break;
      // y-polynomial of this x-node
      long long b0, b1, b2, g0;
      if (p == 0) {
        b0 = F[0]; b1 = F[2]; b2 = F[5]; g0 = H[0];
      } else {
        const bool inner = p <= 2;
        const long long e0 = inner ? eA0 : F[0] + F[3], o0 = inner ? oA0 : F[1] + F[6], e1 = inner ? eA1 : F[2] + F[7],
                        o1 = inner ? oA1 : F[4], o2 = inner ? oA2 : F[8], og = inner ? gA : H[1];
        const bool neg = (p & 1) == 0;
        b0 = neg ? e0 - o0 : e0 + o0;
        b1 = neg ? e1 - o1 : e1 + o1;
        b2 = neg ? F[5] - o2 : F[5] + o2;
        g0 = neg ? H[0] - og : H[0] + og;
      }
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        if (NG > 1 && k != (group & 1)) continue;
        const double* lp = ltile + (25 * k + 5 * p) * PL;
        double* op = otile + (25 * k + 5 * p) * PL;
        double lv[5];
        long long W[5], t[5];
#pragma unroll
        for (int q = 0; q < 5; ++q) {
          lv[q] = __ldg(at(lp + q * PL, off));
          W[q] = active ? *at((const long long*)op + q * PL, off) : 0ll;
        }
        if (k == 0) {
          LimbAcc ev, od;
          rmac<2>(ev, b2);
          rmac<1>(od, b1); rmac<3>(od, F[9]);
          const long long ea = b0 + ev.value8(), oa = od.value8(), eb = b0 + b2, ob = b1 + F[9];
          t[0] = b0; t[1] = ea + oa; t[2] = ea - oa; t[3] = eb + ob; t[4] = eb - ob;
        } else {
          LimbAcc od;
          rmac<1>(od, H[2]);
          const long long oa = od.value8();
          t[0] = g0; t[1] = g0 + oa; t[2] = g0 - oa; t[3] = g0 + H[2]; t[4] = g0 - H[2];
        }
        const int st = (k == 0 ? Ef : Eg) - 1;
#pragma unroll
        for (int q = 0; q < 5; ++q) {
          const double v = collide_advect(a1, lv[q], t[q], st, W[q], s_exp[25 * k + 5 * p + q] + 3);
          if (active) *at(op + q * PL, off) = v;
        }
      }
    }
  }
  // block reduction of the parameter adjoints (fixed order)
  __syncthreads();
  double* sh = (double*)s_xs;
  const int t = threadIdx.y * 32 + threadIdx.x;
  if (!active || group != 0) pb = {0, 0, 0, 0};
  sh[t] = pb.dt_mu; sh[256 + t] = pb.Pr; sh[512 + t] = pb.gm1; sh[768 + t] = pb.epsf;
  __syncthreads();
  for (int n = 128; n > 0; n >>= 1) {
    if (t < n)
#pragma unroll
      for (int k = 0; k < 4; ++k) sh[256 * k + t] += sh[256 * k + t + n];
    __syncthreads();
  }
  if (t == 0) {
    const int b = blockIdx.y * gridDim.x + blockIdx.x;
#pragma unroll
    for (int k = 0; k < 4; ++k) partial[4 * b + k] = sh[256 * k];
  }
}

// ------------------------------------------------------------------- kernels
// One adjoint step in two launches, with the branches derived from the states: a
// general beta, or no memory for the codes.
// k_adjoint_local: Lout = a1 Lin + sum_j mbar_j dm_j/dX (collision part) at
// state X; per-block sums of the parameter adjoints (dt_mu, Pr, gm1, epsf)
// into partial[blk*4 + k].
template <int PRC>
__global__ void __launch_bounds__(256, 2) k_adjoint_local(const double* __restrict__ X, const double* __restrict__ Lin,
                                                       double* __restrict__ Lout, double* __restrict__ partial,
                                                       Geom G, Phys P) {
  const int x = blockIdx.x * 32 + threadIdx.x;
  const int y = blockIdx.y * 8 + threadIdx.y;
  const bool active = x < G.Nx && y < G.Ny;
  __shared__ long long s_cb[21 * 256];
  const int tid = threadIdx.y * 32 + threadIdx.x;
  ParamBar pb = {0, 0, 0, 0};
  if (active) {
    const long long off = cell_index(G, y, x);
    const double* xs = X + off;
    const double* ls = Lin + off;
    double* lo = Lout + off;
    const long long PL = G.plane;
    Moments m = {};
    Coeffs Cb = {};
    double a1b = 0.0;
    {
      // block exponents of the cell's lambda (f and g) for the fixed-point projection
      int ELf = 0, ELg = 0;
#pragma unroll 5
      for (int c = 0; c < 25; ++c) {
        ELf = max(ELf, bexp(__ldg(ls + c * PL)));
        ELg = max(ELg, bexp(__ldg(ls + (25 + c) * PL)));
      }
      long long* cb = s_cb + tid;
#pragma unroll
      for (int k = 0; k < 21; ++k) cb[k * 256] = 0;
      double f[5], g[5], lf[5], lg[5];
#define DVBM_ADJ_A(p)                                                                  \
      _Pragma("unroll") for (int q = 0; q < 5; ++q) {                                  \
        f[q] = __ldg(xs + (5 * p + q) * PL); g[q] = __ldg(xs + (25 + 5 * p + q) * PL);  \
        lf[q] = __ldg(ls + (5 * p + q) * PL); lg[q] = __ldg(ls + (25 + 5 * p + q) * PL); \
        a1b = fma(lf[q], f[q], fma(lg[q], g[q], a1b));                                \
      }                                                                                \
      accumulate_moments<p>(m, f, g);                                                  \
      accumulate_projection_fix<p>(cb, lf, lg, ELf, ELg);
      DVBM_ADJ_A(0) DVBM_ADJ_A(1) DVBM_ADJ_A(2) DVBM_ADJ_A(3) DVBM_ADJ_A(4)
#undef DVBM_ADJ_A
      const bool okf = ELf >= 100, okg = ELg >= 100;
      const int sf = ELf - 1080, sg = ELg - 1080;
      auto cv = [](bool ok, long long v, int sc) { return ok ? ll_to_double_rn(v, sc) : 0.0; };
      Cb.f00 = cv(okf, cb[0 * 256], sf); Cb.f10 = cv(okf, cb[1 * 256], sf); Cb.f01 = cv(okf, cb[2 * 256], sf);
      Cb.f20 = cv(okf, cb[3 * 256], sf); Cb.f11 = cv(okf, cb[4 * 256], sf); Cb.f02 = cv(okf, cb[5 * 256], sf);
      Cb.f30 = cv(okf, cb[6 * 256], sf); Cb.f21 = cv(okf, cb[7 * 256], sf); Cb.f12 = cv(okf, cb[8 * 256], sf);
      Cb.f03 = cv(okf, cb[9 * 256], sf); Cb.f40 = cv(okf, cb[10 * 256], sf); Cb.f31 = cv(okf, cb[11 * 256], sf);
      Cb.f22 = cv(okf, cb[12 * 256], sf); Cb.f13 = cv(okf, cb[13 * 256], sf); Cb.f04 = cv(okf, cb[14 * 256], sf);
      Cb.g00 = cv(okg, cb[15 * 256], sg); Cb.g10 = cv(okg, cb[16 * 256], sg); Cb.g01 = cv(okg, cb[17 * 256], sg);
      Cb.g20 = cv(okg, cb[18 * 256], sg); Cb.g11 = cv(okg, cb[19 * 256], sg); Cb.g02 = cv(okg, cb[20 * 256], sg);
    }
    Moments mb = {};
    const double a1 = collision_coeffs_rev<PRC>(m, P, Cb, a1b, mb, pb);
#define DVBM_ADJ_B(p)                                                                       \
    {                                                                                       \
      double pf[5], pg[5];                                                                  \
      moment_pullback<p>(mb, pf, pg);                                                       \
      _Pragma("unroll") for (int q = 0; q < 5; ++q) {                                       \
        lo[(5 * p + q) * PL] = fma(a1, __ldg(ls + (5 * p + q) * PL), pf[q]);                \
        lo[(25 + 5 * p + q) * PL] = fma(a1, __ldg(ls + (25 + 5 * p + q) * PL), pg[q]);      \
      }                                                                                     \
    }
    DVBM_ADJ_B(0) DVBM_ADJ_B(1) DVBM_ADJ_B(2) DVBM_ADJ_B(3) DVBM_ADJ_B(4)
#undef DVBM_ADJ_B
  }
  // block reduction of the parameter adjoints (fixed order)
  __shared__ double sh[4][256];
  const int t = threadIdx.y * 32 + threadIdx.x;
  sh[0][t] = pb.dt_mu; sh[1][t] = pb.Pr; sh[2][t] = pb.gm1; sh[3][t] = pb.epsf;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (t < w)
#pragma unroll
      for (int k = 0; k < 4; ++k) sh[k][t] += sh[k][t + w];
    __syncthreads();
  }
  if (t == 0) {
    const int b = blockIdx.y * gridDim.x + blockIdx.x;
#pragma unroll
    for (int k = 0; k < 4; ++k) partial[4 * b + k] = sh[k][0];
  }
}

// k_adjoint_adv: Lout += -(dt/dx) v_x sum_c' Lin(c') dF_x(c')/dX(c) - (same in y),
// one thread per (cell, population); blockIdx.z = population.
template <bool RAT>
__global__ void __launch_bounds__(256) k_adjoint_adv(const double* __restrict__ X, const double* __restrict__ Lin,
                                                     double* __restrict__ Lout, Geom G, Phys P) {
  const int x = blockIdx.x * 32 + threadIdx.x;
  const int y = blockIdx.y * 8 + threadIdx.y;
  const int c = blockIdx.z;
  if (x >= G.Nx || y >= G.Ny) return;
  const int pn = (c % 25) / 5, qn = c % 5;
  const int sx = sgn_of(pn), sy = sgn_of(qn);
  if (sx == 0 && sy == 0) return;
  const long long off = cell_index(G, y, x) + (long long)c * G.plane;
  const double* xc = X + off;
  const double* lc = Lin + off;
  double v = Lout[off];
  if constexpr (RAT) {
    if (sx != 0) v = fma(-P.kxr[pn], advection_adjoint_rat(xc, lc, 1, P.lp, P.lq, sx), v);
    if (sy != 0) v = fma(-P.kyr[qn], advection_adjoint_rat(xc, lc, G.pitch, P.lp, P.lq, sy), v);
  } else {
    if (sx != 0) v = fma(-P.kxv[pn], advection_adjoint(xc, lc, 1, P.hq, sx), v);
    if (sy != 0) v = fma(-P.kyv[qn], advection_adjoint(xc, lc, G.pitch, P.hq, sy), v);
  }
  Lout[off] = v;
}

// lambda^N from dL/drho and dL/dT of the final state; partial: gm1 adjoint
__global__ void __launch_bounds__(256) k_adjoint_final(const double* __restrict__ X, const double* __restrict__ rhob,
                                                       const double* __restrict__ Tb, double* __restrict__ Lout,
                                                       double* __restrict__ partial, Geom G, Phys P, Macro M) {
  const int x = blockIdx.x * 32 + threadIdx.x;
  const int y = blockIdx.y * 8 + threadIdx.y;
  const bool active = x < G.Nx && y < G.Ny;
  ParamBar pb = {0, 0, 0, 0};
  if (active) {
    const long long off = cell_index(G, y, x);
    const long long i = (long long)y * G.Nx + x;
    const Moments m = cell_moments<double>(X + off, G.plane, P);
    Moments mb = {};
    macro_rev(m, P, M.T_ref, rhob ? rhob[i] : 0.0, Tb ? Tb[i] : 0.0, mb, pb);
#define DVBM_FIN(p)                                                          \
    {                                                                        \
      double pf[5], pg[5];                                                   \
      moment_pullback<p>(mb, pf, pg);                                        \
      _Pragma("unroll") for (int q = 0; q < 5; ++q) {                        \
        Lout[off + (5 * p + q) * G.plane] = pf[q];                           \
        Lout[off + (25 + 5 * p + q) * G.plane] = pg[q];                      \
      }                                                                      \
    }
    DVBM_FIN(0) DVBM_FIN(1) DVBM_FIN(2) DVBM_FIN(3) DVBM_FIN(4)
#undef DVBM_FIN
  }
  __shared__ double sh[256];
  const int t = threadIdx.y * 32 + threadIdx.x;
  sh[t] = pb.gm1;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (t < w) sh[t] += sh[t + w];
    __syncthreads();
  }
  if (t == 0) partial[blockIdx.y * gridDim.x + blockIdx.x] = sh[0];
}

// adjoint of the equilibrium initial condition: per-cell dL/d(rho0, ux0, uy0, T0)
// and per-block epsf adjoints
__global__ void __launch_bounds__(256) k_adjoint_init(const double* __restrict__ L, const double* __restrict__ rho,
                                                      const double* __restrict__ ux, const double* __restrict__ uy,
                                                      const double* __restrict__ T, double* grho, double* gux,
                                                      double* guy, double* gT, double* __restrict__ partial, Geom G,
                                                      Phys P, Macro M) {
  const int x = blockIdx.x * 32 + threadIdx.x;
  const int y = blockIdx.y * 8 + threadIdx.y;
  const bool active = x < G.Nx && y < G.Ny;
  double epsfb = 0.0;
  if (active) {
    const long long off = cell_index(G, y, x);
    const long long i = (long long)y * G.Nx + x;
    Coeffs Cb = {};
    {
      double lf[5], lg[5];
#define DVBM_INI(p)                                                         \
      _Pragma("unroll") for (int q = 0; q < 5; ++q) {                       \
        lf[q] = L[off + (5 * p + q) * G.plane];                             \
        lg[q] = L[off + (25 + 5 * p + q) * G.plane];                        \
      }                                                                     \
      accumulate_projection<p>(Cb, lf, lg);
      DVBM_INI(0) DVBM_INI(1) DVBM_INI(2) DVBM_INI(3) DVBM_INI(4)
#undef DVBM_INI
    }
    double rb, ub, vb, thb;
    equilibrium_rev(rho[i], ux[i] / M.c, uy[i] / M.c, T[i] / M.T_ref, P, Cb, rb, ub, vb, thb, epsfb);
    grho[i] = rb;
    gux[i] = ub / M.c;
    guy[i] = vb / M.c;
    gT[i] = thb / M.T_ref;
  }
  __shared__ double sh[256];
  const int t = threadIdx.y * 32 + threadIdx.x;
  sh[t] = epsfb;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (t < w) sh[t] += sh[t + w];
    __syncthreads();
  }
  if (t == 0) partial[blockIdx.y * gridDim.x + blockIdx.x] = sh[0];
}

// ------------------------------------------------------------------ wrappers
// partial-sum slots of a launch: the coded step's blocks, at least those of the 8-row kernels
int adjoint_blocks(const Geom& G) {
  const int R = adjoint_tile_rows(G);
  return ((G.Nx + 31) / 32) * ((G.Ny + R - 1) / R);
}

// Branch-code rows next to a band's edges: unpack = 0 copies rows y = 0 (to
// lo) and y = Ny - 1 (to hi) of every population's codes, unpack = 1 copies
// lo and hi into the ghost code rows glo, ghi; layouts [NPOP][Nx] bytes; a
// NULL buffer skips its side.
__global__ void k_code_rows(unsigned char* __restrict__ codes, unsigned char* __restrict__ lo,
                            unsigned char* __restrict__ hi, unsigned char* __restrict__ glo,
                            unsigned char* __restrict__ ghi, int unpack, int Nx, int Ny) {
  const long long n = (long long)NPOP * Nx;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const long long c = i / Nx, x = i % Nx;
    if (unpack) {
      if (lo) glo[i] = lo[i];
      if (hi) ghi[i] = hi[i];
    } else {
      if (lo) lo[i] = codes[(c * Ny) * Nx + x];
      if (hi) hi[i] = codes[(c * Ny + Ny - 1) * Nx + x];
    }
  }
}

cudaError_t launch_code_rows(unsigned char* codes, void* lo, void* hi, unsigned char* glo, unsigned char* ghi,
                             int unpack, const Geom& G, cudaStream_t st) {
  const long long n = (long long)NPOP * G.Nx;
  const int blocks = (int)std::min<long long>((n + 255) / 256, 4096);
  k_code_rows<<<blocks, 256, 0, st>>>(codes, (unsigned char*)lo, (unsigned char*)hi, glo, ghi, unpack, G.Nx, G.Ny);
  return cudaGetLastError();
}

template <int R>
static void launch_adjoint_tile(const double* X, const double* Lin, double* Lout, double* partial,
                                const unsigned char* codes, const double* moms, const unsigned char* glo,
                                const unsigned char* ghi, const Geom& G, const Phys& P, cudaStream_t st) {
  const dim3 b(32, 8), g((G.Nx + 31) / 32, (G.Ny + R - 1) / R);
  if (P.prc < 0) k_adjoint_tile<R, -1><<<g, b, 0, st>>>(X, Lin, Lout, partial, codes, moms, glo, ghi, G, P);
  else if (P.prc > 0) k_adjoint_tile<R, 1><<<g, b, 0, st>>>(X, Lin, Lout, partial, codes, moms, glo, ghi, G, P);
  else k_adjoint_tile<R, 0><<<g, b, 0, st>>>(X, Lin, Lout, partial, codes, moms, glo, ghi, G, P);
}

cudaError_t launch_adjoint_step(const double* X, const double* Lin, double* Lout, double* partial,
                                const unsigned char* codes, const double* moms, const Geom& G, const Phys& P,
                                cudaStream_t st, const unsigned char* glo, const unsigned char* ghi) {
  dim3 block(32, 8), grid((G.Nx + 31) / 32, (G.Ny + 7) / 8);
  if (codes) {
    const int R = adjoint_tile_rows(G);
    if (R == 8) launch_adjoint_tile<8>(X, Lin, Lout, partial, codes, moms, glo, ghi, G, P, st);
    else if (R == 4) launch_adjoint_tile<4>(X, Lin, Lout, partial, codes, moms, glo, ghi, G, P, st);
    else launch_adjoint_tile<2>(X, Lin, Lout, partial, codes, moms, glo, ghi, G, P, st);
    return cudaGetLastError();
  }
  if (P.prc < 0) k_adjoint_local<-1><<<grid, block, 0, st>>>(X, Lin, Lout, partial, G, P);
  else if (P.prc > 0) k_adjoint_local<1><<<grid, block, 0, st>>>(X, Lin, Lout, partial, G, P);
  else k_adjoint_local<0><<<grid, block, 0, st>>>(X, Lin, Lout, partial, G, P);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const dim3 grid3(grid.x, grid.y, NPOP);
  if (P.lq > 0) k_adjoint_adv<true><<<grid3, block, 0, st>>>(X, Lin, Lout, G, P);
  else k_adjoint_adv<false><<<grid3, block, 0, st>>>(X, Lin, Lout, G, P);
  return cudaGetLastError();
}

cudaError_t launch_adjoint_final(const double* X, const double* rhob, const double* Tb, double* Lout, double* partial,
                                 const Geom& G, const Phys& P, const Macro& M, cudaStream_t st) {
  dim3 block(32, 8), grid((G.Nx + 31) / 32, (G.Ny + 7) / 8);
  k_adjoint_final<<<grid, block, 0, st>>>(X, rhob, Tb, Lout, partial, G, P, M);
  return cudaGetLastError();
}

cudaError_t launch_adjoint_init(const double* L, const double* rho, const double* ux, const double* uy,
                                const double* T, double* grho, double* gux, double* guy, double* gT, double* partial,
                                const Geom& G, const Phys& P, const Macro& M, cudaStream_t st) {
  dim3 block(32, 8), grid((G.Nx + 31) / 32, (G.Ny + 7) / 8);
  k_adjoint_init<<<grid, block, 0, st>>>(L, rho, ux, uy, T, grho, gux, guy, gT, partial, G, P, M);
  return cudaGetLastError();
}

}  // namespace dvbm
