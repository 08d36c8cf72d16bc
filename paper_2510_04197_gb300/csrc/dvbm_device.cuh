// dvbm_device.cuh -- device-side building blocks of the GB300 DVBM step.
//
// Model: double-distribution quasi-equilibrium BGK on the D2Q25 Gauss--Hermite
// lattice, internal non-translational energy split (II).  Everything here is
// written in units of c = sqrt(R T_ref): xi = v / c, theta = T / T_ref,
// Hermite coefficients A_ab = a_{x^a y^b} / c^(a+b), so that the Grad
// expansion (Sec. II.D.2, Eq. Grad_g; App. D) factorises into 1-D
// probabilists' Hermite polynomials:
//     F_pq = W_p W_q sum_{a+b<=N} A_ab He_a(xi_p) He_b(xi_q) / (a! b!).
#pragma once
#include <cstdint>
#include <type_traits>
#include <cuda_runtime.h>

namespace dvbm {

// ---- D2Q25 lattice (App. G): 1-D nodes are the roots of He_5 ---------------
// node k: 0, +sqrt(5 - sqrt 10), -sqrt(5 - sqrt 10), +sqrt(5 + sqrt 10), -sqrt(5 + sqrt 10)
constexpr double XA = 1.3556261799742659;   // sqrt(5 - sqrt(10))
constexpr double XB = 2.8569700138728056;   // sqrt(5 + sqrt(10))
// 1-D Gauss--Hermite weights: 8/15 and (7 +- 2 sqrt 10)/60
constexpr double W0 = 0.53333333333333333;  // 8/15
constexpr double WA = 0.22207592200561264;  // (7 + 2 sqrt(10)) / 60
constexpr double WB = 0.011257411327720689; // (7 - 2 sqrt(10)) / 60

constexpr int Q = 25;
constexpr int NPOP = 50;  // f (0..24) and g (25..49); population c = 5 p + q

__host__ __device__ constexpr double xi_of(int k) {
  return k == 0 ? 0.0 : k == 1 ? XA : k == 2 ? -XA : k == 3 ? XB : -XB;
}
__host__ __device__ constexpr double w_of(int k) {
  return k == 0 ? W0 : (k <= 2 ? WA : WB);
}
__host__ __device__ constexpr int sgn_of(int k) { return k == 0 ? 0 : (k == 1 || k == 3) ? 1 : -1; }
// probabilists' Hermite polynomials He_n(x), n <= 4
__host__ __device__ constexpr double he(int n, double x) {
  return n == 0 ? 1.0 : n == 1 ? x : n == 2 ? x * x - 1.0 : n == 3 ? x * x * x - 3.0 * x
                                                                      : x * x * x * x - 6.0 * x * x + 3.0;
}
__host__ __device__ constexpr double inv_fact(int n) {
  return n == 0 ? 1.0 : n == 1 ? 1.0 : n == 2 ? 0.5 : n == 3 ? 1.0 / 6.0 : 1.0 / 24.0;
}
// W_k He_n(xi_k) / n!
__host__ __device__ constexpr double kh(int k, int n) { return w_of(k) * he(n, xi_of(k)) * inv_fact(n); }

// ---- launch-invariant parameters (passed by value, constant bank) ---------
struct Geom {
  int Nx, Ny;
  int pitch;             // elements per row (ghost columns included)
  int xoff;              // element offset of x = 0 inside a row
  long long plane;       // elements per population plane = (Ny + 4) * pitch
  int grid_rows;         // rows of the whole grid (Ny, or more for a band of it): fixes the tile heights
};

struct Phys {
  double c2, inv_c2;     // R T_ref and 1 / (R T_ref)
  double gm1;            // gamma - 1 = R / C_v
  double epsf;           // C_v/R - D/2 = (2 - gamma)/(gamma - 1): eps/(R T) of split II
  double dt, mu, Pr;
  double dt_mu;          // dt / mu
  int prc;               // -1: Pr < 1, 0: Pr == 1, +1: Pr > 1
  double hb;             // beta / 2
  long long hq;          // round(beta/2 * 2^62), integer-pipe limiter (general beta)
  int lp, lq;            // beta = lp / lq exactly (lq <= 64), or lq = 0: use hq
  double kxr[5], kyr[5]; // kxv / (4 lq), kyv / (4 lq): flux factors of the scaled differences
  double kxv[5], kyv[5]; // dt/dx * c * xi_k and dt/dy * c * xi_k
  float kxvf[5], kyvf[5];
  // tile advection of FP64 storage: |kxv|, |kyv| as 2^60-fractions with the
  // limiter's scale folded in (times 2^L / lq, L = ceil(log2 lq); lq counts as 1
  // for a general beta), and the values' extra shift 1 + L below 60 bits
  long long kxq[5], kyq[5];
  int advn;
  double fref0, gref0;   // FP32DEV reference: f_ref = w rho0, g_ref = w rho0 (C_v - R) T0
  double rho_ref_mom;    // unused padding for alignment
};

__device__ __forceinline__ long long cell_index(const Geom& G, int y, int x) {
  return (long long)(y + 2) * G.pitch + x + G.xoff;
}

// ---- macroscopic state and collision coefficients -------------------------
// Raw dimensionless moments of f (mu_ab = sum_i xi_x^a xi_y^b f_i, a + b <= 3)
// and of g (physical units: G00 = sum g, G10/G01 = sum xi g).
struct Moments {
  double m00, m10, m01, m20, m11, m02, m30, m21, m12, m03;
  double g00, g10, g01;
};

// Combined expansion coefficients of one collision:
//   F_new = a1 F + W W sum C_ab He He/(a! b!) - advection,
// with C = (dt/tau1) A^eq + (dt/tau1 - dt/tau2) (A* - A^eq), which equals
// F - (dt/tau1)(F - F*) - (dt/tau2)(F* - F^eq) by linearity of the expansion.
struct Coeffs {
  double f00, f10, f01, f20, f11, f02, f30, f21, f12, f03, f40, f31, f22, f13, f04;
  double g00, g10, g01, g20, g11, g02;  // physical units of g
  double a1;                            // 1 - dt/tau1
  double k1;                            // dt/tau1
  bool bad;                             // rho <= 0, theta <= 0 or not finite
};

// Equilibrium coefficients of f (App. D theta-form) for rho, u (in units of
// c) and s = theta - 1, via the 1-D Hermite recurrences
//   A_{n+1} = u A_n + n s A_{n-1} along each axis.
struct EqF { double a00, a10, a01, a20, a11, a02, a30, a21, a12, a03, a40, a31, a22, a13, a04; };

__device__ __forceinline__ EqF eq_f(double rho, double ux, double uy, double s) {
  EqF e;
  double rs = rho * s;
  e.a00 = rho;
  e.a10 = rho * ux;
  e.a01 = rho * uy;
  e.a20 = fma(e.a10, ux, rs);
  e.a11 = e.a10 * uy;
  e.a02 = fma(e.a01, uy, rs);
  const double rs2 = rs + rs;
  e.a30 = ux * (e.a20 + rs2);
  e.a03 = uy * (e.a02 + rs2);
  e.a21 = e.a20 * uy;
  e.a12 = e.a02 * ux;
  e.a40 = fma(e.a30, ux, 3.0 * s * e.a20);
  e.a04 = fma(e.a03, uy, 3.0 * s * e.a02);
  e.a31 = e.a30 * uy;
  e.a13 = e.a03 * ux;
  e.a22 = e.a20 * fma(uy, uy, s);
  return e;
}

// 1/x with one Halley step from the single-precision reciprocal: relative error
// e = 1 - x r of about 2^-23 becomes e^3 plus rounding (three FP64 instructions;
// the compiler's division takes about three times as many).  Outside the
// single-precision range, and for non-finite x, the plain division.
__device__ __forceinline__ double recip(double x) {
  const unsigned ex = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
  if (ex - 903u >= 240u) return 1.0 / x;  // |x| outside [2^-120, 2^120)
  // x rounded down to 24 bits as a float, and back, by bit manipulation (the
  // hardware conversions run at the FP64 rate)
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const float f = __uint_as_float((hi & 0x80000000u) | (((hi & 0x7fffffffu) - (896u << 20)) << 3) | (lo >> 29));
  const unsigned u = __float_as_uint(__frcp_rn(f));
  const double r = __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))), (int)(u << 29));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// v > 0 (true for +inf, false for NaN) and |v| < 1e300 (false for NaN) on the bit
// patterns: a comparison of doubles takes a slot of the FP64 pipe
__device__ __forceinline__ bool is_positive(double v) {
  return (unsigned long long)__double_as_longlong(v) - 1ull < 0x7ff0000000000000ull;
}
__device__ __forceinline__ bool is_bounded(double v) {
  return (__double_as_longlong(v) & 0x7fffffffffffffffll) < 0x7e37e43c8800759cll;
}

// Collision coefficients from the moments (Sec. II.C relaxation times,
// Table I split-II quasi-equilibria).  PRC selects the Prandtl case at
// compile time: -1 (Pr < 1), 0 (Pr = 1), +1 (Pr > 1).
//   Pr < 1: A*_3 = H_3(f) - S(u, Delta); A*_g1 = sum xi g; else equilibrium.
//   Pr > 1: A*_2 = A^eq_2 + Delta', A*_3 = A^eq_3 + S(u, Delta'),
//           A*_4 = A^eq_4 - [Delta' delta]_cyc; g* = g^eq,
// with Delta = H_2(f) - A^eq_2, Delta' its traceless part and
// S(u, A)_abc = [u_a A_bc]_cyc - tr(A)/(D+2) [u_a d_bc]_cyc, the symmetric
// tensor whose contraction is the heat-flux constraint 2 (A u)_a.
// FP64 work is what bounds this function's kernels, so k1 = dt/tau1 enters at
// the zeroth coefficient and runs through the equilibrium recurrences, and
// k1 A^eq + s1 (A* - A^eq) is written k1 A* + k2 (A^eq - A*) with k2 = Pr k1
// (Pr <= 1) or s1 = k1 - k2 on the deviations alone (Pr > 1): 84 FP64
// instructions instead of 114.
template <int PRC>
__device__ __forceinline__ Coeffs collision_coeffs(const Moments& m, const Phys& P) {
  Coeffs C;
  const double rho = m.m00;
  const double irho = recip(rho);
  const double ux = m.m10 * irho, uy = m.m01 * irho;
  const double Et = fma(0.5, m.m20 + m.m02, m.g00 * P.inv_c2);        // E / c^2
  const double theta = P.gm1 * fma(-0.5, fma(ux, ux, uy * uy), Et * irho);
  const double s = theta - 1.0;
  C.bad = !is_positive(rho) || !is_positive(theta) || !is_bounded(Et);
  const double rt = rho * theta;                                         // p / c^2
  const double kp = (P.dt_mu * P.c2) * rt;                               // dt p / mu
  const double k1 = PRC <= 0 ? kp : kp * P.Pr;                           // dt/tau1
  C.a1 = 1.0 - k1;
  C.k1 = k1;
  const EqF e = eq_f(k1 * rho, ux, uy, s);                               // k1 A^eq
  C.f00 = e.a00; C.f10 = e.a10; C.f01 = e.a01;
  C.f20 = e.a20; C.f11 = e.a11; C.f02 = e.a02;
  C.f30 = e.a30; C.f21 = e.a21; C.f12 = e.a12; C.f03 = e.a03;
  C.f40 = e.a40; C.f31 = e.a31; C.f22 = e.a22; C.f13 = e.a13; C.f04 = e.a04;
  // k1 A^eq of g (split II, physical units): rho eps (1, u, uu + s I)
  const double kr = e.a00 * (theta * (P.epsf * P.c2));
  const double krx = kr * ux, kry = kr * uy, krs = kr * s;
  C.g00 = kr;
  C.g10 = krx;
  C.g01 = kry;
  C.g20 = fma(krx, ux, krs);
  C.g11 = krx * uy;
  C.g02 = fma(kry, uy, krs);
  if (PRC != 0) {
    // Delta = H_2(f) - A^eq_2: mu_20 - rho theta - rho ux^2, mu_11 - rho ux uy, ...
    const double Dxx = fma(-m.m10, ux, m.m20 - rt);
    const double Dxy = fma(-m.m10, uy, m.m11);
    const double Dyy = fma(-m.m01, uy, m.m02 - rt);
    if (PRC < 0) {
      const double s1 = fma(-P.Pr, k1, k1);                             // dt/tau1 - dt/tau2
      const double kap = 0.25 * (Dxx + Dyy);                            // tr(Delta)/(D+2)
      const double Px = Dxx - kap, Py = Dyy - kap;
      // A*_3 = H_3(f) - S(u, Delta); H_3: mu_30 - 3 mu_10, mu_21 - mu_01, mu_12 - mu_10, mu_03 - 3 mu_01
      const double x30 = fma(-3.0 * ux, Px, fma(-3.0, m.m10, m.m30));
      const double x21 = fma(-2.0 * ux, Dxy, fma(-uy, Px, m.m21 - m.m01));
      const double x12 = fma(-2.0 * uy, Dxy, fma(-ux, Py, m.m12 - m.m10));
      const double x03 = fma(-3.0 * uy, Py, fma(-3.0, m.m01, m.m03));
      C.f30 = fma(s1, x30, P.Pr * C.f30);
      C.f21 = fma(s1, x21, P.Pr * C.f21);
      C.f12 = fma(s1, x12, P.Pr * C.f12);
      C.f03 = fma(s1, x03, P.Pr * C.f03);
      // g*: first moment of g
      C.g10 = fma(s1, m.g10, P.Pr * krx);
      C.g01 = fma(s1, m.g01, P.Pr * kry);
    } else {
      const double s1 = k1 - kp;
      const double tx = s1 * (0.5 * (Dxx - Dyy));                       // s1 Delta'_xx = -s1 Delta'_yy
      const double ty = s1 * Dxy;
      C.f20 += tx; C.f11 += ty; C.f02 -= tx;
      C.f30 = fma(3.0 * ux, tx, C.f30);
      C.f21 = fma(uy, tx, fma(2.0 * ux, ty, C.f21));
      C.f12 = fma(-ux, tx, fma(2.0 * uy, ty, C.f12));
      C.f03 = fma(-3.0 * uy, tx, C.f03);
      C.f40 = fma(-6.0, tx, C.f40); C.f31 = fma(-3.0, ty, C.f31);
      C.f13 = fma(-3.0, ty, C.f13); C.f04 = fma(6.0, tx, C.f04);
    }
  }
  return C;
}

// Pure equilibrium coefficients (for initial conditions and wall ghosts):
// same layout as Coeffs with C = A^eq, physical g.
__device__ __forceinline__ Coeffs equilibrium_coeffs(double rho, double ux, double uy, double theta,
                                                     const Phys& P) {
  Coeffs C;
  const double s = theta - 1.0;
  EqF e = eq_f(rho, ux, uy, s);
  C.f00 = e.a00; C.f10 = e.a10; C.f01 = e.a01; C.f20 = e.a20; C.f11 = e.a11; C.f02 = e.a02;
  C.f30 = e.a30; C.f21 = e.a21; C.f12 = e.a12; C.f03 = e.a03;
  C.f40 = e.a40; C.f31 = e.a31; C.f22 = e.a22; C.f13 = e.a13; C.f04 = e.a04;
  const double reps = rho * P.epsf * theta * P.c2;
  C.g00 = reps; C.g10 = reps * ux; C.g01 = reps * uy;
  C.g20 = reps * fma(ux, ux, s); C.g11 = reps * ux * uy; C.g02 = reps * fma(uy, uy, s);
  C.a1 = 0.0; C.k1 = 1.0; C.bad = false;
  return C;
}

// Macroscopic values (rho, u in physical units, T) from moments.
__device__ __forceinline__ void macro_from_moments(const Moments& m, const Phys& P, double c, double T_ref,
                                                   double& rho, double& ux, double& uy, double& T) {
  rho = m.m00;
  const double irho = 1.0 / rho;
  const double uxd = m.m10 * irho, uyd = m.m01 * irho;
  const double Et = fma(0.5, m.m20 + m.m02, m.g00 * P.inv_c2);
  const double theta = P.gm1 * fma(-0.5, fma(uxd, uxd, uyd * uyd), Et * irho);
  ux = uxd * c;
  uy = uyd * c;
  T = theta * T_ref;
}

// ---- sum-factorised moment accumulation -----------------------------------
// Accumulate the contribution of the five populations (p, q = 0..4) of one
// x-node p.  f[q] and g[q] are the values (double).
template <int p>
__device__ __forceinline__ void accumulate_moments(Moments& m, const double (&f)[5], const double (&g)[5]) {
  const double sA = f[1] + f[2], dA = f[1] - f[2], sB = f[3] + f[4], dB = f[3] - f[4];
  const double m0 = f[0] + sA + sB;
  const double m1 = fma(XA, dA, XB * dB);
  const double m2 = fma(XA * XA, sA, (XB * XB) * sB);
  const double m3 = fma(XA * XA * XA, dA, (XB * XB * XB) * dB);
  const double n0 = g[0] + (g[1] + g[2]) + (g[3] + g[4]);
  const double n1 = fma(XA, g[1] - g[2], XB * (g[3] - g[4]));
  m.m00 += m0; m.m01 += m1; m.m02 += m2; m.m03 += m3;
  m.g00 += n0; m.g01 += n1;
  if (p != 0) {
    constexpr double x = xi_of(p);
    m.m10 = fma(x, m0, m.m10);
    m.m11 = fma(x, m1, m.m11);
    m.m12 = fma(x, m2, m.m12);
    m.m20 = fma(x * x, m0, m.m20);
    m.m21 = fma(x * x, m1, m.m21);
    m.m30 = fma(x * x * x, m0, m.m30);
    m.g10 = fma(x, n0, m.g10);
  }
}

// ---- limited slope of the NND reconstruction (Sec. III.A.2) --------------
// sigma(a, b) = (b/2) phi(a/b) = 1/2 minmod3(beta a, (a+b)/2, beta b)
//             = minmod3(hb a, (a+b)/4, hb b),  hb = beta/2,
// (division-free; 0 if a and b differ in sign; b = 0 gives 0).  This float
// form serves the FP32-deviation storage; FP64 storage runs the same limiter
// exactly on integers (below).
__device__ __forceinline__ float limited_slope(float a, float b, float hb) {
  const float x = hb * a, z = hb * b, y = 0.25f * (a + b);
  const float mn = fminf(fminf(fabsf(x), fabsf(y)), fabsf(z));
  return ((__float_as_int(a) ^ __float_as_int(b)) >= 0) ? copysignf(mn, a) : 0.0f;
}

// ---- FP64 advection in block floating point on the integer pipe ----------
// GB300 runs FP64 at 1/64 of the FP32 rate, while integer ops are cheap.  The
// four values of one upwind stencil are brought to their largest exponent E
// as 60-bit integers X = M 2^(e - E + 7) (M the 53-bit significand), so that
// differences, the beta/2 scaling, the minmod selection and the flux
// difference are exact integer arithmetic (truncation only below 2^-60 of the
// largest value); only the result is converted back to double.  The
// conversions are pure bit manipulation.
__device__ __forceinline__ int bexp(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// Zero (and subnormal) inputs need no special case: their shift E - e is 63
// whenever E >= 61, which leaves 0; every caller treats E < 64 as "all values
// negligible" and returns 0 before using the result.
__device__ __forceinline__ long long to_block_fixed(double v, int E) {
  const int hi = __double2hiint(v);
  const unsigned lo = (unsigned)__double2loint(v);
  const int e = (hi >> 20) & 0x7ff;
  const unsigned long long m = ((unsigned long long)((unsigned)(hi & 0xfffff) | 0x100000u) << 32) | lo;
  const unsigned long long mag = (m << 7) >> min(E - e, 63);
  return hi < 0 ? -(long long)mag : (long long)mag;
}

// int64 -> double by bit manipulation (the hardware conversion runs at the FP64
// rate on GB300): |F| is normalised with a count of leading zeros, its top 53
// bits become the significand (truncating the rest, < 2^-52 relative), and
// the exponent is that of F times 2^scale.  F = 0 gives 0.
__device__ __forceinline__ double ll_to_double_scaled(long long F, int scale) {
  if (F == 0) return 0.0;
  const unsigned long long mag = F < 0 ? (unsigned long long)(-F) : (unsigned long long)F;
  const int lz = __clzll(mag);
  const unsigned long long norm = mag << lz;           // leading one at bit 63
  const unsigned long long frac = (norm >> 11) & 0x000fffffffffffffull;
  const int ex = 1023 + 63 - lz + scale;
  const unsigned hi = (unsigned)(frac >> 32) | ((unsigned)ex << 20) | (F < 0 ? 0x80000000u : 0u);
  return __hiloint2double((int)hi, (int)(unsigned)frac);
}

// ---- fixed-point Grad expansion (FP64 storage) ----------------------------
// The expansion t = W W sum C He He /(a! b!) is a fixed linear map of the
// collision coefficients.  On GB300 the FP64 pipe (2 ops / clock / SM) is the
// bottleneck of the step, so the expansion runs in block fixed point on the
// integer pipe: the coefficients of one cell share an exponent (f and g
// separately) as 60-bit integers, the node constants kh(k, n) (all |kh| < 0.54)
// are fractions scaled per node to 62-63 bits (kh(k, n) 2^(63 + kd(k)); the
// outer nodes carry the small weight W_B and gain four bits), each product is
// the high word of the 128-bit product, and the h values of each x-node are
// renormalised to 60 bits before the y-expansion.  Truncation stays below
// 2^-56 of the largest term at each stage; the result is rounded to nearest
// when it goes back to double, so the collision target carries no
// systematic bias into the conserved sums.
__host__ __device__ constexpr int kd(int k) { return k == 0 ? 0 : (k <= 2 ? 1 : 4); }
// int64 -> double rounded to nearest (ties away from zero), value F 2^scale
__device__ __forceinline__ double ll_to_double_rn(long long F, int scale) {
  if (F == 0) return 0.0;
  const unsigned long long mag = F < 0 ? (unsigned long long)(-F) : (unsigned long long)F;
  const int lz = __clzll(mag);
  const unsigned long long norm = mag << lz;                     // leading one at bit 63
  const unsigned long long r = (norm >> 11) + ((norm >> 10) & 1ull);  // 53 or 54 bits after rounding
  const int carry = (int)(r >> 53);                               // rounding reached 2^53
  const unsigned long long frac = (r >> carry) & 0x000fffffffffffffull;
  const int ex = 1023 + 63 - lz + scale + carry;
  const unsigned hi = (unsigned)(frac >> 32) | ((unsigned)ex << 20) | (F < 0 ? 0x80000000u : 0u);
  return __hiloint2double((int)hi, (int)(unsigned)frac);
}

// address of a warp-uniform pointer plus a lane's 32-bit byte offset
template <class T>
__device__ __forceinline__ T* at(T* base, unsigned off) {
  typedef typename std::conditional<std::is_const<T>::value, const char, char>::type B;
  return (T*)((B*)base + off);
}

// ---- kernels chained by programmatic dependent launch ---------------------------
// The short kernels of a step (tiles below 8 rows, ghost layers, walls) are
// launched while the kernel before them in the stream still runs
// (launch_chained), and wait here until it has completed and its writes are
// visible, which spares 1.3 us of a 64^2 step and 1.7 us of one on 4 x 256 with walls.
// Their own successor is let in after that, so that at most one waits.  p: the
// kernel's input, which later loads then depend on; the data changes after the
// kernel's start, so it is read by plain loads (load), never by the read-only path.
template <class T>
__device__ __forceinline__ T* chain_wait(T* p) {
  asm volatile("griddepcontrol.wait;\n\tgriddepcontrol.launch_dependents;" : "+l"(p) : : "memory");
  return p;
}
// NC: in kernels that are not chained, the read-only path (the 8-row step is 7 %
// slower with plain loads: the compiler keeps them in order with its stores)
template <bool NC>
__device__ __forceinline__ double load(const double* p) {
  if (NC) return __ldg(p);
  double v;
  asm("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}
template <bool NC>
__device__ __forceinline__ float load(const float* p) {
  if (NC) return __ldg(p);
  float v;
  asm("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}

// ---- limb products on the integer multiply-add pipe ------------------------
// A 64-bit by 64-bit high-word product (__mul64hi) runs at 3.8 lanes / clock /
// SM on GB300 (measured; it is built from half-rate 32-bit high multiplies),
// a 32 x 32 + 64-bit multiply-add at 62.  Fixed-point factors are therefore
// kept as two signed 32-bit limbs, x = h 2^32 + l with l in [-2^31, 2^31), and
// a sum of products x_i k_i / 2^64 is three wide multiply-adds per product: the
// high products and the two cross products have an accumulator each, the low
// product (below one unit of the result) is left out.
__host__ __device__ constexpr int limb_lo(long long x) { return (int)(unsigned)(unsigned long long)x; }
__host__ __device__ constexpr int limb_hi(long long x) {
  return (int)((x - (long long)limb_lo(x)) >> 32);
}
struct LimbAcc {
  long long hi = 0, mid = 0;
  __device__ __forceinline__ void mac(int xh, int xl, int kh, int kl) {
    // written as the instruction: a compiler's reassociation splits the sums
    // into separate multiplies and adds
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(hi) : "r"(xh), "r"(kh));
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(mid) : "r"(xh), "r"(kl));
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(mid) : "r"(xl), "r"(kh));
  }
  // the sum / 2^64: rounded to nearest or down, or / 2^61 (down)
  __device__ __forceinline__ long long value() const { return hi + ((mid + 0x80000000ll) >> 32); }
  __device__ __forceinline__ long long floor() const { return hi + (mid >> 32); }
  __device__ __forceinline__ long long value8() const { return (hi << 3) + (mid >> 29); }
};
struct Limbs {
  int h, l;
  __device__ __forceinline__ explicit Limbs(long long x) : h((int)(x >> 32) + (int)((unsigned)x >> 31)), l((int)x) {}
};
// limbs packed into one 64-bit word (high word h, low word l)
__device__ __forceinline__ long long pack_limbs(long long x) { return x + ((x & 0x80000000ll) << 1); }

// ---- block fixed point ------------------------------------------------------
// Exponent key of a double: its high word without the sign, so that the largest
// key of a block has the block's largest exponent in bits 20..30.
__device__ __forceinline__ unsigned abs_key(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }
__device__ __forceinline__ unsigned abs_key(float v) { return __float_as_uint(v) & 0x7fffffffu; }

// How a block of largest exponent E enters fixed point.  Below 2^-895 (E < 128) the
// block is negligible: its integers' units would leave the range of doubles, and an
// integer of one unit scaled below the smallest exponent wraps into numbers near
// 2^1000.  Its values become 0, negative ones -1; Signed keeps them from that (exactly 0
// for either sign) where the result is to be 0.  The forward step's kernels do
// without the mask, which costs a 64^2 step 1.6 % and one on 4 x 256 with walls 2.6 %:
// they scale at least at exponent 128, where a unit is below 1e-285.
template <bool Signed>
struct BlockScaleOf {
  int E, n0, sign;  // exponent, dropped bits (63: all), mask of the values' signs
  __device__ __forceinline__ BlockScaleOf(int E_, int bits, int tiny = 128)
      : E(E_), n0(E_ < tiny ? 63 : bits), sign(Signed && E_ < tiny ? 0 : -1) {}
};
typedef BlockScaleOf<true> BlockScale;
typedef BlockScaleOf<false> FlowScale;
// Value v as an integer of 60 - n0 bits at the block exponent E (n0 >= 0):
// v = X 2^(E - 1082 + n0); magnitudes are truncated, negative values are the
// ones' complement of theirs (one unit more).  A value of larger exponent than
// E (only non-finite ones are left out of the block maximum) gives 0 or -1.
template <bool Signed>
__device__ __forceinline__ long long block_fix(double v, const BlockScaleOf<Signed>& B) {
  const int hi = __double2hiint(v);
  const unsigned lo = (unsigned)__double2loint(v);
  const int e = (hi >> 20) & 0x7ff;
  const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
  const unsigned long long m = (((unsigned long long)mh << 32) | lo) << 7;
  const unsigned n = min((unsigned)(B.E - e + B.n0), 63u);
  return (long long)(m >> n) ^ (long long)((hi >> 31) & B.sign);
}
// the same for a float: v = X 2^(E - 186 + n0)
template <bool Signed>
__device__ __forceinline__ long long block_fix(float v, const BlockScaleOf<Signed>& B) {
  const int u = __float_as_int(v);
  const int e = (u >> 23) & 0xff;
  const unsigned mh = (((unsigned)u & 0x7fffffu) | 0x800000u) << 4;
  const unsigned n = min((unsigned)(B.E - e + B.n0), 63u);
  return (long long)(((unsigned long long)mh << 32) >> n) ^ (long long)((u >> 31) & B.sign);
}

// int64 -> double by bit manipulation, value F 2^scale: one count of leading
// zeros on the word that holds the leading one, rounded to nearest (ties away); a
// negative F counts one unit less in magnitude (see block_fix).  The value's
// exponent must lie in the normal range.
__device__ __forceinline__ double fix_to_double(long long F, int scale) {
  const int s = (int)(F >> 63);
  const unsigned hi = (unsigned)(int)(F >> 32) ^ (unsigned)s, lo = (unsigned)F ^ (unsigned)s;
  const bool low = hi == 0u;
  const unsigned top = low ? lo : hi;
  const int n = __clz((int)top) + (low ? 32 : 0);
  // leading one at bit 62 (|F| < 2^62); a carry out of the rounded significand
  // goes into the exponent below, which is exactly right
  const unsigned long long norm = ((((unsigned long long)hi) << 32) | lo) << ((n - 1) & 63);
  const unsigned long long r = (norm + 0x200u) >> 10;
  const unsigned rh = (unsigned)(r >> 32) + ((unsigned)(1023 + 62 - n + scale) << 20);
  const double v = __hiloint2double((int)(rh | ((unsigned)s & 0x80000000u)), (int)(unsigned)r);
  return top == 0u ? 0.0 : v;
}

// ---- moments in block fixed point -------------------------------------------
// The 13 moments of a cell (Sec. II.D.1) without FP64 arithmetic: on GB300 an
// FP64 instruction takes the issue time of 32 integer ones.  The 25 populations
// of f (of g) are brought to their largest exponent as 58-bit integers
// (truncated below 2^-57 of the largest, finer than the rounding of a double
// sum); sums are exact, and the powers of the abscissae are fixed-point factors
// rounded from their exact values to 2^-62 (factors rounded to double leave a
// drift of a few 1e-17 a step between the moments and the equilibria built from
// them).  A non-finite population makes its family's zeroth moment NaN, which
// the caller's checks see.
// XA^n and XB^n times 2^62 / 4, / 16, / 32 (n = 1, 2, 3)
constexpr long long kXA[4] = {0, 1562930575100362931ll, 529687401272071863ll, 359029054183477437ll};
constexpr long long kXB[4] = {0, 3293862167010879573ll, 2352616360245045577ll, 3360677197683338703ll};
// the weighted sum over the two node pairs, (XB^n b + XA^n a) / 16, / 64, / 128 (n = 1, 2, 3)
template <int n>
__device__ __forceinline__ long long pair_sum(long long b, long long a) {
  const Limbs x(b), y(a);
  LimbAcc s;
  s.mac(x.h, x.l, limb_hi(kXB[n]), limb_lo(kXB[n]));
  s.mac(y.h, y.l, limb_hi(kXA[n]), limb_lo(kXA[n]));
  return s.value();
}

template <class S>
struct FixKind {
  static constexpr int kBias = sizeof(S) == 8 ? 1080 : 184;
  static constexpr int kExpBits = sizeof(S) == 8 ? 20 : 23;
  static constexpr unsigned kInf = sizeof(S) == 8 ? 0x7ff00000u : 0x7f800000u;
  static constexpr int kTiny = sizeof(S) == 8 ? 128 : 0;  // blocks below this exponent count as zero
};
template <class S, bool NC = true>
__device__ __forceinline__ void moments_fix_f(const S* __restrict__ s, unsigned off, long long PL, Moments& m) {
  typedef FixKind<S> K;
  S v[25];
  unsigned key = 0;
#pragma unroll
  for (int i = 0; i < 25; ++i) {
    v[i] = load<NC>(at(s + i * PL, off));
    key = max(key, abs_key(v[i]));
  }
  const int E = (int)(key >> K::kExpBits);
  const FlowScale B(E, 2, K::kTiny);
  long long M0[5], M1[5], M2[5], M3s = 0;  // y-sums of each x-node, M1, M2, M3 times 1/16, 1/64, 1/128
#pragma unroll
  for (int p = 0; p < 5; ++p) {
    const long long x0 = block_fix(v[5 * p], B), x1 = block_fix(v[5 * p + 1], B),
                    x2 = block_fix(v[5 * p + 2], B), x3 = block_fix(v[5 * p + 3], B),
                    x4 = block_fix(v[5 * p + 4], B);
    const long long sA = x1 + x2, dA = x1 - x2, sB = x3 + x4, dB = x3 - x4;
    M0[p] = x0 + sA + sB;
    M1[p] = pair_sum<1>(dB, dA);
    M2[p] = pair_sum<2>(sB, sA);
    M3s += pair_sum<3>(dB, dA);
  }
  const long long a0 = M0[1] + M0[2], b0 = M0[3] + M0[4], c0 = M0[1] - M0[2], d0 = M0[3] - M0[4];
  // second factors: the first left four spare bits
  const long long a1 = M1[1] + M1[2], b1 = M1[3] + M1[4], c1 = M1[1] - M1[2], d1 = M1[3] - M1[4];
  const long long a2 = M2[1] + M2[2], b2 = M2[3] + M2[4], c2 = M2[1] - M2[2], d2 = M2[3] - M2[4];
  const int sc = max(E, K::kTiny) - K::kBias;
  m.m00 = fix_to_double(M0[0] + a0 + b0, sc);
  m.m01 = fix_to_double(M1[0] + a1 + b1, sc + 4);
  m.m02 = fix_to_double(M2[0] + a2 + b2, sc + 6);
  m.m03 = fix_to_double(M3s, sc + 7);
  m.m10 = fix_to_double(pair_sum<1>(d0, c0), sc + 4);
  m.m20 = fix_to_double(pair_sum<2>(b0, a0), sc + 6);
  m.m30 = fix_to_double(pair_sum<3>(d0, c0), sc + 7);
  m.m11 = fix_to_double(pair_sum<1>(d1 << 4, c1 << 4), sc + 4);
  m.m21 = fix_to_double(pair_sum<2>(b1 << 4, a1 << 4), sc + 6);
  m.m12 = fix_to_double(pair_sum<1>(d2 << 4, c2 << 4), sc + 6);
  if (key >= K::kInf) m.m00 = __longlong_as_double(0x7ff8000000000000ll);
}
template <class S, bool NC = true>
__device__ __forceinline__ void moments_fix_g(const S* __restrict__ s, unsigned off, long long PL, Moments& m) {
  typedef FixKind<S> K;
  S v[25];
  unsigned key = 0;
#pragma unroll
  for (int i = 0; i < 25; ++i) {
    v[i] = load<NC>(at(s + (25 + i) * PL, off));
    key = max(key, abs_key(v[i]));
  }
  const int E = (int)(key >> K::kExpBits);
  const FlowScale B(E, 2, K::kTiny);
  long long N0[5], N1s = 0;
#pragma unroll
  for (int p = 0; p < 5; ++p) {
    const long long x0 = block_fix(v[5 * p], B), x1 = block_fix(v[5 * p + 1], B),
                    x2 = block_fix(v[5 * p + 2], B), x3 = block_fix(v[5 * p + 3], B),
                    x4 = block_fix(v[5 * p + 4], B);
    N0[p] = x0 + (x1 + x2) + (x3 + x4);
    N1s += pair_sum<1>(x3 - x4, x1 - x2);
  }
  const int sc = max(E, K::kTiny) - K::kBias;
  m.g00 = fix_to_double(N0[0] + (N0[1] + N0[2]) + (N0[3] + N0[4]), sc);
  m.g01 = fix_to_double(N1s, sc + 4);
  m.g10 = fix_to_double(pair_sum<1>(N0[3] - N0[4], N0[1] - N0[2]), sc + 4);
  if (key >= K::kInf) m.g00 = __longlong_as_double(0x7ff8000000000000ll);
}
template <class S>
__device__ __forceinline__ Moments moments_fix(const S* __restrict__ s, unsigned off, long long PL) {
  Moments m;
  moments_fix_f<S>(s, off, PL, m);
  moments_fix_g<S>(s, off, PL, m);
  return m;
}
// moments of the FP32-deviation reference populations w rho0 (f) and w G0 (g):
// sum w = 1, sum w xi^2 = 1 per axis, odd moments vanish
__device__ __forceinline__ void add_reference_f(Moments& m, const Phys& P) {
  m.m00 += P.fref0; m.m20 += P.fref0; m.m02 += P.fref0;
}
__device__ __forceinline__ void add_reference(Moments& m, const Phys& P) {
  add_reference_f(m, P);
  m.g00 += P.gref0;
}

__device__ __forceinline__ long long mhk(long long x, long long k) { return __mul64hi(x, k); }

// int64 -> float rounded to nearest (ties away from zero), value F 2^scale;
// results below the normal float range flush to zero
__device__ __forceinline__ float ll_to_float_rn(long long F, int scale) {
  if (F == 0) return 0.0f;
  const unsigned long long mag = F < 0 ? (unsigned long long)(-F) : (unsigned long long)F;
  const int lz = __clzll(mag);
  const unsigned long long norm = mag << lz;                          // leading one at bit 63
  const unsigned r = (unsigned)(norm >> 40) + (unsigned)((norm >> 39) & 1ull);  // 24 or 25 bits
  const int carry = (int)(r >> 24);
  const unsigned frac = (r >> carry) & 0x7fffffu;
  const int ex = 127 + 63 - lz + scale + carry;
  if (ex <= 0) return 0.0f;
  return __uint_as_float((unsigned)min(ex, 255) << 23 | (ex >= 255 ? 0u : frac) | (F < 0 ? 0x80000000u : 0u));
}

// 52-bit variant: value = X 2^(E - 1074); the magnitude is truncated (toward
// zero) in one shift of the significand
__device__ __forceinline__ long long to_block_fixed52(double v, int E) {
  const int hi = __double2hiint(v);
  const unsigned lo = (unsigned)__double2loint(v);
  const int e = (hi >> 20) & 0x7ff;
  const unsigned long long m = ((unsigned long long)((unsigned)(hi & 0xfffff) | 0x100000u) << 32) | lo;
  const unsigned long long mag = m >> min(E - e + 1, 63);
  return hi < 0 ? -(long long)mag : (long long)mag;
}

// ---- advection of one population over a tile (FP64 storage) -----------------
// The update's flux differences (Sec. III.A.2) of one population over a tile of
// up to 32 x R cells, by one warp, in block fixed point: the tile's cells and
// its upwind halo share one exponent, so every value is converted once (a
// per-cell stencil converts eight values per cell), to integers in units of
// 2^-(58 - L) of the largest (L: Phys::advn - 1; 2^-55 at beta = 6/5): exact for
// values within 2^(6 - L) of it, truncated below.  Differences are exact, and
// each limited slope is computed once and handed to the neighbour (along x by
// a warp shuffle, along y in registers while the warp walks the rows).
//
// The scheme is mirror symmetric, so a tile is walked in the population's own
// direction: stream coordinates i, j run along +v_x and +v_y, and one body
// serves all signs.  With D_j = F_j - F_{j-1} and sigma_j = minmod3(hb D_j,
// (D_j + D_{j+1})/4, hb D_{j+1}) the face value downstream of cell j is
// F_j + sigma_j, and the cell's change is -k ((F_j + sigma_j) - (F_{j-1} + sigma_{j-1})).
// Everything is kept times 4 lq (beta = lp / lq: candidates 2 lp D and
// lq (D + D')); a general beta takes lq = 1 and a fixed-point beta.
constexpr int kCta = 256;                 // threads of a step kernel's CTA
constexpr int kAdvPitch = 36;             // stream columns -2 .. 32 of a tile's row

// x k + y for a small k >= 0: two multiply-adds (a sign-extended 64-bit k takes three)
__device__ __forceinline__ long long mad_small(long long x, unsigned k, long long y) {
  unsigned lo, hi;
  asm("{\n\t.reg .u64 t;\n\tmad.wide.u32 t, %2, %3, %4;\n\tmov.b64 {%0, %1}, t;\n\t}"
      : "=r"(lo), "=r"(hi)
      : "r"((unsigned)x), "r"(k), "l"(y));
  hi += (unsigned)(x >> 32) * k;
  return (long long)(((unsigned long long)hi << 32) | lo);
}

// scaled limited slope 4 lq sigma(a, b)
template <bool RAT>
__device__ __forceinline__ long long slope_fix(long long a, long long b, const Phys& P) {
  const long long t = a + b;
  const bool neg = t < 0;
  const long long m = ((a < b) != neg) ? a : b;  // the smaller in magnitude, where the signs agree
  const bool differ = (a ^ b) < 0;               // else the slope is zero: the first candidate counts as 0
  long long r1, r2;
  if (RAT) {
    r1 = mad_small(m, differ ? 0u : 2u * (unsigned)P.lp, 0);
    r2 = mad_small(t, (unsigned)P.lq, 0);
  } else {
    const Limbs x(differ ? 0ll : m << 3);
    const Limbs h(P.hq);
    LimbAcc s;
    s.mac(x.h, x.l, h.h, h.l);
    r1 = s.floor() << 1;  // 2 beta m
    r2 = t;
  }
  return ((r1 < r2) != neg) ? r1 : r2;
}

// minmod branch of the cell's own slope as the adjoint reads it (backward
// difference first, in grid direction): 0 signs differ, 1 hb Da, 2 (Da + Db)/4,
// 3 hb Db, ties in that order; rational limiter
__device__ __forceinline__ unsigned slope_branch_code(long long a, long long b, bool mirrored, const Phys& P) {
  const long long Da = mirrored ? -b : a, Db = mirrored ? -a : b;
  if ((Da ^ Db) < 0) return 0u;
  const long long ra = Da * (long long)(2 * P.lp), rb = Db * (long long)(2 * P.lp), y = (Da + Db) * (long long)P.lq;
  if (Da >= 0) return (ra <= y && ra <= rb) ? 1u : (y <= rb ? 2u : 3u);
  return (ra >= y && ra >= rb) ? 1u : (y >= rb ? 2u : 3u);
}

struct AdvTile {
  int W, H;          // cells of the tile (ragged at the grid's upper ends)
  bool fx, fy;       // walked against x, against y
  int lane;
};
// What a warp reads of one population: its lane's column in stream rows -2 .. R,
// and one cell of the x-halo.  Read one population ahead, so that the loads'
// latency passes during the walk over the previous one.
template <int R>
struct AdvLoad {
  double v[R + 3], h;
};
// plane: the population's plane at the tile's lowest cell.  Every lane and row
// loads, in ragged tiles the last column and the row after the tile again, so
// that the loads need no predicates.
template <int R>
__device__ __forceinline__ void advect_load(AdvLoad<R>& L, const double* __restrict__ plane, long long PT,
                                            const AdvTile& T) {
  const int i = min(T.lane, T.W - 1);
  const unsigned lx = (unsigned)(T.fx ? T.W - 1 - i : i) * 8u;
  const long long sy = T.fy ? -PT : PT;
  const double* row0 = plane + (T.fy ? (T.H - 1) * PT : 0);  // stream row 0
#pragma unroll
  for (int j = -2; j <= R; ++j) L.v[j + 2] = load<R == 8>(at(row0 + min(j, T.H) * sy, lx));
  const int hr = min(T.lane % R, T.H - 1), hc = T.lane / R;  // halo cell: row hr, stream column -2, -1, W (or 0)
  const int h = hc > 2 ? 0 : hc == 2 ? T.W : hc - 2;
  L.h = load<R == 8>(row0 + hr * sy + (T.fx ? T.W - 1 - h : h));
}

// out: the plane (at the tile's lowest cell, row pitch PT) where the tile's flux
// sums go, kx (x-face difference) + ky (y-face difference) as integers W in
// units of 2^(E - 1079), E the returned block exponent (at least 128); MX, MY: the population
// moves along x, along y; kx, ky: flux factors (Phys::kxq, kyq); xs: this warp's
// [R + 3][kAdvPitch] words of shared memory; code: (CODES) this population's
// branch codes at the tile's lowest cell, row pitch cpitch; next: starts the
// next population's loads into L.
template <int R, bool MX, bool MY, bool RAT, bool CODES, class Next>
__device__ __forceinline__ int advect_tile(AdvLoad<R>& L, const Next& next, long long* out, long long PT, const AdvTile& T,
                                           const Phys& P, long long kx, long long ky, long long* xs,
                                           unsigned char* code, long long cpitch) {
  const int lane = T.lane;
  const bool in = lane < T.W;
  const unsigned lx = in ? (unsigned)(T.fx ? T.W - 1 - lane : lane) : 0u;  // this lane's column of the tile
  const long long sy = T.fy ? -PT : PT;
  constexpr int J0 = MY ? -2 : 0, J1 = MY ? R : R - 1;  // rows this population needs
  const double* v = L.v + (J0 + 2);
  const double vh = L.h;
  const int hr = lane % R, hc = lane / R;
  const bool hin = MX && hc < 3 && hr < T.H;
  // block exponent; non-finite values are left out (their key wraps to 0)
  unsigned key = 0;
#pragma unroll
  for (int j = 0; j <= J1 - J0; ++j) key = max(key, ((unsigned)__double2hiint(v[j]) + 0x100000u) & 0x7fffffffu);
  if (MX) key = max(key, ((unsigned)__double2hiint(vh) + 0x100000u) & 0x7fffffffu);
  key = __reduce_max_sync(0xffffffffu, key);
  const int E = (int)(key >> 20) - 1;
  const FlowScale B(E, P.advn);
  __syncwarp();  // the previous population's reads of xs are done
#pragma unroll
  for (int j = J0; j <= J1; ++j) xs[(j + 2) * kAdvPitch + lane + 2] = block_fix(v[j - J0], B);
  if (MX) {
    __syncwarp();  // column W of a ragged tile is written twice: the halo value last
    if (hin) xs[(hr + 2) * kAdvPitch + (hc == 2 ? T.W + 2 : hc)] = block_fix(vh, B);
  }
  next();
  __syncwarp();
  const unsigned q4 = RAT ? 4u * (unsigned)P.lq : 4u;
  if (MX) {
    // scaled face value upstream of column 0, one row per lane, kept in column -2
    if (lane < T.H) {
      long long* r = xs + (lane + 2) * kAdvPitch;
      const long long a = r[1] - r[0], b = r[2] - r[1];
      r[0] = mad_small(r[1], q4, slope_fix<RAT>(a, b, P));
    }
    __syncwarp();
  }
  const Limbs KX(kx), KY(ky);
  const long long* own = xs + 2 * kAdvPitch + lane + 2;  // (row 0, this column)
  long long c = own[0], dy = 0, gy = 0;
  if (MY) {
    const long long b = own[-kAdvPitch], a = own[-2 * kAdvPitch];
    dy = c - b;
    gy = mad_small(b, q4, slope_fix<RAT>(b - a, dy, P));
  }
  long long* orow = out + (T.fy ? (T.H - 1) * PT : 0);
  unsigned char* crow = CODES ? code + (T.fy ? (T.H - 1) * cpitch : 0) : nullptr;
  const long long csy = T.fy ? -cpitch : cpitch;
#pragma unroll 1
  for (int j = 0; j < T.H; ++j) {
    LimbAcc w;
    unsigned bits = 0;
    if (MX) {
      const long long a = c - own[-1], b = own[1] - c;
      const long long g = mad_small(c, q4, slope_fix<RAT>(a, b, P));
      const long long e = xs[(j + 2) * kAdvPitch];
      long long gl = __shfl_up_sync(0xffffffffu, g, 1);
      if (lane == 0) gl = e;
      const Limbs f(g - gl);
      w.mac(f.h, f.l, KX.h, KX.l);
      if (CODES) bits = slope_branch_code(a, b, T.fx, P);
    }
    const long long cn = own[kAdvPitch];
    if (MY) {
      const long long dn = cn - c;
      const long long g = mad_small(c, q4, slope_fix<RAT>(dy, dn, P));
      const Limbs f(g - gy);
      w.mac(f.h, f.l, KY.h, KY.l);
      if (CODES) bits |= slope_branch_code(dy, dn, T.fy, P) << 2;
      gy = g;
      dy = dn;
    }
    if (in) {
      *at(orow, lx * 8) = w.floor();
      if (CODES) crow[lx] = (unsigned char)bits;
    }
    c = cn;
    own += kAdvPitch;
    orow += sy;
    if (CODES) crow += csy;
  }
  return max(E, 128);
}

// a1 F + target - flux sum of one population: the target t 2^(st - 1079) and
// the flux sum w 2^(sw - 1079) are subtracted as integers at the larger of
// their scales, so that one conversion and one FMA are left.  Both are rounded
// down, so the mean errors cancel in the difference.  The conversion is the
// hardware's: it takes one slot of the FP64 pipe, which the kernel does not
// fill, for about twenty integer instructions.
__device__ __forceinline__ double collide_advect(double a1, double F, long long t, int st, long long w, int sw) {
  const int d = sw - st;
  const double z = __ll2double_rn((t >> min(max(d, 0), 63)) - (w >> min(max(-d, 0), 63)));
  const int zh = __double2hiint(z);
  return fma(a1, F, __hiloint2double(zh == 0 ? 0 : zh + ((max(sw, st) - 1079) << 20), __double2loint(z)));
}

// node constants W_k He_n(xi_k)/n! 2^(61 + kd(k)) (below 2^61), rounded from their
// exact values; nodes 0, +-sqrt(5 - sqrt 10), +-sqrt(5 + sqrt 10)
constexpr long long kKF[3][5] = {
    {1229782938247303441ll, 0ll, -614891469123651721ll, 0ll, 153722867280912930ll},
    {1024144424542654913ll, 1388356993984702056ll, 428974331826690775ll, -268942719741157367ll, -198390030905321379ll},
    {415325171389884787ll, 1186571560667484526ll, 1487337098375687568ll, 1020901976637480698ll, 357337308995267594ll}};
__host__ __device__ constexpr long long kf(int k, int n) {
  return sgn_of(k) < 0 && n % 2 == 1 ? -kKF[(k + 1) / 2][n] : kKF[(k + 1) / 2][n];
}
// as limbs, a constant-bank table for the node loop: [node][n] = {high, low}
static __constant__ int c_kf[5][5][2] = {
#define KF(k, n) {limb_hi(kf(k, n)), limb_lo(kf(k, n))}
#define KROW(k) {KF(k, 0), KF(k, 1), KF(k, 2), KF(k, 3), KF(k, 4)}
    KROW(0), KROW(1), KROW(2), KROW(3), KROW(4)};

// This thread's collision coefficients in block fixed point (60 bits, one
// exponent for f, one for g) as limb pairs in shared memory: field k of thread
// t at [k * kCta + t] (consecutive threads, consecutive words; registers would
// hold 42 words across the node loop).  Field order f00, f10, f01, f20, f11,
// f02, f30, f21, f12, f03, f40, f31, f22, f13, f04, g00, g10, g01, g20, g11, g02.
template <int STRIDE>
struct FixViewOf {
  const long long* b;
  __device__ __forceinline__ void mac(LimbAcc& s, int field, const int (&k)[2]) const {
    const long long x = b[field * STRIDE];
    s.mac((int)(x >> 32), (int)x, k[0], k[1]);
  }
};
typedef FixViewOf<kCta> FixView;
template <int N, int STRIDE = kCta>
__device__ __forceinline__ void fields_to_smem(const double (&f)[N], long long* b, int& E) {
  unsigned key = 0;
#pragma unroll
  for (int k = 0; k < N; ++k) key = max(key, abs_key(f[k]));
  const FlowScale B((int)(key >> 20), 0);
#pragma unroll
  for (int k = 0; k < N; ++k) b[k * STRIDE] = pack_limbs(block_fix(f[k], B));
  E = max(B.E, 128);  // also where collide_advect's result of a zero target is normal
}
// h^b of x-node p: W_p sum_a C_ab He_a(xi_p)/a! (value h 2^(E - 1082 - kd(p)))
template <class V>
__device__ __forceinline__ void hf_node(const V& X, const int (&K)[5][2], long long (&h)[5]) {
  LimbAcc a, b, c, d, e;
  X.mac(a, 0, K[0]); X.mac(a, 1, K[1]); X.mac(a, 3, K[2]); X.mac(a, 6, K[3]); X.mac(a, 10, K[4]);
  X.mac(b, 2, K[0]); X.mac(b, 4, K[1]); X.mac(b, 7, K[2]); X.mac(b, 11, K[3]);
  X.mac(c, 5, K[0]); X.mac(c, 8, K[1]); X.mac(c, 12, K[2]);
  X.mac(d, 9, K[0]); X.mac(d, 13, K[1]);
  X.mac(e, 14, K[0]);
  h[0] = a.value8(); h[1] = b.value8(); h[2] = c.value8(); h[3] = d.value8(); h[4] = e.value8();
}
template <class V>
__device__ __forceinline__ void hg_node(const V& X, const int (&K)[5][2], long long (&h)[3]) {
  LimbAcc a, b, c;
  X.mac(a, 15, K[0]); X.mac(a, 16, K[1]); X.mac(a, 18, K[2]);
  X.mac(b, 17, K[0]); X.mac(b, 19, K[1]);
  X.mac(c, 20, K[0]);
  h[0] = a.value8(); h[1] = b.value8(); h[2] = c.value8();
}
template <int k, int n>
__device__ __forceinline__ void kmac(LimbAcc& s, const Limbs& x) {
  s.mac(x.h, x.l, limb_hi(kf(k, n)), limb_lo(kf(k, n)));
}
// t_q = W_q sum_b h^b He_b(xi_q)/b! of the five y-nodes with the +-xi symmetry:
// value t_q 2^(E - 1079 - kd(p) - kd(q))
__device__ __forceinline__ void expand_node(const long long (&h)[5], long long (&t)[5]) {
  const Limbs h0(h[0]), h1(h[1]), h2(h[2]), h3(h[3]), h4(h[4]);
  LimbAcc c, ea, oa, eb, ob;
  kmac<0, 0>(c, h0); kmac<0, 2>(c, h2); kmac<0, 4>(c, h4);
  kmac<1, 0>(ea, h0); kmac<1, 2>(ea, h2); kmac<1, 4>(ea, h4);
  kmac<1, 1>(oa, h1); kmac<1, 3>(oa, h3);
  kmac<3, 0>(eb, h0); kmac<3, 2>(eb, h2); kmac<3, 4>(eb, h4);
  kmac<3, 1>(ob, h1); kmac<3, 3>(ob, h3);
  t[0] = c.value();
  t[1] = ea.value() + oa.value(); t[2] = ea.value() - oa.value();
  t[3] = eb.value() + ob.value(); t[4] = eb.value() - ob.value();
}
__device__ __forceinline__ void expand_node(const long long (&h)[3], long long (&t)[5]) {
  const Limbs h0(h[0]), h1(h[1]), h2(h[2]);
  LimbAcc c, ea, oa, eb, ob;
  kmac<0, 0>(c, h0); kmac<0, 2>(c, h2);
  kmac<1, 0>(ea, h0); kmac<1, 2>(ea, h2);
  kmac<1, 1>(oa, h1);
  kmac<3, 0>(eb, h0); kmac<3, 2>(eb, h2);
  kmac<3, 1>(ob, h1);
  t[0] = c.value();
  t[1] = ea.value() + oa.value(); t[2] = ea.value() - oa.value();
  t[3] = eb.value() + ob.value(); t[4] = eb.value() - ob.value();
}
__device__ __forceinline__ void load_kf(int p, int (&K)[5][2]) {
#pragma unroll
  for (int n = 0; n < 5; ++n) {
    K[n][0] = c_kf[p][n][0];
    K[n][1] = c_kf[p][n][1];
  }
}

struct Lat25 {
  static constexpr int NQ = 5, POPS = 50, FIELDS = 21, GFIELD = 15, MOMS = 13;  // GFIELD: the first field of g
  typedef Moments Mom;
  typedef int NodeK[5][2];
  __device__ static __forceinline__ bool backward(int k) { return k != 0 && (k & 1) == 0; }
  __device__ static __forceinline__ int kdp(int k) { return k == 0 ? 0 : (k <= 2 ? kd(1) : kd(3)); }
  template <bool NC>
  __device__ static __forceinline__ void moments_f(const double* s, unsigned off, long long PL, Mom& m) {
    moments_fix_f<double, NC>(s, off, PL, m);
  }
  template <bool NC>
  __device__ static __forceinline__ void moments_g(const double* s, unsigned off, long long PL, Mom& m) {
    moments_fix_g<double, NC>(s, off, PL, m);
  }
  template <int PRC>
  __device__ static __forceinline__ Coeffs coeffs(const Mom& m, const Phys& P) { return collision_coeffs<PRC>(m, P); }
  __device__ static __forceinline__ void to_smem(const Coeffs& C, long long* b, int& Ef, int& Eg) {
    const double f[15] = {C.f00, C.f10, C.f01, C.f20, C.f11, C.f02, C.f30, C.f21,
                          C.f12, C.f03, C.f40, C.f31, C.f22, C.f13, C.f04};
    const double g[6] = {C.g00, C.g10, C.g01, C.g20, C.g11, C.g02};
    fields_to_smem<15>(f, b, Ef);
    fields_to_smem<6>(g, b + 15 * kCta, Eg);
  }
  // the fields in order; the moments that a sum over f (k = 0) or g yields, and back
  template <class Put>
  __device__ static __forceinline__ void fields(const Coeffs& C, const Put& put) {
    const double v[21] = {C.f00, C.f10, C.f01, C.f20, C.f11, C.f02, C.f30, C.f21, C.f12, C.f03, C.f40,
                          C.f31, C.f22, C.f13, C.f04, C.g00, C.g10, C.g01, C.g20, C.g11, C.g02};
#pragma unroll
    for (int k = 0; k < 21; ++k) put(k, v[k]);
  }
  template <class Put>
  __device__ static __forceinline__ void put(const Mom& m, int k, const Put& put) {
    if (k == 0) {
      put(0, m.m00); put(1, m.m10); put(2, m.m01); put(3, m.m20); put(4, m.m11); put(5, m.m02); put(6, m.m30);
      put(7, m.m21); put(8, m.m12); put(9, m.m03);
    } else {
      put(10, m.g00); put(11, m.g10); put(12, m.g01);
    }
  }
  template <class Get>
  __device__ static __forceinline__ void get(Mom& m, const Get& get) {
    m.m00 = get(0); m.m10 = get(1); m.m01 = get(2); m.m20 = get(3); m.m11 = get(4); m.m02 = get(5); m.m30 = get(6);
    m.m21 = get(7); m.m12 = get(8); m.m03 = get(9); m.g00 = get(10); m.g10 = get(11); m.g01 = get(12);
  }
  __device__ static __forceinline__ void load_k(int p, NodeK& K) { load_kf(p, K); }
  template <class V>
  __device__ static __forceinline__ void target_f(const V& X, const NodeK& K, long long (&t)[5]) {
    long long h[5];
    hf_node(X, K, h);
    expand_node(h, t);
  }
  template <class V>
  __device__ static __forceinline__ void target_g(const V& X, const NodeK& K, long long (&t)[5]) {
    long long h[3];
    hg_node(X, K, h);
    expand_node(h, t);
  }
};

// ---- the FP64 step over tiles --------------------------------------------------
// Two phases per 32 x R tile, 256 threads.  Advection, one population per warp:
// the warp walks the tile and writes the flux sums (advect_tile) as integers into
// the new state's space, from where they come back out of L2.  Collision, one
// cell per thread: moments, combined coefficients, the collision target of each
// population in fixed point, and the update with the flux sum (collide_advect).
// Low tiles (R < 8, small grids) also write the periodic and zero-gradient ghost
// images of the cells next to the grid's edge, so that a step without walls is
// one launch (4 us less at 64^2).  In the 8-row kernel the same code costs 6 %: its
// divergent tail keeps the compiler off the uniform registers for addresses.
//  * Advection: warp w does f (w < 4) or g.  D2Q25: x-node p = 1 + w % 4, its four
//    populations that move along both axes, (p, 0) along x only and (0, p) along
//    y only, so that all eight warps have the same work; the resting population
//    needs none.  D2Q16: the four populations of x-node w % 4.
//  * Collision with R < 8: a cell has 8 / R threads, which share its populations
//    (in units of an x-node's f or g).
struct GhostKinds {
  int k[4];  // xlo, xhi, ylo, yhi: 0 periodic, 1 zero gradient, else not written here
};
// is the cell the source of a ghost image?
__device__ __forceinline__ bool on_edge(int x, int y, const Geom& G, const GhostKinds& B) {
  return ((x < 2 && B.k[0] < 2) || (x >= G.Nx - 2 && B.k[1] < 2) || (y < 2 && B.k[2] < 2) || (y >= G.Ny - 2 && B.k[3] < 2));
}
// copies N planes' values of cell (x, y) to the cell's ghost images; p: the cell in
// the first of them
template <int N, class S>
__device__ __forceinline__ void write_images(S* p, long long PL, int x, int y, const Geom& G, const GhostKinds& B) {
  S v[N];
#pragma unroll
  for (int q = 0; q < N; ++q) v[q] = p[q * PL];
  auto put = [&](long long o) {
#pragma unroll
    for (int q = 0; q < N; ++q) p[q * PL + o] = v[q];
  };
  const long long PT = G.pitch;
  if (B.k[0] == 0) {
    if (x < 2) put(G.Nx);
    if (x >= G.Nx - 2) put(-G.Nx);
  }
  if (B.k[0] == 1 && x == 0) put(-1), put(-2);
  if (B.k[1] == 1 && x == G.Nx - 1) put(1), put(2);
  if (B.k[2] == 0) {
    if (y < 2) put(G.Ny * PT);
    if (y >= G.Ny - 2) put(-G.Ny * PT);
  }
  if (B.k[2] == 1 && y == 0) put(-PT), put(-2 * PT);
  if (B.k[3] == 1 && y == G.Ny - 1) put(PT), put(2 * PT);
}

// What bounds it: the integer ALU (about two thirds busy) beside the FP64 pipe
// (57 %) and the latency between them; DRAM is at 38 % of its rate (the flux sums
// leave L2 in part: about 1.6 kB a cell).  D2Q25: 13.2 k instructions and 186 FP64 ones
// a cell (conversions counted), against 26.8 k and 407 of a thread per cell with its
// own stencils: 15.5 -> 8.4 ms a step at 4096^2, 1.02 -> 0.54 ms at 1024^2.  D2Q16: 10.5 -> 5.6 ms and 0.70 -> 0.37 ms.  Three CTAs of 80
// registers; four of 64 measured 1 % slower.
// L: the lattice (Lat25, Lat16).  PRC: Prandtl branch; RAT: rational limiter;
// CODES: also the branch codes of every population's slopes (one byte x | y << 2
// at codes[pop][y][x]) and, unless moms is null, the cells' moments.
template <class L, int R, int PRC, bool RAT, bool CODES>
__global__ void __launch_bounds__(kCta, R == 8 ? 3 : 1) k_step_tile(const double* __restrict__ src, double* dst, Geom G, Phys P,
                                                       GhostKinds B, unsigned int* __restrict__ flag,
                                                       unsigned char* codes, double* __restrict__ moms) {
  __shared__ long long s_buf[L::FIELDS * kCta];  // the advection's tiles, then the collision coefficients
  __shared__ int s_exp[L::POPS];                 // block exponents of the flux sums
  static_assert(8 * (R + 3) * kAdvPitch <= L::FIELDS * kCta, "the advection tiles fit the coefficients' space");
  constexpr int NQ = L::NQ, NF = NQ * NQ;
  const int x0 = blockIdx.x * 32, y0 = blockIdx.y * R;
  const long long PL = G.plane;
  const long long PT = G.pitch;
  const long long cplane = (long long)G.Nx * G.Ny;
  if constexpr (R < 8) src = chain_wait(src);
  const double* stile = src + cell_index(G, y0, x0);
  double* dtile = dst + cell_index(G, y0, x0);
  {
    const int w = __shfl_sync(0xffffffffu, (int)threadIdx.y, 0), c0 = NF * (w >> 2);
    AdvTile T;
    T.W = min(32, G.Nx - x0);
    T.H = min(R, G.Ny - y0);
    T.lane = threadIdx.x;
    long long* xs = s_buf + w * ((R + 3) * kAdvPitch);
    unsigned char* ctile = CODES ? codes + (long long)y0 * G.Nx + x0 : nullptr;
    int E;
    AdvLoad<R> V;
    // the walk directions of population (p, q): sign of each velocity component
    auto tile = [&](int p, int q) {
      AdvTile t = T;
      t.fx = L::backward(p);
      t.fy = L::backward(q);
      return t;
    };
    auto load = [&](int p, int q) { advect_load<R>(V, stile + (c0 + NQ * p + q) * PL, PT, tile(p, q)); };
    auto out = [&](int c) { return (long long*)(dtile + c * PL); };
    auto code = [&](int c) { return CODES ? ctile + c * cplane : nullptr; };
    if constexpr (NQ == 5) {
      const int p = 1 + (w & 3);
      load(p, 0);
      {
        const int c = c0 + 5 * p;
        E = advect_tile<R, true, false, RAT, CODES>(V, [&] { load(p, 1); }, out(c), PT, tile(p, 0), P, P.kxq[p], 0, xs,
                                                    code(c), G.Nx);
        if (T.lane == 0) s_exp[c] = E;
      }
#pragma unroll 1
      for (int q = 1; q < 5; ++q) {
        const int c = c0 + 5 * p + q;
        E = advect_tile<R, true, true, RAT, CODES>(V, [&] { load(q < 4 ? p : 0, q < 4 ? q + 1 : p); }, out(c), PT,
                                                   tile(p, q), P, P.kxq[p], P.kyq[q], xs, code(c), G.Nx);
        if (T.lane == 0) s_exp[c] = E;
      }
      {
        const int c = c0 + p;
        E = advect_tile<R, false, true, RAT, CODES>(V, [] {}, out(c), PT, tile(0, p), P, 0, P.kyq[p], xs, code(c), G.Nx);
        if (T.lane == 0) s_exp[c] = E;
      }
      if (p == 1) {  // the resting population: no flux, and no slopes the adjoint uses
        if (T.lane == 0) s_exp[c0] = 0;
        if (T.lane < T.W)
          for (int j = 0; j < T.H; ++j) {
            ((long long*)dtile)[c0 * PL + j * PT + T.lane] = 0;
            if (CODES) ctile[c0 * cplane + (long long)j * G.Nx + T.lane] = 0;
          }
      }
    } else {
      const int p = w & 3;
      load(p, 0);
#pragma unroll 1
      for (int q = 0; q < 4; ++q) {
        const int c = c0 + 4 * p + q;
        E = advect_tile<R, true, true, RAT, CODES>(V, [&] { load(p, min(q + 1, 3)); }, out(c), PT, tile(p, q), P, P.kxq[p],
                                                   P.kyq[q], xs, code(c), G.Nx);
        if (T.lane == 0) s_exp[c] = E;
      }
    }
  }
  __syncthreads();
  constexpr int NG = 8 / R;  // threads of a cell
  const int row = threadIdx.y % R, group = threadIdx.y / R;
  const int x = x0 + threadIdx.x, y = y0 + row;
  const unsigned off = (row * (unsigned)PT + threadIdx.x) * 8u;  // this cell's byte offset in the tile
  const int cell = row * 32 + threadIdx.x;
  const FixView X{s_buf + cell};
  const bool inside = x < G.Nx && y < G.Ny;
  int Ef, Eg;
  double a1;
  auto collision = [&](const typename L::Mom& m) {
    if constexpr (CODES) {
      // the recomputing adjoint also keeps the cell's moments (13 planes of
      // Nx * Ny doubles, Moments field order) for its collision part
      if (moms) {
        const long long ci = (long long)y * G.Nx + x;
        const double v[13] = {m.m00, m.m10, m.m01, m.m20, m.m11, m.m02, m.m30,
                              m.m21, m.m12, m.m03, m.g00, m.g10, m.g01};
#pragma unroll
        for (int k = 0; k < 13; ++k) moms[k * cplane + ci] = v[k];
      }
    }
    const auto C = L::template coeffs<PRC>(m, P);
    if (C.bad) atomicOr(flag, 1u);
    L::to_smem(C, s_buf + cell, Ef, Eg);
    a1 = C.a1;
  };
  if constexpr (NG == 1) {
    if (!inside) return;
    typename L::Mom m;
    L::template moments_f<true>(stile, off, PL, m);
    L::template moments_g<true>(stile, off, PL, m);
    collision(m);
  } else {
    // the first group sums f and forms the coefficients, the second sums g: all
    // groups doing all of it would share the FP64 pipe (6 us more at 64^2)
    __shared__ double s_share[4][32 * R];
    __shared__ int s_block[2][32 * R];
    typename L::Mom m;
    if (inside && group == 0) L::template moments_f<false>(stile, off, PL, m);
    if (inside && group == 1) {
      L::template moments_g<false>(stile, off, PL, m);
      s_share[0][cell] = m.g00; s_share[1][cell] = m.g10; s_share[2][cell] = m.g01;
    }
    __syncthreads();
    if (inside && group == 0) {
      m.g00 = s_share[0][cell]; m.g10 = s_share[1][cell]; m.g01 = s_share[2][cell];
      collision(m);
      s_share[3][cell] = a1;
      s_block[0][cell] = Ef;
      s_block[1][cell] = Eg;
    }
    __syncthreads();
    if (!inside) return;
    a1 = s_share[3][cell];
    Ef = s_block[0][cell];
    Eg = s_block[1][cell];
  }
#pragma unroll 1
  for (int p0 = 0; p0 < NQ; p0 += NG > 2 ? NG / 2 : 1) {
    // NG = 1: an x-node's f and g in turn; NG = 2: one of them; NG = 4: of every second x-node
    const int p = NG > 2 ? p0 + (group >> 1) : p0;
    if (NG > 2 && p >= NQ) break;
    typename L::NodeK K;
    L::load_k(p, K);
    const int dp = L::kdp(p);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (NG > 1 && k != (group & 1)) continue;
      const double* sp = stile + (NF * k + NQ * p) * PL;
      double* dp_ = dtile + (NF * k + NQ * p) * PL;
      double F[NQ];
      long long W[NQ], t[NQ];
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        F[q] = load<R == 8>(at(sp + q * PL, off));
        W[q] = *at((const long long*)dp_ + q * PL, off);
      }
      if (k == 0) L::target_f(X, K, t);
      else L::target_g(X, K, t);
      const int st = (k == 0 ? Ef : Eg) - dp;
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        *at(dp_ + q * PL, off) = collide_advect(a1, F[q], t[q], st - L::kdp(q), W[q], s_exp[NF * k + NQ * p + q]);
      }
    }
  }
  if constexpr (R < 8) {
    if (on_edge(x, y, G, B)) {
      // of the units this thread has written
      for (int p = NG > 2 ? group >> 1 : 0; p < NQ; p += NG > 2 ? NG / 2 : 1)
        write_images<NQ>(at(dtile + (NF * (group & 1) + NQ * p) * PL, off), PL, x, y, G, B);
    }
  }
}

// Flux difference F_{j+1/2} - F_{j-1/2} of the upwind-limited face values
// along a stride (float, FP32-deviation storage); SGN = sign of the velocity
// component (never 0 here).
//   v > 0: faces f_{j-1} + sigma_{j-1}, f_j + sigma_j
//   v < 0: faces f_j - sigma_j, f_{j+1} - sigma_{j+1}
template <int SGN, class T>
__device__ __forceinline__ T flux_difference(const T* __restrict__ ptr, long long stride, T hb) {
  static_assert(sizeof(T) == 4, "FP64 storage uses the integer flux differences");
  if (SGN > 0) {
    const T fm2 = __ldg(ptr - 2 * stride), fm1 = __ldg(ptr - stride), f0 = __ldg(ptr), fp1 = __ldg(ptr + stride);
    const T Dm = fm1 - fm2, D0 = f0 - fm1, Dp = fp1 - f0;
    return D0 + limited_slope(D0, Dp, hb) - limited_slope(Dm, D0, hb);
  } else {
    const T fm1 = __ldg(ptr - stride), f0 = __ldg(ptr), fp1 = __ldg(ptr + stride), fp2 = __ldg(ptr + 2 * stride);
    const T D0 = f0 - fm1, Dp = fp1 - f0, Dpp = fp2 - fp1;
    return Dp - limited_slope(Dp, Dpp, hb) + limited_slope(D0, Dp, hb);
  }
}

}  // namespace dvbm
