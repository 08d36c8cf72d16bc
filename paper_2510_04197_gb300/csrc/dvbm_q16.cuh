// dvbm_q16.cuh -- the total-energy split (I) on the D2Q16 lattice: lattice,
// moments, equilibria and quasi-equilibria, Grad expansion (double and block
// fixed point).  Shared by the D2Q16 step kernel (dvbm_d2q16.cu) and the
// lattice-templated auxiliary kernels (dvbm_aux.cu).
//
// Same time step as the D2Q25 / split II kernels (Eq. finalDiscretePDE), with
//  * the D2Q16 Gauss--Hermite lattice (App. G, Table "D2Q16"): 1-D nodes
//    +-sqrt(3 -+ sqrt 6) with weights (3 +- sqrt 6)/12;
//  * E = sum g (Eq. eq_quadratur3 (I)), f^eq to third order and g^eq to
//    second order (Sec. II.D.3, App. E), g^eq built from the split-I moments
//    of App. A: M0 = E, M1 = u (E + rho R T), M2 = rho R T uu + (E + rho R T)(uu + R T I);
//  * the split-I quasi-equilibria of Table I: Pr < 1: f* = f^eq,
//    M1(g*) = M1(g) - u.(M2(f) - M2(f^eq)); Pr > 1: M2(f*) = M2(f),
//    M1(g*) = M1(g^eq) + u.(M2(f) - M2(f^eq)); Pr = 1: equilibria.
// Populations: c = 4 p + q for f (0..15), 16 + 4 p + q for g, x-node p and
// y-node q in the order (+a, -a, +b, -b), a = sqrt(3 - sqrt 6), b = sqrt(3 + sqrt 6).
// FP64 storage; advection in block floating point on the integer pipe.
#pragma once
#include "dvbm_device.cuh"

namespace dvbm {
namespace q16 {

constexpr double YA = 0.7419637843027258;   // sqrt(3 - sqrt 6)
constexpr double YB = 2.3344142183389773;   // sqrt(3 + sqrt 6)
constexpr double VA = 0.45412414523193151;  // (3 + sqrt 6)/12
constexpr double VB = 0.045875854768068492; // (3 - sqrt 6)/12
constexpr int NP = 32;

__host__ __device__ constexpr double xi(int k) { return k == 0 ? YA : k == 1 ? -YA : k == 2 ? YB : -YB; }
__host__ __device__ constexpr double w(int k) { return k < 2 ? VA : VB; }
__host__ __device__ constexpr int sgn(int k) { return (k % 2 == 0) ? 1 : -1; }

struct Mom { double m00, m10, m01, m20, m11, m02, g00, g10, g01; };
struct Co {
  double f00, f10, f01, f20, f11, f02, f30, f21, f12, f03;
  double g00, g10, g01, g20, g11, g02;  // physical energy units
  double a1;
  bool bad;
};

struct Eq3 { double a00, a10, a01, a20, a11, a02, a30, a21, a12, a03; };
struct EqG { double A00, A10, A01, A20, A11, A02; };

__device__ __forceinline__ Eq3 eq_f3(double rho, double ux, double uy, double s) {
  Eq3 e;
  const double rs = rho * s;
  e.a00 = rho; e.a10 = rho * ux; e.a01 = rho * uy;
  e.a20 = fma(e.a10, ux, rs); e.a11 = e.a10 * uy; e.a02 = fma(e.a01, uy, rs);
  e.a30 = fma(e.a20, ux, 2.0 * s * e.a10); e.a03 = fma(e.a02, uy, 2.0 * s * e.a01);
  e.a21 = e.a20 * uy; e.a12 = e.a02 * ux;
  return e;
}

// g^eq coefficients of split I in physical units: E the total energy, pRT = rho R T
__device__ __forceinline__ EqG eq_g1(double E, double pRT, double ux, double uy, double theta) {
  EqG q;
  const double Ep = E + pRT;
  q.A00 = E;
  q.A10 = ux * Ep;
  q.A01 = uy * Ep;
  q.A20 = fma(pRT, ux * ux, Ep * fma(ux, ux, theta)) - E;
  q.A11 = (pRT + Ep) * ux * uy;
  q.A02 = fma(pRT, uy * uy, Ep * fma(uy, uy, theta)) - E;
  return q;
}

// Collision coefficients (Table I split I): k1 A^eq + (k1 - k2)(A* - A^eq) with the
// equilibria of f and g at k1, as in collision_coeffs: k1 = dt/tau1 enters at the
// zeroth coefficients, and A20, A11, A02 of g share (H + p) u:
//   A20 = (H + p) ux^2 + H theta - E,  A11 = (H + p) ux uy,  H = E + p.
// 58 FP64 instructions instead of 91 in a kernel whose FP64 pipe is about 70 % busy:
// 12 steps at 2048^2 19.07 -> 18.50 ms.
template <int PRC>
__device__ __forceinline__ Co coeffs(const Mom& m, const Phys& P) {
  Co C;
  const double rho = m.m00;
  const double irho = recip(rho);
  const double ux = m.m10 * irho, uy = m.m01 * irho;
  const double E = m.g00;
  const double theta = P.gm1 * fma(-0.5, fma(ux, ux, uy * uy), E * P.inv_c2 * irho);
  const double s = theta - 1.0;
  C.bad = !is_positive(rho) || !is_positive(theta) || !is_bounded(E);
  const double rt = rho * theta, pRT = rt * P.c2;
  const double kp = P.dt_mu * pRT;                // dt p / mu
  const double k1 = PRC <= 0 ? kp : kp * P.Pr;    // dt/tau1
  C.a1 = 1.0 - k1;
  const Eq3 e = eq_f3(k1 * rho, ux, uy, s);       // k1 A^eq
  C.f00 = e.a00; C.f10 = e.a10; C.f01 = e.a01; C.f20 = e.a20; C.f11 = e.a11; C.f02 = e.a02;
  C.f30 = e.a30; C.f21 = e.a21; C.f12 = e.a12; C.f03 = e.a03;
  const double p = k1 * pRT, H = fma(k1, E, p), S = H + p;
  const double Sx = S * ux, Sy = S * uy;
  C.g00 = k1 * E;
  const double z = fma(H, theta, -C.g00);
  C.g10 = ux * H; C.g01 = uy * H;
  C.g20 = fma(Sx, ux, z); C.g11 = Sx * uy; C.g02 = fma(Sy, uy, z);
  if (PRC != 0) {
    // Delta = H_2(f) - A^eq_2 and u . Delta
    const double Dxx = fma(-m.m10, ux, m.m20 - rt), Dxy = fma(-m.m10, uy, m.m11), Dyy = fma(-m.m01, uy, m.m02 - rt);
    const double cx = fma(ux, Dxx, uy * Dxy), cy = fma(ux, Dxy, uy * Dyy);
    if (PRC < 0) {
      const double s1 = fma(-P.Pr, k1, k1);       // dt/tau1 - dt/tau2
      C.g10 = fma(s1, fma(-P.c2, cx, m.g10), P.Pr * C.g10);
      C.g01 = fma(s1, fma(-P.c2, cy, m.g01), P.Pr * C.g01);
    } else {
      const double s1 = k1 - kp, sc = s1 * P.c2;
      C.f20 = fma(s1, Dxx, C.f20); C.f11 = fma(s1, Dxy, C.f11); C.f02 = fma(s1, Dyy, C.f02);
      C.g10 = fma(sc, cx, C.g10); C.g01 = fma(sc, cy, C.g01);
    }
  }
  return C;
}

// equilibrium populations (k1 = 1, no quasi-equilibrium part)
__device__ __forceinline__ Co equilibrium(double rho, double ux, double uy, double theta, const Phys& P) {
  Co C;
  const Eq3 e = eq_f3(rho, ux, uy, theta - 1.0);
  const double pRT = rho * P.c2 * theta;
  const double E = rho * P.c2 * (theta * recip(P.gm1) + 0.5 * fma(ux, ux, uy * uy));
  const EqG q = eq_g1(E, pRT, ux, uy, theta);
  C.f00 = e.a00; C.f10 = e.a10; C.f01 = e.a01; C.f20 = e.a20; C.f11 = e.a11; C.f02 = e.a02;
  C.f30 = e.a30; C.f21 = e.a21; C.f12 = e.a12; C.f03 = e.a03;
  C.g00 = q.A00; C.g10 = q.A10; C.g01 = q.A01; C.g20 = q.A20; C.g11 = q.A11; C.g02 = q.A02;
  C.a1 = 0.0;
  C.bad = false;
  return C;
}

__device__ __forceinline__ void macro(const Mom& m, const Phys& P, double c, double T_ref, double& rho, double& ux,
                                      double& uy, double& T) {
  rho = m.m00;
  const double irho = 1.0 / rho;
  const double a = m.m10 * irho, b = m.m01 * irho;
  const double theta = P.gm1 * fma(-0.5, fma(a, a, b * b), m.g00 * P.inv_c2 * irho);
  ux = a * c;
  uy = b * c;
  T = theta * T_ref;
}

// ---- the step over tiles (k_step_tile) -----------------------------------------

// node constants W_k He_n(xi_k)/n! 2^(61 + kdq(k)), rounded from their exact values
// (the +-sqrt(3 + sqrt 6) nodes carry the small weight and gain two bits)
__host__ __device__ constexpr int kdq(int k) { return k < 2 ? 0 : 2; }
constexpr long long kKQ[2][4] = {
    {1047138985598193535ll, 776939204445353226ll, -235339116647385024ll, -317184102009169216ll},
    {423130076034613764ll, 987760865702054896ll, 941356466589540094ll, 403251684809969295ll}};
__host__ __device__ constexpr long long kqf(int k, int n) {
  return sgn(k) < 0 && n % 2 == 1 ? -kKQ[k / 2][n] : kKQ[k / 2][n];
}
static __constant__ int c_kqf[4][4][2] = {
#define KQ(k, n) {limb_hi(kqf(k, n)), limb_lo(kqf(k, n))}
#define KQROW(k) {KQ(k, 0), KQ(k, 1), KQ(k, 2), KQ(k, 3)}
    KQROW(0), KQROW(1), KQROW(2), KQROW(3)};
#undef KQROW
#undef KQ

// YA^n and YB^n times 2^62 / 4, / 8 (n = 1, 2): pair sums / 16, / 32
constexpr long long kYA[3] = {0, 855426002562088766ll, 317347557025960323ll};
constexpr long long kYB[3] = {0, 2691396352982990230ll, 3141416956794580605ll};
template <int n>
__device__ __forceinline__ long long pair_sum16(long long b, long long a) {
  const Limbs x(b), y(a);
  LimbAcc s;
  s.mac(x.h, x.l, limb_hi(kYB[n]), limb_lo(kYB[n]));
  s.mac(y.h, y.l, limb_hi(kYA[n]), limb_lo(kYA[n]));
  return s.value();
}

// moments in block fixed point, as moments_fix for D2Q25: of f (k = 0) or g (k = 1)
template <int k, bool NC = true>
__device__ __forceinline__ void moments_fix16(const double* __restrict__ s, unsigned off, long long PL, Mom& m) {
  double v[16];
  unsigned key = 0;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    v[i] = load<NC>(at(s + (16 * k + i) * PL, off));
    key = max(key, abs_key(v[i]));
  }
  const int E = (int)(key >> 20);
  const FlowScale B(E, 2);
  const int sc = max(E, 128) - 1080;
  long long M0[4], M1[4], M2s = 0;  // y-sums of each x-node, M1 and M2 times 1/16, 1/32
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const long long x0 = block_fix(v[4 * p], B), x1 = block_fix(v[4 * p + 1], B),
                    x2 = block_fix(v[4 * p + 2], B), x3 = block_fix(v[4 * p + 3], B);
    const long long sA = x0 + x1, dA = x0 - x1, sB = x2 + x3, dB = x2 - x3;
    M0[p] = sA + sB;
    M1[p] = pair_sum16<1>(dB, dA);
    if (k == 0) M2s += pair_sum16<2>(sB, sA);
  }
  const long long a0 = M0[0] + M0[1], b0 = M0[2] + M0[3], c0 = M0[0] - M0[1], d0 = M0[2] - M0[3];
  const double s00 = key < 0x7ff00000u ? fix_to_double(a0 + b0, sc) : __longlong_as_double(0x7ff8000000000000ll);
  const double s10 = fix_to_double(pair_sum16<1>(d0, c0), sc + 4);
  const double s01 = fix_to_double((M1[0] + M1[1]) + (M1[2] + M1[3]), sc + 4);
  if (k == 0) {
    m.m00 = s00; m.m10 = s10; m.m01 = s01;
    m.m20 = fix_to_double(pair_sum16<2>(b0, a0), sc + 5);
    m.m02 = fix_to_double(M2s, sc + 5);
    m.m11 = fix_to_double(pair_sum16<1>((M1[2] - M1[3]) << 4, (M1[0] - M1[1]) << 4), sc + 4);
  } else {
    m.g00 = s00; m.g10 = s10; m.g01 = s01;
  }
}
template <int k, int n>
__device__ __forceinline__ void kqmac(LimbAcc& s, const Limbs& x) {
  s.mac(x.h, x.l, limb_hi(kqf(k, n)), limb_lo(kqf(k, n)));
}
}  // namespace q16

struct Lat16 {
  static constexpr int NQ = 4, POPS = 32, FIELDS = 16, GFIELD = 10, MOMS = 9;
  typedef q16::Mom Mom;
  typedef int NodeK[4][2];
  __device__ static __forceinline__ bool backward(int k) { return (k & 1) != 0; }
  __device__ static __forceinline__ int kdp(int k) { return q16::kdq(k); }
  template <bool NC>
  __device__ static __forceinline__ void moments_f(const double* s, unsigned off, long long PL, Mom& m) {
    q16::moments_fix16<0, NC>(s, off, PL, m);
  }
  template <bool NC>
  __device__ static __forceinline__ void moments_g(const double* s, unsigned off, long long PL, Mom& m) {
    q16::moments_fix16<1, NC>(s, off, PL, m);
  }
  template <int PRC>
  __device__ static __forceinline__ q16::Co coeffs(const Mom& m, const Phys& P) { return q16::coeffs<PRC>(m, P); }
  // fields f00, f10, f01, f20, f11, f02, f30, f21, f12, f03, g00, g10, g01, g20, g11, g02
  __device__ static __forceinline__ void to_smem(const q16::Co& C, long long* b, int& Ef, int& Eg) {
    const double f[10] = {C.f00, C.f10, C.f01, C.f20, C.f11, C.f02, C.f30, C.f21, C.f12, C.f03};
    const double g[6] = {C.g00, C.g10, C.g01, C.g20, C.g11, C.g02};
    fields_to_smem<10>(f, b, Ef);
    fields_to_smem<6>(g, b + 10 * kCta, Eg);
  }
  template <class Put>
  __device__ static __forceinline__ void fields(const q16::Co& C, const Put& put) {
    const double v[16] = {C.f00, C.f10, C.f01, C.f20, C.f11, C.f02, C.f30, C.f21,
                          C.f12, C.f03, C.g00, C.g10, C.g01, C.g20, C.g11, C.g02};
#pragma unroll
    for (int k = 0; k < 16; ++k) put(k, v[k]);
  }
  template <class Put>
  __device__ static __forceinline__ void put(const Mom& m, int k, const Put& put) {
    if (k == 0) {
      put(0, m.m00); put(1, m.m10); put(2, m.m01); put(3, m.m20); put(4, m.m11); put(5, m.m02);
    } else {
      put(6, m.g00); put(7, m.g10); put(8, m.g01);
    }
  }
  template <class Get>
  __device__ static __forceinline__ void get(Mom& m, const Get& get) {
    m.m00 = get(0); m.m10 = get(1); m.m01 = get(2); m.m20 = get(3); m.m11 = get(4); m.m02 = get(5);
    m.g00 = get(6); m.g10 = get(7); m.g01 = get(8);
  }
  __device__ static __forceinline__ void load_k(int p, NodeK& K) {
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      K[n][0] = q16::c_kqf[p][n][0];
      K[n][1] = q16::c_kqf[p][n][1];
    }
  }
  template <class V>
  __device__ static __forceinline__ void target_f(const V& X, const NodeK& K, long long (&t)[4]) {
    LimbAcc a, b, c, d;
    X.mac(a, 0, K[0]); X.mac(a, 1, K[1]); X.mac(a, 3, K[2]); X.mac(a, 6, K[3]);
    X.mac(b, 2, K[0]); X.mac(b, 4, K[1]); X.mac(b, 7, K[2]);
    X.mac(c, 5, K[0]); X.mac(c, 8, K[1]);
    X.mac(d, 9, K[0]);
    const Limbs h0(a.value8()), h1(b.value8()), h2(c.value8()), h3(d.value8());
    LimbAcc ea, oa, eb, ob;
    q16::kqmac<0, 0>(ea, h0); q16::kqmac<0, 2>(ea, h2);
    q16::kqmac<0, 1>(oa, h1); q16::kqmac<0, 3>(oa, h3);
    q16::kqmac<2, 0>(eb, h0); q16::kqmac<2, 2>(eb, h2);
    q16::kqmac<2, 1>(ob, h1); q16::kqmac<2, 3>(ob, h3);
    t[0] = ea.value() + oa.value(); t[1] = ea.value() - oa.value();
    t[2] = eb.value() + ob.value(); t[3] = eb.value() - ob.value();
  }
  template <class V>
  __device__ static __forceinline__ void target_g(const V& X, const NodeK& K, long long (&t)[4]) {
    LimbAcc a, b, c;
    X.mac(a, 10, K[0]); X.mac(a, 11, K[1]); X.mac(a, 13, K[2]);
    X.mac(b, 12, K[0]); X.mac(b, 14, K[1]);
    X.mac(c, 15, K[0]);
    const Limbs h0(a.value8()), h1(b.value8()), h2(c.value8());
    LimbAcc ea, oa, eb, ob;
    q16::kqmac<0, 0>(ea, h0); q16::kqmac<0, 2>(ea, h2);
    q16::kqmac<0, 1>(oa, h1);
    q16::kqmac<2, 0>(eb, h0); q16::kqmac<2, 2>(eb, h2);
    q16::kqmac<2, 1>(ob, h1);
    t[0] = ea.value() + oa.value(); t[1] = ea.value() - oa.value();
    t[2] = eb.value() + ob.value(); t[3] = eb.value() - ob.value();
  }
};

}  // namespace dvbm
