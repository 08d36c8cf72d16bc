// dvbm_lattice.cuh -- what the auxiliary kernels (initial conditions, ghost
// layers, field and total diagnostics) need from a lattice / energy split, so
// that dvbm_aux.cu writes each of those kernels once for both models:
//   L25: D2Q25, internal non-translational energy split (II), FP64 or
//        FP32-deviation storage;
//   L16: D2Q16, total-energy split (I), FP64 storage.
#pragma once
#include "dvbm_cellmom.cuh"
#include "dvbm_internal.h"
#include "dvbm_q16.cuh"

namespace dvbm {

// macroscopic state of one cell: rho, momentum density jx, jy and total energy
// density E (physical units, per unit volume), velocity u and temperature T
struct CellState {
  double rho, jx, jy, E, ux, uy, T;
};

struct L25 {
  static constexpr int NPOP = 50;
  typedef Lat25 Tile;
  // the sums over f and over g of one cell
  template <class S, bool NC = true>
  __device__ static void sum_f(const S* p, long long PL, Moments& m, const Phys& P) {
    moments_fix_f<S, NC>(p, 0u, PL, m);
    if constexpr (sizeof(S) == 4) add_reference_f(m, P);
  }
  template <class S, bool NC = true>
  __device__ static void sum_g(const S* p, long long PL, Moments& m, const Phys& P) {
    moments_fix_g<S, NC>(p, 0u, PL, m);
    if constexpr (sizeof(S) == 4) m.g00 += P.gref0;
  }
  __device__ static CellState state_of(const Moments& m, const Phys& P, const Macro& M) {
    CellState c;
    macro_from_moments(m, P, M.c, M.T_ref, c.rho, c.ux, c.uy, c.T);
    c.jx = m.m10 * M.c;
    c.jy = m.m01 * M.c;
    c.E = m.g00 + 0.5 * P.c2 * (m.m20 + m.m02);  // split II: E = sum g + sum v^2/2 f
    return c;
  }
  template <class S>
  __device__ static CellState state(const S* p, long long PL, const Phys& P, const Macro& M) {
    Moments m;
    sum_f<S>(p, PL, m, P);
    sum_g<S>(p, PL, m, P);
    return state_of(m, P, M);
  }
  // the same in units of c and T_ref, and its equilibrium coefficients
  __device__ static void reduced_state(const Moments& m, const Phys& P, double& rho, double& ux, double& uy,
                                       double& theta) {
    rho = m.m00;
    const double irho = recip(rho);
    ux = m.m10 * irho;
    uy = m.m01 * irho;
    theta = P.gm1 * fma(-0.5, fma(ux, ux, uy * uy), fma(0.5, m.m20 + m.m02, m.g00 * P.inv_c2) * irho);
  }
  __device__ static Coeffs reduced_equilibrium(double rho, double ux, double uy, double theta, const Phys& P) {
    return equilibrium_coeffs(rho, ux, uy, theta, P);
  }
  // equilibrium coefficients of (rho, u, T) (Sec. III.A.3 initial conditions)
  __device__ static Coeffs equilibrium(double rho, double ux, double uy, double T, const Phys& P, const Macro& M) {
    return equilibrium_coeffs(rho, ux / M.c, uy / M.c, T / M.T_ref, P);
  }
};

struct L16 {
  static constexpr int NPOP = 32;
  typedef Lat16 Tile;
  template <class S, bool NC = true>
  __device__ static void sum_f(const S* p, long long PL, q16::Mom& m, const Phys&) {
    static_assert(sizeof(S) == 8, "the D2Q16 / split I model has FP64 storage only");
    q16::moments_fix16<0, NC>(p, 0u, PL, m);
  }
  template <class S, bool NC = true>
  __device__ static void sum_g(const S* p, long long PL, q16::Mom& m, const Phys&) {
    q16::moments_fix16<1, NC>(p, 0u, PL, m);
  }
  __device__ static CellState state_of(const q16::Mom& m, const Phys& P, const Macro& M) {
    CellState c;
    q16::macro(m, P, M.c, M.T_ref, c.rho, c.ux, c.uy, c.T);
    c.jx = m.m10 * M.c;
    c.jy = m.m01 * M.c;
    c.E = m.g00;  // split I: E = sum g
    return c;
  }
  template <class S>
  __device__ static CellState state(const S* p, long long PL, const Phys& P, const Macro& M) {
    q16::Mom m;
    sum_f<S>(p, PL, m, P);
    sum_g<S>(p, PL, m, P);
    return state_of(m, P, M);
  }
  __device__ static void reduced_state(const q16::Mom& m, const Phys& P, double& rho, double& ux, double& uy,
                                       double& theta) {
    rho = m.m00;
    const double irho = recip(rho);
    ux = m.m10 * irho;
    uy = m.m01 * irho;
    theta = P.gm1 * fma(-0.5, fma(ux, ux, uy * uy), m.g00 * P.inv_c2 * irho);
  }
  __device__ static q16::Co reduced_equilibrium(double rho, double ux, double uy, double theta, const Phys& P) {
    return q16::equilibrium(rho, ux, uy, theta, P);
  }
  __device__ static q16::Co equilibrium(double rho, double ux, double uy, double T, const Phys& P, const Macro& M) {
    return q16::equilibrium(rho, ux / M.c, uy / M.c, T / M.T_ref, P);
  }
};

}  // namespace dvbm
