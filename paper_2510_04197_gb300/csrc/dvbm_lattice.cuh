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
  template <class S>
  __device__ static CellState state(const S* p, long long PL, const Phys& P, const Macro& M) {
    Moments m = moments_fix<S>(p, 0u, PL);
    if constexpr (sizeof(S) == 4) add_reference(m, P);
    CellState c;
    macro_from_moments(m, P, M.c, M.T_ref, c.rho, c.ux, c.uy, c.T);
    c.jx = m.m10 * M.c;
    c.jy = m.m01 * M.c;
    c.E = m.g00 + 0.5 * P.c2 * (m.m20 + m.m02);  // split II: E = sum g + sum v^2/2 f
    return c;
  }
  // equilibrium coefficients of (rho, u, T) (Sec. III.A.3 initial conditions)
  __device__ static Coeffs equilibrium(double rho, double ux, double uy, double T, const Phys& P, const Macro& M) {
    return equilibrium_coeffs(rho, ux / M.c, uy / M.c, T / M.T_ref, P);
  }
  __device__ static void subtract(Coeffs& A, const Coeffs& B) {
    A.f00 -= B.f00; A.f10 -= B.f10; A.f01 -= B.f01; A.f20 -= B.f20; A.f11 -= B.f11; A.f02 -= B.f02; A.f30 -= B.f30;
    A.f21 -= B.f21; A.f12 -= B.f12; A.f03 -= B.f03; A.f40 -= B.f40; A.f31 -= B.f31; A.f22 -= B.f22; A.f13 -= B.f13;
    A.f04 -= B.f04;
    A.g00 -= B.g00; A.g10 -= B.g10; A.g01 -= B.g01; A.g20 -= B.g20; A.g11 -= B.g11; A.g02 -= B.g02;
  }
};

struct L16 {
  static constexpr int NPOP = 32;
  typedef Lat16 Tile;
  template <class S>
  __device__ static CellState state(const S* p, long long PL, const Phys& P, const Macro& M) {
    static_assert(sizeof(S) == 8, "the D2Q16 / split I model has FP64 storage only");
    const q16::Mom m = q16::moments_fix16(p, 0u, PL);
    CellState c;
    q16::macro(m, P, M.c, M.T_ref, c.rho, c.ux, c.uy, c.T);
    c.jx = m.m10 * M.c;
    c.jy = m.m01 * M.c;
    c.E = m.g00;  // split I: E = sum g
    return c;
  }
  __device__ static q16::Co equilibrium(double rho, double ux, double uy, double T, const Phys& P, const Macro& M) {
    return q16::equilibrium(rho, ux / M.c, uy / M.c, T / M.T_ref, P);
  }
  __device__ static void subtract(q16::Co& A, const q16::Co& B) {
    A.f00 -= B.f00; A.f10 -= B.f10; A.f01 -= B.f01; A.f20 -= B.f20; A.f11 -= B.f11; A.f02 -= B.f02;
    A.f30 -= B.f30; A.f21 -= B.f21; A.f12 -= B.f12; A.f03 -= B.f03;
    A.g00 -= B.g00; A.g10 -= B.g10; A.g01 -= B.g01; A.g20 -= B.g20; A.g11 -= B.g11; A.g02 -= B.g02;
  }
};

}  // namespace dvbm
