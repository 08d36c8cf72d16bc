// dvbm_internal.h -- launch wrappers shared by the translation units of libdvbm.
#pragma once
#include <cuda_runtime.h>
#include "dvbm_device.cuh"

namespace dvbm {

struct BCDev {
  int kind[4];          // xlo, xhi, ylo, yhi (0 periodic, 1 zero-gradient, 2 wall, 3 external: not filled here)
  double uw[4][2];      // wall velocity
  double Tw[4];         // wall temperature
};

// launch of a kernel that begins with chain_wait
template <class... P, class... A>
inline void launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t st, A... args) {
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = block;
  c.stream = st;
  c.attrs = &at;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, kernel, (P)args...);  // an error is left for cudaGetLastError, as by <<<>>>
}

struct Macro {          // constants needed to turn moments into physical fields
  double c, T_ref, R, gamma;
};

// ghost layers the step kernels write themselves: periodic and zero-gradient sides
inline GhostKinds ghost_kinds(const BCDev& bc) {
  GhostKinds B;
  for (int s = 0; s < 4; ++s) B.k[s] = bc.kind[s];
  return B;
}
// Tile height of the FP64 step.  8 rows share their halo best (2.2 times the rate of
// 2 rows on a full chip); lower tiles spread a small grid over more SMs and shorten
// a tile's serial chain.  4 rows as long as the 8-row tiles fit in one wave (three
// CTAs on each of 152 SMs), 2 rows as long as each SM gets one of them.  Measured,
// periodic, us a step with 2 / 4 / 8 rows.  D2Q25: 64^2 15.7 / 20.6 / 37.4, 96^2
// 16.6 / 20.8 / 37.8, 128^2 30.3 / 21.0 / 37.9, 192^2 58 / 31.6 / 39.3, 224^2
// 81 / 45.7 / 56.5, 288^2 - / 70.4 / 76.4, 352^2 - / 96.4 / 96.8, 416^2 - / 123 / 118,
// 512^2 - / 184 / 160.  D2Q16: 64^2 11.2 / 15.0 / 27.4, 128^2 14.8 / 15.3 / 27.6, 192^2
// 28.0 / 21.6 / 27.4, 288^2 - / 50.1 / 53.8, 352^2 - / 67.7 / 66.4, 512^2 - / 131 / 108.
// A band counts the tiles of the whole grid: a tile's cells share a block exponent,
// so bands of whole 8-row tiles are bitwise the undecomposed run only with its tiles
// (a band of 192 rows of 192 columns then takes 39.3 us a step instead of 31.6 where
// the whole grid has 8-row tiles).
inline long long tiles8(const Geom& G) { return (long long)((G.Nx + 31) / 32) * ((G.grid_rows + 7) / 8); }
inline int tile_rows(const Geom& G) {
  const long long tiles = tiles8(G);
  return 4 * tiles <= 152 ? 2 : tiles <= 3 * 152 ? 4 : 8;
}
// Tile height of the coded adjoint step: 4 rows only while each SM gets one of
// them (the low tiles' kernel has one CTA of 214 registers on an SM, the 8-row
// kernel two of 128).
inline int adjoint_tile_rows(const Geom& G) {
  const long long tiles = tiles8(G);
  return 4 * tiles <= 152 ? 2 : 2 * tiles <= 152 ? 4 : 8;
}
// Does the step kernel write the ghost layers of periodic and zero-gradient sides?
// Then only wall sides are left for launch_ghost, else all.
inline bool step_writes_images(int storage, const Geom& G) { return storage == 0 && tile_rows(G) < 8; }
cudaError_t launch_step(int storage, const void* src, void* dst, const Geom& G, const Phys& P, const BCDev& bc,
                        unsigned int* flag, cudaStream_t st);
// FP64 step with the rational limiter that also records the minmod branch
// codes of every population's x and y slopes: codes[pop][y][x] = x | y << 2
// moms (nullable): also store the 13 moments of each cell of the input state,
// moms[k][y][x] in Moments field order
cudaError_t launch_step_codes(const void* src, void* dst, const Geom& G, const Phys& P, const BCDev& bc,
                              unsigned int* flag, unsigned char* codes, double* moms, cudaStream_t st);
// auxiliary kernels, written once for both models: lattice 0 = D2Q25 / split II
// (storage 0 FP64, 1 FP32-deviation), lattice 1 = D2Q16 / split I (FP64)
cudaError_t launch_init(int lattice, int storage, void* dst, const double* rho, const double* ux, const double* uy,
                        const double* T, const Geom& G, const Phys& P, const Macro& M, cudaStream_t st);
cudaError_t launch_ghost(int lattice, int storage, void* buf, const Geom& G, const Phys& P, const Macro& M,
                         const BCDev& bc, cudaStream_t st);
cudaError_t launch_moments(int lattice, int storage, const void* src, double* rho, double* ux, double* uy, double* T,
                           const Geom& G, const Phys& P, const Macro& M, cudaStream_t st);
// per-block partial sums: out[blk*6 + {mass, momx, momy, energy, bad, 0}]
cudaError_t launch_totals(int lattice, int storage, const void* src, double* partial, int nblocks, const Geom& G,
                          const Phys& P, const Macro& M, cudaStream_t st);
// per-block maxima of |u| + sqrt(gamma R T) and of p = rho R T, and a bad-input count:
// out[blk*3 + {max speed, bad, max p}]
cudaError_t launch_speed(const double* rho, const double* ux, const double* uy, const double* T, long long n,
                         double* partial, int nblocks, const Macro& M, cudaStream_t st);
// halo rows of a slab: unpack = 0: rows y = 0, 1 -> lo and y = Ny - 2, Ny - 1 -> hi;
// unpack = 1: lo -> ghost rows y = -2, -1 and hi -> y = Ny, Ny + 1; layout [npop][2][Nx]
// of elem-byte elements (8: double, 4: float); a NULL buffer skips its side
cudaError_t launch_halo(int elem, void* buf, void* lo, void* hi, int unpack, const Geom& G, int npop,
                        cudaStream_t st);
cudaError_t launch_pack(int storage, const void* buf, void* packed, int to_packed, const Geom& G, int npop,
                        cudaStream_t st);

// D2Q16, total-energy split (I), FP64 storage
cudaError_t launch_step16(const void* src, void* dst, const Geom& G, const Phys& P, const BCDev& bc, unsigned int* flag,
                          cudaStream_t st);

// adjoint (FP64 storage, periodic)
int adjoint_blocks(const Geom& G);
// codes: the branch codes recorded by launch_step_codes for this step, or
// nullptr (the advection adjoint then derives the branches from X)
// glo, ghi: the neighbouring bands' code rows next to a band's edges ([NPOP][Nx]
// each, coded path only), or nullptr: the codes wrap periodically in y
cudaError_t launch_adjoint_step(const double* X, const double* Lin, double* Lout, double* partial,
                                const unsigned char* codes, const double* moms, const Geom& G, const Phys& P,
                                cudaStream_t st, const unsigned char* glo = nullptr,
                                const unsigned char* ghi = nullptr);
// branch-code rows of a band's edges: unpack = 0: rows y = 0 -> lo, y = Ny - 1 -> hi of
// every population's codes; unpack = 1: lo -> glo, hi -> ghi; [NPOP][Nx] bytes, NULL skips
cudaError_t launch_code_rows(unsigned char* codes, void* lo, void* hi, unsigned char* glo, unsigned char* ghi,
                             int unpack, const Geom& G, cudaStream_t st);
cudaError_t launch_adjoint_final(const double* X, const double* rhob, const double* Tb, double* Lout, double* partial,
                                 const Geom& G, const Phys& P, const Macro& M, cudaStream_t st);
cudaError_t launch_adjoint_init(const double* L, const double* rho, const double* ux, const double* uy,
                                const double* T, double* grho, double* gux, double* guy, double* gT, double* partial,
                                const Geom& G, const Phys& P, const Macro& M, cudaStream_t st);

}  // namespace dvbm
