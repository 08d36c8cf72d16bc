// dvbm_d2q16.cu -- the time step with the total-energy split (I) on D2Q16: the
// tiled FP64 step of dvbm_device.cuh (k_step_tile) on the lattice traits Lat16 of
// dvbm_q16.cuh.
#include "dvbm_internal.h"
#include "dvbm_q16.cuh"

namespace dvbm {

template <int R, bool RAT>
static void launch_tile16(const double* s, double* d, const Geom& G, const Phys& P, const GhostKinds& B,
                          unsigned int* flag, cudaStream_t st) {
  const dim3 block(32, 8), grid((G.Nx + 31) / 32, (G.Ny + R - 1) / R);
  const auto k = P.prc < 0   ? k_step_tile<Lat16, R, -1, RAT, false>
                 : P.prc > 0 ? k_step_tile<Lat16, R, 1, RAT, false>
                             : k_step_tile<Lat16, R, 0, RAT, false>;
  unsigned char* codes = nullptr;
  double* moms = nullptr;
  if (R < 8) launch_chained(k, grid, block, st, s, d, G, P, B, flag, codes, moms);
  else k<<<grid, block, 0, st>>>(s, d, G, P, B, flag, codes, moms);
}

cudaError_t launch_step16(const void* src, void* dst, const Geom& G, const Phys& P, const BCDev& bc, unsigned int* flag,
                          cudaStream_t st) {
  const double* s = (const double*)src;
  double* d = (double*)dst;
  const GhostKinds B = ghost_kinds(bc);
  const bool rat = P.lq > 0;
  const int R = tile_rows(G);
  if (rat) {
    if (R == 8) launch_tile16<8, true>(s, d, G, P, B, flag, st);
    else if (R == 4) launch_tile16<4, true>(s, d, G, P, B, flag, st);
    else launch_tile16<2, true>(s, d, G, P, B, flag, st);
  } else {
    if (R == 8) launch_tile16<8, false>(s, d, G, P, B, flag, st);
    else if (R == 4) launch_tile16<4, false>(s, d, G, P, B, flag, st);
    else launch_tile16<2, false>(s, d, G, P, B, flag, st);
  }
  return cudaGetLastError();
}

}  // namespace dvbm
