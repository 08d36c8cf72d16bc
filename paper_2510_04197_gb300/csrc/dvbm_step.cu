// dvbm_step.cu -- the fused time step (Sec. III.A.1, Eq. finalDiscretePDE):
//     F_new = (1 - dt/tau1) F + W W sum C He He - (dt/dx) v_x dF_x - (dt/dy) v_y dF_y
// over tiles of cells: moments, combined collision coefficients, the
// collision target of every population (sum-factorised Grad expansion) and its
// upwind-limited flux differences.  GB300 has two FP64 lanes per SM, so FP64
// storage does all of this but the collision coefficients in fixed point on the
// integer pipes (k_step_tile); FP32-deviation storage keeps float deviations from
// a reference state, with the advection in float (k_step32).
#include "dvbm_device.cuh"
#include "dvbm_internal.h"

namespace dvbm {

// ---- FP32-deviation storage ----------------------------------------------------
// One thread per cell: moments and coefficients as above, the collision target
// of each population rounded to float, the upwind-limited flux differences in
// float on the deviations from L1-cached neighbours.
// the five targets t_q 2^(scale - kd(q)) of an x-node as floats: the hardware's
// conversion (one slot of the FP64 pipe, which this kernel does not fill, for
// about fifteen integer instructions) and two exact power-of-two factors
__device__ __forceinline__ float pow2f(int e) { return __int_as_float(min(max(e + 127, 0), 254) << 23); }
__device__ __forceinline__ void to_floats(const long long (&t)[5], int scale, float (&f)[5]) {
  const int s1 = scale >> 1;
  const float m1 = pow2f(s1), m2 = pow2f(scale - s1);
#pragma unroll
  for (int q = 0; q < 5; ++q) f[q] = (__ll2float_rn(t[q]) * m1) * (m2 * (1.0f / (float)(1 << kd(q))));
}

// The ten populations (f and g, y-nodes q = 0..4) of x-node p; CENTER: p = 0
// (xi_x = 0, no x-flux), otherwise p = 1..4 at run time, so that one copy of
// this body serves the four moving x-nodes and the kernel's code stays small
// enough for the instruction cache.  The y-node loop stays unrolled (rolled it
// measured 2 % slower at 4096^2).
template <bool CENTER>
__device__ __forceinline__ void node_update32(int p, const float* __restrict__ s, float* __restrict__ d, const Geom& G,
                                              const FixView& X, int Ef, int Eg, const Phys& P, float a1f) {
  const long long PL = G.plane, PT = G.pitch;
  const int dp = (CENTER || p == 0) ? 0 : (p <= 2 ? kd(1) : kd(3));
  float tf[5], tg[5];
  {
    int K[5][2];
    load_kf(p, K);
    long long hf[5], hg[3], t[5];
    hf_node(X, K, hf);
    expand_node(hf, t);
    to_floats(t, Ef - 1079 - dp, tf);
    hg_node(X, K, hg);
    expand_node(hg, t);
    to_floats(t, Eg - 1079 - dp, tg);
  }
  // x-node sign and flux factor (p = 1, 3: +xi; p = 2, 4: -xi); warp-uniform selects
  const int sx = (p & 1) ? 1 : -1;
  const int pa = (p + 1) >> 1;  // 1 for p = 1, 2; 2 for p = 3, 4
  float kxf = 0.f;
  if (!CENTER) kxf = (pa == 1 ? P.kxvf[1] : P.kxvf[3]) * (float)sx;
  const float hb = (float)P.hb;
  const long long pbase = (long long)(5 * p) * PL;
#pragma unroll 1
  for (int k = 0; k < 2; ++k) {  // f then g: one copy of the body for both
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      const long long co = pbase + (long long)(q + 25 * k) * PL;
      const float t = k == 0 ? tf[q] : tg[q];
      const float* pc = s + co;
      float fx = 0, fy = 0;
      if (!CENTER) fx = sx > 0 ? flux_difference<1, float>(pc, 1, hb) : flux_difference<-1, float>(pc, 1, hb);
      if (sgn_of(q) > 0) fy = flux_difference<1, float>(pc, PT, hb);
      if (sgn_of(q) < 0) fy = flux_difference<-1, float>(pc, PT, hb);
      float adv = 0.f;
      if (!CENTER) adv = kxf * fx;
      if (sgn_of(q) != 0) adv = fmaf(P.kyvf[q], fy, adv);
      d[co] = fmaf(a1f, __ldg(pc), t) - adv;
    }
  }
}

template <int PRC>
__global__ void __launch_bounds__(kCta, 1024 / kCta) k_step32(const float* __restrict__ src, float* __restrict__ dst,
                                                             Geom G, Phys P,
                                                             unsigned int* __restrict__ flag) {
  const int x = blockIdx.x * 32 + threadIdx.x;
  const int y = blockIdx.y * 8 + threadIdx.y;
  if (x >= G.Nx || y >= G.Ny) return;
  const long long off = cell_index(G, y, x);
  const float* s = src + off;
  float* d = dst + off;
  const long long PL = G.plane;
  Moments m = moments_fix<float>(s, 0u, PL);
  add_reference(m, P);
  Coeffs C = collision_coeffs<PRC>(m, P);
  if (C.bad) atomicOr(flag, 1u);
  // the expansion then yields t - (dt/tau1) F_ref directly: the reference
  // populations w rho0 and w G0 have only a zeroth Hermite coefficient
  C.f00 -= C.k1 * P.fref0;
  C.g00 -= C.k1 * P.gref0;
  // new deviation = a1 * dev + (t - k1 * ref) - advection, with the bracket
  // (equilibrium evaluation minus the relaxed reference) at FP64-or-better
  // precision, rounded to float only in the update
  const float a1f = (float)C.a1;
  __shared__ long long s_fix[Lat25::FIELDS * kCta];
  const int tid = threadIdx.y * 32 + threadIdx.x;
  int Ef, Eg;
  Lat25::to_smem(C, s_fix + tid, Ef, Eg);
  const FixView X{s_fix + tid};
  node_update32<true>(0, s, d, G, X, Ef, Eg, P, a1f);
#pragma unroll 1
  for (int p = 1; p < 5; ++p) node_update32<false>(p, s, d, G, X, Ef, Eg, P, a1f);
}

template <int R, bool RAT, bool CODES>
static void launch_tile(const double* s, double* d, const Geom& G, const Phys& P, const GhostKinds& B, unsigned int* flag,
                        unsigned char* codes, double* moms, cudaStream_t st) {
  const dim3 block(32, 8), grid((G.Nx + 31) / 32, (G.Ny + R - 1) / R);
  const auto k = P.prc < 0   ? k_step_tile<Lat25, R, -1, RAT, CODES>
                 : P.prc > 0 ? k_step_tile<Lat25, R, 1, RAT, CODES>
                             : k_step_tile<Lat25, R, 0, RAT, CODES>;
  if (R < 8) launch_chained(k, grid, block, st, s, d, G, P, B, flag, codes, moms);
  else k<<<grid, block, 0, st>>>(s, d, G, P, B, flag, codes, moms);
}
template <bool RAT, bool CODES>
static void launch_tiles(const double* s, double* d, const Geom& G, const Phys& P, const GhostKinds& B,
                         unsigned int* flag, unsigned char* codes, double* moms, cudaStream_t st) {
  const int R = tile_rows(G);
  if (R == 8) launch_tile<8, RAT, CODES>(s, d, G, P, B, flag, codes, moms, st);
  else if (R == 4) launch_tile<4, RAT, CODES>(s, d, G, P, B, flag, codes, moms, st);
  else launch_tile<2, RAT, CODES>(s, d, G, P, B, flag, codes, moms, st);
}

cudaError_t launch_step_codes(const void* src, void* dst, const Geom& G, const Phys& P, const BCDev& bc,
                              unsigned int* flag, unsigned char* codes, double* moms, cudaStream_t st) {
  if (!(P.lq > 0) || !codes) return cudaErrorInvalidValue;
  launch_tiles<true, true>((const double*)src, (double*)dst, G, P, ghost_kinds(bc), flag, codes, moms, st);
  return cudaGetLastError();
}

cudaError_t launch_step(int storage, const void* src, void* dst, const Geom& G, const Phys& P, const BCDev& bc,
                        unsigned int* flag, cudaStream_t st) {
  const GhostKinds B = ghost_kinds(bc);
  if (storage == 0) {
    const double* s = (const double*)src;
    double* d = (double*)dst;
    if (P.lq > 0) launch_tiles<true, false>(s, d, G, P, B, flag, nullptr, nullptr, st);
    else launch_tiles<false, false>(s, d, G, P, B, flag, nullptr, nullptr, st);
  } else {
    const dim3 block(32, 8), grid((G.Nx + 31) / 32, (G.Ny + 7) / 8);
    const float* s = (const float*)src;
    float* d = (float*)dst;
    if (P.prc < 0) k_step32<-1><<<grid, block, 0, st>>>(s, d, G, P, flag);
    else if (P.prc > 0) k_step32<1><<<grid, block, 0, st>>>(s, d, G, P, flag);
    else k_step32<0><<<grid, block, 0, st>>>(s, d, G, P, flag);
  }
  return cudaGetLastError();
}

}  // namespace dvbm
