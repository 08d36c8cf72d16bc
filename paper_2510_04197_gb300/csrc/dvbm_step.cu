// dvbm_step.cu -- the fused time step (Sec. III.A.1, Eq. finalDiscretePDE):
//     F_new = (1 - dt/tau1) F + W W sum C He He - (dt/dx) v_x dF_x - (dt/dy) v_y dF_y
// over 32 x 8-cell tiles: moments, combined collision coefficients, the
// collision target of every population (sum-factorised Grad expansion) and its
// upwind-limited flux differences.  GB300 has two FP64 lanes per SM, so FP64
// storage does all of this but the collision coefficients in fixed point on the
// integer pipes (k_step64); FP32-deviation storage keeps float deviations from
// a reference state, with the advection in float (k_step32).
#include "dvbm_device.cuh"
#include "dvbm_internal.h"

namespace dvbm {

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
__constant__ int c_kf[5][5][2] = {
#define KF(k, n) {limb_hi(kf(k, n)), limb_lo(kf(k, n))}
#define KROW(k) {KF(k, 0), KF(k, 1), KF(k, 2), KF(k, 3), KF(k, 4)}
    KROW(0), KROW(1), KROW(2), KROW(3), KROW(4)};

// This thread's collision coefficients in block fixed point (60 bits, one
// exponent for f, one for g) as limb pairs in shared memory: field k of thread
// t at [k * kCta + t] (consecutive threads, consecutive words; registers would
// hold 42 words across the node loop).  Field order f00, f10, f01, f20, f11,
// f02, f30, f21, f12, f03, f40, f31, f22, f13, f04, g00, g10, g01, g20, g11, g02.
constexpr int kFixFields = 21;
struct FixView {
  const long long* b;
  __device__ __forceinline__ void mac(LimbAcc& s, int field, const int (&k)[2]) const {
    const long long x = b[field * kCta];
    s.mac((int)(x >> 32), (int)x, k[0], k[1]);
  }
};
__device__ __forceinline__ void coeffs_to_smem(const Coeffs& C, long long* b, int& Ef, int& Eg) {
  const double f[15] = {C.f00, C.f10, C.f01, C.f20, C.f11, C.f02, C.f30, C.f21,
                        C.f12, C.f03, C.f40, C.f31, C.f22, C.f13, C.f04};
  const double g[6] = {C.g00, C.g10, C.g01, C.g20, C.g11, C.g02};
  unsigned kf_ = 0, kg_ = 0;
#pragma unroll
  for (int k = 0; k < 15; ++k) kf_ = max(kf_, abs_key(f[k]));
#pragma unroll
  for (int k = 0; k < 6; ++k) kg_ = max(kg_, abs_key(g[k]));
  Ef = (int)(kf_ >> 20);
  Eg = (int)(kg_ >> 20);
  const int nf = Ef < 128 ? 63 : 0, ng = Eg < 128 ? 63 : 0;  // negligible coefficients: target 0
#pragma unroll
  for (int k = 0; k < 15; ++k) b[k * kCta] = pack_limbs(block_fix(f[k], Ef, nf));
#pragma unroll
  for (int k = 0; k < 6; ++k) b[(15 + k) * kCta] = pack_limbs(block_fix(g[k], Eg, ng));
}

// h^b of x-node p: W_p sum_a C_ab He_a(xi_p)/a! (value h 2^(E - 1082 - kd(p)))
__device__ __forceinline__ void hf_node(const FixView& X, const int (&K)[5][2], long long (&h)[5]) {
  LimbAcc a, b, c, d, e;
  X.mac(a, 0, K[0]); X.mac(a, 1, K[1]); X.mac(a, 3, K[2]); X.mac(a, 6, K[3]); X.mac(a, 10, K[4]);
  X.mac(b, 2, K[0]); X.mac(b, 4, K[1]); X.mac(b, 7, K[2]); X.mac(b, 11, K[3]);
  X.mac(c, 5, K[0]); X.mac(c, 8, K[1]); X.mac(c, 12, K[2]);
  X.mac(d, 9, K[0]); X.mac(d, 13, K[1]);
  X.mac(e, 14, K[0]);
  h[0] = a.value8(); h[1] = b.value8(); h[2] = c.value8(); h[3] = d.value8(); h[4] = e.value8();
}
__device__ __forceinline__ void hg_node(const FixView& X, const int (&K)[5][2], long long (&h)[3]) {
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

// ---- FP64 storage ------------------------------------------------------------
// Two phases per 32 x 8 tile.  Advection, one population per warp: the warp
// walks the tile and writes the flux sums (advect_tile) as integers into the new
// state's space, from where they come back out of L2.  Collision, one cell per
// thread: moments, combined coefficients, the collision target of each
// population in fixed point, and the update with the flux sum (collide_advect).
// In the advection warp w does f (w < 4) or g of x-node p = 1 + w % 4: the four
// populations that move along both axes, (p, 0) along x only and (0, p) along y
// only, so that all eight warps have the same work; the resting population
// needs none.
// What bounds it: the integer ALU (about two thirds busy) beside the FP64 pipe
// (about half) and the latency between them; DRAM is at a fifth of its rate.
// 12.4 k instructions and 186 FP64 ones a cell, against 26.8 k and 407 of a
// thread per cell with its own stencils: 15.5 -> 8.5 ms a step at 4096^2, 1.02 ->
// 0.57 ms at 1024^2.  Three CTAs of 80 registers; four of 64 measured 1 % slower.
template <int PRC, bool RAT, bool CODES>
__global__ void __launch_bounds__(kCta, 3) k_step64(const double* __restrict__ src, double* dst, Geom G, Phys P,
                                                    unsigned int* __restrict__ flag, unsigned char* codes,
                                                    double* __restrict__ moms) {
  __shared__ long long s_buf[kFixFields * kCta];  // the advection's tiles, then the collision coefficients
  __shared__ int s_exp[NPOP];                     // block exponents of the flux sums
  static_assert(8 * kAdvRows * kAdvPitch <= kFixFields * kCta, "the advection tiles fit the coefficients' space");
  const int x0 = blockIdx.x * 32, y0 = blockIdx.y * kTileY;
  const long long PL = G.plane;
  const long long PT = G.pitch;
  const long long cplane = (long long)G.Nx * G.Ny;
  const double* stile = src + cell_index(G, y0, x0);
  double* dtile = dst + cell_index(G, y0, x0);
  {
    const int w = __shfl_sync(0xffffffffu, (int)threadIdx.y, 0), c0 = 25 * (w >> 2), p = 1 + (w & 3);
    AdvTile T;
    T.W = min(32, G.Nx - x0);
    T.H = min(kTileY, G.Ny - y0);
    T.lane = threadIdx.x;
    long long* xs = s_buf + w * (kAdvRows * kAdvPitch);
    unsigned char* ctile = CODES ? codes + (long long)y0 * G.Nx + x0 : nullptr;
    int E;
    AdvLoad L;
    // the walk directions of population (p, q): sign of each velocity component
    auto tile = [&](int pp, int q) {
      AdvTile t = T;
      t.fx = pp != 0 && (pp & 1) == 0;
      t.fy = q != 0 && (q & 1) == 0;
      return t;
    };
    auto load = [&](int pp, int q) {
      advect_load(L, stile + (c0 + 5 * pp + q) * PL, PT, tile(pp, q));
    };
    auto out = [&](int c) { return (long long*)(dtile + c * PL); };
    auto code = [&](int c) { return CODES ? ctile + c * cplane : nullptr; };
    load(p, 0);
    {
      const int c = c0 + 5 * p;
      E = advect_tile<true, false, RAT, CODES>(L, [&] { load(p, 1); }, out(c), PT, tile(p, 0), P, P.kxq[p], 0, xs, code(c),
                                               G.Nx);
      if (T.lane == 0) s_exp[c] = E;
    }
#pragma unroll 1
    for (int q = 1; q < 5; ++q) {
      const int c = c0 + 5 * p + q;
      E = advect_tile<true, true, RAT, CODES>(L, [&] { load(q < 4 ? p : 0, q < 4 ? q + 1 : p); }, out(c), PT, tile(p, q), P,
                                              P.kxq[p], P.kyq[q], xs, code(c), G.Nx);
      if (T.lane == 0) s_exp[c] = E;
    }
    {
      const int c = c0 + p;
      E = advect_tile<false, true, RAT, CODES>(L, [] {}, out(c), PT, tile(0, p), P, 0, P.kyq[p], xs, code(c), G.Nx);
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
  }
  __syncthreads();
  const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
  if (x >= G.Nx || y >= G.Ny) return;
  const unsigned off = (threadIdx.y * (unsigned)PT + threadIdx.x) * 8u;  // this cell's byte offset in the tile
  const Moments m = moments_fix<double>(stile, off, PL);
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
  const Coeffs C = collision_coeffs<PRC>(m, P);
  if (C.bad) atomicOr(flag, 1u);
  const int tid = threadIdx.y * 32 + threadIdx.x;
  int Ef, Eg;
  coeffs_to_smem(C, s_buf + tid, Ef, Eg);
  const FixView X{s_buf + tid};
  const double a1 = C.a1;
#pragma unroll 1
  for (int p = 0; p < 5; ++p) {
    int K[5][2];
    load_kf(p, K);
    const int dp = p == 0 ? 0 : (p <= 2 ? kd(1) : kd(3));
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const double* sp = stile + (25 * k + 5 * p) * PL;
      double* dp_ = dtile + (25 * k + 5 * p) * PL;
      double F[5];
      long long W[5], t[5];
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        F[q] = __ldg(at(sp + q * PL, off));
        W[q] = *at((const long long*)dp_ + q * PL, off);
      }
      if (k == 0) {
        long long h[5];
        hf_node(X, K, h);
        expand_node(h, t);
      } else {
        long long h[3];
        hg_node(X, K, h);
        expand_node(h, t);
      }
      const int st = (k == 0 ? Ef : Eg) - dp;
#pragma unroll
      for (int q = 0; q < 5; ++q)
        *at(dp_ + q * PL, off) = collide_advect(a1, F[q], t[q], st - kd(q), W[q], s_exp[25 * k + 5 * p + q]);
    }
  }
}

// ---- FP32-deviation storage ----------------------------------------------------
// One thread per cell: moments and coefficients as above, the collision target
// of each population rounded to float, the upwind-limited flux differences in
// float on the deviations from L1-cached neighbours.
// The ten populations (f and g, y-nodes q = 0..4) of x-node p; CENTER: p = 0
// (xi_x = 0, no x-flux), otherwise p = 1..4 at run time, so that one copy of
// this body serves the four moving x-nodes and the kernel's code stays small
// enough for the instruction cache.  The y-node loop stays unrolled (1754 vs
// 1722 MLUPS rolled at 4096^2).
template <bool CENTER>
__device__ __forceinline__ void node_update32(int p, const float* __restrict__ s, float* __restrict__ d, long long PL,
                                              long long PT, const FixView& X, int Ef, int Eg, const Phys& P, float a1f) {
  const int dp = (CENTER || p == 0) ? 0 : (p <= 2 ? kd(1) : kd(3));
  float tf[5], tg[5];
  {
    int K[5][2];
    load_kf(p, K);
    long long hf[5], hg[3], t[5];
    hf_node(X, K, hf);
    expand_node(hf, t);
#pragma unroll
    for (int q = 0; q < 5; ++q) tf[q] = ll_to_float_rn(t[q], Ef - 1079 - dp - kd(q));
    hg_node(X, K, hg);
    expand_node(hg, t);
#pragma unroll
    for (int q = 0; q < 5; ++q) tg[q] = ll_to_float_rn(t[q], Eg - 1079 - dp - kd(q));
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
                                                             Geom G, Phys P, unsigned int* __restrict__ flag) {
  const int x = blockIdx.x * 32 + threadIdx.x;
  const int y = blockIdx.y * kTileY + threadIdx.y;
  if (x >= G.Nx || y >= G.Ny) return;
  const long long off = cell_index(G, y, x);
  const float* s = src + off;
  float* d = dst + off;
  const long long PL = G.plane;
  const long long PT = G.pitch;
  Moments m = moments_fix<float>(s, 0u, PL);
  // moments of the reference populations w rho0 (f) and w G0 (g):
  // sum w = 1, sum w xi^2 = 1 per axis, odd moments vanish
  m.m00 += P.fref0; m.m20 += P.fref0; m.m02 += P.fref0;
  m.g00 += P.gref0;
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
  __shared__ long long s_fix[kFixFields * kCta];
  const int tid = threadIdx.y * 32 + threadIdx.x;
  int Ef, Eg;
  coeffs_to_smem(C, s_fix + tid, Ef, Eg);
  const FixView X{s_fix + tid};
  node_update32<true>(0, s, d, PL, PT, X, Ef, Eg, P, a1f);
#pragma unroll 1
  for (int p = 1; p < 5; ++p) node_update32<false>(p, s, d, PL, PT, X, Ef, Eg, P, a1f);
}

template <bool RAT, bool CODES>
static void launch_step64(dim3 grid, dim3 block, const double* s, double* d, const Geom& G, const Phys& P,
                          unsigned int* flag, unsigned char* codes, double* moms, cudaStream_t st) {
  if (P.prc < 0) k_step64<-1, RAT, CODES><<<grid, block, 0, st>>>(s, d, G, P, flag, codes, moms);
  else if (P.prc > 0) k_step64<1, RAT, CODES><<<grid, block, 0, st>>>(s, d, G, P, flag, codes, moms);
  else k_step64<0, RAT, CODES><<<grid, block, 0, st>>>(s, d, G, P, flag, codes, moms);
}

cudaError_t launch_step_codes(const void* src, void* dst, const Geom& G, const Phys& P, unsigned int* flag,
                              unsigned char* codes, double* moms, cudaStream_t st) {
  if (!(P.lq > 0) || !codes) return cudaErrorInvalidValue;
  dim3 block(32, kTileY);
  dim3 grid((G.Nx + 31) / 32, (G.Ny + kTileY - 1) / kTileY);
  launch_step64<true, true>(grid, block, (const double*)src, (double*)dst, G, P, flag, codes, moms, st);
  return cudaGetLastError();
}

cudaError_t launch_step(int storage, const void* src, void* dst, const Geom& G, const Phys& P, unsigned int* flag,
                        cudaStream_t st) {
  dim3 block(32, kTileY);
  dim3 grid((G.Nx + 31) / 32, (G.Ny + kTileY - 1) / kTileY);
  if (storage == 0) {
    if (P.lq > 0) launch_step64<true, false>(grid, block, (const double*)src, (double*)dst, G, P, flag, nullptr, nullptr, st);
    else launch_step64<false, false>(grid, block, (const double*)src, (double*)dst, G, P, flag, nullptr, nullptr, st);
  } else {
    const float* s = (const float*)src;
    float* d = (float*)dst;
    if (P.prc < 0) k_step32<-1><<<grid, block, 0, st>>>(s, d, G, P, flag);
    else if (P.prc > 0) k_step32<1><<<grid, block, 0, st>>>(s, d, G, P, flag);
    else k_step32<0><<<grid, block, 0, st>>>(s, d, G, P, flag);
  }
  return cudaGetLastError();
}

}  // namespace dvbm
