// dvbm_aux.cu -- initial conditions, ghost layers, diagnostics.
//
// Each kernel below is written once for both models: templated on the
// lattice traits L25 / L16 of dvbm_lattice.cuh and on the storage type.
//
//  k_init     equilibrium populations of given (rho, u, T) fields (Sec. III.A.3),
//             by the step kernels' block-fixed-point Grad expansion
//  k_ghost    two ghost layers per side: periodic wrap or zero-gradient copy
//  k_wall     the ghost layers of no-slip isothermal walls by ghost node +
//             non-equilibrium extrapolation (Sec. III.E): rho_G = rho_B, u_G = 2 u_W - u_B,
//             T_G = 2 T_W - T_B, F_G = F^eq(G) + (F_B - F^eq(B)); ghost k
//             mirrors interior cell k (k = 1, 2)
//  k_moments  rho, u, T fields
//  k_totals   per-block sums of mass, momentum, total energy (+ bad-cell count)
//  k_speed    per-block maxima of |u| + sqrt(gamma R T) (CFL rule) and of p = rho R T
//             (shortest relaxation time), and a bad-input count
//  k_pack     padded <-> packed [50][Ny][Nx] state copies
#include "dvbm_lattice.cuh"

namespace dvbm {

// Bound by the integer pipes (about 3 k instructions a cell: equilibrium
// coefficients in FP64, 21 of them to fixed point, the expansion by limb
// products, 50 conversions); the whole dvbm_init call 6.5 -> 3.4 ms at 4096^2 FP64, of which 1 ms is the write.
template <class L, class S>
__global__ void __launch_bounds__(kCta, 3) k_init(S* __restrict__ dst, const double* __restrict__ rho,
                                               const double* __restrict__ ux, const double* __restrict__ uy,
                                               const double* __restrict__ T, Geom G, Phys P, Macro M) {
  typedef typename L::Tile LT;
  constexpr int NQ = LT::NQ, NF = NQ * NQ;
  __shared__ long long s_buf[LT::FIELDS * kCta];
  const int x = blockIdx.x * 32 + threadIdx.x;
  const int y = blockIdx.y * 8 + threadIdx.y;
  if (x >= G.Nx || y >= G.Ny) return;
  const long long i = (long long)y * G.Nx + x;
  long long* b = s_buf + threadIdx.y * 32 + threadIdx.x;
  int Ef, Eg;
  {
    auto C = L::equilibrium(rho[i], ux[i], uy[i], T[i], P, M);
    if constexpr (sizeof(S) == 4) {
      // the reference populations w rho0 and w G0 carry only a zeroth Hermite
      // coefficient: without it the expansion yields the deviations
      C.f00 -= P.fref0;
      C.g00 -= P.gref0;
    }
    LT::to_smem(C, b, Ef, Eg);
  }
  const FixView X{b};
  const long long PL = G.plane;
  S* d = dst + cell_index(G, y, x);
#pragma unroll 1
  for (int p = 0; p < NQ; ++p) {
    typename LT::NodeK K;
    LT::load_k(p, K);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      long long t[NQ];
      if (k == 0) LT::target_f(X, K, t);
      else LT::target_g(X, K, t);
      const int sc = (k == 0 ? Ef : Eg) - 1079 - LT::kdp(p);
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        S* o = d + (NF * k + NQ * p + q) * PL;
        if constexpr (sizeof(S) == 8) *o = fix_to_double(t[q], sc - LT::kdp(q));
        else *o = ll_to_float_rn(t[q], sc - LT::kdp(q));
      }
    }
  }
}

// Ghost layer k (1 or 2) of position j along a side: the ghost cell (gx, gy) and its
// source, by kind: periodic wrap, zero gradient, or a wall's mirror cell (ghost k
// mirrors interior cell k).  Sides 0..3 = xlo, xhi, ylo, yhi.
__device__ __forceinline__ void ghost_cells(int side, int kind, int k, int j, const Geom& G, int& gx, int& gy, int& bx,
                                            int& by) {
  const bool lo = (side % 2) == 0;
  const int n = side < 2 ? G.Nx : G.Ny;
  const int gi = lo ? -k : n - 1 + k;  // coordinate along the normal
  int bi;
  if (kind == 0) bi = lo ? n - k : k - 1;
  else if (kind == 1) bi = lo ? 0 : n - 1;
  else bi = lo ? k - 1 : n - k;
  if (side < 2) { gx = gi; gy = j; bx = bi; by = j; }
  else          { gx = j; gy = gi; bx = j; by = bi; }
}

// periodic and zero-gradient sides, one thread per (side, layer, position, population)
template <class S>
__global__ void k_ghost(S* __restrict__ buf, Geom G, BCDev bc) {
  buf = chain_wait(buf);
  const int side = blockIdx.y, kind = bc.kind[side], pop = blockIdx.z;
  if (kind > 1) return;
  const int len = side < 2 ? G.Ny : G.Nx;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 2 * len) return;
  int gx, gy, bx, by;
  ghost_cells(side, kind, 1 + t / len, t % len, G, gx, gy, bx, by);
  buf[pop * G.plane + cell_index(G, gy, gx)] = buf[pop * G.plane + cell_index(G, by, bx)];
}

// Isothermal no-slip walls: F_G = F^eq(rho_B, 2 u_W - u_B, 2 T_W - T_B) + (F_B - F^eq(B)),
// i.e. F_B plus the expansion of the difference of the two equilibria's
// coefficients, in the step kernels' fixed point.  The work is small and all
// latency, FP64 chains first (one FP64 warp instruction occupies its scheduler's
// pipe for 64 cycles), so a ghost cell has one thread in each of the block's
// eight warps: warps 0 and 1 sum f and g, then form the equilibria of the mirror
// cell and of the ghost, then bring the differences to fixed point (f, g); all
// share the populations (units of an x-node's f or g).  Velocities and temperatures
// are in units of c and T_ref (bc's too), which spares four FP64 divisions
// a cell (a step there 28.1 -> 25.7 us).  At 4 x 256 one thread a
// cell took 33 us of a 55 us step; this takes 11.
template <class L, class S>
__global__ void __launch_bounds__(kCta, 2) k_wall(S* __restrict__ buf, Geom G, Phys P, BCDev bc) {
  typedef typename L::Tile LT;
  constexpr int NQ = LT::NQ, NF = NQ * NQ, N = LT::FIELDS;
  __shared__ long long s_fix[N * 32];
  __shared__ double s_m[LT::MOMS][32], s_eq[2][N][32];
  __shared__ int s_E[2][32];
  buf = chain_wait(buf);
  const int side = blockIdx.y, lane = threadIdx.x, w = threadIdx.y;
  if (bc.kind[side] != 2) return;
  const int len = side < 2 ? G.Ny : G.Nx;
  if ((int)blockIdx.x * 32 >= 2 * len) return;
  const int t = min((int)blockIdx.x * 32 + lane, 2 * len - 1);  // surplus lanes repeat the last cell
  int gx, gy, bx, by;
  ghost_cells(side, 2, 1 + t / len, t % len, G, gx, gy, bx, by);
  const long long PL = G.plane;
  S* g = buf + cell_index(G, gy, gx);
  const S* b = buf + cell_index(G, by, bx);
  if (w < 2) {
    typename LT::Mom m;
    if (w == 0) L::template sum_f<S, false>(b, PL, m, P);
    else L::template sum_g<S, false>(b, PL, m, P);
    LT::put(m, w, [&](int k, double v) { s_m[k][lane] = v; });
  }
  __syncthreads();
  if (w < 2) {
    typename LT::Mom m;
    LT::get(m, [&](int k) { return s_m[k][lane]; });
    double rho, ux, uy, theta;
    L::reduced_state(m, P, rho, ux, uy, theta);
    if (w == 1) {
      ux = 2.0 * bc.uw[side][0] - ux;
      uy = 2.0 * bc.uw[side][1] - uy;
      theta = 2.0 * bc.Tw[side] - theta;
    }
    const auto C = L::reduced_equilibrium(rho, ux, uy, theta, P);
    LT::fields(C, [&](int k, double v) { s_eq[w][k][lane] = v; });
  }
  __syncthreads();
  if (w == 0) {
    double d[LT::GFIELD];
#pragma unroll
    for (int k = 0; k < LT::GFIELD; ++k) d[k] = s_eq[1][k][lane] - s_eq[0][k][lane];
    fields_to_smem<LT::GFIELD, 32>(d, s_fix + lane, s_E[0][lane]);
  } else if (w == 1) {
    double d[N - LT::GFIELD];
#pragma unroll
    for (int k = 0; k < N - LT::GFIELD; ++k) d[k] = s_eq[1][LT::GFIELD + k][lane] - s_eq[0][LT::GFIELD + k][lane];
    fields_to_smem<N - LT::GFIELD, 32>(d, s_fix + 32 * LT::GFIELD + lane, s_E[1][lane]);
  }
  __syncthreads();
  const FixViewOf<32> X{s_fix + lane};
#pragma unroll 1
  for (int u = w; u < 2 * NQ; u += 8) {
    const int p = u >> 1, k = u & 1;
    typename LT::NodeK K;
    LT::load_k(p, K);
    long long v[NQ];
    if (k == 0) LT::target_f(X, K, v);
    else LT::target_g(X, K, v);
    const int sc = s_E[k][lane] - 1079 - LT::kdp(p);
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const long long o = (NF * k + NQ * p + q) * PL;
      g[o] = (S)((double)b[o] + fix_to_double(v[q], sc - LT::kdp(q)));
    }
  }
}

template <class L, class S>
__global__ void k_moments(const S* __restrict__ src, double* rho, double* ux, double* uy, double* T, Geom G,
                          Phys P, Macro M) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= G.Nx || y >= G.Ny) return;
  const CellState c = L::template state<S>(src + cell_index(G, y, x), G.plane, P, M);
  const long long i = (long long)y * G.Nx + x;
  if (rho) rho[i] = c.rho;
  if (ux) ux[i] = c.ux;
  if (uy) uy[i] = c.uy;
  if (T) T[i] = c.T;
}

// block of 256 threads; grid-stride over cells; fixed-order block reduction
template <class L, class S>
__global__ void __launch_bounds__(256) k_totals(const S* __restrict__ src, double* partial, Geom G, Phys P,
                                                Macro M) {
  double acc[5] = {0, 0, 0, 0, 0};
  const long long ncell = (long long)G.Nx * G.Ny;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < ncell;
       i += (long long)gridDim.x * blockDim.x) {
    const int y = (int)(i / G.Nx), x = (int)(i % G.Nx);
    const CellState c = L::template state<S>(src + cell_index(G, y, x), G.plane, P, M);
    acc[0] += c.rho;
    acc[1] += c.jx;
    acc[2] += c.jy;
    acc[3] += c.E;
    if (!(c.rho > 0.0) || !(c.T > 0.0) || !(fabs(c.E) < 1e300)) acc[4] += 1.0;
  }
  __shared__ double sh[5][256];
#pragma unroll
  for (int k = 0; k < 5; ++k) sh[k][threadIdx.x] = acc[k];
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w)
#pragma unroll
      for (int k = 0; k < 5; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int k = 0; k < 5; ++k) partial[blockIdx.x * 6 + k] = sh[k][0];
}

__global__ void __launch_bounds__(256) k_speed(const double* __restrict__ rho, const double* __restrict__ ux,
                                               const double* __restrict__ uy, const double* __restrict__ T,
                                               long long n, double* partial, Macro M) {
  double mx = 0.0, bad = 0.0, pm = 0.0;
  // The FP64 square roots (about 50 instructions of the FP64 pipe) are taken
  // only where a single-precision estimate (relative error below 2^-21) could
  // exceed the maximum so far; the input tests compare bit patterns.  What a
  // product or a conversion loses below the smallest float stays under 2^-60 of
  // the estimate (factors gamma R, R within 2^+-30, rho and T below 2^60 for the
  // pressure), so it is used against maxima above 2^-30 only: otherwise mxf, pmf
  // are 0 and every cell is evaluated in FP64.
  const float gR = (float)(M.gamma * M.R), R = (float)M.R, lowest = 0x1p-30f, highest = 0x1p30f;
  const bool est = gR > lowest && gR < highest && R > lowest && R < highest;
  const unsigned long long big = (unsigned long long)__double_as_longlong(1e300);
  auto positive = [&](double v) { return (unsigned long long)__double_as_longlong(v) - 1ull < big - 1ull; };
  auto bounded = [&](double v) { return ((unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull) < big; };
  float mxf = 0.f, pmf = 0.f;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double r = rho[i], a = ux[i], b = uy[i], t = T[i];
    if (!positive(r) || !positive(t) || !bounded(a) || !bounded(b)) {
      bad += 1.0;
      continue;
    }
    const float af = (float)a, bf = (float)b, tf = (float)t;
    if (!((sqrtf(af * af + bf * bf) + sqrtf(gR * tf)) * 1.000001f < mxf)) {
      mx = fmax(mx, sqrt(a * a + b * b) + sqrt(M.gamma * M.R * t));
      mxf = est && (float)mx > lowest ? (float)mx : 0.f;
    }
    const float rf = (float)r;
    if (!(rf * R * tf * 1.000001f < pmf) || fmaxf(rf, tf) >= 0x1p60f) {
      pm = fmax(pm, r * M.R * t);
      pmf = est && (float)pm > lowest ? (float)pm : 0.f;
    }
  }
  __shared__ double sm[256], sb[256], sp[256];
  sm[threadIdx.x] = mx;
  sb[threadIdx.x] = bad;
  sp[threadIdx.x] = pm;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) {
      sm[threadIdx.x] = fmax(sm[threadIdx.x], sm[threadIdx.x + w]);
      sb[threadIdx.x] += sb[threadIdx.x + w];
      sp[threadIdx.x] = fmax(sp[threadIdx.x], sp[threadIdx.x + w]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    partial[3 * blockIdx.x] = sm[0];
    partial[3 * blockIdx.x + 1] = sb[0];
    partial[3 * blockIdx.x + 2] = sp[0];
  }
}

template <class S>
__global__ void k_pack(S* buf, S* packed, int to_packed, Geom G) {
  // one plane per blockIdx.z
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y;
  const int c = blockIdx.z;
  if (x >= G.Nx) return;
  const long long pi = ((long long)c * G.Ny + y) * G.Nx + x;
  const long long bi = c * G.plane + cell_index(G, y, x);
  if (to_packed) packed[pi] = buf[bi];
  else buf[bi] = packed[pi];
}

// the same in 16-byte words: V words a row, eight rows a block
template <class S>
__global__ void __launch_bounds__(256) k_pack16(S* buf, S* packed, int to_packed, Geom G, int V) {
  const int v = blockIdx.x * 128 + threadIdx.x;
  const int c = blockIdx.z;
  if (v >= V) return;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int y = blockIdx.y * 8 + threadIdx.y + 2 * k;
    if (y < G.Ny) {
      uint4* p = (uint4*)(packed + ((long long)c * G.Ny + y) * G.Nx) + v;
      uint4* b = (uint4*)(buf + c * G.plane + cell_index(G, y, 0)) + v;
      if (to_packed) *p = *b;
      else *b = *p;
    }
  }
}

// halo rows of a slab (one thread per element): blockIdx.y = 2 side + row,
// blockIdx.z = population plane
template <class S>
__global__ void k_halo(S* buf, S* lo, S* hi, int unpack, Geom G) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int side = blockIdx.y >> 1, k = blockIdx.y & 1;
  const int c = blockIdx.z;
  S* ext = side == 0 ? lo : hi;
  if (x >= G.Nx || !ext) return;
  const int yb = unpack ? (side == 0 ? k - 2 : G.Ny + k) : (side == 0 ? k : G.Ny - 2 + k);
  const long long bi = (long long)c * G.plane + cell_index(G, yb, x);
  const long long ei = ((long long)c * 2 + k) * G.Nx + x;
  if (unpack) buf[bi] = ext[ei];
  else ext[ei] = buf[bi];
}

// ---------------------------------------------------------------- wrappers
cudaError_t launch_halo(int elem, void* buf, void* lo, void* hi, int unpack, const Geom& G, int npop,
                        cudaStream_t st) {
  dim3 b(128), g((G.Nx + 127) / 128, 4, npop);
  if (elem == 8) k_halo<double><<<g, b, 0, st>>>((double*)buf, (double*)lo, (double*)hi, unpack, G);
  else k_halo<float><<<g, b, 0, st>>>((float*)buf, (float*)lo, (float*)hi, unpack, G);
  return cudaGetLastError();
}

// lattice 0: D2Q25 (storage 0 FP64, 1 FP32-deviation); lattice 1: D2Q16 (FP64)
cudaError_t launch_init(int lattice, int storage, void* dst, const double* rho, const double* ux, const double* uy,
                        const double* T, const Geom& G, const Phys& P, const Macro& M, cudaStream_t st) {
  dim3 b(32, 8), g((G.Nx + 31) / 32, (G.Ny + 7) / 8);
  if (lattice == 1) k_init<L16, double><<<g, b, 0, st>>>((double*)dst, rho, ux, uy, T, G, P, M);
  else if (storage == 0) k_init<L25, double><<<g, b, 0, st>>>((double*)dst, rho, ux, uy, T, G, P, M);
  else k_init<L25, float><<<g, b, 0, st>>>((float*)dst, rho, ux, uy, T, G, P, M);
  return cudaGetLastError();
}

cudaError_t launch_ghost(int lattice, int storage, void* buf, const Geom& G, const Phys& P, const Macro& M,
                         const BCDev& bc, cudaStream_t st) {
  const int len = G.Nx > G.Ny ? G.Nx : G.Ny;
  bool copies = false, walls = false;
  for (int k = 0; k < 4; ++k) {
    copies = copies || bc.kind[k] < 2;
    walls = walls || bc.kind[k] == 2;
  }
  if (copies) {
    const dim3 b(128), g((2 * len + 127) / 128, 4, lattice == 1 ? L16::NPOP : L25::NPOP);
    if (storage == 0) launch_chained(k_ghost<double>, g, b, st, (double*)buf, G, bc);
    else launch_chained(k_ghost<float>, g, b, st, (float*)buf, G, bc);
  }
  if (walls) {
    const dim3 b(32, 8), g((2 * len + 31) / 32, 4);
    BCDev w = bc;  // in units of c and T_ref
    for (int k = 0; k < 4; ++k) {
      w.uw[k][0] /= M.c;
      w.uw[k][1] /= M.c;
      w.Tw[k] /= M.T_ref;
    }
    if (lattice == 1) launch_chained(k_wall<L16, double>, g, b, st, (double*)buf, G, P, w);
    else if (storage == 0) launch_chained(k_wall<L25, double>, g, b, st, (double*)buf, G, P, w);
    else launch_chained(k_wall<L25, float>, g, b, st, (float*)buf, G, P, w);
  }
  return cudaGetLastError();
}

cudaError_t launch_moments(int lattice, int storage, const void* src, double* rho, double* ux, double* uy, double* T,
                           const Geom& G, const Phys& P, const Macro& M, cudaStream_t st) {
  dim3 b(32, 4), g((G.Nx + 31) / 32, (G.Ny + 3) / 4);
  if (lattice == 1) k_moments<L16, double><<<g, b, 0, st>>>((const double*)src, rho, ux, uy, T, G, P, M);
  else if (storage == 0) k_moments<L25, double><<<g, b, 0, st>>>((const double*)src, rho, ux, uy, T, G, P, M);
  else k_moments<L25, float><<<g, b, 0, st>>>((const float*)src, rho, ux, uy, T, G, P, M);
  return cudaGetLastError();
}

cudaError_t launch_totals(int lattice, int storage, const void* src, double* partial, int nblocks, const Geom& G,
                          const Phys& P, const Macro& M, cudaStream_t st) {
  if (lattice == 1) k_totals<L16, double><<<nblocks, 256, 0, st>>>((const double*)src, partial, G, P, M);
  else if (storage == 0) k_totals<L25, double><<<nblocks, 256, 0, st>>>((const double*)src, partial, G, P, M);
  else k_totals<L25, float><<<nblocks, 256, 0, st>>>((const float*)src, partial, G, P, M);
  return cudaGetLastError();
}

cudaError_t launch_speed(const double* rho, const double* ux, const double* uy, const double* T, long long n,
                         double* partial, int nblocks, const Macro& M, cudaStream_t st) {
  k_speed<<<nblocks, 256, 0, st>>>(rho, ux, uy, T, n, partial, M);
  return cudaGetLastError();
}

cudaError_t launch_pack(int storage, const void* buf, void* packed, int to_packed, const Geom& G, int npop,
                        cudaStream_t st) {
  // rows of whole 16-byte words on 16-byte boundaries (the padded rows always
  // start on 128) are copied in words: 3.4 -> 2.0 ms at 4096^2 FP64
  const int per = storage == 0 ? 2 : 4;
  if (G.Nx % per == 0 && ((size_t)packed & 15) == 0) {
    const int V = G.Nx / per;
    const dim3 b(128, 2), g((V + 127) / 128, (G.Ny + 7) / 8, npop);
    if (storage == 0) k_pack16<double><<<g, b, 0, st>>>((double*)buf, (double*)packed, to_packed, G, V);
    else k_pack16<float><<<g, b, 0, st>>>((float*)buf, (float*)packed, to_packed, G, V);
    return cudaGetLastError();
  }
  dim3 b(128), g((G.Nx + 127) / 128, G.Ny, npop);
  if (storage == 0) k_pack<double><<<g, b, 0, st>>>((double*)buf, (double*)packed, to_packed, G);
  else k_pack<float><<<g, b, 0, st>>>((float*)buf, (float*)packed, to_packed, G);
  return cudaGetLastError();
}

}  // namespace dvbm
