// aux.cuh -- ghost fill, restriction, CFL reduction, refinement flags, conservation sums,
// host-layout packing and regrid kernels.
#pragma once
#include "chain.cuh"
#include "map_internal.hpp"
#include "physics.cuh"
#include "step.cuh"

namespace mapgb {

// W neighbouring values moved by one access
template <typename T, int W>
struct alignas(W * sizeof(T)) Pack {
  T v[W];
};

// Ghost fill of the leaves of one level (Sec. 4.3): every ghost cell gathers from the
// block its region resolves to -- a copy from a same-level block, or the conservative
// minmod prolongation of the covering coarser leaf (whose ghosts an earlier level pass
// filled).  Region tables come from the host tree.
//
// A thread takes a pair of x-neighbours (2p, 2p + 1) of one leaf, all variables: the two
// ghost columns of a side, like every pair inside the block's x range, lie in one region, and
// every unclamped index map shifts x by an even number, so a copied pair is one 8-byte (FP32)
// load and store per variable and a prolonged pair has one coarse cell, whose slopes it
// shares.  Pairs are numbered over all leaves, so small blocks leave no threads idle.
// Latency- and instruction-bound before (one cell per thread, one CTA per leaf); a fill of
// every region: 256^3 FP32 456 us -> 402, octree of 9472 8^3 leaves, finest level 222 ->
// 191, 32640 16^2 blocks 181 -> 154.
template <int NDIM, int NB>
struct Shell {
  static constexpr int NP = NB + 4;
  static constexpr int ROW = NP / 2;                                 // pairs of a padded row
  static constexpr int PLANE = NP * ROW;
  static constexpr int PLANE_GHOSTS = 2 * NG * ROW + NB * NG;        // pairs: ghost rows, then ghost columns
  static constexpr int COUNT = NDIM == 3 ? 2 * NG * PLANE + NB * PLANE_GHOSTS : PLANE_GHOSTS;
  // g-th ghost pair of a block -> padded (i, j, k) of its first cell: the 2*NG full ghost
  // planes first (3D), then per interior plane its NG ghost rows on each side and the pair of
  // ghost columns on each side
  static __device__ __forceinline__ void pair(int g, int& i, int& j, int& k) {
    if (NDIM == 3) {
      if (g < 2 * NG * PLANE) {
        const int pl = g / PLANE, c = g % PLANE;
        k = pl < NG ? pl : NB + pl;
        j = c / ROW;
        i = 2 * (c % ROW);
        return;
      }
      g -= 2 * NG * PLANE;
      k = NG + g / PLANE_GHOSTS;
      g %= PLANE_GHOSTS;
    } else {
      k = 0;
    }
    constexpr int ROWS = 2 * NG * ROW;
    if (g < ROWS) {
      const int r = g / ROW;
      j = r < NG ? r : NB + r;
      i = 2 * (g % ROW);
    } else {
      g -= ROWS;
      j = NG + g / 2;
      i = g % 2 ? NB + NG : 0;
    }
  }
};

// EONLY: the energy alone (between conduction substeps)
template <typename T, int NDIM, int NB, bool EONLY>
__global__ void __launch_bounds__(256) fill_kernel(T* __restrict__ u, const int* __restrict__ blocks,
                                                   int n, const GhostRegion* __restrict__ regions, int skip_pushed) {
  using G = Geo<NDIM, NB>;
  using SH = Shell<NDIM, NB>;
  using P = Pack<T, 2>;
  constexpr int NP = G::NP, P2 = G::P2, S = G::S;
  constexpr int V0 = EONLY ? EN : 0, V1 = EONLY ? EN + 1 : NV;
  static_assert(NG == 2 && NP % 2 == 0, "the ghost columns of a side are one aligned pair");
  chain_begin();
  // (32-bit: a pool that fills the device's memory has under 2^30 ghost pairs)
  const unsigned item = blockIdx.x * blockDim.x + threadIdx.x;
  const int leaf = (int)(item / SH::COUNT), g = (int)(item % SH::COUNT);
  if (leaf >= n) return;
  const int blk = blocks[leaf];
  int i, j, k;
  SH::pair(g, i, j, k);
  const int c = (k * NP + j) * NP + i;
  const int rx = i < NG ? 0 : (i >= NG + NB ? 2 : 1);
  const int ry = j < NG ? 0 : (j >= NG + NB ? 2 : 1);
  const int rz = NDIM == 3 ? (k < NG ? 0 : (k >= NG + NB ? 2 : 1)) : 1;
  const GhostRegion gr = regions[(size_t)blk * 27 + rx + 3 * ry + 9 * rz];
  if (skip_pushed && gr.pushed) return;            // written by the source's step kernel
  T* ub = u + (size_t)blk * NV * S + c;
  const T* sb = u + (size_t)gr.src * NV * S;
  const int gi = gr.m[0] * i + gr.a[0], gj = gr.m[1] * j + gr.a[1];
  const int gk = NDIM == 3 ? gr.m[2] * k + gr.a[2] : 0;
  const bool mapped = gr.m[0] == 1;                // else both cells clamp to one x index
  if (gr.kind == 0) {
    const T* f = sb + (gk * NP + gj) * NP + gi;
    P val[NV];
#pragma unroll
    for (int v = V0; v < V1; ++v) {
      if (mapped) val[v] = *reinterpret_cast<const P*>(f + (size_t)v * S);
      else val[v].v[0] = val[v].v[1] = f[(size_t)v * S];
    }
#pragma unroll
    for (int v = V0; v < V1; ++v) *reinterpret_cast<P*>(ub + (size_t)v * S) = val[v];
  } else {
    const int ci = (gi >> 1) - gr.corg[0] + NG, cj = (gj >> 1) - gr.corg[1] + NG;
    const int ck = NDIM == 3 ? (gk >> 1) - gr.corg[2] + NG : 0;
    const T* fc = sb + (ck * NP + cj) * NP + ci;
    // mapped: gi is even, so the pair covers both halves of coarse cell ci
    const T ox0 = (gi & 1) ? T(0.25) : T(-0.25), ox1 = mapped ? T(0.25) : ox0;
    const T oy = (gj & 1) ? T(0.25) : T(-0.25);
    const T oz = (gk & 1) ? T(0.25) : T(-0.25);
#pragma unroll
    for (int v = V0; v < V1; ++v) {
      const T* f = fc + (size_t)v * S;
      const T f0 = f[0];
      const T sx = minmod<T>(f[1] - f0, f0 - f[-1]);
      const T sy = minmod<T>(f[NP] - f0, f0 - f[-NP]);
      const T sz = NDIM == 3 ? minmod<T>(f[P2] - f0, f0 - f[-P2]) : T(0);
      P val;
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        T t = f0;
        t += sx * (x ? ox1 : ox0);
        t += sy * oy;
        if (NDIM == 3) t += sz * oz;
        val.v[x] = t;
      }
      *reinterpret_cast<P*>(ub + (size_t)v * S) = val;
    }
  }
}

// Parents of one level become the mean of their 2^ndim children (Sec. 4.3 step (1)).  A thread
// takes one variable of ITEMS parent cells, and a parent is spread over several CTAs (its
// cells and variables are a whole number of CTAs): levels hold few parents.  The two
// x-children of a cell are one aligned pair.  One CTA per parent with the variables in
// sequence was bound by their load latencies: 2D 16^2, 680, 232 and 64 parents: 10, 8
// and 8 us -> 9.5, 5.4 and 4.7 (cold caches; a quadtree step does six); 1088 8^3 parents 60 -> 54.
struct RestrictShape {
  static constexpr int THREADS = 192, ITEMS = 3, PER_CTA = THREADS * ITEMS;
};

template <typename T, int NDIM, int NB>
__global__ void __launch_bounds__(RestrictShape::THREADS) restrict_kernel(T* __restrict__ u, const int* __restrict__ parents,
                                                                              const int* __restrict__ children) {
  using G = Geo<NDIM, NB>;
  using P = Pack<T, 2>;
  constexpr int NP = G::NP, S = G::S;
  constexpr int NI = NDIM == 3 ? NB * NB * NB : NB * NB;
  constexpr int NZC = NDIM == 3 ? 2 : 1;
  constexpr int N = RestrictShape::ITEMS, M = NV * NI / RestrictShape::PER_CTA;   // CTAs per parent
  static_assert(NV * NI % RestrictShape::PER_CTA == 0, "a parent is a whole number of CTAs");
  chain_begin();
  const int par = parents[blockIdx.x / M];
  T* dst[N];
  P f[N][NZC][2];
#pragma unroll
  for (int q = 0; q < N; ++q) {
    const int r = (blockIdx.x % M) * RestrictShape::PER_CTA + q * RestrictShape::THREADS + threadIdx.x;
    const int v = r / NI, c = r % NI;
    const int i = c % NB, j = (c / NB) % NB, k = NDIM == 3 ? c / (NB * NB) : 0;
    const int fi = 2 * i, fj = 2 * j, fk = 2 * k;
    // both halves of a cell's children lie in one child block (NB is even)
    const int cb = (fi / NB) | ((fj / NB) << 1) | ((NDIM == 3 ? fk / NB : 0) << 2);
    const T* src = u + (size_t)children[(size_t)par * 8 + cb] * NV * S + (size_t)v * S +
                   ((NDIM == 3 ? fk % NB + NG : 0) * NP + fj % NB + NG) * NP + fi % NB + NG;
    dst[q] = u + (size_t)par * NV * S + (size_t)v * S + ((NDIM == 3 ? k + NG : 0) * NP + j + NG) * NP + i + NG;
#pragma unroll
    for (int dz = 0; dz < NZC; ++dz)
#pragma unroll
      for (int dy = 0; dy < 2; ++dy) f[q][dz][dy] = *reinterpret_cast<const P*>(src + (dz * NP + dy) * NP);
  }
#pragma unroll
  for (int q = 0; q < N; ++q) {
    T sum = T(0);
#pragma unroll
    for (int dz = 0; dz < NZC; ++dz)
#pragma unroll
      for (int dy = 0; dy < 2; ++dy) {
        sum += f[q][dz][dy].v[0];
        sum += f[q][dz][dy].v[1];
      }
    *dst[q] = sum / T(1 << NDIM);
  }
}

// Maximum that keeps a NaN from either side (fmax drops it): a NaN cell anywhere makes the
// reduced signal speed NaN, so the time step built from it is rejected.
template <typename T>
__device__ __forceinline__ T nan_max(T a, T b) {
  return (a != a) ? a : ((b != b) ? b : fmax(a, b));
}

template <typename T>
__device__ __forceinline__ void load_global(const T* b, size_t S, int c, T* w) {
#pragma unroll
  for (int v = 0; v < NV; ++v) w[v] = b[(size_t)v * S + c];
}

// alpha_g: max over leaf interior cells and directions of |v_d| + c_f,d (Sec. 3.7), one leaf
// per CTA, two x-neighbours per thread (8-byte FP32 loads, two chains of roots).  The maxima
// stay in T until one thread widens the leaf's for the atomic (a maximum is exact in any
// precision, and widening is exact and monotone): FP64 on every warp, at 1/64 of the FP32
// rate, had cost more than the cells of a 16^2 block.  32640 16^2 blocks: 228 us -> 63;
// 256^3: 135 -> 106 (floor 89 and 44 us for one read of the state).
//
// A leaf goes to as many CTAs as give each thread four pairs (four for a 16^3 leaf): few
// leaves then still reach every SM.  64 16^3 FP64 leaves, one CTA each: 200 us -> 103.
template <int NDIM, int NB>
__host__ __device__ constexpr int cfl_threads() {
  constexpr int pairs = (NDIM == 3 ? NB * NB * NB : NB * NB) / 2;
  return pairs < 128 ? pairs : 128;
}

template <int NDIM, int NB>
__host__ __device__ constexpr int cfl_parts() {
  constexpr int rounds = (NDIM == 3 ? NB * NB * NB : NB * NB) / 2 / cfl_threads<NDIM, NB>();
  return rounds > 4 ? rounds / 4 : 1;
}

template <typename T, int NDIM, int NB>
__global__ void __launch_bounds__(cfl_threads<NDIM, NB>()) cfl_kernel(const T* __restrict__ u,
                                                                      const int* __restrict__ blocks,
                                                                      const BlockGeo* __restrict__ geo, ProbDyn* dyn,
                                                                      T gamma, T gm1, T kappa0) {
  using G = Geo<NDIM, NB>;
  using V = Pack<T, 2>;
  constexpr int NP = G::NP, S = G::S, NT = cfl_threads<NDIM, NB>(), PARTS = cfl_parts<NDIM, NB>();
  constexpr int NI = NDIM == 3 ? NB * NB * NB : NB * NB;
  __shared__ T red[32], redk[32];
  Phys<T> P;
  P.gamma = gamma;
  P.gm1 = gm1;
  P.ch = T(0);
  P.tau = T(0);
  const bool cond = kappa0 > T(0);
  chain_begin();
  const int blk = blocks[blockIdx.x / PARTS], part = blockIdx.x % PARTS;
  const T* ub = u + (size_t)blk * NV * S;
  T am = T(0), km = T(0);
  for (int c = part * (NI / PARTS) + 2 * threadIdx.x; c < (part + 1) * (NI / PARTS); c += 2 * NT) {
    const int i = c % NB, j = (c / NB) % NB, k = NDIM == 3 ? c / (NB * NB) : 0;
    const T* cell = ub + ((NDIM == 3 ? k + NG : 0) * NP + j + NG) * NP + i + NG;
    V q[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) q[v] = *reinterpret_cast<const V*>(cell + (size_t)v * S);
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      T w[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) w[v] = q[v].v[x];
      const T p = pressure<T>(w, P);
      T a = alpha_p<T, 0>(w, p, P);
      a = nan_max<T>(a, alpha_p<T, 1>(w, p, P));
      if (NDIM == 3) a = nan_max<T>(a, alpha_p<T, 2>(w, p, P));
      am = nan_max<T>(am, a);
      if (cond) {
        // kappa T / p read as kappa / rho, kappa = kappa0 T^(5/2), T = max(p, 0) / rho
        const T tt = (p < T(0) ? T(0) : p) / w[RHO];
        const T kr = kappa0 * (tt * tt * sqrt(tt)) / w[RHO];
        km = nan_max<T>(km, kr);
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    am = nan_max<T>(am, __shfl_xor_sync(0xffffffffu, am, o));
    if (cond) km = nan_max<T>(km, __shfl_xor_sync(0xffffffffu, km, o));
  }
  if ((threadIdx.x & 31) == 0) {
    red[threadIdx.x >> 5] = am;
    redk[threadIdx.x >> 5] = km;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < NT / 32; ++q) {
      am = nan_max<T>(am, red[q]);
      km = nan_max<T>(km, redk[q]);
    }
    ProbDyn* d = dyn + geo[blk].problem;
    atomicMax(&d->alpha_bits, (unsigned long long)__double_as_longlong((double)am));
    if (cond) atomicMax(&d->kmax_bits, (unsigned long long)__double_as_longlong((double)km));
  }
}

// Per-block maxima of alpha (the allocation-free CFL variant): partial[b] = max over the
// interior cells of block b and the directions of |v_d| + c_f,d.
template <typename T, int NDIM, int NB>
__global__ void __launch_bounds__(256) cfl_partial_kernel(const T* __restrict__ u, int nblocks, T gamma, T gm1,
                                                          double* __restrict__ partial) {
  using G = Geo<NDIM, NB>;
  constexpr int NP = G::NP, S = G::S;
  constexpr int NI = NDIM == 3 ? NB * NB * NB : NB * NB;
  __shared__ double red[32];
  Phys<T> P;
  P.gamma = gamma;
  P.gm1 = gm1;
  P.ch = T(0);
  P.tau = T(0);
  for (int blk = blockIdx.x; blk < nblocks; blk += gridDim.x) {
    const T* ub = u + (size_t)blk * NV * S;
    T am = T(0);                     // in T within each warp, as in cfl_kernel
    for (int c = threadIdx.x; c < NI; c += blockDim.x) {
      const int i = c % NB, j = (c / NB) % NB, k = NDIM == 3 ? c / (NB * NB) : 0;
      const int cc = ((NDIM == 3 ? k + NG : 0) * NP + j + NG) * NP + i + NG;
      T w[NV];
      load_global<T>(ub, S, cc, w);
      const T p = pressure<T>(w, P);
      T a = alpha_p<T, 0>(w, p, P);
      a = nan_max<T>(a, alpha_p<T, 1>(w, p, P));
      if (NDIM == 3) a = nan_max<T>(a, alpha_p<T, 2>(w, p, P));
      am = nan_max<T>(am, a);
    }
    for (int o = 16; o > 0; o >>= 1) am = nan_max<T>(am, __shfl_xor_sync(0xffffffffu, am, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = am;
    __syncthreads();
    if (threadIdx.x == 0) {
      double a = 0.0;
      for (int q = 0; q < (int)(blockDim.x + 31) / 32; ++q) a = nan_max<double>(a, red[q]);
      partial[blk] = a;     // every slot < nblocks is written before it is read
    }
    __syncthreads();
  }
}

// Refinement estimator (Sec. 4.5) in the pool's precision, over the interior and the first
// ghost ring; block maximum -> flag.  The parameters come rounded to that precision (FlagArgs)
// and one thread rounds the leaf's spacings: FP64 operations and conversions on every thread,
// at 1/64 of the FP32 rate, had kept an FP32 pool's kernel on the FP64 pipe (84 % busy).
// 9472 8^3 leaves, |J| criterion: 176 -> 66 us.
template <typename T, int NDIM, int NB>
__global__ void __launch_bounds__(256) flags_kernel(FlagArgs<T> L) {
  // the estimator runs in the pool's precision: FP64 pools bitwise as the FP64 formula, FP32
  // pools in FP32 (decisions then differ from FP64 only within float rounding of a threshold)
  using R = T;
  using G = Geo<NDIM, NB>;
  constexpr int NP = G::NP, P2 = G::P2, S = G::S;
  constexpr int NR = NDIM == 3 ? (NB + 2) * (NB + 2) * (NB + 2) : (NB + 2) * (NB + 2);
  __shared__ R red[32];
  __shared__ R two_dx[3];
  __shared__ R mindx_s;
  const T* u = L.u;
  const R bias = L.bias, filt = L.filter;
  const R half_sqrt3 = (R)(1.7320508075688772 / 2.0);
  // the pool's pressure recovery (FP32 pools: with its FP64 fallback at low e_int / e)
  Phys<T> PP;
  PP.gamma = L.gamma;
  PP.gm1 = L.gm1;
  PP.ch = T(0);
  PP.tau = L.tau;
  auto pres = [&](const T* ub, int c) -> R {
    R w[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) w[v] = (R)ub[(size_t)v * S + c];
    return pressure<T>(w, PP);
  };
  const int offs[3] = {1, NP, P2};
  for (int bi = blockIdx.x; bi < L.nblocks; bi += gridDim.x) {
    const int blk = L.blocks[bi];
    const int level = L.geo[blk].level;
    const T* ub = u + (size_t)blk * NV * S;
    if (threadIdx.x == 0) {
      const BlockGeo gg = L.geo[blk];
      R least = (R)gg.dx[0];                       // rounding keeps the order
      for (int d = 0; d < 3; ++d) {
        const R dx = (R)gg.dx[d];
        two_dx[d] = d < NDIM ? R(2) * dx : R(1);   // doubling is exact
        if (d < NDIM) least = fmin(least, dx);
      }
      mindx_s = least;
    }
    __syncthreads();
    const R mindx = mindx_s;
    const R lvf = L.level_factor[level < 16 ? level : 15];
    R emax = R(0);
    for (int q = threadIdx.x; q < NR; q += blockDim.x) {
      const int i = 1 + q % (NB + 2), j = 1 + (q / (NB + 2)) % (NB + 2);
      const int k = NDIM == 3 ? 1 + q / ((NB + 2) * (NB + 2)) : 0;
      const int c = (k * NP + j) * NP + i;
      auto est = [&](auto field, R eps) -> R {
        R s1 = R(0), s2 = R(0);
        const R f0 = field(c);
        for (int d = 0; d < NDIM; ++d) {
          const R fp = field(c + offs[d]), fm = field(c - offs[d]);
          const R d1 = fp - fm;
          const R d2 = fp - R(2) * f0 + fm;
          s1 += d1 * d1;
          s2 += d2 * d2;
        }
        const R du = half_sqrt3 * sqrt(s1);
        const R d2u = sqrt(s2);
        const R au = fabs(f0) + eps;
        const R e = bias * du / au + (R(1) - bias) * d2u / (du + filt * au);
        return e * lvf;
      };
      if (L.var_mask & 1) emax = fmax(emax, est([&](int cc) { return (R)ub[RHO * (size_t)S + cc]; }, L.eps_rho));
      if (L.var_mask & 2) emax = fmax(emax, est([&](int cc) { return pres(ub, cc); }, L.eps_p));
      if (L.var_mask & 4) {
        auto cd = [&](int comp, int d) -> R {
          if (d >= NDIM) return R(0);
          return ((R)ub[(size_t)comp * S + c + offs[d]] - (R)ub[(size_t)comp * S + c - offs[d]]) / two_dx[d];
        };
        const R jx = cd(BZ, 1) - cd(BY, 2);
        const R jy = cd(BX, 2) - cd(BZ, 0);
        const R jz = cd(BY, 0) - cd(BX, 1);
        const R bx = ub[(size_t)BX * S + c], by = ub[(size_t)BY * S + c], bz = ub[(size_t)BZ * S + c];
        const R e = sqrt(jx * jx + jy * jy + jz * jz) * mindx / (sqrt(bx * bx + by * by + bz * bz) + L.eps_b);
        emax = fmax(emax, e);
      }
    }
    for (int o = 16; o > 0; o >>= 1) emax = fmax(emax, __shfl_xor_sync(0xffffffffu, emax, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = emax;
    __syncthreads();
    if (threadIdx.x == 0) {
      R er = R(0);
      for (int q = 0; q < (int)(blockDim.x + 31) / 32; ++q) er = fmax(er, red[q]);
      const double e = (double)er;
      int8_t f = 0;
      if (e > L.thr && level < L.max_level) f = 1;
      else if (e < L.coarsen_thr && level > 0) f = -1;
      L.flags[bi] = f;
      if (L.est) L.est[bi] = e;
    }
    __syncthreads();
  }
}

// FP64 conservation sums of the leaf interiors: sum U * cell volume per problem.
template <typename T, int NDIM, int NB>
__global__ void __launch_bounds__(256) sums_kernel(SumLaunch L) {
  using G = Geo<NDIM, NB>;
  constexpr int NP = G::NP, S = G::S;
  constexpr int NI = NDIM == 3 ? NB * NB * NB : NB * NB;
  __shared__ double red[NV][32];
  const T* u = (const T*)L.u;
  for (int bi = blockIdx.x; bi < L.nblocks; bi += gridDim.x) {
    const int blk = L.blocks[bi];
    const BlockGeo gg = L.geo[blk];
    const T* ub = u + (size_t)blk * NV * S;
    double s[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) s[v] = 0.0;
    for (int c = threadIdx.x; c < NI; c += blockDim.x) {
      const int i = c % NB, j = (c / NB) % NB, k = NDIM == 3 ? c / (NB * NB) : 0;
      const int cc = ((NDIM == 3 ? k + NG : 0) * NP + j + NG) * NP + i + NG;
#pragma unroll
      for (int v = 0; v < NV; ++v) s[v] += (double)ub[(size_t)v * S + cc];
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      for (int o = 16; o > 0; o >>= 1) s[v] += __shfl_xor_sync(0xffffffffu, s[v], o);
      if ((threadIdx.x & 31) == 0) red[v][threadIdx.x >> 5] = s[v];
    }
    __syncthreads();
    if (threadIdx.x < NV) {
      double t = 0.0;
      for (int q = 0; q < (int)(blockDim.x + 31) / 32; ++q) t += red[threadIdx.x][q];
      const double vol = gg.dx[0] * gg.dx[1] * (NDIM == 3 ? gg.dx[2] : 1.0);
      atomicAdd(&L.sums[gg.problem * NV + threadIdx.x], t * vol);
    }
    __syncthreads();
  }
}

// Host layout [n][9][nz][nb][nb] <-> pool interiors.  A copy, bound by HBM: a thread moves
// QUADS groups of four x-neighbours, one 16-byte (FP32) access on the dense side and two
// 8-byte ones on the padded side (an interior row starts two cells into its padded row), all
// loads before the first store.  576 groups per CTA divide every block shape.  W = 1 is the
// same walk with single values, for a caller's buffer that is not aligned to four of them.
// 256^3 FP32 to the pool and back: 343 + 445 us one value per access -> 197 + 320 (floor 178
// each at the copy rate).
struct PackShape {
  static constexpr int THREADS = 192, QUADS = 3, PER_CTA = THREADS * QUADS;
};

template <typename T, typename H, int NDIM, int NB, int W, bool TO_POOL>
__global__ void __launch_bounds__(PackShape::THREADS) pack_kernel(T* __restrict__ u, H* __restrict__ dense,
                                                                  const int* __restrict__ blocks, int nblocks) {
  using G = Geo<NDIM, NB>;
  constexpr int NP = G::NP, S = G::S;
  constexpr int NI = NDIM == 3 ? NB * NB * NB : NB * NB;
  constexpr int PER = NV * NI / W;                 // groups of one block
  constexpr int HALF = W == 4 ? 2 : 1;             // values per padded-side access
  constexpr int N = PackShape::QUADS;
  static_assert(NB % W == 0 && (PER % PackShape::PER_CTA == 0 || PackShape::PER_CTA % PER == 0), "whole blocks per CTA");
  T* pool[N];
  H* host[N];
  bool on[N];
#pragma unroll
  for (int q = 0; q < N; ++q) {
    const int r = q * PackShape::THREADS + threadIdx.x;
    int leaf, g;
    if (PER >= PackShape::PER_CTA) {
      constexpr int M = PER >= PackShape::PER_CTA ? PER / PackShape::PER_CTA : 1;
      leaf = blockIdx.x / M;
      g = (blockIdx.x % M) * PackShape::PER_CTA + r;
    } else {
      leaf = blockIdx.x * (PackShape::PER_CTA / PER) + r / PER;
      g = r % PER;
    }
    on[q] = leaf < nblocks;
    const int e = g * W, v = e / NI, c = e % NI;
    const int i = c % NB, j = (c / NB) % NB, k = NDIM == 3 ? c / (NB * NB) : 0;
    const int cc = ((NDIM == 3 ? k + NG : 0) * NP + j + NG) * NP + i + NG;
    pool[q] = u + (on[q] ? (size_t)blocks[leaf] * NV * S : 0) + (size_t)v * S + cc;
    host[q] = dense + (size_t)leaf * NV * NI + e;
  }
  if (TO_POOL) {
    Pack<H, W> h[N];
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (on[q]) h[q] = *reinterpret_cast<const Pack<H, W>*>(host[q]);
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (on[q]) {
#pragma unroll
        for (int b = 0; b < W; b += HALF) {
          Pack<T, HALF> t;
#pragma unroll
          for (int x = 0; x < HALF; ++x) t.v[x] = (T)h[q].v[b + x];
          *reinterpret_cast<Pack<T, HALF>*>(pool[q] + b) = t;
        }
      }
  } else {
    Pack<T, HALF> t[N][W / HALF];
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (on[q]) {
#pragma unroll
        for (int b = 0; b < W; b += HALF) t[q][b / HALF] = *reinterpret_cast<const Pack<T, HALF>*>(pool[q] + b);
      }
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (on[q]) {
        Pack<H, W> h;
#pragma unroll
        for (int b = 0; b < W; ++b) h.v[b] = (H)t[q][b / HALF].v[b % HALF];
        *reinterpret_cast<Pack<H, W>*>(host[q]) = h;
      }
  }
}

// Regrid: copy kept / coarsened leaves, prolong new children from their old parent leaf
// (Sec. 4.3 formula applied to interior cells; the old parent's ghosts are filled).
template <typename T, int NDIM, int NB>
__global__ void __launch_bounds__(256) regrid_kernel(RegridLaunch L) {
  using G = Geo<NDIM, NB>;
  constexpr int NP = G::NP, P2 = G::P2, S = G::S;
  constexpr int NI = NDIM == 3 ? NB * NB * NB : NB * NB;
  const T* uo = (const T*)L.u_old;
  T* un = (T*)L.u_new;
  for (int ti = blockIdx.x; ti < L.ntasks; ti += gridDim.x) {
    const RegridTask tk = L.tasks[ti];
    const T* sb = uo + (size_t)tk.src * NV * S;
    T* db = un + (size_t)tk.dst * NV * S;
    const int bx = tk.cb & 1, by = (tk.cb >> 1) & 1, bz = (tk.cb >> 2) & 1;
    for (int c = threadIdx.x; c < NI; c += blockDim.x) {
      const int i = c % NB, j = (c / NB) % NB, k = NDIM == 3 ? c / (NB * NB) : 0;
      const int dc = ((NDIM == 3 ? k + NG : 0) * NP + j + NG) * NP + i + NG;
      if (tk.kind == 0) {
#pragma unroll
        for (int v = 0; v < NV; ++v) db[(size_t)v * S + dc] = sb[(size_t)v * S + dc];
      } else {
        const int gi = bx * NB + i, gj = by * NB + j, gk = bz * NB + k;
        const int cc = ((NDIM == 3 ? (gk >> 1) + NG : 0) * NP + (gj >> 1) + NG) * NP + (gi >> 1) + NG;
        const T ox = (gi & 1) ? T(0.25) : T(-0.25);
        const T oy = (gj & 1) ? T(0.25) : T(-0.25);
        const T oz = (gk & 1) ? T(0.25) : T(-0.25);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const T* f = sb + (size_t)v * S;
          T val = f[cc];
          val += minmod<T>(f[cc + 1] - f[cc], f[cc] - f[cc - 1]) * ox;
          val += minmod<T>(f[cc + NP] - f[cc], f[cc] - f[cc - NP]) * oy;
          if (NDIM == 3) val += minmod<T>(f[cc + P2] - f[cc], f[cc] - f[cc - P2]) * oz;
          db[(size_t)v * S + dc] = val;
        }
      }
    }
  }
}


// Reflux (Sec. 4.2, boundary step (2), after Berger and Colella): one CTA per coarse leaf
// with coarse/fine faces.  For every face cell of such a face the coarse flux recorded by the
// step kernel is replaced by the mean of the fine fluxes covering the cell:
//   u_c += lam (F_fine - F_coarse) on a low face, u_c -= lam (F_fine - F_coarse) on a high one
// (lam = dt / dx_d of the coarse leaf; psi's correction carries the damping factor the step
// already applied).  A thread takes a corrected cell: it applies the faces the cell lies on in
// the order (d, low then high), checks the cell, stores it again into the ghost regions of the
// same-level leaves that copy it and, in the fused form, adds it to alpha_g and the FP64 sums
// (the step kernel left these cells out).
//
// The kernel is bound by latency -- a few hundred cells per leaf, each a chain of register
// loads -- and by FP64, at 1/64 of the FP32 rate: so no face waits for another, dt/dx is one
// division on one warp, and the sums of a warp are reduced by halving the number of variables
// with the number of lanes that hold them (16 additions instead of 45).  Faces one after the
// other with a barrier each, and every sum through all lanes: 27 -> 15 us per launch on the
// rotor's quadtree (16^2), 57 -> 26 on a 9472-leaf octree (8^3).
//
// A thread per corrected cell of a leaf with its usual coarse/fine faces: up to four of 16 cells
// (16^2), three of 64 (8^3, at a corner of the fine region), one of 256 (16^3); a leaf with more
// takes a second round.  The choice weighs little: rotor, four steps, 32 / 64 / 128 threads 583.7 /
// 583.8 / 585.7 us; octree, four steps, 128 / 192 / 256 threads 4069 / 4078 / 4109.
template <int NDIM, int NB>
__host__ __device__ constexpr int reflux_threads() {
  return NDIM == 2 ? 64 : (NB == 8 ? 192 : 256);
}

template <typename T, int NDIM, int NB>
__global__ void __launch_bounds__(reflux_threads<NDIM, NB>()) reflux_kernel(RefluxLaunch L) {
  using G = Geo<NDIM, NB>;
  constexpr int NP = G::NP, S = G::S, NT = reflux_threads<NDIM, NB>(), NW = NT / 32;
  constexpr int NF = NDIM == 3 ? NB * NB : NB;          // face cells per face
  constexpr int H = NB / 2;
  constexpr size_t NB2 = (size_t)NB * NB;
  constexpr size_t PER = (size_t)2 * NDIM * NV * NB2;   // one register slot
  __shared__ double red[NV + 1][NW];
  __shared__ T lam_s[3];
  __shared__ RefluxTask tk;
  chain_begin();
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  {
    constexpr int words = sizeof(RefluxTask) / sizeof(int);
    static_assert(sizeof(RefluxTask) % sizeof(int) == 0 && words <= 32, "one word per lane");
    if (tid < words) reinterpret_cast<int*>(&tk)[tid] = reinterpret_cast<const int*>(L.tasks + blockIdx.x)[tid];
  }
  __syncthreads();
  const int q = tk.coarse;
  const int prob = L.geo[q].problem;
  if (L.nsub && L.it >= L.nsub[prob]) return;              // no substep for this problem
  if (wid == 0) {
    const double dtp = L.hsub ? L.hsub[prob] : L.dyn[prob].dt;
    const double l = dtp / L.geo[q].dx[lane < NDIM ? lane : 0];
    if (lane < NDIM) lam_s[lane] = (T)l;
  }
  __syncthreads();
  T* ub = (T*)L.u + (size_t)q * NV * S;
  const T* freg = (const T*)L.freg;
  const T damp = (T)L.dyn[prob].damp;
  int mask = 0;
#pragma unroll
  for (int f = 0; f < 2 * NDIM; ++f)
    if (tk.fslot[f][0] >= 0) mask |= 1 << f;
  Phys<T> P;
  P.gamma = (T)L.gamma;
  P.gm1 = (T)(L.gamma - 1.0);
  P.ch = T(0);
  P.tau = (T)L.tau;
  unsigned errbits = 0;
  T am = T(0);
  double sum[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) sum[v] = 0.0;
  for (int item = tid; item < __popc(mask) * NF; item += NT) {
    int f = 0, rank = item / NF;                           // the face of this item: the rank-th in the mask
#pragma unroll
    for (int f2 = 0; f2 < 2 * NDIM; ++f2)
      if ((mask >> f2) & 1) {
        if (rank == 0) f = f2;
        --rank;
      }
    const int d0 = f >> 1, s0 = f & 1, idx = item % NF;
    int ci[3] = {0, 0, 0};
    {
      const int t0 = idx % NB, t1 = NDIM == 3 ? idx / NB : 0;
      ci[0] = d0 == 0 ? (s0 ? NB - 1 : 0) : t0;
      ci[1] = d0 == 1 ? (s0 ? NB - 1 : 0) : (d0 == 0 ? t0 : t1);
      ci[2] = NDIM == 3 ? (d0 == 2 ? (s0 ? NB - 1 : 0) : t1) : 0;
    }
    // a cell on several such faces is taken with the first of them
    bool first = true;
#pragma unroll
    for (int f2 = 0; f2 < 2 * NDIM; ++f2)
      if (f2 < f && ((mask >> f2) & 1) && ci[f2 >> 1] == ((f2 & 1) ? NB - 1 : 0)) first = false;
    if (!first) continue;
    const int c = ((NDIM == 3 ? ci[2] + NG : 0) * NP + ci[1] + NG) * NP + ci[0] + NG;
    T w[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) w[v] = ub[(size_t)v * S + c];
#pragma unroll
    for (int d = 0; d < NDIM; ++d) {
      const int t0 = d == 0 ? ci[1] : ci[0], t1 = NDIM == 3 ? (d == 2 ? ci[1] : ci[2]) : 0;
      const int k = t0 / H + (NDIM == 3 ? 2 * (t1 / H) : 0);
      const int f0 = 2 * (t0 % H), f1 = NDIM == 3 ? 2 * (t1 % H) : 0;
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        const int fs = 2 * d + side;
        if (!((mask >> fs) & 1) || ci[d] != (side ? NB - 1 : 0)) continue;
        const T* rc = freg + (size_t)tk.cslot * PER + (size_t)fs * NV * NB2 + t1 * NB + t0;
        const T* rf = freg + (size_t)tk.fslot[fs][k] * PER + (size_t)(2 * d + 1 - side) * NV * NB2 + f1 * NB + f0;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          if (v < L.v0 || v >= L.v1) continue;
          const T* fv = rf + (size_t)v * NB2;
          T ff;
          if (NDIM == 2) ff = T(0.5) * (fv[0] + fv[1]);
          else ff = T(0.25) * ((fv[0] + fv[1]) + (fv[NB] + fv[NB + 1]));
          T corr = lam_s[d] * (ff - rc[(size_t)v * NB2]);
          if (v == PSI) corr = corr * damp;
          w[v] = side ? w[v] - corr : w[v] + corr;
        }
      }
    }
    bool fin = true;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      if (v >= L.v0 && v < L.v1) ub[(size_t)v * S + c] = w[v];
      fin = fin && isfinite(w[v]);
    }
    if (!fin) {
      errbits |= 1u;
      am = (T)NAN;
    } else {
      const T pr = pressure<T>(w, P);
      if (!(w[RHO] > T(0)) || pr < T(0)) errbits |= 2u;
      if (L.dyn_next) {
        T a = alpha_p<T, 0>(w, pr, P);
        a = dmax<T>(a, alpha_p<T, 1>(w, pr, P));
        if (NDIM == 3) a = dmax<T>(a, alpha_p<T, 2>(w, pr, P));
        if (!(am != am)) am = dmax<T>(am, a);
      }
    }
    if (L.sums) {
#pragma unroll
      for (int v = 0; v < NV; ++v) sum[v] += (double)w[v];
    }
    // the same-level leaves that copy this cell into their ghosts
    const int x = ci[0] + NG, y = ci[1] + NG, z = NDIM == 3 ? ci[2] + NG : 0;
    const int fx = x < 2 * NG ? -1 : (x >= NB ? 1 : 0);
    const int fy = y < 2 * NG ? -1 : (y >= NB ? 1 : 0);
    const int fz = NDIM == 3 ? (z < 2 * NG ? -1 : (z >= NB ? 1 : 0)) : 0;
    for (int kz = 0; kz < (fz ? 2 : 1); ++kz)
      for (int ky = 0; ky < (fy ? 2 : 1); ++ky)
        for (int kx = 0; kx < (fx ? 2 : 1); ++kx) {
          const int ex = kx ? fx : 0, ey = ky ? fy : 0, ez = kz ? fz : 0;
          if (!(ex | ey | ez)) continue;
          const PushEntry pe = L.pushes[(size_t)q * 27 + (ex + 1) + 3 * (ey + 1) + 9 * (ez + 1)];
          if (pe.dst < 0) continue;
          T* db = (T*)L.u + (size_t)pe.dst * NV * S;
          const size_t dc = ((size_t)(z + pe.off[2]) * NP + (y + pe.off[1])) * NP + (x + pe.off[0]);
#pragma unroll
          for (int v = 0; v < NV; ++v) db[(size_t)v * S + dc] = w[v];
        }
  }
  unsigned e = errbits;
  for (int o = 16; o > 0; o >>= 1) e |= __shfl_xor_sync(0xffffffffu, e, o);
  if (lane == 0 && e) atomicOr(L.err_word, e);
  if (!L.dyn_next && !L.sums) return;
  for (int o = 16; o > 0; o >>= 1) am = nan_max<T>(am, __shfl_xor_sync(0xffffffffu, am, o));
  // the warp's sums of sixteen values (nine in use): after the exchange over lane bit b a lane
  // keeps the half of its values whose index agrees with that bit, so lanes v and v + 16 end
  // with the halves of value v
  double s[16];
#pragma unroll
  for (int v = 0; v < 16; ++v) s[v] = v < NV ? sum[v < NV ? v : 0] : 0.0;
#pragma unroll
  for (int b = 3; b >= 0; --b) {
    const int half = 1 << b;
    const bool up = (lane >> b) & 1;
#pragma unroll
    for (int v = 0; v < half; ++v) {
      const double give = up ? s[v] : s[v + half], keep = up ? s[v + half] : s[v];
      s[v] = keep + __shfl_xor_sync(0xffffffffu, give, half);
    }
  }
  s[0] += __shfl_xor_sync(0xffffffffu, s[0], 16);
  if (lane < NV) red[lane][wid] = s[0];
  if (lane == NV) red[NV][wid] = (double)am;
  __syncthreads();
  if (tid == NV && L.dyn_next) {
    double a = 0.0;
    for (int k = 0; k < NW; ++k) a = nan_max<double>(a, red[NV][k]);
    atomicMax(&L.dyn_next[prob].alpha_bits, (unsigned long long)__double_as_longlong(a));
  }
  if (tid < NV && L.sums) {
    const BlockGeo gg = L.geo[q];
    const double vol = gg.dx[0] * gg.dx[1] * (NDIM == 3 ? gg.dx[2] : 1.0);
    double t = 0.0;
    for (int k = 0; k < NW; ++k) t += red[tid][k];
    atomicAdd(&L.sums[prob * NV + tid], t * vol);
  }
}


// Thermal conduction (Sec. 3.6), one substep on one leaf per CTA, in place on the energy:
//   e_i += h sum_d (F_d,i+1/2 - F_d,i-1/2) / dx_d,  kappa = kappa0 T^(5/2), T = max(p,0)/rho,
//   isotropic:     F = sqrt(kappa_l kappa_r) (T_r - T_l) / dx_d,
//   along B:       F = sqrt(kappa_l kappa_r) b_d (b . grad T), b = B_f / |B_f| with B_f the
//                  mean of the two cells' B, transverse derivatives the mean of the two
//                  cells' central differences (no flux where B_f = 0),
// face gradients clipped to +-grad_t_max when it is > 0.  T and kappa of the interior and its
// one-cell ring are staged in shared memory first; other leaves read this leaf's energy only
// through their own ghost copies, so the in-place write is safe.  Boundary face fluxes go to
// the face register's energy slot as fluxes of e along +d (-F) for reflux.

// Products that are not contracted into a sum, so that both conduction kernels round alike
// wherever the compiler would fuse one of them differently; quotients by a fixed b likewise: the
// plain quotient in FP64, the product with the reciprocal rb = qdiv(1, b) in FP32.
__device__ __forceinline__ float pmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double pmul(double a, double b) { return a * b; }
__device__ __forceinline__ float pquo(float a, float, float rb) { return __fmul_rn(a, rb); }
__device__ __forceinline__ double pquo(double a, double b, double) { return a / b; }

// pressure<T> with every rounding spelled out, for the same reason (the loop keeps the parts
// of it that conduction leaves alone, which no product may be fused across)
__device__ __forceinline__ double cond_pressure(const double* w, const Phys<double>& P) { return pressure<double>(w, P); }
__device__ __forceinline__ float cond_pressure(const float* w, const Phys<float>& P) {
  const float m2 = __fmaf_rn(w[MZ], w[MZ], __fmaf_rn(w[MY], w[MY], __fmul_rn(w[MX], w[MX])));
  const float b2 = __fmaf_rn(w[BZ], w[BZ], __fmaf_rn(w[BY], w[BY], __fmul_rn(w[BX], w[BX])));
  const float kin = __fmul_rn(0.5f * m2, qdiv(1.0f, w[RHO]));
  const float eint = __fadd_rn(__fadd_rn(w[EN], -kin), -0.5f * b2);
  if (eint < P.tau * w[EN]) return pressure_fp64(w[RHO], w[MX], w[MY], w[MZ], w[BX], w[BY], w[BZ], w[EN], P.gm1);
  return __fmul_rn(P.gm1, eint);
}

// T and kappa of one cell from its state
template <typename T>
__device__ __forceinline__ void cond_tk(const T* w, const Phys<T>& P, T k0, T& tt, T& kk) {
  T p = cond_pressure(w, P);
  if (p < T(0)) p = T(0);
  tt = pquo(p, w[RHO], sizeof(T) == 4 ? qdiv<T>(T(1), w[RHO]) : T(0));
  kk = pmul(k0, pmul(pmul(tt, tt), sqrt(tt)));
}

// The two faces of a cell in direction d: their mean field and |B|^2 (unused for the isotropic
// form), which conduction leaves as they are.
template <typename T>
struct CondFaces {
  T b[2][3], b2[2];
};

// B: the three components, S apart; c: the cell's index; po: the stride of direction d
template <typename T>
__device__ __forceinline__ void cond_faces(const T* B, size_t S, int c, int po, CondFaces<T>& f) {
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    const int cl = side ? c : c - po, cr = cl + po;
    f.b2[side] = T(0);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      f.b[side][j] = pmul(T(0.5), B[(size_t)j * S + cl] + B[(size_t)j * S + cr]);
      f.b2[side] += pmul(f.b[side][j], f.b[side][j]);
    }
  }
}

// Spacings of a leaf in T, with their reciprocals and those of twice the spacing.
template <typename T>
struct CondDx {
  T dx[3], rdx[3], rdx2[3];
  __device__ __forceinline__ explicit CondDx(const BlockGeo& g) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      dx[d] = (T)g.dx[d];
      rdx[d] = sizeof(T) == 4 ? qdiv<T>(T(1), dx[d]) : T(0);
      rdx2[d] = T(0.5) * rdx[d];
    }
  }
};

// The energy rate of one interior cell: r its ring-region index (strides ro), sT / sK the
// ring's T and kappa, faces(d) the faces of direction d, face(d, F) sees their two fluxes (the
// reflux registers take them).  Both conduction kernels call it, so their arithmetic is the
// same.
template <typename T, int NDIM, typename BF, typename FF>
__device__ __forceinline__ T cond_rate(const T* sT, const T* sK, int r, const int* ro, const CondDx<T>& X,
                                       T gmax, int mode, BF faces, FF face) {
  T acc = T(0);
#pragma unroll
  for (int d = 0; d < NDIM; ++d) {
    T F[2];
    const CondFaces<T> cf = faces(d);
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const int rl = side ? r : r - ro[d], rr = rl + ro[d];
      T gn = pquo(sT[rr] - sT[rl], X.dx[d], X.rdx[d]);
      if (gmax > T(0)) gn = fmax(-gmax, fmin(gmax, gn));
      const T kf = sqrt(pmul(sK[rl], sK[rr]));
      if (mode == 1) {
        F[side] = pmul(kf, gn);
      } else {
        const T* bf = cf.b[side];
        const T b2 = cf.b2[side];
        if (!(b2 > T(0))) {
          F[side] = T(0);
        } else {
          T bg = pmul(bf[d], gn);
#pragma unroll
          for (int t = 0; t < NDIM; ++t) {
            if (t == d) continue;
            T gt = pmul(T(0.5), pquo(sT[rl + ro[t]] - sT[rl - ro[t]], T(2) * X.dx[t], X.rdx2[t]) +
                                    pquo(sT[rr + ro[t]] - sT[rr - ro[t]], T(2) * X.dx[t], X.rdx2[t]));
            if (gmax > T(0)) gt = fmax(-gmax, fmin(gmax, gt));
            bg += pmul(bf[t], gt);
          }
          F[side] = qdiv<T>(pmul(pmul(kf, bf[d]), bg), b2);
        }
      }
    }
    face(d, F);
    acc += pquo(F[1] - F[0], X.dx[d], X.rdx[d]);
  }
  return acc;
}

template <typename T, int NDIM, int NB>
__global__ void __launch_bounds__(256) conduction_kernel(CondLaunch L) {
  using G = Geo<NDIM, NB>;
  constexpr int NP = G::NP, S = G::S;
  constexpr int R = NB + 2;
  constexpr int NR = NDIM == 3 ? R * R * R : R * R;
  constexpr int NI = NDIM == 3 ? NB * NB * NB : NB * NB;
  constexpr size_t NB2 = (size_t)NB * NB;
  extern __shared__ __align__(16) unsigned char csm[];
  T* sT = reinterpret_cast<T*>(csm);
  T* sK = sT + NR;
  chain_begin();
  const int blk = L.blocks[blockIdx.x];
  const BlockGeo gg = L.geo[blk];
  if (L.it >= L.nsub[gg.problem]) return;
  const T h = (T)L.hsub[gg.problem];
  T* ub = (T*)L.u + (size_t)blk * NV * S;
  Phys<T> P;
  P.gamma = (T)L.gamma;
  P.gm1 = (T)(L.gamma - 1.0);
  P.ch = T(0);
  P.tau = (T)L.tau;
  const T k0 = (T)L.kappa0, gmax = (T)L.grad_t_max;
  // region cell r = (ri, rj, rk) is padded cell (ri+1, rj+1, rk+1)
  for (int r = threadIdx.x; r < NR; r += blockDim.x) {
    const int ri = r % R, rj = (r / R) % R, rk = NDIM == 3 ? r / (R * R) : 0;
    const int c = ((NDIM == 3 ? rk + 1 : 0) * NP + rj + 1) * NP + ri + 1;
    T w[NV];
    load_global<T>(ub, S, c, w);
    cond_tk<T>(w, P, k0, sT[r], sK[r]);
  }
  __syncthreads();
  const int slot = L.freg ? L.refl[blk].slot : -1;
  T* R0 = slot >= 0 ? (T*)L.freg + (size_t)slot * (2 * NDIM * NV * NB2) : nullptr;
  const int ro[3] = {1, R, R * R};
  const int po[3] = {1, NP, NP * NP};
  const CondDx<T> X(gg);
  for (int q = threadIdx.x; q < NI; q += blockDim.x) {
    const int i = q % NB, j = (q / NB) % NB, k = NDIM == 3 ? q / (NB * NB) : 0;
    const int r = ((NDIM == 3 ? k + 1 : 0) * R + j + 1) * R + i + 1;
    const int c = ((NDIM == 3 ? k + NG : 0) * NP + j + NG) * NP + i + NG;
    const int ic[3] = {i, j, k};
    auto faces = [&](int d) {
      CondFaces<T> f;
      if (L.mode != 1) cond_faces<T>(ub + (size_t)BX * S, S, c, po[d], f);
      return f;
    };
    auto face = [&](int d, const T* F) {
      if (R0) {
        const int da = d == 0 ? 1 : 0, db = d == 2 ? 1 : 2;
        const int t0 = ic[da], t1 = NDIM == 3 ? ic[db] : 0;
        if (ic[d] == 0) R0[(size_t)(2 * d) * NV * NB2 + (size_t)EN * NB2 + t1 * NB + t0] = -F[0];
        if (ic[d] == NB - 1) R0[(size_t)(2 * d + 1) * NV * NB2 + (size_t)EN * NB2 + t1 * NB + t0] = -F[1];
      }
    };
    const T acc = cond_rate<T, NDIM>(sT, sK, r, ro, X, gmax, L.mode, faces, face);
    ub[(size_t)EN * S + c] = ub[(size_t)EN * S + c] + pmul(h, acc);
  }
}

// Exchange words of the conduction loop: a value with the number of the substep that made it,
// in one 64-bit word (two for FP64), so the reader that finds the number it waits for has the
// value with it -- no fence, flag or barrier between the two.
__device__ __forceinline__ void put_word(unsigned long long* p, unsigned tag, unsigned bits) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(((unsigned long long)tag << 32) | bits) : "memory");
}
// waits for tag in *p (giving up after ~2^31 clock cycles, about a second, or at once for the
// test hook)
__device__ __forceinline__ bool get_word(const unsigned long long* p, unsigned tag, int give_up, unsigned& bits) {
  if (give_up) return false;
  const long long t0 = clock64();
  for (;;) {
    unsigned long long x;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(x) : "l"(p) : "memory");
    if ((unsigned)(x >> 32) == tag) {
      bits = (unsigned)x;
      return true;
    }
    if (clock64() - t0 > (1ll << 31)) return false;
  }
}
template <typename T>
struct XWords { static constexpr int N = sizeof(T) / 4; };
__device__ __forceinline__ void put_value(unsigned long long* p, unsigned tag, float x) {
  put_word(p, tag, __float_as_uint(x));
}
__device__ __forceinline__ void put_value(unsigned long long* p, unsigned tag, double x) {
  put_word(p, tag, (unsigned)__double2loint(x));
  put_word(p + 1, tag, (unsigned)__double2hiint(x));
}
__device__ __forceinline__ bool get_value(const unsigned long long* p, unsigned tag, int give_up, float& x) {
  unsigned b = 0;
  const bool ok = get_word(p, tag, give_up, b);
  x = __uint_as_float(b);
  return ok;
}
__device__ __forceinline__ bool get_value(const unsigned long long* p, unsigned tag, int give_up, double& x) {
  unsigned lo = 0, hi = 0;
  const bool ok = get_word(p, tag, give_up, lo) && get_word(p + 1, tag, give_up, hi);
  x = __hiloint2double((int)hi, (int)lo);
  return ok;
}

// Shape of the loop's CTA: one thread per interior cell and one per ring cell of the leaf
// (3D 8^3: the same threads take a cell of each kind).
template <int NDIM, int NB>
struct CondLoopShape {
  static constexpr int R = NB + 2;
  static constexpr int NR = NDIM == 3 ? R * R * R : R * R;
  static constexpr int NI = NDIM == 3 ? NB * NB * NB : NB * NB;
  static constexpr int NG1 = NR - NI;                          // ghost cells of the ring region
  static constexpr int RING0 = NI + NG1 <= 512 ? NI : 0;       // first thread with a ring cell
  static constexpr int THREADS = ((RING0 + NG1 > NI ? RING0 + NG1 : NI) + 31) / 32 * 32;
  // every leaf's CTA has to be resident: in FP32 the registers are held to three 2D 16^2 or two
  // 3D 8^3 leaves per SM (456 and 304 leaves on 152 SMs)
  static constexpr int MIN_CTAS = NB == 8 ? (NDIM == 3 ? 2 : 6) : 3;
  // the faces' mean field: 2D in registers over the loop; 3D (24 of them) from B in shared memory
  static constexpr bool FACES_KEPT = NDIM == 2;
  // k-th ghost cell of the ring region -> region coordinates
  static __device__ __forceinline__ void ghost(int k, int& ri, int& rj, int& rk) {
    rk = NDIM == 3 ? 0 : 1;
    if (NDIM == 3) {
      constexpr int PER = R * R - NB * NB;                      // ghosts of an inner plane
      if (k < 2 * R * R) {
        rk = k < R * R ? 0 : R - 1;
        k %= R * R;
        rj = k / R;
        ri = k % R;
        return;
      }
      k -= 2 * R * R;
      rk = 1 + k / PER;
      k %= PER;
    }
    if (k < 2 * R) {
      rj = k < R ? 0 : R - 1;
      ri = k % R;
    } else {
      k -= 2 * R;
      rj = 1 + k / 2;
      ri = k % 2 ? R - 1 : 0;
    }
  }
};

// The substep loop of one step (CondLoopLaunch), one leaf per CTA of a cooperative launch.
// A thread keeps its cell's state -- an interior cell's, a ring cell's -- in registers over
// the loop; T and kappa of the region are in shared memory.  Per substep: the interior
// energies (cond_rate, as conduction_kernel), their new T and kappa, and, of the cells next to
// the leaf's faces, the energy as an exchange word; each ring thread waits for the word of the
// interior cell its ghost copies (all regions are copies here, whose first ghost layer reads
// interior cells) and takes T and kappa of it.  Words alternate between two slots: a leaf
// writes slot it & 1 again only after its neighbours' words of the substep between, which they
// write after they have read that slot.  Leaves of different problems never wait for one
// another, so each runs its own problem's substeps.
//
// A substep is latency: two CTA barriers and one trip of a word through L2.  256^2 (256 leaves
// of 16^2, FP32): 6.4 us per substep with a grid barrier and the energies in the spare state
// buffers -> 1.8 us.
template <typename T, int NDIM, int NB>
__global__ void __launch_bounds__(CondLoopShape<NDIM, NB>::THREADS, sizeof(T) == 4 ? CondLoopShape<NDIM, NB>::MIN_CTAS : 1)
cond_loop_kernel(CondLoopLaunch L) {
  using G = Geo<NDIM, NB>;
  using SH = CondLoopShape<NDIM, NB>;
  constexpr int NP = G::NP, S = G::S, R = SH::R, NR = SH::NR, NI = SH::NI, W = XWords<T>::N;
  extern __shared__ __align__(16) unsigned char csm[];
  T* sT = reinterpret_cast<T*>(csm);
  T* sK = sT + NR;
  T* sB = sK + NR;                                    // 3D: [3][NR]
  __shared__ int failed;
  const int blk = L.blocks[blockIdx.x], tid = threadIdx.x;
  const BlockGeo gg = L.geo[blk];
  const int ns = L.nsub[gg.problem];
  const T h = (T)L.hsub[gg.problem];
  T* ub = (T*)L.u + (size_t)blk * NV * S;
  Phys<T> P;
  P.gamma = (T)L.gamma;
  P.gm1 = (T)(L.gamma - 1.0);
  P.ch = T(0);
  P.tau = (T)L.tau;
  const T k0 = (T)L.kappa0, gmax = (T)L.grad_t_max;
  const CondDx<T> X(gg);
  const int ro[3] = {1, R, R * R};
  const int po[3] = {1, NP, NP * NP};
  unsigned long long* const slot[2] = {L.words, L.words + (size_t)L.nblocks * NI * W};
  if (tid == 0) failed = 0;

  // the interior cell
  const bool inner = tid < NI;
  int r = 0, c = 0;
  bool shown = false;                                 // its energy is read by other leaves
  T w[NV];
  CondFaces<T> cf[SH::FACES_KEPT ? NDIM : 1];
  if (inner) {
    const int i = tid % NB, j = (tid / NB) % NB, k = NDIM == 3 ? tid / (NB * NB) : 0;
    r = ((NDIM == 3 ? k + 1 : 0) * R + j + 1) * R + i + 1;
    c = ((NDIM == 3 ? k + NG : 0) * NP + j + NG) * NP + i + NG;
    shown = i == 0 || i == NB - 1 || j == 0 || j == NB - 1 || (NDIM == 3 && (k == 0 || k == NB - 1));
    load_global<T>(ub, S, c, w);
    if (SH::FACES_KEPT && L.mode != 1) {
#pragma unroll
      for (int d = 0; d < NDIM; ++d) cond_faces<T>(ub + (size_t)BX * S, S, c, po[d], cf[SH::FACES_KEPT ? d : 0]);
    }
    cond_tk<T>(w, P, k0, sT[r], sK[r]);
  }
  auto keep_b = [&](int at, const T* q) {
    if (!SH::FACES_KEPT)
#pragma unroll
      for (int j = 0; j < 3; ++j) sB[j * NR + at] = q[BX + j];
  };
  if (inner) keep_b(r, w);
  // the ring cell, and the word of the interior cell it copies
  const bool ring = tid >= SH::RING0 && tid < SH::RING0 + SH::NG1;
  int rg = 0;
  size_t src = 0;
  constexpr bool ONE_CELL = SH::RING0 == NI;          // no thread has a cell of each kind
  T w2[ONE_CELL ? 1 : NV];
  T* const wg = ONE_CELL ? w : w2;
  if (ring) {
    int ri, rj, rk;
    SH::ghost(tid - SH::RING0, ri, rj, rk);
    rg = ((NDIM == 3 ? rk : 0) * R + rj) * R + ri;
    load_global<T>(ub, S, ((NDIM == 3 ? rk + 1 : 0) * NP + rj + 1) * NP + ri + 1, wg);
    cond_tk<T>(wg, P, k0, sT[rg], sK[rg]);
    keep_b(rg, wg);
    const int rx = ri == 0 ? 0 : (ri == R - 1 ? 2 : 1), ry = rj == 0 ? 0 : (rj == R - 1 ? 2 : 1);
    const int rz = NDIM == 3 ? (rk == 0 ? 0 : (rk == R - 1 ? 2 : 1)) : 1;
    const GhostRegion g = L.regions[(size_t)blk * 27 + rx + 3 * ry + 9 * rz];
    const int si = g.m[0] * (ri + 1) + g.a[0] - NG, sj = g.m[1] * (rj + 1) + g.a[1] - NG;
    const int sk = NDIM == 3 ? g.m[2] * (rk + 1) + g.a[2] - NG : 0;
    src = ((size_t)g.src * NI + (sk * NB + sj) * NB + si) * W;
  }
  const size_t own = ((size_t)blk * NI + tid) * W;
  __syncthreads();
  bool ok = true;
  for (int it = 0; it < ns; ++it) {
    const unsigned tag = L.tag0 + (unsigned)it;
    const bool more = it + 1 < ns;
    if (inner) {
      auto faces = [&](int d) {
        if (SH::FACES_KEPT) return cf[SH::FACES_KEPT ? d : 0];
        CondFaces<T> f;
        if (L.mode != 1) cond_faces<T>(sB, NR, r, ro[d], f);
        return f;
      };
      auto face = [](int, const T*) {};
      const T acc = cond_rate<T, NDIM>(sT, sK, r, ro, X, gmax, L.mode, faces, face);
      w[EN] = w[EN] + pmul(h, acc);
      if (shown && more) put_value(slot[it & 1] + own, tag, w[EN]);
    }
    if (!more) break;
    __syncthreads();                                  // every rate has read T and kappa
    if (inner) cond_tk<T>(w, P, k0, sT[r], sK[r]);
    if (ring) {
      if (get_value(slot[it & 1] + src, tag, L.fail_waits, wg[EN])) cond_tk<T>(wg, P, k0, sT[rg], sK[rg]);
      else failed = 1;
    }
    __syncthreads();
    if (failed) {
      ok = false;
      break;
    }
  }
  if (!ok) {
    if (tid == 0) atomicOr(L.err_word, 4u);
    return;
  }
  if (ns > 0 && inner) ub[(size_t)EN * S + c] = w[EN];
}

}  // namespace mapgb
