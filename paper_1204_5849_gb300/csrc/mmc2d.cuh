// mmc2d.cuh -- the 2D MMC update of one block plane (Sec. 3.1) with every flux evaluated once.
//
// MMC splits the fluxes of u and of u~ at every face with that face's speeds, so a face reads
// the flux and speed of four u cells and two u~ cells, and the predictor those of three per
// direction.  Evaluated where they are used, each cell's flux is computed about 3.5 times
// over; the step is bound by instruction issue, so that was most of its time.  Here
//   1. cell_fluxes: flux and speed of u, both directions, once per padded cell, into shared
//      memory (six components: those of rho, B_d and psi are m_d, psi and c_h^2 B_d);
//   2. predict: u~ on the ring from them;
//   3. faces: a thread walks a few consecutive faces of one grid line, so u's values slide
//      through registers and the flux of u~ is evaluated once per cell and line.
// y lines run on exchanged states: F_y(U) = P F_x(P U), the same operations (exch_xy).
//
// 32640 16^2 blocks, FP32: 967 us per step with every face and predictor on its own (3012
// thread instructions per cell) -> 893 us (2363).
#pragma once
#include "physics.cuh"

namespace mapgb {
namespace mmc2d {

// flux components kept per cell and direction, in the frame of the direction (N normal, T the
// other in-plane one), and the speed
enum { FMN = 0, FMT = 1, FMZ = 2, FBT = 3, FBZ = 4, FEN = 5, SPD = 6, NQ = 7 };

// components of the state in the frame of direction yd: variable of the k-th
__device__ __forceinline__ int var_of(bool yd, int v) {
  return v == MX ? (yd ? MY : MX) : v == MY ? (yd ? MX : MY) : v == BX ? (yd ? BY : BX) : v == BY ? (yd ? BX : BY) : v;
}

template <typename T>
__device__ __forceinline__ void keep(const T* f, T* q) {       // f in the direction's frame
  q[FMN] = f[MX];
  q[FMT] = f[MY];
  q[FMZ] = f[MZ];
  q[FBT] = f[BY];
  q[FBZ] = f[BZ];
  q[FEN] = f[EN];
}

// the whole flux from the kept components and the state, both in the direction's frame
template <typename T>
__device__ __forceinline__ T flux_of(int v, const T* q, const T* w, const Phys<T>& P) {
  switch (v) {
    case RHO: return w[MX];
    case MX: return q[FMN];
    case MY: return q[FMT];
    case MZ: return q[FMZ];
    case BX: return w[PSI];
    case BY: return q[FBT];
    case BZ: return q[FBZ];
    case EN: return q[FEN];
    default: return P.ch * P.ch * w[BX];
  }
}

// 1. R[2][NQ][P2] of the padded plane su[9][P2] (its corner 2x2 cells are not read)
template <typename T, int NB, int NT>
__device__ __forceinline__ void cell_fluxes(const T* su, T* R, const Phys<T>& P, int tid) {
  constexpr int NP = NB + 4, P2 = NP * NP;
  for (int c = tid; c < P2; c += NT) {
    T w[NV], f[NV], q[NQ];
#pragma unroll
    for (int v = 0; v < NV; ++v) w[v] = su[v * P2 + c];
    const T p = pressure<T>(w, P);
    flux_p<T, 0>(w, p, P, f);
    keep<T>(f, q);
    q[SPD] = alpha_p<T, 0>(w, p, P);
#pragma unroll
    for (int k = 0; k < NQ; ++k) R[k * P2 + c] = q[k];
    flux_p<T, 1>(w, p, P, f);
    const T fy[NV] = {f[RHO], f[MY], f[MX], f[MZ], f[BY], f[BX], f[BZ], f[EN], f[PSI]};
    keep<T>(fy, q);
    q[SPD] = alpha_p<T, 1>(w, p, P);
#pragma unroll
    for (int k = 0; k < NQ; ++k) R[(NQ + k) * P2 + c] = q[k];
  }
}

// 2. u~ at padded cell c: u - sum_d lam_d (h_{i+1/2} - h_{i-1/2}), h = f+_i + f-_{i+1}
template <typename T, int NB>
__device__ __forceinline__ void predict(const T* su, const T* R, int c, const T* lam, const Phys<T>& P, T* acc) {
  constexpr int NP = NB + 4, P2 = NP * NP;
  T u[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = u[v] = su[v * P2 + c];
#pragma unroll
  for (int d = 0; d < 2; ++d) {
    const int st = d ? NP : 1;
    const T* Rd = R + d * NQ * P2;
    T w[NV], wm[NV], wp[NV], q[NQ], qm[NQ], qp[NQ];   // in the frame of d
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int s = var_of(d == 1, v);
      w[v] = u[s];
      wm[v] = su[s * P2 + c - st];
      wp[v] = su[s * P2 + c + st];
    }
#pragma unroll
    for (int k = 0; k < NQ; ++k) {
      if (k == SPD || sizeof(T) == 8) q[k] = Rd[k * P2 + c];
      qm[k] = Rd[k * P2 + c - st];
      qp[k] = Rd[k * P2 + c + st];
    }
    const T am = qm[SPD] > q[SPD] ? qm[SPD] : q[SPD], ap = q[SPD] > qp[SPD] ? q[SPD] : qp[SPD];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int s = var_of(d == 1, v);
      const bool glm = v == BX || v == PSI;
      const T sm = glm ? P.ch : am, sp = glm ? P.ch : ap;
      const T fm = flux_of<T>(v, qm, wm, P), fp = flux_of<T>(v, qp, wp, P);
      if (sizeof(T) == 8) {
        // the order of the split form
        const T f0 = flux_of<T>(v, q, w, P);
        const T hp = T(0.5) * (f0 + sp * w[v]) + T(0.5) * (fp - sp * wp[v]);
        const T hm = T(0.5) * (fm + sm * wm[v]) + T(0.5) * (f0 - sm * w[v]);
        acc[s] -= lam[d] * (hp - hm);
      } else {
        // h_{i+1/2} - h_{i-1/2} with the cell's own flux cancelled and the dissipation taken on
        // differences
        const T g = (fp - fm) - sp * (wp[v] - w[v]) + sm * (w[v] - wm[v]);
        acc[s] -= (T(0.5) * lam[d]) * g;
      }
    }
  }
}

// one face from the states and kept fluxes of u_{i-1}..u_{i+2} (w, q) and u~_i, u~_{i+1}
// (t, g); the operations of mmc_face, in its order in FP64
template <typename T, int LIM>
__device__ __forceinline__ void face(const T (&w)[4][NV], const T (&q)[4][NQ], const T (&t)[2][NV],
                                     const T (&g)[2][NQ], const Phys<T>& P, T* F) {
  const T alpha = q[1][SPD] > q[2][SPD] ? q[1][SPD] : q[2][SPD];
  const T alphat = g[0][SPD] > g[1][SPD] ? g[0][SPD] : g[1][SPD];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const bool glm = v == BX || v == PSI;
    const T a = glm ? P.ch : alpha, b = glm ? P.ch : alphat;
    const T f0 = flux_of<T>(v, q[0], w[0], P), f1 = flux_of<T>(v, q[1], w[1], P);
    const T f2 = flux_of<T>(v, q[2], w[2], P), f3 = flux_of<T>(v, q[3], w[3], P);
    const T g0 = flux_of<T>(v, g[0], t[0], P), g1 = flux_of<T>(v, g[1], t[1], P);
    if (sizeof(T) == 8) {
      const T fp = T(0.5) * (f1 + a * w[1][v]), fm = T(0.5) * (f2 - a * w[2][v]);
      const T gpl = T(0.5) * (g0 + b * t[0][v]) + -(T(0.5) * (f0 + a * w[0][v]));
      const T gmc = fm - T(0.5) * (g0 - b * t[0][v]);
      const T gpc = T(0.5) * (g1 + b * t[1][v]) - fp;
      const T gmr = T(0.5) * (f3 - a * w[3][v]) - T(0.5) * (g1 - b * t[1][v]);
      F[v] = (fp + fm) + T(0.5) * (limiter<T, LIM>(gpl, gpc) - limiter<T, LIM>(gmr, gmc));
    } else {
      // twice the split fluxes (the limiters scale): the halves go into the last two factors
      const T fp = f1 + a * w[1][v], fm = f2 - a * w[2][v];
      const T gpl = (g0 + b * t[0][v]) - (f0 + a * w[0][v]);
      const T gmc = fm - (g0 - b * t[0][v]);
      const T gpc = (g1 + b * t[1][v]) - fp;
      const T gmr = (f3 - a * w[3][v]) - (g1 - b * t[1][v]);
      F[v] = T(0.5) * (fp + fm) + T(0.25) * (limiter<T, LIM>(gpl, gpc) - limiter<T, LIM>(gmr, gmc));
    }
  }
}

// 3. faces of the plane into sfx / sfy (layout of the step kernel's face buffer): thread tid
// takes a segment of one of the 2 NB grid lines.  The first faces of the segments of a warp
// differ modulo 4, which spreads the lines' rows (strides 20 and 12) over the banks.
template <int NB, int SEG>
__device__ __forceinline__ int segment_start(int s) {
  if (SEG == 4) return NB == 16 ? (s == 0 ? 0 : s == 1 ? 5 : s == 2 ? 9 : s == 3 ? 14 : 17)
                                : (s == 0 ? 0 : s == 1 ? 3 : s == 2 ? 5 : s == 3 ? 6 : 9);
  return s * (NB + 1) / SEG;
}

template <typename T, int NB, int NT, int LIM>
__device__ __forceinline__ void faces(const T* su, const T* st, const T* R, T* sfx, T* sfy, const Phys<T>& P, int tid) {
  constexpr int NP = NB + 4, P2 = NP * NP, RW = NB + 2, RING = RW * RW, NFACE = NB * (NB + 1);
  constexpr int SEG = NT / (2 * NB);
  static_assert(NT % (2 * NB) == 0, "whole segments per line");
  const int line = tid % NB, seg = (tid / NB) % SEG;
  const bool yd = tid >= NB * SEG;
  const int k0 = segment_start<NB, SEG>(seg), k1 = segment_start<NB, SEG>(seg + 1);
  const int us = yd ? NP : 1, rs = yd ? RW : 1;                  // strides along the line
  // face k lies between padded cells k + 1 and k + 2 of the line, ring cells k and k + 1
  int c = yd ? k0 * NP + line + 2 : (line + 2) * NP + k0;        // padded cell k0
  int r = yd ? k0 * RW + line + 1 : (line + 1) * RW + k0;        // ring cell k0
  const T* Rd = R + (yd ? NQ * P2 : 0);
  T w[4][NV], q[4][NQ], t[2][NV], g[2][NQ];
  auto load_u = [&](int at, T* x, T* y) {
#pragma unroll
    for (int v = 0; v < NV; ++v) x[v] = su[var_of(yd, v) * P2 + at];
#pragma unroll
    for (int k = 0; k < NQ; ++k) y[k] = Rd[k * P2 + at];
  };
  auto load_t = [&](int at, T* x, T* y) {
#pragma unroll
    for (int v = 0; v < NV; ++v) x[v] = st[var_of(yd, v) * RING + at];
    const T p = pressure<T>(x, P);
    T f[NV];
    flux_p<T, 0>(x, p, P, f);
    keep<T>(f, y);
    y[SPD] = alpha_p<T, 0>(x, p, P);
  };
  load_u(c, w[0], q[0]);
  load_u(c + us, w[1], q[1]);
  load_u(c + 2 * us, w[2], q[2]);
  load_t(r, t[0], g[0]);
#pragma unroll 1
  for (int k = k0; k < k1; ++k) {
    load_u(c + 3 * us, w[3], q[3]);
    load_t(r + rs, t[1], g[1]);
    T F[NV];
    face<T, LIM>(w, q, t, g, P, F);
    T* dst = yd ? sfy + k * NB + line : sfx + line * (NB + 1) + k;
#pragma unroll
    for (int v = 0; v < NV; ++v) dst[var_of(yd, v) * NFACE] = F[v];
    c += us;
    r += rs;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      w[0][v] = w[1][v];
      w[1][v] = w[2][v];
      w[2][v] = w[3][v];
      t[0][v] = t[1][v];
    }
#pragma unroll
    for (int v = 0; v < NQ; ++v) {
      q[0][v] = q[1][v];
      q[1][v] = q[2][v];
      q[2][v] = q[3][v];
      g[0][v] = g[1][v];
    }
  }
}

}  // namespace mmc2d
}  // namespace mapgb
