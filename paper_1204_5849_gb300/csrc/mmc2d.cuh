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
// thread instructions per cell) -> 893 us (2363) -> 867 us (1932) with the components of the
// FP32 form in pairs.  Three CTAs reside per SM (68 KB each); what is left between the issue
// slots (48 % busy) is dependent latency and the barriers of the four phases.
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

// FP32: the frame's components as pairs (the GLM pair last, then the energy alone), so the
// split fluxes of two components are one paired operation each
enum { PA = 0, PB = 1, PC = 2, PG = 3, NPAIR = 4 };     // (rho, B_T), (m_N, m_T), (m_Z, B_Z), (B_N, psi)
struct Comps {
  float2 p[NPAIR];
  float e;
};
// the pair components of a state (frame order w[NV]) and of its flux
__device__ __forceinline__ void pairs_of(const float* w, Comps& c) {
  c.p[PA] = make_float2(w[RHO], w[BY]);
  c.p[PB] = make_float2(w[MX], w[MY]);
  c.p[PC] = make_float2(w[MZ], w[BZ]);
  c.p[PG] = make_float2(w[BX], w[PSI]);
  c.e = w[EN];
}
__device__ __forceinline__ void flux_pairs_of(const float* q, const Comps& w, float ch2, Comps& c) {
  c.p[PA] = make_float2(w.p[PB].x, q[FBT]);
  c.p[PB] = make_float2(q[FMN], q[FMT]);
  c.p[PC] = make_float2(q[FMZ], q[FBZ]);
  c.p[PG] = make_float2(w.p[PG].y, ch2 * w.p[PG].x);
  c.e = q[FEN];
}

// 1. in FP32: two x-neighbours per thread, one in each lane of the paired operations; of the
// outermost rows only the pairs over the interior columns are read
template <int NB, int NT>
__device__ __forceinline__ void cell_fluxes(const float* su, float* R, const Phys<float>& P, int tid) {
  constexpr int NP = NB + 4, P2 = NP * NP, EDGE = NB / 2, FULL = NP / 2;
  constexpr int TOTAL = 2 * EDGE + (NB + 2) * FULL;
  for (int g = tid; g < TOTAL; g += NT) {
    int row, col;
    if (g < 2 * EDGE) {
      row = g < EDGE ? 0 : NP - 1;
      col = NG + 2 * (g % EDGE);
    } else {
      row = 1 + (g - 2 * EDGE) / FULL;
      col = 2 * ((g - 2 * EDGE) % FULL);
    }
    const int c = row * NP + col;
    float2 w[NV], f[NV], al;
#pragma unroll
    for (int v = 0; v < NV; ++v) w[v] = *reinterpret_cast<const float2*>(su + v * P2 + c);
    auto put = [&](int k, float2 x) { *reinterpret_cast<float2*>(R + k * P2 + c) = x; };
    pair::flux2<0>(w, P, f, &al);
    put(FMN, f[MX]);
    put(FMT, f[MY]);
    put(FMZ, f[MZ]);
    put(FBT, f[BY]);
    put(FBZ, f[BZ]);
    put(FEN, f[EN]);
    put(SPD, al);
    pair::flux2<1>(w, P, f, &al);
    put(NQ + FMN, f[MY]);
    put(NQ + FMT, f[MX]);
    put(NQ + FMZ, f[MZ]);
    put(NQ + FBT, f[BX]);
    put(NQ + FBZ, f[BZ]);
    put(NQ + FEN, f[EN]);
    put(NQ + SPD, al);
  }
}

// 2. in FP32: h_{i+1/2} - h_{i-1/2} with the cell's own flux cancelled and the dissipation
// taken on differences, two components at a time
template <int NB>
__device__ __forceinline__ void predict(const float* su, const float* R, int c, const float* lam, const Phys<float>& P,
                                        float* acc) {
  constexpr int NP = NB + 4, P2 = NP * NP;
  const float ch2 = P.ch * P.ch;
  float u[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) u[v] = acc[v] = su[v * P2 + c];
#pragma unroll
  for (int d = 0; d < 2; ++d) {
    const int st = d ? NP : 1;
    const float* Rd = R + d * NQ * P2 + c;
    float x[NV], q[NQ];
    Comps w, wm, wp, fm, fp;
    auto state = [&](int o, Comps& s) {
#pragma unroll
      for (int v = 0; v < NV; ++v) x[v] = su[var_of(d == 1, v) * P2 + c + o];
      pairs_of(x, s);
    };
    auto flux = [&](int o, const Comps& s, Comps& f) {
#pragma unroll
      for (int k = 0; k < SPD; ++k) q[k] = Rd[k * P2 + o];
      flux_pairs_of(q, s, ch2, f);
    };
#pragma unroll
    for (int v = 0; v < NV; ++v) x[v] = u[var_of(d == 1, v)];
    pairs_of(x, w);
    state(-st, wm);
    state(st, wp);
    flux(-st, wm, fm);
    flux(st, wp, fp);
    const float a0 = Rd[SPD * P2];
    const float am = dmax(Rd[SPD * P2 - st], a0), ap = dmax(a0, Rd[SPD * P2 + st]);
    const float hl = -0.5f * lam[d];
    auto upd = [&](int k, float sm, float sp, float& o0, float& o1) {
      float2 g = pair::sub(fp.p[k], fm.p[k]);
      g = pair::fma(pair::splat(-sp), pair::sub(wp.p[k], w.p[k]), g);
      g = pair::fma(pair::splat(sm), pair::sub(w.p[k], wm.p[k]), g);
      const float2 o = pair::fma(pair::splat(hl), g, make_float2(o0, o1));
      o0 = o.x;
      o1 = o.y;
    };
    upd(PA, am, ap, acc[RHO], acc[d ? BX : BY]);
    upd(PB, am, ap, acc[d ? MY : MX], acc[d ? MX : MY]);
    upd(PC, am, ap, acc[MZ], acc[BZ]);
    upd(PG, P.ch, P.ch, acc[d ? BY : BX], acc[PSI]);
    const float ge = (fp.e - fm.e) - ap * (wp.e - w.e) + am * (w.e - wm.e);
    acc[EN] += hl * ge;
  }
}

// FP32 minmod as max(min(a, b), 0) + min(max(a, b), 0), the inner two handing a NaN on (a gradient
// without a value limits to 0, as minmod_lim's): one operation more on the ALU pipe than
// minmod_lim, one of the five on the FMA pipe, and faster in this walk (32640 16^2 blocks, four
// steps: 3819 us against 3858)
template <int LIM>
__device__ __forceinline__ float limit(float a, float b) {
  if (LIM != 0) return limiter<float, LIM>(a, b);
  float lo, hi;
  asm("min.ftz.NaN.f32 %0, %1, %2;" : "=f"(lo) : "f"(a), "f"(b));
  asm("max.ftz.NaN.f32 %0, %1, %2;" : "=f"(hi) : "f"(a), "f"(b));
  return fmaxf(lo, 0.0f) + fminf(hi, 0.0f);
}
template <int LIM>
__device__ __forceinline__ float2 limit2(float2 a, float2 b) {
  if (LIM != 0) return pair::limiter2<LIM>(a, b);
  return make_float2(limit<LIM>(a.x, b.x), limit<LIM>(a.y, b.y));
}

// one component (pair) of a face: twice the split fluxes (the limiters scale), the halves in
// the last two factors
template <int LIM>
__device__ __forceinline__ float2 combine(float2 a, float2 b, float2 w0, float2 w1, float2 w2, float2 w3, float2 f0,
                                          float2 f1, float2 f2, float2 f3, float2 t0, float2 t1, float2 g0, float2 g1) {
  const float2 na = make_float2(-a.x, -a.y), nb = make_float2(-b.x, -b.y);
  const float2 fp = pair::fma(a, w1, f1), fm = pair::fma(na, w2, f2);
  const float2 gpl = pair::sub(pair::fma(b, t0, g0), pair::fma(a, w0, f0));
  const float2 gmc = pair::sub(fm, pair::fma(nb, t0, g0));
  const float2 gpc = pair::sub(pair::fma(b, t1, g1), fp);
  const float2 gmr = pair::sub(pair::fma(na, w3, f3), pair::fma(nb, t1, g1));
  const float2 l = pair::sub(limit2<LIM>(gpl, gpc), limit2<LIM>(gmr, gmc));
  return pair::fma(pair::splat(0.25f), l, pair::mul(pair::splat(0.5f), pair::add(fp, fm)));
}

// 1. R[2][NQ][P2] of the padded plane su[9][P2]
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
      q[k] = Rd[k * P2 + c];
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
      const T f0 = flux_of<T>(v, q, w, P);
      const T hp = T(0.5) * (f0 + sp * w[v]) + T(0.5) * (fp - sp * wp[v]);
      const T hm = T(0.5) * (fm + sm * wm[v]) + T(0.5) * (f0 - sm * w[v]);
      acc[s] -= lam[d] * (hp - hm);
    }
  }
}

// one face from the states and kept fluxes of u_{i-1}..u_{i+2} (w, q) and u~_i, u~_{i+1}
// (t, g); the operations of mmc_face, in its order
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
    const T fp = T(0.5) * (f1 + a * w[1][v]), fm = T(0.5) * (f2 - a * w[2][v]);
    const T gpl = T(0.5) * (g0 + b * t[0][v]) + -(T(0.5) * (f0 + a * w[0][v]));
    const T gmc = fm - T(0.5) * (g0 - b * t[0][v]);
    const T gpc = T(0.5) * (g1 + b * t[1][v]) - fp;
    const T gmr = T(0.5) * (f3 - a * w[3][v]) - T(0.5) * (g1 - b * t[1][v]);
    F[v] = (fp + fm) + T(0.5) * (limiter<T, LIM>(gpl, gpc) - limiter<T, LIM>(gmr, gmc));
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

// the longest segment
template <int NB, int SEG>
__host__ __device__ constexpr int segment_most() {
  return SEG == 4 ? (NB == 16 ? 5 : 3) : (NB + SEG) / SEG;
}

// FP32: the walk unrolled, so the values of the line's cells stay where they are
template <int NB, int NT, int LIM>
__device__ __forceinline__ void faces_f32(const float* su, const float* st, const float* R, float* sfx, float* sfy,
                                          const Phys<float>& P, int tid) {
  constexpr int NP = NB + 4, P2 = NP * NP, RW = NB + 2, RING = RW * RW, NFACE = NB * (NB + 1);
  constexpr int SEG = NT / (2 * NB), MOST = segment_most<NB, SEG>();
  static_assert(NT % (2 * NB) == 0, "whole segments per line");
  const int line = tid % NB, seg = (tid / NB) % SEG;
  const bool yd = tid >= NB * SEG;
  const int k0 = segment_start<NB, SEG>(seg), n = segment_start<NB, SEG>(seg + 1) - k0;
  const int us = yd ? NP : 1, rs = yd ? RW : 1;                  // strides along the line
  const float* uc = su + (yd ? k0 * NP + line + 2 : (line + 2) * NP + k0);
  const float* rc = st + (yd ? k0 * RW + line + 1 : (line + 1) * RW + k0);
  const float* Rc = R + (yd ? NQ * P2 + k0 * NP + line + 2 : (line + 2) * NP + k0);
  float* dst = yd ? sfy + k0 * NB + line : sfx + line * (NB + 1) + k0;
  const int ds = yd ? NB : 1;
  const float ch2 = P.ch * P.ch;
  Comps w[4], f[4], t[2], g[2];
  float al[4], at[2];
  auto load_u = [&](int k, Comps& s, Comps& fl, float& a) {
    float x[NV], q[NQ];
#pragma unroll
    for (int v = 0; v < NV; ++v) x[v] = uc[var_of(yd, v) * P2 + k * us];
#pragma unroll
    for (int j = 0; j < SPD; ++j) q[j] = Rc[j * P2 + k * us];
    a = Rc[SPD * P2 + k * us];
    pairs_of(x, s);
    flux_pairs_of(q, s, ch2, fl);
  };
  auto load_t = [&](int k, Comps& s, Comps& fl, float& a) {
    float x[NV], y[NV], q[NQ];
#pragma unroll
    for (int v = 0; v < NV; ++v) x[v] = rc[var_of(yd, v) * RING + k * rs];
    const float p = pressure<float>(x, P);
    flux_p<float, 0>(x, p, P, y);
    keep<float>(y, q);
    a = alpha_p<float, 0>(x, p, P);
    pairs_of(x, s);
    flux_pairs_of(q, s, ch2, fl);
  };
  load_u(0, w[0], f[0], al[0]);
  load_u(1, w[1], f[1], al[1]);
  load_u(2, w[2], f[2], al[2]);
  load_t(0, t[0], g[0], at[0]);
#pragma unroll
  for (int k = 0; k < MOST; ++k) {
    if (k >= n) break;
    const int c0 = k & 3, c1 = (k + 1) & 3, c2 = (k + 2) & 3, c3 = (k + 3) & 3, e0 = k & 1, e1 = e0 ^ 1;
    load_u(k + 3, w[c3], f[c3], al[c3]);
    load_t(k + 1, t[e1], g[e1], at[e1]);
    // (a face whose u~ has no speed on its right takes the first-order flux: its gradients are NaN)
    const float a = dmax(al[c1], al[c2]), b = dmax(at[e0], at[e1]);
    float F[NV];
    auto comb = [&](int p, float sa, float sb, float& o0, float& o1) {
      const float2 x = combine<LIM>(pair::splat(sa), pair::splat(sb), w[c0].p[p], w[c1].p[p], w[c2].p[p], w[c3].p[p],
                                    f[c0].p[p], f[c1].p[p], f[c2].p[p], f[c3].p[p], t[e0].p[p], t[e1].p[p], g[e0].p[p],
                                    g[e1].p[p]);
      o0 = x.x;
      o1 = x.y;
    };
    comb(PA, a, b, F[RHO], F[BY]);
    comb(PB, a, b, F[MX], F[MY]);
    comb(PC, a, b, F[MZ], F[BZ]);
    comb(PG, P.ch, P.ch, F[BX], F[PSI]);
    {
      const float fp = f[c1].e + a * w[c1].e, fm = f[c2].e - a * w[c2].e;
      const float gpl = (g[e0].e + b * t[e0].e) - (f[c0].e + a * w[c0].e);
      const float gmc = fm - (g[e0].e - b * t[e0].e);
      const float gpc = (g[e1].e + b * t[e1].e) - fp;
      const float gmr = (f[c3].e - a * w[c3].e) - (g[e1].e - b * t[e1].e);
      F[EN] = 0.5f * (fp + fm) + 0.25f * (limit<LIM>(gpl, gpc) - limit<LIM>(gmr, gmc));
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) dst[var_of(yd, v) * NFACE + k * ds] = F[v];
  }
}

}  // namespace mmc2d
}  // namespace mapgb
