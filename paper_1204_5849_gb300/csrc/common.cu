// common.cu -- per-problem time-step finalisation (precision independent).
#include <math.h>

#include "chain.cuh"
#include "map_internal.hpp"

namespace mapgb {

// dt, c_h, c_p and the psi damping factor of each problem from its alpha_g (Sec. 3.7
// time step; Sec. 2 c_h and c_p; eq. MHD-5 damping exp(-dt c_h^2/c_p^2)).  Resets the
// running alpha maximum for the next reduction and, for a fused step, zeroes the
// conservation sums that the step accumulates.
//
// One problem per CTA of two warps.  The kernel is a chain of dependent FP64 operations (a
// quotient, root, logarithm or exponential is 10-20 of them, each some 50 cycles on a pipe
// of 1/64 of the FP32 rate), so its time is the longest chain: warp 0 takes dt and the three
// dt/dx0 quotients, one per lane of a single division; warp 1 takes log(c_d) before dt is
// known and then c_p and the damping.  (One thread per problem, everything in sequence, and a
// memset of the sums beside it: 5.2 us more per step; 128^2 MMC, ten steps and state in and
// out: 299 -> 247 us.)
__global__ void __launch_bounds__(64) finalize_kernel(FinalizeLaunch L) {
  const int p = blockIdx.x, lane = threadIdx.x & 31;
  const bool dt_warp = threadIdx.x < 32;
  const double log_cd = !dt_warp && L.cp_mode == MAP_CP_FROM_CD ? log(L.c_d) : 0.0;
  chain_release();
  chain_begin();
  const ProbDyn d = L.dyn[p];
  __syncthreads();                       // both warps hold the maxima before they are reset
  const double ag = __longlong_as_double((long long)d.alpha_bits);
  double sig = ag;
  if (L.ch_mode == MAP_CH_FIXED && L.ch_fixed > sig) sig = L.ch_fixed;
  double dt = L.c_cfl * d.mindx / ((double)L.ndim * sig);
  if (L.eta > 0.0) {
    const double dtr = L.c_cfl * d.mindx * d.mindx / (2.0 * (double)L.ndim * L.eta);
    if (dtr < dt) dt = dtr;
  }
  // thermal conduction (Sec. 3.6): dt_c = c_cfl min(dx)^2 / (n_dim max(kappa T / p)), the
  // rate read as kappa / rho; without the subcycle it bounds dt
  double dtc = __longlong_as_double(0x7ff0000000000000ll);
  const double kmax = __longlong_as_double((long long)d.kmax_bits);
  if (L.conduction && kmax > 0.0) dtc = L.c_cfl * d.mindx * d.mindx / ((double)L.ndim * kmax);
  if (L.conduction && !L.subcycle && dtc < dt) dt = dtc;
  if (L.dt_override > 0.0) dt = L.dt_override;
  double ch;
  if (L.ch_mode == MAP_CH_AUTO) ch = ag;
  else if (L.ch_mode == MAP_CH_PAPER) ch = L.c_cfl * d.mindx / dt;
  else ch = L.ch_fixed;
  ProbDyn* o = L.dyn + p;
  if (dt_warp) {
    // per-dimension dt/dx at level 0; a level-L block takes 2^L of it, which is dt/dx_L
    // exactly (dx_L = dx0 / 2^L as the host computes it), so blocks divide nothing
    const double q = dt / (lane == 0 ? d.dx0[0] : lane == 1 ? d.dx0[1] : d.dx0[2]);
    if (lane < 3) o->lam0[lane] = q;
    if (lane == 0) {
      o->dt = dt;
      o->ch = ch;
      o->alpha_g = ag;
      o->dtc = dtc;
      o->alpha_bits = 0ull;
      o->kmax_bits = 0ull;
    }
  } else {
    const double cp = L.cp_mode == MAP_CP_FROM_CD ? sqrt(-dt * ch * ch / log_cd) : L.cp_fixed;
    const double damp = cp > 0.0 ? exp(-dt * ch * ch / (cp * cp)) : 1.0;
    if (lane == 0) {
      o->cp = cp;
      o->damp = damp;
    }
    if (L.sums && lane < kNV) L.sums[(size_t)p * kNV + lane] = 0.0;
  }
}

__global__ void zero_alpha_kernel(ProbDyn* dyn, int n) {
  chain_begin();
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < n) {
    dyn[p].alpha_bits = 0ull;
    dyn[p].kmax_bits = 0ull;
  }
}

// dt, c_h, c_p, damping and alpha_g of every problem, stored by the GPU itself into host
// memory it can address (page-locked and mapped): no copy engine takes part, so the store does
// not queue behind the large state copies that the copy engines may be running.
__global__ void speeds_out_kernel(const ProbDyn* __restrict__ dyn, int n, double* __restrict__ out) {
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
    double* o = out + 5 * (size_t)p;
    o[0] = dyn[p].dt;
    o[1] = dyn[p].ch;
    o[2] = dyn[p].cp;
    o[3] = dyn[p].damp;
    o[4] = dyn[p].alpha_g;
  }
}

cudaError_t launch_speeds_out(const ProbDyn* dyn, int n, double* out, cudaStream_t s, long long* cnt) {
  if (cnt) ++*cnt;
  speeds_out_kernel<<<1, 128, 0, s>>>(dyn, n, out);
  return cudaGetLastError();
}

cudaError_t launch_finalize(const FinalizeLaunch& L, cudaStream_t s, long long* cnt) {
  if (cnt) ++*cnt;
  return launch_chained(finalize_kernel, L.nprob, 64, 0, s, L);
}

cudaError_t launch_zero_alpha(ProbDyn* dyn, int n, cudaStream_t s, long long* cnt) {
  if (cnt) ++*cnt;
  return launch_chained(zero_alpha_kernel, (n + 127) / 128, 128, 0, s, dyn, n);
}

}  // namespace mapgb
