// Internal declarations of the two-phase kernels (step_mp.cu).
#pragma once
#include <cuda_runtime.h>

namespace lbmk {

// Constants of a two-phase solve in the working precision R (host-filled, so the
// FP32 kernels convert nothing per thread on GB300's slow FP64 pipe).
template <typename R>
struct MpConst {
  R c, rho_g, rho_g_lo, drl, drl_lo;  // drl = rho_l - rho_g; _lo: what R rounds off
  R hdt_ic, Fx, Fy;                   // dt / (2 c), body force
  R kb, kl, kg;                       // dt / (2 c) mu grad phi and (dt / 2) c grad rho from the
                                      // stencil sums r = 36 dx / 3 grad phi (see mp_macro)
  R tau0, dtau, zg, dzeta;            // tau / dt = tau0 + phi dtau, or (zg + phi dzeta) / rho + 1/2
  R om_h, hom_h, s1, s2;              // dt / tau_phi and half of it; sources of the odd h pairs
};

// Two-phase solve; each axis periodic or bounded by resting half-way walls on both
// sides.  State planes: z_0..8, h_0..4, (phi u)_x, (phi u)_y of the previous step.
struct MpParams {
  int nx, ny, pitch;
  long long plane;
  double c, cs2, dt, dx, inv_c;
  double rho_l, rho_g, nu_l, nu_g;
  double kappa, beta, W, tauphi;
  int nu_rule, z_mrt, qy_literal;
  int xwall, ywall;  // 1: the axis ends at resting walls (bounce-back, mirrored phi)
  double Fx, Fy;
  int forced;        // a body force or a force field acts
  MpConst<double> kd;
  MpConst<float> kf;
  const void *force;  // 2 planes or null
  int local;          // 1: src holds the pre-collision state itself (after init)
  const void *src;
  void *dst;
};

template <typename R>
__device__ __forceinline__ const MpConst<R> &KM(const MpParams &P);
template <>
__device__ __forceinline__ const MpConst<double> &KM<double>(const MpParams &P) { return P.kd; }
template <>
__device__ __forceinline__ const MpConst<float> &KM<float>(const MpParams &P) { return P.kf; }

cudaError_t mp_step(const MpParams &P, int prec, cudaStream_t s);
// Equilibria of the given fields (pre-collision state of time 0) into P.dst.
cudaError_t mp_init(const MpParams &P, int prec, const double *phi0, const double *ux0, const double *uy0,
                    const double *p0, cudaStream_t s);
cudaError_t mp_moments(const MpParams &P, int prec, unsigned mask, double *out, cudaStream_t s);
cudaError_t mp_integrals(const MpParams &P, int prec, double *partials, int max_blocks, double *out5, const double *flag,
                         cudaStream_t s);
int mp_integral_blocks(int nx, int ny);

}  // namespace lbmk
