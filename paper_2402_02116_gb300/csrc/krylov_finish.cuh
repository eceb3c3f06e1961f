// The once-per-problem scalar steps of BiCGSTAB, as device functions of a CTA: run by the last CTA of
// the launch that makes their partials (krylov.cuh, KrylovFinish), or by a one-warp kernel of their
// own (uneven batches and the paper-literal form).
#pragma once

#include "krylov.cuh"
#include "reduce.cuh"
#include "vec.cuh"

namespace dbi {

// A pair of FP64 scalars of the state as the type C of the vectors (FP32: the rounded copies).
template <typename C> __device__ __forceinline__ C state_value(double re, double im, const float (&f)[2]) {
  if constexpr (sizeof(C) == sizeof(float2)) return mk<C>(f[0], f[1]);
  else return mk<C>(re, im);
}
template <typename C> __device__ __forceinline__ C state_alpha(const KState &k) {
  return state_value<C>(k.alpha_re, k.alpha_im, k.al_f);
}
template <typename C> __device__ __forceinline__ C state_omega(const KState &k) {
  return state_value<C>(k.om_re, k.om_im, k.om_f);
}
template <typename C> __device__ __forceinline__ C state_beta(const KState &k) {
  return state_value<C>(k.beta_re, k.beta_im, k.be_f);
}
// The FP32 copies at the values of the FP64 scalars.
__device__ __forceinline__ void round_state(KState &k) {
  k.al_f[0] = float(k.alpha_re); k.al_f[1] = float(k.alpha_im);
  k.om_f[0] = float(k.om_re); k.om_f[1] = float(k.om_im);
  k.be_f[0] = float(k.beta_re); k.be_f[1] = float(k.beta_im);
}

// alpha = rho / <rhat, A p> of problem b from the operator's `nparts` partials. Every thread of the
// CTA must call it.
__device__ __forceinline__ void finish_alpha(KState *st, int b, const double *part, int nparts) {
  double sg[2];
  gather_n<2>(part, nparts, sg);
  if (threadIdx.x == 0) {
    const double2 sigma = make_double2(sg[0], sg[1]);
    const double2 alpha = (sigma.x == 0.0 && sigma.y == 0.0)
                              ? make_double2(0.0, 0.0)
                              : zdiv(make_double2(st[b].rho_re, st[b].rho_im), sigma);
    st[b].alpha_re = alpha.x;
    st[b].alpha_im = alpha.y;
    st[b].al_f[0] = float(alpha.x);
    st[b].al_f[1] = float(alpha.y);
  }
}

// omega = <t, s> / ||t||^2 (zero when the half step already met tol) of problem b from the second
// operator pass's partials and those of ||s||^2.
__device__ __forceinline__ void finish_omega(KState *st, int b, const double *part, int nparts, const double *partS,
                                             int nS, double tol) {
  double q[3], sn[1];
  gather_n<3>(part, nparts, q);
  gather_n<1>(partS, nS, sn);
  if (threadIdx.x == 0) {
    const int half = sn[0] <= tol * tol * st[b].bnorm2;
    const double2 om = (half || q[2] == 0.0) ? make_double2(0.0, 0.0)
                                             : make_double2(q[0] / q[2], q[1] / q[2]);
    st[b].om_re = om.x;
    st[b].om_im = om.y;
    st[b].om_f[0] = float(om.x);
    st[b].om_f[1] = float(om.y);
    st[b].half = half;
    st[b].snorm2 = sn[0];
  }
}

// End of an inverse row tile of problem b that stored its partials (EPI 1 or 2): the last of the
// problem's `tiles` CTAs does the scalar step.
template <int EPI>
__device__ __forceinline__ void finish_tile(const KrylovFinish &fin, int b, const double *part, int tiles) {
  if (EPI == 0 || !fin.st) return;
  if (!last_cta(fin.arrived + b, tiles)) return;
  if constexpr (EPI == 1) finish_alpha(fin.st, b, part, tiles);
  else finish_omega(fin.st, b, part, tiles, fin.partS + size_t(b) * kRedBlocks * kRedSlots, fin.nS, fin.tol);
}

}  // namespace dbi
