// learned_arith.cuh -- the 2D FP32 arithmetic of the corrected scheme: primitive
// recovery, limited slopes and the plain HLL / HLLC face flux.
//
// The same formulas as hydro_device.cuh with other roundings.  The network
// reads its features in BF16, so a state that differs by one rounding can
// round a feature the other way and move the correction by 2^-9 of itself;
// over tens of steps that grows far above FP32 rounding (5e-5 relative after
// 32 steps of a 256^2 shear layer).  The corrected scheme therefore keeps the
// roundings its runs have had, while the plain solver's flux has its own.
#pragma once

#include "hydro_device.cuh"

namespace gh {
namespace lf {

__device__ __forceinline__ float limited_slope(float wm, float wc, float wp, const Geo<float>& g) {
  return minmod3((wc - wm) * g.ticm, (wp - wm) * g.ipm, (wp - wc) * g.tipc);
}

__device__ __forceinline__ float fdiv(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ float frcp(float x) { return __fdividef(1.0f, x); }
__device__ __forceinline__ float sound_speed(float gamma, float p, float n) {
  const float gp = gamma * p;
  return gp * rsqrtf(gp * n);
}

// e D = G D - |S|^2 / 2 in FP64 (products of FP32 values are exact in FP64).
// Kept out of line so that only lanes that need it execute FP64 instructions.
static __device__ __noinline__ float energy_density_times_n_fp64(float n, float s1, float s2, float s3, float G) {
  const double s2d = fma((double)s1, (double)s1, fma((double)s2, (double)s2, (double)s3 * (double)s3));
  return (float)fma(-0.5, s2d, (double)G * (double)n);
}

// e in FP32 where the kinetic energy is at most half of G, else through FP64.
__device__ __forceinline__ void recover(const float (&u)[4], float (&w)[4]) {
  const float rn = frcp(u[0]);
  float s2 = 0.0f;
#pragma unroll
  for (int q = 0; q < 2; ++q) s2 = fmaf(u[1 + q], u[1 + q], s2);
  const float ke = 0.5f * s2 * rn;
  float e = u[3] - ke;
  if (__builtin_expect(!(ke <= 0.5f * u[3]), 0)) {
    const float eD = energy_density_times_n_fp64(u[0], u[1], u[2], 0.0f, u[3]);
    e = eD * rn;
  }
  w[0] = u[0];
#pragma unroll
  for (int q = 0; q < 2; ++q) w[1 + q] = u[1 + q] * rn;
  w[3] = e;
}

// Conserved state U(W) and physical flux F^Q(U) of one side of a face.
template <int Q>
__device__ __forceinline__ void side_state(const float (&w)[4], float p, float (&u)[4], float (&f)[4]) {
  const float n = w[0], vq = w[1 + Q];
  float v2 = 0.0f;
#pragma unroll
  for (int q = 0; q < 2; ++q) v2 += w[1 + q] * w[1 + q];
  u[0] = n;
#pragma unroll
  for (int q = 0; q < 2; ++q) u[1 + q] = n * w[1 + q];
  u[3] = w[3] + 0.5f * n * v2;
#pragma unroll
  for (int v = 0; v < 3; ++v) f[v] = u[v] * vq;
  f[1 + Q] += p;
  f[3] = (u[3] + p) * vq;
}

// Face flux along axis Q: Eq. FluxHLL, or the middle state of the side that
// alpha_m selects, F* = F_K + S_K (U* - U_K) (see hydro_device.cuh).
template <int Q, int SOLVER>
__device__ __forceinline__ void face_flux(const float (&wl)[4], const float (&wr)[4], float gamma, float gm1,
                                          float (&F)[4]) {
  const float nl = wl[0], nr = wr[0];
  const float pl = gm1 * wl[3], pr = gm1 * wr[3];
  const float vl = wl[1 + Q], vr = wr[1 + Q];
  const float cl = sound_speed(gamma, pl, nl);
  const float cr = sound_speed(gamma, pr, nr);
  const float ap = max0(vl + cl, vr + cr);
  const float am = max0(cl - vl, cr - vr);
  if constexpr (SOLVER == SOLVER_HLL) {
    float ul[4], ur[4], fl[4], fr[4];
    side_state<Q>(wl, pl, ul, fl);
    side_state<Q>(wr, pr, ur, fr);
    const float inv = frcp(ap + am);
    const float apam = ap * am;
#pragma unroll
    for (int v = 0; v < 4; ++v) F[v] = (ap * fl[v] + am * fr[v] - apam * (ur[v] - ul[v])) * inv;
  } else {
    const float sl = am + vl;
    const float sr = ap - vr;
    const float ml = nl * vl, mr = nr * vr;
    const float alpha_m = fdiv(mr * sr + ml * sl - (pr - pl), nr * sr + nl * sl);
    const bool left = is_zero(am) || (!is_zero(ap) && nonneg(alpha_m));
    const float SK = left ? -am : ap;
    const float pK = left ? pl : pr;
    float wK[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) wK[v] = left ? wl[v] : wr[v];
    const float nK = wK[0], vK = wK[1 + Q];
    float uK[4], fK[4];
    side_state<Q>(wK, pK, uK, fK);
    const float dK = SK - vK;
    const float rden = is_zero(SK) ? 0.0f : frcp(SK - alpha_m);
    const float Ds = nK * dK * rden;
    const float ps = pK + nK * dK * (alpha_m - vK);
    float us[4];
    us[0] = Ds;
#pragma unroll
    for (int q = 0; q < 2; ++q) us[1 + q] = Ds * (q == Q ? alpha_m : wK[1 + q]);
    us[3] = (dK * uK[3] - pK * vK + ps * alpha_m) * rden;
#pragma unroll
    for (int v = 0; v < 4; ++v) F[v] = fK[v] + SK * (us[v] - uK[v]);
  }
}

}  // namespace lf
}  // namespace gh
