// hydro_device.cuh -- device-side arithmetic of the finite-volume hydro update
// (GenASiS, Cardall et al., arXiv:1207.3392, Secs. 3.1-3.5) for sm_103a.
//
// Variables: conserved U = (D, S_1..S_ndim, G), primitive W = (n, v_1..v_ndim, e),
// auxiliary p = (gamma-1) e, m = 1 (Sec. 3.5).  NV = ndim + 2 per cell.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "dword.cuh"

namespace gh {

enum : int { BC_PERIODIC = 0, BC_REFLECT = 1, BC_OUTFLOW = 2 };
// SOLVER_HLLC_SW: HLLC, with HLL on faces transverse to a shock (Sec. 3.2)
enum : int { SOLVER_HLL = 0, SOLVER_HLLC = 1, SOLVER_HLLC_SW = 2 };
enum : unsigned { STATUS_NONPHYS = 1u, STATUS_TIMEOUT = 2u };

// Programmatic dependent launch: a kernel of a step's chain is launched while
// its predecessor's last CTAs still run.  chain_wait() returns when the
// predecessor has finished and its writes are visible, and lets the successor's
// CTAs be placed; a kernel of the chain calls it before any access to memory
// that a kernel writes.  Without the launch attribute it is a no-op.
// Such memory is then read with plain loads: __ldg, and const __restrict__
// parameters, promise that nobody writes it while the kernel runs, which in a
// chain begins before the wait, and would let the compiler load ahead of it.
__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Per-cell reconstruction geometry along one axis (Eq. MinMod with
// non-uniform centre distances): theta / (q_c - q_-), 1 / (q_+ - q_-),
// theta / (q_+ - q_c), and the half width (face offset from the geometric
// centre).  The limiter parameter theta is folded into the one-sided terms.
template <class T>
struct __align__(sizeof(T) * 4) Geo {
  T ticm, ipm, tipc, h;
};

// Ghost-cell source along one axis: periodic wrap, reflecting mirror (normal
// momentum negated), or outflow copy of the edge cell.  Indices beyond the two
// ghost layers are clamped onto the outermost ghost so every load stays in
// bounds (such cells only ever feed discarded results).
__device__ __forceinline__ int bc_map(int c, int n, int bc_lo, int bc_hi, bool& flip) {
  flip = false;
  if (c >= 0 && c < n) return c;
  if (c < 0) {
    c = c < -2 ? -2 : c;
    if (bc_lo == BC_PERIODIC) return c + n;
    if (bc_lo == BC_REFLECT) { flip = true; return -1 - c; }
    return 0;
  }
  c = c > n + 1 ? n + 1 : c;
  if (bc_hi == BC_PERIODIC) return c - n;
  if (bc_hi == BC_REFLECT) { flip = true; return 2 * n - 1 - c; }
  return n - 1;
}

// Three-argument minmod: zero unless all arguments share a strict sign, else
// the one of smallest magnitude (Eq. MinMod).
template <class T>
__device__ __forceinline__ T minmod3(T a, T b, T c) {
  T lo = fmin(a, fmin(b, c));
  T hi = fmax(a, fmax(b, c));
  return lo > T(0) ? lo : (hi < T(0) ? hi : T(0));
}

// FP32: the extremes from the three-input min/max of sm_100+, and the case
// split as max(lo, 0) + min(hi, 0) (one of the two terms is zero): the same
// value as the template above in five instructions instead of eight.
__device__ __forceinline__ float minmod3(float a, float b, float c) {
  float lo, hi;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(lo) : "f"(a), "f"(b), "f"(c));
  asm("max.f32 %0, %1, %2, %3;" : "=f"(hi) : "f"(a), "f"(b), "f"(c));
  return fmaxf(lo, 0.0f) + fminf(hi, 0.0f);
}

// FP64: the extremes and sign tests on the integer pipe.  GB300's FP64 pipe
// is the bound of the FP64 path (~2 operations per clock per SM), its integer
// ALU far from it.  A double's bits, with the magnitude bits flipped when the
// sign is set, order as signed integers like the doubles (NaN aside); -0.0
// maps to -1 and +0.0 to 0.  The values returned are the operands themselves.
__device__ __forceinline__ long long okey(double x) {
  const long long i = __double_as_longlong(x);
  return i ^ ((i >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double minmod3(double a, double b, double c) {
  const long long ka = okey(a), kb = okey(b), kc = okey(c);
  long long klo = ka, khi = ka;
  double lo = a, hi = a;
  if (kb < klo) { klo = kb; lo = b; }
  if (kb > khi) { khi = kb; hi = b; }
  if (kc < klo) { klo = kc; lo = c; }
  if (kc > khi) { khi = kc; hi = c; }
  return klo > 0 ? lo : (khi < -1 ? hi : 0.0);  // strictly positive / strictly negative
}

// Double word: one comparison orders b and c, and a normalised pair has the
// sign of its high part.
__device__ __forceinline__ dw minmod3(dw a, dw b, dw c) {
  const bool l = b < c;
  dw lo = l ? b : c, hi = l ? c : b;
  if (a < lo) lo = a;
  if (hi < a) hi = a;
  return lo.hi > 0.0f ? lo : (hi.hi < 0.0f ? hi : dw(0.0f, 0.0f));
}

// max(0, a, b) for the wave speeds: plain for float and double word, on the
// integer pipe for double.
template <class T>
__device__ __forceinline__ T max0(T a, T b) { return fmax(T(0), fmax(a, b)); }
__device__ __forceinline__ double max0(double a, double b) {
  const long long ka = okey(a), kb = okey(b);
  const double m = ka < kb ? b : a;
  return (ka < kb ? kb : ka) > 0 ? m : 0.0;
}

// The same with 2^-120 (FP64 2^-500) in place of 0, far below any speed, and
// |x| <= that: HLLC's upwind test.  With it S_K - v_K is not zero where v_K and S_K are.
__device__ __forceinline__ float max_floor(float a, float b) { return fmaxf(0x1p-120f, fmaxf(a, b)); }
__device__ __forceinline__ dw max_floor(dw a, dw b) { return fmax(dw(0x1p-120f, 0.0f), fmax(a, b)); }
__device__ __forceinline__ double max_floor(double a, double b) {
  const long long ka = okey(a), kb = okey(b);
  const double m = ka < kb ? b : a;
  return (ka < kb ? kb : ka) > 0x20b0000000000000ll ? m : 0x1p-500;
}
__device__ __forceinline__ bool at_floor(float x) { return fabsf(x) <= 0x1p-120f; }
__device__ __forceinline__ bool at_floor(dw x) { return fabsf(x.hi) <= 0x1p-120f; }
__device__ __forceinline__ bool at_floor(double x) {  // to within the high word
  return (unsigned)((unsigned long long)__double_as_longlong(x) >> 32 & 0x7fffffffu) <= 0x20b00000u;
}

// max(a, b) of a CFL speed a >= 0 that ignores a NaN b, x > 0, |x| < infinity,
// x == 0 and x >= 0; FP64: on the integer pipe.
template <class T>
__device__ __forceinline__ T max_speed(T a, T b) { return fmax(a, b); }
__device__ __forceinline__ double max_speed(double a, double b) {
  const long long ka = __double_as_longlong(a), kb = __double_as_longlong(b);
  return kb > ka && kb <= 0x7ff0000000000000ll ? b : a;
}
template <class T>
__device__ __forceinline__ bool positive(T x) { return x > T(0); }
__device__ __forceinline__ bool positive(double x) {  // false for NaN, whose bits lie above infinity's
  const long long b = __double_as_longlong(x);
  return b > 0 && b <= 0x7ff0000000000000ll;
}
template <class T>
__device__ __forceinline__ bool finite(T x) { return fabs(x) < T(INFINITY); }
__device__ __forceinline__ bool finite(double x) {
  return (__double_as_longlong(x) & 0x7fffffffffffffffll) < 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool is_zero(float x) { return x == 0.0f; }
__device__ __forceinline__ bool nonneg(float x) { return x >= 0.0f; }
__device__ __forceinline__ bool nonneg(dw x) { return x.hi >= 0.0f; }
__device__ __forceinline__ bool nonneg(double x) { return okey(x) >= -1; }

// Correctly rounded operations that the compiler may neither fuse nor split.
// Every kernel family (tiles, batch, one-launch, learned, multilevel) inlines
// the functions below, and writing the roundings out keeps the same cell and
// face bitwise the same in all of them, whatever surrounds the call.
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub_rn(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ dw add_rn(dw a, dw b) { return a + b; }
__device__ __forceinline__ dw sub_rn(dw a, dw b) { return a - b; }
__device__ __forceinline__ dw mul_rn(dw a, dw b) { return a * b; }
__device__ __forceinline__ dw fma_rn(dw a, dw b, dw c) { return fma(a, b, c); }
// a / 2 (exact) and c - a / 2
__device__ __forceinline__ float half_of(float a) { return __fmul_rn(0.5f, a); }
__device__ __forceinline__ double half_of(double a) {  // normal numbers: one off the exponent, on the integer pipe
  const long long b = __double_as_longlong(a);
  const unsigned ex = (unsigned)((unsigned long long)b >> 52) & 0x7ffu;
  return ex - 2u < 0x7fdu ? __longlong_as_double(b - (1ll << 52)) : __dmul_rn(0.5, a);
}
__device__ __forceinline__ dw half_of(dw a) { return dw(__fmul_rn(0.5f, a.hi), __fmul_rn(0.5f, a.lo)); }
__device__ __forceinline__ float sub_half(float c, float a) { return __fmaf_rn(-0.5f, a, c); }
__device__ __forceinline__ double sub_half(double c, double a) { return __fma_rn(-0.5, a, c); }
__device__ __forceinline__ dw sub_half(dw c, dw a) { return c - half_of(a); }

// Values a distance h s below and above wc (the two faces of a cell), alone and
// as a pair; double word forms h s once for both.
template <class T>
__device__ __forceinline__ T face_lo(T s, T h, T wc) { return fma_rn(-s, h, wc); }
template <class T>
__device__ __forceinline__ T face_hi(T s, T h, T wc) { return fma_rn(s, h, wc); }
__device__ __forceinline__ dw face_lo(dw s, dw h, dw wc) { return wc - s * h; }
__device__ __forceinline__ dw face_hi(dw s, dw h, dw wc) { return wc + s * h; }
template <class T>
__device__ __forceinline__ void face_pair(T s, T h, T wc, T& lo, T& hi) {
  lo = face_lo(s, h, wc);
  hi = face_hi(s, h, wc);
}
__device__ __forceinline__ void face_pair(dw s, dw h, dw wc, dw& lo, dw& hi) {
  const dw d = s * h;
  lo = wc - d;
  hi = wc + d;
}

// Limited slope of cell c from its neighbours (Eq. MinMod; theta is in g).
template <class T>
__device__ __forceinline__ T limited_slope(T wm, T wc, T wp, const Geo<T>& g) {
  return minmod3(mul_rn(sub_rn(wc, wm), g.ticm), mul_rn(sub_rn(wp, wm), g.ipm), mul_rn(sub_rn(wp, wc), g.tipc));
}

// Division, reciprocal and square root used by the flux arithmetic.  FP64
// takes Newton-type reciprocals from an FP32 seed (a few ulp, far inside its
// 1e-10 parity bar); FP32 uses the hardware approximations (a few ulp, far
// inside its 1e-5 bar).
//
// FP64 seeds: conversions between the formats of values in the normal FP32
// range, on the integer pipe (rebias the exponent, move the mantissa; the
// truncation to FP32 costs a relative 2^-23 at most, which the correction
// steps below remove), because GB300 runs an FP64 conversion at the rate of
// its slow FP64 pipe.
__device__ __forceinline__ float seed_float(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
  const unsigned mag = __funnelshift_l(lo, (hi & 0x7fffffffu) - (896u << 20), 3);
  return __uint_as_float((hi & 0x80000000u) | mag);
}
__device__ __forceinline__ double seed_double(float f) {
  const unsigned u = __float_as_uint(f);
  const unsigned hi = (u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20));
  return __longlong_as_double((long long)(((unsigned long long)hi << 32) | (unsigned long long)(u << 29)));
}
// Biased exponent in [900, 1146] (|x| ~ 1e-37 .. 1e37): the range in which the
// seeds and their reciprocals are normal FP32 numbers.
__device__ __forceinline__ bool seed_range(double x) {
  const unsigned ex = (unsigned)((unsigned long long)__double_as_longlong(x) >> 52) & 0x7ffu;
  return ex - 900u <= 246u;
}
// The same of a positive x: a negative x (a limited density below zero) has no root.
__device__ __forceinline__ bool root_range(double x) {
  return (unsigned)((unsigned long long)__double_as_longlong(x) >> 52) - 900u <= 246u;
}
// Hardware FP32 reciprocal and reciprocal square root (relative error about
// 2^-23); arguments above 2^126 give 0.
__device__ __forceinline__ float frcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float frsqrt(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// FP64 reciprocal: seed r with relative error ~2^-22, then 1/x = r (1 + e +
// e^2 + ...) with the exact residual e = 1 - x r: the cubic step r + r (e +
// e^2) leaves e^3 ~ 2^-66, below the FP64 rounding level, in three FP64 FMAs
// in place of an IEEE division on GB300's slow FP64 pipe.  Arguments outside
// the normal FP32 range (and 0, infinities, NaN) take the IEEE division.
__device__ __forceinline__ double frcp(double x) {
  if (!seed_range(x)) return 1.0 / x;
  const double r = seed_double(frcp(seed_float(x)));
  const double e = fma_rn(-x, r, 1.0);
  return fma_rn(r, fma_rn(e, e, e), r);
}
// a / b from the reciprocal and one residual correction q + r (a - b q).
__device__ __forceinline__ double fdiv(double a, double b) {
  const double r = frcp(b);
  const double q = mul_rn(a, r);
  return fma_rn(r, fma_rn(-b, q, a), q);
}
__device__ __forceinline__ float fdiv(float a, float b) { return mul_rn(a, frcp(b)); }
// double-word: the operations of dword.cuh
__device__ __forceinline__ dw fdiv(dw a, dw b) { return a / b; }
__device__ __forceinline__ dw frcp(dw x) { return dw(1.0f, 0.0f) / x; }

// Sound speed c = sqrt(gamma p / n) (Sec. 3.5) as gp rsqrt(gp n), gp = gamma p.
// FP64: seed r = rsqrt(x) with relative error ~2^-22, residual e = 1 - x r^2,
// then x^(-1/2) = r (1 - e)^(-1/2) = r (1 + e/2 + 3 e^2/8 + ...), which leaves
// 5 e^3/16 ~ 2^-65: seven FP64 operations; CUDA's rsqrt outside the seed range
// (NaN for gp n < 0, which the wave speeds leave out), and 0 where gamma p is not positive.  FP32: the hardware approximation.
// Double word: the same form with one correction (34 -> 26 operations), the
// quotient and square root of dword.cuh where gp n nears the ends of FP32 or both
// factors are limited below zero.
__device__ __forceinline__ dw sound_speed(dw gamma, dw p, dw n) {
  const dw gp = gamma * p;
  const float x = mul_rn(gp.hi, n.hi);
  if (!(x > 1e-30f && x < 1e30f && gp.hi > 0.0f)) return sqrt(gamma * (p / n));
  // c0 = gp rsqrt(gp n) and one Newton correction (gp - n c0^2) / (2 n c0) from
  // the exact residual, 1 / (n c0) = rsqrt(gp n)
  const float r = frsqrt(x), c0 = mul_rn(gp.hi, r);
  float q, qe, ph, pl, zh, zl;
  two_prod(c0, c0, q, qe);
  two_prod(n.hi, q, ph, pl);
  pl = fma_rn(n.hi, qe, fma_rn(n.lo, q, pl));
  const float res = add_rn(sub_rn(sub_rn(gp.hi, ph), pl), gp.lo);  // gp.hi - ph exact
  fast_two_sum(c0, mul_rn(res, mul_rn(0.5f, r)), zh, zl);
  return dw(zh, zl);
}
__device__ __forceinline__ float sound_speed(float gamma, float p, float n) {
  const float gp = mul_rn(gamma, p);
  return mul_rn(gp, frsqrt(mul_rn(gp, n)));
}
__device__ __forceinline__ double sound_speed(double gamma, double p, double n) {
  const double gp = mul_rn(gamma, p), x = mul_rn(gp, n);
  if (!(okey(gp) > 0)) return 0.0;
  if (!root_range(x)) return mul_rn(gp, rsqrt(x));
  const double r = seed_double(frsqrt(seed_float(x)));
  const double e = fma_rn(-mul_rn(x, r), r, 1.0);
  const double c = mul_rn(gp, r);
  return fma_rn(mul_rn(c, e), fma_rn(0.375, e, 0.5), c);
}

// ---------------------------------------------------------------------------
// Conserved -> primitive recovery: v = S / D, e = G - S.v / 2.
//
// FP64 and double word: as written.
// Mixed path (FP32 storage): the difference cancels when the kinetic energy is
// a large part of G.  Where it is at most half of G the FP32 difference loses
// at most one bit and is used as is.  Elsewhere v is extended by its residual,
// v = v_r + v_l with v_l = (S - v_r D) / D, every product S v_r is split into
// its rounded value and rounding error, and the sums carry their rounding
// errors (Knuth's TwoSum), so that S.v / 2 is known to about 2^-46; the leading
// difference G - s/2 is exact there (the two lie within a factor 2), and its
// correction is added last.  The result is as exact as the FP32 state allows
// (a rounding of G alone moves e by 2^-25 G), without the FP64 pipe, which an
// earlier FP64 branch here kept 44% busy in the FP32 batch kernel (Riemann
// problems carry much kinetic energy): 256 problems, 20 steps with their
// copies in and out, 20.97 -> 17.85 ms.
// ---------------------------------------------------------------------------
template <int NDIM, class T>
__device__ __forceinline__ void recover(const T (&u)[NDIM + 2], T (&w)[NDIM + 2]) {
  constexpr int NV = NDIM + 2;
  const T rn = frcp(u[0]);
  w[0] = u[0];
#pragma unroll
  for (int q = 0; q < NDIM; ++q) w[1 + q] = mul_rn(u[1 + q], rn);
  T sv = mul_rn(u[1], w[1]);
#pragma unroll
  for (int q = 1; q < NDIM; ++q) sv = fma_rn(u[1 + q], w[1 + q], sv);
  w[NV - 1] = sub_half(u[NV - 1], sv);
}

// e of a cell whose kinetic energy exceeds half of G: the compensated form
// (v_r: the rounded velocities, rn: the reciprocal of D).
template <int NDIM>
__device__ __forceinline__ float energy_compensated(const float (&u)[NDIM + 2], const float (&vr)[NDIM], float rn) {
  float s = 0.0f, t = 0.0f;  // S.v = s + t
#pragma unroll
  for (int q = 0; q < NDIM; ++q) {
    const float S = u[1 + q];
    const float vl = mul_rn(fma_rn(-vr[q], u[0], S), rn);
    const float p = mul_rn(S, vr[q]);
    const float pe = fma_rn(S, vl, fma_rn(S, vr[q], -p));
    if (q == 0) {
      s = p;
      t = pe;
    } else {
      float z, ze;
      two_sum(s, p, z, ze);
      s = z;
      t = add_rn(t, add_rn(ze, pe));
    }
  }
  return sub_half(sub_half(u[NDIM + 1], s), t);
}

template <int NDIM>
__device__ __forceinline__ void recover(const float (&u)[NDIM + 2], float (&w)[NDIM + 2]) {
  constexpr int NV = NDIM + 2;
  const float rn = frcp(u[0]);
  float vr[NDIM];
#pragma unroll
  for (int q = 0; q < NDIM; ++q) vr[q] = mul_rn(u[1 + q], rn);
  float sv = mul_rn(u[1], vr[0]);
#pragma unroll
  for (int q = 1; q < NDIM; ++q) sv = fma_rn(u[1 + q], vr[q], sv);
  float e = sub_half(u[NV - 1], sv);
  if (__builtin_expect(!(e >= half_of(u[NV - 1])), 0)) e = energy_compensated<NDIM>(u, vr, rn);
  w[0] = u[0];
#pragma unroll
  for (int q = 0; q < NDIM; ++q) w[1 + q] = vr[q];
  w[NV - 1] = e;
}

// ---------------------------------------------------------------------------
// Face flux along axis Q from reconstructed primitive states on the left (wl)
// and right (wr) of the face (Eqs. conservedLeft..conservedRight).
//   wave speeds  alpha_+ = max(0, v_L + c_L, v_R + c_R),
//                alpha_- = max(0, c_L - v_L, c_R - v_R)         (Sec. 3.2, 3.5)
//   HLL          Eq. FluxHLL
//   HLLC         Eq. MiddleWaveSpeed for alpha_m, then one middle state on the
//                side selected by the sign of alpha_m (Eq. FluxHLLC), written
//                with the signed outer wave speed S_K (S_L = -alpha_-,
//                S_R = alpha_+), d_K = S_K - v_K and a_K = D_K d_K:
//                  D* = a_K / (S_K - alpha_m)
//                  p* = p_K + a_K (alpha_m - v_K)
//                  G* = (d_K G_K - p_K v_K + p* alpha_m) / (S_K - alpha_m)
//                     = (d_K G_K + (alpha_m - v_K)(p_K + a_K alpha_m))
//                       / (S_K - alpha_m)
//                which are the outer jump conditions of Sec. 3.2 solved for the
//                middle state (this form satisfies p*_L = p*_R).  The middle
//                state moves with alpha_m, so its flux is
//                  F* = alpha_m U* + p* (0, e_Q, alpha_m):
//                D* alpha_m, that times (alpha_m, transverse v_K) plus p* in
//                the normal momentum, and (G* + p*) alpha_m; neither F_K nor U_K
//                beyond G_K is formed, about 20 operations a face fewer than
//                F_K + S_K (U* - U_K).  Measured with the shorter reciprocal
//                and sound speed above, ms per RK2 step, HLLC: FP64 128^3
//                4.90 -> 4.22 (bound by the FP64 pipe), double word 128^3
//                1.36 -> 1.14, FP32 256^3 1.436 -> 1.383 (bound by issue).
//                alpha_- = 0 gives F_L, alpha_+ = 0 gives F_R (upwind): there
//                S_K = 0, and alpha_m is replaced by v_K, for which U* = U_K
//                and the formulas above are F_K.  (The code's S_K is then not 0
//                but 2^-120, 2^-500 in FP64: that changes no bit of F_K, and the
//                side may also be at rest, where 1 / (S_K - v_K) of S_K = 0 would
//                make the vanishing terms NaN: a limited pressure at or
//                below 0 on a stretched mesh.)
// ---------------------------------------------------------------------------
// Conserved state U(W) and physical flux F^Q(U) of one side of a face
// (Sec. 3.5): p is its pressure, w[1 + Q] its normal velocity.
template <class T, int NDIM, int Q>
__device__ __forceinline__ void side_state(const T (&w)[NDIM + 2], T p, T (&u)[NDIM + 2], T (&f)[NDIM + 2]) {
  constexpr int NV = NDIM + 2;
  const T n = w[0], vq = w[1 + Q];
  T v2 = mul_rn(w[1], w[1]);
#pragma unroll
  for (int q = 1; q < NDIM; ++q) v2 = fma_rn(w[1 + q], w[1 + q], v2);
  u[0] = n;
#pragma unroll
  for (int q = 0; q < NDIM; ++q) u[1 + q] = mul_rn(n, w[1 + q]);
  u[NV - 1] = fma_rn(half_of(n), v2, w[NV - 1]);
#pragma unroll
  for (int v = 0; v < NV - 1; ++v) f[v] = v == 1 + Q ? fma_rn(u[v], vq, p) : mul_rn(u[v], vq);
  f[NV - 1] = mul_rn(add_rn(u[NV - 1], p), vq);
}

template <class T, int NDIM, int Q, int SOLVER>
__device__ __forceinline__ void face_flux(const T (&wl)[NDIM + 2], const T (&wr)[NDIM + 2],
                                          T gamma, T gm1, T (&F)[NDIM + 2]) {
  constexpr int NV = NDIM + 2;
  const T nl = wl[0], nr = wr[0];
  const T pl = mul_rn(gm1, wl[NV - 1]), pr = mul_rn(gm1, wr[NV - 1]);
  const T vl = wl[1 + Q], vr = wr[1 + Q];
  const T cl = sound_speed(gamma, pl, nl);
  const T cr = sound_speed(gamma, pr, nr);

  if constexpr (SOLVER == SOLVER_HLL) {
    const T ap = max0(add_rn(vl, cl), add_rn(vr, cr));
    const T am = max0(sub_rn(cl, vl), sub_rn(cr, vr));
    T ul[NV], ur[NV], fl[NV], fr[NV];
    side_state<T, NDIM, Q>(wl, pl, ul, fl);
    side_state<T, NDIM, Q>(wr, pr, ur, fr);
    const T inv = frcp(add_rn(ap, am));
    const T apam = mul_rn(ap, am);
#pragma unroll
    for (int v = 0; v < NV; ++v)
      F[v] = mul_rn(fma_rn(-apam, sub_rn(ur[v], ul[v]), fma_rn(am, fr[v], mul_rn(ap, fl[v]))), inv);
  } else {
    const T ap = max_floor(add_rn(vl, cl), add_rn(vr, cr));
    const T am = max_floor(sub_rn(cl, vl), sub_rn(cr, vr));
    const T sl = add_rn(am, vl);  // = -(S_L - v_L) > 0
    const T sr = sub_rn(ap, vr);  // =   S_R - v_R  > 0
    const T al = mul_rn(nl, sl), ar = mul_rn(nr, sr);
    const T alpha = fdiv(fma_rn(ar, vr, fma_rn(al, vl, sub_rn(pl, pr))), add_rn(ar, al));
    const bool left = at_floor(am) || (!at_floor(ap) && nonneg(alpha));
    const T SK = left ? -am : ap;
    const T dK = left ? -sl : sr;
    const T aK = left ? -al : ar;
    const T pK = left ? pl : pr;
    T wK[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) wK[v] = left ? wl[v] : wr[v];
    const T vK = wK[1 + Q];
    const T a = at_floor(SK) ? vK : alpha;
    const T dv = sub_rn(a, vK);
    T v2 = mul_rn(wK[1], wK[1]);
#pragma unroll
    for (int q = 1; q < NDIM; ++q) v2 = fma_rn(wK[1 + q], wK[1 + q], v2);
    const T GK = fma_rn(half_of(wK[0]), v2, wK[NV - 1]);
    const T r = frcp(sub_rn(SK, a));
    const T ps = fma_rn(aK, dv, pK);
    const T Gs = mul_rn(fma_rn(dK, GK, mul_rn(dv, fma_rn(aK, a, pK))), r);
    const T m = mul_rn(mul_rn(aK, r), a);  // D* alpha_m
    F[0] = m;
#pragma unroll
    for (int q = 0; q < NDIM; ++q) F[1 + q] = q == Q ? fma_rn(m, a, ps) : mul_rn(m, wK[1 + q]);
    F[NV - 1] = mul_rn(add_rn(Gs, ps), a);
  }
}

// Column sums of the conserved totals.  FP64 state: plain FP64 FMA.  FP32
// state: a compensated pair of floats (Knuth's TwoSum plus the exact rounding
// error of each product from an FMA), about 48 significant bits, so no FP64
// instruction runs per cell; the pair is folded into FP64 once per column.
template <class T>
struct ColumnSum;

template <>
struct ColumnSum<double> {
  double s = 0.0;
  __device__ __forceinline__ void add_product(double u, double dz_hi, double) { s = fma(u, dz_hi, s); }
  __device__ __forceinline__ double value() const { return s; }
};

template <>
struct ColumnSum<float> {
  float hi = 0.0f, lo = 0.0f;
  // add u * (dz_hi + dz_lo)
  __device__ __forceinline__ void add_product(float u, float dz_hi, float dz_lo) {
    const float p = mul_rn(u, dz_hi);
    const float pe = fma_rn(u, dz_lo, fma_rn(u, dz_hi, -p));
    float t, err;
    two_sum(hi, p, t, err);
    hi = t;
    lo = add_rn(lo, add_rn(err, pe));
  }
  __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

// Double-word state: the column sum in double-word arithmetic (dz as a pair).
template <>
struct ColumnSum<dw> {
  dw s = dw(0.0f, 0.0f);
  __device__ __forceinline__ void add_product(dw u, dw dz, dw) { s = fma(u, dz, s); }
  __device__ __forceinline__ double value() const { return (double)s; }
};

// Deterministic block reductions (fixed shuffle tree, then warps in order).
template <class T>
__device__ __forceinline__ T warp_sum(T x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
template <class T>
__device__ __forceinline__ T warp_max(T x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = fmax(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}

}  // namespace gh
