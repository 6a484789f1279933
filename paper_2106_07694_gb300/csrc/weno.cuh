// WENO reconstruction arithmetic of the transport kernels (Supplement Eqs. S9-S16, the order
// raised to five): face values from split fluxes kept divided by the Lax-Friedrichs alpha, so
// epsilon = 1e-6 here is epsilon = 1e-6 alpha^2 on the unscaled flux.
//
// WENO5-JS is written on the first differences d1..d4 of the five upwind-side values
// a, b, c, d, e and their second differences s_k = d_{k+2} - d_{k+1}.  With the smoothness
// indicators multiplied by 3/4 (only ratios of (eps + beta_k)^2 enter, so eps is too):
//   beta_0 = s0^2 + 3/4 d2 (d2 + s0),  beta_1 = s1^2 + 3/4 d2 d3,  beta_2 = s2^2 + 3/4 d3 (d3 - s2);
// candidates relative to the centre value, over one half:
//   2 (q_0 - c) = d2 + 2/3 s0,  2 (q_1 - c) = d2 + 2/3 s1,  2 (q_2 - c) = d3 - 1/3 s2;
// with A_k = (eps + beta_k)^2 the weights are A1 A2 : 6 A0 A2 : 3 A0 A1 (linear weights times
// ten), one numerator and one denominator: face value = c + num / (2 den).
// 25 FP32 operations against 28 for the squares of s and t = 3 d2 - d1, d2 + d3, d4 - 3 d3 and
// the candidates over six.  Its FP32 error against FP64 is that of the longer form (rms 8.3e-9
// on a noisy front of height 1/2, 6.6e-9 on smooth data, both forms).
//
// The reciprocal is the hardware's approximate one (1 ulp) without the range handling that
// __fdividef carries: den is at least 10 (3/4 1e-6)^4 = 3e-24, and past 2^126 both give 0.
// Rounding is sign-symmetric, so a mirrored (h-) reconstruction may pass the negated
// differences of the stored order and gets the bits of the reversed values.
#pragma once
#include "common.cuh"

namespace lw {

__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// 1 / x in FP64 for the weights' denominators, positive and from 10 (3/4 1e-6)^4 = 3e-24 up: the
// hardware's approximation, of relative error e0, and one step r (1 + e + e^2) with e = 1 - x r,
// the third-order hyperpower iteration for an inverse (Altman 1960).  x r (1 + e + e^2) =
// (1 - e)(1 + e + e^2) = 1 - e^3, so e0^3 is left beside the last rounding: with e0 of 2^-20 under
// 0.51 units in the last place (tested: within one unit of IEEE division from 3e-24 to 1e60, the
// quotient within two).  Four operations with the product, where an IEEE division takes about ten
// of the narrow FP64 pipe: a step on 128 x 256 takes 68.6 us, 74.9 with divisions.  c and u are no
// further from a long-double run with it (300 x 133 after 1500 steps: c 3.98e-14 both, 128 x 256
// after 8000: 2.76e-14 both; with division and the 12/13 form of the indicators 3.98e-14, 2.79e-14).
__device__ __forceinline__ double rcp_newton(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

template <typename T>
struct Recon {
  T num, den;  // face value = centre value + num / (2 den)
};

template <typename T>
__device__ __forceinline__ Recon<T> weno5_recon(T d1, T d2, T d3, T d4, T s0, T s1, T s2) {
  const T eps = T(0.75e-6), g2 = T(0.75) * d2, g3 = T(0.75) * d3;
  T A0 = fma_t(g2, d2 + s0, fma_t(s0, s0, eps));
  T A1 = fma_t(g2, d3, fma_t(s1, s1, eps));
  T A2 = fma_t(g3, d3 - s2, fma_t(s2, s2, eps));
  A0 *= A0;
  A1 *= A1;
  A2 *= A2;
  const T r0 = fma_t(T(2.0 / 3.0), s0, d2), r1 = fma_t(T(2.0 / 3.0), s1, d2), r2 = fma_t(T(-1.0 / 3.0), s2, d3);
  const T A02x6 = T(6) * (A0 * A2);
  return {fma_t(A1, fma_t(T(3) * A0, r2, A2 * r0), A02x6 * r1), fma_t(A1, fma_t(T(3), A0, A2), A02x6)};
}

template <typename T>
__device__ __forceinline__ Recon<T> weno5_recon(T a, T b, T c, T d, T e) {
  const T d1 = b - a, d2 = c - b, d3 = d - c, d4 = e - d;
  return weno5_recon<T>(d1, d2, d3, d4, d2 - d1, d3 - d2, d4 - d3);
}

// The paper's third-order WENO (Supplement Eqs. S10, S11, S14-S16) on the upwind-side values
// a, b, c = h_{i-1}, h_i, h_{i+1}: candidates (b + c)/2 and (3b - a)/2, indicators (c - b)^2
// and (b - a)^2, linear weights 2/3 and 1/3, on the differences d1 = b - a, d2 = c - b and
// A_k = (eps + d_k^2)^2 of them: the weights are 2 A1 : A2.
template <typename T>
__device__ __forceinline__ Recon<T> weno3_recon(T d1, T d2, T A1, T A2) {
  return {fma_t(A2, d1, (T(2) * A1) * d2), fma_t(T(2), A1, A2)};
}
template <typename T>
__device__ __forceinline__ T weno3_smooth(T d) {
  const T b = fma_t(d, d, T(1e-6));
  return b * b;
}
template <typename T>
__device__ __forceinline__ Recon<T> weno3_recon(T a, T b, T c) {
  const T d1 = b - a, d2 = c - b;
  return weno3_recon<T>(d1, d2, weno3_smooth(d1), weno3_smooth(d2));
}

// Face value of one reconstruction about the centre value c.
__device__ __forceinline__ float recon_value(Recon<float> r, float c) {
  return fmaf(0.5f, r.num * rcp_approx(r.den), c);
}
__device__ __forceinline__ double recon_value(Recon<double> r, double c) {
  return fma(0.5, r.num * rcp_newton(r.den), c);
}

// Sum of two face values (h+ about the centre value cp, h- about cm), each rounded at its own
// size.  Summing the two corrections first, one operation less, kept more of them than c can
// take up a step: the drift of c against 64 bits on 128 x 256 grew by 3 % (8000 steps: 9.84e-6
// -> 1.017e-5 relative, 9.87e-6 in this form).
__device__ __forceinline__ float recon_sum(Recon<float> p, float cp, Recon<float> m, float cm) {
  return fmaf(0.5f, p.num * rcp_approx(p.den), cp) + fmaf(0.5f, m.num * rcp_approx(m.den), cm);
}
// In FP64, where the pipe is narrow, the corrections are summed first: a face is then 6e-18 from the
// exact one (rms on a noisy front) against 2.7e-17, and over 8000 steps c drifts no more than with
// the values rounded one by one (2.758e-14 against 2.761e-14).
__device__ __forceinline__ double recon_sum(Recon<double> p, double cp, Recon<double> m, double cm) {
  return fma(0.5, fma(p.num, rcp_newton(p.den), m.num * rcp_newton(m.den)), cp + cm);
}

// Face flux divided by alpha: h+ from the left-biased values p0..p4, h- from the right-biased
// values m0..m4 (already mirrored), diffusion kd (cl - cr) with kd = kappa / alpha.  The stage
// kernels difference the faces and multiply by alpha once, in the combination.
template <typename T>
__device__ __forceinline__ T face_flux_x(T p0, T p1, T p2, T p3, T p4, T m0, T m1, T m2, T m3, T m4, T kd, T cl, T cr) {
  return fma_t(kd, cl - cr, recon_sum(weno5_recon(p0, p1, p2, p3, p4), p2, weno5_recon(m0, m1, m2, m3, m4), m2));
}

// Face flux (divided by alpha) of a transport-scheme variant (SCHEME = kSchemeWeno3 |
// kSchemeSignSplit bits; 0 is the Lax-Friedrichs WENO5 of face_flux_x) from the staged pairs
// of the six points i-2 .. i+3 around the face i+1/2 (p[k], m[k] = point i-2+k).
// Lax-Friedrichs schemes stage p = h+/alpha, m = h-/alpha; the sign split stages
// p = w c/alpha, m = w/alpha and reconstructs w c from the side the face velocity
// (w_i + w_{i+1})/2 comes from (ties to the left).  T = float or double.
template <int SCHEME, typename T>
__device__ __forceinline__ T face_flux_scheme(const T (&p)[6], const T (&m)[6], T kd, T cl, T cr) {
  constexpr bool W3 = (SCHEME & kSchemeWeno3) != 0, SIGN = (SCHEME & kSchemeSignSplit) != 0;
  T h;
  if (SIGN) {
    const bool left = m[2] + m[3] >= T(0);
    const T c = left ? p[2] : p[3];
    if (W3)
      h = recon_value(weno3_recon<T>(left ? p[1] : p[4], c, left ? p[3] : p[2]), c);
    else
      h = recon_value(weno5_recon<T>(left ? p[0] : p[5], left ? p[1] : p[4], c, left ? p[3] : p[2], left ? p[4] : p[1]),
                      c);
  } else if (W3) {
    h = recon_sum(weno3_recon<T>(p[1], p[2], p[3]), p[2], weno3_recon<T>(m[4], m[3], m[2]), m[3]);
  } else {
    h = recon_sum(weno5_recon<T>(p[0], p[1], p[2], p[3], p[4]), p[2], weno5_recon<T>(m[5], m[4], m[3], m[2], m[1]), m[3]);
  }
  return fma_t(kd, cl - cr, h);
}

// The Shu-Osher combination of a stage (Eqs. S21-S23) at one node: ch the stage input there,
// Lk = -div of the face fluxes divided by alpha, cn = c^n.  The last stage is s + (c - s)/3, not
// c/3 + 2 s/3: the FP32 roundings of 1/3 and 2/3 sum to 1 + 3e-8, which would add a bias to c
// every step.
template <int STAGE, typename T>
__device__ __forceinline__ T rk_finish(T s, T cn) {
  if (STAGE == 1) return s;
  if (STAGE == 2) return fma_t(T(0.75), cn, T(0.25) * s);
  return fma_t(T(1) / T(3), cn - s, s);
}
template <int STAGE, typename T>
__device__ __forceinline__ T rk_combine(T ch, T Lk, T alpha, T cn) {
  return rk_finish<STAGE>(fma_t(alpha, Lk, ch), cn);
}
// The same on the floor row, less its settling outflow vs ch.  The outflow joins the increment,
// and the sum is rounded once at the size of c: c less the outflow rounded first, and the rest then,
// biased the floor's c and the deposit.  Relative error of the deposit in FP32, 40 lattices of
// 256 x 512 with Vs from 2e-4 to 4e-3: 4.5e-7 rms after 1000 steps so, 3.1e-7 in this form (10 of
// 2304 x 2048: 5.4e-7 and 2.0e-7).
template <int STAGE, typename T>
__device__ __forceinline__ T rk_combine_floor(T ch, T Lk, T alpha, T cn, T vs) {
  return rk_finish<STAGE>(ch + fma_t(-vs, ch, alpha * Lk), cn);
}

}  // namespace lw
