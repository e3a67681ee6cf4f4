// One edge of the wave-propagation method, in the form the row-walking
// update kernels (walk, band) evaluate it: per edge the upwind normal flux
// with its MC-limited second-order correction, and the two fluctuations
// that the transverse terms carry into the neighbouring edges (the flux form
// of the unsplit method of Sec. 5, with the correction waves propagated
// transversely when transverse = 2).
//
// Units: an edge speed s enters as the half Courant number c = s dt / (2 h)
// (capacity form: c = phi dt / 2) and every flux and fluctuation carries the
// same factor dt / (2 h) (dt / 2).  With it no separate dt/h is left in the
// inner loop:
//   correction        1/2 |s| (1 - |s| dt/h) lim   ->  |c| (1/2 - |c|) lim
//   transverse share  1/2 dt/h s X                 ->  c X
//   update            q - dt/h (dF + dG)           ->  q - 2 (dF + dG)
// and 2 lim = min(|W + Wup|, 4 |W|, 4 |Wup|) takes the limiter's factors.
// The FP64 pipe issues 1/64 of an SM's slots, so what bounds the FP64 update
// is its count of FP64 instructions: about 25 a cell in this form, of 66 in
// the speeds' own units with min, max and compares in FP64 -- the minima,
// signs and selections are taken on the bits by integer instructions.
// Measured on one GB300, a coarse step before and after: swirl forest of 496
// 32^2 patches in FP64 1.32 -> 0.87 ms (FP32 0.136 -> 0.123 ms), 64 forests
// of 16^2 patches in FP64 5.7 -> 3.7 ms, 256 forests of 32^2 patches in FP32
// 6.5 -> 6.0 ms.
#pragma once

#include "device_util.cuh"

namespace fc {

// The scheme's options.  FULL (second order, MC limiter, transverse
// propagation of both: what runs by default): constants, so the inner loop
// holds no selection by option (8 instructions a cell in FP32).
template <typename real, bool FULL>
struct Scheme {
  real k0 = real(0.25);  // correction |c| (k0 - k1 |c|) m, m = 2 lim (MC) or W (unlimited):
  real k1 = real(0.5);   //   1/4, 1/2 with MC; 1/2, 1 unlimited; 0, 0 first order
  bool mc_ = true;       // MC limiter
  bool t1_ = true, t2_ = true;  // transverse fluctuations; their corrections too
  __device__ __forceinline__ bool mc() const { return FULL || mc_; }
  __device__ __forceinline__ bool t1() const { return FULL || t1_; }
  __device__ __forceinline__ bool t2() const { return FULL || t2_; }
  __device__ __forceinline__ real c0() const { return FULL ? real(0.25) : k0; }
  __device__ __forceinline__ real c1() const { return FULL ? real(0.5) : k1; }
};

inline bool full_scheme(int order, int limiter, int transverse) {
  return order > 1 && limiter != 0 && transverse > 1;
}

template <typename real, bool FULL>
__device__ __forceinline__ Scheme<real, FULL> make_scheme(int order, int limiter,
                                                          int transverse) {
  Scheme<real, FULL> sc;
  if (!FULL) {
    sc.mc_ = limiter != 0;
    sc.k0 = order > 1 ? (sc.mc_ ? real(0.25) : real(0.5)) : real(0);
    sc.k1 = real(2) * sc.k0;
    sc.t1_ = transverse > 0;
    sc.t2_ = transverse > 1;
  }
  return sc;
}

// A launch's scalars in the field's precision, converted on the host: one
// FP64 conversion or product on every thread of a CTA takes the FP64 pipe
// 16 cycles a warp (and a division some thirty times that).
template <typename real>
struct AdvConst {
  real h;       // cell width
  real cu, cv;  // half Courant numbers of a constant velocity
  real hdt;     // dt / 2 (capacity form)
  real bfac;    // recorded flux / flux in this file's units: 2 h / dt (capacity form: 2 / dt)
  real alpha;   // time-interpolation weight
};
template <typename real>
inline AdvConst<real> adv_const(const DevForest<real>& D, const AdvArgs& a) {
  AdvConst<real> c;
  c.h = real(a.h);
  c.cu = real(D.vel[0] * 0.5 * a.nu);
  c.cv = real(D.vel[1] * 0.5 * a.nu);
  c.hdt = real(0.5 * a.dt);
  c.bfac = real(2.0 / (D.metric ? a.dt : a.nu));
  c.alpha = real(a.alpha);
  return c;
}

// does the edge's flow come from its left / lower cell (a zero speed's sign
// does not matter: every use is multiplied by it)
__device__ __forceinline__ bool upwind_left(float c) { return c >= 0.f; }
__device__ __forceinline__ bool upwind_left(double c) { return __double2hiint(c) >= 0; }

// twice the MC-limited wave: 0 unless W and Wup share a sign, else
// sign(W) min(|W + Wup|, 4 |W|, 4 |Wup|).  (A zero wave gives a zero minimum,
// so the signs' bits decide.)
__device__ __forceinline__ float mc_twice(float W, float Wup) {
  const float m = fminf(fabsf(W + Wup), 4.f * fminf(fabsf(W), fabsf(Wup)));
  return (__float_as_int(W) ^ __float_as_int(Wup)) >= 0 ? copysignf(m, W) : 0.f;
}
// one FP64 instruction (the sum): magnitudes compare as integers, 4 x adds 2
// to the exponent; a minimum below the normal range counts as zero
__device__ __forceinline__ double mc_twice(double W, double Wup) {
  constexpr unsigned long long kMag = 0x7fffffffffffffffull;
  const unsigned long long w = (unsigned long long)__double_as_longlong(W);
  const unsigned long long u = (unsigned long long)__double_as_longlong(Wup);
  const unsigned long long aw = w & kMag, au = u & kMag;
  const unsigned long long mn = aw < au ? aw : au;
  const unsigned long long a = (unsigned long long)__double_as_longlong(W + Wup) & kMag;
  const unsigned long long m4 = mn + (2ull << 52);
  unsigned long long m = a < m4 ? a : m4;
  if ((long long)(w ^ u) < 0 || mn < (1ull << 52)) m = 0;
  return __longlong_as_double((long long)(m | (w & ~kMag)));
}

// the correction's factor of m; w: sum of the two cells' 1/kappa in the
// capacity form, where the correction is 1/2 |c| (1 - |c| w) lim
template <typename real, bool FULL>
__device__ __forceinline__ real corr_factor(real c, const Scheme<real, FULL>& sc) {
  const real a = fabs(c);
  return a * fma(-sc.c1(), a, sc.c0());
}
template <typename real, bool FULL>
__device__ __forceinline__ real corr_factor_cap(real c, real w, const Scheme<real, FULL>& sc) {
  const real a = fabs(c);
  return a * fma(-sc.c0() * a, w, sc.c0());
}

// the edge between cells qb and qc (W = qc - qb, Wup the upwind edge's jump,
// k the correction's factor): normal flux and the fluctuations entering the
// right / upper (P) and the left / lower (M) cell
template <bool FULL>
__device__ __forceinline__ void edge_flux(float c, float W, float Wup, float qb, float qc, float k,
                                          const Scheme<float, FULL>& sc, float& Fn, float& P, float& M) {
  const float cp = fmaxf(c, 0.f), cm = fminf(c, 0.f);
  const float Ft = k * (sc.mc() ? mc_twice(W, Wup) : W);
  const float T = sc.t2() ? Ft : 0.f;
  Fn = fmaf(cp, qb, fmaf(cm, qc, Ft));
  P = fmaf(cp, W, -T);
  M = fmaf(cm, W, T);
}
// (one of the two products with max(c, 0), min(c, 0) is zero: selected)
template <bool FULL>
__device__ __forceinline__ void edge_flux(double c, double W, double Wup, double qb, double qc,
                                          double k, const Scheme<double, FULL>& sc, double& Fn,
                                          double& P, double& M) {
  const bool up = upwind_left(c);
  const double Ft = k * (sc.mc() ? mc_twice(W, Wup) : W);
  const double T = sc.t2() ? Ft : 0.0;
  Fn = fma(c, up ? qb : qc, Ft);
  const double Ts = up ? -T : T;
  const double A = fma(c, W, Ts);
  P = up ? A : -T;
  M = up ? T : A;
}

// the jump on the upwind side of an edge from its four cells
__device__ __forceinline__ float upwind_jump(float c, float qa, float qb, float qc, float qd) {
  return upwind_left(c) ? qb - qa : qd - qc;
}
__device__ __forceinline__ double upwind_jump(double c, double qa, double qb, double qc,
                                              double qd) {
  const bool up = upwind_left(c);
  return (up ? qb : qd) - (up ? qa : qc);
}

// an edge from its four cells qa..qd
template <typename real, bool FULL>
__device__ __forceinline__ void edge(real c, real qa, real qb, real qc, real qd, real k,
                                     const Scheme<real, FULL>& sc, real& Fn, real& P, real& M) {
  edge_flux(c, qc - qb, upwind_jump(c, qa, qb, qc, qd), qb, qc, k, sc, Fn, P, M);
}

// final flux: the normal flux F less the transverse shares of the fluctuation
// sums Xm, Xp in the cells before and beyond the edge
template <bool FULL>
__device__ __forceinline__ float final_flux(float c, float Xm, float Xp, float F,
                                            const Scheme<float, FULL>& sc) {
  const float ct = sc.t1() ? c : 0.f;
  return fmaf(-fmaxf(ct, 0.f), Xm, fmaf(-fminf(ct, 0.f), Xp, F));
}
template <bool FULL>
__device__ __forceinline__ double final_flux(double c, double Xm, double Xp, double F,
                                             const Scheme<double, FULL>& sc) {
  const double X = upwind_left(c) ? Xm : Xp;
  return fma(-c, sc.t1() ? X : 0.0, F);
}

}  // namespace fc
