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
// and the limiter's factors go into the correction's.
// The FP64 pipe issues 1/64 of an SM's slots, so what bounds the FP64 update
// is its count of FP64 instructions: about 25 a cell in this form, of 66 in
// the speeds' own units with min, max and compares in FP64 -- the minima,
// signs and selections are taken on the bits by integer instructions.
// Measured on one GB300, a coarse step before and after: swirl forest of 496
// 32^2 patches in FP64 1.32 -> 0.87 ms (FP32 0.136 -> 0.123 ms), 64 forests
// of 16^2 patches in FP64 5.7 -> 3.7 ms, 256 forests of 32^2 patches in FP32
// 6.5 -> 6.0 ms.  (Those bits have to be taken as magnitude_bits() does.)
#pragma once

#include <algorithm>
#include <limits>

#include "device_util.cuh"

namespace fc {

// The scheme's options.  FULL (second order, MC limiter, transverse
// propagation of both: what runs by default): constants, so the inner loop
// holds no selection by option (8 instructions a cell in FP32).
template <typename real, bool FULL>
struct Scheme {
  // the correction's factor |c| (k0 - k1 |c|) of the limited wave, k1 = 2 k0:
  // MC in FP32 of lim / 2 (k0 = 1), in FP64 of 2 lim (1/4: fewer FP64
  // instructions, see limited()); unlimited of W (1/2); first order 0
  static constexpr real kMC = sizeof(real) == 4 ? real(1) : real(0.25);
  real k0 = kMC, k1 = real(2) * kMC;
  bool mc_ = true;       // MC limiter
  bool t1_ = true, t2_ = true;  // transverse fluctuations; their corrections too
  __device__ __forceinline__ bool mc() const { return FULL || mc_; }
  __device__ __forceinline__ bool t1() const { return FULL || t1_; }
  __device__ __forceinline__ bool t2() const { return FULL || t2_; }
  __device__ __forceinline__ real c0() const { return FULL ? kMC : k0; }
  __device__ __forceinline__ real c1() const { return FULL ? real(2) * kMC : k1; }
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
    sc.k0 = order > 1 ? (sc.mc_ ? sc.kMC : real(0.5)) : real(0);
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
  // (a step so short that this leaves the type's range changes no value: its
  // flux times dt / h is below every field's last bit, but inf times a zero
  // flux is not)
  c.bfac = real(std::min(2.0 / (D.metric ? a.dt : a.nu),
                         double(std::numeric_limits<real>::max())));
  c.alpha = real(a.alpha);
  return c;
}

// does the edge's flow come from its left / lower cell (a zero speed's sign
// does not matter: every use is multiplied by it)
__device__ __forceinline__ bool upwind_left(float c) { return c >= 0.f; }
__device__ __forceinline__ bool upwind_left(double c) { return __double2hiint(c) >= 0; }

// minima and maxima that are NaN where an operand is
__device__ __forceinline__ float min_nan(float a, float b) {
  float m;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(m) : "f"(a), "f"(b));
  return m;
}
__device__ __forceinline__ float min_nan(float a, float b, float c) {
  float m;
  asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(a), "f"(b), "f"(c));
  return m;
}
__device__ __forceinline__ float max_nan(float a, float b, float c) {
  float m;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(a), "f"(b), "f"(c));
  return m;
}

// The MC-limited wave, 0 unless W and Wup share a sign (and where a NaN cell
// leaves no wave), else sign(W) min(|W + Wup| / 2, 2 |W|, 2 |Wup|), up to the
// factor above: half of it in FP32, twice it in FP64.  FP32: the smaller
// magnitude comes with the product of the signs, so the maximum with 0 settles
// both exceptions without a comparison.
__device__ __forceinline__ float limited(float W, float Wup) {
  const float m = min_nan(fabsf(0.25f * (W + Wup)), min_mag_signs(W, Wup));
  return copysignf(fmaxf(m, 0.f), W);
}
// one FP64 instruction (the sum): magnitudes compare as integers, 4 x adds 2
// to the exponent; a minimum below the normal range counts as zero, and a NaN
// sum (an operand was NaN)
__device__ __forceinline__ double limited(double W, double Wup) {
  constexpr unsigned long long kInf = 0x7ff0000000000000ull;
  const unsigned long long aw = magnitude_bits(W), au = magnitude_bits(Wup);
  const unsigned long long mn = aw < au ? aw : au;
  const unsigned long long a = magnitude_bits(W + Wup);
  const unsigned long long m4 = mn + (2ull << 52);
  unsigned long long m = a < m4 ? a : m4;
  const int w = __double2hiint(W);
  if ((w ^ __double2hiint(Wup)) < 0 || mn < (1ull << 52) || a > kInf) m = 0;
  return __hiloint2double((int)(m >> 32) | (w & (int)0x80000000), (int)m);
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

// The edge between cells qb and qc (W = qc - qb, Wup the upwind edge's jump,
// k the correction's factor): normal flux F and the fluctuations P entering
// the right / upper cell, as nP = -P, and M entering the left / lower cell.
// Sums of fluctuations are carried with their sign turned (nX = -X): every
// step is then an addition or a fused multiply-add without a negation of its
// own (an FP64 instruction in FP64, two integer ones in the packed form).
template <bool FULL>
__device__ __forceinline__ void edge_flux(float c, float W, float Wup, float qb, float qc, float k,
                                          const Scheme<float, FULL>& sc, float& F, float& nP,
                                          float& M) {
  const float cp = fmaxf(c, 0.f), cm = fminf(c, 0.f);
  const float Ft = k * (sc.mc() ? limited(W, Wup) : W);
  const float T = sc.t2() ? Ft : 0.f;
  F = fmaf(cp, qb, fmaf(cm, qc, Ft));
  nP = fmaf(-cp, W, T);
  M = fmaf(cm, W, T);
}
// (one of the two fluctuations is the correction alone: selected)
template <bool FULL>
__device__ __forceinline__ void edge_flux(double c, double W, double Wup, double qb, double qc,
                                          double k, const Scheme<double, FULL>& sc, double& F,
                                          double& nP, double& M) {
  const bool up = upwind_left(c);
  const double Ft = k * (sc.mc() ? limited(W, Wup) : W);
  const double T = sc.t2() ? Ft : 0.0;
  F = fma(c, up ? qb : qc, Ft);
  const double B = fma(-fabs(c), W, T);
  nP = up ? B : T;
  M = up ? T : B;
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
                                     const Scheme<real, FULL>& sc, real& F, real& nP, real& M) {
  edge_flux(c, qc - qb, upwind_jump(c, qa, qb, qc, qd), qb, qc, k, sc, F, nP, M);
}

// final flux: the normal flux F less the transverse shares of the fluctuation
// sums in the cells before and beyond the edge (nXm, nXp: turned)
template <bool FULL>
__device__ __forceinline__ float final_flux(float c, float nXm, float nXp, float F,
                                            const Scheme<float, FULL>& sc) {
  const float ct = sc.t1() ? c : 0.f;
  return fmaf(fmaxf(ct, 0.f), nXm, fmaf(fminf(ct, 0.f), nXp, F));
}
template <bool FULL>
__device__ __forceinline__ double final_flux(double c, double nXm, double nXp, double F,
                                             const Scheme<double, FULL>& sc) {
  const double X = upwind_left(c) ? nXm : nXp;
  return fma(c, sc.t1() ? X : 0.0, F);
}

// final_flux as A + B nXm, from the side that is known (nXp)
template <bool FULL>
__device__ __forceinline__ void edge_affine(float c, float nXp, float F,
                                            const Scheme<float, FULL>& sc, float& A, float& B) {
  const float ct = sc.t1() ? c : 0.f;
  A = fmaf(fminf(ct, 0.f), nXp, F);
  B = fmaxf(ct, 0.f);
}
template <bool FULL>
__device__ __forceinline__ void edge_affine(double c, double nXp, double F,
                                            const Scheme<double, FULL>& sc, double& A,
                                            double& B) {
  const bool up = upwind_left(c);
  A = up || !sc.t1() ? F : fma(c, nXp, F);
  B = up && sc.t1() ? c : 0.0;
}

}  // namespace fc

// ------------------------------------------------ the walk's packed form
//
// The FP32 walk computes two cells at a time in packed registers (float2:
// add, sub, mul and fma are one instruction for both), the FP64 walk one
// (double).
namespace fc {

__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 vsub(float2 a, float2 b) {
  float2 r;
  asm("{\n .reg .b64 a, b, c;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n"
      " sub.rn.f32x2 c, a, b;\n mov.b64 {%0, %1}, c;\n}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ double vadd(double a, double b) { return a + b; }
__device__ __forceinline__ double vsub(double a, double b) { return a - b; }
__device__ __forceinline__ double vmul(double a, double b) { return a * b; }
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }

template <typename real>
struct Packed;
template <>
struct Packed<float> {
  using V = float2;
  static constexpr int N = 2;
  static __device__ __forceinline__ V all(float a) { return make_float2(a, a); }
  static __device__ __forceinline__ V make(float a, float b) { return make_float2(a, b); }
  static __device__ __forceinline__ float get(V v, int k) { return k ? v.y : v.x; }
};
template <>
struct Packed<double> {
  using V = double;
  static constexpr int N = 1;
  static __device__ __forceinline__ V all(double a) { return a; }
  static __device__ __forceinline__ V make(double a, double) { return a; }
  static __device__ __forceinline__ double get(V v, int) { return v; }
};

// a half Courant number, split by sign where the products with both parts
// are cheaper than a selection (FP32)
template <typename V>
struct Speed;
template <>
struct Speed<float2> {
  float2 c, p, m;  // p + m = c
  Speed() = default;
  __device__ __forceinline__ explicit Speed(float2 v) : c(v) {
    p = make_float2(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f));
    m = vsub(v, p);
  }
};
template <>
struct Speed<double> {
  double c;
  Speed() = default;
  __device__ __forceinline__ explicit Speed(double v) : c(v) {}
};

// limited() of both packed cells: the same value, by ordering (fewer
// instructions; the form above has the shorter chain, which the band update
// with its few warps waits for: 0.139 against 0.123 ms a coarse step)
__device__ __forceinline__ float2 limited(float2 W, float2 U) {
  const float2 s4 = vmul(vadd(W, U), make_float2(0.25f, 0.25f));
  const float2 lo = make_float2(fmaxf(min_nan(s4.x, W.x, U.x), 0.f),
                                fmaxf(min_nan(s4.y, W.y, U.y), 0.f));
  const float2 hi = make_float2(fminf(max_nan(s4.x, W.x, U.x), 0.f),
                                fminf(max_nan(s4.y, W.y, U.y), 0.f));
  return vadd(lo, hi);
}

// one edge for both packed cells: normal flux F, nP = -P and M
template <bool FULL>
__device__ __forceinline__ void vedge(const Speed<float2>& s, float2 W, float2 U, float2 qb,
                                      float2 qc, const Scheme<float, FULL>& sc, float2& F,
                                      float2& nP, float2& M) {
  const float2 ab = vsub(s.p, s.m);  // |c|
  const float c0 = sc.c0(), c1 = -sc.c1();
  const float2 k = vmul(ab, vfma(make_float2(c1, c1), ab, make_float2(c0, c0)));
  const float2 Ft = vmul(k, sc.mc() ? limited(W, U) : W);
  const float2 T = sc.t2() ? Ft : make_float2(0.f, 0.f);
  F = vfma(s.p, qb, vfma(s.m, qc, Ft));
  nP = vfma(s.p, vsub(qb, qc), T);
  M = vfma(s.m, W, T);
}
template <bool FULL>
__device__ __forceinline__ void vedge(const Speed<double>& s, double W, double U, double qb,
                                      double qc, const Scheme<double, FULL>& sc, double& F,
                                      double& nP, double& M) {
  edge_flux(s.c, W, U, qb, qc, corr_factor(s.c, sc), sc, F, nP, M);
}

__device__ __forceinline__ float2 vselect(float2 c, float2 a, float2 b) {
  return make_float2(upwind_left(c.x) ? a.x : b.x, upwind_left(c.y) ? a.y : b.y);
}
__device__ __forceinline__ double vselect(double c, double a, double b) {
  return upwind_left(c) ? a : b;
}
// the jump on the upwind side from an edge's four cells
__device__ __forceinline__ float2 vupwind(float2 c, float2 qa, float2 qb, float2 qc, float2 qd) {
  return vselect(c, vsub(qb, qa), vsub(qd, qc));
}
__device__ __forceinline__ double vupwind(double c, double qa, double qb, double qc, double qd) {
  return upwind_jump(c, qa, qb, qc, qd);
}

// final flux from the turned sums nXm, nXp
template <bool FULL>
__device__ __forceinline__ float2 vfinal(const Speed<float2>& s, float2 nXm, float2 nXp, float2 F,
                                         const Scheme<float, FULL>& sc) {
  return sc.t1() ? vfma(s.p, nXm, vfma(s.m, nXp, F)) : F;
}
template <bool FULL>
__device__ __forceinline__ double vfinal(const Speed<double>& s, double nXm, double nXp, double F,
                                         const Scheme<double, FULL>& sc) {
  return final_flux(s.c, nXm, nXp, F, sc);
}

}  // namespace fc
