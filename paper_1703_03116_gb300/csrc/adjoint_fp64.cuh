// The FP64 transpose of a patch's update, in the forward kernels' units
// (walk_edge.cuh): an edge speed s enters as c = s dt / (2 h), and fluxes and
// fluctuations carry dt / (2 h), so no separate dt/h is left: the update is
// q - 2 (dF + dG), a fluctuation's transverse share c X.  The velocity-scale
// derivative sum_e dL/ds_e s_e = sum_e dL/dc_e c_e is the same in either.
//
// The FP64 pipe (1/64 of an SM's issue slots) bounds these kernels: minima,
// signs and selections are taken on the bits, and an edge's forward values
// and its transpose together take about 27 FP64 instructions, half of what
// the form in the speeds' own units takes.  4 coarse steps of 229 patches of
// 32^2 and their gradient: 5.0 -> 3.7 ms, 3.2 ms with magnitudes and
// negations on the bits too (magnitude_bits()), 3.1 ms with a column's factors
// kept over its rows and one addition less an edge.
//
// FP32 keeps that form (adjoint.cu): in the adjoint of a global step its
// instructions are 2% (in the multirate reverse, which this does not say
// anything of, its transposes are what the time goes to).  Its velocity-scale
// derivative is summed in FP32 by a thread and a warp and in FP64 from there
// on; other roundings of the terms move it by 1e-7.
#pragma once

#include "walk_edge.cuh"

namespace fc {
namespace half {

struct AdjScheme {
  bool o2, mc, t1, t2;  // second order, MC limiter, transverse fluctuations, corrections
};

// |a|, -a
__device__ __forceinline__ double magnitude(double a) {
  return __longlong_as_double((long long)magnitude_bits(a));
}
__device__ __forceinline__ double turned(double a) {
  int hi;
  asm("xor.b32 %0, %1, 0x80000000;" : "=r"(hi) : "r"(__double2hiint(a)));
  return __hiloint2double(hi, __double2loint(a));
}

// Forward values of an edge that its transpose reads: jump W, limited wave L
// and its partials dW, dU with respect to W and the upwind jump on the piece
// the data select, the correction's factor kap and the correction Ft = kap L,
// and the fluctuations (P turned).
template <typename real>
struct EdgeFw {
  real W, L, dW, dU, kap, Ft, nP, M;
  bool up;
};

template <typename real>
__device__ __forceinline__ EdgeFw<real> edge_fw(const AdjScheme& sc, real c, real qa, real qb,
                                                real qc, real qd) {
  EdgeFw<real> e;
  e.up = upwind_left(c);
  e.W = qc - qb;
  const real a = magnitude(c);
  if (sc.mc) {
    const real U = upwind_jump(c, qa, qb, qc, qd);
    const real S = e.W + U;
    // the pieces (W + U) / 2, 2 W, 2 U; ties take the first.  A wave that
    // the forward limiter drops has no partials: jumps of two signs, one below
    // the normal range (where adding 2 to the exponent is not 4 x), a NaN
    constexpr unsigned long long kInf = 0x7ff0000000000000ull, kMin = 1ull << 52;
    const unsigned long long mW = magnitude_bits(e.W), mU = magnitude_bits(U);
    const unsigned long long mS = magnitude_bits(S), k4 = 2ull << 52;  // (4 x: exponent + 2)
    const bool on = (__double2hiint(e.W) ^ __double2hiint(U)) >= 0 && mW >= kMin && mU >= kMin &&
                    mS <= kInf;
    const bool half = mS <= mW + k4 && mS <= mU + k4, byW = mW <= mU;
    const real f = half ? real(0.5) : real(2);
    e.L = on ? f * (half ? S : byW ? e.W : U) : real(0);
    e.dW = on && (half || byW) ? f : real(0);
    e.dU = on && (half || !byW) ? f : real(0);
  } else {
    e.L = e.W;
    e.dW = real(1);
    e.dU = real(0);
  }
  e.kap = a * (real(0.5) - a);
  if (!sc.o2) e.kap = e.L = real(0);
  e.Ft = e.kap * e.L;
  const real T = sc.t2 ? e.Ft : real(0);
  const real B = fma(-a, e.W, T);
  e.nP = e.up ? B : T;
  e.M = e.up ? T : B;
  return e;
}

// One edge's transpose: e is the forward edge at half Courant number c between
// cells a, b, c, d along its normal (qb, qc the middle two); lF, lP, lM the
// adjoints of its normal flux and of the fluctuations it sends into c's and
// b's side.  Returns the four cells' adjoint contributions and c lF, and adds
// the derivative with respect to the edge speed times the speed to ds.
template <typename real>
struct EdgeAdj {
  real a, b, c, d, cF;
};

template <typename real>
__device__ __forceinline__ EdgeAdj<real> edge_transpose(const EdgeFw<real>& e, const AdjScheme& sc,
                                                       real c, real qb, real qc, real lF,
                                                       real lP, real lM, real& ds) {
  const real lFt = sc.t2 ? lF + (lM - lP) : lF;
  const real a = magnitude(c);
  const real lsel = sc.t1 ? (e.up ? lP : lM) : real(0);
  const real cl = c * lsel, g = e.kap * lFt;
  EdgeAdj<real> o;
  o.cF = c * lF;
  const real lW = fma(e.dW, g, cl), lU = e.dU * g;
  const real nU = turned(lU), nW = turned(lW);
  // on the upwind cell, then with the jump's share of its side
  const real v = (o.cF + (e.up ? lU : nU)) + (e.up ? nW : lW);
  o.b = e.up ? v : nW;
  o.c = e.up ? lW : v;
  o.a = e.up ? nU : real(0);
  o.d = e.up ? real(0) : lU;
  // d(kap)/dc c = |c| (1/2 - 2 |c|) = kap - |c|^2
  const real u = fma(-a, a * e.L, e.Ft);
  ds = fma(lFt, u, fma(cl, e.W, fma(o.cF, e.up ? qb : qc, ds)));
  return o;
}

template <typename real>
__device__ __forceinline__ real pos(real c) { return upwind_left(c) ? c : real(0); }
template <typename real>
__device__ __forceinline__ real neg(real c) { return upwind_left(c) ? real(0) : c; }

// The edges' half Courant numbers: a factor of the column times one of the
// row (swirl), or constant.
template <typename real>
struct AdjSpeeds {
  const real *Sx, *Sy, *Tx, *Ty;  // the patch's tables, node k at [k + 1]
  real uc, cu, cv;
  bool swirl;
  __device__ __forceinline__ real xfac(int i) const { return swirl ? uc * Sx[i + 1] : real(0); }
  __device__ __forceinline__ real yfac(int i) const { return swirl ? -uc * Tx[i + 1] : real(0); }
  __device__ __forceinline__ real u(real f, int j) const { return swirl ? f * Ty[j + 1] : cu; }
  __device__ __forceinline__ real v(real f, int j) const { return swirl ? f * Sy[j + 1] : cv; }
};

// Transpose of the update of one patch (its final fluxes, their transverse
// increments and every edge), as a row walk: thread tid's lane li owns
// column li of the band of R rows starting at r0 = (tid / MX) R and walks
// rows r0 - 1 .. r0 + R, recomputing the forward edges it needs from the
// tile Q (x-edge (li, j) and y-edge (li, j + 1) at row j), taking the
// neighbouring column's values by shuffles, and transposing the x-edges of
// rows [r0, r0 + R) and the y-edges of rows [r0, r0 + R) (band 0 also the
// x-edges of row -1, the last band those of row MX and its y-edges).  The
// contributions to a cell's adjoint gather in a four-row register window of
// the lane's column and reach LQ (zeroed) by one shared atomic add per cell
// and band; ghost columns take theirs directly.  The edges of column MX (x)
// and of ghost columns -1 and MX (y) are side_transpose's.  LN: twice the
// adjoint of the new interior (the update's factor); XMe[j + 1]: forward M
// of x-edge (MX, j); YPm[j], YMm[j]: forward P (turned), M of y-edge (-1, j).
// Returns the lane's share of sum ds.
template <typename real, int MX, int R>
__device__ __forceinline__ real band_transpose(const real* Q, real* LQ, const real* LN,
                                               const real* XMe, const real* YPm, const real* YMm,
                                               const AdjScheme& sc, const AdjSpeeds<real>& sp,
                                               int tid) {
  constexpr int S = MX + 4;
  constexpr unsigned kAll = 0xffffffffu;
  const int li = tid % MX, r0 = (tid / MX) * R, r1 = r0 + R;
  const bool last = r1 == MX;
  // a column's factors, kept (the tables would be read and multiplied again
  // after every atomic add)
  const real ux = sp.xfac(li), uxE = sp.xfac(MX), vy = sp.yfac(li);
  auto uvel = [&](int j) -> real { return sp.u(ux, j); };
  auto vvel = [&](int j) -> real { return sp.v(vy, j); };
  auto q = [&](int i, int j) -> real { return Q[(j + kMbc) * S + i + kMbc]; };
  auto ln = [&](int j) -> real { return (j >= 0 && j < MX) ? LN[j * MX + li] : real(0); };
  auto flush = [&](int row, real v) {
    if (row >= -kMbc && row <= MX + 1) atomicAdd(&LQ[(row + kMbc) * S + li + kMbc], v);
  };
  real dsum = 0;
  real A0 = 0, A1 = 0, A2 = 0, A3 = 0;  // contributions to rows j-2 .. j+1
  real qa = q(li, r0 - 2), qb = q(li, r0 - 1), qc = q(li, r0), qd = 0;
  real ln_cur = ln(r0 - 1);
  real v_cur = r0 - 1 >= 0 ? vvel(r0 - 1) : real(0);
  real lGf_cur = r0 - 1 >= 0 ? ln_cur - ln(r0 - 2) : real(0);
  real nP_prev = 0, nX_prev = 0, lY_prev = 0;
  EdgeFw<real> ey{};  // forward y-edge (li, j)
#pragma unroll(R <= 8 ? R + 2 : 2)
  for (int it = 0; it < R + 2; ++it) {
    const int j = r0 - 1 + it;
    const bool xrow = (j >= r0 && j < r1) || j == -1 || (last && j == MX);
    const bool yrow = (j >= r0 && j < r1) || (last && j == MX);
    if (j + 2 <= MX + 1) qd = q(li, j + 2);
    // forward: x-edge (li, j), y-edge (li, j + 1)
    const real su = uvel(j);
    const real ql = q(li - 1, j);
    const EdgeFw<real> ex = edge_fw(sc, su, q(li - 2, j), ql, qb, q(li + 1, j));
    real vn = 0;
    EdgeFw<real> eyn{};
    if (j + 1 <= MX) {
      vn = vvel(j + 1);
      eyn = edge_fw(sc, vn, qa, qb, qc, qd);
    }
    // adjoints of the final fluxes and of the fluctuation sums
    const real ln_next = ln(j + 1);
    const real lGf_next = j + 1 <= MX ? ln_next - ln_cur : real(0);  // y-edge (li, j+1)
    real ln_left = __shfl_up_sync(kAll, ln_cur, 1, MX);
    if (li == 0) ln_left = real(0);
    const bool frow = j >= 0 && j < MX;
    const real lFf = frow ? ln_cur - ln_left : real(0);  // x-edge (li, j)
    real lFf_r = __shfl_down_sync(kAll, lFf, 1, MX);     // x-edge (li+1, j)
    real su_r = __shfl_down_sync(kAll, su, 1, MX);
    if (li == MX - 1) {
      lFf_r = frow ? turned(ln_cur) : real(0);
      su_r = sp.u(uxE, j);
    }
    // (turned: nlY, nlX the negated adjoints of Y(li, j), X(li, j))
    const real nlY = frow && sc.t1 ? fma(pos(su_r), lFf_r, neg(su) * lFf) : real(0);
    const real nlX =
        sc.t1 ? fma(pos(vn), lGf_next, j >= 0 ? neg(v_cur) * lGf_cur : real(0)) : real(0);
    const real lY = turned(nlY), lX = turned(nlX);
    real lX_l = __shfl_up_sync(kAll, lX, 1, MX);  // X(li-1, j)
    if (li == 0) lX_l = real(0);
    // forward fluctuation sums, turned: X(li, j), Y(li, j), Y(li-1, j)
    real XM_r = __shfl_down_sync(kAll, ex.M, 1, MX);
    if (li == MX - 1) XM_r = XMe[j + 1];
    const real nX = ex.nP - XM_r;
    const real nY = nP_prev - eyn.M;
    real nY_l = __shfl_up_sync(kAll, nY, 1, MX);
    if (li == 0) nY_l = frow ? YPm[j] - YMm[j + 1] : real(0);
    // x-edge (li, j)
    EdgeAdj<real> ox{0, 0, 0, 0, 0};
    if (xrow) ox = edge_transpose(ex, sc, su, ql, qb, lFf, lX, lX_l, dsum);
    if (sc.t1 && xrow && frow) dsum = fma(ox.cF, ex.up ? nY_l : nY, dsum);
    real T = ox.c;
    {
      const real b1 = __shfl_down_sync(kAll, ox.b, 1, MX);
      const real a2 = __shfl_down_sync(kAll, ox.a, 2, MX);
      const real d1 = __shfl_up_sync(kAll, ox.d, 1, MX);
      if (li + 1 < MX) T += b1;
      if (li + 2 < MX) T += a2;
      if (li >= 1) T += d1;
    }
    if (xrow) {  // contributions to the ghost columns
      if (li == 0) {
        atomicAdd(&LQ[(j + kMbc) * S + 0], ox.a);
        atomicAdd(&LQ[(j + kMbc) * S + 1], ox.b);
      }
      if (li == 1) atomicAdd(&LQ[(j + kMbc) * S + 1], ox.a);
      if (li == MX - 1) atomicAdd(&LQ[(j + kMbc) * S + MX + kMbc], ox.d);
    }
    // y-edge (li, j)
    if (yrow) {
      const EdgeAdj<real> oy = edge_transpose(ey, sc, v_cur, qa, qb, lGf_cur,
                                              j < MX ? lY : real(0), j > 0 ? lY_prev : real(0),
                                              dsum);
      if (sc.t1) dsum = fma(oy.cF, ey.up ? nX_prev : nX, dsum);
      A0 += oy.a;
      A1 += oy.b;
      A2 += oy.c;
      A3 += oy.d;
    }
    A2 += T;
    if (j >= r0 && j < r1) A2 = fma(real(0.5), ln_cur, A2);  // the update's identity part
    flush(j - 2, A0);
    A0 = A1;
    A1 = A2;
    A2 = A3;
    A3 = real(0);
    nX_prev = nX;
    lY_prev = lY;
    ey = eyn;
    nP_prev = eyn.nP;
    v_cur = vn;
    lGf_cur = lGf_next;
    ln_cur = ln_next;
    qa = qb;
    qb = qc;
    qc = qd;
  }
  const int jl = r0 + R;  // the last row walked
  flush(jl - 1, A0);
  flush(jl, A1);
  flush(jl + 1, A2);
  return dsum;
}

// The edges band_transpose leaves: x-edge (MX, j), j in [-1, MX], and the
// y-edges of ghost columns -1 and MX, j in [0, MX] (threads tid, stride
// nt, one edge each, contributions by shared atomic adds).  Returns the
// threads' share of sum ds.
template <typename real, int MX, class UV, class VV>
__device__ __forceinline__ real side_transpose(const real* Q, real* LQ, const real* LN,
                                               const AdjScheme& sc, UV uvel, VV vvel, int tid,
                                               int nt) {
  constexpr int S = MX + 4;
  auto q = [&](int i, int j) -> real { return Q[(j + kMbc) * S + i + kMbc]; };
  auto ln = [&](int i, int j) -> real {
    return (i >= 0 && i < MX && j >= 0 && j < MX) ? LN[j * MX + i] : real(0);
  };
  auto add = [&](int i, int j, real v) { atomicAdd(&LQ[(j + kMbc) * S + i + kMbc], v); };
  // adjoints of the final fluxes of x-edge (i, j) and y-edge (i, j)
  auto lFf = [&](int i, int j) -> real {
    return (j >= 0 && j < MX) ? ln(i, j) - ln(i - 1, j) : real(0);
  };
  auto lGf = [&](int i, int j) -> real {
    return (i >= 0 && i < MX && j >= 0 && j <= MX) ? ln(i, j) - ln(i, j - 1) : real(0);
  };
  auto yedge = [&](int c, int j) {
    return edge_fw(sc, vvel(c, j), q(c, j - 2), q(c, j - 1), q(c, j), q(c, j + 1));
  };
  real dsum = 0;
  for (int k = tid; k < 3 * MX + 4; k += nt) {
    if (k < MX + 2) {  // x-edge (MX, j): its P enters no updated cell; M enters (MX-1, j)
      const int j = k - 1;
      const real s = uvel(MX, j);
      const EdgeFw<real> e =
          edge_fw(sc, s, q(MX - 2, j), q(MX - 1, j), q(MX, j), q(MX + 1, j));
      const real lF = lFf(MX, j);
      real nlM = 0;
      if (sc.t1)
        nlM = (j + 1 <= MX ? pos(vvel(MX - 1, j + 1)) * lGf(MX - 1, j + 1) : real(0)) +
              (j >= 0 ? neg(vvel(MX - 1, j)) * lGf(MX - 1, j) : real(0));
      const EdgeAdj<real> o =
          edge_transpose(e, sc, s, q(MX - 1, j), q(MX, j), lF, real(0), turned(nlM), dsum);
      add(MX - 2, j, o.a);
      add(MX - 1, j, o.b);
      add(MX, j, o.c);
      add(MX + 1, j, o.d);
      if (sc.t1 && j >= 0 && j < MX) {  // its transverse increment's speed
        const int c = e.up ? MX - 1 : MX;
        dsum = fma(o.cF, yedge(c, j).nP - yedge(c, j + 1).M, dsum);
      }
    } else {  // y-edge (c, j) of ghost column c = -1 or MX (no flux of its own updates a cell)
      const bool right = k >= 2 * MX + 3;
      const int j = k - (right ? 2 * MX + 3 : MX + 2);
      const int c = right ? MX : -1;
      const real s = vvel(c, j);
      const EdgeFw<real> e = yedge(c, j);
      // adjoint of Y(c, r): from x-edge (0, r)'s u+ (c = -1) or (MX, r)'s u- (c = MX)
      auto lY = [&](int r) -> real {
        if (r < 0 || r >= MX || !sc.t1) return real(0);
        return turned(right ? neg(uvel(MX, r)) * lFf(MX, r) : pos(uvel(0, r)) * lFf(0, r));
      };
      const EdgeAdj<real> o =
          edge_transpose(e, sc, s, q(c, j - 1), q(c, j), real(0), lY(j), lY(j - 1), dsum);
      add(c, j - 2, o.a);
      add(c, j - 1, o.b);
      add(c, j, o.c);
      add(c, j + 1, o.d);
    }
  }
  return dsum;
}

}  // namespace half
}  // namespace fc
