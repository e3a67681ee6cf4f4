// Cubed-sphere metric terms (Sec. 5.3: advection on the mapped unit sphere).
//
// The wave-propagation update on a mapped grid runs in capacity form: each
// cell carries its area kappa on the sphere, each edge the volume flux of
// the velocity through it.  For the solid-body rotation u = omega x X the
// velocity has the stream function psi = -omega . X on the unit sphere, so
// the flux through an edge is a difference of psi at its two end points;
// across an x-edge (from its lower end a to its upper end b) it is
// omega . (X_b - X_a), across a y-edge (from its left end a to its right end
// b) omega . (X_a - X_b), positive along +x and +y.  The difference is taken
// of the end points before the dot product (psi itself is O(1), the flux
// O(h)).  Cells are bounded by great circles (gnomonic grid lines), so the
// area is exactly that of two spherical triangles, each by the formula of
// Van Oosterom and Strackee (1983): tan(E/2) = |a . (b x c)| /
// (1 + a.b + b.c + c.a).
//
// The metrics of a patch cover its ghost cells too (the patch's own mapping
// extended past its block) and are computed in FP64 once per layout: kappa
// is kept in FP64, the update's block (1/kappa, phi_x, phi_y) in the field's
// precision.
//
// The deformational flow of Sec. 5.3 has a time-dependent streamfunction
// psi = k sin^2(rho - 2 pi t/T) cos^2(theta) cos(pi t/T) - 2 pi sin(theta)/T_f.
// With s = Y cos a - X sin a (a = 2 pi t/T), which is sin(rho - a) cos(theta),
// and sin(theta) = Z, psi = k c s^2 - (2 pi/T_f) Z (c = cos(pi t/T)); an edge
// flux psi(b) - psi(a) = k c (s_b - s_a)(s_b + s_a) - (2 pi/T_f)(Z_b - Z_a) is
// again formed from the end points' differences: (s_b - s_a)(s_b + s_a) =
// cos^2 a E1 - cos a sin a E2 + sin^2 a E3 with E1 = dY SY, E2 = dY SX + dX SY,
// E3 = dX SX (d the difference, S the sum over the end points), and E4 = dZ.
// These four are kept per edge, so a substep's flux is four multiply-adds an
// edge instead of the twelve of the end points' form (the FP64 pipe bounds the
// refresh), and the time's sine and cosines are taken once per CTA, by three
// threads of three warps.  432 patches of 32^2: 47 -> 20 us.  They take more
// memory than the corners (71.8 against 29.4 KB a 32^2 patch), so a layout
// whose coefficients exceed the forest's budget keeps the corners and forms
// the same values at each refresh: the same bits.  A global step of 1536
// patches of 32^2, FP32 and FP64: 63 and 202 us from coefficients, 141 and 279
// from corners (the end points' form from corners: 210 and 592).
#include <atomic>
#include <cmath>

#include "device_util.cuh"

namespace fc {
namespace {

__device__ __forceinline__ double axis_component(int code, int k) {
  return (code == k + 1) ? 1.0 : (code == -(k + 1)) ? -1.0 : 0.0;
}

// the triple product as a . ((b - a) x (c - a)): equal to a . (b x c), but
// without cancelling from O(1) terms down to O(h^2) for a small triangle
__device__ __forceinline__ double tri_area(const double* a, const double* b, const double* c) {
  const double u0 = b[0] - a[0], u1 = b[1] - a[1], u2 = b[2] - a[2];
  const double v0 = c[0] - a[0], v1 = c[1] - a[1], v2 = c[2] - a[2];
  const double w0 = u1 * v2 - u2 * v1;
  const double w1 = u2 * v0 - u0 * v2;
  const double w2 = u0 * v1 - u1 * v0;
  const double num = fabs(a[0] * w0 + a[1] * w1 + a[2] * w2);
  const double ab = a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
  const double bcd = b[0] * c[0] + b[1] * c[1] + b[2] * c[2];
  const double ca = c[0] * a[0] + c[1] * a[1] + c[2] * a[2];
  return 2.0 * atan2(num, 1.0 + ab + bcd + ca);
}

// an edge's four coefficients from its end points a, b; sg: the sign of psi(b)
// less psi(a) in the flux (the roundings written out: the kept and the
// refresh's own are the same bits)
struct EdgeCoef {
  double e1, e2, e3, e4;
};
__device__ __forceinline__ EdgeCoef edge_coef(const double* a, const double* b, double sg) {
  const double dX = sg * (b[0] - a[0]), dY = sg * (b[1] - a[1]);
  const double sX = a[0] + b[0], sY = a[1] + b[1];
  return EdgeCoef{dY * sY, fma(dY, sX, __dmul_rn(dX, sY)), dX * sX, sg * (b[2] - a[2])};
}

// one CTA per patch; X: the (S+1)^2 grid corners on the sphere, in shared
// memory as three planes.  After a regrid (rm != null) a patch that kept its
// quadrant copies its blocks from the old layout's store instead.
template <typename real>
__global__ void __launch_bounds__(256) metrics_kernel(const PatchMeta* meta, int npatch, int mx,
                                                      double w0, double w1, double w2,
                                                      double* metric, real* umetric,
                                                      const RemapEntry* rm,
                                                      const double* old_metric,
                                                      const real* old_umetric, double* coef,
                                                      bool corners) {
  extern __shared__ double Xs[];
  const int S = mx + 2 * kMbc, SN = S + 1, NE = S * SN;
  double* X0 = Xs;
  double* X1 = X0 + SN * SN;
  double* X2 = X1 + SN * SN;
  for (int p = blockIdx.x; p < npatch; p += gridDim.x) {
    double* K = metric + (size_t)p * S * S;
    real* U = umetric + (size_t)p * umetric_stride(S);
    if (rm && rm[p].kind == RM_COPY) {
      const double2* sk = reinterpret_cast<const double2*>(old_metric + (size_t)rm[p].src[0] * S * S);
      for (int k = threadIdx.x; k < S * S / 2; k += blockDim.x)
        reinterpret_cast<double2*>(K)[k] = sk[k];
      const double2* su = reinterpret_cast<const double2*>(
          old_umetric + (size_t)rm[p].src[0] * umetric_stride(S));
      const int n2 = umetric_stride(S) * (int)sizeof(real) / (int)sizeof(double2);
      for (int k = threadIdx.x; k < n2; k += blockDim.x) reinterpret_cast<double2*>(U)[k] = su[k];
      continue;
    }
    const PatchMeta pm = meta[p];
    int n, ex, ey;
    cube_face(pm.block, &n, &ex, &ey);
    const double h = 1.0 / ldexp((double)mx, pm.level);
    for (int k = threadIdx.x; k < SN * SN; k += blockDim.x) {
      const int i = k % SN, j = k / SN;
      const double x = ((double)pm.x * mx + (i - kMbc)) * h;
      const double y = ((double)pm.y * mx + (j - kMbc)) * h;
      const double ta = tan((x - 0.5) * M_PI / 2.0), tb = tan((y - 0.5) * M_PI / 2.0);
      double P[3];
      for (int c = 0; c < 3; ++c)
        P[c] = axis_component(n, c) + ta * axis_component(ex, c) + tb * axis_component(ey, c);
      const double len = sqrt(P[0] * P[0] + P[1] * P[1] + P[2] * P[2]);
      X0[k] = P[0] / len;
      X1[k] = P[1] / len;
      X2[k] = P[2] / len;
    }
    __syncthreads();
    auto corner = [&](int i, int j, double* v) {
      const int k = j * SN + i;
      v[0] = X0[k];
      v[1] = X1[k];
      v[2] = X2[k];
    };
    for (int k = threadIdx.x; k < S * S; k += blockDim.x) {
      const int i = k % S, j = k / S;
      double a[3], b[3], c[3], d[3];
      corner(i, j, a);
      corner(i + 1, j, b);
      corner(i + 1, j + 1, c);
      corner(i, j + 1, d);
      K[k] = tri_area(a, b, c) + tri_area(a, c, d);
      U[k] = real(1) / real(K[k]);
    }
    for (int k = threadIdx.x; k < 2 * NE; k += blockDim.x) {
      // x-edge i-1/2 of row j: corners (i, j) below (a), (i, j+1) above (b);
      // y-edge j-1/2 of column i: corners (i, j) left (a), (i+1, j) right (b)
      const bool y = k >= NE;
      const int e = y ? k - NE : k, w = y ? S : SN;
      const int i = e % w, j = e / w;
      double a[3], b[3];
      corner(i, j, a);
      corner(y ? i + 1 : i, y ? j : j + 1, b);
      if (y) {
        U[S * S + k] = real(w0 * (a[0] - b[0]) + w1 * (a[1] - b[1]) + w2 * (a[2] - b[2]));
      } else {
        U[S * S + k] = real(w0 * (b[0] - a[0]) + w1 * (b[1] - a[1]) + w2 * (b[2] - a[2]));
      }
      // of the edges an update reads: the flux is psi's difference
      // of the lower less the upper end of an x-edge, the right less the left
      // end of a y-edge
      const int ei = i - kMbc, ej = j - kMbc;
      if (coef && !corners && ei >= (y ? -1 : 0) && ei <= mx && ej >= (y ? 0 : -1) && ej <= mx) {
        const EdgeCoef c = edge_coef(a, b, y ? 1.0 : -1.0);
        const int NK = 2 * edges_read(mx);
        double* C = coef + (size_t)p * coef_stride(mx, false) +
                    (y ? NK / 2 + ej * (mx + 2) + ei + 1 : (ej + 1) * (mx + 1) + ei);
        C[0] = c.e1;
        C[NK] = c.e2;
        C[2 * NK] = c.e3;
        C[3 * NK] = c.e4;
      }
    }
    if (coef && corners) {
      const int M = mx + 3;  // nodes -1..mx+1
      double* C = coef + (size_t)p * coef_stride(mx, true);
      for (int k = threadIdx.x; k < M * M; k += blockDim.x)
        for (int c = 0; c < 3; ++c)
          C[c * M * M + k] = (c == 0 ? X0 : c == 1 ? X1 : X2)[(k / M + 1) * SN + k % M + 1];
    }
    __syncthreads();
  }
}

// phi_x, phi_y of the update's blocks of patches [p0, p1) at time t, of the
// edges an update reads; CORNERS: coef holds the grid corners (the coefficients
// are formed here: 13 FP64 instructions an edge instead of 4)
template <typename real, int MX, bool CORNERS>
__global__ void __launch_bounds__(512) deform_fluxes_kernel(int p0, int p1,
                                                            const double* __restrict__ coef,
                                                            real* __restrict__ umetric, double kc,
                                                            double T, double rot, double t_half,
                                                            const double* t0_dev, double t_off) {
  constexpr int S = MX + 2 * kMbc, SN = S + 1, NE = S * SN, NK = 2 * edges_read(MX);
  constexpr int M = MX + 3;
  __shared__ double tr[3];
  const double t = t0_dev ? *t0_dev + t_off : t_half;
  if (threadIdx.x == 0) tr[0] = cospi(2.0 * t / T);
  if (threadIdx.x == 32) tr[1] = sinpi(2.0 * t / T);
  if (threadIdx.x == 64) tr[2] = kc * cospi(t / T);
  __syncthreads();
  const double c1 = tr[2] * tr[0] * tr[0], c2 = -tr[2] * tr[0] * tr[1],
               c3 = tr[2] * tr[1] * tr[1];
  for (int p = p0 + blockIdx.x; p < p1; p += gridDim.x) {
    const double* C = coef + (size_t)p * coef_stride(MX, CORNERS);
    real* U = umetric + (size_t)p * umetric_stride(S) + S * S;
    for (int k = threadIdx.x; k < NK; k += blockDim.x) {
      const bool y = k >= NK / 2;
      const int e = y ? k - NK / 2 : k;
      // x-edges: MX + 1 a row, rows 1..MX + 2 of the extended range; y-edges:
      // MX + 2 a row
      const int o = y ? NE + (e / (MX + 2) + 2) * S + e % (MX + 2) + 1
                      : (e / (MX + 1) + 1) * SN + e % (MX + 1) + 2;
      if constexpr (CORNERS) {
        const double* A = C + (y ? (e / (MX + 2) + 1) * M + e % (MX + 2)
                                 : (e / (MX + 1)) * M + e % (MX + 1) + 1);
        const double* B = A + (y ? 1 : M);
        const double a[3] = {A[0], A[M * M], A[2 * M * M]};
        const double b[3] = {B[0], B[M * M], B[2 * M * M]};
        const EdgeCoef f = edge_coef(a, b, y ? 1.0 : -1.0);
        U[o] = real(fma(-rot, f.e4, fma(c1, f.e1, fma(c2, f.e2, c3 * f.e3))));
      } else {  // (written out: through an EdgeCoef a refresh took 0.3 us longer)
        U[o] = real(
            fma(-rot, C[3 * NK + k], fma(c1, C[k], fma(c2, C[NK + k], c3 * C[2 * NK + k]))));
      }
    }
  }
}

template <typename real, int MX>
void deform_launch(int p0, int p1, const double* coef, bool corners, real* umetric, double kc,
                   double T, double rot, double t_half, const double* t0_dev, double t_off,
                   cudaStream_t s) {
  // (an SM's share of the patches by one CTA of as many threads as a patch
  // feeds for some rounds: the time's functions once a CTA)
  const int n = p1 - p0, grid = n < 304 ? n : 304;
  auto kern = corners ? deform_fluxes_kernel<real, MX, true> : deform_fluxes_kernel<real, MX, false>;
  kern<<<grid, MX == 32 ? 512 : 128, 0, s>>>(p0, p1, coef, umetric, kc, T, rot, t_half, t0_dev,
                                             t_off);
}

}  // namespace

template <typename real>
cudaError_t launch_deform_fluxes(int p0, int p1, int mx, const double* coef, bool corners,
                                 real* umetric, double kc, double T, double rot, double t_half,
                                 const double* t0_dev, double t_off, cudaStream_t s) {
  if (p1 <= p0) return cudaSuccess;
  auto launch = mx == 8    ? deform_launch<real, 8>
                : mx == 16 ? deform_launch<real, 16>
                : mx == 32 ? deform_launch<real, 32>
                           : nullptr;
  if (!launch) return cudaErrorInvalidValue;
  launch(p0, p1, coef, corners, umetric, kc, T, rot, t_half, t0_dev, t_off, s);
  ++launch_counter();
  return cudaGetLastError();
}

template <typename real>
cudaError_t launch_sphere_metrics(const PatchMeta* meta, int npatch, int mx, const double* omega,
                                  double* metric, real* umetric, const RemapEntry* rm,
                                  const double* old_metric, const real* old_umetric, double* coef,
                                  bool corners, cudaStream_t s) {
  if (npatch <= 0) return cudaSuccess;
  const int SN = mx + 2 * kMbc + 1;
  const size_t smem = sizeof(double) * 3 * (size_t)SN * SN;
  // set once per process; concurrent first calls both set it (idempotent)
  static std::atomic<bool> attr_set{false};
  if (!attr_set.load(std::memory_order_acquire)) {
    cudaError_t e = cudaFuncSetAttribute(metrics_kernel<real>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024);
    if (e != cudaSuccess) return e;
    attr_set.store(true, std::memory_order_release);
  }
  if (smem > 64 * 1024) return cudaErrorInvalidValue;
  const int grid = npatch < 65535 * 8 ? npatch : 65535 * 8;
  metrics_kernel<real><<<grid, 256, smem, s>>>(meta, npatch, mx, omega[0], omega[1], omega[2],
                                               metric, umetric, rm, old_metric, old_umetric, coef,
                                               corners);
  ++launch_counter();
  return cudaGetLastError();
}

#define FC_INSTANTIATE(real)                                                                     \
  template cudaError_t launch_deform_fluxes<real>(int, int, int, const double*, bool, real*,     \
                                                  double, double, double, double, const double*, \
                                                  double, cudaStream_t);                         \
  template cudaError_t launch_sphere_metrics<real>(const PatchMeta*, int, int, const double*,    \
                                                   double*, real*, const RemapEntry*,            \
                                                   const double*, const real*, double*, bool,    \
                                                   cudaStream_t);

FC_INSTANTIATE(float)
FC_INSTANTIATE(double)

}  // namespace fc
