// The wave-propagation patch update, "band" variant (sm_103a).
//
// One CTA per patch, as in the staged variant, so that a launch of few
// patches still takes about one patch's latency; inside the CTA the update
// is the walk variant's row walk, divided among the warps.  Warp segment b
// (MX lanes) owns the band of R rows [bR, (b+1)R): lane li owns column li and
// walks the band's rows, keeping a four-row register window of its column,
// taking the neighbouring column's edge results by warp shuffles and writing
// each finished row of cells straight to HBM.  A band also computes the
// x-edges of the row below it and of the row above it, which the transverse
// increments of its first and last y-edge read: R + 2 rows of x-edges and
// R + 1 rows of y-edges per band.  The staged variant instead passes over
// every edge in shared memory, with a CTA barrier between phases.
//
// Before the walk, the CTA fills the tile's ghost ring (Alg. 1: the
// neighbour reads are made while the tile's TMA copy is in flight). It then
// computes what every band reads at the patch's sides: for each row, the
// x = MX edge (normal flux, speed, and the fluctuation into the last
// column); and the fluctuations of the y-edges of ghost columns -1 and MX.
// Then the bands run with no further CTA barrier.
//
// Refluxing: the final fluxes through the patch's faces are recorded as the
// staged variant does.
#include <atomic>
#include <cstdint>

#include "ghost_ring.cuh"
#include "walk_edge.cuh"

namespace fc {
namespace {

// threads of a CTA: one per column of each band, and one for each task of the
// ghost ring and each entry of the tables (64 patches of 16^2, FP64, a global
// step: 10.1 us with a thread per ghost cell, 9.0 us so)
template <typename real, int MX, int R>
constexpr int band_threads() {
  constexpr int ring = ring_threads<MX>(), tab = 4 * (MX + 3);
  constexpr int most = ((ring > tab ? ring : tab) + 31) / 32 * 32;
  return MX * MX / R > most ? MX * MX / R : most;
}

// resident CTAs the register budget is sized for: as many whole CTAs as 1024
// FP32 / 512 FP64 threads hold (FP32 mx = 32: 4 of 256 threads, at most 64
// registers a thread; FP64 in bands of 8 rows: 2 of 192, at most 168, 141 used)
template <typename real, int MX, int R>
constexpr int band_min_blocks() {
  return (sizeof(real) == 4 ? 1024 : 512) / band_threads<real, MX, R>() > 0
             ? (sizeof(real) == 4 ? 1024 : 512) / band_threads<real, MX, R>()
             : 1;
}

// CAP: the capacity form of the cubed sphere (Sec. 5.3) -- the patch's block
// of metrics in the field's precision (1/kappa, phi_x, phi_y, formed once
// from the FP64 ones) arrives in dynamic shared memory by a second bulk copy;
// edge speeds are the edge volume fluxes phi, the correction's 2 |c| is |c|
// (1/kappa_L + 1/kappa_R), a fluctuation sum and the update are divided by the
// area of the cell they enter.  The FP64 block itself, converted and divided
// by where it was read, was 31.7 KB a 32^2 patch (15.8 KB in FP32) and bound
// the FP32 update: a coarse step of 1806 patches (levels 1-7) 2.30 -> 1.66 ms.
template <typename real, int MX, int R, bool SWIRL, bool CAP, bool FULL>
__global__ void __launch_bounds__(band_threads<real, MX, R>(), band_min_blocks<real, MX, R>())
    advance_band_kernel(DevForest<real> D, int p0, int p1, AdvArgs a, AdvConst<real> ac,
                        int* err) {
  constexpr int S = MX + 4;
  constexpr int MS = CAP ? umetric_stride(S) : 0;
  constexpr uint32_t mbytes = sizeof(real) * MS;
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  const real* Ms = reinterpret_cast<const real*>(dyn_smem);  // CAP: 1/kappa, phi_x, phi_y
  constexpr int NT = band_threads<real, MX, R>();
  constexpr int NW = MX * MX / R;  // threads that walk a band
  constexpr int NV = MX + 3;  // corner nodes -1..MX+1 of a row or column
  constexpr int NG = num_ghosts<MX>();
  constexpr unsigned kAll = 0xffffffffu;
  constexpr uint32_t bytes = sizeof(real) * S * S;
  static_assert(NT >= 4 * NV && NT >= ring_threads<MX>(), "a thread per table entry and task");
  static_assert(MX % R == 0 && NW % 32 == 0 && NT % 32 == 0, "bands of R rows, whole warps");
  __shared__ __align__(128) real Q[S * S];
  __shared__ __align__(8) uint64_t bar;
  __shared__ real ucoef_s;
  // ghost values gathered while the tile loads: the whole ring, or the cells
  // beyond coarse patches' interiors (ghost_ring.cuh)
  __shared__ real ring[CAP ? NG : 24];
  __shared__ bool ring_w[CAP ? NG : 1];
  // streamfunction tables over corner nodes k = 0..MX+2 (index k - 1):
  // Sx = sin^2(pi x_node), Tx = sin(pi (x_{c} + x_{c+1})) of column c = k - 1
  __shared__ real Sx[NV], Sy[NV], Tx[NV], Ty[NV];
  // the patch's sides: x-edge MX of rows -1..MX at [r + 1] (final-flux
  // inputs: normal flux, speed; fluctuation into cell MX - 1), and the
  // y-edges of ghost columns -1 / MX at rows 0..MX (fluctuations up / down)
  __shared__ real FeN[MX + 2], FeU[MX + 2], XMe[MX + 2];
  __shared__ real YPm[MX + 1], YMm[MX + 1], YPp[MX + 1], YMp[MX + 1];
  // FP64: the jumps of x-edges -1 and MX of rows -1..MX (between them a lane
  // takes the neighbouring lanes' instead of another subtraction: a coarse step
  // of the swirl forest 605 -> 591 us)
  constexpr bool kLaneJump = sizeof(real) == 8;
  __shared__ real WL[kLaneJump ? MX + 2 : 1], WR[kLaneJump ? MX + 2 : 1];

  const int tid = threadIdx.x;
  const int li = tid % MX;  // column of this lane
  const int r0 = (tid / MX) * R;  // first row of this lane's band
  // thread 0 initialises the copy barrier, issues the copies and waits for
  // them; the other threads touch the barrier only after a CTA barrier
  if (tid == 0) mbar_init(&bar, 1);
  const real cu = ac.cu, cv = ac.cv, h = ac.h;
  const Scheme<real, FULL> sc = make_scheme<real, FULL>(D.order, D.limiter, D.transverse);
  const real hdt = ac.hdt, bfac = ac.bfac;
  const real* tab = static_cast<const real*>(a.trig);  // the level's streamfunction factors
  auto q = [&](int i, int j) -> real { return Q[(j + kMbc) * S + (i + kMbc)]; };
  // capacity form: 1/kappa of cell (i, j), volume flux of x-edge (i, j) /
  // y-edge (i, j) times dt / 2
  auto ik = [&](int i, int j) -> real { return Ms[(j + kMbc) * S + i + kMbc]; };
  auto phx = [&](int i, int j) -> real {
    return hdt * Ms[S * S + (j + kMbc) * (S + 1) + i + kMbc];
  };
  auto phy = [&](int i, int j) -> real {
    return hdt * Ms[S * S + S * (S + 1) + (j + kMbc) * S + i + kMbc];
  };

  uint32_t parity = 0;
  for (int p = p0 + blockIdx.x; p < p1; p += gridDim.x, parity ^= 1) {
    const PatchMeta pm = D.meta[p];
    // (the launch's level: the copy does not wait for the patch's record)
    const real* src = D.buf[D.cur[a.level]] + (size_t)p * S * S;
    real* dst = D.buf[D.cur[a.level] ^ 1] + (size_t)p * S * S;
    if (tid == 0) {
      fence_proxy_async();
      mbar_expect_tx(&bar, bytes + mbytes);
      bulk_load(Q, src, bytes, &bar);
      if (CAP) bulk_load(dyn_smem, D.umetric + (size_t)p * MS, mbytes, &bar);
    }
    // the swirl coefficient, by the last thread (it gathers at most one
    // ghost); read after the barrier below
    if (SWIRL && tid == NT - 1 && p == p0 + (int)blockIdx.x) {
      const double t = a.t0_dev ? *a.t0_dev + a.t_off : a.t_half;
      ucoef_s = cospi_ratio<real>(t, a.period) * real(a.sfac * 0.5 * a.nu);
    }
    // the tables, one entry a thread: read (FP64) or computed (FP32: cheaper
    // than the read by 1%) now, stored after the gather, whose reads are not
    // to wait for this one's
    real tv = real(0);
    const int tk = NT - 1 - tid;  // (the first threads start the gather's longest reads)
    if (SWIRL && tk < 4 * NV) {
      const int tb = tk / NV, c = tk % NV;
      const int z = (tb & 1 ? pm.y : pm.x) * MX + c - 1;
      if (sizeof(real) == 8 && tab) {
        tv = tab[(tb < 2 ? 0 : a.trig_len) + z + 1];
      } else if (tb < 2) {
        tv = sinpi_r(real(z) * h);
        tv *= tv;
      } else {
        tv = sinpi_r(real(2 * z + 1) * h);
      }
    }
    // each gathering thread reads its region's entry from the table itself: no
    // staging pass, no barrier before the gather
    RingPart<real> part;
    const bool each = CAP && (pm.flags & 2);  // ghost by ghost: a neighbour's axes are turned
    if (a.gather) {
      if (each)
        gather_ring<real, MX>(
            D, [&](int r) { return D.nbr[(size_t)p * 8 + r]; }, p, pm, a.tlevel, ac.alpha,
            a.direct != 0, ring, ring_w, tid, NT, static_cast<real*>(a.keep_t), a.keep_t_p0);
      else
        part = ring_read<real, MX, CAP>(D, p, pm, a.level, a.tlevel, ac.alpha, a.direct != 0, ring,
                                   tid, static_cast<real*>(a.keep_t), a.keep_t_p0);
    }
    if (SWIRL && tk < 4 * NV) {
      const int tb = tk / NV, c = tk % NV;
      (tb == 0 ? Sx : tb == 1 ? Sy : tb == 2 ? Tx : Ty)[c] = tv;
    }
    // thread 0 observes the copy's completion (bounded), the others after the
    // barrier (at once); the CTA leaves together if it gave up
    const bool landed = tid == 0 ? mbar_wait(&bar, parity, a.wait_limit) : true;
    if (!__syncthreads_and(landed)) {
      if (tid == 0) atomicOr(err, kErrTimeout);
      mbar_wait(&bar, parity, kWaitLimit);  // let the copy land before leaving
      return;
    }
    if (tid != 0) mbar_wait(&bar, parity, kWaitLimit);
    if (a.gather) {
      if (each)
        store_ring<real, MX>(Q, ring, ring_w, tid, NT);
      else
        ring_store<real, MX, CAP>(D, part, a.level, a.tlevel, ac.alpha, a.direct != 0, Q, ring, tid,
                             static_cast<real*>(a.keep_t), a.keep_t_p0, p);
      __syncthreads();
      // (uniform over the CTA: does the patch touch a wall?)
      const int last_q = (1 << a.level) - 1;
      if (D.domain == FC_DOMAIN_WALLS &&
          (pm.x == 0 || pm.y == 0 || pm.x == last_q || pm.y == last_q)) {
        wall_bc<real, MX>(pm, Q, tid, NT);
        __syncthreads();
      }
      if (each) {  // corners beyond a cube vertex
        corner3_fill_k<real, MX>([&](int r) { return D.nbr[(size_t)p * 8 + r].kind; }, Q, tid,
                                 NT);
        __syncthreads();
      }
    }
    if (a.keep) {  // the adjoint's replay keeps the ghost-filled input tile
      real* kp = static_cast<real*>(a.keep) + (size_t)(p - a.keep_p0) * S * S;
      for (int k = tid; k < S * S; k += NT) kp[k] = Q[k];
    }
    const real ucoef = SWIRL ? ucoef_s : real(0);
    // the sides: x-edge MX of rows -1..MX, y-edges of ghost columns -1 and
    // MX at rows 0..MX (one edge a thread)
    for (int k = tid; k < (kLaneJump ? 4 * MX + 6 : 3 * MX + 4); k += NT) {
      real Fn, nP, M;
      if (kLaneJump && k >= 3 * MX + 4) {
        const int r = k - (3 * MX + 4) - 1;
        WL[r + 1] = q(-1, r) - q(-2, r);
      } else if (k < MX + 2) {
        const int r = k - 1;
        const real c = CAP ? phx(MX, r) : SWIRL ? (ucoef * Sx[MX + 1]) * Ty[r + 1] : cu;
        const real kf = CAP ? corr_factor_cap(c, ik(MX - 1, r) + ik(MX, r), sc) : corr_factor(c, sc);
        edge(c, q(MX - 2, r), q(MX - 1, r), q(MX, r), q(MX + 1, r), kf, sc, Fn, nP, M);
        FeN[k] = Fn;
        FeU[k] = c;
        XMe[k] = M;
        if (kLaneJump) WR[k] = q(MX, r) - q(MX - 1, r);
      } else {
        const bool right = k >= 2 * MX + 3;
        const int r = k - (right ? 2 * MX + 3 : MX + 2);
        const int i = right ? MX : -1;
        const real c = CAP ? phy(i, r) : SWIRL ? (-ucoef * Tx[i + 1]) * Sy[r + 1] : cv;
        const real kf = CAP ? corr_factor_cap(c, ik(i, r - 1) + ik(i, r), sc) : corr_factor(c, sc);
        edge(c, q(i, r - 2), q(i, r - 1), q(i, r), q(i, r + 1), kf, sc, Fn, nP, M);
        (right ? YPp : YPm)[r] = nP;
        (right ? YMp : YMm)[r] = M;
      }
    }
    __syncthreads();
    // the band walk: iteration it works on row r = r0 - 1 + it; it computes
    // x-edge (li, r) and y-edge (li, r + 1), finishes the final fluxes of
    // row r and updates cell (li, r - 1)
    real* bf = a.bflux ? static_cast<real*>(a.bflux) + ((size_t)p * 2 + a.bslot) * 4 * MX
                       : nullptr;
    if (tid < NW) {  // (the warps beyond the bands only gathered ghosts)
      const real ux = SWIRL ? ucoef * Sx[li + 1] : real(0);   // times Ty of the row: x-edge
      const real vy = SWIRL ? -ucoef * Tx[li + 1] : real(0);  // times Sy of the row: y-edge
      real qa = q(li, r0 - 2), qb = q(li, r0 - 1), qc = q(li, r0), qd = 0;
      real Wa = qb - qa, Wb = qc - qb;  // jumps of y-edges (li, r), (li, r + 1)
      // turned fluctuation sums into cells (capacity form: over the cell's
      // area) and final fluxes carried from row to row
      real nX_prev = 0, Gn_cur = 0, v_cur = 0, nP_cur = 0, Gf_prev = 0, dF_prev = 0;
      // capacity form: 1/kappa of this column's cells in rows r-1, r
      real ik_prev = CAP ? ik(li, r0 - 2) : real(0), ik_cur = CAP ? ik(li, r0 - 1) : real(0);
#pragma unroll(R <= 8 ? R + 2 : 2)
      for (int it = 0; it < R + 2; ++it) {
        const int r = r0 - 1 + it;
        if (it <= R) qd = q(li, r + 2);
        const real Wc = qd - qc;  // jump of y-edge (li, r + 2)
        const real ik_next = CAP && it <= R ? ik(li, r + 1) : real(0);
        real ik_left = CAP ? __shfl_up_sync(kAll, ik_cur, 1, MX) : real(0);  // cell (li-1, r)
        if (CAP && li == 0) ik_left = ik(-1, r);
        // x-edge (li, r): cells (li-1, r) | (li, r)
        const real cx = CAP ? phx(li, r) : SWIRL ? ux * Ty[r + 1] : cu;
        real Fn_r, nP_r, XM_r;
        const real kf = CAP ? corr_factor_cap(cx, ik_left + ik_cur, sc) : corr_factor(cx, sc);
        if constexpr (kLaneJump) {
          const real ql = q(li - 1, r), W = qb - ql;
          const real Wl = __shfl_up_sync(kAll, W, 1, MX), Wr = __shfl_down_sync(kAll, W, 1, MX);
          edge_flux(cx, W,
                    upwind_left(cx) ? (li == 0 ? WL[r + 1] : Wl) : (li == MX - 1 ? WR[r + 1] : Wr),
                    ql, qb, kf, sc, Fn_r, nP_r, XM_r);
        } else {
          edge(cx, q(li - 2, r), q(li - 1, r), qb, q(li + 1, r), kf, sc, Fn_r, nP_r, XM_r);
        }
        real XMn = __shfl_down_sync(kAll, XM_r, 1, MX);
        if (li == MX - 1) XMn = XMe[r + 1];
        const real nX_r = CAP ? (nP_r - XMn) * ik_cur : nP_r - XMn;  // into cell (li, r)
        // y-edge (li, r+1): cells (li, r) | (li, r+1); the last row's is the
        // next band's
        real Gn_n = 0, nP_n = 0, YM_n = 0, v_n = 0;
        if (it <= R) {
          v_n = CAP ? phy(li, r + 1) : SWIRL ? vy * Sy[r + 2] : cv;
          edge_flux(v_n, Wb, upwind_left(v_n) ? Wa : Wc, qb, qc,
                    CAP ? corr_factor_cap(v_n, ik_cur + ik_next, sc) : corr_factor(v_n, sc), sc,
                    Gn_n, nP_n, YM_n);
        }
        // final flux at y-edge (li, r)
        real Gf_r = 0;
        if (it >= 1) {
          Gf_r = final_flux(v_cur, nX_prev, nX_r, Gn_cur, sc);
          if (bf && r == 0) bf[2 * MX + li] = Gf_r * bfac;
          if (bf && r == MX) bf[3 * MX + li] = Gf_r * bfac;
        }
        // final fluxes at x-edges (li, r) and (li+1, r), rows of the band
        real dF_r = 0;
        if (it >= 1 && it <= R) {
          // turned y-fluctuation sum into cell (li, r)
          const real nY_r = CAP ? (nP_cur - YM_n) * ik_cur : nP_cur - YM_n;
          real nYl = __shfl_up_sync(kAll, nY_r, 1, MX);
          if (li == 0) nYl = CAP ? (YPm[r] - YMm[r + 1]) * ik_left : YPm[r] - YMm[r + 1];
          const real Ff = final_flux(cx, nYl, nY_r, Fn_r, sc);
          real Fr = __shfl_down_sync(kAll, Ff, 1, MX);
          if (li == MX - 1) {
            const real nYr = CAP ? (YPp[r] - YMp[r + 1]) * ik(MX, r) : YPp[r] - YMp[r + 1];
            Fr = final_flux(FeU[r + 1], nY_r, nYr, FeN[r + 1], sc);
          }
          dF_r = Fr - Ff;
          if (bf && li == 0) bf[r] = Ff * bfac;
          if (bf && li == MX - 1) bf[MX + r] = Fr * bfac;
        }
        // conservative update of cell (li, r-1)
        if (it >= 2) {
          const real d = dF_prev + (Gf_r - Gf_prev);
          dst[(r + 1) * S + (li + kMbc)] = fma(real(-2), CAP ? d * ik_prev : d, qa);
        }
        nX_prev = nX_r;
        Gn_cur = Gn_n;
        v_cur = v_n;
        nP_cur = nP_n;
        Gf_prev = Gf_r;
        dF_prev = dF_r;
        qa = qb;
        qb = qc;
        qc = qd;
        Wa = Wb;
        Wb = Wc;
        ik_prev = ik_cur;
        ik_cur = ik_next;
      }
    }
    __syncthreads();  // the next patch's copy overwrites the tile
  }
}

template <typename real, int MX, int R, bool SWIRL, bool CAP, bool FULL>
cudaError_t band_launch_t(const DevForest<real>& D, int p0, int p1, const AdvArgs& a, int* err,
                          cudaStream_t s) {
  constexpr size_t dyn = CAP ? sizeof(real) * (size_t)umetric_stride(MX + 4) : 0;
  auto kern = advance_band_kernel<real, MX, R, SWIRL, CAP, FULL>;
  if (CAP) {  // set once per process; concurrent first calls both set it (idempotent)
    static std::atomic<bool> attr_set{false};
    if (!attr_set.load(std::memory_order_acquire)) {
      cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)dyn);
      if (e != cudaSuccess) return e;
      attr_set.store(true, std::memory_order_release);
    }
  }
  kern<<<p1 - p0, band_threads<real, MX, R>(), dyn, s>>>(D, p0, p1, a, adv_const(D, a), err);
  ++launch_counter();
  return cudaGetLastError();
}

template <typename real, int MX, int R, bool FULL>
cudaError_t band_launch_f(const DevForest<real>& D, int p0, int p1, const AdvArgs& a, int* err,
                        cudaStream_t s) {
  if (D.metric) return band_launch_t<real, MX, R, false, true, FULL>(D, p0, p1, a, err, s);
  if (D.vel_kind == FC_VEL_SWIRL)
    return band_launch_t<real, MX, R, true, false, FULL>(D, p0, p1, a, err, s);
  return band_launch_t<real, MX, R, false, false, FULL>(D, p0, p1, a, err, s);
}

template <typename real, int MX, int R>
cudaError_t band_launch(const DevForest<real>& D, int p0, int p1, const AdvArgs& a, int* err,
                        cudaStream_t s) {
  return full_scheme(D.order, D.limiter, D.transverse)
             ? band_launch_f<real, MX, R, true>(D, p0, p1, a, err, s)
             : band_launch_f<real, MX, R, false>(D, p0, p1, a, err, s);
}

}  // namespace

// rows per band from the requested warps per CTA: a.warps x 32 threads, at
// most one lane per interior cell
template <typename real>
cudaError_t launch_advance_band(const DevForest<real>& D, int p0, int p1, const AdvArgs& a,
                                int* err, cudaStream_t s) {
  switch (D.mx) {
    case 8: return band_launch<real, 8, 1>(D, p0, p1, a, err, s);
    case 16:
      return a.warps <= 2 ? band_launch<real, 16, 4>(D, p0, p1, a, err, s)
             : a.warps == 4 ? band_launch<real, 16, 2>(D, p0, p1, a, err, s)
                            : band_launch<real, 16, 1>(D, p0, p1, a, err, s);
    case 32:
      return a.warps <= 4  ? band_launch<real, 32, 8>(D, p0, p1, a, err, s)
             : a.warps == 8 ? band_launch<real, 32, 4>(D, p0, p1, a, err, s)
                            : band_launch<real, 32, 2>(D, p0, p1, a, err, s);
    default: return cudaErrorInvalidValue;
  }
}

// (compiled once per precision, see build.py)
template cudaError_t launch_advance_band<FC_REAL>(const DevForest<FC_REAL>&, int, int,
                                                  const AdvArgs&, int*, cudaStream_t);

}  // namespace fc
