// The ghost ring of one patch by a CTA, side by side: the band update's
// gather for patches whose neighbours keep orientation (every patch of a
// square domain; on the cubed sphere those away from the cube's edges, the
// others take the ring ghost by ghost).
//
// A launch of a few hundred patches waits for each patch's chain of dependent
// reads and instructions, not for bandwidth.  Ghost by ghost, with each
// ghost's own entry and transform, the kinds of a warp's ghosts ran one after
// another; here a group of MX threads takes one face, whose ghosts share their
// entry and rule, so a warp runs one or two kinds; a coarser neighbour's cells
// beside the face are read once for their four ghosts, and the few cells an
// interpolation needs beyond the coarse patch's interior are found by threads
// of their own at the same time.  Measured (one GB300): the update of 248
// patches of 32^2 in FP32 10.4 -> 7.2 us, a coarse step of the swirl forest
// (496 patches, 16 finest substeps one after another) 0.124 -> 0.104 ms; on
// the sphere (1806 patches, levels 1-7) 1.66 -> 1.21 ms.
//
// Threads: [0, 4 MX) ghosts (or coarse cells) of the faces; [4 MX, 4 MX + 16)
// corner ghosts; from the next whole warp on 24 cells beyond coarse interiors:
// [side] past the end of a coarse face neighbour's half that the face covers,
// [4 + 5 corner + m] the five stencil cells of a coarse corner neighbour.
#pragma once

#include "ghost_gather.cuh"

namespace fc {

template <int MX>
__host__ __device__ constexpr int ring_cells_from() {
  return (4 * MX + 16 + 31) / 32 * 32;
}
template <int MX>
__host__ __device__ constexpr int ring_threads() {
  return ring_cells_from<MX>() + 24;
}

// what a thread carries from its reads to its stores (across the wait for
// the patch's own tile)
template <typename real>
struct RingPart {
  int kind;             // of its region's neighbour; 0: nothing to store
  real v0, v1, v2, v3;  // two ghosts, or the coarse cell, its neighbours in, lo, hi
  real v4;              // coarse, mapped grid: the cell towards the owner
  int t, n0;            // coarse: index along the face, patch
  bool own;             // coarse: the cell towards the owner is the owner's average
};

// Eq. ghost_coarse of four cells, the first at offset o of patch n (mapped
// grid: weighted by their areas)
template <bool CAP, typename real>
__device__ __forceinline__ real ring_average(const DevForest<real>& D, int n, int o, real s0,
                                             real s1, real s2, real s3) {
  if (!CAP) return real(0.25) * (((s0 + s1) + s2) + s3);
  const double* K = D.metric + (size_t)n * D.S * D.S + o;
  const double k0 = K[0], k1 = K[1], k2 = K[D.S], k3 = K[D.S + 1];
  return real((((k0 * double(s0) + k1 * double(s1)) + k2 * double(s2)) + k3 * double(s3)) /
              (((k0 + k1) + k2) + k3));
}

// interior cell at offset o of a patch at qo / qn (older / newer state) of
// the level read at weight alpha (0 and 1: one state alone, see src_interior)
template <typename real>
__device__ __forceinline__ real ring_time(const real* qo, const real* qn, real alpha, bool one,
                                          int o) {
  const real v = (alpha == real(1) ? qn : qo)[o];
  return one ? v : (real(1) - alpha) * v + alpha * qn[o];
}

// The reads of patch p (level L), before its tile is needed.  direct: a
// coarser neighbour is read as its fill would leave it at tlevel = L - 1 and
// alpha (interpolate_direct_entry), else from its filled tile (D.qT at
// tlevel, else the store).  cells: 24 values in shared memory.  keep_t: the
// cells an interpolation reads are also stored in the kept coarse tiles.
template <typename real, int MX, bool CAP>
__device__ __forceinline__ RingPart<real> ring_read(const DevForest<real>& D, int p,
                                                    const PatchMeta& pm, int L, int tlevel,
                                                    real alpha, bool direct, real* cells, int tid,
                                                    real* keep_t, int keep_t_p0) {
  constexpr int S = MX + 4, SS = S * S;
  RingPart<real> w;
  w.kind = 0;
  const bool one = alpha == real(0) || alpha == real(1);
  const NbrEntry* E = D.nbr + (size_t)p * 8;
  if (tid < 4 * MX) {
    const int f = tid / MX, li = tid % MX;
    const NbrEntry e = E[f];
    const bool X = f < 2, low = (f & 1) == 0;
    const int sn = X ? 1 : S, st = X ? S : 1;  // strides across and along the face
    if (e.kind == NB_SAME) {
      w.kind = NB_SAME;
      const real* c = D.buf[D.cur[L]] + (size_t)e.n0 * SS + (li + kMbc) * st + (low ? MX : 2) * sn;
      w.v0 = c[0];
      w.v1 = c[sn];
    } else if (e.kind == NB_FINE) {
      // n0 holds the face's lower half, n1 the upper; a ghost's four cells are
      // summed in the order (0,0), (1,0), (0,1), (1,1)
      w.kind = NB_SAME;
      const int half = li >= MX / 2 ? 1 : 0;
      const int n = half ? e.n1 : e.n0;
      const int o = (2 * li - half * MX + kMbc) * st + (low ? MX - 2 : 2) * sn;
      const real* c = D.buf[D.cur[L + 1]] + (size_t)n * SS + o;
      real u[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) u[k] = c[(k >> 2) * 2 * sn + (k & 1) + ((k >> 1) & 1) * S];
      w.v0 = ring_average<CAP>(D, n, o, u[0], u[1], u[2], u[3]);
      w.v1 = ring_average<CAP>(D, n, o + 2 * sn, u[4], u[5], u[6], u[7]);
    } else if (e.kind == NB_COARSE && li < MX / 2) {
      w.kind = NB_COARSE;
      const int t0 = X ? ((pm.y * MX + e.fy) >> 1) - e.y0 * MX
                       : ((pm.x * MX + e.fx) >> 1) - e.x0 * MX;
      const int t = t0 + li;
      const int o = (t + kMbc) * st + ((low ? MX - 1 : 0) + kMbc) * sn;
      const int ol = t > 0 ? o - st : o, oh = t < MX - 1 ? o + st : o;  // (inside the patch)
      const int d = low ? -sn : sn;
      w.t = t;
      w.n0 = e.n0;
      w.own = direct && (e.code[0] & kSrcComplete);
      const int c = D.cur[L - 1];
      if (direct) {
        const real* qo = D.buf[c ^ 1] + (size_t)e.n0 * SS;
        const real* qn = D.buf[c] + (size_t)e.n0 * SS;
        w.v0 = ring_time(qo, qn, alpha, one, o);
        w.v1 = ring_time(qo, qn, alpha, one, o + d);
        w.v2 = ring_time(qo, qn, alpha, one, ol);
        w.v3 = ring_time(qo, qn, alpha, one, oh);
        if (CAP && w.own) {
          const int b = (2 * li + kMbc) * st + (low ? kMbc : MX) * sn;
          const real* u = D.buf[D.cur[L]] + (size_t)p * SS + b;
          w.v4 = ring_average<CAP>(D, p, b, u[0], u[1], u[S], u[S + 1]);
        }
      } else {
        const real* q = patch_ptr(tlevel == L - 1 ? D.qT : D.buf[c], e.n0, S);
        w.v0 = q[o];
        w.v1 = q[o + d];
        w.v2 = q[ol];
        w.v3 = q[oh];
      }
    }
  } else if (tid < 4 * MX + 16) {
    const int k = tid - 4 * MX, r = 4 + (k >> 2), x = k & 1, y = (k >> 1) & 1;
    const NbrEntry e = E[r];
    if (e.kind == NB_SAME) {
      w.kind = NB_SAME;
      w.v0 = D.buf[D.cur[L]][(size_t)e.n0 * SS + (((r & 2) ? 0 : MX - 2) + y + kMbc) * S +
                             ((r & 1) ? 0 : MX - 2) + x + kMbc];
    } else if (e.kind == NB_FINE) {
      w.kind = NB_SAME;
      const int o = (((r & 2) ? 0 : MX - 4) + 2 * y + kMbc) * S + ((r & 1) ? 0 : MX - 4) + 2 * x +
                    kMbc;
      const real* c = D.buf[D.cur[L + 1]] + (size_t)e.n0 * SS + o;
      w.v0 = ring_average<CAP>(D, e.n0, o, c[0], c[1], c[S], c[S + 1]);
    } else if (e.kind == NB_COARSE) {
      w.kind = NB_COARSE;
    }
  } else if (tid >= ring_cells_from<MX>() && tid < ring_threads<MX>()) {
    const int k = tid - ring_cells_from<MX>();
    const int r = k < 4 ? k : 4 + (k - 4) / 5;
    const NbrEntry e = E[r];
    if (e.kind == NB_COARSE) {
      // the region's first ghost, its coarse cell, and the cell wanted
      const int gi = (r == 1 || (r >= 4 && (r & 1))) ? MX : (r == 0 || r >= 4) ? -2 : 0;
      const int gj = (r == 3 || (r >= 4 && (r & 2))) ? MX : (r == 2 || r >= 4) ? -2 : 0;
      int ci = ((pm.x * MX + gi + e.fx) >> 1) - e.x0 * MX;
      int cj = ((pm.y * MX + gj + e.fy) >> 1) - e.y0 * MX;
      int ui = gi, uj = gj;  // the ghost group that reads the cell
      if (k < 4) {  // the face's half of the coarse patch starts at 0 or ends at its side
        if (r < 2) {
          if (cj > 0) uj = MX - 2;
          cj = cj > 0 ? MX : -1;
        } else {
          if (ci > 0) ui = MX - 2;
          ci = ci > 0 ? MX : -1;
        }
      } else {
        const int m = (k - 4) % 5;
        ci += m == 1 ? 1 : m == 2 ? -1 : 0;
        cj += m == 3 ? 1 : m == 4 ? -1 : 0;
      }
      const int at = (cj + kMbc) * S + ci + kMbc;
      const int c = D.cur[L - 1];
      real v;
      if (direct) {
        const PatchMeta cm{e.lev, e.x0, e.y0, 0, 0, 0};
        v = coarse_cell_interior<real, MX>(D, cm, ci, cj)
                ? ring_time(D.buf[c ^ 1] + (size_t)e.n0 * SS, D.buf[c] + (size_t)e.n0 * SS, alpha,
                            one, (cj + kMbc) * S + ci + kMbc)
                : coarse_ghost_at<real, MX>(D, e, cm, p, tlevel, alpha, ui, uj, ci, cj);
        if (keep_t) keep_t[(size_t)(e.n0 - keep_t_p0) * SS + at] = v;  // (unclamped place)
      } else {
        v = patch_ptr(tlevel == L - 1 ? D.qT : D.buf[c], e.n0, S)[at];
      }
      cells[k] = v;
    }
  }
  return w;
}

// The stores into the landed tile T (cells and T's interior visible to all).
template <typename real, int MX, bool CAP>
__device__ __forceinline__ void ring_store(const DevForest<real>& D, const RingPart<real>& w,
                                           int L, int tlevel, real alpha, bool direct, real* T,
                                           const real* cells, int tid, real* keep_t,
                                           int keep_t_p0, int p) {
  constexpr int S = MX + 4, SS = S * S;
  if (w.kind == 0) return;
  if (tid >= 4 * MX) {  // a corner ghost
    const int k = tid - 4 * MX, r = 4 + (k >> 2), x = k & 1, y = (k >> 1) & 1;
    real v = w.v0;
    if (w.kind == NB_COARSE) {
      const real* c = cells + 4 + 5 * (r - 4);
      const real sx = minmod(c[1] - c[0], c[0] - c[2]), sy = minmod(c[3] - c[0], c[0] - c[4]);
      v = c[0] + real(0.25) * ((x ? sx : -sx) + (y ? sy : -sy));
    }
    T[(((r & 2) ? MX : -2) + y + kMbc) * S + ((r & 1) ? MX : -2) + x + kMbc] = v;
    return;
  }
  const int f = tid / MX, li = tid % MX;
  const bool X = f < 2, low = (f & 1) == 0;
  const int sn = X ? 1 : S, st = X ? S : 1;
  real* g = T + (low ? 0 : MX + 2) * sn + kMbc * st;
  if (w.kind == NB_SAME) {
    g[li * st] = w.v0;
    g[li * st + sn] = w.v1;
    return;
  }
  const int t = w.t;
  const real q0 = w.v0, in = w.v1;
  const real lo = t == 0 ? cells[f] : w.v2, hi = t == MX - 1 ? cells[f] : w.v3;
  real out;
  if (CAP && w.own) {
    out = w.v4;
  } else if (w.own) {  // towards the owner: the average of its own cells
    const real* u = T + (2 * li + kMbc) * st + (low ? kMbc : MX) * sn;
    out = real(0.25) * (((u[0] + u[1]) + u[S]) + u[S + 1]);
  } else if (direct) {
    const NbrEntry e = D.nbr[(size_t)p * 8 + f];
    const PatchMeta cm{e.lev, e.x0, e.y0, 0, 0, 0};
    const int n = low ? MX : -1;
    out = coarse_ghost<real, MX>(D, cm, w.n0, tlevel, alpha, X ? n : t, X ? t : n);
  } else {
    out = patch_ptr(tlevel == L - 1 ? D.qT : D.buf[D.cur[L - 1]], w.n0,
                    S)[(t + kMbc) * st + ((low ? MX : -1) + kMbc) * sn];
  }
  if (keep_t && direct) {
    real* K = keep_t + (size_t)(w.n0 - keep_t_p0) * SS + (t + kMbc) * st +
              ((low ? MX - 1 : 0) + kMbc) * sn;
    const int d = low ? -sn : sn;
    K[0] = q0;
    K[d] = in;
    K[-d] = out;
    K[-st] = lo;
    K[st] = hi;
  }
  // slopes towards higher index, across the face and along it
  const real sc = low ? minmod(out - q0, q0 - in) : minmod(in - q0, q0 - out);
  const real sl = minmod(hi - q0, q0 - lo);
  const real sx = X ? sc : sl, sy = X ? sl : sc;
  real* u = g + 2 * li * st;
#pragma unroll
  for (int k = 0; k < 4; ++k)
    u[(k & 1) + (k >> 1) * S] =
        q0 + real(0.25) * (((k & 1) ? sx : -sx) + ((k >> 1) ? sy : -sy));
}

}  // namespace fc
