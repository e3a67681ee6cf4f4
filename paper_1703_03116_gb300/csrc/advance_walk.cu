// The wave-propagation patch update, "walk" variant (sm_103a), for launches
// that fill the GPU: what bounds them is the instructions a cell takes, not
// memory (9 bytes a cell move in FP32 at mx = 32, 1/5 of what HBM could).
//
//  * A lane owns an interior column and walks up the rows with a register
//    window; per row it computes its x-edge (left edge of its cell) and the
//    y-edge above; the neighbouring column's results arrive by warp shuffles.
//  * In FP32 a lane works on two cells at once in packed registers
//    (walk_edge.cuh): at mx = 32 rows r and r + 16 of one patch (a warp), at
//    mx = 16 and 8 the same row of two patches (four and eight a warp).  FP64
//    is bound by its pipe and takes one.
//  * What a patch's ghosts come from is the same along a face, so the ghost
//    ring is filled face by face without divergence; from a coarser
//    neighbour each of the mx/2 coarse cells beside the face is computed
//    once for its four ghosts, from the states before and after that level's
//    step, so that no fill kernel runs before the update.  (Ghost by ghost,
//    with each ghost's own neighbour entry and index transform, the ring took
//    as many instructions as the update itself.)
//  * The x-edge and the two y-edge columns outside the lanes (x-edge MX,
//    ghost columns -1 and MX) are 3 MX + 4 independent edges spread over the
//    lanes before the walk.
//  * Tile and neighbour entries arrive by 1D bulk copies; one buffer a warp
//    and as many warps as fit hide the copies and the gathers' reads.  The
//    streamfunction's factors come from a table per level.
//
// Measured on one GB300 against the form before it (ghost by ghost after a
// fill launch, one cell a lane, two tile buffers a warp), a coarse step with
// its field moves: 256 forests (67168 patches of 32^2, FP32) 6.0 -> 2.6 ms,
// 64 forests (13852 patches of 16^2, FP64) 3.7 -> 2.0 ms; 16384 patches of
// 32^2 at one level 94 -> 67 us.  About 3500 warp instructions a 32^2 patch
// (of 6200), at 58% of the issue slots with 24 warps an SM; its sides are one
// loop over strides because as four copies of the code they overflowed the
// instruction cache (4.1 against 2.7 ms).
//
// The entries of a square domain's layout keep orientation (a = 0: only the
// cubed sphere turns axes, and its capacity form runs band or staged).
#include <atomic>
#include <cstdint>

#include "ghost_gather.cuh"
#include "walk_edge.cuh"

namespace fc {
namespace {

template <typename real>
struct Vec2;
template <>
struct Vec2<float> {
  using T = float2;
};
template <>
struct Vec2<double> {
  using T = double2;
};
// x-edge MX of a row: fluctuation M into cell MX - 1 and the final flux as
// A + B nY, nY the turned y-fluctuation sum of cell MX - 1; W: the edge's jump
template <typename real>
struct alignas(16) EdgeRec {
  real M, A, B, W;
};

// Shared memory of one patch: its tile, its eight neighbour entries, and per
// row the streamfunction's factors and the edges beside the lanes.  The
// stride between patches of a warp is MX modulo 32 elements, so that the
// segments of a warp read different banks.
template <typename real, int MX>
struct Slot {
  static constexpr int S = MX + 4;
  static constexpr int tile = 0;
  static constexpr int nbr = tile + (int)sizeof(real) * S * S;
  static constexpr int rows = nbr + 8 * (int)sizeof(NbrEntry);       // real2 (MX + 2 rows -1..MX)
  static constexpr int rec = (rows + 2 * (int)sizeof(real) * (MX + 2) + 15) & ~15;
  static constexpr int yl = rec + (int)sizeof(EdgeRec<real>) * (MX + 2);  // rows -1..MX at [r + 1]
  static constexpr int ye = yl + (int)sizeof(real) * (MX + 2);       // P, M of columns -1, MX
  static constexpr int wl = ye;  // (then, FP64: jumps of x-edge -1 at rows -1..MX)
  static constexpr int end = ye + (int)sizeof(real) * 4 * (MX + 1);
  // bytes, congruent to MX elements modulo 32 elements, a multiple of 16
  static constexpr int row = 32 * (int)sizeof(real);
  static constexpr int bytes = (end - MX * (int)sizeof(real) + row - 1) / row * row +
                               MX * (int)sizeof(real);
};

// interior cell (i, j) of a patch of the interpolated level at weight alpha
template <typename real, int MX>
__device__ __forceinline__ real coarse_interior(const real* qo, const real* qn, real alpha, int i,
                                                int j) {
  const int o = (j + kMbc) * (MX + 4) + i + kMbc;
  // (0: the newer state may still be written beside this kernel; 1: a step
  // of all levels at one time has no older state)
  if (alpha == real(0)) return qo[o];
  if (alpha == real(1)) return qn[o];
  return (real(1) - alpha) * qo[o] + alpha * qn[o];
}

// A patch's ghost ring, by the MX lanes (li) of its segment, in two parts
// with a warp barrier between them.  Sides and corners are told apart by
// strides, not by code: the walk's instructions and these share a cache.
//
// Part 1: ghosts from same-size neighbours (every read issued before any is
// stored), and into `cells` what the interpolations need beyond the coarse
// patches' interiors: for each coarser face neighbour the coarse cell past
// the end of the face at [side], for each coarser corner neighbour the five
// cells of its stencil at [4 + 5 corner + m].  direct: a coarser neighbour on
// tlevel is read as its fill would leave it (interpolate_direct_entry), else
// from its filled tile.
template <typename real, int MX>
__device__ __forceinline__ void gather_part1(const DevForest<real>& D, const NbrEntry* E,
                                             const PatchMeta& pm, int p, int tlevel, real alpha,
                                             bool direct, bool mixed, real* T, real* cells,
                                             int li) {
  constexpr int S = MX + 4, SS = S * S;
  constexpr int NC = (16 + MX - 1) / MX;  // corner ghosts a lane
  real v0[4], v1[4], vc[NC];
#pragma unroll
  for (int f = 0; f < 4; ++f) {  // rows / columns mx - 2, mx - 1 or 0, 1 of the neighbour
    const int sn = f < 2 ? 1 : S, st = f < 2 ? S : 1;
    if (E[f].kind == NB_SAME) {
      const real* src = D.buf[D.cur[E[f].lev]] + (size_t)E[f].n0 * SS + (li + kMbc) * st +
                        ((f & 1) ? 2 : MX) * sn;
      v0[f] = src[0];
      v1[f] = src[sn];
    }
  }
#pragma unroll
  for (int u = 0; u < NC; ++u) {
    const int k = li + u * MX, r = 4 + (k >> 2);
    if (k < 16 && E[r].kind == NB_SAME) {
      const int i = ((r & 1) ? 0 : MX - 2) + (k & 1), j = ((r & 2) ? 0 : MX - 2) + ((k >> 1) & 1);
      vc[u] = D.buf[D.cur[E[r].lev]][(size_t)E[r].n0 * SS + (j + kMbc) * S + i + kMbc];
    }
  }
  if (mixed) {
#pragma unroll 1
    for (int k = li; k < 24; k += MX) {
      const int r = k < 4 ? k : 4 + (k - 4) / 5;
      const NbrEntry& e = E[r];
      if (e.kind != NB_COARSE) continue;
      // the first ghost of the region, its coarse cell, and the cell wanted
      const int gi = (r == 1 || (r >= 4 && (r & 1))) ? MX : (r == 0 || r >= 4) ? -2 : 0;
      const int gj = (r == 3 || (r >= 4 && (r & 2))) ? MX : (r == 2 || r >= 4) ? -2 : 0;
      int ci = ((pm.x * MX + gi + e.fx) >> 1) - e.x0 * MX;
      int cj = ((pm.y * MX + gj + e.fy) >> 1) - e.y0 * MX;
      int ui = gi, uj = gj;  // the ghost group that reads the cell
      if (k < 4) {  // the face's half of the coarse patch starts at 0 or ends at its side
        int& c = r < 2 ? cj : ci;
        int& u = r < 2 ? uj : ui;
        if (c > 0) u = MX - 2;
        c = c > 0 ? MX : -1;
      } else {
        const int m = (k - 4) % 5;
        ci += m == 1 ? 1 : m == 2 ? -1 : 0;
        cj += m == 3 ? 1 : m == 4 ? -1 : 0;
      }
      real v;
      if (direct && e.lev == tlevel) {
        const PatchMeta cm{e.lev, e.x0, e.y0, 0, 0, 0};
        if (coarse_cell_interior<real, MX>(D, cm, ci, cj)) {
          const int c = D.cur[tlevel];
          v = coarse_interior<real, MX>(D.buf[c ^ 1] + (size_t)e.n0 * SS,
                                        D.buf[c] + (size_t)e.n0 * SS, alpha, ci, cj);
        } else {
          v = coarse_ghost_at<real, MX>(D, e, cm, p, tlevel, alpha, ui, uj, ci, cj);
        }
      } else {
        v = patch_ptr(e.lev == tlevel ? D.qT : D.buf[D.cur[e.lev]], e.n0,
                      S)[(cj + kMbc) * S + ci + kMbc];
      }
      cells[k] = v;
    }
  }
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    const int sn = f < 2 ? 1 : S, st = f < 2 ? S : 1;
    if (E[f].kind == NB_SAME) {
      real* g = T + (li + kMbc) * st + ((f & 1) ? MX + 2 : 0) * sn;
      g[0] = v0[f];
      g[sn] = v1[f];
    }
  }
#pragma unroll
  for (int u = 0; u < NC; ++u) {
    const int k = li + u * MX, r = 4 + (k >> 2);
    if (k < 16 && E[r].kind == NB_SAME) {
      const int i = ((r & 1) ? MX : -2) + (k & 1), j = ((r & 2) ? MX : -2) + ((k >> 1) & 1);
      T[(j + kMbc) * S + i + kMbc] = vc[u];
    }
  }
}

// Eq. ghost_fine for the four fine cells of a coarse cell: (dx, dy) = (-+1, -+1)
template <typename real>
__device__ __forceinline__ real fine_value(real q0, real sx, real sy, int x, int y) {
  return q0 + real(0.25) * ((x ? sx : -sx) + (y ? sy : -sy));
}

// Part 2: ghosts from finer and coarser neighbours.
template <typename real, int MX>
__device__ __forceinline__ void gather_part2(const DevForest<real>& D, const NbrEntry* E,
                                             const PatchMeta& pm, int p, int tlevel, real alpha,
                                             bool direct, real* T, const real* cells, int li) {
  constexpr int S = MX + 4, SS = S * S;
#pragma unroll 1
  for (int f = 0; f < 4; ++f) {
    const NbrEntry& e = E[f];
    const bool X = f < 2, low = (f & 1) == 0;
    const int sn = X ? 1 : S, st = X ? S : 1;          // strides across and along the face
    real* g = T + (low ? 0 : MX + 2) * sn + kMbc * st;  // its first ghost, outer or inner
    if (e.kind == NB_FINE) {
      // n0 holds the face's lower half, n1 the upper; lane li takes ghosts li;
      // a ghost's four cells are summed in the order (0,0), (1,0), (0,1), (1,1)
      const int half = li >= MX / 2 ? 1 : 0;
      const real* c = D.buf[D.cur[e.lev]] + (size_t)(half ? e.n1 : e.n0) * SS +
                      (2 * li - half * MX + kMbc) * st + (low ? MX - 2 : 2) * sn;
      real w[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) w[k] = c[(k >> 2) * 2 * sn + (k & 1) + ((k >> 1) & 1) * S];
      g[li * st] = real(0.25) * (((w[0] + w[1]) + w[2]) + w[3]);
      g[li * st + sn] = real(0.25) * (((w[4] + w[5]) + w[6]) + w[7]);
    } else if (e.kind == NB_COARSE && li < MX / 2) {
      // the coarse cell beside rows / columns 2 li, 2 li + 1, the cells away
      // from (in) and towards the owner (out), and along the face (lo, hi)
      const int t0 = X ? ((pm.y * MX + e.fy) >> 1) - e.y0 * MX
                       : ((pm.x * MX + e.fx) >> 1) - e.x0 * MX;
      const int t = t0 + li;
      const bool viaT = e.lev == tlevel;
      const int o = (t + kMbc) * st + ((low ? MX - 1 : 0) + kMbc) * sn;
      const int ol = t > 0 ? o - st : o, oh = t < MX - 1 ? o + st : o;  // (inside the patch)
      const int d = low ? -sn : sn;
      real q0, in, out, lo, hi;
      if (direct && viaT) {
        const int c = D.cur[tlevel];
        const real* qo = D.buf[c ^ 1] + (size_t)e.n0 * SS;
        const real* qn = D.buf[c] + (size_t)e.n0 * SS;
        if (alpha == real(0) || alpha == real(1)) {  // (see coarse_interior)
          const real* q = alpha == real(0) ? qo : qn;
          q0 = q[o];
          in = q[o + d];
          lo = q[ol];
          hi = q[oh];
        } else {
          const real b = real(1) - alpha;
          q0 = b * qo[o] + alpha * qn[o];
          in = b * qo[o + d] + alpha * qn[o + d];
          lo = b * qo[ol] + alpha * qn[ol];
          hi = b * qo[oh] + alpha * qn[oh];
        }
        if (e.code[0] & kSrcComplete) {  // towards the owner: the average of its own cells
          const real* w = T + (2 * li + kMbc) * st + (low ? kMbc : MX) * sn;
          const int a = X ? sn : st, b2 = X ? st : sn;
          out = real(0.25) * (((w[0] + w[a]) + w[b2]) + w[a + b2]);
        } else {
          const PatchMeta cm{e.lev, e.x0, e.y0, 0, 0, 0};
          const int n = low ? MX : -1;
          out = coarse_ghost<real, MX>(D, cm, e.n0, tlevel, alpha, X ? n : t, X ? t : n);
        }
      } else {
        const real* q = patch_ptr(viaT ? D.qT : D.buf[D.cur[e.lev]], e.n0, S);
        q0 = q[o];
        in = q[o + d];
        out = q[o - d];
        lo = q[ol];
        hi = q[oh];
      }
      if (t == 0) lo = cells[f];
      if (t == MX - 1) hi = cells[f];
      // slopes towards higher index, across the face and along it
      const real sc = low ? minmod(out - q0, q0 - in) : minmod(in - q0, q0 - out);
      const real sl = minmod(hi - q0, q0 - lo);
      const real sx = X ? sc : sl, sy = X ? sl : sc;
      real* w = g + 2 * li * st;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        w[(k & 1) + (k >> 1) * S] = fine_value(q0, sx, sy, k & 1, k >> 1);
    }
  }
#pragma unroll 1
  for (int k = li; k < 16; k += MX) {  // the corners
    const int r = 4 + (k >> 2), x = k & 1, y = (k >> 1) & 1;
    const NbrEntry& e = E[r];
    real v;
    if (e.kind == NB_FINE) {
      const real* w = D.buf[D.cur[e.lev]] + (size_t)e.n0 * SS +
                      (((r & 2) ? 0 : MX - 4) + 2 * y + kMbc) * S + ((r & 1) ? 0 : MX - 4) + 2 * x +
                      kMbc;
      v = real(0.25) * (((w[0] + w[1]) + w[S]) + w[S + 1]);
    } else if (e.kind == NB_COARSE) {
      const real* c = cells + 4 + 5 * (r - 4);
      const real sx = minmod(c[1] - c[0], c[0] - c[2]), sy = minmod(c[3] - c[0], c[0] - c[4]);
      v = fine_value(c[0], sx, sy, x, y);
    } else {
      continue;
    }
    T[(((r & 2) ? MX : -2) + y + kMbc) * S + ((r & 1) ? MX : -2) + x + kMbc] = v;
  }
}

template <typename real, int MX>
struct WalkShape {
  static constexpr int PK = Packed<real>::N;        // cells a lane works on at once
  static constexpr bool SPLIT = PK == 2 && MX == 32;  // of one patch (two halves of its rows)
  static constexpr int NPS = SPLIT ? 1 : PK;        // patches of a segment of MX lanes
  static constexpr int PPW = (32 / MX) * NPS;       // patches of a warp
  static constexpr int R = SPLIT ? MX / 2 : MX;     // rows a lane walks
};

// CTAs an SM is to hold of 8 warps each: FP32 24 warps of at most 80
// registers, FP64 16 of 128 (its pipe, not latency, bounds it)
template <typename real, int MX, bool SWIRL, bool FULL>
__global__ void __launch_bounds__(256, sizeof(real) == 4 ? 3 : 2)
    advance_walk_kernel(const __grid_constant__ DevForest<real> D, int p0, int p1,
                        const __grid_constant__ AdvArgs a, AdvConst<real> ac, int* err) {
  using W = WalkShape<real, MX>;
  using PV = Packed<real>;
  using V = typename PV::V;
  using SL = Slot<real, MX>;
  constexpr int S = MX + 4, TILE = S * S, PPW = W::PPW, NSEG = 32 / MX;
  constexpr unsigned kAll = 0xffffffffu;
  constexpr uint32_t tbytes = sizeof(real) * TILE, nbytes = 8 * sizeof(NbrEntry);
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bars[8];
  __shared__ real ucoef_s;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, NW = blockDim.x >> 5;
  const int seg = lane / MX, li = lane % MX;
  unsigned char* wbase = smem_raw + (size_t)warp * PPW * SL::bytes;
  auto slot = [&](int s) { return wbase + s * SL::bytes; };

  if (threadIdx.x == 0 && SWIRL) {
    const double t = a.t0_dev ? *a.t0_dev + a.t_off : a.t_half;
    ucoef_s = cospi_ratio<real>(t, a.period) * real(a.sfac * 0.5 * a.nu);
  }
  if (lane == 0) mbar_init(&bars[warp], 1);
  __syncthreads();

  const real ucoef = SWIRL ? ucoef_s : real(0);
  const Scheme<real, FULL> sc = make_scheme<real, FULL>(D.order, D.limiter, D.transverse);
  const real h = ac.h;
  const real* tab = static_cast<const real*>(a.trig);
  auto sin2 = [&](int z) -> real {  // sin^2(pi x) at node z
    if (tab) return tab[z + 1];
    const real s = sinpi_r(real(z) * h);
    return s * s;
  };
  auto sin1 = [&](int z) -> real {  // sin(pi (x_z + x_{z+1}))
    return tab ? tab[a.trig_len + z + 1] : sinpi_r(real(2 * z + 1) * h);
  };

  const int ngroups = (p1 - p0 + PPW - 1) / PPW;
  const int TW = gridDim.x * NW;
  uint32_t par = 0;
  for (int g = blockIdx.x * NW + warp; g < ngroups; g += TW) {
    const int pg = p0 + g * PPW, nvalid = min(PPW, p1 - pg);
    if (lane == 0) {
      fence_proxy_async();
      mbar_expect_tx(&bars[warp], nvalid * (tbytes + (a.gather ? nbytes : 0)));
      for (int s = 0; s < nvalid; ++s) {
        const int p = pg + s;
        bulk_load(slot(s) + SL::tile, D.buf[D.cur[a.level]] + (size_t)p * TILE, tbytes, &bars[warp]);
        if (a.gather) bulk_load(slot(s) + SL::nbr, D.nbr + (size_t)p * 8, nbytes, &bars[warp]);
      }
    }
    // this lane's patches (beyond the range: the group's first, not stored)
    int pk[W::NPS];
    bool ok[W::NPS];
    real ux[W::NPS], vy[W::NPS];          // factors of the lane's x- and y-edges
    real uxE[W::NPS], vyM[W::NPS], vyP[W::NPS];  // of x-edge MX and of columns -1, MX
#pragma unroll
    for (int k = 0; k < W::NPS; ++k) {
      const int s = k * NSEG + seg;
      ok[k] = s < nvalid;
      pk[k] = ok[k] ? pg + s : pg;
      ux[k] = vy[k] = uxE[k] = vyM[k] = vyP[k] = real(0);
      if (SWIRL) {
        const PatchMeta pm = D.meta[pk[k]];
        const int x0 = pm.x * MX, y0 = pm.y * MX;
        ux[k] = ucoef * sin2(x0 + li);
        vy[k] = -ucoef * sin1(x0 + li);
        uxE[k] = ucoef * sin2(x0 + MX);
        vyM[k] = -ucoef * sin1(x0 - 1);
        vyP[k] = -ucoef * sin1(x0 + MX);
        // row r: factor of its x-edges, and of the y-edges above it
        real* rw = reinterpret_cast<real*>(slot(ok[k] ? s : 0) + SL::rows);
        if (ok[k])
          for (int r = li - 1; r <= MX; r += MX) {
            rw[2 * (r + 1)] = sin1(y0 + r);
            rw[2 * (r + 1) + 1] = sin2(y0 + r + 1);
          }
      }
    }
    const bool landed = mbar_wait(&bars[warp], par, a.wait_limit);
    if (!__all_sync(kAll, landed)) {
      if (lane == 0) atomicOr(err, kErrTimeout);
      mbar_wait(&bars[warp], par, kWaitLimit);  // let the copies in flight land before leaving
      return;
    }
    par ^= 1;
    if (a.gather) {  // Alg. 1 for the warp's patches, into their tiles' ghost rings
      bool mixed = false, wall = false;
#pragma unroll
      for (int k = 0; k < W::NPS; ++k) {
        const int s = k * NSEG + seg;
        if (s < nvalid)
          for (int r = li; r < 8; r += MX) {
            const int kind = reinterpret_cast<const NbrEntry*>(slot(s) + SL::nbr)[r].kind;
            mixed |= kind == NB_FINE || kind == NB_COARSE;
            wall |= kind == NB_EXTERIOR;
          }
      }
      mixed = __any_sync(kAll, mixed);
      wall = __any_sync(kAll, wall);
#pragma unroll 1
      for (int k = 0; k < W::NPS; ++k) {
        const int s = k * NSEG + seg;
        if (s < nvalid)
          gather_part1<real, MX>(D, reinterpret_cast<const NbrEntry*>(slot(s) + SL::nbr),
                                 D.meta[pg + s], pg + s, a.tlevel, ac.alpha, a.direct != 0, mixed,
                                 reinterpret_cast<real*>(slot(s) + SL::tile),
                                 reinterpret_cast<real*>(slot(s) + SL::ye), li);
      }
      __syncwarp();
      if (mixed) {
#pragma unroll 1
        for (int k = 0; k < W::NPS; ++k) {
          const int s = k * NSEG + seg;
          if (s < nvalid)
            gather_part2<real, MX>(D, reinterpret_cast<const NbrEntry*>(slot(s) + SL::nbr),
                                   D.meta[pg + s], pg + s, a.tlevel, ac.alpha, a.direct != 0,
                                   reinterpret_cast<real*>(slot(s) + SL::tile),
                                   reinterpret_cast<const real*>(slot(s) + SL::ye), li);
        }
        __syncwarp();
      }
      if (wall && D.domain == FC_DOMAIN_WALLS) {
#pragma unroll 1
        for (int k = 0; k < W::NPS; ++k) {
          const int s = k * NSEG + seg;
          if (s < nvalid)
            wall_bc<real, MX>(D.meta[pg + s], reinterpret_cast<real*>(slot(s) + SL::tile), li, MX);
        }
        __syncwarp();
      }
    } else {
      __syncwarp();  // the rows' factors
    }
    if (a.keep)  // the adjoint's replay keeps the ghost-filled input tile
      for (int k = 0; k < W::NPS; ++k) {
        const int s = k * NSEG + seg;
        if (s >= nvalid) continue;
        const real* T = reinterpret_cast<const real*>(slot(s) + SL::tile);
        real* kp = static_cast<real*>(a.keep) + (size_t)(pg + s - a.keep_p0) * TILE;
        for (int c = li; c < TILE; c += MX) kp[c] = T[c];
      }
    // packed views: component k of a lane reads slot sk at row offset rk
    const unsigned char* b0 = slot(ok[0] ? seg : 0);
    const unsigned char* b1 =
        W::SPLIT ? b0 : W::NPS == 2 ? slot(ok[W::NPS - 1] ? NSEG + seg : 0) : b0;
    const real* T0 = reinterpret_cast<const real*>(b0 + SL::tile);
    const real* T1 = reinterpret_cast<const real*>(b1 + SL::tile);
    constexpr int r1 = W::SPLIT ? W::R : 0;  // row offset of component 1
    constexpr int kl = W::NPS - 1;           // patch of component 1

    // the edges beside the lanes: x-edge MX of rows -1..MX, y-edges of ghost
    // columns -1 and MX at rows 0..MX, one (packed: two) a lane and round; in
    // the split form a lane takes edges t and t + NT, else edge t of both patches
    {
      constexpr int NTASK = 3 * MX + 4;
      constexpr int NT = W::SPLIT ? (NTASK + 1) / 2 : NTASK;
      for (int t = li; t < NT; t += MX) {
        V c, qa, qb, qc, qd;
        const int ts[2] = {t, W::SPLIT ? t + NT : t};
        real cc[2], v[2][4];
#pragma unroll
        for (int k = 0; k < PV::N; ++k) {
          const int q = min(ts[k], NTASK - 1);
          const bool x = q < MX + 2;
          const bool right = q >= 2 * MX + 3;
          const int r = x ? q - 1 : q - (right ? 2 * MX + 3 : MX + 2);
          const real* T = k ? T1 : T0;
          const real* rw = reinterpret_cast<const real*>((k ? b1 : b0) + SL::rows);
          const real* o = T + (r + kMbc) * S + ((x || right) ? MX : -1) + kMbc;
          const int st = x ? 1 : S;
          const int w = k ? kl : 0;
          // (y-edge row r takes the factor stored with row r - 1)
          cc[k] = SWIRL ? (x ? uxE[w] * rw[2 * (r + 1)]
                             : (right ? vyP[w] : vyM[w]) * rw[2 * r + 1])
                        : (x ? ac.cu : ac.cv);
          v[k][0] = o[-2 * st];
          v[k][1] = o[-st];
          v[k][2] = o[0];
          v[k][3] = o[st];
        }
        constexpr int z = PV::N - 1;
        c = PV::make(cc[0], cc[z]);
        qa = PV::make(v[0][0], v[z][0]);
        qb = PV::make(v[0][1], v[z][1]);
        qc = PV::make(v[0][2], v[z][2]);
        qd = PV::make(v[0][3], v[z][3]);
        V F, nP, M;
        const Speed<V> sp(c);
        const V W = vsub(qc, qb);
        vedge(sp, W, vupwind(c, qa, qb, qc, qd), qb, qc, sc, F, nP, M);
#pragma unroll
        for (int k = 0; k < PV::N; ++k) {
          const int q = ts[k];
          if (q >= NTASK || !ok[W::SPLIT ? 0 : k]) continue;
          unsigned char* b = const_cast<unsigned char*>(k ? b1 : b0);
          if (q < MX + 2) {
            EdgeRec<real>* e = reinterpret_cast<EdgeRec<real>*>(b + SL::rec) + q;
            e->M = PV::get(M, k);
            e->A = PV::get(F, k);  // (the normal flux and the speed, until both columns are known)
            e->B = PV::get(c, k);
            if (sizeof(real) == 8) e->W = PV::get(W, k);
          } else {
            const bool right = q >= 2 * MX + 3;
            const int r = q - (right ? 2 * MX + 3 : MX + 2);
            real* y = reinterpret_cast<real*>(b + SL::ye) + (right ? 2 * (MX + 1) : 0);
            y[r] = PV::get(nP, k);
            y[MX + 1 + r] = PV::get(M, k);
          }
        }
      }
      __syncwarp();
#pragma unroll
      for (int k = 0; k < W::NPS; ++k) {
        if (!ok[k]) continue;
        unsigned char* b = const_cast<unsigned char*>(k ? b1 : b0);
        const real* y = reinterpret_cast<const real*>(b + SL::ye);
        reinterpret_cast<real*>(b + SL::yl)[li + 1] = y[li] - y[MX + 1 + li + 1];
        EdgeRec<real>& e = reinterpret_cast<EdgeRec<real>*>(b + SL::rec)[li + 1];
        const real nYE = y[2 * (MX + 1) + li] - y[3 * (MX + 1) + li + 1];  // of ghost cell MX
        edge_affine(e.B, nYE, e.A, sc, e.A, e.B);
      }
      __syncwarp();
      if (sizeof(real) == 8) {  // the jumps of x-edge -1, over the P, M that no lane reads now
        if (ok[0])
          for (int r = li; r < MX + 2; r += MX)
            reinterpret_cast<real*>(const_cast<unsigned char*>(b0) + SL::wl)[r] =
                T0[(r + 1) * S + 1] - T0[(r + 1) * S];
        __syncwarp();
      }
    }

    // the walk: iteration it works on row r = it - 1 (of each component's
    // rows): x-edge (li, r), y-edge (li, r + 1), the final fluxes of row r
    // and the update of row r - 1.  Rows outside the patch's are computed
    // from whatever shared memory holds there and used by no stored cell.
    auto col = [&](int i, int r) -> V {  // cell (li + i, r) of each component
      const int o = (r + kMbc) * S + li + i + kMbc;
      return PV::make(T0[o], T1[o + r1 * S]);
    };
    const V uxv = PV::make(ux[0], ux[kl]), vyv = PV::make(vy[0], vy[kl]);
    const real* rw0 = reinterpret_cast<const real*>(b0 + SL::rows);
    const real* rw1 = reinterpret_cast<const real*>(b1 + SL::rows) + 2 * r1;
    const EdgeRec<real>* ec0 = reinterpret_cast<const EdgeRec<real>*>(b0 + SL::rec);
    const EdgeRec<real>* ec1 = reinterpret_cast<const EdgeRec<real>*>(b1 + SL::rec) + r1;
    const real* yl0 = reinterpret_cast<const real*>(b0 + SL::yl);
    const real* yl1 = reinterpret_cast<const real*>(b1 + SL::yl) + r1;
    const real* wl0 = reinterpret_cast<const real*>(b0 + SL::wl);
    real* dst = D.buf[D.cur[a.level] ^ 1];
    real* dst0 = dst + (size_t)pk[0] * TILE + li + kMbc;
    real* dst1 = dst + (size_t)pk[kl] * TILE + r1 * S + li + kMbc;
    const bool okl = ok[kl];
    auto up = [&](V v) -> V {  // of the lane to the left
      return PV::make(__shfl_up_sync(kAll, PV::get(v, 0), 1, MX),
                      PV::N == 2 ? __shfl_up_sync(kAll, PV::get(v, 1), 1, MX) : real(0));
    };
    auto down = [&](V v) -> V {
      return PV::make(__shfl_down_sync(kAll, PV::get(v, 0), 1, MX),
                      PV::N == 2 ? __shfl_down_sync(kAll, PV::get(v, 1), 1, MX) : real(0));
    };
    const bool first = li == 0, last = li == MX - 1;
    V qa = col(0, -2), qb = col(0, -1), qc = col(0, 0);
    V Wa = vsub(qb, qa), Wb = vsub(qc, qb);
    const V zero = PV::all(real(0));
    V nX_prev = zero, G_cur = zero, nP_cur = zero, Gf_prev = zero, dF_prev = zero;
    Speed<V> v_cur(zero);
#pragma unroll(sizeof(real) == 4 ? 6 : 2)  // (FP32, 256 forests: 2.72 ms by 2, 2.68 by 6)
    for (int it = 0; it < W::R + 2; ++it) {
      const int r = it - 1;
      const V qd = col(0, r + 2);
      const V Wc = vsub(qd, qc);
      V fx, fy;  // speeds of x-edge (li, r) and y-edge (li, r + 1)
      if (SWIRL) {
        using V2 = typename Vec2<real>::T;
        const V2 f0 = reinterpret_cast<const V2*>(rw0)[it], f1 = reinterpret_cast<const V2*>(rw1)[it];
        fx = vmul(uxv, PV::make(f0.x, f1.x));
        fy = vmul(vyv, PV::make(f0.y, f1.y));
      } else {
        fx = PV::all(ac.cu);
        fy = PV::all(ac.cv);
      }
      const Speed<V> sx(fx), sy(fy);
      V F, nP, M;
      const EdgeRec<real> e0 = ec0[it], e1 = ec1[it];
      {
        const V ql = col(-1, r), W = vsub(qb, ql);
        V U;  // the jump on the upwind side
        if constexpr (PV::N == 1) {  // (FP64: the neighbouring lanes' instead of another
                                     // subtraction: 64 forests of 16^2 patches 2.03 -> 1.97 ms)
          const V Wl = up(W), Wr = down(W);
          U = vselect(fx, first ? wl0[it] : Wl, last ? e0.W : Wr);
        } else {
          U = vupwind(fx, col(-2, r), ql, qb, col(1, r));
        }
        vedge(sx, W, U, ql, qb, sc, F, nP, M);
      }
      V Mr = down(M);
      if (last) Mr = PV::make(e0.M, e1.M);
      const V nX = vsub(nP, Mr);  // turned x-fluctuation sum of cell (li, r)
      // (FP64: the last row's y-edge and the first and last rows' x-fluxes,
      // which nothing uses, are left out; FP32 has no branch here)
      constexpr bool kAll2 = PV::N == 2;
      V Gn = zero, nPn = zero, Mn = zero;
      if (kAll2 || it <= W::R) vedge(sy, Wb, vselect(fy, Wa, Wc), qb, qc, sc, Gn, nPn, Mn);
      // final flux of y-edge (li, r)
      const V Gf = vfinal(v_cur, nX_prev, nX, G_cur, sc);
      // final fluxes of x-edges (li, r) and (li + 1, r)
      V dF = zero;
      if (kAll2 || (it >= 1 && it <= W::R)) {
        const V nY = vsub(nP_cur, Mn);  // turned y-fluctuation sum of cell (li, r)
        V nYl = up(nY);
        if (first) nYl = PV::make(yl0[it], yl1[it]);
        const V Ff = vfinal(sx, nYl, nY, F, sc);
        V Fr = down(Ff);
        const V Fe = vfma(PV::make(e0.B, e1.B), nY, PV::make(e0.A, e1.A));
        if (last) Fr = Fe;
        dF = vsub(Fr, Ff);
      }
      if (it >= 2) {  // the update of cell (li, r - 1)
        const V n = vfma(PV::all(real(-2)), vadd(dF_prev, vsub(Gf, Gf_prev)), qa);
        if (ok[0]) dst0[(r + 1) * S] = PV::get(n, 0);
        if (PV::N == 2 && okl) dst1[(r + 1) * S] = PV::get(n, PV::N - 1);
      }
      nX_prev = nX;
      G_cur = Gn;
      v_cur = sy;
      nP_cur = nPn;
      Gf_prev = Gf;
      dF_prev = dF;
      qa = qb;
      qb = qc;
      qc = qd;
      Wa = Wb;
      Wb = Wc;
    }
    __syncwarp();  // the next group's copies overwrite the slots
  }
}

template <typename real, int MX, bool SWIRL, bool FULL>
cudaError_t walk_launch(const DevForest<real>& D, int p0, int p1, const AdvArgs& a, int* err,
                        cudaStream_t s) {
  using W = WalkShape<real, MX>;
  auto kern = advance_walk_kernel<real, MX, SWIRL, FULL>;
  // warps of a CTA: those asked for, at most what shared memory holds
  constexpr size_t per_warp = (size_t)W::PPW * Slot<real, MX>::bytes;
  constexpr int most = (int)(227 * 1024 / per_warp) < 8 ? (int)(227 * 1024 / per_warp) : 8;
  const int nw = a.warps < most ? a.warps : most;
  const size_t smem = nw * per_warp;
  // set once per process; concurrent first calls set the same
  static std::atomic<int> max_ctas[9];
  int cap = max_ctas[nw].load(std::memory_order_acquire);
  if (cap == 0) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(most * per_warp));
    if (e != cudaSuccess) return e;
    int dev = 0, nsm = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, nw * 32, smem);
    if (e != cudaSuccess) return e;
    cap = nsm * (per_sm > 0 ? per_sm : 1);
    max_ctas[nw].store(cap, std::memory_order_release);
  }
  const int groups = (p1 - p0 + W::PPW - 1) / W::PPW;
  int ctas = (groups + nw - 1) / nw;
  if (a.ctas > 0) cap = a.ctas;
  if (ctas > cap) ctas = cap;
  kern<<<ctas, nw * 32, smem, s>>>(D, p0, p1, a, adv_const(D, a), err);
  ++launch_counter();
  return cudaGetLastError();
}

template <typename real, int MX>
cudaError_t walk_opt(const DevForest<real>& D, int p0, int p1, const AdvArgs& a, int* err,
                     cudaStream_t s) {
  const bool full = full_scheme(D.order, D.limiter, D.transverse);
  if (D.vel_kind == FC_VEL_SWIRL)
    return full ? walk_launch<real, MX, true, true>(D, p0, p1, a, err, s)
                : walk_launch<real, MX, true, false>(D, p0, p1, a, err, s);
  return full ? walk_launch<real, MX, false, true>(D, p0, p1, a, err, s)
              : walk_launch<real, MX, false, false>(D, p0, p1, a, err, s);
}

}  // namespace

template <typename real>
cudaError_t launch_advance_walk(const DevForest<real>& D, int p0, int p1, const AdvArgs& a,
                                int* err, cudaStream_t s) {
  switch (D.mx) {
    case 8: return walk_opt<real, 8>(D, p0, p1, a, err, s);
    case 16: return walk_opt<real, 16>(D, p0, p1, a, err, s);
    case 32: return walk_opt<real, 32>(D, p0, p1, a, err, s);
    default: return cudaErrorInvalidValue;
  }
}

// (compiled once per precision, see build.py)
template cudaError_t launch_advance_walk<FC_REAL>(const DevForest<FC_REAL>&, int, int,
                                                  const AdvArgs&, int*, cudaStream_t);

}  // namespace fc
