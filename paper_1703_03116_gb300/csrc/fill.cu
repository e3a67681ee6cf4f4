// Standalone ghost-cell fill kernels (Alg. 1, Sec. 2.3), one CTA per target
// patch, writing the ghost ring of the patch arrays in HBM.
//
// fill_coarse: phases 1-2 -- copy from same-size neighbours, average fine
//   neighbours, then the physical boundary condition.  Patches on the
//   time-interpolated level also receive their interior (1 - alpha) q_old +
//   alpha q_new (multirate: the coarse data a finer level interpolates from).
// fill_fine: phases 3-4 -- interpolation from the coarser neighbour, then
//   the boundary condition again.
// On the cubed sphere the corner ghosts beyond a cube vertex are set last,
// by whichever kernel finishes the patch's edge ghosts.
//
// The rules themselves live in ghost_gather.cuh, shared with the patch-update
// kernels, which apply them to the tile they hold in shared memory.
// fill_tag: the whole of Alg. 1 for every patch at one time, and the regrid
//   indicator, in one launch: a coarser neighbour's cells are computed where
//   they are read (as the updates do), so no patch waits for another's ghosts,
//   and the indicator is taken from the tile in shared memory.
#include "ghost_ring.cuh"

namespace fc {
namespace {

// One CTA per patch: its tile by a bulk copy, its ghost ring (ghost_ring.cuh,
// or ghost by ghost where a neighbour's axes are turned), the wall condition
// and the corners beyond a cube vertex; the ghosts go back to the patch's
// array, the indicator (kind 0: max over cells of |grad q| / 2, 1: max q - min
// q; tag_kernel's values) to delta if it is set.  Three launches took their
// latency one after another (496 patches of 32^2, FP32: 20 us and two gaps, now
// 6 us; the tag with its copy to the host 47 -> 29 us).
template <typename real, int MX, bool CAP>
__global__ void __launch_bounds__(288) fill_tag_kernel(const __grid_constant__ DevForest<real> D,
                                                       int kind, double* delta, uint32_t wait_limit,
                                                       int* err) {
  constexpr int S = MX + 4, NT = 288, NG = num_ghosts<MX>();
  constexpr uint32_t bytes = sizeof(real) * S * S;
  __shared__ __align__(128) real Q[S * S];
  __shared__ __align__(8) uint64_t bar;
  __shared__ real ring[CAP ? NG : 24];
  __shared__ bool ring_w[CAP ? NG : 1];
  __shared__ real red[2][NT / 32];
  const int tid = threadIdx.x, p = blockIdx.x;
  if (tid == 0) mbar_init(&bar, 1);
  const PatchMeta pm = D.meta[p];
  const int L = pm.level;
  real* P = D.buf[D.cur[L]] + (size_t)p * S * S;
  if (tid == 0) {
    fence_proxy_async();
    mbar_expect_tx(&bar, bytes);
    bulk_load(Q, P, bytes, &bar);
  }
  const bool each = CAP && (pm.flags & 2);
  RingPart<real> part;
  if (each)
    gather_ring<real, MX>(D, [&](int r) { return D.nbr[(size_t)p * 8 + r]; }, p, pm, L - 1,
                          real(1), true, ring, ring_w, tid, NT);
  else
    part = ring_read<real, MX, CAP>(D, p, pm, L, L - 1, real(1), true, ring, tid, nullptr, 0);
  const bool landed = tid == 0 ? mbar_wait(&bar, 0, wait_limit) : true;
  if (!__syncthreads_and(landed)) {
    if (tid == 0) atomicOr(err, kErrTimeout);
    mbar_wait(&bar, 0, kWaitLimit);  // let the copy land before leaving
    return;
  }
  if (tid != 0) mbar_wait(&bar, 0, kWaitLimit);
  if (each)
    store_ring<real, MX>(Q, ring, ring_w, tid, NT);
  else
    ring_store<real, MX, CAP>(D, part, L, L - 1, real(1), true, Q, ring, tid, nullptr, 0, p);
  __syncthreads();
  const int last_q = (1 << L) - 1;
  if (D.domain == FC_DOMAIN_WALLS &&
      (pm.x == 0 || pm.y == 0 || pm.x == last_q || pm.y == last_q)) {
    wall_bc<real, MX>(pm, Q, tid, NT);
    __syncthreads();
  }
  if (each) {
    corner3_fill_k<real, MX>([&](int r) { return D.nbr[(size_t)p * 8 + r].kind; }, Q, tid, NT);
    __syncthreads();
  }
  for (int k = tid; k < NG; k += NT) {
    int i, j;
    ghost_ij<MX>(k, i, j);
    const int o = (j + kMbc) * S + i + kMbc;
    P[o] = Q[o];
  }
  if (!delta) return;
  real hi = kind == 1 ? Q[2 * S + 2] : real(0), lo = hi;
  for (int k = tid; k < MX * MX; k += NT) {
    const real* c = Q + (k / MX + 2) * S + k % MX + 2;
    real v = c[0];
    if (kind == 0) {
      const real gx = c[1] - c[-1], gy = c[S] - c[-S];
      v = gx * gx + gy * gy;
    }
    hi = v > hi ? v : hi;
    lo = v < lo ? v : lo;
  }
  for (int w = 16; w > 0; w >>= 1) {
    const real a = __shfl_down_sync(0xffffffffu, hi, w), b = __shfl_down_sync(0xffffffffu, lo, w);
    hi = a > hi ? a : hi;
    lo = b < lo ? b : lo;
  }
  if ((tid & 31) == 0) {
    red[0][tid >> 5] = hi;
    red[1][tid >> 5] = lo;
  }
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < NT / 32; ++w) {
      hi = red[0][w] > hi ? red[0][w] : hi;
      lo = red[1][w] < lo ? red[1][w] : lo;
    }
    delta[p] = kind == 1 ? (double)hi - (double)lo : 0.5 * sqrt((double)hi);
  }
}

template <typename real, int MX>
__global__ void __launch_bounds__(256) fill_coarse_kernel(DevForest<real> D, FillArgs A) {
  constexpr int S = MX + 4;
  __shared__ NbrStage st;
  const real alpha = real(A.alpha);
  for (int t = blockIdx.x; t < A.ntargets; t += gridDim.x) {
    const int p = A.targets[t];
    stage_neighbours(D.meta, D.nbr, p, st, threadIdx.x);
    const PatchMeta pm = D.meta[p];
    __syncthreads();
    real* Q = patch_ptr((pm.level == A.tlevel) ? D.qT : D.buf[D.cur[pm.level]], p, S);
    if (pm.level == A.tlevel) {
      if (A.full_interior) {
        for (int k = threadIdx.x; k < MX * MX; k += blockDim.x) {
          const int i = k % MX, j = k / MX;
          Q[(j + kMbc) * S + i + kMbc] = src_interior(D, A.tlevel, alpha, p, pm.level, i, j);
        }
      } else {
        // the cells within two of the patch's edge: rows 0, 1, MX-2, MX-1,
        // then columns 0, 1, MX-2, MX-1 of the rows between
        constexpr int NR = 4 * MX + 4 * (MX - 4);
        for (int k = threadIdx.x; k < NR; k += blockDim.x) {
          int i, j;
          if (k < 4 * MX) {
            const int r = k / MX;
            j = r < 2 ? r : MX - 4 + r;
            i = k % MX;
          } else {
            const int c = (k - 4 * MX) & 3;
            j = 2 + ((k - 4 * MX) >> 2);
            i = c < 2 ? c : MX - 4 + c;
          }
          Q[(j + kMbc) * S + i + kMbc] = src_interior(D, A.tlevel, alpha, p, pm.level, i, j);
        }
      }
    }
    for (int k = threadIdx.x; k < num_ghosts<MX>(); k += blockDim.x) {
      int i, j;
      ghost_ij<MX>(k, i, j);
      real v;
      if (copy_or_average<real, MX>(D, st, pm, A.tlevel, alpha, i, j, v))
        Q[(j + kMbc) * S + i + kMbc] = v;
    }
    if (D.domain == FC_DOMAIN_WALLS) {
      __syncthreads();
      wall_bc<real, MX>(pm, Q, threadIdx.x, blockDim.x);
    }
    if (D.domain == FC_DOMAIN_SPHERE && !(pm.flags & 1)) {  // edge ghosts are final
      __syncthreads();
      corner3_fill<real, MX>(st, Q, threadIdx.x, blockDim.x);
    }
    __syncthreads();
  }
}

template <typename real, int MX>
__global__ void __launch_bounds__(256) fill_fine_kernel(DevForest<real> D, FillArgs A) {
  constexpr int S = MX + 4;
  __shared__ NbrStage st;
  for (int t = blockIdx.x; t < A.ntargets; t += gridDim.x) {
    const int p = A.targets[t];
    stage_neighbours(D.meta, D.nbr, p, st, threadIdx.x);
    const PatchMeta pm = D.meta[p];
    __syncthreads();
    real* Q = patch_ptr((pm.level == A.tlevel) ? D.qT : D.buf[D.cur[pm.level]], p, S);
    for (int k = threadIdx.x; k < num_ghosts<MX>(); k += blockDim.x) {
      int i, j;
      ghost_ij<MX>(k, i, j);
      real v;
      if (interpolate<real, MX>(D, st, pm, A.tlevel, i, j, v)) Q[(j + kMbc) * S + i + kMbc] = v;
    }
    if (D.domain == FC_DOMAIN_WALLS) {
      __syncthreads();
      wall_bc<real, MX>(pm, Q, threadIdx.x, blockDim.x);
    }
    if (D.domain == FC_DOMAIN_SPHERE) {
      __syncthreads();
      corner3_fill<real, MX>(st, Q, threadIdx.x, blockDim.x);
    }
    __syncthreads();
  }
}

inline int grid_for(int n) { return n < 1 ? 1 : (n < 65535 * 8 ? n : 65535 * 8); }

template <typename real, int MX>
cudaError_t fill_mx(const DevForest<real>& D, const FillArgs& A, bool fine, cudaStream_t s) {
  constexpr int threads = MX >= 32 ? 256 : 128;
  if (fine)
    fill_fine_kernel<real, MX><<<grid_for(A.ntargets), threads, 0, s>>>(D, A);
  else
    fill_coarse_kernel<real, MX><<<grid_for(A.ntargets), threads, 0, s>>>(D, A);
  ++launch_counter();
  return cudaGetLastError();
}

template <typename real>
cudaError_t fill_dispatch(const DevForest<real>& D, const FillArgs& A, bool fine,
                          cudaStream_t s) {
  if (A.ntargets <= 0) return cudaSuccess;
  switch (D.mx) {
    case 8: return fill_mx<real, 8>(D, A, fine, s);
    case 16: return fill_mx<real, 16>(D, A, fine, s);
    case 32: return fill_mx<real, 32>(D, A, fine, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

template <typename real>
cudaError_t launch_fill_coarse(const DevForest<real>& D, const FillArgs& A, cudaStream_t s) {
  return fill_dispatch(D, A, false, s);
}

template <typename real>
cudaError_t launch_fill_fine(const DevForest<real>& D, const FillArgs& A, cudaStream_t s) {
  return fill_dispatch(D, A, true, s);
}

template <typename real>
cudaError_t launch_fill_tag(const DevForest<real>& D, int kind, double* delta,
                            uint32_t wait_limit, int* err, cudaStream_t s) {
  if (D.npatch <= 0) return cudaSuccess;
  const bool cap = D.metric != nullptr;
  switch (D.mx) {
    case 8:
      if (cap)
        fill_tag_kernel<real, 8, true><<<D.npatch, 288, 0, s>>>(D, kind, delta, wait_limit, err);
      else
        fill_tag_kernel<real, 8, false><<<D.npatch, 288, 0, s>>>(D, kind, delta, wait_limit, err);
      break;
    case 16:
      if (cap)
        fill_tag_kernel<real, 16, true><<<D.npatch, 288, 0, s>>>(D, kind, delta, wait_limit, err);
      else
        fill_tag_kernel<real, 16, false><<<D.npatch, 288, 0, s>>>(D, kind, delta, wait_limit, err);
      break;
    case 32:
      if (cap)
        fill_tag_kernel<real, 32, true><<<D.npatch, 288, 0, s>>>(D, kind, delta, wait_limit, err);
      else
        fill_tag_kernel<real, 32, false><<<D.npatch, 288, 0, s>>>(D, kind, delta, wait_limit, err);
      break;
    default: return cudaErrorInvalidValue;
  }
  ++launch_counter();
  return cudaGetLastError();
}

template cudaError_t launch_fill_tag<float>(const DevForest<float>&, int, double*, uint32_t,
                                            int*, cudaStream_t);
template cudaError_t launch_fill_tag<double>(const DevForest<double>&, int, double*, uint32_t,
                                             int*, cudaStream_t);
template cudaError_t launch_fill_coarse<float>(const DevForest<float>&, const FillArgs&,
                                               cudaStream_t);
template cudaError_t launch_fill_coarse<double>(const DevForest<double>&, const FillArgs&,
                                                cudaStream_t);
template cudaError_t launch_fill_fine<float>(const DevForest<float>&, const FillArgs&,
                                             cudaStream_t);
template cudaError_t launch_fill_fine<double>(const DevForest<double>&, const FillArgs&,
                                              cudaStream_t);

}  // namespace fc
