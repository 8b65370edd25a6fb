// lbm_batch.cuh -- the step of many independent domains (an ensemble of
// uneven grids, each with its own species constants and reference state)
// by one launch per kernel: persistent blocks walk a list of tiles (domain,
// first node), taking the domain's parameters into shared memory whenever
// the domain changes.  Each domain's collide is the one its own step would take
// (collide_node, or split_tile of lbm_split.cuh), and the stencils add up in the
// same order with the same rounding (lbm_stencil.cuh): a domain's state is that
// of the same domain stepped alone, whichever launch plan the batch runs.  With
// split_tile bit for bit; collide_node is compiled apart for the batch (its
// parameters in shared memory), which the compiler contracts differently in
// places, so there the two agree to rounding (seven steps, M <= 3: FP64 2e-16,
// FP32 5e-8, 16-bit storage 7e-7 of the largest population).
#pragma once

#include "lbm_collide.cuh"
#include "lbm_split.cuh"

namespace lbm {

template <int M, class Real, class Store, int PAR>
__global__ void __launch_bounds__(collide_block<M, Real, 0, Store>(), collide_min_blocks<M, Real, 0, Store>())
collide_batch_kernel(const DevParams<Real>* __restrict__ params, void* const* __restrict__ pops,
                     void* const* __restrict__ side, const int2* __restrict__ tiles, int ntiles,
                     unsigned* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ __align__(16) DevParams<Real> sp;
  static_assert(sizeof(DevParams<Real>) % 8 == 0, "8-byte words");
  int cur = -1;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int2 tl = tiles[t];
    if (tl.x != cur) {                       // block-uniform
      __syncthreads();
      const unsigned long long* src = reinterpret_cast<const unsigned long long*>(params + tl.x);
      unsigned long long* dst = reinterpret_cast<unsigned long long*>(&sp);
      for (int k = threadIdx.x; k < (int)(sizeof(DevParams<Real>) / 8); k += blockDim.x) dst[k] = src[k];
      __syncthreads();
      cur = tl.x;
    }
    collide_node<M, Real, Store, PAR, 0>(sp, static_cast<Store*>(pops[cur]), static_cast<Real*>(side[cur]), err,
                                         nullptr, nullptr, (long long)tl.y + threadIdx.x, smem_raw);
  }
}

// The same for the domains whose step takes the split collide; tiles of 32 nodes.
template <int M, class Real, class Store, int PAR>
__global__ void __launch_bounds__(Split<M>::THREADS, split_min_blocks<M, Real>())
collide_split_batch_kernel(const DevParams<Real>* __restrict__ params, void* const* __restrict__ pops,
                           void* const* __restrict__ side, const int2* __restrict__ tiles, int ntiles,
                           unsigned* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ __align__(16) DevParams<Real> sp;
  __shared__ PlaneOffsets po;
  Real* const sm = reinterpret_cast<Real*>(smem_raw);
  int cur = -1;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int2 tl = tiles[t];
    if (tl.x != cur) {                       // block-uniform; the tile before ended on a barrier
      const unsigned long long* src = reinterpret_cast<const unsigned long long*>(params + tl.x);
      unsigned long long* dst = reinterpret_cast<unsigned long long*>(&sp);
      for (int k = threadIdx.x; k < (int)(sizeof(DevParams<Real>) / 8); k += blockDim.x) dst[k] = src[k];
      __syncthreads();
      for (int k = threadIdx.x; k < (M + 2) * Q; k += blockDim.x) po.off[k] = (long long)k * sp.N * (long long)sizeof(Store);
      split_constants<M, Real>(sp, sm);
      __syncthreads();
      cur = tl.x;
    }
    split_tile<M, Real, Store, PAR, 0>(sp, static_cast<Store*>(pops[cur]), static_cast<Real*>(side[cur]), err, po, sm,
                                       tl.y / 32);
  }
}

template <class Real>
__global__ void __launch_bounds__(BLOCK_LIGHT)
grad_GK_batch_kernel(const BatchGeom* __restrict__ geom, void* const* __restrict__ side,
                     const int2* __restrict__ tiles, int ntiles) {
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int2 tl = tiles[t];
    const BatchGeom g = geom[tl.x];
    Real* const s = static_cast<Real*>(side[tl.x]);
    if (g.nx % ROWV == 0) grad_GK_node<Real, true>(g, s, (long long)tl.y + threadIdx.x);
    else grad_GK_node<Real, false>(g, s, (long long)tl.y + threadIdx.x);
  }
}

template <class Real>
__global__ void __launch_bounds__(BLOCK_LIGHT)
grad_X_batch_kernel(const BatchGeom* __restrict__ geom, void* const* __restrict__ side,
                    const int2* __restrict__ tiles, int ntiles) {
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int2 tl = tiles[t];
    const BatchGeom g = geom[tl.x];
    Real* const s = static_cast<Real*>(side[tl.x]);
    if (g.nx % ROWV == 0) grad_X_node<Real, true>(g, s, (long long)tl.y + threadIdx.x);
    else grad_X_node<Real, false>(g, s, (long long)tl.y + threadIdx.x);
  }
}

}  // namespace lbm
