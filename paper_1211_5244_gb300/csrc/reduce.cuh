// Block and grid reductions of the Hartree energy (FP64, deterministic order).
#pragma once

#include "common.cuh"

namespace ps {

__device__ __forceinline__ double block_sum(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  const int nw = (blockDim.x + 31) >> 5;
  v = (threadIdx.x < nw) ? sh[threadIdx.x] : 0.0;
  if (wid == 0) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  }
  return v;  // valid in thread 0
}

// Deterministic grid reduction: every CTA stores its partial; the CTA that
// arrives last sums all partials in index order and resets the counter.
__device__ inline void energy_finish(double part, double* partials, unsigned* counter,
                              double scale, double* E) {
  __shared__ double sh[32];
  __shared__ unsigned s_last;
  const int nblk = gridDim.x * gridDim.y;
  const int bid = blockIdx.y * gridDim.x + blockIdx.x;
  double bs = block_sum(part, sh);
  if (threadIdx.x == 0) {
    partials[bid] = bs;
    __threadfence();
    const unsigned prev = atomicAdd(counter, 1u);
    s_last = (prev == (unsigned)(nblk - 1)) ? 1u : 0u;
  }
  __syncthreads();
  if (s_last) {
    __threadfence();
    double acc = 0.0;
    for (int i = threadIdx.x; i < nblk; i += blockDim.x) acc += __ldcg(partials + i);
    double tot = block_sum(acc, sh);
    if (threadIdx.x == 0) {
      *E = scale * tot;
      *counter = 0u;
    }
  }
}

// The energy of a solve in two halves. The z pass (or the fused pass along
// another axis) stores one partial per CTA and is done; one CTA of the last pass adds them
// in a fixed order (four strided sums per thread, then the CTA's sum: the same
// partials give the same bits), beside the other CTAs: CTA 0 after its own rows in
// the register and Stockham kernels, one without lines of its own in the tile kernels. A
// last-arriving CTA in the z pass itself cost its fence, its atomic and the sum at
// the end of the pass, where nothing else runs (128^3 wire FP32: 40.8 us per solve
// against 37.1 without the energy).
__device__ inline void energy_partial(double part, double* partials) {
  __shared__ double sh[32];
  const double bs = block_sum(part, sh);
  if (threadIdx.x == 0) partials[blockIdx.y * gridDim.x + blockIdx.x] = bs;
}

// ... for an FP32 per-thread value: FP32 within each warp, the warp sums
// added in FP64 by one thread
__device__ inline void energy_partial_f32(float part, double* partials) {
  __shared__ float wsum[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    double bs = 0.0;
    for (int w = 0; w < (int)((blockDim.x + 31) >> 5); ++w) bs += (double)wsum[w];
    partials[blockIdx.y * gridDim.x + blockIdx.x] = bs;
  }
}

// The last pass's half: every thread of one CTA calls it.
__device__ inline void energy_total(const double* partials, int n, double scale, double* E) {
  __shared__ double sh[32];
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for (int i = threadIdx.x; i < n; i += 4 * blockDim.x)
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = i + u * blockDim.x;
      if (j < n) acc[u] += __ldcg(partials + j);
    }
  const double tot = block_sum((acc[0] + acc[1]) + (acc[2] + acc[3]), sh);
  if (threadIdx.x == 0) *E = scale * tot;
}

}  // namespace ps
