// Block sums of the Wilson kernels, in a header of their own that a host compiler takes too: tests/test_block_sums.py runs
// the block thread by thread under the schedules that a GPU may choose.
#pragma once

// Per-block partial sums: warp level in the iteration precision, across warps in FP64; quantity q goes to
// part[q gy + blockIdx.y].  Masked kernels call this once per slot in a loop, so the block meets again before it returns:
// a warp that has no sites of the next slot would otherwise store its next sums while warp 0 still adds these.
template <typename R, int NQ, int NT>
__device__ __forceinline__ void reduce_partials(R (&v)[NQ], double* part, int gy) {
  __shared__ double sh[NQ][NT / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    R t = v[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (lane == 0) sh[q][warp] = (double)t;
  }
  __syncthreads();
  if (threadIdx.x < NQ) {   // one thread per quantity: NT / 32 FP64 warp instructions a block, not NQ NT / 32
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) t += sh[threadIdx.x][w];
    part[(size_t)threadIdx.x * gy + blockIdx.y] = t;
  }
  __syncthreads();
}
