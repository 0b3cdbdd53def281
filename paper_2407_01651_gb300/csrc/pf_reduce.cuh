// pf_reduce.cuh -- the block-level end of the FP64 reductions.
//
// Every reduction writes one record of NQ sums per block; one block of 256
// threads then adds the records.  A single warp that walks 1024 records one
// after the other waits for 1024 dependent FP64 additions (109 us measured);
// 256 threads with at most a few records each and a shuffle tree take about
// 3 us.  The order is fixed by the block and thread indices, so a result does
// not depend on scheduling.
#pragma once

#include <cuda_runtime.h>

namespace pf {

constexpr int RED_THREADS = 256;

// Sum over the 256 threads of a block (QMAX: the quantity that takes the
// maximum instead, -1 for none).  The result is valid in thread q for
// quantity q, as the return value.
template <int NQ, int QMAX = -1>
__device__ __forceinline__ double block_sum256(double (&acc)[NQ]) {
  __shared__ double sh[NQ][RED_THREADS / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int half = 16; half > 0; half >>= 1) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const double o = __shfl_down_sync(0xffffffffu, acc[q], half);
      acc[q] = q == QMAX ? fmax(acc[q], o) : acc[q] + o;
    }
  }
  __syncthreads();   // a second use of sh within one kernel
  if (lane == 0)
#pragma unroll
    for (int q = 0; q < NQ; ++q) sh[q][warp] = acc[q];
  __syncthreads();
  double r = 0.0;
  if ((int)threadIdx.x < NQ) {
    r = sh[threadIdx.x][0];
#pragma unroll
    for (int w = 1; w < RED_THREADS / 32; ++w) {
      const double o = sh[threadIdx.x][w];
      r = (int)threadIdx.x == QMAX ? fmax(r, o) : r + o;
    }
  }
  return r;
}

// Sum of nb records of NQ doubles by one block of 256 threads; thread q
// returns quantity q.
template <int NQ, int QMAX = -1>
__device__ __forceinline__ double sum_records256(const double* partial, int nb) {
  double acc[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) acc[q] = 0.0;
  for (int b = threadIdx.x; b < nb; b += RED_THREADS) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      // written by other blocks of the same launch in the one-launch form
      const double v = __ldcg(partial + (size_t)b * NQ + q);
      acc[q] = q == QMAX ? fmax(acc[q], v) : acc[q] + v;
    }
  }
  return block_sum256<NQ, QMAX>(acc);
}

// True in every thread of the block that finishes last.  ctr starts at 0 and
// is 0 again afterwards.  Call after this block's record was written.
__device__ __forceinline__ bool last_block(unsigned int* ctr) {
  __shared__ bool last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicInc(ctr, gridDim.x - 1) == gridDim.x - 1;
    __threadfence();
  }
  __syncthreads();
  return last;
}

// out[0..NQ) = the sum of nb records, one block of 256 threads.
template <int NQ>
static __global__ void __launch_bounds__(RED_THREADS) k_sum_records(
    const double* __restrict__ partial, int nb, double* __restrict__ out) {
  const double r = sum_records256<NQ>(partial, nb);
  if ((int)threadIdx.x < NQ) out[threadIdx.x] = r;
}

}  // namespace pf
