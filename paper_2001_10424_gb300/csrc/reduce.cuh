// reduce.cuh - deterministic grid-wide reductions with a fused finaliser.
//
// Every block reduces its values (shared memory, then one warp's shuffles) and
// writes one partial per value; the last block to arrive (atomic ticket)
// sums the partials in a fixed order and runs the finaliser, which updates
// the solver scalars on the device. The order of every addition depends only
// on the launch shape, so results are bitwise reproducible run to run.
#pragma once
#include <cuda_runtime.h>
#include "common.cuh"
#include "state.cuh"

namespace gkb {

struct RedBuf {
  double* partial;        // >= max blocks * 4 doubles
  unsigned int* ticket;   // one counter, zero between launches
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// sums over the block (of at most 256 threads) of v[0..NV-1], value i to lane 0
// of warp i. Through shared memory: a warp adds the block's values eight (or
// so) to a lane, then across its lanes; shuffles in every warp first would
// issue four times as many FP64 additions, each of which holds the SM's FP64
// unit for 16 cycles (1024^2 product with dot, 4257 blocks: tile kernel 42.4 ->
// 41.3 us; in FP64 78.9 -> 72.1 us).
template <int NV>
__device__ __forceinline__ double block_sum(const double (&v)[NV], double (*sh)[256], int tid, int nthr) {
  const int lane = tid & 31, warp = tid >> 5;
#pragma unroll
  for (int i = 0; i < NV; ++i) sh[i][tid] = v[i];
  __syncthreads();
  double s = 0.0;
  if (warp < NV) {
    for (int t = lane; t < nthr; t += 32) s += sh[warp][t];
    s = warp_sum(s);
  }
  return s;
}

// All threads of every block of the problem's grid B must call this exactly
// once.
template <int NV>
__device__ void grid_reduce(double (&v)[NV], RedBuf red, int fin, void* st, const Blk& B) {
  __shared__ double sh[NV][256];
  __shared__ double tot[NV];
  __shared__ bool am_last;
  const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
  const int nthr = blockDim.x * blockDim.y * blockDim.z;
  const int lane = tid & 31, warp = tid >> 5;
  const unsigned bid = B.x + B.nx * (B.y + B.ny * B.z);
  const unsigned nblk = B.nx * B.ny * B.nz;
  double s = block_sum<NV>(v, sh, tid, nthr);
  if (warp < NV && lane == 0) red.partial[(size_t)bid * NV + warp] = s;
  __syncthreads();
  if (tid == 0) {
    __threadfence();  // the block's partials, ordered before its ticket
    unsigned t = atomicAdd(red.ticket, 1u);
    am_last = (t == nblk - 1);
  }
  __syncthreads();
  if (!am_last) return;
  __threadfence();
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    v[i] = 0.0;
    for (unsigned b = tid; b < nblk; b += nthr) v[i] += __ldcg(red.partial + (size_t)b * NV + i);
  }
  s = block_sum<NV>(v, sh, tid, nthr);
  if (warp < NV && lane == 0) tot[warp] = s;
  __syncthreads();
  if (tid == 0) {
    double fin_v[4] = {0, 0, 0, 0};
#pragma unroll
    for (int i = 0; i < NV; ++i) fin_v[i] = tot[i];
    finalize(fin, fin_v, st);
    *red.ticket = 0u;
  }
}

// the same over the launch's own grid
template <int NV>
__device__ __forceinline__ void grid_reduce(double (&v)[NV], RedBuf red, int fin, void* st) {
  grid_reduce<NV>(v, red, fin, st, native_blk());
}

}  // namespace gkb
