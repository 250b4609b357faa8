// Deterministic reductions in FP64: block sums in a fixed order, and the sum of
// the fused step's tile partials into the per-step records.
#pragma once

#include <cuda_runtime.h>

#include "vplbm_params.h"

namespace vplbm {

// Programmatic dependent launch (launch_pdl). pdl_trigger: the next launch's
// blocks may take free slots from here on. pdl_wait: returns once all earlier
// work on the stream is complete and its writes are visible.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum of v[0..2] over the block of NT threads, fixed order; result valid in
// thread 0.
template <int NT = kThreads>
__device__ __forceinline__ void block_sum3(double v[3], double (*sm)[3]) {
  const int tid = threadIdx.x + threadIdx.y * blockDim.x;
  constexpr int n_warps = NT / 32;
  const int lane = tid & 31, warp = tid >> 5;
#pragma unroll
  for (int k = 0; k < 3; ++k) v[k] = warp_sum(v[k]);
  if (lane == 0) {
    sm[warp][0] = v[0];
    sm[warp][1] = v[1];
    sm[warp][2] = v[2];
  }
  __syncthreads();
  if (warp == 0) {  // a component a lane
    double s = 0.0;
    for (int w = 0; w < n_warps; ++w) s += sm[w][lane % 3];
#pragma unroll
    for (int k = 0; k < 3; ++k) v[k] = __shfl_sync(0xffffffffu, s, k);
  }
  __syncthreads();
}

// Tile i's partial of a step. Record units lie by unit and component, tile after
// tile, so that the threads' loads are contiguous (a tile's units one after the
// other cost four times the sectors, through one SM); a unit's density is an FP32
// number where the collision is, so that it is not converted back and forth on
// the FP64 pipe. A single step's sum is a chain of latencies that nothing hides:
// with this, and a component a lane in block_sum3's last sum, one 1024 x 256 FP32
// step with its record, alone, went from 22.1 to 20.5 us (three runs of each,
// apart by 0.4 and 0.8), the sum itself from 8.5 to 7.9. Leaving out the additions of
// zero forces by votes made it longer (8.2; 10.8 against 9.3 on 4096 x 1024).
__device__ __forceinline__ void tile_partial(const ReduceArgs& a, const double* src, int i, double v[3]) {
  if (!a.units) {
    for (int k = 0; k < 3; ++k) v[k] = __ldcg(src + 3ll * i + k);
    return;
  }
  double m64 = 0.0;
  float m32 = 0.f;
  v[0] = v[1] = 0.0;
  const long long nt = a.n_tiles;
  constexpr int kBatch = 4;  // units whose loads are under way at once (a tile has 4 or 8)
  for (int w0 = 0; w0 < a.units; w0 += kBatch) {
    double x[kBatch][3];
#pragma unroll
    for (int w = 0; w < kBatch; ++w) {
#pragma unroll
      for (int k = 0; k < 3; ++k) x[w][k] = __ldcg(src + nt * (3 * (w0 + w) + k) + i);
    }
#pragma unroll
    for (int w = 0; w < kBatch; ++w) {
      v[0] += x[w][0];
      v[1] += x[w][1];
      if (a.f64)
        m64 += x[w][2];
      else
        m32 += __int_as_float(__double2loint(x[w][2]));
    }
  }
  const int x0 = i % a.tiles_x * a.tile_x, y0 = i / a.tiles_x * a.tile_y;
  // sum rho = active nodes + sum drho
  v[2] = double(min(a.tile_x, a.nx - x0) * min(a.tile_y, a.ny - y0)) + (a.f64 ? m64 : double(m32));
}

// Records of the steps of one window: block (x, y) adds the partials of chunk
// y of step x's tiles (each thread its strided share in increasing order,
// then the block in a fixed order); with more than one chunk, the step's last
// block to finish adds the chunk sums the same way. The order depends on the
// tile count alone, so a solver's records do not depend on how its steps were
// batched, and a record is that of the single launch that wrote its partials.
// The sums stand apart from the step so that no block of the step waits for
// another: fence, arrival count and the last block's dependent FP64 sums at
// the end of every step cost 3.7 us of 12.8 on a 1024 x 256 FP32 grid, and
// 8 of 70 us on 4096 x 1024, where they also held resident-block slots. One
// launch per window of kWindow steps costs a few us per window.
__device__ __forceinline__ void reduce_steps(const ReduceArgs& a, int step, int chunk, double (*sm)[3],
                                             int* s_last) {
  const int tid = threadIdx.x;
  const int n_chunks = reduce_chunks(a.n_tiles);
  const double* src = a.partials + 3ll * a.n_tiles * (a.units ? a.units : 1) * step;
  const int end = min(a.n_tiles, (chunk + 1) * kChunkTiles);
  double v[3] = {0.0, 0.0, 0.0};
#pragma unroll 2
  for (int i = chunk * kChunkTiles + tid; i < end; i += kThreads) {
    double t[3];
    tile_partial(a, src, i, t);
    v[0] += t[0];
    v[1] += t[1];
    v[2] += t[2];
  }
  block_sum3(v, sm);
  if (n_chunks > 1) {
    double* cs = a.chunk_sums + 3ll * n_chunks * step;
    if (tid == 0) {
      for (int k = 0; k < 3; ++k) __stcg(cs + 3 * chunk + k, v[k]);
      __threadfence();
      *s_last = atomicAdd(a.counters + step, 1u) == unsigned(n_chunks - 1);
    }
    __syncthreads();
    if (!*s_last) return;
    __threadfence();
    v[0] = v[1] = v[2] = 0.0;
    for (int c = tid; c < n_chunks; c += kThreads)
      for (int k = 0; k < 3; ++k) v[k] += __ldcg(cs + 3 * c + k);
    block_sum3(v, sm);
    if (tid == 0) a.counters[step] = 0u;  // ready for the next window
  }
  // a ring shorter than the window keeps its latest steps
  if (tid == 0 && step + a.ring_len >= a.steps) {
    double* r = a.ring + 3ll * ((a.t0 + step) % a.ring_len);
    r[0] = v[0];
    r[1] = v[1];
    r[2] = a.reduce_mass ? v[2] : 0.0;
  }
}

}  // namespace vplbm
