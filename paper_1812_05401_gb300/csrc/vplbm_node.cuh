// The fused step with one node per thread, for grids too small to fill the GPU
// with a vector of nodes per thread.
#pragma once

#include "vplbm_device.cuh"

namespace vplbm {

// A block takes the nodes of one record unit: the rows y0 + w, y0 + w + W, ...
// of a tile that warp w of the vector kernel (step_tile) adds up, each TX
// nodes wide. A node's arithmetic is the vector kernel's and the unit's sums
// are formed in its order (N nodes of a row after the other, row after row,
// then across lanes), so both kernels give the same bits.
//
// A small grid's step is bound by latency: launch, load, one node's dependent
// chain, record. The vector kernel has a quarter of the warps, each with four
// nodes' instructions and the neighbour exchange in one chain, and in boundary
// tiles the fix-ups of a row's ends; here every lane loads its own neighbours
// (coalesced, unaligned). Per step, FP32 channel, vector against node kernel:
// 128 x 64 5.6 / 2.5 us, 640 x 320 6.3 / 4.3, 1024 x 512 8.1 / 8.0, 2048 x 512
// 12.2 / 14.4; FP16 128 x 64 8.1 / 2.9, 800 x 400 7.9 / 6.9, 1024 x 512
// 8.7 / 9.3; FP64, bound by each SM's FP64 pipe, over which the smaller blocks
// spread better: 300 x 100 33.4 / 11.7, 1000 x 400 98.8 / 84.8, 4096 x 1024
// 808 / 786. Hence the line in nodewise_rule.
template <int STORE, int COLL, int MODE>
__global__ void __launch_bounds__(kNodeThreads, kNodeBlocks)
    node_step_kernel(const __grid_constant__ StepParams p) {
  using S = Store<STORE>;
  using T = typename S::T;
  using E = typename S::E;
  constexpr int N = npt(STORE), TX = tile_x(STORE), W = warps_per_block(STORE);
  constexpr bool REF = S::kElements;
  __shared__ T s_dm[kNodeThreads], s_fx[kNodeThreads], s_fy[kNodeThreads];
  const int tile = blockIdx.x / W, w = blockIdx.x % W;
  const int tx = tile % p.tiles_x, ty = tile / p.tiles_x;
  const int r = threadIdx.x / TX;
  const int x0 = tx * TX;
  const int x = x0 + threadIdx.x % TX, y = ty * p.tile_y + w + W * r;
  const bool active = x < p.nx && y < p.ny;
  T drho = T(0), fpx = T(0), fpy = T(0);
  bool solid = false;
  pdl_wait();
  if (active) {
    constexpr bool AA = MODE == kModeAAPush;
    const E* src = static_cast<const E*>(p.src);
    // sources of the directions with xi_y = 1 and -1 (uniform across a warp)
    int yd = y - 1, yu = y + 1;
    bool wall_d = false, wall_u = false;
    if (yd < 0) {
      wall_d = p.bc_y != kBcPeriodic;
      yd = wall_d ? y : yd + p.ny;
    }
    if (yu >= p.ny) {
      wall_u = p.bc_y != kBcPeriodic;
      yu = wall_u ? y : yu - p.ny;
    }
    int xl = x - 1, xr = x + 1;
    bool inlet = false, outlet = false;
    if (xl < 0) {
      inlet = p.bc_x != kBcPeriodic;
      xl = inlet ? x : xl + p.nx;
    }
    if (xr >= p.nx) {
      // in place, the last column's values come from the side copy
      outlet = p.bc_x == kBcInletConvective || (AA && p.bc_x != kBcPeriodic);
      xr = p.bc_x == kBcPeriodic ? xr - p.nx : p.nx - 1;  // zero gradient: the last column
    }
    const long long i = (long long)y * p.pitch + x;
    const uint8_t m = p.mask[i];
    T h[9];
    if constexpr (MODE == kModeAALocal) {
#pragma unroll
      for (int a = 0; a < 9; ++a) h[a] = S::in_e(src[(long long)a * p.plane + i], a);
      if (x == 0 || x == p.nx - 1) aa_local_boundary<S, true>(p, h, x, y, true);
    } else {
#pragma unroll
      for (int a = 0; a < 9; ++a) {
        const bool wall = cy(a) == 1 ? wall_d : (cy(a) == -1 ? wall_u : false);
        const int as = wall ? mirror_y(a) : a;
        const int ys = cy(a) == 1 ? yd : (cy(a) == -1 ? yu : y);
        const int xs = cx(a) == 1 ? xl : (cx(a) == -1 ? xr : x);
        // in place, a value from beyond an open side would be another node's slot
        const bool none = AA && ((inlet && cx(a) == 1) || (outlet && cx(a) == -1));
        h[a] = none ? T(0)
                    : S::in_e(src[(long long)(AA ? opposite(as) : as) * p.plane + (long long)ys * p.pitch + xs], a);
      }
      if (inlet) {
#pragma unroll
        for (int a = 0; a < 9; ++a)
          if (cx(a) == 1) {
            const int as = (cy(a) == 1 && wall_d) || (cy(a) == -1 && wall_u) ? mirror_y(a) : a;
            h[a] = consts<T>(p).heq_in[as] - sref<S>(p, a);
          }
      }
      if (outlet) {
#pragma unroll
        for (int a = 0; a < 9; ++a)
          if (cx(a) == -1) {
            const bool wall = cy(a) == 1 ? wall_d : (cy(a) == -1 ? wall_u : false);
            const int ys = cy(a) == 1 ? yd : (cy(a) == -1 ? yu : y);
            const int as = wall ? mirror_y(a) : a;
            h[a] = AA ? outlet_ghost_aa<S, true>(p, as, ys, true)
                      : outlet_ghost<S>(p, src, as, ys, true) - sref<S>(p, a);
          }
      }
    }
    Macro<T> q;
    if (COLL == kTrt && p.force_free && m == 0) {
      if (interior_tile<STORE>(p, tx, ty)) {
        q = macros<T, kFree, REF>(p, h, 0, x, y);
        collide_trt<T, kFree, REF>(p, h, q);
      } else {
        q = macros<T, kFluid, REF>(p, h, 0, x, y);
        collide_trt<T, kFluid, REF>(p, h, q);
      }
    } else if (COLL == kTrt) {
      q = macros<T, kGeneral, REF>(p, h, m, x, y);
      collide_trt<T, kGeneral, REF>(p, h, q);
    } else {
      if constexpr (REF) {
#pragma unroll
        for (int a = 0; a < 9; ++a) h[a] = h[a] + sref<S>(p, a);
      }
      q = macros<T>(p, h, m, x, y);
      collide_mrt<T>(p, h, q);
      if constexpr (REF) {
#pragma unroll
        for (int a = 0; a < 9; ++a) h[a] = h[a] - sref<S>(p, a);
      }
    }
    if (!sound_density(q.rho)) atomicOr(p.flag, 1);
    drho = q.drho;
    if (m) {
      solid = true;
      fpx = q.fpx;
      fpy = q.fpy;
    }
    const bool sr = S::kSixteen && p.stochastic;
    unsigned nb[1];
    round_words(p, x, y, round_bits(unsigned(p.t), p.round_key), sr, nb);
    E* dst = static_cast<E*>(p.dst);
    typename S::R e[9];
#pragma unroll
    for (int a = 0; a < 9; ++a) e[a] = S::round_e(h[a], a, nb[0], x & 1, sr);
    if constexpr (MODE == kModeAAPush) {
      const bool inside = x >= 1 && x <= p.nx - 2 && y >= 1 && y <= p.ny - 2;
#pragma unroll
      for (int a = 0; a < 9; ++a) {
        if (inside)
          store_raw<S>(dst + (long long)a * p.plane + i + cy(a) * p.pitch + cx(a), e[a]);
        else
          push_one<S>(p, dst, a, x, y, e[a]);
      }
      if (x == p.nx - 1 && p.bc_x != kBcPeriodic) {
        push_outlet_copy<S>(p, dst, 3, y, e[3]);
        push_outlet_copy<S>(p, dst, 6, y, e[6]);
        push_outlet_copy<S>(p, dst, 7, y, e[7]);
      }
    } else {
#pragma unroll
      for (int a = 0; a < 9; ++a)
        store_raw<S>(dst + (long long)(MODE == kModeAALocal ? opposite(a) : a) * p.plane + i, e[a]);
      if (MODE == kModeAALocal && x == p.nx - 1 && p.bc_x != kBcPeriodic) {
        typename S::R* z = static_cast<typename S::R*>(p.z);
        z[0 * p.ny + y] = e[3];
        z[1 * p.ny + y] = e[6];
        z[2 * p.ny + y] = e[7];
      }
    }
  }
  pdl_trigger();
  s_dm[threadIdx.x] = drho;
  s_fx[threadIdx.x] = fpx;
  s_fy[threadIdx.x] = fpy;
  const int any_solid = __syncthreads_or(solid);
  if (threadIdx.x >= kLanes) return;
  const int rows = blockDim.x / TX;
  T dm = T(0), fx = T(0), fy = T(0);
  for (int j = 0; j < rows; ++j) {
    const int at = j * TX + N * threadIdx.x;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      dm += s_dm[at + k];
      if (any_solid) {
        fx -= s_fx[at + k];
        fy -= s_fy[at + k];
      }
    }
  }
  double bfx = 0.0, bfy = 0.0;
  dm = warp_sum(dm);
  if (any_solid) {
    bfx = warp_sum(double(fx));
    bfy = warp_sum(double(fy));
  }
  if (threadIdx.x == 0) {
    double* out = p.partials + 3ll * p.n_tiles * w + tile;
    out[0] = bfx;
    out[p.n_tiles] = bfy;
    *reinterpret_cast<T*>(out + 2ll * p.n_tiles) = dm;
  }
}

}  // namespace vplbm
