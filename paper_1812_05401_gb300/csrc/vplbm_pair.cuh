// Two fused steps in one launch, for grids whose step is bound by HBM.
#pragma once

#include "vplbm_device.cuh"

namespace vplbm {

// A block takes one tile, kPairRows rows at a time, through the steps of pp.a
// and pp.b: it collides those rows and the ring of nodes around them (the
// ring's results are worked out again by the tiles they belong to), keeps the
// populations the rows pull next in shared memory, and pulls, collides and
// stores those. The grid's populations are then read and written once for two
// steps. Every node's values and every tile's record sums are formed by the
// single step's code in its order: two steps here give the bits of two single
// steps.
//
// A single step is bound by HBM (16384 x 4096: 0.734 ms, 73 bytes a node); this
// kernel moves half the bytes and is bound by instruction issue and latency at 24
// warps an SM (IPC 1.95). Per step of long calls, single against pair: 16384 x
// 4096 734 -> 578 us, 4096 x 1024 49.4 -> 43.1, 6048 x 2016 (SRT, convective)
// 142 -> 126 (pair_rule has the line). What it took, on 16384 x 4096 with a moving
// cylinder (us a step of batches of 20 with their mask updates and the field read
// at the end; tiles of one part):
// - direct loads in the first step, a row at a time: 766 (latency); the rows on
//   their way to shared memory at once (stage): 658;
// - a lane's nodes one after the other (collide_row's ONE): 110 registers become
//   80 without spills, three blocks an SM: 602 (two blocks an SM: 673; two nodes
//   at a time, 80 bytes of spills: 622);
// - edges and masks of both rows loaded ahead: 602, not kept.
// Tiles of 32 rows in two parts, for the order of the single step's records,
// cost 625 against 598 as tiles of 16, on the same measure.
//
// Shared memory: v[a][j][TX], the populations of direction a that row j of the
// part pulls, by the column they come from, and halo[side][k][j], those that
// enter the row from the columns beside it (directions 1, 5, 8 from the left and
// 3, 6, 7 from the right). Only what is pulled is kept: 75 KB with the sums,
// three blocks an SM; 16 rows for that reason (18 rows of work for 16). A wall's
// mirror image is put in the place of the row beyond it, so that the second step
// pulls without regard to y.
template <int STORE>
struct PairTile {
  static constexpr int TX = tile_x(STORE), R = kPairRows;
  typename Store<STORE>::T v[9][R][TX];
  typename Store<STORE>::T halo[2][3][R];
  TileSums<STORE> sums[2];
  typename Store<STORE>::T dm[2][threads_per_block(STORE)];  // a thread's sum of drho in each step
};

// The first step of halo node j (row y0 + j of the grid) of a side, one node per lane.
// ANY: the node may lie beside or beyond a boundary.
template <int STORE, bool ANY>
__device__ __forceinline__ void pair_halo(const StepParams& p, PairTile<STORE>& sm, int side, int j, int x0, int y0) {
  using S = Store<STORE>;
  using T = typename S::T;
  using E = typename S::E;
  constexpr int TX = PairTile<STORE>::TX, R = kPairRows;
  const E* src = static_cast<const E*>(p.src);
  int x = side ? x0 + TX : x0 - 1, y = y0 + j;
  T h[9];
  bool inlet = false;
  if (ANY) {
    if (y < 0 || y >= p.ny) {
      if (p.bc_y != kBcPeriodic || y > p.ny) return;
      y = y < 0 ? y + p.ny : y - p.ny;
    }
    if (x < 0) {
      inlet = p.bc_x != kBcPeriodic;
      x += p.nx;
    } else if (x >= p.nx) {
      if (p.bc_x != kBcPeriodic) return;  // the outlet's values come from the last column
      x = 0;
    }
  }
  if (ANY && inlet) {
#pragma unroll
    for (int a = 0; a < 9; ++a) h[a] = consts<T>(p).heq_in[a];
  } else {
    if (ANY) {
      pull_node<S>(p, src, x, y, h);
    } else {
      const E* at = src + (long long)y * p.pitch + x;
#pragma unroll
      for (int a = 0; a < 9; ++a) h[a] = S::in_e(at[(long long)a * p.plane - cy(a) * p.pitch - cx(a)], a);
    }
    const uint8_t m = p.mask[(long long)y * p.pitch + x];
    Macro<T> q;
    if (m == 0 && free_form<STORE>(p, x, y)) {
      q = macros<T, kFree>(p, h, 0, x, y);
      collide_trt<T, kFree>(p, h, q);
    } else {
      q = macros<T, kGeneral>(p, h, m, x, y);
      collide_trt<T, kGeneral>(p, h, q);
    }
    if (!sound_density(q.rho)) atomicOr(p.flag, 1);
  }
  const T o0 = side ? h[3] : h[1], o1 = side ? h[6] : h[5], o2 = side ? h[7] : h[8];
  T(*to)[R] = sm.halo[side];
  if (j >= 0 && j < R) to[0][j] = o0;
  if (j + 1 < R) to[1][j + 1] = o1;
  if (j >= 1) to[2][j - 1] = o2;
  if (ANY && p.bc_y != kBcPeriodic) {
    if (y == 0) to[1][j] = o2;
    if (y == p.ny - 1 && j < R) to[2][j] = o1;
  }
}

// 16 bytes from global to shared memory, in the background (past L1).
__device__ __forceinline__ void copy16_async(void* to, const void* from) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(unsigned(__cvta_generic_to_shared(to))), "l"(from)
               : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void copy_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
}

template <int STORE>
__global__ void __launch_bounds__(threads_per_block(STORE), min_blocks_per_sm(STORE))
    pair_step_kernel(const __grid_constant__ PairParams pp) {
  using S = Store<STORE>;
  using T = typename S::T;
  using E = typename S::E;
  constexpr int N = npt(STORE), TX = tile_x(STORE), W = warps_per_block(STORE), R = kPairRows;
  static_assert(STORE == kF32, "the first step's populations are kept as FP32 elements hold them");
  extern __shared__ __align__(16) unsigned char raw[];
  PairTile<STORE>& sm = *reinterpret_cast<PairTile<STORE>*>(raw);
  const StepParams& p = pp.a;  // grid, boundaries and constants: those of pp.b as well
  const int lane = threadIdx.x, warp = threadIdx.y;
  const int tile = blockIdx.x, tx = tile % p.tiles_x, ty = tile / p.tiles_x;
  const int x0 = tx * TX, xb = x0 + lane * N;
  const bool free = p.force_free && interior_tile<STORE>(p, tx, ty);
  int y0 = ty * p.tile_y;  // first row of the part at work
  const E* src = static_cast<const E*>(p.src);
  E* dst = static_cast<E*>(pp.b.dst);
  // What a thread adds up for each step's record, out of the registers that the
  // rows' populations need: the densities in shared memory, the forces (rarely
  // touched: solid nodes) in local memory.
  const int tid = lane + warp * kLanes;
  volatile T force[2][2] = {{T(0), T(0)}, {T(0), T(0)}};
  bool solid[2] = {false, false};
  sm.dm[0][tid] = sm.dm[1][tid] = T(0);
  auto sums_of = [&](int step, unsigned mw) {
    RowSums<T> sums;
    sums.dm = sm.dm[step][tid];
    if (mw) {
      sums.fx = force[step][0];
      sums.fy = force[step][1];
    }
    return sums;
  };
  auto keep_sums = [&](int step, unsigned mw, const RowSums<T>& sums) {
    sm.dm[step][tid] = sums.dm;
    if (mw) {
      force[step][0] = sums.fx;
      force[step][1] = sums.fy;
      solid[step] = true;
    }
  };
  pdl_wait();

  // Where the warp keeps direction a of row j (of the part) in the first step,
  // its source before and its result after the collision: the place the row's
  // result is pulled from, which no other row uses; for what leaves the part,
  // the place of what enters there (the ring rows' results, which the same
  // warps put there afterwards, or the wall's mirror images).
  auto place = [&](int a, int j) -> T* {
    const int jj = j + cy(a);
    const bool out = cy(a) == 1 ? jj == R : (cy(a) == -1 ? jj < 0 : false);
    return &sm.v[out ? mirror_y(a) : a][out ? j : jj][lane * N];
  };
  // The source rows of the warp's own rows, all on their way at once.
  auto stage = [&](int j, auto gen) {
    constexpr bool GEN = decltype(gen)::value;
    int y = y0 + j;
    if (GEN && y >= p.ny) {
      if (p.bc_y != kBcPeriodic || y > p.ny) y = -1;
      else y = 0;
    }
    if (!GEN || (y >= 0 && xb < p.nx)) {
#pragma unroll
      for (int a = 0; a < 9; ++a) copy16_async(place(a, j), source_row<S, GEN>(p, src, a, y) + xb);
    }
    copy_commit();
  };
  // First step of the warp's rows: two of the part, and a ring row (-1 and R)
  // for the first and the last warp.
  auto first = [&](auto gen, const auto& el) {
    constexpr bool GEN = decltype(gen)::value;
    const bool lane_active = !GEN || xb < p.nx;
#pragma unroll 1
    for (int r = 0; r < 3; ++r) {
      if (r == 2 && warp != 0 && warp != W - 1) break;
      const int j = r < 2 ? warp + r * W : (warp == 0 ? -1 : R);
      int y = y0 + j;
      bool own = r < 2;
      if (GEN && (y < 0 || y >= p.ny)) {
        if (p.bc_y != kBcPeriodic || y > p.ny) continue;
        y = y < 0 ? y + p.ny : y - p.ny;
        own = false;
      }
      const T edge = el.value(p, src, x0, y, lane);
      const unsigned mw = lane_active ? mask_word<N>(p.mask + (long long)y * p.pitch + xb) : 0u;
      T v[9][N], h[N][9];
      if (r < 2) {
        if (r == 0)
          copy_wait<1>();
        else
          copy_wait<0>();
#pragma unroll
        for (int a = 0; a < 9; ++a) {
          S::load_h(place(a, j), v[a], a);
#pragma unroll
          for (int k = 0; k < N; ++k)
            if (GEN && !lane_active) v[a][k] = T(0);
        }
      } else {
        load_row<S, N, GEN>(p, src, xb, y, lane_active, v);
      }
      shift_row<S, N, GEN>(p.nx, x0, lane, v, edge, h);
      if (!lane_active) continue;
      RowSums<T> sums = sums_of(0, mw);
      collide_row<STORE, kTrt, GEN, N, true>(p, h, mw, xb, y, r == 2 || GEN ? free_form<STORE>(p, x0, y) : free, sums);
      if (own) keep_sums(0, mw, sums);
      auto keep = [&](int a, int jj, int from) {
        T o[N];
#pragma unroll
        for (int k = 0; k < N; ++k) o[k] = h[k][from];
        S::store_h(&sm.v[a][jj][lane * N], o, a, nullptr, false);
      };
#pragma unroll
      for (int a = 0; a < 9; ++a) {
        const int jj = j + cy(a);
        if (cy(a) == 0 ? j >= 0 && j < R : (cy(a) == 1 ? jj < R : jj >= 0)) keep(a, jj, a);
      }
      if (GEN && p.bc_y != kBcPeriodic) {
        if (y == 0) {
          keep(2, j, 4);
          keep(5, j, 8);
          keep(6, j, 7);
        }
        if (y == p.ny - 1 && own) {
          keep(4, j, 2);
          keep(7, j, 6);
          keep(8, j, 5);
        }
      }
    }
  };
  // second step, row j of the part
  auto second = [&](int j, auto gen) {
    constexpr bool GEN = decltype(gen)::value;
    const int y = y0 + j;
    const bool last = GEN && x0 + TX >= p.nx;
    const bool lane_active = !GEN || xb < p.nx;
    T v[9][N], h[N][9];
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      S::load_h(&sm.v[a][j][lane * N], v[a], a);
#pragma unroll
      for (int k = 0; k < N; ++k)
        if (GEN && !lane_active) v[a][k] = T(0);
    }
    T edge = T(0);
    if (lane < (last ? 3 : 6)) {
      edge = sm.halo[lane < 3 ? 0 : 1][lane % 3][j];
    } else if (last && lane >= 6 && lane < 9) {
      // what enters the domain's last column
      const int m = lane - 6, a = m == 0 ? 3 : (m == 1 ? 6 : 7);
      if (p.bc_x == kBcPeriodic) {
        edge = sm.halo[1][m][j];
      } else {
        edge = sm.v[a][j][p.nx - 1 - x0];  // zero gradient: the last column's
        if (p.bc_x == kBcInletConvective) {
          // the state of the first step once more, and the second step's from it
          int as = a, ys = y - (m == 0 ? 0 : (m == 1 ? 1 : -1));
          if (ys < 0 || ys >= p.ny) {
            if (p.bc_y == kBcPeriodic) {
              ys = ys < 0 ? ys + p.ny : ys - p.ny;
            } else {
              as = m == 1 ? 7 : 6;
              ys = y;
            }
          }
          const Consts<T>& c = consts<T>(p);
          const T g = outlet_ghost<S>(p, src, as, ys, false);
          edge = mul(mad(c.u_conv, edge, g), c.conv_inv);
          static_cast<T*>(pp.b.ghost_dst)[(long long)(as == 3 ? 0 : (as == 6 ? 1 : 2)) * p.ny + ys] = edge;
        }
      }
    }
    shift_row<S, N, GEN>(p.nx, x0, lane, v, edge, h);
    if (!lane_active) return;
    const long long i = (long long)y * p.pitch + xb;
    const unsigned mw = mask_word<N>(pp.b.mask + i);
    RowSums<T> sums = sums_of(1, mw);
    collide_row<STORE, kTrt, GEN, N, true>(pp.b, h, mw, xb, y, free, sums);
    keep_sums(1, mw, sums);
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      T o[N];
#pragma unroll
      for (int k = 0; k < N; ++k) o[k] = h[k][a];
      S::store_h(dst + (long long)a * p.plane + i, o, a, nullptr, false);
    }
  };

  // Rows of the tile by warp as in the single step; the ring's columns go to
  // the second and third warp, a node per lane.
  static_assert(R == 2 * W, "two rows a warp");
#pragma unroll 1
  for (const int end = min(p.ny, y0 + p.tile_y);;) {
    // neither the part nor its ring of nodes touches a boundary
    const bool inner = x0 >= 2 && x0 + TX <= p.nx - 2 && y0 >= 2 && y0 + R <= p.ny - 2;
    if (inner) {
      stage(warp, std::false_type());
      stage(warp + W, std::false_type());
      if ((warp == 1 || warp == 2) && lane < R + 2) pair_halo<STORE, false>(p, sm, warp - 1, lane - 1, x0, y0);
      first(std::false_type(), EdgeLane<S, TX, false>(p, src, x0, lane));
    } else {
      stage(warp, std::true_type());
      stage(warp + W, std::true_type());
      if ((warp == 1 || warp == 2) && lane < R + 2) pair_halo<STORE, true>(p, sm, warp - 1, lane - 1, x0, y0);
      first(std::true_type(), EdgeLane<S, TX, true>(p, src, x0, lane));
    }
    __syncthreads();
    if (inner) {
#pragma unroll 1
      for (int j = warp; j < R; j += W) second(j, std::false_type());
    } else {
#pragma unroll 1
      for (int j = warp; j < R && y0 + j < p.ny; j += W) second(j, std::true_type());
    }
    y0 += R;
    if (y0 >= end) break;
    __syncthreads();  // the next part takes the places over
  }
  y0 = ty * p.tile_y;
  pdl_trigger();
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    RowSums<T> sums;
    sums.dm = sm.dm[k][tid];
    if (solid[k]) {
      sums.fx = force[k][0];
      sums.fy = force[k][1];
      sums.solid = true;
    }
    warp_records<STORE>(p, sums, sm.sums[k]);
  }
  __syncthreads();
  if (lane == 0 && warp < 2)
    tile_record<STORE>(p, tile, x0, y0, true, sm.sums[warp], warp == 0 ? pp.a.partials : pp.b.partials);
}

inline cudaError_t prepare_pair(const void* kernel, int bytes) {
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  return e == cudaSuccess ? cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                                 cudaSharedmemCarveoutMaxShared)
                          : e;
}

}  // namespace vplbm
