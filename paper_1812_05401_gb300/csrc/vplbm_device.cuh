// Device side of the VP-LBM solver: storage traits, the fused
// stream-penalize-collide-reduce step, the mask update for moving bodies, and
// the initialisation / read-back kernels. Included by one translation unit per
// storage type (kernels_<storage>.cu).
//
// Arithmetic form. The kernel works on offsets h_alpha = f_alpha - w_alpha
// (w: the D2Q9 weights). Equilibrium, forcing and both collision operators are
// affine in f with the rest state w as a fixed point, so colliding h is the
// same operation, and it keeps the small deviations from the rest state out of
// the rounding of numbers near w. FP32 and the 16-bit storage forms store h
// itself; FP64 storage stores f.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "vplbm_params.h"
#include "vplbm_reduce.cuh"

namespace vplbm {

// D2Q9 velocity set in the order of Eq. vecteurs_D2Q9.
__device__ __host__ constexpr int cx(int a) {
  return a == 1 || a == 5 || a == 8 ? 1 : (a == 3 || a == 6 || a == 7 ? -1 : 0);
}
__device__ __host__ constexpr int cy(int a) {
  return a == 2 || a == 5 || a == 6 ? 1 : (a == 4 || a == 7 || a == 8 ? -1 : 0);
}
// Direction with the same x and opposite y velocity (free-slip reflection).
__device__ __host__ constexpr int mirror_y(int a) {
  return a == 2 ? 4 : a == 4 ? 2 : a == 5 ? 8 : a == 8 ? 5 : a == 6 ? 7 : a == 7 ? 6 : a;
}
// Direction with the opposite velocity.
__device__ __host__ constexpr int opposite(int a) {
  return a == 0 ? 0 : (a <= 4 ? (a + 1) % 4 + 1 : (a - 3) % 4 + 5);
}
// Weights, Eq. anex_eq19.
template <class T>
__device__ __forceinline__ constexpr T wgt(int a) {
  return a == 0 ? T(4.0 / 9.0) : (a <= 4 ? T(1.0 / 9.0) : T(1.0 / 36.0));
}

// ---------------------------------------------------------------------------
// Storage traits: E is the element in HBM, T the arithmetic type, h = f - w
// the offset of a population. An element holds h - ref (sref), ref a
// per-direction reference: FP32 elements hold h, FP64 elements h + w = f. The
// fused step works on the elements' values e = h - ref as they are (load_h,
// store_h, round_e, in_e: no reference), its collision taking ref through
// constant sums; in, out, to_f64 and from_f64 convert to and from h and f.
// ---------------------------------------------------------------------------
template <int S> struct Store;
template <> struct Store<kF64> {
  using E = double;
  using T = double;
  static constexpr bool kSixteen = false;
  static constexpr bool kElements = true;
  static __device__ __forceinline__ T in(E e, int, T ref) { return e + ref; }
  static __device__ __forceinline__ T in_e(E e, int) { return e; }
  static __device__ __forceinline__ E out(T h, int, T ref) { return h - ref; }
  static __device__ __forceinline__ double to_f64(const E* p, int, T) { return *p; }
  static __device__ __forceinline__ void from_f64(E* p, double f, int, T) { *p = f; }
  // npt = 2 consecutive elements as one 16-byte access
  static __device__ __forceinline__ void load_h(const E* p, T e[2], int) {
    const double2 v = *reinterpret_cast<const double2*>(p);
    e[0] = v.x;
    e[1] = v.y;
  }
  static __device__ __forceinline__ void store_h(E* p, const T e[2], int, const unsigned*, bool) {
    *reinterpret_cast<double2*>(p) = make_double2(e[0], e[1]);
  }
  // one element's raw bits, rounded as store_h rounds it (r: the word of the
  // element's node pair, k: the element's place in the lane's vector)
  using R = unsigned long long;
  static __device__ __forceinline__ R round_e(T e, int, unsigned, int, bool) {
    return static_cast<R>(__double_as_longlong(e));
  }
};
template <> struct Store<kF32> {
  // FP32 elements hold the offsets h = f - w as well: the same bytes as f,
  // with the rounding step of |h| <~ 0.1 instead of that of f ~ w.
  using E = float;
  using T = float;
  static constexpr bool kSixteen = false;
  static constexpr bool kElements = false;
  static __device__ __forceinline__ T in(E e, int, T) { return e; }
  static __device__ __forceinline__ T in_e(E e, int) { return e; }
  static __device__ __forceinline__ E out(T h, int, T) { return h; }
  static __device__ __forceinline__ double to_f64(const E* p, int a, T) {
    return wgt<double>(a) + double(*p);
  }
  static __device__ __forceinline__ void from_f64(E* p, double f, int a, T) {
    *p = float(f - wgt<double>(a));
  }
  // npt = 4 consecutive elements as one 16-byte access
  static __device__ __forceinline__ void load_h(const E* p, T h[4], int) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    h[0] = v.x;
    h[1] = v.y;
    h[2] = v.z;
    h[3] = v.w;
  }
  static __device__ __forceinline__ void store_h(E* p, const T h[4], int, const unsigned*, bool) {
    *reinterpret_cast<float4*>(p) = make_float4(h[0], h[1], h[2], h[3]);
  }
  using R = unsigned;
  static __device__ __forceinline__ R round_e(T h, int, unsigned, int, bool) { return __float_as_uint(h); }
};
// 16-bit offset forms: npt = 4 elements as one 8-byte access.
// Multipliers deriving each direction's rounding bits from the node's word
// (distinct odd constants: a bijection of 32-bit words per direction).
__device__ __forceinline__ constexpr unsigned round_mul(int a) {
  return a == 0 ? 0x9e3779b1u : a == 1 ? 0x85ebca77u : a == 2 ? 0xc2b2ae3du : a == 3 ? 0x27d4eb2fu
       : a == 4 ? 0x165667b1u : a == 5 ? 0xd3a2646du : a == 6 ? 0xfd7046c5u : a == 7 ? 0xb55a4f09u
       : 0x68e31da5u;
}

// Packed conversion of two FP32 values to two 16-bit values in one register
// (lo in the low half, the lower address): round to nearest even.
__device__ __forceinline__ unsigned pack_f16_rn(float lo, float hi) {
  unsigned d;
  asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}
__device__ __forceinline__ unsigned pack_bf16_rn(float lo, float hi) {
  unsigned d;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}
// Stochastic rounding of two FP32 values to two 16-bit values with the
// hardware conversion (cvt.rs): each result adds random bits below its kept
// significand bits and truncates, so the magnitude rounds up with probability
// equal to its distance from the lower neighbour. The low result takes its
// bits from the low half of rbits, the high result from the high half (the
// lowest 13 bits of each half for FP16, all 16 for BF16).
__device__ __forceinline__ unsigned pack_f16_rs(float lo, float hi, unsigned rbits) {
  unsigned d;
  asm("cvt.rs.f16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(hi), "f"(lo), "r"(rbits));
  return d;
}
__device__ __forceinline__ unsigned pack_bf16_rs(float lo, float hi, unsigned rbits) {
  unsigned d;
  asm("cvt.rs.bf16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(hi), "f"(lo), "r"(rbits));
  return d;
}
// Rounding bits of direction a for a pair of nodes: their 32-bit pair word
// times the direction's odd constant; the low half goes to the first node,
// the high half to the second. The pair word is a full 32-bit hash, so the
// two halves are independent; each direction's bits are a different
// bijection of them.
__device__ __forceinline__ unsigned pair_bits(unsigned pair_word, int a) {
  return pair_word * round_mul(a);
}

// 16-bit offset forms: npt = 4 elements as one 8-byte access; an element
// holds h - ref (FP32 arithmetic on both sides of the conversion).
template <class H>
struct Store16 {
  using E = H;
  using T = float;
  static constexpr bool kSixteen = true;
  static constexpr bool kElements = true;
};
template <> struct Store<kF16> : Store16<__half> {
  static __device__ __forceinline__ void load_h(const E* p, T e[4], int) {
    unpack(*reinterpret_cast<const uint2*>(p), e);
  }
  static __device__ __forceinline__ void unpack(const uint2 v, T e[4]) {
    const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&v.x));
    const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&v.y));
    e[0] = a.x;
    e[1] = a.y;
    e[2] = b.x;
    e[3] = b.y;
  }
  // r[j]: the rounding word of node pair j (stochastic rounding only)
  static __device__ __forceinline__ void store_h(E* p, const T e[4], int a, const unsigned* r,
                                                 bool sr) {
    uint2 v;
    if (sr) {
      v.x = pack_f16_rs(e[0], e[1], pair_bits(r[0], a));
      v.y = pack_f16_rs(e[2], e[3], pair_bits(r[1], a));
    } else {
      v.x = pack_f16_rn(e[0], e[1]);
      v.y = pack_f16_rn(e[2], e[3]);
    }
    *reinterpret_cast<uint2*>(p) = v;
  }
  static __device__ __forceinline__ T in_e(E e, int) { return __half2float(e); }
  static __device__ __forceinline__ T in(E e, int, T ref) { return __half2float(e) + ref; }
  static __device__ __forceinline__ E out(T h, int, T ref) { return __float2half_rn(h - ref); }
  // one element as store_h rounds it (the packed conversions round each half alike)
  using R = unsigned short;
  static __device__ __forceinline__ R round_e(T e, int a, unsigned r, int k, bool sr) {
    return sr ? (unsigned short)(pack_f16_rs(e, 0.f, pair_bits(r, a) >> (16 * (k & 1))) & 0xffffu)
              : __half_as_ushort(__float2half_rn(e));
  }
  // f of a stored element: w + (element + ref), the offset as the kernel forms it
  static __device__ __forceinline__ double to_f64(const E* p, int a, T ref) {
    return wgt<double>(a) + double(__half2float(*p) + ref);
  }
  static __device__ __forceinline__ void from_f64(E* p, double f, int a, T ref) {
    *p = __double2half(f - wgt<double>(a) - double(ref));
  }
};
template <> struct Store<kBF16> : Store16<__nv_bfloat16> {
  static __device__ __forceinline__ void load_h(const E* p, T e[4], int) {
    unpack(*reinterpret_cast<const uint2*>(p), e);
  }
  // a bf16 is the upper half of an FP32: widening is a shift or a mask
  static __device__ __forceinline__ void unpack(const uint2 v, T e[4]) {
    e[0] = __uint_as_float(v.x << 16);
    e[1] = __uint_as_float(v.x & 0xffff0000u);
    e[2] = __uint_as_float(v.y << 16);
    e[3] = __uint_as_float(v.y & 0xffff0000u);
  }
  static __device__ __forceinline__ void store_h(E* p, const T e[4], int a, const unsigned* r,
                                                 bool sr) {
    uint2 v;
    if (sr) {
      v.x = pack_bf16_rs(e[0], e[1], pair_bits(r[0], a));
      v.y = pack_bf16_rs(e[2], e[3], pair_bits(r[1], a));
    } else {
      v.x = pack_bf16_rn(e[0], e[1]);
      v.y = pack_bf16_rn(e[2], e[3]);
    }
    *reinterpret_cast<uint2*>(p) = v;
  }
  static __device__ __forceinline__ T in_e(E e, int) { return __bfloat162float(e); }
  static __device__ __forceinline__ T in(E e, int, T ref) { return __bfloat162float(e) + ref; }
  static __device__ __forceinline__ E out(T h, int, T ref) { return __float2bfloat16_rn(h - ref); }
  using R = unsigned short;
  static __device__ __forceinline__ R round_e(T e, int a, unsigned r, int k, bool sr) {
    return sr ? (unsigned short)(pack_bf16_rs(e, 0.f, pair_bits(r, a) >> (16 * (k & 1))) & 0xffffu)
              : __bfloat16_as_ushort(__float2bfloat16_rn(e));
  }
  static __device__ __forceinline__ double to_f64(const E* p, int a, T ref) {
    return wgt<double>(a) + double(__bfloat162float(*p) + ref);
  }
  static __device__ __forceinline__ void from_f64(E* p, double f, int a, T ref) {
    *p = __double2bfloat16(f - wgt<double>(a) - double(ref));
  }
};

// The reference of direction a's stored elements: an element holds h - sref
// (16-bit stores: h - h_ref; FP64: h + w = f; FP32: h).
template <class S>
__device__ __forceinline__ typename S::T sref(const StepParams& p, int a) {
  if constexpr (S::kSixteen)
    return p.cf.h_ref[a];
  else if constexpr (S::kElements)
    return -wgt<typename S::T>(a);
  else
    return typename S::T(0);
}

// Scalar offset load/store of one population of direction a.
template <class S>
__device__ __forceinline__ typename S::T load_h(const StepParams& p, const typename S::E* ptr, int a) {
  return S::in(*ptr, a, sref<S>(p, a));
}
template <class S>
__device__ __forceinline__ void store_h(const StepParams& p, typename S::E* ptr, typename S::T h, int a) {
  *ptr = S::out(h, a, sref<S>(p, a));
}

// Random bits of the stochastic rounding: the MurmurHash3 32-bit finalizer
// (Appleby) of the node's index mixed with the step's key gives one uniform
// 32-bit word per node; direction alpha uses the word times a distinct odd
// constant (a bijection of 32-bit words, so each direction's bits are again
// uniform) and takes its top bits.
__device__ __forceinline__ unsigned round_bits(unsigned counter, unsigned key) {
  unsigned h = counter ^ key;
  h ^= h >> 16;
  h *= 0x85ebca6bu;
  h ^= h >> 13;
  h *= 0xc2b2ae35u;
  h ^= h >> 16;
  return h;
}



// Explicitly rounded operations. The collision is written with them so that
// no instance of it depends on which products the compiler contracts: a node
// has the same bits in every kernel (single, in-place, grouped, paired steps)
// that computes it.
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mad(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double mad(double a, double b, double c) { return __fma_rn(a, b, c); }

// Convective outlet (Section 3.3, after Yang): the ghost column x = nx of
// direction as (3, 6 or 7), row ys, advanced by the implicit upwind step of
// dg/dt + U_c dg/dx = 0 from the last column's f*(t):
// g^t = (g^{t-1} + U_c f*(nx - 1)) / (1 + U_c), in offsets (the weights cancel).
// The step's one reader of each entry writes g^t to ghost_dst (write = true).
template <class S>
__device__ __forceinline__ typename S::T outlet_ghost(const StepParams& p,
                                                      const typename S::E* src, int as, int ys,
                                                      bool write) {
  using T = typename S::T;
  const Consts<T>& c = consts<T>(p);
  const long long gi = (long long)(as == 3 ? 0 : (as == 6 ? 1 : 2)) * p.ny + ys;
  const T f_last = load_h<S>(p, src + (long long)as * p.plane + (long long)ys * p.pitch + (p.nx - 1), as);
  const T g = mul(mad(c.u_conv, f_last, static_cast<const T*>(p.ghost_src)[gi]), c.conv_inv);
  if (write && p.ghost_dst) static_cast<T*>(p.ghost_dst)[gi] = g;
  return g;
}

// The same ghost value in the in-place (AA) push step, whose store no longer
// holds the last column intact (the neighbours' pushes overwrite it): the
// stored f*(nx - 1) comes from the side copy z that the local step wrote.
// ESP: the value as an element (offset minus the reference) instead of an
// offset; the convective state itself is always kept as offsets.
template <class S, bool ESP = false>
__device__ __forceinline__ typename S::T outlet_ghost_aa(const StepParams& p, int as, int ys,
                                                         bool write) {
  using T = typename S::T;
  const long long gi = (long long)(as == 3 ? 0 : (as == 6 ? 1 : 2)) * p.ny + ys;
  const typename S::E ze = static_cast<const typename S::E*>(p.z)[gi];
  if (p.bc_x != kBcInletConvective)  // zero gradient
    return ESP ? S::in_e(ze, as) : S::in(ze, as, sref<S>(p, as));
  const T f_last = S::in(ze, as, sref<S>(p, as));
  const Consts<T>& c = consts<T>(p);
  const T g = mul(mad(c.u_conv, f_last, static_cast<const T*>(p.ghost_src)[gi]), c.conv_inv);
  if (write && p.ghost_dst) static_cast<T*>(p.ghost_dst)[gi] = g;
  return ESP ? g - sref<S>(p, as) : g;
}

// ---------------------------------------------------------------------------
// Pull with boundary conditions (streaming, left-hand side of Eq. LatticeBoltz)
// ---------------------------------------------------------------------------
template <class S, int A>
__device__ __forceinline__ typename S::T pull_bc(const StepParams& p, const typename S::E* src,
                                                 int x, int y) {
  using T = typename S::T;
  int as = A;
  int xs = x - cx(A);
  int ys = y - cy(A);
  if (ys < 0 || ys >= p.ny) {
    if (p.bc_y == kBcPeriodic) {
      ys = ys < 0 ? ys + p.ny : ys - p.ny;
    } else {  // free slip: the mirror of the population that left this row
      as = mirror_y(A);
      ys = y;
    }
  }
  if (xs < 0 || xs >= p.nx) {
    if (p.bc_x == kBcPeriodic) {
      xs = xs < 0 ? xs + p.nx : xs - p.nx;
    } else if (xs < 0) {  // inlet ghost column at f_eq(1, u_in)
      const Consts<T>& c = consts<T>(p);
      return as == A ? c.heq_in[A] : c.heq_in[mirror_y(A)];
    } else if (p.bc_x == kBcInletConvective) {  // read only: the step writes the state
      return outlet_ghost<S>(p, src, as, ys, false);
    } else {  // zero-gradient outlet ghost column
      xs = p.nx - 1;
    }
  }
  return load_h<S>(p, src + (long long)as * p.plane + (long long)ys * p.pitch + xs, as);
}

// The nine pulled populations of node (x, y), one at a time with the boundary
// rules (the diagnostics' scalar pull; the fused step pulls whole vectors).
template <class S>
__device__ __forceinline__ void pull_node(const StepParams& p, const typename S::E* src, int x,
                                          int y, typename S::T h[9]) {
  h[0] = pull_bc<S, 0>(p, src, x, y);
  h[1] = pull_bc<S, 1>(p, src, x, y);
  h[2] = pull_bc<S, 2>(p, src, x, y);
  h[3] = pull_bc<S, 3>(p, src, x, y);
  h[4] = pull_bc<S, 4>(p, src, x, y);
  h[5] = pull_bc<S, 5>(p, src, x, y);
  h[6] = pull_bc<S, 6>(p, src, x, y);
  h[7] = pull_bc<S, 7>(p, src, x, y);
  h[8] = pull_bc<S, 8>(p, src, x, y);
}

// ---------------------------------------------------------------------------
// Density, implicit velocity and penalization force of one node
// (Eqs. density, velocity, 17 and 18).
//   d = j + rho g / 2 - rho u_s,  u = u_s + d / (rho (1 + a)),
//   f_pen = -kappa d,  a = chi/(2 eta),  kappa = (chi/eta)/(1 + a).
// This is Eq. 18 rewritten so that neither u - u_s nor a rho u_s appear:
// the 1/eta factor never multiplies a rounding error.
// ---------------------------------------------------------------------------
// Correctly rounded reciprocal.
__device__ __forceinline__ float recip(float v) { return __frcp_rn(v); }
__device__ __forceinline__ double recip(double v) { return __drcp_rn(v); }

// Whether a density is sound: positive and below 1e30 (a NaN is not). FP64: the
// bits of positive numbers are ordered as the numbers, and integer comparisons
// leave the FP64 pipe alone.
__device__ __forceinline__ bool sound_density(float rho) { return rho > 0.f && rho < 1e30f; }
__device__ __forceinline__ bool sound_density(double rho) {
  return static_cast<unsigned long long>(__double_as_longlong(rho)) - 1ull <
         static_cast<unsigned long long>(__double_as_longlong(1e30)) - 1ull;
}

template <class T>
struct Macro {
  T drho, rho, ux, uy, fpx, fpy, Fx, Fy;
};

template <class T>
__device__ __forceinline__ void solid_velocity(const StepParams& p, uint8_t m, int x, int y,
                                               T& usx, T& usy) {
  if (m == kStaticSolid) {
    if (p.us) {
      const long long i = (long long)y * p.pitch + x;
      if (sizeof(T) == 8) {
        const double2 v = reinterpret_cast<const double2*>(p.us)[i];
        usx = T(v.x);
        usy = T(v.y);
      } else {
        const float2 v = reinterpret_cast<const float2*>(p.us)[i];
        usx = T(v.x);
        usy = T(v.y);
      }
    }
  } else if (m <= p.n_bodies) {
    const T* b = consts<T>(p).body[m - 1];
    const T dx = T(x) - b[0];
    const T dy = T(y) - b[1];
    usx = mad(-b[4], dy, b[2]);
    usy = mad(b[4], dx, b[3]);
  }
  // any other label (only a caller-written mask can hold one) is solid at rest
}

// Sum and difference of the offsets of the opposite pair k ((1,3), (2,4),
// (5,7), (6,8)) whose values the kernel holds in ha, hb: offsets themselves,
// or (REF) the elements of a 16-bit or FP64 store. The 16-bit reference is odd
// in xi, so the pair sum of the elements is that of the offsets, and the
// difference is decoded with the pair's reference difference (exact in FP32).
// FP64 elements are f = h + w: the difference needs no decoding, and the sum
// takes 2 w off one of the two, which is exact near w. The step thus converts
// only the rest population between f and h: 12 of some 115 FP64 operations a
// node less than with every population converted in and out, on a kernel bound
// by the FP64 pipe (with sound_density 1024 x 256 57.3 -> 50.2 us per step,
// 128 x 128 Couette 12.6 -> 12.1); one rounding less per population, and errors
// against plain 64-bit torch as before (mean over 12 seeds, force of the Couette
// box 4.2e-12 / 4.1e-12, its fields 1.8e-14).
template <class T, bool REF>
__device__ __forceinline__ T pair_s(T ha, T hb, int k) {
  if constexpr (REF && sizeof(T) == 8)
    return (ha - T(2) * wgt<T>(k < 2 ? 1 : 5)) + hb;
  else
    return ha + hb;
}
// The rest population's offset and back.
template <class T, bool REF>
__device__ __forceinline__ T rest_in(T h0) {
  return REF && sizeof(T) == 8 ? h0 - wgt<T>(0) : h0;
}
template <class T, bool REF>
__device__ __forceinline__ T rest_out(T h0) {
  return REF && sizeof(T) == 8 ? h0 + wgt<T>(0) : h0;
}
template <class T, bool REF>
__device__ __forceinline__ T pair_d(const Consts<T>& c, T ha, T hb, int k) {
  if constexpr (REF && sizeof(T) == 4)
    return (ha - hb) + c.r_d[k];
  else
    return ha - hb;
}

// Forms of a node's step. kGeneral: any node. A fluid node (m = 0) without
// body force (g = 0), for which Eqs. 17 and 18 reduce to f_pen = 0 and
// u = j / rho, needs half the operations: kFluid gives the general form's
// bits, which computes the same values through zero terms; kFree rounds the
// collision's last products in another order. Which of the two a node takes
// depends on its place alone (free_form), not on the kernel.
// REF: h holds the stored elements of a 16-bit (h - h_ref) or FP64 (h + w) store.
enum { kGeneral = 0, kFluid = 1, kFree = 2 };

template <class T, int FORM = kGeneral, bool REF = false>
__device__ __forceinline__ Macro<T> macros(const StepParams& p, const T h[9], uint8_t m, int x,
                                           int y) {
  Macro<T> r;
  const Consts<T>& c = consts<T>(p);
  // sums and differences of opposite populations (the two-rate collision
  // reuses them)
  const T s13 = pair_s<T, REF>(h[1], h[3], 0), s24 = pair_s<T, REF>(h[2], h[4], 1);
  const T s57 = pair_s<T, REF>(h[5], h[7], 2), s68 = pair_s<T, REF>(h[6], h[8], 3);
  const T d13 = pair_d<T, REF>(c, h[1], h[3], 0), d24 = pair_d<T, REF>(c, h[2], h[4], 1);
  const T d57 = pair_d<T, REF>(c, h[5], h[7], 2), d68 = pair_d<T, REF>(c, h[6], h[8], 3);
  r.drho = rest_in<T, REF>(h[0]) + ((s13 + s24) + (s57 + s68));
  r.rho = T(1) + r.drho;
  const T jx = d13 + (d57 - d68);
  const T jy = d24 + (d57 + d68);
  if constexpr (FORM != kGeneral) {
    const T inv = recip(r.rho);
    r.ux = mul(jx, inv);
    r.uy = mul(jy, inv);
    r.fpx = r.fpy = r.Fx = r.Fy = T(0);
    return r;
  }
  T usx = T(0), usy = T(0), a = T(0), kap = T(0);
  if (m) {
    a = c.a_s;
    kap = c.kappa_s;
    solid_velocity<T>(p, m, x, y, usx, usy);
  }
  const T gx = c.gx, gy = c.gy;
  const T half = mul(T(0.5), r.rho);
  const T dx = mad(-r.rho, usx, mad(half, gx, jx));
  const T dy = mad(-r.rho, usy, mad(half, gy, jy));
  const T inv = recip(mul(r.rho, T(1) + a));
  r.ux = mad(dx, inv, usx);
  r.uy = mad(dy, inv, usy);
  r.fpx = mul(-kap, dx);
  r.fpy = mul(-kap, dy);
  r.Fx = mad(r.rho, gx, r.fpx);
  r.Fy = mad(r.rho, gy, r.fpy);
  return r;
}

// ---------------------------------------------------------------------------
// Collision on offsets, two-rate form.
// The printed S relaxes the even moments (e, eps, p_xx, p_xy: symmetric under
// xi -> -xi) at s+ = s_n and the odd ones (q_x, q_y) at s- = s_q; the rates of
// rho, j_x and j_y do not change the result (rho = rho_eq, and j* = j + F for
// any rate because m_eq uses the half-force velocity). Splitting each pair of
// opposite populations into its even and odd parts, h+- = (h_a +- h_abar)/2,
// Eq. equa_lbl_mrt with Eq. Guo2 is then, per pair,
//   h*_a    = h_a    + P + Q,   h*_abar = h_abar + P - Q,
//   P = -s+ (h+ - heq+) + (1 - s+/2) G+,   Q = -s- (h- - heq-) + (1 - s-/2) G-,
// with heq+ = w (drho - 1.5 rho u.u + 4.5 rho (xi.u)^2), heq- = 3 w rho xi.u,
// G+ = w (9 (xi.u)(xi.F) - 3 u.F), G- = 3 w xi.F (the even and odd parts of
// Eq. Guo2's F_a), and for the rest population h*_0 = (1 - s+) h_0 + w_0 K,
// K = s+ (drho - 1.5 rho u.u) - 3 (1 - s+/2) u.F. SRT with Eq. Guo1 is the
// same with s+ = s- = 1/tau. This is the moment-space operator rearranged,
// not an approximation of it.
// On stored elements (REF) the update of a pair is the same, e*_a = e_a + P + Q.
// 16-bit: e = h - r with r odd in xi, so the pair sums s and the rest population
// need no decoding, the differences d take the pair's constant (pair_d). FP64:
// e = h + w with w even in xi, so d needs none, and s and the rest population
// take the weights off (pair_s, rest_in, rest_out).
// ---------------------------------------------------------------------------
// w: the weight of the pair's directions.
template <class T, int FORM>
__device__ __forceinline__ void trt_pair(T& ha, T& hb, T s, T d, T xu, T xF, T K, T w, T aw, T bw,
                                         T amw, T bmw, T hsp, T hsm) {
  // P = w (s+ heq+ + c+ G+) - (s+/2) s and Q = w (s- heq- + c- G-) - (s-/2) d;
  // without a force G+- = 0
  T P, Q;
  if constexpr (FORM == kFree) {
    P = mad(-hsp, s, mad(xu, mul(aw, xu), mul(K, w)));
    Q = mad(amw, xu, -mul(hsm, d));
  } else if constexpr (FORM == kFluid) {
    P = mad(-hsp, s, mad(K, w, mul(xu, mul(aw, xu))));
    Q = mad(-hsm, d, mul(amw, xu));
  } else {
    P = mad(-hsp, s, mad(K, w, mul(xu, mad(aw, xu, mul(bw, xF)))));
    Q = mad(-hsm, d, mad(amw, xu, mul(bmw, xF)));
  }
  ha = ha + (P + Q);
  hb = hb + (P - Q);
}

template <class T, int FORM = kGeneral, bool REF = false>
__device__ __forceinline__ void collide_trt(const StepParams& p, T h[9], const Macro<T>& q) {
  const Consts<T>& c = consts<T>(p);
  const T ux = q.ux, uy = q.uy, Fx = q.Fx, Fy = q.Fy, rho = q.rho;
  const T w9 = T(1.0 / 9.0), w36 = T(1.0 / 36.0);
  const T uu = mad(ux, ux, mul(uy, uy));
  const T e = mad(-mul(T(1.5), rho), uu, q.drho);
  const T K = FORM != kGeneral ? mul(c.t_sp, e) : mad(c.t_sp, e, -mul(c.t_c3p, mad(ux, Fx, mul(uy, Fy))));
  const T a9 = mul(c.t_a[0], rho), a36 = mul(c.t_a[1], rho);
  const T am9 = mul(c.t_am[0], rho), am36 = mul(c.t_am[1], rho);
  // the pair sums and differences as macros() formed them
  const T s13 = pair_s<T, REF>(h[1], h[3], 0), s24 = pair_s<T, REF>(h[2], h[4], 1);
  const T s57 = pair_s<T, REF>(h[5], h[7], 2), s68 = pair_s<T, REF>(h[6], h[8], 3);
  const T d13 = pair_d<T, REF>(c, h[1], h[3], 0), d24 = pair_d<T, REF>(c, h[2], h[4], 1);
  const T d57 = pair_d<T, REF>(c, h[5], h[7], 2), d68 = pair_d<T, REF>(c, h[6], h[8], 3);
  h[0] = rest_out<T, REF>(mad(T(4.0 / 9.0), K, mul(c.t_1msp, rest_in<T, REF>(h[0]))));
  trt_pair<T, FORM>(h[1], h[3], s13, d13, ux, Fx, K, w9, a9, c.t_b[0], am9, c.t_bm[0], c.t_hsp, c.t_hsm);
  trt_pair<T, FORM>(h[2], h[4], s24, d24, uy, Fy, K, w9, a9, c.t_b[0], am9, c.t_bm[0], c.t_hsp, c.t_hsm);
  trt_pair<T, FORM>(h[5], h[7], s57, d57, ux + uy, Fx + Fy, K, w36, a36, c.t_b[1], am36, c.t_bm[1],
                    c.t_hsp, c.t_hsm);
  trt_pair<T, FORM>(h[6], h[8], s68, d68, uy - ux, Fy - Fx, K, w36, a36, c.t_b[1], am36, c.t_bm[1],
                    c.t_hsp, c.t_hsm);
}

// MRT (Eq. equa_lbl_mrt with Lu forcing, Eq. Guo2), on the moments of h, for
// rates without the two-rate structure.
// m = M h with M of Eq. eq1.7; since M w = (1, -2, 1, 0, ...), the equilibrium
// moments of h are m_eq(rho, u) - M w. The forcing moments M F are
// (0, 6 u.F, -6 u.F, F_x, -F_x, F_y, -F_y, 2 (u F_x - v F_y), u F_y + v F_x).
// Rates of the conserved moments (rho, j_x, j_y) do not change the result
// (j* = j + F for any rate, because m_eq uses the half-force velocity).
// f* = M^-1 m* with M^-1 = M^T diag(1/9, 1/36, 1/36, 1/6, 1/12, 1/6, 1/12, 1/4, 1/4).
// Products that are rounded, or whose fusing shows in the result, are written
// out (mul, mad); the plain ones are by powers of two, exact either way.
template <class T>
__device__ __forceinline__ void collide_mrt(const StepParams& p, T h[9], const Macro<T>& q) {
  const Consts<T>& c = consts<T>(p);
  const T s1 = c.s_e, s2 = c.s_eps, s4 = c.s_qx, s6 = c.s_qy, s7 = c.s_pxx, s8 = c.s_pxy;
  const T sum14 = (h[1] + h[2]) + (h[3] + h[4]);
  const T sum58 = (h[5] + h[6]) + (h[7] + h[8]);
  const T e = -T(4) * h[0] - sum14 + T(2) * sum58;
  const T eps = T(4) * h[0] - T(2) * sum14 + sum58;
  const T jx = (h[1] - h[3]) + (h[5] - h[6]) + (h[8] - h[7]);
  const T qx = T(2) * (h[3] - h[1]) + (h[5] - h[6]) + (h[8] - h[7]);
  const T jy = (h[2] - h[4]) + (h[5] + h[6]) - (h[7] + h[8]);
  const T qy = T(2) * (h[4] - h[2]) + (h[5] + h[6]) - (h[7] + h[8]);
  const T pxx = (h[1] - h[2]) + (h[3] - h[4]);
  const T pxy = (h[5] - h[6]) + (h[7] - h[8]);

  const T rho = q.rho, ux = q.ux, uy = q.uy, Fx = q.Fx, Fy = q.Fy;
  const T uu = mad(ux, ux, mul(uy, uy));
  const T uF = mad(ux, Fx, mul(uy, Fy));
  const T rho3 = mul(T(3), rho), rux = mul(rho, ux);
  const T e_eq = mad(rho3, uu, -T(2) * q.drho);
  const T eps_eq = mad(-rho3, uu, q.drho);

  const T es = mad(mul(T(1) - T(0.5) * s1, T(6)), uF, mad(-s1, e - e_eq, e));
  const T epss = mad(-mul(T(1) - T(0.5) * s2, T(6)), uF, mad(-s2, eps - eps_eq, eps));
  const T jxs = jx + Fx;
  const T jys = jy + Fy;
  const T qxs = mad(-(T(1) - T(0.5) * s4), Fx, mad(-s4, qx + rux, qx));
  const T qys = mad(-(T(1) - T(0.5) * s6), Fy, mad(-s6, mad(rho, uy, qy), qy));
  const T pxxs = mad((T(1) - T(0.5) * s7) * T(2), mad(ux, Fx, -mul(uy, Fy)),
                     mad(-s7, mad(-rho, mad(ux, ux, -mul(uy, uy)), pxx), pxx));
  const T pxys = mad(T(1) - T(0.5) * s8, mad(ux, Fy, mul(uy, Fx)), mad(-s8, mad(-rux, uy, pxy), pxy));

  const T a0 = mul(q.drho, T(1.0 / 9.0));
  const T a1 = mul(es, T(1.0 / 36.0));
  const T a2 = mul(epss, T(1.0 / 36.0));
  const T a4 = mul(qxs, T(1.0 / 12.0));
  const T a6 = mul(qys, T(1.0 / 12.0));
  const T a7 = pxxs * T(0.25);
  const T a8 = pxys * T(0.25);
  // j*/6 - q*/6 (directions 1..4) and j*/6 + q*/12 (5..8)
  const T x14 = mad(jxs, T(1.0 / 6.0), -T(2) * a4), x58 = mad(jxs, T(1.0 / 6.0), a4);
  const T y14 = mad(jys, T(1.0 / 6.0), -T(2) * a6), y58 = mad(jys, T(1.0 / 6.0), a6);

  const T b14 = a0 - a1 - T(2) * a2;  // common part of directions 1..4
  const T b58 = a0 + T(2) * a1 + a2;  // common part of directions 5..8
  h[0] = a0 - T(4) * a1 + T(4) * a2;
  h[1] = b14 + x14 + a7;
  h[2] = b14 + y14 - a7;
  h[3] = b14 - x14 + a7;
  h[4] = b14 - y14 - a7;
  h[5] = b58 + x58 + y58 + a8;
  h[6] = b58 - x58 + y58 - a8;
  h[7] = b58 - x58 - y58 + a8;
  h[8] = b58 + x58 - y58 - a8;
}

// ---------------------------------------------------------------------------
// The fused time step of one tile: (32 N) x tile_y nodes, N = npt(STORE). Lane
// l of warp w takes nodes x0 + N l .. x0 + N l + N - 1 of rows y0 + w + W r,
// r = 0..rows_per_warp-1, W = warps_per_block(STORE).
//
// Every direction is pulled with one N-element vector load per lane: a
// direction with xi_x = +1 takes its first node's value from the lane to the
// left (warp shuffle), one with xi_x = -1 its last node's value from the lane
// to the right. The values from beside the tile come with one more load, one
// value per lane (EdgeLane), and are handed to the edge lanes by shuffles.
// Interior tiles (no boundary within one node) do nothing else. Tiles touching
// a boundary (GEN) also remap: the source row of each direction (periodic wrap
// or free-slip mirror, uniform across the warp), the values from beside the
// tile (periodic wrap, inlet ghost, outlet copy), and those entering the
// domain's last column; lanes past the last column load and store nothing.
// ---------------------------------------------------------------------------
// The value of direction as from (xs, ys), through the x boundary rules (the
// caller has applied the y rules to as and ys).
// AA: the push step reads f*_as(xs, ys) from the opposite slot of the source
// node (where the local step put it).
// ESP: the value as an element (offset minus the reference), as the fused step
// works on them; the reference is even in xi_y, so the mirrored source as of a
// free-slip wall has the pulled direction's reference.
template <class S, bool AA = false, bool ESP = false>
__device__ __forceinline__ typename S::T edge_pull(const StepParams& p, const typename S::E* src,
                                                   int as, int ys, int xs) {
  using T = typename S::T;
  if (xs < 0 || xs >= p.nx) {
    if (p.bc_x == kBcPeriodic) {
      xs %= p.nx;
      if (xs < 0) xs += p.nx;
    } else if (xs < 0) {  // inlet ghost column at f_eq(1, u_in)
      const T h = consts<T>(p).heq_in[as];
      return ESP ? h - sref<S>(p, as) : h;
    } else if (AA) {
      return outlet_ghost_aa<S, ESP>(p, as, ys, xs == p.nx);
    } else if (p.bc_x == kBcInletConvective) {
      // xs == nx: the last column's own pull (the entry's one reader)
      const T g = outlet_ghost<S>(p, src, as, ys, xs == p.nx);
      return ESP ? g - sref<S>(p, as) : g;
    } else {  // zero-gradient outlet ghost column
      xs = p.nx - 1;
    }
  }
  const typename S::E e = src[(long long)(AA ? opposite(as) : as) * p.plane + (long long)ys * p.pitch + xs];
  return ESP ? S::in_e(e, as) : S::in(e, as, sref<S>(p, as));
}

// Place of a direction with xi_x != 0 among the three of its side (1, 5, 8 and
// 3, 6, 7: xi_y = 0, 1, -1).
__device__ __forceinline__ constexpr int side_slot(int a) {
  return a == 1 || a == 3 ? 0 : (a == 5 || a == 6 ? 1 : 2);
}

// The values that enter a row of a tile from beside it, one per lane (so that
// one load covers them all): lanes 0..2 take directions 1, 5, 8 from x0 - 1,
// lanes 3..5 directions 3, 6, 7 from x0 + TX, and in the tile of the domain's
// last column (GEN) lanes 6..8 directions 3, 6, 7 from beyond that column. As
// one load per direction by the edge lane alone they were six more loads per
// row of an interior tile, and in boundary tiles nine instances of the
// boundary rules, run one after the other. With it, per step: 1001 x 701 BF16
// 19.7 -> 14.1 us, 4096 x 1024 FP32 58.3 -> 51.7 and FP16 43.8 -> 36.7 us,
// 16384 x 4096 FP16 0.483 -> 0.454 ms, 32 mixed solves 344 -> 284 us (with
// the branch-free rows of collide_row for FP32). The interior tiles' source is
// kept as one pointer: worked out anew in each row, the 16384 x 4096 FP16 step
// took 0.51 ms; three loads by lanes 0 and 31 in place of one and six shuffles
// likewise.
template <class S, int TX, bool GEN, bool AA = false>
struct EdgeLane {
  using T = typename S::T;
  using E = typename S::E;
  const E* at;  // interior tiles: the lane's source in row 0 (null: none)
  __device__ __forceinline__ EdgeLane(const StepParams& p, const E* src, int x0, int lane) {
    if constexpr (!GEN) {
      const int m = lane % 3;
      const bool left = lane < 3;
      const int a = m == 0 ? (left ? 1 : 3) : (m == 1 ? (left ? 5 : 6) : (left ? 8 : 7));
      const int dy = m == 0 ? 0 : (m == 1 ? -1 : 1);
      at = lane < 6 ? src + (long long)(AA ? opposite(a) : a) * p.plane + dy * p.pitch + (left ? x0 - 1 : x0 + TX)
                    : nullptr;
    }
  }
  __device__ __forceinline__ T value(const StepParams& p, const E* src, int x0, int y, int lane) const {
    if constexpr (!GEN) {
      return at ? S::in_e(at[(long long)y * p.pitch], 1) : T(0);
    } else {
      const bool last = x0 + TX >= p.nx;
      if (lane >= 9 || (last ? lane >= 3 && lane < 6 : lane >= 6)) return T(0);
      const int m = lane % 3;
      const bool left = lane < 3;
      int as = m == 0 ? (left ? 1 : 3) : (m == 1 ? (left ? 5 : 6) : (left ? 8 : 7));
      int ys = y - (m == 0 ? 0 : (m == 1 ? 1 : -1));
      if (ys < 0 || ys >= p.ny) {
        if (p.bc_y == kBcPeriodic) {
          ys = ys < 0 ? ys + p.ny : ys - p.ny;
        } else {
          as = m == 1 ? (left ? 8 : 7) : (left ? 5 : 6);
          ys = y;
        }
      }
      return edge_pull<S, AA, true>(p, src, as, ys, left ? x0 - 1 : (last ? p.nx : x0 + TX));
    }
  }
};

// Node k's pulled value from the loaded vectors: its own place's for xi_x = 0,
// the left or right neighbour's for xi_x = +-1 (from the neighbouring lane, or
// from edge, the values of EdgeLane, at the row's ends).
template <class S, int N, bool GEN>
__device__ __forceinline__ void shift_row(int nx, int x0, int lane, const typename S::T (&v)[9][N],
                                          typename S::T edge, typename S::T (&h)[N][9]) {
  using T = typename S::T;
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    if (cx(a) == 0) {
#pragma unroll
      for (int k = 0; k < N; ++k) h[k][a] = v[a][k];
    } else if (cx(a) == 1) {
      const T left = __shfl_up_sync(0xffffffffu, v[a][N - 1], 1);
      const T e = __shfl_sync(0xffffffffu, edge, side_slot(a));
      h[0][a] = lane == 0 ? e : left;
#pragma unroll
      for (int k = 1; k < N; ++k) h[k][a] = v[a][k - 1];
    } else {
      const T right = __shfl_down_sync(0xffffffffu, v[a][0], 1);
      const T e = __shfl_sync(0xffffffffu, edge, 3 + side_slot(a));
#pragma unroll
      for (int k = 0; k < N - 1; ++k) h[k][a] = v[a][k + 1];
      h[N - 1][a] = lane == kLanes - 1 ? e : right;
      if (GEN && x0 + kLanes * N >= nx) {  // the domain's last column
        const T beyond = __shfl_sync(0xffffffffu, edge, 6 + side_slot(a));
        const int at = nx - 1 - x0 - lane * N;
#pragma unroll
        for (int k = 0; k < N; ++k)
          if (k == at) h[k][a] = beyond;
      }
    }
  }
}

// The source row of direction a's population for row y of nodes.
template <class S, bool GEN, bool AA = false>
__device__ __forceinline__ const typename S::E* source_row(const StepParams& p, const typename S::E* src, int a,
                                                           int y) {
  int as = a, ys = y - cy(a);
  if (GEN && (ys < 0 || ys >= p.ny)) {
    if (p.bc_y == kBcPeriodic) {
      ys = ys < 0 ? ys + p.ny : ys - p.ny;
    } else {  // free slip: the mirror of the population that left this row
      as = mirror_y(a);
      ys = y;
    }
  }
  return src + (long long)(AA ? opposite(as) : as) * p.plane + (long long)ys * p.pitch;
}

// The values a lane's N nodes xb .. xb + N - 1 of row y pull, by the column
// they come from.
template <class S, int N, bool GEN, bool AA = false>
__device__ __forceinline__ void load_row(const StepParams& p, const typename S::E* src, int xb, int y,
                                         bool lane_active, typename S::T (&v)[9][N]) {
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    const typename S::E* row = source_row<S, GEN, AA>(p, src, a, y);
    if (!GEN || lane_active) {
      S::load_h(row + xb, v[a], a);
    } else {
#pragma unroll
      for (int k = 0; k < N; ++k) v[a][k] = typename S::T(0);
    }
  }
}

// The pulled populations of a lane's N nodes xb .. xb + N - 1 of row y.
template <class S, int N, bool GEN, bool AA = false>
__device__ __forceinline__ void pull_row(const StepParams& p, const typename S::E* src,
                                         const EdgeLane<S, kLanes * N, GEN, AA>& el, int x0, int y, int lane,
                                         bool lane_active, typename S::T (&h)[N][9]) {
  using T = typename S::T;
  const T edge = el.value(p, src, x0, y, lane);
  T v[9][N];
  load_row<S, N, GEN, AA>(p, src, x0 + lane * N, y, lane_active, v);
  shift_row<S, N, GEN>(p.nx, x0, lane, v, edge, h);
}

// ---------------------------------------------------------------------------
// In-place (AA-pattern) streaming on one buffer. A push step reads each
// population from the opposite slot of its source node (where the previous
// local step put it), collides, and writes f*_a to slot a of the node it
// streams to; a local step reads a node's own slots, collides, and writes f*_a
// to the node's opposite slot. Every location a push step reads is written by
// the same node, after its read: in the vector layout both happen in the lane
// that owns the location's aligned vector (or the edge lane's extra element),
// so the buffer can be updated in place. Each value is rounded with the bits
// of its node, direction and step, as the A/B scheme rounds it, so the two
// schemes give bitwise the same populations.
// ---------------------------------------------------------------------------
template <class S>
__device__ __forceinline__ void store_raw(typename S::E* p, typename S::R w) {
  *reinterpret_cast<typename S::R*>(p) = w;
}
// N raw elements to an aligned vector (16 bytes, or 8 for 16-bit storage)
template <class S, int N>
__device__ __forceinline__ void store_raw_vec(typename S::E* p, const typename S::R (&w)[N]) {
  if constexpr (sizeof(typename S::E) == 2) {
    uint2 v;
    v.x = unsigned(w[0]) | (unsigned(w[1 % N]) << 16);
    v.y = unsigned(w[2 % N]) | (unsigned(w[3 % N]) << 16);
    *reinterpret_cast<uint2*>(p) = v;
  } else if constexpr (sizeof(typename S::E) == 4) {
    *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1 % N], w[2 % N], w[3 % N]);
  } else {
    *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(w[0], w[1 % N]);
  }
}
template <class R>
__device__ __forceinline__ R shfl_up_raw(R v) {
  if constexpr (sizeof(R) == 8)
    return __shfl_up_sync(0xffffffffu, v, 1);
  else
    return R(__shfl_up_sync(0xffffffffu, unsigned(v), 1));
}
template <class R>
__device__ __forceinline__ R shfl_down_raw(R v) {
  if constexpr (sizeof(R) == 8)
    return __shfl_down_sync(0xffffffffu, v, 1);
  else
    return R(__shfl_down_sync(0xffffffffu, unsigned(v), 1));
}

// Slot of the value that a push step sends out through an open x side:
// lost[side][k][y], side 0 = x = nx - 1 (alpha = 1, 5, 8), 1 = x = 0 (alpha = 3, 6, 7).
__device__ __forceinline__ long long lost_index(const StepParams& p, int a, int y, bool left) {
  const int k = left ? (a == 3 ? 0 : (a == 6 ? 1 : 2)) : (a == 1 ? 0 : (a == 5 ? 1 : 2));
  return (long long)((left ? 3 : 0) + k) * p.ny + y;
}

// Where a push step puts f*_a of node (x, y): the pull's boundary rules read
// backwards (periodic wrap; a free-slip wall returns it as mirror_y(a) in the
// same row at x + cx(a)). Returns false when it leaves through an open x side.
__device__ __forceinline__ bool push_target(const StepParams& p, int a, int x, int y, int* ap,
                                            int* xt, int* yt) {
  *ap = a;
  *xt = x + cx(a);
  *yt = y + cy(a);
  if (*yt < 0 || *yt >= p.ny) {
    if (p.bc_y == kBcPeriodic) {
      *yt = *yt < 0 ? *yt + p.ny : *yt - p.ny;
    } else {
      *ap = mirror_y(a);
      *yt = y;
    }
  }
  if (*xt < 0 || *xt >= p.nx) {
    if (p.bc_x != kBcPeriodic) return false;
    *xt = *xt < 0 ? *xt + p.nx : *xt - p.nx;
  }
  return true;
}

template <class S>
__device__ __forceinline__ void push_one(const StepParams& p, typename S::E* buf, int a, int x, int y,
                                         typename S::R e) {
  int ap, xt, yt;
  if (push_target(p, a, x, y, &ap, &xt, &yt))
    store_raw<S>(buf + (long long)ap * p.plane + (long long)yt * p.pitch + xt, e);
  else
    store_raw<S>(static_cast<typename S::E*>(p.lost) + lost_index(p, a, y, x + cx(a) < 0), e);
}

// The outlet's ghost column (a copy of the last column) streams its
// populations alpha = 3, 6, 7 into the last column: the push step writes them
// where the next local step reads them (that step turns them into the
// zero-gradient or convective ghost values).
template <class S>
__device__ __forceinline__ void push_outlet_copy(const StepParams& p, typename S::E* buf, int as,
                                                 int y, typename S::R e) {
  int ap = as, yt = y + cy(as);
  if (yt < 0 || yt >= p.ny) {
    if (p.bc_y == kBcPeriodic) {
      yt = yt < 0 ? yt + p.ny : yt - p.ny;
    } else {
      ap = mirror_y(as);
      yt = y;
    }
  }
  store_raw<S>(buf + (long long)ap * p.plane + (long long)yt * p.pitch + (p.nx - 1), e);
}

// Interior tiles: the push of direction a as one aligned vector store per
// lane (the x-shifted element from the neighbouring lane); the edge lanes
// write the element that crosses into the next tile, and leave the one the
// neighbouring tile writes.
template <class S, int N>
__device__ __forceinline__ void push_dir_vec(const StepParams& p, typename S::E* buf, int a, int xb,
                                             int y, int lane, const typename S::R (&e)[N]) {
  using R = typename S::R;
  typename S::E* row = buf + (long long)a * p.plane + (long long)(y + cy(a)) * p.pitch;
  if (cx(a) == 0) {
    store_raw_vec<S, N>(row + xb, e);
  } else if (cx(a) == 1) {  // element j of this lane's vector receives node xb + j - 1
    R w[N];
    w[0] = shfl_up_raw(e[N - 1]);
#pragma unroll
    for (int j = 1; j < N; ++j) w[j] = e[j - 1];
    if (lane == 0) {
#pragma unroll
      for (int j = 1; j < N; ++j) store_raw<S>(row + xb + j, w[j]);
    } else {
      store_raw_vec<S, N>(row + xb, w);
    }
    if (lane == kLanes - 1) store_raw<S>(row + xb + N, e[N - 1]);
  } else {  // element j receives node xb + j + 1
    R w[N];
#pragma unroll
    for (int j = 0; j < N - 1; ++j) w[j] = e[j + 1];
    w[N - 1] = shfl_down_raw(e[0]);
    if (lane == kLanes - 1) {
#pragma unroll
      for (int j = 0; j < N - 1; ++j) store_raw<S>(row + xb + j, w[j]);
    } else {
      store_raw_vec<S, N>(row + xb, w);
    }
    if (lane == 0) store_raw<S>(row + xb - 1, e[0]);
  }
}

// Local step at the open x sides: the values the A/B pull would take from the
// ghost columns. Inlet: f_eq(1, u_in) for the directions entering at x = 0.
// Outlet: h holds the ghost column's copy of f*(nx - 1) (pushed there by the
// previous push step); the convective outlet advances its state from it.
// ESP: h holds elements (offsets minus the reference) instead of offsets.
template <class S, bool ESP = false>
__device__ __forceinline__ void aa_local_boundary(const StepParams& p, typename S::T h[9], int x,
                                                  int y, bool write) {
  using T = typename S::T;
  if (p.bc_x == kBcPeriodic) return;
  const Consts<T>& c = consts<T>(p);
#pragma unroll
  for (int a = 1; a < 9; ++a) {
    if (!((cx(a) == 1 && x == 0) || (cx(a) == -1 && x == p.nx - 1))) continue;
    int as = a, ys = y - cy(a);
    if (ys < 0 || ys >= p.ny) {
      if (p.bc_y == kBcPeriodic) {
        ys = ys < 0 ? ys + p.ny : ys - p.ny;
      } else {
        as = mirror_y(a);
        ys = y;
      }
    }
    if (cx(a) == 1) {
      h[a] = ESP ? c.heq_in[as] - sref<S>(p, a) : c.heq_in[as];
    } else if (p.bc_x == kBcInletConvective) {
      const long long gi = (long long)(as == 3 ? 0 : (as == 6 ? 1 : 2)) * p.ny + ys;
      const T f_last = ESP ? h[a] + sref<S>(p, a) : h[a];
      const T g = mul(mad(c.u_conv, f_last, static_cast<const T*>(p.ghost_src)[gi]), c.conv_inv);
      if (write) static_cast<T*>(p.ghost_dst)[gi] = g;
      h[a] = ESP ? g - sref<S>(p, a) : g;
    }
  }
}

// f*_a(x, y) as stored, whatever the scheme and phase (for the diagnostics:
// export, momentum exchange, outlet state).
template <class S>
__device__ __forceinline__ typename S::E fstar_e(const StepParams& p, const typename S::E* buf, int a,
                                                 int x, int y) {
  if (p.mode == kModeAB) return buf[(long long)a * p.plane + (long long)y * p.pitch + x];
  if (p.mode == kModeAAPush)  // after a local step: the node's opposite slot
    return buf[(long long)opposite(a) * p.plane + (long long)y * p.pitch + x];
  int ap, xt, yt;  // after a push step: where it was pushed
  if (push_target(p, a, x, y, &ap, &xt, &yt))
    return buf[(long long)ap * p.plane + (long long)yt * p.pitch + xt];
  return static_cast<const typename S::E*>(p.lost)[lost_index(p, a, y, x + cx(a) < 0)];
}

// What a thread adds up for a step's record over the rows it collides: sum of
// drho, and the force on its solid nodes (at most 16, or 32 of a 16-bit store,
// whose blocks have half the warps), in the arithmetic type.
template <class T>
struct RowSums {
  T dm = T(0), fx = T(0), fy = T(0);
  bool solid = false;
};

// The N mask bytes of a lane's nodes, byte k for node k (kept in one register:
// the collision's registers are the kernel's tightest budget).
template <int N>
__device__ __forceinline__ unsigned mask_word(const uint8_t* m) {
  return N == 4 ? *reinterpret_cast<const unsigned*>(m) : unsigned(*reinterpret_cast<const unsigned short*>(m));
}

// Whether the tile at column tx and row ty of tiles touches no boundary: none
// of its nodes pulls from outside the grid.
template <int STORE>
__device__ __forceinline__ bool interior_tile(const StepParams& p, int tx, int ty) {
  const int x0 = tx * tile_x(STORE), y0 = ty * p.tile_y;
  return x0 >= 1 && x0 + tile_x(STORE) <= p.nx - 1 && y0 >= 1 && y0 + p.tile_y <= p.ny - 1;
}

// Whether fluid node (x, y) takes the force-free form of the step: those of
// tiles that touch no boundary do.
template <int STORE>
__device__ __forceinline__ bool free_form(const StepParams& p, int x, int y) {
  return p.force_free && interior_tile<STORE>(p, x / tile_x(STORE), y / p.tile_y);
}

// Storages whose rows of fluid nodes are collided without branches: FP32, and
// FP64 (1024 x 256 step 82.0 -> 79.0 us). The 16-bit kernels, at 64 registers,
// lose by it (4096 x 1024 FP16 batch of 50 steps 2.00 -> 2.03 ms).
__host__ __device__ constexpr bool straight_rows(int storage) { return storage == kF32 || storage == kF64; }

// Collide one row's N pulled nodes of a lane whose first node lies in the
// domain. free: fluid nodes take the force-free form (free_form of their tile).
// ONE: a lane's nodes one after the other, for kernels short of registers (the
// paired step at 80 registers spills 216 bytes otherwise).
template <int STORE, int COLL, bool GEN, int N, bool ONE = false>
__device__ __forceinline__ void collide_row(const StepParams& p, typename Store<STORE>::T (&h)[N][9],
                                            unsigned mw, int xb, int y, bool free,
                                            RowSums<typename Store<STORE>::T>& acc) {
  using S = Store<STORE>;
  using T = typename S::T;
  constexpr bool REF = S::kElements;  // h holds elements
  auto finish_node = [&](const Macro<T>& q, uint8_t m) {
    // a NaN or infinite population makes rho NaN, infinite or non-positive
    if (!sound_density(q.rho)) atomicOr(p.flag, 1);
    acc.dm += q.drho;
    if (m) {
      acc.solid = true;
      acc.fx -= q.fpx;
      acc.fy -= q.fpy;
    }
  };
  // A row of fluid nodes only, without body force (a warp's usual row): the
  // lane's nodes one beside the other without a branch between them, so that
  // their dependent chains overlap. Interior tiles take kFree there and
  // boundary tiles kFluid.
  if (COLL == kTrt && straight_rows(STORE) && p.force_free && free != GEN &&
      (!GEN || xb + (kLanes - int(threadIdx.x)) * N <= p.nx) && !__any_sync(0xffffffffu, mw != 0)) {
    constexpr int FORM = GEN ? kFluid : kFree;
    bool sound = true;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      if (ONE && k > 0 && mw != 0) break;  // never: keeps the nodes' instructions apart
      const Macro<T> q = macros<T, FORM, REF>(p, h[k], 0, xb + k, y);
      collide_trt<T, FORM, REF>(p, h[k], q);
      sound = sound && sound_density(q.rho);
      acc.dm += q.drho;
    }
    if (!sound) atomicOr(p.flag, 1);
    return;
  }
  auto node = [&](T(&hk)[9], int x, uint8_t m) {
    if (GEN && x >= p.nx) return;  // past the last column: padding, stored as pulled
    if (COLL == kTrt && free && m == 0) {
      // a fluid node without body force
      const Macro<T> q = macros<T, kFree, REF>(p, hk, 0, x, y);
      collide_trt<T, kFree, REF>(p, hk, q);
      finish_node(q, 0);
    } else if (COLL == kTrt) {
      const Macro<T> q = macros<T, kGeneral, REF>(p, hk, m, x, y);
      collide_trt<T, kGeneral, REF>(p, hk, q);
      finish_node(q, m);
    } else {
      // the moment-space form works on offsets
      if constexpr (REF) {
#pragma unroll
        for (int a = 0; a < 9; ++a) hk[a] = hk[a] + sref<S>(p, a);
      }
      const Macro<T> q = macros<T>(p, hk, m, x, y);
      collide_mrt<T>(p, hk, q);
      finish_node(q, m);
      if constexpr (REF) {
#pragma unroll
        for (int a = 0; a < 9; ++a) hk[a] = hk[a] - sref<S>(p, a);
      }
    }
  };
#pragma unroll
  for (int k = 0; k < N; ++k) node(h[k], xb + k, uint8_t(mw >> (8 * k)));
}

// The rounding word of each of a lane's node pairs (16-bit stores): pairs
// (xb, xb + 1), (xb + 2, xb + 3) are numbered row by row.
template <int NW>
__device__ __forceinline__ void round_words(const StepParams& p, int xb, int y, unsigned key, bool sr,
                                            unsigned (&nb)[NW]) {
#pragma unroll
  for (int j = 0; j < NW; ++j)
    nb[j] = sr ? round_bits(unsigned((long long)y * ((p.nx + 1) >> 1) + (xb >> 1) + j), key) : 0u;
}

// A tile's share of a step's records (reduce_kernel adds the tiles): the force
// on the solid nodes, summed per thread in the arithmetic type (at most 16 nodes,
// or 32 of a 16-bit store) and in FP64 from the thread up; the total density, in
// the arithmetic type within the block and FP64 from the tile up. Warps and
// blocks without solid nodes skip the FP64 work (on GB300 FP64 runs at a small
// fraction of the FP32 rate).
template <int STORE>
struct TileSums {  // in shared memory, by warp
  double f[warps_per_block(STORE)][2];
  typename Store<STORE>::T dm[warps_per_block(STORE)];
};
template <int STORE>
__device__ __forceinline__ void warp_records(const StepParams& p, const RowSums<typename Store<STORE>::T>& acc,
                                             TileSums<STORE>& sums) {
  const bool warp_solid = __any_sync(0xffffffffu, acc.solid);
  typename Store<STORE>::T dm = acc.dm;
  double bfx = 0.0, bfy = 0.0;
  if (p.reduce_mass) dm = warp_sum(dm);
  if (warp_solid) {
    bfx = warp_sum(double(acc.fx));
    bfy = warp_sum(double(acc.fy));
  }
  if (threadIdx.x == 0) {
    sums.dm[threadIdx.y] = dm;
    sums.f[threadIdx.y][0] = bfx;
    sums.f[threadIdx.y][1] = bfy;
  }
}
// One thread, once every warp's sums stand (solid: whether any warp has solid nodes).
template <int STORE>
__device__ __forceinline__ void tile_record(const StepParams& p, int tile, int x0, int y0, bool solid,
                                            const TileSums<STORE>& sums, double* partials) {
  using T = typename Store<STORE>::T;
  constexpr int W = warps_per_block(STORE);
  constexpr int TX = tile_x(STORE);
  double ts[3] = {0.0, 0.0, 0.0};
  T msum = T(0);
#pragma unroll
  for (int w = 0; w < W; ++w) msum += sums.dm[w];
  if (solid) {
#pragma unroll
    for (int w = 0; w < W; ++w) {
      ts[0] += sums.f[w][0];
      ts[1] += sums.f[w][1];
    }
  }
  if (p.reduce_mass) {
    // sum rho = active nodes + sum drho
    const int nact = min(TX, p.nx - x0) * min(p.tile_y, p.ny - y0);
    ts[2] = double(nact) + double(msum);
  }
  double* out = partials + 3ll * tile;
  out[0] = ts[0];
  out[1] = ts[1];
  out[2] = ts[2];
}

// MODE: kModeAB (pull from p.src, store to p.dst), or one of the two in-place
// AA steps on the one buffer p.dst (== p.src).
template <int STORE, int COLL, int MODE = kModeAB>
__device__ __forceinline__ void step_tile(const StepParams& p, int tile, long long t,
                                          double* partials) {
  using S = Store<STORE>;
  using T = typename S::T;
  using E = typename S::E;
  constexpr int N = npt(STORE);
  constexpr int TX = kLanes * N;
  constexpr int W = warps_per_block(STORE);

  const int lane = threadIdx.x, warp = threadIdx.y;
  const int tx = tile % p.tiles_x;
  const int ty = tile / p.tiles_x;
  const int x0 = tx * TX, y0 = ty * p.tile_y;
  const int xb = x0 + lane * N;
  const bool interior = interior_tile<STORE>(p, tx, ty);
  // Plain pointers and loads: the previous step's stores may complete while
  // this kernel's blocks already wait (pdl_wait), so a load must not be taken
  // for one of memory that stays unchanged for the whole kernel.
  const E* src = static_cast<const E*>(p.src);
  E* dst = static_cast<E*>(p.dst);
  E* buf = static_cast<E*>(p.dst);  // the in-place modes' one buffer

  RowSums<T> acc;
  const unsigned key = round_bits(unsigned(t), p.round_key);

  // Collide and store one row of pulled populations (lane_active: the lane's
  // first node lies in the domain).
  auto process_row = [&](int y, auto& h, auto gen) {
    constexpr bool GEN = decltype(gen)::value;
    const long long i = (long long)y * p.pitch + xb;
    const unsigned mw = mask_word<N>(p.mask + i);
    const bool sr = S::kSixteen && p.stochastic;
    collide_row<STORE, COLL, GEN>(p, h, mw, xb, y, !GEN && p.force_free, acc);
    unsigned nb[(N + 1) / 2];
    round_words(p, xb, y, key, sr, nb);
    if constexpr (MODE == kModeAB) {
#pragma unroll
      for (int a = 0; a < 9; ++a) {
        T o[N];
#pragma unroll
        for (int k = 0; k < N; ++k) o[k] = h[k][a];
        S::store_h(dst + (long long)a * p.plane + i, o, a, nb, sr);
      }
    } else if constexpr (MODE == kModeAALocal) {
#pragma unroll
      for (int a = 0; a < 9; ++a) {
        T o[N];
#pragma unroll
        for (int k = 0; k < N; ++k) o[k] = h[k][a];
        S::store_h(buf + (long long)opposite(a) * p.plane + i, o, a, nb, sr);
      }
      if (GEN && p.bc_x != kBcPeriodic) {
        // the outlet column's stored f* of alpha = 3, 6, 7, for the next push step
#pragma unroll
        for (int k = 0; k < N; ++k) {
          if (xb + k != p.nx - 1) continue;
          typename S::R* z = static_cast<typename S::R*>(p.z);
          z[0 * p.ny + y] = S::round_e(h[k][3], 3, nb[k >> 1], k, sr);
          z[1 * p.ny + y] = S::round_e(h[k][6], 6, nb[k >> 1], k, sr);
          z[2 * p.ny + y] = S::round_e(h[k][7], 7, nb[k >> 1], k, sr);
        }
      }
    } else {  // push step
      // vector pushes wherever every target of the row lies in the grid: all
      // of an interior tile, and the rows of a boundary tile that touches
      // neither x side nor the first or last row (warp-uniform)
      const bool vec = !GEN || (x0 >= 1 && x0 + TX <= p.nx - 1 && y >= 1 && y <= p.ny - 2);
#pragma unroll
      for (int a = 0; a < 9; ++a) {
        typename S::R e[N];
#pragma unroll
        for (int k = 0; k < N; ++k) e[k] = S::round_e(h[k][a], a, nb[k >> 1], k, sr);
        if (vec) {
          push_dir_vec<S, N>(p, buf, a, xb, y, lane, e);
        } else {
#pragma unroll
          for (int k = 0; k < N; ++k)
            if (xb + k < p.nx) push_one<S>(p, buf, a, xb + k, y, e[k]);
        }
      }
      if (GEN && p.bc_x != kBcPeriodic) {
#pragma unroll
        for (int k = 0; k < N; ++k) {
          if (xb + k != p.nx - 1) continue;
          push_outlet_copy<S>(p, buf, 3, y, S::round_e(h[k][3], 3, nb[k >> 1], k, sr));
          push_outlet_copy<S>(p, buf, 6, y, S::round_e(h[k][6], 6, nb[k >> 1], k, sr));
          push_outlet_copy<S>(p, buf, 7, y, S::round_e(h[k][7], 7, nb[k >> 1], k, sr));
        }
      }
    }
  };

  constexpr bool AA = MODE == kModeAAPush;
  const E* from = AA ? buf : src;
  auto do_row = [&](int y, auto gen, const auto& el) {
    constexpr bool GEN = decltype(gen)::value;
    const bool lane_active = !GEN || xb < p.nx;
    T h[N][9];
    if constexpr (MODE == kModeAALocal) {
      if (!lane_active) return;
      const long long i = (long long)y * p.pitch + xb;
#pragma unroll
      for (int a = 0; a < 9; ++a) {
        T v[N];
        S::load_h(buf + (long long)a * p.plane + i, v, a);
#pragma unroll
        for (int k = 0; k < N; ++k) h[k][a] = v[k];
      }
      if (GEN) {
#pragma unroll
        for (int k = 0; k < N; ++k)
          if (xb + k < p.nx) aa_local_boundary<S, true>(p, h[k], xb + k, y, true);
      }
    } else {
      pull_row<S, N, GEN, AA>(p, from, el, x0, y, lane, lane_active, h);
      if (!lane_active) return;
    }
    process_row(y, h, gen);
  };

  if (interior) {
    const EdgeLane<S, TX, false, AA> el(p, from, x0, lane);
#pragma unroll 1
    for (int r = 0; r < p.rows_per_warp; ++r) do_row(y0 + warp + r * W, std::false_type(), el);
  } else {
    const EdgeLane<S, TX, true, AA> el(p, from, x0, lane);
#pragma unroll 1
    for (int r = 0; r < p.rows_per_warp; ++r) {
      const int y = y0 + warp + r * W;
      if (y >= p.ny) break;  // warp-uniform: a warp is one row
      do_row(y, std::true_type(), el);
    }
  }

  pdl_trigger();
  __shared__ TileSums<STORE> sums;
  warp_records<STORE>(p, acc, sums);
  const bool solid = __syncthreads_or(acc.solid);
  if (lane + warp * kLanes == 0) tile_record<STORE>(p, tile, x0, y0, solid, sums, partials);
}

// Consecutive steps are launched dependently (launch_pdl): once every block has
// stored its populations (pdl_trigger in step_tile), the next step's blocks
// take the freed slots and wait there for this one's completion, so that the
// launch latency and the block start-up overlap the end of the previous step:
// 1024 x 256 FP32 9.0 -> 7.1 us per step, 4096 x 1024 FP32 62.1 -> 58.4.
// Triggered at the start of the kernel instead, the next step's blocks crowd
// onto the SMs with free slots while others still work: 8.4 us, and small FP64
// grids, bound by each SM's FP64 pipe, lost up to half.
template <int STORE, int COLL, int MODE = kModeAB>
__global__ void __launch_bounds__(threads_per_block(STORE), min_blocks_per_sm(STORE))
    fused_step_kernel(const __grid_constant__ StepParams p) {
  pdl_wait();
  step_tile<STORE, COLL, MODE>(p, blockIdx.x, p.t, p.partials);
}

// Grouped launch for serving: block b runs tile table[b].tile of solver
// table[b].solver at that solver's k-th step of the batch. Each solver has two
// parameter sets in a device array, for even and odd k (source and destination
// buffers swapped); params[].t is the solver's step index at k = 0. The block
// copies its solver's parameters to shared memory first (they are read many
// times per node), and takes the collision operator from them, so one launch
// covers SRT and MRT solvers of one storage type. MODE: the streaming step of
// every solver in the launch (in-place solvers are grouped by phase).
template <int STORE, int MODE = kModeAB>
__global__ void __launch_bounds__(threads_per_block(STORE), min_blocks_per_sm(STORE))
    fused_group_kernel(const StepParams* __restrict__ params, const GroupTile* __restrict__ table,
                       long long k) {
  __shared__ StepParams sp;
  // the table and the parameters were copied before the group's first launch:
  // read while the previous step's last blocks run
  const GroupTile gt = table[blockIdx.x];
  const StepParams* g = params + 2 * gt.solver + int(k & 1);
  {
    static_assert(sizeof(StepParams) % sizeof(int) == 0, "StepParams is copied in 4-byte words");
    const int* from = reinterpret_cast<const int*>(g);
    int* to = reinterpret_cast<int*>(&sp);
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    for (int w = tid; w < int(sizeof(StepParams) / sizeof(int)); w += threads_per_block(STORE))
      to[w] = __ldg(from + w);
  }
  __syncthreads();
  pdl_wait();
  double* partials = sp.partials + 3ll * sp.n_tiles * (k % kWindow);
  if (sp.collision == kTrt)
    step_tile<STORE, kTrt, MODE>(sp, gt.tile, sp.t + k, partials);
  else
    step_tile<STORE, kMrt, MODE>(sp, gt.tile, sp.t + k, partials);
}

// ---------------------------------------------------------------------------
// Moments: the density and implicit velocity the next step computes.
// ---------------------------------------------------------------------------
// The populations the next step pulls, in any scheme and phase (read only:
// the caller's parameters carry no ghost_dst).
template <class S, int A>
__device__ __forceinline__ typename S::T pull_aa(const StepParams& p, const typename S::E* buf, int x,
                                                 int y) {
  int as = A, ys = y - cy(A);
  if (ys < 0 || ys >= p.ny) {
    if (p.bc_y == kBcPeriodic) {
      ys = ys < 0 ? ys + p.ny : ys - p.ny;
    } else {
      as = mirror_y(A);
      ys = y;
    }
  }
  return edge_pull<S, true>(p, buf, as, ys, x - cx(A));
}
template <class S>
__device__ __forceinline__ void pull_node_any(const StepParams& p, int x, int y, typename S::T h[9]) {
  const typename S::E* buf = static_cast<const typename S::E*>(p.src);
  if (p.mode == kModeAB) {
    pull_node<S>(p, buf, x, y, h);
  } else if (p.mode == kModeAALocal) {
#pragma unroll
    for (int a = 0; a < 9; ++a)
      h[a] = S::in(buf[(long long)a * p.plane + (long long)y * p.pitch + x], a, sref<S>(p, a));
    aa_local_boundary<S>(p, h, x, y, false);
  } else {
    h[0] = pull_aa<S, 0>(p, buf, x, y);
    h[1] = pull_aa<S, 1>(p, buf, x, y);
    h[2] = pull_aa<S, 2>(p, buf, x, y);
    h[3] = pull_aa<S, 3>(p, buf, x, y);
    h[4] = pull_aa<S, 4>(p, buf, x, y);
    h[5] = pull_aa<S, 5>(p, buf, x, y);
    h[6] = pull_aa<S, 6>(p, buf, x, y);
    h[7] = pull_aa<S, 7>(p, buf, x, y);
    h[8] = pull_aa<S, 8>(p, buf, x, y);
  }
}

template <int STORE>
__global__ void moments_kernel(const __grid_constant__ StepParams p, double* rho, double* ux,
                               double* uy) {
  using S = Store<STORE>;
  using T = typename S::T;
  const int x = blockIdx.x * kBlockX + threadIdx.x;
  const int y = blockIdx.y * kBlockY + threadIdx.y;
  if (x >= p.nx || y >= p.ny) return;
  T h[9];
  pull_node_any<S>(p, x, y, h);
  const uint8_t m = p.mask[(long long)y * p.pitch + x];
  const Macro<T> q = macros<T>(p, h, m, x, y);
  const long long o = (long long)y * p.nx + x;
  rho[o] = double(q.rho);
  ux[o] = double(q.ux);
  uy[o] = double(q.uy);
}

// ---------------------------------------------------------------------------
// Momentum exchange (Section 3.3, after Ladd). Over every link from a fluid
// node x_f to a solid node x_s = x_f + xi_a the momentum
// xi_a [f*_a(x_f) + f*_abar(x_s)] of the store f*(t) crosses into the solid.
// Threads take the solid nodes of the box and look back along each direction
// for a fluid node; a link whose start lies outside a non-periodic side does
// not exist. The grid is fixed (kMeBlocks) and each thread walks its nodes
// grid-stride, so the share of each thread depends on the box alone; sums are
// FP64 in fixed order (thread, warp, block, then the last block to finish
// adds the block partials in block order).
// ---------------------------------------------------------------------------
template <int STORE>
__global__ void __launch_bounds__(kThreads)
    momentum_exchange_kernel(const __grid_constant__ StepParams p, const MeArgs m) {
  using S = Store<STORE>;
  using E = typename S::E;
  __shared__ double sm[kThreads / 32][3];
  __shared__ int s_last;
  const E* src = static_cast<const E*>(p.src);
  int x0 = m.x0, y0 = m.y0, x1 = m.x1, y1 = m.y1;
  {
    const int sx0 = m.static_box[0], sy0 = m.static_box[1];
    const int sx1 = m.static_box[2], sy1 = m.static_box[3];
    if (sx1 >= sx0 && sy1 >= sy0) {
      if (x1 < x0 || y1 < y0) {
        x0 = sx0, y0 = sy0, x1 = sx1, y1 = sy1;
      } else {
        x0 = min(x0, sx0), y0 = min(y0, sy0), x1 = max(x1, sx1), y1 = max(y1, sy1);
      }
    }
  }
  double fx = 0.0, fy = 0.0;
  if (x1 >= x0 && y1 >= y0) {
    const int w = x1 - x0 + 1;
    const long long n = (long long)w * (y1 - y0 + 1);
    for (long long i = (long long)blockIdx.x * kThreads + threadIdx.x; i < n;
         i += (long long)gridDim.x * kThreads) {
      const int x = x0 + int(i % w), y = y0 + int(i / w);
      if (p.mask[(long long)y * p.pitch + x] == 0) continue;
#pragma unroll
      for (int a = 1; a < 9; ++a) {
        int xf = x - cx(a), yf = y - cy(a);
        if (xf < 0 || xf >= p.nx) {
          if (p.bc_x != kBcPeriodic) continue;
          xf = xf < 0 ? xf + p.nx : xf - p.nx;
        }
        if (yf < 0 || yf >= p.ny) {
          if (p.bc_y != kBcPeriodic) continue;
          yf = yf < 0 ? yf + p.ny : yf - p.ny;
        }
        if (p.mask[(long long)yf * p.pitch + xf] != 0) continue;
        const int o = opposite(a);
        const E ef = fstar_e<S>(p, src, a, xf, yf), es = fstar_e<S>(p, src, o, x, y);
        const double flow = S::to_f64(&ef, a, sref<S>(p, a)) + S::to_f64(&es, o, sref<S>(p, o));
        fx += double(cx(a)) * flow;
        fy += double(cy(a)) * flow;
      }
    }
  }
  double v[3] = {fx, fy, 0.0};
  block_sum3(v, sm);
  if (threadIdx.x == 0) {
    __stcg(m.partials + 2 * blockIdx.x + 0, v[0]);
    __stcg(m.partials + 2 * blockIdx.x + 1, v[1]);
    __threadfence();
    s_last = atomicAdd(m.counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double u[3] = {0.0, 0.0, 0.0};
  for (int b = threadIdx.x; b < (int)gridDim.x; b += kThreads) {
    u[0] += __ldcg(m.partials + 2 * b + 0);
    u[1] += __ldcg(m.partials + 2 * b + 1);
  }
  block_sum3(u, sm);
  if (threadIdx.x == 0) {
    m.out[0] = u[0];
    m.out[1] = u[1];
    *m.counter = 0u;
  }
}

// f*(t) := f_eq(rho0, u(x)), u from a device [2][ny][nx] array or uniform.
template <int STORE>
__global__ void init_kernel(const __grid_constant__ StepParams p, void* dst, const double* u,
                            double rho0, double u0x, double u0y) {
  using S = Store<STORE>;
  using T = typename S::T;
  const int x = blockIdx.x * kBlockX + threadIdx.x;
  const int y = blockIdx.y * kBlockY + threadIdx.y;
  if (x >= p.nx || y >= p.ny) return;
  const long long o = (long long)y * p.nx + x;
  const long long nn = (long long)p.nx * p.ny;
  const T ux = T(u ? u[o] : u0x), uy = T(u ? u[nn + o] : u0y), rho = T(rho0);
  const T drho = rho - T(1);
  const T common = drho - T(1.5) * rho * (ux * ux + uy * uy);
  typename S::E* d = static_cast<typename S::E*>(dst);
  const long long i = (long long)y * p.pitch + x;
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    const T xu = T(cx(a)) * ux + T(cy(a)) * uy;
    const T heq = wgt<T>(a) * (common + rho * xu * (T(3) + T(4.5) * xu));
    // in place (AA), a state before a push step keeps f*_a in the opposite slot
    const int slot = p.mode == kModeAB ? a : opposite(a);
    store_h<S>(p, d + (long long)slot * p.plane + i, heq, a);
  }
}

// Convective outlet state g := the offsets of the last column of the store
// (a zero-gradient start), [3][ny] rows alpha = 3, 6, 7.
// In place (AA), also the side copy z of those stored values (either output
// may be null).
template <int STORE>
__global__ void ghost_init_kernel(const __grid_constant__ StepParams p, const void* srcv, void* ghostv,
                                  void* zv) {
  using S = Store<STORE>;
  using T = typename S::T;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 3 * p.ny) return;
  const int k = i / p.ny, y = i - k * p.ny;
  const int a = k == 0 ? 3 : (k == 1 ? 6 : 7);
  const typename S::E e = fstar_e<S>(p, static_cast<const typename S::E*>(srcv), a, p.nx - 1, y);
  if (ghostv) static_cast<T*>(ghostv)[i] = S::in(e, a, sref<S>(p, a));
  if (zv) static_cast<typename S::E*>(zv)[i] = e;
}

// Store <-> dense FP64 [9][ny][nx].
template <int STORE>
__global__ void export_kernel(const __grid_constant__ StepParams p, const void* srcv, double* f) {
  using S = Store<STORE>;
  const int x = blockIdx.x * kBlockX + threadIdx.x;
  const int y = blockIdx.y * kBlockY + threadIdx.y;
  if (x >= p.nx || y >= p.ny) return;
  const typename S::E* src = static_cast<const typename S::E*>(srcv);
  const long long i = (long long)y * p.pitch + x;
  const long long o = (long long)y * p.nx + x;
  const long long nn = (long long)p.nx * p.ny;
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    const typename S::E e = fstar_e<S>(p, src, a, x, y);
    f[a * nn + o] = S::to_f64(&e, a, sref<S>(p, a));
  }
  (void)i;
}

template <int STORE>
__global__ void import_kernel(const __grid_constant__ StepParams p, void* dstv, const double* f) {
  using S = Store<STORE>;
  const int x = blockIdx.x * kBlockX + threadIdx.x;
  const int y = blockIdx.y * kBlockY + threadIdx.y;
  if (x >= p.nx || y >= p.ny) return;
  typename S::E* dst = static_cast<typename S::E*>(dstv);
  const long long i = (long long)y * p.pitch + x;
  const long long o = (long long)y * p.nx + x;
  const long long nn = (long long)p.nx * p.ny;
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    const int slot = p.mode == kModeAB ? a : opposite(a);  // in place: before a push step
    S::from_f64(dst + slot * p.plane + i, f[a * nn + o], a, sref<S>(p, a));
  }
}

}  // namespace vplbm
