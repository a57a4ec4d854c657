// levelops.cu — geometric multigrid building blocks on the vertex-nested
// hierarchy (the preconditioner of the BiCGSTAB stage solve; the paper's
// Sec. 5 setup paragraph names BiCGSTAB + GMG without further detail):
//   - residual r = b - A x, damped point-block Jacobi, multicolour block
//     Gauss-Seidel (2^d colours by coordinate parity), all with the 2x2 block
//     stencil read as coalesced 16/32-byte loads in parity-split order;
//   - full-weighting restriction P^T and trilinear prolongation P (per
//     component; Dirichlet p_w unknowns excluded from the correction space);
//   - Galerkin coarse operators J_c = P^T J P, M_c = P^T M P in FP64;
//   - packing of A = shift*M - J into FP64 / FP32 / FP16-with-row-scales
//     storage and the 2x2 diagonal-block inverses;
//   - the coarsest level's dense LU (partial pivoting) and explicit inverse.
// All of these are HBM-bandwidth kernels except the set-up ones.
#include <cooperative_groups.h>
#include <algorithm>
#include <type_traits>
#include <vector>

#include "cluster_plan.h"
#include "rf_common.cuh"
#include "rf_kernels.h"

namespace cg = cooperative_groups;

namespace rf {

// ----------------------------------------------------------------- loads
template <int KIND> struct Ty;
template <> struct Ty<STORE_F64> { typedef double T; typedef double S; };
template <> struct Ty<STORE_F32> { typedef float T; typedef float S; };
template <> struct Ty<STORE_F16> { typedef float T; typedef __half S; };

// Streaming read of matrix data: read-only path, not kept in L1, and first in
// line for eviction from L2 (an L2 cache-hint policy), so that the x vector,
// which every colour launch gathers from its neighbours, keeps its place
// there.  -DRF_NO_L2_HINTS builds the loads without the L2 policies.
__device__ __forceinline__ uint64_t l2_policy_first() {
  uint64_t pol;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ uint64_t l2_policy_last() {
  uint64_t pol;
  asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
#ifdef RF_NO_L2_HINTS
__device__ __forceinline__ float4 ld_stream_f4(const float4* p) {
  float4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0,%1,%2,%3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ double2 ld_stream_d2(const double2* p) {
  double2 v;
  asm volatile("ld.global.nc.L1::no_allocate.v2.f64 {%0,%1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ uint2 ld_stream_u2(const uint2* p) {
  uint2 v;
  asm volatile("ld.global.nc.L1::no_allocate.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ uint4 ld_stream_u4(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
template <typename V>
__device__ __forceinline__ V ld_keep(const V* p) { return *p; }
#else
__device__ __forceinline__ float4 ld_stream_f4(const float4* p) {
  float4 v;
  asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.f32 {%0,%1,%2,%3}, [%4], %5;"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p), "l"(l2_policy_first()));
  return v;
}
__device__ __forceinline__ double2 ld_stream_d2(const double2* p) {
  double2 v;
  asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v2.f64 {%0,%1}, [%2], %3;"
               : "=d"(v.x), "=d"(v.y) : "l"(p), "l"(l2_policy_first()));
  return v;
}
__device__ __forceinline__ uint2 ld_stream_u2(const uint2* p) {
  uint2 v;
  asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v2.u32 {%0,%1}, [%2], %3;"
               : "=r"(v.x), "=r"(v.y) : "l"(p), "l"(l2_policy_first()));
  return v;
}
__device__ __forceinline__ uint4 ld_stream_u4(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0,%1,%2,%3}, [%4], %5;"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p), "l"(l2_policy_first()));
  return v;
}
// Neighbour values of x: kept in L1 (neighbouring threads share them) and
// last in line for eviction from L2.  Only values this launch does not write
// are read this way (GS reads other colours; residual / Jacobi read an input).
// Volatile and not .nc: the preceding launch may write x until rf_pdl_begin() has
// waited for it, so the loads may not move ahead of that, nor is x read-only for
// as long as the kernel runs.
__device__ __forceinline__ float2 ld_keep(const float2* p) {
  float2 v;
  asm volatile("ld.global.L2::cache_hint.v2.f32 {%0,%1}, [%2], %3;" : "=f"(v.x), "=f"(v.y) : "l"(p), "l"(l2_policy_last()));
  return v;
}
__device__ __forceinline__ double2 ld_keep(const double2* p) {
  double2 v;
  asm volatile("ld.global.L2::cache_hint.v2.f64 {%0,%1}, [%2], %3;" : "=d"(v.x), "=d"(v.y) : "l"(p), "l"(l2_policy_last()));
  return v;
}
#endif
// Values that another thread of this block has just written (behind a block
// barrier, which the load may not cross): at L2, past this SM's L1.
__device__ __forceinline__ float2 ld_written(const float2* p) {
  float2 v;
  asm volatile("ld.global.cg.v2.f32 {%0,%1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ double2 ld_written(const double2* p) {
  double2 v;
  asm volatile("ld.global.cg.v2.f64 {%0,%1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p) : "memory");
  return v;
}

// Stencil blocks that reach the other x-parity run of the vertex's own x-line
// (dx = -1, +1 with dy = dz = 0).  In a launch that sweeps a pair of colours
// differing only in x parity (k_gs_pair) these are the only neighbours of the
// second colour that the first one writes; the second colour reads them
// coherently at L2 (SAME = true), never through the read-only path.
template <int NB>
__host__ __device__ constexpr bool same_line_block(int b) {
  return NB == 27 ? (b == 12 || b == 14) : (b == 3 || b == 5);
}
template <bool SAME, int NB, typename V>
__device__ __forceinline__ V ld_xn(const V* p, int b) {
  if (SAME && same_line_block<NB>(b)) return ld_written(p);
  return ld_keep(p);
}
template <bool SAME, int NB, typename V>
__device__ __forceinline__ V ld_xn_plain(const V* p, int b) {
  if (SAME && same_line_block<NB>(b)) return ld_written(p);
  return *p;
}

// One stored 2x2 block as loaded (FP64: two double2; FP32: a float4; FP16:
// four halves), and its entries in the arithmetic type (FP16: times the row's
// per-entry FP32 scales).  Loading and unpacking are split so that a batch of
// loads can be issued before any of them is unpacked.
template <int KIND> struct RawBlock;
template <> struct RawBlock<STORE_F64> { double2 u, w; };
template <> struct RawBlock<STORE_F32> { float4 u; };
template <> struct RawBlock<STORE_F16> { uint2 u; };

template <int KIND>
__device__ __forceinline__ void load_raw(const void* A, int64_t nv, int b, int64_t p, RawBlock<KIND>& r) {
  const int64_t o = (int64_t)b * nv + p;
  if constexpr (KIND == STORE_F64) {
    const double2* q = reinterpret_cast<const double2*>(A) + o * 2;
    r.u = ld_stream_d2(q);
    r.w = ld_stream_d2(q + 1);
  } else if constexpr (KIND == STORE_F32) {
    r.u = ld_stream_f4(reinterpret_cast<const float4*>(A) + o);
  } else {
    r.u = ld_stream_u2(reinterpret_cast<const uint2*>(A) + o);
  }
}

template <int KIND>
__device__ __forceinline__ void unpack_block(const RawBlock<KIND>& r, const float4& sc, typename Ty<KIND>::T (&a)[4]) {
  if constexpr (KIND == STORE_F64) {
    a[0] = r.u.x; a[1] = r.u.y; a[2] = r.w.x; a[3] = r.w.y;
  } else if constexpr (KIND == STORE_F32) {
    a[0] = r.u.x; a[1] = r.u.y; a[2] = r.u.z; a[3] = r.u.w;
  } else {
    uint2 u = r.u;
    __half2 h01 = *reinterpret_cast<__half2*>(&u.x), h23 = *reinterpret_cast<__half2*>(&u.y);
    float2 f01 = __half22float2(h01), f23 = __half22float2(h23);
    a[0] = f01.x * sc.x; a[1] = f01.y * sc.y; a[2] = f23.x * sc.z; a[3] = f23.y * sc.w;
  }
}

template <int KIND>
__device__ __forceinline__ void load_block(const void* A, int64_t nv, int b, int64_t p, const float4& sc,
                                           typename Ty<KIND>::T (&a)[4]) {
  RawBlock<KIND> r;
  load_raw<KIND>(A, nv, b, p, r);
  unpack_block<KIND>(r, sc, a);
}

// A row's sum of a_0 x_0 + a_1 x_1 over its blocks, in explicit operations, so
// that every kernel applying a block (per-block, batched, shared-matrix) rounds
// it identically, whatever the compiler would otherwise contract.  FP32: one
// product, one multiply-add, one sum per block (a chain of one add per block).
// FP64: a multiply-add for each of two sums, of the a_0 x_0 and of the a_1 x_1, added
// at the end, as these kernels are bound by the FP64 pipe (65^3 Jacobi: 104 us a sweep
// with three operations per block, 70 us with two; its 108 multiply-adds per vertex
// take 56 us).  One sum through both products rounds twice as long a chain: its mean
// error against 113 bits, in units of sum |a x|, is 9.2e-17 at 17^3 and 6.6e-17 at
// 33 x 17, with two sums 6.8e-17 and 5.2e-17 (the three operations: 7.2e-17, 6.0e-17).
template <typename T> struct RowAcc;
template <> struct RowAcc<float> {
  float s = 0.f;
  __device__ __forceinline__ void add(float a0, float a1, float2 x) {
    s = __fadd_rn(s, __fmaf_rn(a0, x.x, __fmul_rn(a1, x.y)));
  }
  __device__ __forceinline__ float value() const { return s; }
};
template <> struct RowAcc<double> {
  double u = 0.0, v = 0.0;
  __device__ __forceinline__ void add(double a0, double a1, double2 x) {
    u = __fma_rn(a0, x.x, u);
    v = __fma_rn(a1, x.y, v);
  }
  __device__ __forceinline__ double value() const { return __dadd_rn(u, v); }
};

// FP16 storage holds the blocks of a row in pairs, one 16-byte load per pair
// (a warp reads 512 contiguous bytes per load, as with FP32 blocks): slot s
// of row p is half s % 2 of uint4 number (s / 2) * nv + p.  The two blocks of
// a pair have offsets of the same parity in every axis, so they reach
// vertices of the same colour: the first sweep from zero, which skips the
// blocks of colours not yet visited, skips whole pairs.  Slots (3D): the
// pairs dx = -1, +1 for each (dy, dz); then the dx = 0 pairs (dy = -1, +1 at
// dz = 0), (dz = -1, +1 at dy = 0), (dy = -1, +1 at dz = -1), (dy = -1, +1 at
// dz = +1); then the centre and an empty slot.  2D: dx = -1, +1 for each dy,
// then (dy = -1, +1 at dx = 0), then the centre and an empty slot.  A sweep
// that skips the centre reads none of the last pair.
__host__ __device__ constexpr int f16_block_of_slot(int nb, int s) {
  if (nb == 27) {
    if (s < 18) return ((s & 1) ? 2 : 0) + 3 * ((s >> 1) % 3) + 9 * ((s >> 1) / 3);
    switch (s) {
      case 18: return 10; case 19: return 16;   // (0, -1, 0), (0, +1, 0)
      case 20: return 4;  case 21: return 22;   // (0, 0, -1), (0, 0, +1)
      case 22: return 1;  case 23: return 7;    // (0, -1, -1), (0, +1, -1)
      case 24: return 19; case 25: return 25;   // (0, -1, +1), (0, +1, +1)
      case 26: return 13;                       // centre
      default: return -1;
    }
  }
  if (s < 6) return ((s & 1) ? 2 : 0) + 3 * (s >> 1);
  return s == 6 ? 1 : s == 7 ? 7 : s == 8 ? 4 : -1;
}
__host__ __device__ constexpr int f16_slot_of_block(int nb, int b) {
  int s = 0;
  while (s < nb && f16_block_of_slot(nb, s) != b) ++s;
  return s;
}

__device__ __forceinline__ void f16_half(const uint4& u, int h, const float4& sc, float (&a)[4]) {
  RawBlock<STORE_F16> r;
  r.u = h ? make_uint2(u.z, u.w) : make_uint2(u.x, u.y);
  unpack_block<STORE_F16>(r, sc, a);
}

// The FP16 stencil sum, slot by slot: CP pairs (2 CP blocks) and their x values
// loaded per memory round trip, then summed.  Per-block, batched and
// shared-matrix FP16 kernels all sum in this slot order with RowAcc.
template <int NB, int CP, bool SAME = false>
__device__ __forceinline__ void stencil_sum_f16(const LevelOp& L, int64_t p, int par,
                                                const float2* __restrict__ x, bool skip_centre, uint32_t skipmask,
                                                float& s0, float& s1) {
  constexpr int C = NB == 27 ? 13 : 4, NP = (NB + 1) / 2;
  const float4 sc = reinterpret_cast<const float4*>(L.scale)[p];
  const uint4* __restrict__ A = reinterpret_cast<const uint4*>(L.A);
  RowAcc<float> a0, a1;
#pragma unroll
  for (int q0 = 0; q0 < NP; q0 += CP) {
    uint4 raw[CP];
    float2 xv[CP][2];
    bool use[CP][2];
#pragma unroll
    for (int c = 0; c < CP; ++c) {
      const int q = q0 + c;
      if (q >= NP) break;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int b = f16_block_of_slot(NB, 2 * q + h);
        use[c][h] = b >= 0 && !(skip_centre && b == C) && !((skipmask >> (b >= 0 ? b : 0)) & 1u);
      }
      if (use[c][0] || use[c][1]) raw[c] = ld_stream_u4(A + (int64_t)q * L.d.nv + p);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int b = f16_block_of_slot(NB, 2 * q + h);
        if (use[c][h]) xv[c][h] = ld_xn<SAME, NB>(x + p + (par ? L.nb.off[1][b] : L.nb.off[0][b]), b);
      }
    }
#pragma unroll
    for (int c = 0; c < CP; ++c) {
      if (q0 + c >= NP) break;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (!use[c][h]) continue;
        float a[4];
        f16_half(raw[c], h, sc, a);
        a0.add(a[0], a[1], xv[c][h]);
        a1.add(a[2], a[3], xv[c][h]);
      }
    }
  }
  s0 = a0.value();
  s1 = a1.value();
}

// sum over the stencil of blocks * x (centre optionally skipped)
template <int KIND, int NB, bool SAME = false>
__device__ __forceinline__ void stencil_sum(const LevelOp& L, int64_t p, int par,
                                            const typename V2<typename Ty<KIND>::T>::t* __restrict__ x,
                                            bool skip_centre, uint32_t skipmask, typename Ty<KIND>::T& s0,
                                            typename Ty<KIND>::T& s1) {
  typedef typename Ty<KIND>::T T;
  constexpr int C = NB == 27 ? 13 : 4;
  float4 sc = make_float4(1.f, 1.f, 1.f, 1.f);
  if (KIND == STORE_F16) sc = reinterpret_cast<const float4*>(L.scale)[p];
  RowAcc<T> a0, a1;
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    if (skip_centre && b == C) continue;
    if ((skipmask >> b) & 1u) continue;   // neighbour known to be zero
    T a[4];
    load_block<KIND>(L.A, L.d.nv, b, p, sc, a);
    const int off = par ? L.nb.off[1][b] : L.nb.off[0][b];
    const typename V2<T>::t xv = ld_xn_plain<SAME, NB>(x + p + off, b);
    a0.add(a[0], a[1], xv);
    a1.add(a[2], a[3], xv);
  }
  s0 = a0.value();
  s1 = a1.value();
}

// stencil_sum with the loads of CH blocks (and their x values) issued before
// any is used: one memory round trip per CH blocks instead of one per block.
// The block loads are the `volatile` streaming loads of load_raw, which the
// compiler keeps in source order, so placing all CH of them ahead of the sums
// is what batches them (ordinary loads get sunk back next to their uses).
// The same blocks are summed in the same order with the same RowAcc, so the
// sums equal stencil_sum's bit for bit.
// This is what the small levels need, where a thread's chain of round trips,
// not bandwidth, sets the time.
// Stencil blocks (FP16: block pairs) whose loads a batched kernel issues per
// memory round trip; an unbatched FP16 kernel loads one pair per round trip.
// Batched FP16 is for small levels, where a thread's round trips set the time:
// seven pairs (GS at 17^3: 12.7 us a pair launch unbatched, 6.8 us so).
__host__ __device__ constexpr int chunk_of(int kind) { return kind == STORE_F16 ? 7 : 9; }

template <int KIND, int NB, int CH, bool SAME = false>
__device__ __forceinline__ void stencil_sum_batched(const LevelOp& L, int64_t p, int par,
                                                    const typename V2<typename Ty<KIND>::T>::t* __restrict__ x,
                                                    bool skip_centre, uint32_t skipmask, typename Ty<KIND>::T& s0,
                                                    typename Ty<KIND>::T& s1) {
  typedef typename Ty<KIND>::T T;
  typedef typename V2<T>::t V;
  constexpr int C = NB == 27 ? 13 : 4;
  float4 sc = make_float4(1.f, 1.f, 1.f, 1.f);
  if (KIND == STORE_F16) sc = reinterpret_cast<const float4*>(L.scale)[p];
  RowAcc<T> a0, a1;
#pragma unroll
  for (int b0 = 0; b0 < NB; b0 += CH) {
    RawBlock<KIND> raw[CH];
    bool skip[CH];
    V xv[CH];
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      const int b = b0 + c;
      if (b >= NB) break;
      skip[c] = (skip_centre && b == C) || ((skipmask >> b) & 1u);
      if (!skip[c]) {
        load_raw<KIND>(L.A, L.d.nv, b, p, raw[c]);
        xv[c] = ld_xn<SAME, NB>(x + p + (par ? L.nb.off[1][b] : L.nb.off[0][b]), b);
      }
    }
    // unpacked only now: an FP16 block's scaling waits for its load, which
    // would otherwise hold back the loads issued after it
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      if (b0 + c >= NB) break;
      if (skip[c]) continue;   // as in the per-block sum
      T a[4];
      unpack_block<KIND>(raw[c], sc, a);
      a0.add(a[0], a[1], xv[c]);
      a1.add(a[2], a[3], xv[c]);
    }
  }
  s0 = a0.value();
  s1 = a1.value();
}

template <int KIND, int NB, int CH, bool SAME = false>
__device__ __forceinline__ void stencil_sum_any(const LevelOp& L, int64_t p, int par,
                                                const typename V2<typename Ty<KIND>::T>::t* __restrict__ x,
                                                bool skip_centre, uint32_t skipmask, typename Ty<KIND>::T& s0,
                                                typename Ty<KIND>::T& s1) {
  if constexpr (KIND == STORE_F16)
    stencil_sum_f16<NB, (CH > 0 ? CH : 1), SAME>(L, p, par, x, skip_centre, skipmask, s0, s1);
  else if constexpr (CH > 0)
    stencil_sum_batched<KIND, NB, CH, SAME>(L, p, par, x, skip_centre, skipmask, s0, s1);
  else
    stencil_sum<KIND, NB, SAME>(L, p, par, x, skip_centre, skipmask, s0, s1);
}

// (A x)_p, with A = shift*M - J on the fine level (blocks hold J)
template <int KIND, bool FINE, int NB, int CH = 0>
__device__ __forceinline__ void apply_row(const LevelOp& L, int64_t p, int par,
                                          const typename V2<typename Ty<KIND>::T>::t* __restrict__ x,
                                          typename Ty<KIND>::T& s0, typename Ty<KIND>::T& s1) {
  typedef typename Ty<KIND>::T T;
  // batched: the mask is L.nomask (always zero) read at run time, which keeps
  // each block's load in its own conditional branch and so stops the compiler
  // from interleaving the batch's loads with the sums (it does that with a
  // constant zero mask, and the batch is lost)
  stencil_sum_any<KIND, NB, CH>(L, p, par, x, false, CH > 0 ? L.nomask : 0u, s0, s1);
  if (FINE) {
    const double2 m = reinterpret_cast<const double2*>(L.mdiag)[p];
    const T xs = x[p].y, sh = (T)L.shift;
    s0 = (T)(sh * (T)m.x) * xs - s0;
    s1 = (T)(sh * (T)m.y) * xs - s1;
  }
}

template <typename T>
__device__ __forceinline__ void dinv_apply(const T* Dinv, int64_t p, T r0, T r1, T& y0, T& y1) {
  const T* D = Dinv + p * 4;
  y0 = D[0] * r0 + D[1] * r1;
  y1 = D[2] * r0 + D[3] * r1;
}

// ----------------------------------------------------------------- residual
template <int KIND, bool FINE, int NB, int CH = 0>
__device__ __forceinline__ void residual_point(const LevelOp& L, const typename V2<typename Ty<KIND>::T>::t* __restrict__ b,
                                               const typename V2<typename Ty<KIND>::T>::t* __restrict__ x,
                                               typename V2<typename Ty<KIND>::T>::t* __restrict__ r, int64_t p) {
  typedef typename Ty<KIND>::T T;
  const int par = (int)((uint32_t)p % (uint32_t)L.d.nx) >= L.d.E;   // nv < 2^31
  const typename V2<T>::t bv = b[p];
  T s0, s1;
  apply_row<KIND, FINE, NB, CH>(L, p, par, x, s0, s1);
  typename V2<T>::t o;
  o.x = bv.x - s0;
  o.y = bv.y - s1;
  r[p] = o;
}

template <int KIND, bool FINE, int NB, int CH>
__global__ void __launch_bounds__(CH > 0 ? 256 : 512) k_residual(LevelOp L, const typename V2<typename Ty<KIND>::T>::t* __restrict__ b,
                                                  const typename V2<typename Ty<KIND>::T>::t* __restrict__ x,
                                                  typename V2<typename Ty<KIND>::T>::t* __restrict__ r) {
  rf_pdl_begin(b, x);
  int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= L.d.nv) return;
  residual_point<KIND, FINE, NB, CH>(L, b, x, r, p);
}

// ----------------------------------------------------------------- Jacobi
template <int KIND, bool FINE, int NB, int CH = 0>
__device__ __forceinline__ void jacobi_point(const LevelOp& L, const typename V2<typename Ty<KIND>::T>::t* __restrict__ b,
                                             const typename V2<typename Ty<KIND>::T>::t* __restrict__ xin,
                                             typename V2<typename Ty<KIND>::T>::t* __restrict__ xout, double omega,
                                             int zero_x, int64_t p) {
  typedef typename Ty<KIND>::T T;
  const typename V2<T>::t bv = b[p];
  T r0 = bv.x, r1 = bv.y, x0 = 0, x1 = 0;
  if (!zero_x) {
    const int par = (int)((uint32_t)p % (uint32_t)L.d.nx) >= L.d.E;   // nv < 2^31
    T s0, s1;
    apply_row<KIND, FINE, NB, CH>(L, p, par, xin, s0, s1);
    r0 -= s0;
    r1 -= s1;
    x0 = xin[p].x;
    x1 = xin[p].y;
  }
  T y0, y1;
  dinv_apply<T>(reinterpret_cast<const T*>(L.Dinv), p, r0, r1, y0, y1);
  typename V2<T>::t o;
  o.x = x0 + (T)omega * y0;
  o.y = x1 + (T)omega * y1;
  xout[p] = o;
}

template <int KIND, bool FINE, int NB, int CH>
__global__ void __launch_bounds__(CH > 0 ? 256 : 512) k_jacobi(LevelOp L, const typename V2<typename Ty<KIND>::T>::t* __restrict__ b,
                                                const typename V2<typename Ty<KIND>::T>::t* __restrict__ xin,
                                                typename V2<typename Ty<KIND>::T>::t* __restrict__ xout, double omega,
                                                int zero_x) {
  rf_pdl_begin(b, xin);
  int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= L.d.nv) return;
  jacobi_point<KIND, FINE, NB, CH>(L, b, xin, xout, omega, zero_x, p);
}

// ----------------------------------------------------------------- multicolour GS
// One vertex p (x parity px) of a colour: x_p <- D_p^-1 (b_p - sum_{q != p} A_pq x_q).
template <int KIND, bool FINE, int NB, int CH = 0, bool SAME = false>
__device__ __forceinline__ void gs_vertex(const LevelOp& L, const typename V2<typename Ty<KIND>::T>::t* __restrict__ b,
                                          typename V2<typename Ty<KIND>::T>::t* __restrict__ x, int px, int64_t p,
                                          uint32_t skipmask) {
  typedef typename Ty<KIND>::T T;
  const typename V2<T>::t bv = b[p];
  T s0, s1;
  stencil_sum_any<KIND, NB, CH, SAME>(L, p, px, x, true, skipmask, s0, s1);
  // off-diagonal part of A: fine level A_pq = -J_pq (q != p), coarse A_pq
  const T r0 = FINE ? bv.x + s0 : bv.x - s0;
  const T r1 = FINE ? bv.y + s1 : bv.y - s1;
  T y0, y1;
  dinv_apply<T>(reinterpret_cast<const T*>(L.Dinv), p, r0, r1, y0, y1);
  typename V2<T>::t o;
  o.x = y0;
  o.y = y1;
  x[p] = o;
}

// One colour (px,py,pz) of the sweep.
// Work item t of the colour: t enumerates the colour's x-runs line by line.
template <int KIND, bool FINE, int NB, int CH = 0>
__device__ __forceinline__ void gs_point(const LevelOp& L, const typename V2<typename Ty<KIND>::T>::t* __restrict__ b,
                                         typename V2<typename Ty<KIND>::T>::t* __restrict__ x, int px, int py, int pz,
                                         int cnt_x, int lines_y, int64_t t, uint32_t skipmask) {
  typedef typename Ty<KIND>::T T;
  // 32-bit index arithmetic: a colour has fewer than 2^31 vertices
  const uint32_t tt = (uint32_t)t, line = tt / (uint32_t)cnt_x, kl = line / (uint32_t)lines_y;
  const int pos = (int)(tt - line * (uint32_t)cnt_x);
  const int jj = (int)(line - kl * (uint32_t)lines_y), kk = (int)kl;
  const int j = 2 * jj + py, k = 2 * kk + pz;
  const int64_t p = ((int64_t)j + (int64_t)L.d.ny * k) * L.d.nx + (px ? L.d.E : 0) + pos;
  gs_vertex<KIND, FINE, NB, CH>(L, b, x, px, p, skipmask);
}

template <int KIND, bool FINE, int NB, int CH>
__global__ void __launch_bounds__(CH > 0 ? 256 : 512) k_gs_colour(LevelOp L, const typename V2<typename Ty<KIND>::T>::t* __restrict__ b,
                                                   typename V2<typename Ty<KIND>::T>::t* __restrict__ x, int px, int py,
                                                   int pz, int cnt_x, int lines_y, int64_t count, uint32_t skipmask,
                                                   int reverse) {
  rf_pdl_begin(b, x);
  // reverse: blocks take the colour's vertices from the end (see gs_zigzag)
  const int64_t bx = reverse ? (int64_t)(gridDim.x - 1 - blockIdx.x) : (int64_t)blockIdx.x;
  int64_t t = bx * blockDim.x + threadIdx.x;
  if (t >= count) return;
  gs_point<KIND, FINE, NB, CH>(L, b, x, px, py, pz, cnt_x, lines_y, t, skipmask);
}

// Threads of a colour-pair block (k_gs_pair) at most.
constexpr int GS_PAIR_MAX_THREADS = 320;

// Vertex of item v of a pair block's run: line l0 + v / cnt of the pair's
// lines (enumerated y first), position v % cnt in the run of parity px.
__device__ __forceinline__ int64_t pair_vertex(const Dims& d, int l0, int v, int cnt, int px, int py, int pz,
                                               int lines_y) {
  const int li = v / cnt, pos = v - li * cnt;
  const int line = l0 + li, kl = line / lines_y;
  const int j = 2 * (line - kl * lines_y) + py, k = 2 * kl + pz;
  return ((int64_t)j + (int64_t)d.ny * k) * d.nx + (px ? d.E : 0) + pos;
}

// Two consecutive colours of a sweep that differ only in x parity,
// (first_px, py, pz) then (1 - first_px, py, pz), in one launch.  A vertex of
// either colour reaches the other one only on its own x-line (dx = -1, +1 with
// dy = dz = 0); all its other neighbours have colours that neither of the two
// writes.  So a block that owns whole x-lines updates the first colour's run
// of each of its lines, passes a block barrier, and then updates the second
// colour's runs, reading the just-written neighbours at L2: every vertex sees
// the values that the two separate colour launches give it, and the sums are
// the same operations in the same order.  One launch instead of two, and the
// other colours' x values are gathered once for both.  Block b owns lines
// [b * lpb, b * lpb + lpb) of the pair (reversed block order: see gs_zigzag).
template <int KIND, bool FINE, int NB, int CH, int FPX>
__global__ void __launch_bounds__(GS_PAIR_MAX_THREADS) k_gs_pair(LevelOp L, const typename V2<typename Ty<KIND>::T>::t* __restrict__ b,
                                                  typename V2<typename Ty<KIND>::T>::t* __restrict__ x,
                                                  int py, int pz, int lines_y, int nlines, int lpb,
                                                  uint32_t skip_first, uint32_t skip_second, int reverse) {
  rf_pdl_begin(b, x);
  const int bx = reverse ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x;
  const int l0 = bx * lpb;
  const int nl = min(lpb, nlines - l0);
  // one vertex per thread and run: the launch gives every block at least
  // lpb * (nx + 1) / 2 threads (a loop here would make the compiler hoist
  // the stencil's address arithmetic and double the registers)
  const int v = threadIdx.x;
  {
    const int cnt = FPX ? L.d.nx / 2 : (L.d.nx + 1) / 2;
    if (v < nl * cnt)
      gs_vertex<KIND, FINE, NB, CH, false>(L, b, x, FPX, pair_vertex(L.d, l0, v, cnt, FPX, py, pz, lines_y), skip_first);
  }
  __syncthreads();
  {
    const int cnt = FPX ? (L.d.nx + 1) / 2 : L.d.nx / 2;
    if (v < nl * cnt)
      gs_vertex<KIND, FINE, NB, CH, true>(L, b, x, 1 - FPX, pair_vertex(L.d, l0, v, cnt, 1 - FPX, py, pz, lines_y), skip_second);
  }
}

// ----------------------------------------------------------------- small FP32 levels
// On levels that cannot fill the GPU a launch costs its chain of latencies, not
// its bytes: the launch itself, the round trips to L2, the last block.  These
// forms of the FP32 kernels load a row's whole stencil and D^-1 before
// griddepcontrol.wait (matrices do not change during a solve, so this overlaps
// the predecessor's tail), then gather b and all neighbours in one round trip.
// 27 float4 and 27 float2 take up to 200 registers, which the few blocks of such
// a level afford.  Same sums in the same order as the kernels above.
template <int NB>
struct RowF32 {
  float4 a[NB], d;
};
template <int NB, bool CENTRE>
__device__ __forceinline__ void row_load(const LevelOp& L, int64_t p, uint32_t mask, RowF32<NB>& R) {
  const float4* A = reinterpret_cast<const float4*>(L.A) + p;
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    if (!CENTRE && b == (NB == 27 ? 13 : 4)) continue;
    if (!((mask >> b) & 1u)) R.a[b] = __ldg(A + (int64_t)b * L.d.nv);
  }
  R.d = __ldg(reinterpret_cast<const float4*>(L.Dinv) + p);
}
template <int NB, bool CENTRE, bool SAME>
__device__ __forceinline__ void row_sum(const LevelOp& L, int64_t p, int par, const float2* __restrict__ x, uint32_t mask,
                                        const RowF32<NB>& R, float& s0, float& s1) {
  float2 xv[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    if (!CENTRE && b == (NB == 27 ? 13 : 4)) continue;
    if (!((mask >> b) & 1u)) xv[b] = ld_xn<SAME, NB>(x + p + (par ? L.nb.off[1][b] : L.nb.off[0][b]), b);
  }
  RowAcc<float> a0, a1;
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    if ((!CENTRE && b == (NB == 27 ? 13 : 4)) || ((mask >> b) & 1u)) continue;
    a0.add(R.a[b].x, R.a[b].y, xv[b]);
    a1.add(R.a[b].z, R.a[b].w, xv[b]);
  }
  s0 = a0.value();
  s1 = a1.value();
}
// (A x)_p with A = shift*M - J on the finest level, as apply_row
template <int NB, bool FINE>
__device__ __forceinline__ void row_apply(const LevelOp& L, int64_t p, const float2* __restrict__ x, const RowF32<NB>& R,
                                          float& s0, float& s1) {
  const int par = (int)((uint32_t)p % (uint32_t)L.d.nx) >= L.d.E;   // nv < 2^31
  row_sum<NB, true, false>(L, p, par, x, 0u, R, s0, s1);
  if (FINE) {
    const double2 m = reinterpret_cast<const double2*>(L.mdiag)[p];
    const float xs = x[p].y, sh = (float)L.shift;
    s0 = (sh * (float)m.x) * xs - s0;
    s1 = (sh * (float)m.y) * xs - s1;
  }
}

template <int NB, bool FINE>
__global__ void __launch_bounds__(64) k_residual_small(const __grid_constant__ LevelOp L, const float2* __restrict__ b,
                                                       const float2* __restrict__ x, float2* __restrict__ r) {
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  RowF32<NB> R;
  if (p < L.d.nv) row_load<NB, true>(L, p, 0u, R);
  rf_pdl_begin(b, x);
  if (p >= L.d.nv) return;
  const float2 bv = b[p];
  float s0, s1;
  row_apply<NB, FINE>(L, p, x, R, s0, s1);
  r[p] = make_float2(bv.x - s0, bv.y - s1);
}

template <int NB, bool FINE>
__global__ void __launch_bounds__(64) k_jacobi_small(const __grid_constant__ LevelOp L, const float2* __restrict__ b,
                                                     const float2* __restrict__ xin, float2* __restrict__ xout, double omega) {
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  RowF32<NB> R;
  if (p < L.d.nv) row_load<NB, true>(L, p, 0u, R);
  rf_pdl_begin(b, xin);
  if (p >= L.d.nv) return;
  const float2 bv = b[p], x0 = xin[p];
  float s0, s1;
  row_apply<NB, FINE>(L, p, xin, R, s0, s1);
  const float r0 = bv.x - s0, r1 = bv.y - s1;
  const float y0 = R.d.x * r0 + R.d.y * r1, y1 = R.d.z * r0 + R.d.w * r1;
  xout[p] = make_float2(x0.x + (float)omega * y0, x0.y + (float)omega * y1);
}

template <int NB, bool FINE, int FPX>
__global__ void __launch_bounds__(GS_PAIR_MAX_THREADS) k_gs_pair_small(const __grid_constant__ LevelOp L,
                                                                       const float2* __restrict__ b, float2* __restrict__ x,
                                                                       int py, int pz, int lines_y,
                                                                       uint32_t skip_first, uint32_t skip_second) {
  // one line per block, one vertex per thread and run
  const int l0 = blockIdx.x, v = threadIdx.x;
  const int cnt0 = FPX ? L.d.nx / 2 : (L.d.nx + 1) / 2, cnt1 = FPX ? (L.d.nx + 1) / 2 : L.d.nx / 2;
  const bool on0 = v < cnt0, on1 = v < cnt1;
  const int64_t p0 = on0 ? pair_vertex(L.d, l0, v, cnt0, FPX, py, pz, lines_y) : 0;
  const int64_t p1 = on1 ? pair_vertex(L.d, l0, v, cnt1, 1 - FPX, py, pz, lines_y) : 0;
  RowF32<NB> R;
  if (on0) row_load<NB, false>(L, p0, skip_first, R);
  rf_pdl_begin(b, x);
  auto update = [&](int64_t p, float2 bv, float s0, float s1) {
    const float r0 = FINE ? bv.x + s0 : bv.x - s0, r1 = FINE ? bv.y + s1 : bv.y - s1;   // as gs_vertex
    x[p] = make_float2(R.d.x * r0 + R.d.y * r1, R.d.z * r0 + R.d.w * r1);
  };
  float s0, s1;
  const float2 b0 = on0 ? b[p0] : make_float2(0.f, 0.f), b1 = on1 ? b[p1] : make_float2(0.f, 0.f);
  if (on0) {
    row_sum<NB, false, false>(L, p0, FPX, x, skip_first, R, s0, s1);
    update(p0, b0, s0, s1);
  }
  if (on1) row_load<NB, false>(L, p1, skip_second, R);
  __syncthreads();
  if (on1) {
    row_sum<NB, false, true>(L, p1, 1 - FPX, x, skip_second, R, s0, s1);
    update(p1, b1, s0, s1);
  }
}

// ----------------------------------------------------------------- small FP64 levels
// Two neighbouring lanes per vertex, lane h its row h: a small FP64 level has
// fewer warps than the GPU has FP64 schedulers (one warp instruction takes 64
// cycles on each), so half the chain per thread is half the time.  As in the
// FP32 forms the matrix rows are loaded before griddepcontrol.wait.  Same sums in
// the same order; D^-1 and the updates as dinv_apply's callers.
template <int NB>
struct RowF64 {
  double2 a[NB], d;
};
template <int NB, bool CENTRE>
__device__ __forceinline__ void row_load(const LevelOp& L, int64_t p, int h, uint32_t mask, RowF64<NB>& R) {
  const double2* A = reinterpret_cast<const double2*>(L.A) + p * 2 + h;
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    if (!CENTRE && b == (NB == 27 ? 13 : 4)) continue;
    if (!((mask >> b) & 1u)) R.a[b] = __ldg(A + (int64_t)b * L.d.nv * 2);
  }
  R.d = __ldg(reinterpret_cast<const double2*>(L.Dinv) + p * 2 + h);
}
template <int NB, bool CENTRE, bool SAME>
__device__ __forceinline__ double row_sum(const LevelOp& L, int64_t p, int par, const double2* __restrict__ x, uint32_t mask,
                                          const RowF64<NB>& R) {
  RowAcc<double> s;
#pragma unroll
  for (int b0 = 0; b0 < NB; b0 += 9) {
    double2 xv[9];
#pragma unroll
    for (int c = 0; c < 9; ++c) {
      const int b = b0 + c;
      if ((!CENTRE && b == (NB == 27 ? 13 : 4)) || ((mask >> b) & 1u)) continue;
      xv[c] = ld_xn<SAME, NB>(x + p + (par ? L.nb.off[1][b] : L.nb.off[0][b]), b);
    }
#pragma unroll
    for (int c = 0; c < 9; ++c) {
      const int b = b0 + c;
      if ((!CENTRE && b == (NB == 27 ? 13 : 4)) || ((mask >> b) & 1u)) continue;
      s.add(R.a[b].x, R.a[b].y, xv[c]);
    }
  }
  return s.value();
}
// row h of A x at p with A = shift*M - J on the finest level, as apply_row
template <int NB, bool FINE>
__device__ __forceinline__ double row_apply(const LevelOp& L, int64_t p, int h, const double2* __restrict__ x, const RowF64<NB>& R) {
  const int par = (int)((uint32_t)p % (uint32_t)L.d.nx) >= L.d.E;   // nv < 2^31
  const double s = row_sum<NB, true, false>(L, p, par, x, 0u, R);
  if (!FINE) return s;
  const double m = L.mdiag[2 * p + h];
  return (L.shift * m) * x[p].y - s;
}
__device__ __forceinline__ double pair_other(double v) { return __shfl_xor_sync(3u << (threadIdx.x & 30), v, 1); }

template <int NB, bool FINE>
__global__ void __launch_bounds__(64) k_residual_small64(const __grid_constant__ LevelOp L, const double2* __restrict__ b,
                                                         const double2* __restrict__ x, double2* __restrict__ r) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, p = t >> 1;
  const int h = (int)(t & 1);
  RowF64<NB> R;
  if (p < L.d.nv) row_load<NB, true>(L, p, h, 0u, R);
  rf_pdl_begin(b, x);
  if (p >= L.d.nv) return;
  const double bv = reinterpret_cast<const double*>(b)[t];
  reinterpret_cast<double*>(r)[t] = bv - row_apply<NB, FINE>(L, p, h, x, R);
}

template <int NB, bool FINE>
__global__ void __launch_bounds__(64) k_jacobi_small64(const __grid_constant__ LevelOp L, const double2* __restrict__ b,
                                                       const double2* __restrict__ xin, double2* __restrict__ xout, double omega) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, p = t >> 1;
  const int h = (int)(t & 1);
  RowF64<NB> R;
  if (p < L.d.nv) row_load<NB, true>(L, p, h, 0u, R);
  rf_pdl_begin(b, xin);
  if (p >= L.d.nv) return;
  const double bv = reinterpret_cast<const double*>(b)[t], x0 = reinterpret_cast<const double*>(xin)[t];
  const double mine = bv - row_apply<NB, FINE>(L, p, h, xin, R), other = pair_other(mine);
  const double y = h ? R.d.x * other + R.d.y * mine : R.d.x * mine + R.d.y * other;
  reinterpret_cast<double*>(xout)[t] = x0 + omega * y;
}

template <int NB, bool FINE, int FPX>
__global__ void __launch_bounds__(NB == 27 ? 128 : 288) k_gs_pair_small64(const __grid_constant__ LevelOp L, const double2* __restrict__ b,
                                                        double2* __restrict__ x, int py, int pz, int lines_y,
                                                        uint32_t skip_first, uint32_t skip_second) {
  // one line per block (longer runs in several rounds)
  const int cnt0 = FPX ? L.d.nx / 2 : (L.d.nx + 1) / 2, cnt1 = FPX ? (L.d.nx + 1) / 2 : L.d.nx / 2;
  const int h = threadIdx.x & 1, v0 = threadIdx.x >> 1, step = blockDim.x >> 1;
  RowF64<NB> R;
  auto load = [&](int v, int cnt, int px, uint32_t skip) {
    const int64_t p = pair_vertex(L.d, blockIdx.x, v, cnt, px, py, pz, lines_y);
    row_load<NB, false>(L, p, h, skip, R);
    return p;
  };
  auto update = [&](auto same, int64_t p, int px, uint32_t skip) {
    const double bv = reinterpret_cast<const double*>(b)[2 * p + h];
    const double s = row_sum<NB, false, decltype(same)::value>(L, p, px, x, skip, R);
    const double mine = FINE ? bv + s : bv - s, other = pair_other(mine);   // as gs_vertex
    reinterpret_cast<double*>(x)[2 * p + h] = h ? R.d.x * other + R.d.y * mine : R.d.x * mine + R.d.y * other;
  };
  int64_t p = v0 < cnt0 ? load(v0, cnt0, FPX, skip_first) : 0;
  rf_pdl_begin(b, x);
  for (int v = v0; v < cnt0;) {
    update(std::false_type{}, p, FPX, skip_first);
    v += step;
    if (v < cnt0) p = load(v, cnt0, FPX, skip_first);
  }
  __syncthreads();
  for (int v = v0; v < cnt1; v += step) {
    p = load(v, cnt1, 1 - FPX, skip_second);
    update(std::true_type{}, p, 1 - FPX, skip_second);
  }
}

// ----------------------------------------------------------------- transfers
template <typename T>
__device__ __forceinline__ typename V2<T>::t restrict_value(const Dims& df, const Dims& dc, const uint8_t* __restrict__ dmf,
                                                            const uint8_t* __restrict__ dmc,
                                                            const typename V2<T>::t* rf, int64_t pc, int I, int J, int K) {
  typedef typename V2<T>::t V;
  const bool mc = dmc[pc] != 0;
  // all 3^d fine values and masks are loaded first (one memory round trip),
  // then summed in the fixed (dz, dy, dx) order
  V r[27];
  uint8_t m[27];
  bool in[27];
#pragma unroll
  for (int q = 0; q < 27; ++q) {
    const int dx = q % 3 - 1, dy = (q / 3) % 3 - 1, dz = q / 9 - 1;
    const int fi = 2 * I + dx, fj = 2 * J + dy, fk = df.dim == 3 ? 2 * K + dz : 0;
    in[q] = (df.dim == 3 || dz == 0) && fi >= 0 && fi < df.nx && fj >= 0 && fj < df.ny && fk >= 0 && fk < df.nz;
    if (in[q]) {
      const int64_t pf = pidx(df, fi, fj, fk);
      r[q] = rf[pf];
      m[q] = dmf[pf];
    } else {
      r[q].x = 0;
      r[q].y = 0;
      m[q] = 1;
    }
  }
  T s0 = 0, s1 = 0;
#pragma unroll
  for (int q = 0; q < 27; ++q) {
    if (!in[q]) continue;
    const int dx = q % 3 - 1, dy = (q / 3) % 3 - 1, dz = q / 9 - 1;
    const T w = (T)((dx ? 0.5 : 1.0) * (dy ? 0.5 : 1.0) * (dz ? 0.5 : 1.0));
    if (!(mc || m[q])) s0 += w * r[q].x;
    s1 += w * r[q].y;
  }
  V o;
  o.x = s0;
  o.y = s1;
  return o;
}

template <typename T>
__device__ __forceinline__ void restrict_point(const Dims& df, const Dims& dc, const uint8_t* __restrict__ dmf,
                                               const uint8_t* __restrict__ dmc, const typename V2<T>::t* __restrict__ rf,
                                               typename V2<T>::t* __restrict__ bc, int64_t pc) {
  int I, J, K;
  pcoords(dc, pc, I, J, K);
  bc[pc] = restrict_value<T>(df, dc, dmf, dmc, rf, pc, I, J, K);
}

template <typename T>
__global__ void __launch_bounds__(256) k_restrict(Dims df, Dims dc, const uint8_t* __restrict__ dmf,
                                                  const uint8_t* __restrict__ dmc,
                                                  const typename V2<T>::t* __restrict__ rf,
                                                  typename V2<T>::t* __restrict__ bc) {
  rf_pdl_begin(rf);
  int64_t pc = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (pc >= dc.nv) return;
  restrict_point<T>(df, dc, dmf, dmc, rf, bc, pc);
}

// the corrected fine value x_f + (P x_c)
template <typename T, typename XC>
__device__ __forceinline__ typename V2<T>::t prolong_value(const Dims& df, const Dims& dc, const uint8_t* __restrict__ dmf,
                                                           const uint8_t* __restrict__ dmc, XC xc,
                                                           const typename V2<T>::t* xf, int64_t pf, int fi, int fj, int fk) {
  typedef typename V2<T>::t V;
  const bool mf = dmf[pf] != 0;
  // the (up to) 2^d coarse parents, loaded first, summed in (K, J, I) order
  V c[8];
  uint8_t m[8];
  bool in[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int K = (fk >> 1) + ((q >> 2) & 1), J = (fj >> 1) + ((q >> 1) & 1), I = (fi >> 1) + (q & 1);
    in[q] = ((q & 1) == 0 || (fi & 1)) && (((q >> 1) & 1) == 0 || (fj & 1)) &&
            (((q >> 2) & 1) == 0 || (fk & 1)) && K < dc.nz && J < dc.ny && I < dc.nx;
    if (in[q]) {
      const int64_t pc = pidx(dc, I, J, K);
      c[q] = xc((int)pc);
      m[q] = dmc[pc];
    } else {
      c[q].x = 0;
      c[q].y = 0;
      m[q] = 1;
    }
  }
  const T wz = (df.dim == 3 && (fk & 1)) ? (T)0.5 : (T)1;
  const T wy = (fj & 1) ? (T)0.5 : (T)1;
  const T w = ((fi & 1) ? (T)0.5 : (T)1) * wy * wz;
  T s0 = 0, s1 = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    if (!in[q]) continue;
    if (!(mf || m[q])) s0 += w * c[q].x;
    s1 += w * c[q].y;
  }
  V o = xf[pf];
  o.x += s0;
  o.y += s1;
  return o;
}

template <typename T>
__device__ __forceinline__ void prolong_point(const Dims& df, const Dims& dc, const uint8_t* __restrict__ dmf,
                                              const uint8_t* __restrict__ dmc, const typename V2<T>::t* __restrict__ xc,
                                              typename V2<T>::t* __restrict__ xf, int64_t pf) {
  int fi, fj, fk;
  pcoords(df, pf, fi, fj, fk);
  xf[pf] = prolong_value<T>(df, dc, dmf, dmc, [&](int pc) { return xc[pc]; }, xf, pf, fi, fj, fk);
}

template <typename T>
__global__ void __launch_bounds__(256) k_prolong(Dims df, Dims dc, const uint8_t* __restrict__ dmf,
                                                 const uint8_t* __restrict__ dmc,
                                                 const typename V2<T>::t* __restrict__ xc,
                                                 typename V2<T>::t* __restrict__ xf) {
  rf_pdl_begin(xc, xf);
  int64_t pf = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (pf >= df.nv) return;
  prolong_point<T>(df, dc, dmf, dmc, xc, xf, pf);
}

// The same transfers, organised for memory-level parallelism.  The per-point
// kernels above put each gathered load behind its own bounds branch.  These
// issue every load before the first sum: a value outside the grid is read at
// an in-grid address and then skipped.  They also take the vertex from the
// launch shape (a plane per blockIdx.y, the position within it by one 32-bit
// division) and compute the gathered lines' offsets once per vertex, instead
// of pcoords and a 64-bit pidx per value.  Loads, masks, weights and the order
// of the sums are those of restrict_point / prolong_point, so the results are
// bitwise equal.  At 257^3 the transfers take 3.14 ms per solve against 4.14.
template <typename T>
__device__ __forceinline__ void restrict_planes_body(const Dims& df, const Dims& dc, const uint8_t* __restrict__ dmf,
                                                     const uint8_t* __restrict__ dmc,
                                                     const typename V2<T>::t* __restrict__ rf,
                                                     typename V2<T>::t* __restrict__ bc) {
  rf_pdl_begin(rf);
  typedef typename V2<T>::t V;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= dc.nx * dc.ny) return;
  const int J = t / dc.nx, pos = t - J * dc.nx, K = blockIdx.y;
  const int I = pos < dc.E ? 2 * pos : 2 * (pos - dc.E) + 1;
  // 32-bit vertex indices: a grid has at most 2^31 vertices (rf_grid_create)
  const int pc = (J + dc.ny * K) * dc.nx + pos;
  const bool mc = dmc[pc] != 0;
  int xo[3];
  bool xin[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int fi = 2 * I + a - 1;
    xin[a] = fi >= 0 && fi < df.nx;
    xo[a] = (fi & 1) ? df.E + (fi >> 1) : (fi >> 1);
  }
  int lo[9];
  bool lin[9];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int fj = 2 * J + b - 1, fk = df.dim == 3 ? 2 * K + c - 1 : 0;
      lin[3 * c + b] = (df.dim == 3 || c == 1) && fj >= 0 && fj < df.ny && fk >= 0 && fk < df.nz;
      lo[3 * c + b] = lin[3 * c + b] ? (fj + df.ny * fk) * df.nx : 0;   // (no overflow outside the grid)
    }
  // every load is issued, without a branch, before the first sum: a value
  // outside the grid is read at the vertex's own fine position (always
  // inside) and then skipped, so the 27 loads are one memory round trip
  const int pf0 = lo[4] + xo[1];
  V r[27];
  uint8_t m[27];
  bool in[27];
#pragma unroll
  for (int q = 0; q < 27; ++q) {
    const int a = q % 3, bc3 = q / 3;   // bc3 = 3 * (dz + 1) + (dy + 1)
    in[q] = lin[bc3] && xin[a];
    const int pf = in[q] ? lo[bc3] + xo[a] : pf0;
    r[q] = rf[pf];
    m[q] = dmf[pf];
  }
  T s0 = 0, s1 = 0;
#pragma unroll
  for (int q = 0; q < 27; ++q) {
    if (!in[q]) continue;
    const int dx = q % 3 - 1, dy = (q / 3) % 3 - 1, dz = q / 9 - 1;
    const T w = (T)((dx ? 0.5 : 1.0) * (dy ? 0.5 : 1.0) * (dz ? 0.5 : 1.0));
    if (!(mc || m[q])) s0 += w * r[q].x;
    s1 += w * r[q].y;
  }
  V o;
  o.x = s0;
  o.y = s1;
  bc[pc] = o;
}

template <typename T>
__global__ void __launch_bounds__(256) k_restrict_planes(Dims df, Dims dc, const uint8_t* __restrict__ dmf,
                                                         const uint8_t* __restrict__ dmc,
                                                         const typename V2<T>::t* __restrict__ rf,
                                                         typename V2<T>::t* __restrict__ bc) {
  restrict_planes_body<T>(df, dc, dmf, dmc, rf, bc);
}

// Prolongation and correction x_f += P x_c, two fine vertices per thread:
// thread (I, fj, fk) updates fine vertex 2I (even half of the parity-split
// line) and 2I + 1 (odd half), whose coarse parents along x are I, and I and
// I + 1.  Their (up to 8) parents are loaded once, before the first sum (one
// memory round trip; a parent outside the coarse grid is read at coarse
// vertex 0 and skipped).  Each fine value then sums its parents in the
// (K, J, I) order of prolong_point with the same expressions, so the results
// are the per-point kernel's bit for bit.  The pairing halves the gathered
// loads and the index arithmetic per fine vertex (the one-vertex-per-thread
// form issued ~330 instructions per vertex and was issue-bound).
template <typename T>
__device__ __forceinline__ void prolong_pairs_body(const Dims& df, const Dims& dc, const uint8_t* __restrict__ dmf,
                                                   const uint8_t* __restrict__ dmc,
                                                   const typename V2<T>::t* __restrict__ xc,
                                                   typename V2<T>::t* __restrict__ xf) {
  rf_pdl_begin(xc, xf);
  typedef typename V2<T>::t V;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= dc.nx * df.ny) return;
  const int fj = t / dc.nx, I = t - fj * dc.nx, fk = blockIdx.y;
  const int J0 = fj >> 1, K0 = fk >> 1;
  const bool oy = (fj & 1) != 0, oz = df.dim == 3 && (fk & 1) != 0;
  const bool odd = 2 * I + 1 < df.nx;   // fine vertex 2I + 1 exists
  // 32-bit vertex indices: a grid has at most 2^31 vertices (rf_grid_create)
  const int fline = (fj + df.ny * fk) * df.nx;
  const int pe = fline + I, po = fline + df.E + I;
  const int xo[2] = {(I & 1) ? dc.E + (I >> 1) : (I >> 1), ((I + 1) & 1) ? dc.E + ((I + 1) >> 1) : ((I + 1) >> 1)};
  V c8[8];
  uint8_t m[8];
  bool in[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int ib = q & 1, jb = (q >> 1) & 1, kb = (q >> 2) & 1;
    in[q] = (!jb || oy) && (!kb || oz) && (!ib || odd) && K0 + kb < dc.nz && J0 + jb < dc.ny && I + ib < dc.nx;
    const int pc = in[q] ? ((J0 + jb) + dc.ny * (K0 + kb)) * dc.nx + xo[ib] : 0;
    c8[q] = xc[pc];
    m[q] = dmc[pc];
  }
  const V xe = xf[pe];
  const bool me = dmf[pe] != 0;
  V xo_v = xe;
  bool mo = false;
  if (odd) {
    xo_v = xf[po];
    mo = dmf[po] != 0;
  }
  const T wz = oz ? (T)0.5 : (T)1;
  const T wy = oy ? (T)0.5 : (T)1;
  {
    const T w = (T)1 * wy * wz;   // fine x even
    T s0 = 0, s1 = 0;
#pragma unroll
    for (int q = 0; q < 8; q += 2) {
      if (!in[q]) continue;
      if (!(me || m[q])) s0 += w * c8[q].x;
      s1 += w * c8[q].y;
    }
    V o = xe;
    o.x += s0;
    o.y += s1;
    xf[pe] = o;
  }
  if (odd) {
    const T w = (T)0.5 * wy * wz;   // fine x odd
    T s0 = 0, s1 = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      if (!in[q]) continue;
      if (!(mo || m[q])) s0 += w * c8[q].x;
      s1 += w * c8[q].y;
    }
    V o = xo_v;
    o.x += s0;
    o.y += s1;
    xf[po] = o;
  }
}

template <typename T>
__global__ void __launch_bounds__(256) k_prolong_planes(Dims df, Dims dc, const uint8_t* __restrict__ dmf,
                                                        const uint8_t* __restrict__ dmc,
                                                        const typename V2<T>::t* __restrict__ xc,
                                                        typename V2<T>::t* __restrict__ xf) {
  prolong_pairs_body<T>(df, dc, dmf, dmc, xc, xf);
}

// ----------------------------------------------------------------- coarsest solve
// x = A^-1 b on the coarsest level: one warp per row of the explicit
// inverse, lanes over its columns (coalesced), FP64 sums.
template <typename T>
__device__ __forceinline__ void coarse_solve_body(int N, const double* __restrict__ Ainv, const T* __restrict__ b,
                                                  T* __restrict__ x) {
  rf_pdl_begin(b);
  extern __shared__ double sb[];
  for (int t = threadIdx.x; t < N; t += blockDim.x) sb[t] = (double)b[t];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (r >= N) return;
  const double* row = Ainv + (int64_t)r * N;
  double s = 0.0;
  for (int c = lane; c < N; c += 32) s += row[c] * sb[c];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) x[r] = (T)s;
}

template <typename T>
__global__ void __launch_bounds__(256) k_coarse_solve(int N, const double* __restrict__ Ainv,
                                                      const T* __restrict__ b, T* __restrict__ x) {
  coarse_solve_body<T>(N, Ainv, b, x);
}

// ----------------------------------------------------------------- V-cycle tail
// Levels below a few 10^4 vertices cannot fill the GPU: launched one kernel per
// GS colour, each costs a launch gap.  Here one launch runs the whole V-cycle
// from level `first` down to the coarsest and back up, its phases separated by
// barriers (every thread reaches every barrier: all loop bounds below are
// uniform across the launch).  Two forms:
//   k_vcycle_tail: ONE thread-block cluster, hardware cluster barriers;
//   k_vcycle_coop: a cooperative launch of every co-resident block, grid
//     barriers in global memory whose waits give up after P.limit_ns (the
//     block then sets *P.status = 1 and leaves; the others see the flag in
//     their own waits and leave too, so the kernel always ends).

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Grid barrier of a cooperative launch: bar[0] counts this generation's
// arrivals, bar[1] is the generation.  `gen` (held by thread 0) is the
// generation this block last passed.  The last block to arrive resets the
// count and then publishes gen + 1; the others wait for it, at most limit_ns.
// Returns false when the wait gave up or another block already had.
__device__ __forceinline__ bool grid_sync_bounded(unsigned* bar, unsigned expected, unsigned& gen,
                                                  double* status, long long limit_ns) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    const unsigned want = gen + 1;
    __threadfence();   // this block's phase results before its arrival
    if (atomicAdd(&bar[0], 1u) == expected - 1) {
      atomicExch(&bar[0], 0u);
      __threadfence();
      atomicExch(&bar[1], want);
    } else {
      const unsigned long long t0 = global_ns();
      while (*(volatile unsigned*)&bar[1] != want) {
        if (*(volatile double*)status != 0.0 || (long long)(global_ns() - t0) > limit_ns) {
          *(volatile double*)status = 1.0;
          ok = 0;
          break;
        }
        __nanosleep(64);
      }
    }
    __threadfence();   // the other blocks' results are read after the barrier
    gen = want;
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// The V-cycle below level P.first; sync() separates phases and returns false
// when the launch must end (coop: a barrier gave up).
template <int KIND, int NB, typename Sync>
__device__ __forceinline__ void vcycle_tail_body(const TailParams& P, int64_t gt, int64_t nthr, Sync&& sync) {
  typedef typename Ty<KIND>::T T;
  typedef typename V2<T>::t V;
  // batched stencil loads (a thread's round trips set a phase's time); FP64
  // blocks three at a time, which keeps the whole V-cycle within the registers
  constexpr int CH = KIND == STORE_F64 ? 3 : chunk_of(KIND);
  const int ncol = 1 << P.L[P.first].op.d.dim;
  V* curs[RF_MAXL];
  auto gs_sweep = [&](const LevelOp& op, const V* b, V* x, bool forward, bool zero_start) {
    for (int cc = 0; cc < ncol; ++cc) {
      const int col = forward ? cc : ncol - 1 - cc;
      const int px = col & 1, py = (col >> 1) & 1, pz = (col >> 2) & 1;
      const int cnt_x = px ? op.d.nx / 2 : (op.d.nx + 1) / 2;
      const int lines_y = (op.d.ny - py + 1) / 2;
      const int lines_z = op.d.dim == 3 ? (op.d.nz - pz + 1) / 2 : 1;
      const int64_t count = (int64_t)cnt_x * lines_y * lines_z;
      const uint32_t skip = (zero_start && forward) ? P.zmask[col] : 0u;
      for (int64_t t = gt; t < count; t += nthr) gs_point<KIND, false, NB, CH>(op, b, x, px, py, pz, cnt_x, lines_y, t, skip);
      if (!sync()) return false;
    }
    return true;
  };
  auto jacobi_sweep = [&](const LevelOp& op, const V* b, const V* xin, V* xout, bool zero_x) {
    for (int64_t p = gt; p < op.d.nv; p += nthr) jacobi_point<KIND, false, NB, CH>(op, b, xin, xout, P.omega, zero_x, p);
    return sync();
  };
  for (int l = P.first; l < P.coarsest; ++l) {
    const TailLevel& Lv = P.L[l];
    const TailLevel& Lc = P.L[l + 1];
    const V* b = (const V*)Lv.b;
    V* x = (V*)Lv.x;
    V* tmp = (V*)Lv.t;
    V* cur = x;
    if (P.smoother == 1) {
      for (int sw = 0; sw < P.nu1; ++sw)
        if (!gs_sweep(Lv.op, b, x, true, sw == 0)) return;
    } else {
      V* first = ((P.nu1 + P.nu2) & 1) ? x : tmp;
      if (!jacobi_sweep(Lv.op, b, nullptr, first, true)) return;
      cur = first;
      for (int sw = 1; sw < P.nu1; ++sw) {
        V* dst = (cur == x) ? tmp : x;
        if (!jacobi_sweep(Lv.op, b, cur, dst, false)) return;
        cur = dst;
      }
    }
    curs[l] = cur;
    for (int64_t p = gt; p < Lv.op.d.nv; p += nthr) residual_point<KIND, false, NB, CH>(Lv.op, b, cur, (V*)Lv.r, p);
    if (!sync()) return;
    for (int64_t p = gt; p < Lc.op.d.nv; p += nthr)
      restrict_point<T>(Lv.op.d, Lc.op.d, Lv.op.dmask, Lc.op.dmask, (const V*)Lv.r, (V*)Lc.b, p);
    if (!sync()) return;
  }
  {
    // x = A^-1 b on the coarsest level, one warp per row with lanes over the
    // columns and the xor-shuffle sum of coarse_solve_body: the same values
    // as the coarse-solve kernel, so the tail equals the V-cycle of
    // one launch per phase bit for bit
    const T* bc = (const T*)P.L[P.coarsest].b;
    T* xc = (T*)P.L[P.coarsest].x;
    const int lane = (int)(gt & 31);
    for (int64_t r = gt >> 5; r < P.N; r += nthr >> 5) {   // uniform per warp: nthr is a multiple of 32
      const double* row = P.Ainv + r * P.N;
      double s = 0.0;
      for (int c = lane; c < P.N; c += 32) s += row[c] * (double)bc[c];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) xc[r] = (T)s;
    }
    if (!sync()) return;
  }
  for (int l = P.coarsest - 1; l >= P.first; --l) {
    const TailLevel& Lv = P.L[l];
    const TailLevel& Lc = P.L[l + 1];
    const V* b = (const V*)Lv.b;
    V* x = (V*)Lv.x;
    V* tmp = (V*)Lv.t;
    V* cur = curs[l];
    for (int64_t p = gt; p < Lv.op.d.nv; p += nthr)
      prolong_point<T>(Lv.op.d, Lc.op.d, Lv.op.dmask, Lc.op.dmask, (const V*)Lc.x, cur, p);
    if (!sync()) return;
    if (P.smoother == 1) {
      for (int sw = 0; sw < P.nu2; ++sw)
        if (!gs_sweep(Lv.op, b, x, false, false)) return;
    } else {
      for (int sw = 0; sw < P.nu2; ++sw) {
        V* dst = (cur == x) ? tmp : x;
        if (!jacobi_sweep(Lv.op, b, cur, dst, false)) return;
        cur = dst;
      }
    }
  }
}

template <int KIND, int NB>
__global__ void __launch_bounds__(TAIL_THREADS) k_vcycle_tail(const __grid_constant__ TailParams P) {
  cg::cluster_group cl = cg::this_cluster();
  const int64_t nthr = (int64_t)cl.num_blocks() * blockDim.x;
  const int64_t gt = (int64_t)cl.block_rank() * blockDim.x + threadIdx.x;
  vcycle_tail_body<KIND, NB>(P, gt, nthr, [&]() {
    cl.sync();
    return true;
  });
}

// The cluster tail with its vectors in shared memory.  Every CTA of the cluster
// keeps a copy of x (Jacobi: of both iterates) of every tail level, zero halo
// included, and owns the x-lines rank + cs * i of each level: it computes their
// values and stores each into the copies of the CTAs that own a neighbouring line
// (distributed shared memory), so a phase reads x and b from its own shared
// memory and costs one cluster barrier.
// The blocks and D^-1 of the own lines are copied to shared memory too (cp.async,
// before the predecessor's results are waited for), the smallest levels first
// as far as they fit; other levels stream them from L2.  GS sweeps colour
// pairs as k_gs_pair does (all kinds: here the pair saves a barrier): the pair's
// second colour reaches the first only on its own line, so a block barrier
// lies between them.  r crosses through global memory (one phase per level).
// Sums, order and operations per vertex are those of the launch-per-phase
// kernels, bit for bit.  Bound by latency: at 17^3 and below a pair phase is two
// chains of 26 blocks from shared memory (0.3 us each), 5 remote stores and the
// barrier (0.4 us).  With x read through L2 the V-cycle from 17^3 down took 180 us
// (FP32 GS), now 100; FP64 GS, then 32 launches a level, 33^3 solve's coarse part
// 690 -> 270 us a V-cycle, 2D from 129 x 65 down 430 -> 230 us.
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// What a CTA of k_vcycle_cl needs of one level, read from the parameters once
// per level and sweep: indexed reads of them in the row loops (a neighbour
// table, say) cost more than the sums.
struct ClLevel {
  int nx, ny, pl, E, xl0, xr0, xl1, xr1;   // pl = nx ny; x offsets of dx = -1, +1 for even and odd vertices
  int rows, lines, nlines;
  float inv_nx;
  uint32_t peers;                          // CTAs that own a line next to one of this CTA's, this one included
  int64_t nv;
  const void* A;
  const void* Dinv;
  const float4* sA;
};

// a / d for 0 <= a < 2^20 with inv = 1.0f / d: the quotient's distance to the
// next whole number, at least 1 / (2 d), is beyond the rounding of the product
__device__ __forceinline__ int cl_div(int a, float inv) { return (int)(((float)a + 0.5f) * inv); }

// Residual b - (stencil sum) of local row lr = vertex p, x and b in shared memory,
// the blocks there or (L.sA null) in global memory, CH at a time: their loads
// first (MASKED: blocks of skipmask left out; a sweep that skips none keeps
// its loads free of branches), then the sums in stencil order.  FP64: a pair of
// neighbouring lanes shares a vertex, lane h sums its row h (an SM's FP64 pipe
// takes 64 cycles per warp instruction on each of its four schedulers, and a
// cluster's few rows leave most of them idle); both get both residuals.
template <int KIND, int NB, bool CENTRE, bool MASKED>
__device__ __forceinline__ void cl_residual(const ClLevel& L, int lr, int p, int par, int h,
                                            const typename V2<typename Ty<KIND>::T>::t* x,
                                            const typename V2<typename Ty<KIND>::T>::t bv, uint32_t skipmask,
                                            typename Ty<KIND>::T& r0, typename Ty<KIND>::T& r1) {
  typedef typename Ty<KIND>::T T;
  constexpr int C = NB == 27 ? 13 : 4;
  const int xl = par ? L.xl1 : L.xl0, xr = par ? L.xr1 : L.xr0;
  auto xat = [&](int b) {
    const int dx = b % 3 - 1, dy = (b / 3) % 3 - 1, dz = b / 9 - (NB == 27 ? 1 : 0);
    return x[p + (dx < 0 ? xl : dx > 0 ? xr : 0) + dy * L.nx + dz * L.pl];
  };
  auto skipped = [&](int b) { return (!CENTRE && b == C) || (MASKED && ((skipmask >> b) & 1u)); };
  if constexpr (KIND == STORE_F64) {
    const double2* sm = reinterpret_cast<const double2*>(L.sA) + h * L.rows + lr;
    const double2* gm = reinterpret_cast<const double2*>(L.A) + (int64_t)p * 2 + h;
    RowAcc<double> a0;
    auto sum = [&](auto shared) {
      constexpr int CH = decltype(shared)::value ? 3 : 9;
#pragma unroll
      for (int b0 = 0; b0 < NB; b0 += CH) {
        double2 a[CH], xv[CH];
#pragma unroll
        for (int c = 0; c < CH; ++c)
          if (!skipped(b0 + c)) a[c] = decltype(shared)::value ? sm[2 * (b0 + c) * L.rows] : __ldg(gm + (int64_t)(b0 + c) * L.nv * 2);
#pragma unroll
        for (int c = 0; c < CH; ++c)
          if (!skipped(b0 + c)) xv[c] = xat(b0 + c);
#pragma unroll
        for (int c = 0; c < CH; ++c)
          if (!skipped(b0 + c)) a0.add(a[c].x, a[c].y, xv[c]);
      }
    };
    if (L.sA) sum(std::true_type{});
    else sum(std::false_type{});
    const double mine = (h ? bv.y : bv.x) - a0.value();
    const double other = __shfl_xor_sync(3u << (threadIdx.x & 30), mine, 1);
    r0 = h ? other : mine;
    r1 = h ? mine : other;
  } else {
    RowAcc<T> a0, a1;
    auto sum = [&](auto shared) {
      constexpr int CH = 9;
#pragma unroll
      for (int b0 = 0; b0 < NB; b0 += CH) {
        float4 a[CH];
        float2 xv[CH];
#pragma unroll
        for (int c = 0; c < CH; ++c)
          if (!skipped(b0 + c))
            a[c] = decltype(shared)::value ? L.sA[(b0 + c) * L.rows + lr]
                                           : __ldg(reinterpret_cast<const float4*>(L.A) + (int64_t)(b0 + c) * L.nv + p);
#pragma unroll
        for (int c = 0; c < CH; ++c)
          if (!skipped(b0 + c)) xv[c] = xat(b0 + c);
#pragma unroll
        for (int c = 0; c < CH; ++c)
          if (!skipped(b0 + c)) {
            a0.add(a[c].x, a[c].y, xv[c]);
            a1.add(a[c].z, a[c].w, xv[c]);
          }
      }
    };
    if (L.sA) sum(std::true_type{});
    else sum(std::false_type{});
    r0 = bv.x - a0.value();
    r1 = bv.y - a1.value();
  }
}

template <int KIND, int NB>
__global__ void __launch_bounds__(TAIL_THREADS, 1) k_vcycle_cl(const __grid_constant__ TailParams P) {
  typedef typename Ty<KIND>::T T;
  typedef typename V2<T>::t V;
  constexpr int PARTS = KIND == STORE_F64 ? 2 : 1;   // 16-byte parts of a block
  constexpr int RS = PARTS;                          // threads per vertex
  extern __shared__ __align__(16) unsigned char cl_raw[];
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), cs = P.cl_cs, tid = threadIdx.x, nt = blockDim.x;
  auto xbuf = [&](int l) { return reinterpret_cast<V*>(cl_raw + P.cl_x[l]); };   // interior (after the halo)
  auto tbuf = [&](int l) { return reinterpret_cast<V*>(cl_raw + P.cl_t[l]); };
  auto bbuf = [&](int l) { return reinterpret_cast<V*>(cl_raw + P.cl_b[l]); };   // own rows (coarsest: all)
  // the own lines of level l by (y, z) parity: their counts, then their numbers
  auto list = [&](int l, int cls) { return reinterpret_cast<int*>(cl_raw + P.cl_list[l]) + 4 + cls * (P.cl_rows[l] / P.L[l].op.d.nx); };
  auto count = [&](int l, int cls) { return reinterpret_cast<int*>(cl_raw + P.cl_list[l])[cls]; };
  auto level = [&](int l) {
    const LevelOp& op = P.L[l].op;
    ClLevel L;
    L.nx = op.d.nx; L.ny = op.d.ny; L.E = op.d.E; L.pl = NB == 27 ? op.d.nx * op.d.ny : 0;
    L.xl0 = L.E - 1; L.xr0 = L.E; L.xl1 = -L.E; L.xr1 = 1 - L.E;
    L.rows = P.cl_rows[l];
    L.inv_nx = 1.0f / (float)L.nx;
    L.lines = cl_div(L.rows, L.inv_nx);
    L.nlines = op.d.ny * (NB == 27 ? op.d.nz : 1);
    L.nv = op.d.nv;
    L.A = op.A;
    L.Dinv = op.Dinv;
    L.sA = P.cl_a[l] >= 0 ? reinterpret_cast<const float4*>(cl_raw + P.cl_a[l]) : nullptr;
    // line Ln = rank + cs * i, so its neighbours' owners are the same for every own line
    L.peers = 0;
#pragma unroll
    for (int c = -1; c <= 1; ++c) {
      const int o = rank + (NB == 27 ? c * L.ny : 0);
      L.peers |= 1u << ((o - 1) & (cs - 1)) | 1u << (o & (cs - 1)) | 1u << ((o + 1) & (cs - 1));
    }
    return L;
  };
  auto put = [&](uint32_t peers, auto* dst, auto v) {   // into the copies of these CTAs
    for (uint32_t m = peers; m; m &= m - 1) *cl.map_shared_rank(dst, __ffs(m) - 1) = v;
  };
  const uint32_t everyone = cs == 32 ? ~0u : (1u << cs) - 1;
  // zeros in every vector (reads of neighbours outside the grid, and of colours
  // not yet visited, must meet finite values), the matrices, the line lists
  for (int t = tid; t < P.cl_vec_bytes / 16; t += nt) reinterpret_cast<float4*>(cl_raw)[t] = make_float4(0.f, 0.f, 0.f, 0.f);
  __syncthreads();
  for (int l = P.first; l < P.coarsest; ++l) {
    const ClLevel L = level(l);
    if (L.sA) {
      float4* dst = const_cast<float4*>(L.sA);
      const float4* A = reinterpret_cast<const float4*>(L.A);
      const float4* D = reinterpret_cast<const float4*>(L.Dinv);
      for (int lr = tid; lr < L.rows; lr += nt) {
        const int i = cl_div(lr, L.inv_nx), Ln = rank + cs * i, p = Ln * L.nx + (lr - i * L.nx);
        if (Ln >= L.nlines) continue;
        for (int b = 0; b < NB; ++b)
#pragma unroll
          for (int h = 0; h < PARTS; ++h) cp_async16(dst + (b * PARTS + h) * L.rows + lr, A + ((int64_t)b * L.nv + p) * PARTS + h);
#pragma unroll
        for (int h = 0; h < PARTS; ++h) cp_async16(dst + (NB * PARTS + h) * L.rows + lr, D + (int64_t)p * PARTS + h);
      }
    }
    if (tid < 4) {
      int n = 0;
      for (int i = 0; i < L.lines; ++i) {
        const int Ln = rank + cs * i;
        if (Ln >= L.nlines) break;
        const int k = Ln / L.ny, j = Ln - k * L.ny;
        if (((j & 1) | (k & 1) << 1) == tid) list(l, tid)[n++] = i;
      }
      reinterpret_cast<int*>(cl_raw + P.cl_list[l])[tid] = n;
    }
  }
  __syncthreads();
  rf_pdl_begin();
  {
    const ClLevel L = level(P.first);
    const V* b = (const V*)P.L[P.first].b;
    V* sb = bbuf(P.first);
    for (int lr = tid; lr < L.rows; lr += nt) {
      const int i = cl_div(lr, L.inv_nx), Ln = rank + cs * i;
      if (Ln < L.nlines) sb[lr] = b[Ln * L.nx + (lr - i * L.nx)];
    }
  }
  cp_async_wait_all();
  cl.sync();               // every CTA's vectors are zero before a peer writes into them

  // D^-1 r of a row (FP64: the component of row h), then out = x + w D^-1 r (w = 0:
  // out = D^-1 r) into the peers' copies
  auto update = [&](const ClLevel& L, int lr, int p, int h, T r0, T r1, V* out, bool add, V xv, T w) {
    if constexpr (KIND == STORE_F64) {
      const double2 D = L.sA ? reinterpret_cast<const double2*>(L.sA)[(2 * NB + h) * L.rows + lr]
                             : __ldg(reinterpret_cast<const double2*>(L.Dinv) + (int64_t)p * 2 + h);
      const T y = D.x * r0 + D.y * r1;
      put(L.peers, reinterpret_cast<T*>(out + p) + h, add ? (h ? xv.y : xv.x) + w * y : y);
    } else {
      const float4 D = L.sA ? L.sA[NB * L.rows + lr] : __ldg(reinterpret_cast<const float4*>(L.Dinv) + p);
      const T y0 = D.x * r0 + D.y * r1, y1 = D.z * r0 + D.w * r1;
      V o;
      o.x = add ? xv.x + w * y0 : y0;
      o.y = add ? xv.y + w * y1 : y1;
      put(L.peers, out + p, o);
    }
  };
  auto gs_sweep = [&](int l, V* x, bool forward, bool zero_start) {
    const ClLevel L = level(l);
    const V* sb = bbuf(l);
    const int ncol = NB == 27 ? 8 : 4;
    const float inv_e = 1.0f / (float)L.E, inv_o = 1.0f / (float)(L.nx - L.E);
    V none;
    none.x = 0;
    none.y = 0;
#pragma unroll 1
    for (int cc = 0; cc < ncol; cc += 2) {
      const int c1 = forward ? cc : ncol - 1 - cc, cls = c1 >> 1, nln = count(l, cls);
      const int* ln = list(l, cls);
#pragma unroll 1
      for (int half = 0; half < 2; ++half) {
        const int col = half ? (c1 ^ 1) : c1, px = col & 1;
        const int cnt = px ? L.nx - L.E : L.E;
        const float inv = px ? inv_o : inv_e;
        const uint32_t skip = (zero_start && forward) ? P.zmask[col] : 0u;
        for (int t = tid; t < nln * cnt * RS; t += nt) {
          const int it = t / RS, h = t % RS, li = cl_div(it, inv), i = ln[li], u = (px ? L.E : 0) + it - li * cnt;
          const int p = (rank + cs * i) * L.nx + u, lr = i * L.nx + u;
          T r0, r1;
          if (skip) cl_residual<KIND, NB, false, true>(L, lr, p, px, h, x, sb[lr], skip, r0, r1);   // coarse level: A_pq as stored
          else cl_residual<KIND, NB, false, false>(L, lr, p, px, h, x, sb[lr], 0u, r0, r1);
          update(L, lr, p, h, r0, r1, x, false, none, (T)0);
        }
        if (half == 0) __syncthreads();
      }
      cl.sync();
    }
  };
  auto jacobi_sweep = [&](int l, const V* xin, V* xout, bool zero_x) {
    const ClLevel L = level(l);
    const V* sb = bbuf(l);
    for (int t = tid; t < L.rows * RS; t += nt) {
      const int lr = t / RS, h = t % RS, i = cl_div(lr, L.inv_nx), Ln = rank + cs * i, u = lr - i * L.nx, p = Ln * L.nx + u;
      if (Ln >= L.nlines) continue;
      T r0 = sb[lr].x, r1 = sb[lr].y;
      V x0;
      x0.x = 0;
      x0.y = 0;
      if (!zero_x) {
        cl_residual<KIND, NB, true, false>(L, lr, p, u >= L.E, h, xin, sb[lr], 0u, r0, r1);
        x0 = xin[p];
      }
      update(L, lr, p, h, r0, r1, xout, true, x0, (T)P.omega);
    }
    cl.sync();
  };

  const bool gs = P.smoother == 1;
  const bool first_x = ((P.nu1 + P.nu2) & 1) != 0;   // Jacobi: which buffer the first sweep fills
  // one place for each direction's sweeps (the kernel holds them once)
  auto sweeps = [&](int l, V* cur, int n, bool forward, bool zero_start) {
#pragma unroll 1
    for (int sw = 0; sw < n; ++sw) {
      if (gs) {
        gs_sweep(l, cur, forward, zero_start && sw == 0);
      } else {
        const bool zero = zero_start && sw == 0;
        V* dst = zero ? cur : cur == xbuf(l) ? tbuf(l) : xbuf(l);
        jacobi_sweep(l, cur, dst, zero);
        cur = dst;
      }
    }
    return cur;
  };
#pragma unroll 1
  for (int l = P.first; l < P.coarsest; ++l) {
    V* cur = sweeps(l, gs || first_x ? xbuf(l) : tbuf(l), P.nu1, true, true);
    const ClLevel L = level(l);
    const LevelOp& op = P.L[l].op;
    const V* sb = bbuf(l);
    V* r = (V*)P.L[l].r;
    for (int t = tid; t < L.rows * RS; t += nt) {
      const int lr = t / RS, h = t % RS, i = cl_div(lr, L.inv_nx), Ln = rank + cs * i, u = lr - i * L.nx, p = Ln * L.nx + u;
      if (Ln >= L.nlines) continue;
      V o;
      cl_residual<KIND, NB, true, false>(L, lr, p, u >= L.E, h, cur, sb[lr], 0u, o.x, o.y);
      if (h == 0) r[p] = o;
    }
    cl.sync();
    const LevelOp& oc = P.L[l + 1].op;
    const bool last = l + 1 == P.coarsest;
    V* bc = bbuf(l + 1);
    const int nxc = oc.d.nx, n = last ? (int)oc.d.nv : P.cl_rows[l + 1];
    const float inv = 1.0f / (float)nxc;
    for (int t = last ? rank * nt + tid : tid; t < n; t += last ? cs * nt : nt) {
      // the coarsest level's b goes to everyone, another level's own rows stay
      const int q = cl_div(t, inv), Ln = last ? q : rank + cs * q, u = t - q * nxc;
      const int K = NB == 27 ? Ln / oc.d.ny : 0, J = Ln - K * oc.d.ny, I = u < oc.d.E ? 2 * u : 2 * (u - oc.d.E) + 1;
      if (NB == 27 ? K >= oc.d.nz : J >= oc.d.ny) continue;
      const V o = restrict_value<T>(op.d, oc.d, op.dmask, oc.dmask, r, Ln * nxc + u, I, J, K);
      if (last) put(everyone, bc + t, o);
      else bc[t] = o;
    }
    if (last) cl.sync();
    else __syncthreads();
  }
  {
    // x = A^-1 b on the coarsest level: one warp per row, the xor-shuffle sum of coarse_solve_body
    const T* bc = reinterpret_cast<const T*>(bbuf(P.coarsest));
    T* xc = reinterpret_cast<T*>(xbuf(P.coarsest));
    const int lane = tid & 31;
    for (int r = rank * (nt >> 5) + (tid >> 5); r < P.N; r += cs * (nt >> 5)) {
      const double* row = P.Ainv + (int64_t)r * P.N;
      double s = 0.0;
      for (int c = lane; c < P.N; c += 32) s += row[c] * (double)bc[c];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane < cs) *cl.map_shared_rank(xc + r, lane) = (T)s;
    }
    cl.sync();
  }
  // where a level's iterate lies after n sweeps
  auto after = [&](int l, int n) { return gs || first_x == ((n & 1) != 0) ? xbuf(l) : tbuf(l); };
#pragma unroll 1
  for (int l = P.coarsest - 1; l >= P.first; --l) {
    const ClLevel L = level(l);
    const LevelOp& op = P.L[l].op;
    const LevelOp& oc = P.L[l + 1].op;
    V* cur = after(l, P.nu1);
    const bool last = l + 1 == P.coarsest;
    const V* xc = last ? xbuf(l + 1) : after(l + 1, P.nu1 + P.nu2);
    const float inv_nxc = 1.0f / (float)oc.d.nx;
    for (int lr = tid; lr < L.rows; lr += nt) {
      const int i = cl_div(lr, L.inv_nx), Ln = rank + cs * i, u = lr - i * L.nx;
      if (Ln >= L.nlines) continue;
      const int k = NB == 27 ? Ln / L.ny : 0, j = Ln - k * L.ny;
      put(L.peers, cur + Ln * L.nx + u,
          prolong_value<T>(op.d, oc.d, op.dmask, oc.dmask, [&](int pc) {
            // a level's values from the CTA that owns their line (the coarsest: from the own copy)
            return last ? xc[pc] : *cl.map_shared_rank(xc + pc, cl_div(pc, inv_nxc) & (cs - 1));
          }, cur, Ln * L.nx + u, u < L.E ? 2 * u : 2 * (u - L.E) + 1, j, k));
    }
    cl.sync();
    cur = sweeps(l, cur, P.nu2, false, false);
    if (l == P.first) {
      V* xg = (V*)P.L[l].x;
      for (int lr = tid; lr < L.rows; lr += nt) {
        const int i = cl_div(lr, L.inv_nx), Ln = rank + cs * i, p = Ln * L.nx + (lr - i * L.nx);
        if (Ln < L.nlines) xg[p] = cur[p];
      }
    }
  }
}

template <int KIND, int NB>
__global__ void __launch_bounds__(TAIL_THREADS) k_vcycle_coop(const __grid_constant__ TailParams P) {
  const int64_t nthr = (int64_t)gridDim.x * blockDim.x;
  const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned gen = 0;
  if (threadIdx.x == 0) gen = *(volatile unsigned*)&P.bar[1];   // cannot move before every block has read it
  vcycle_tail_body<KIND, NB>(P, gt, nthr, [&]() { return grid_sync_bounded(P.bar, gridDim.x, gen, P.status, P.limit_ns); });
}

// `rounds` bounded grid barriers expecting `gridDim.x + extra` arrivals (a
// check of the barrier: with extra > 0 every wait gives up after limit_ns).
__global__ void __launch_bounds__(256) k_barrier_check(unsigned* bar, int rounds, int extra, double* status,
                                                      long long limit_ns, unsigned* passed) {
  unsigned gen = 0;
  if (threadIdx.x == 0) gen = *(volatile unsigned*)&bar[1];
  for (int r = 0; r < rounds; ++r) {
    if (!grid_sync_bounded(bar, gridDim.x + (unsigned)extra, gen, status, limit_ns)) return;
    if (threadIdx.x == 0) atomicAdd(passed, 1u);
  }
}

template <typename K>
static int coop_blocks(K kernel, int threads) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    return 0;
  }
  return per_sm * num_sms();
}

template <typename K, typename... A>
static cudaError_t coop_launch(K kernel, int blocks, int threads, void* s, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks, 1, 1);
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = (cudaStream_t)s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  count_launch();
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

int coop_tail_blocks(int kind, int nb) {
  if (nb == 27) {
    if (kind == STORE_F64) return coop_blocks(k_vcycle_coop<STORE_F64, 27>, TAIL_THREADS);
    if (kind == STORE_F32) return coop_blocks(k_vcycle_coop<STORE_F32, 27>, TAIL_THREADS);
    return coop_blocks(k_vcycle_coop<STORE_F16, 27>, TAIL_THREADS);
  }
  if (kind == STORE_F64) return coop_blocks(k_vcycle_coop<STORE_F64, 9>, TAIL_THREADS);
  if (kind == STORE_F32) return coop_blocks(k_vcycle_coop<STORE_F32, 9>, TAIL_THREADS);
  return coop_blocks(k_vcycle_coop<STORE_F16, 9>, TAIL_THREADS);
}

cudaError_t launch_vcycle_coop(const TailParams& P, int kind, int nb, int blocks, void* s) {
  if (nb == 27) {
    if (kind == STORE_F64) return coop_launch(k_vcycle_coop<STORE_F64, 27>, blocks, TAIL_THREADS, s, P);
    if (kind == STORE_F32) return coop_launch(k_vcycle_coop<STORE_F32, 27>, blocks, TAIL_THREADS, s, P);
    return coop_launch(k_vcycle_coop<STORE_F16, 27>, blocks, TAIL_THREADS, s, P);
  }
  if (kind == STORE_F64) return coop_launch(k_vcycle_coop<STORE_F64, 9>, blocks, TAIL_THREADS, s, P);
  if (kind == STORE_F32) return coop_launch(k_vcycle_coop<STORE_F32, 9>, blocks, TAIL_THREADS, s, P);
  return coop_launch(k_vcycle_coop<STORE_F16, 9>, blocks, TAIL_THREADS, s, P);
}

cudaError_t launch_barrier_check(unsigned* bar, int rounds, int extra, double* status, long long limit_ns,
                                 unsigned* passed, int* blocks_out, void* s) {
  const int blocks = coop_blocks(k_barrier_check, 256);
  if (blocks_out) *blocks_out = blocks;
  if (blocks < 1) return cudaErrorInvalidConfiguration;
  return coop_launch(k_barrier_check, blocks, 256, s, bar, rounds, extra, status, limit_ns, passed);
}

static uint32_t zero_start_mask(int dim, int col);

template <int KIND, int NB>
static cudaLaunchConfig_t tail_config(int csize, void* s, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(csize, 1, 1);
  cfg.blockDim = dim3(TAIL_THREADS, 1, 1);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = (cudaStream_t)s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = csize;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

template <int KIND, int NB>
static cudaError_t tail_launch(const TailParams& P, int csize, void* s) {
  cudaError_t e = cudaFuncSetAttribute(k_vcycle_tail<KIND, NB>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = tail_config<KIND, NB>(csize, s, attr);
  count_launch();
  return cudaLaunchKernelEx(&cfg, k_vcycle_tail<KIND, NB>, P);
}

template <int KIND, int NB>
static int tail_size_t() {
  cudaFuncSetAttribute(k_vcycle_tail<KIND, NB>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  const int sizes[2] = {16, 8};
  for (int q = 0; q < 2; ++q) {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = tail_config<KIND, NB>(sizes[q], nullptr, attr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_vcycle_tail<KIND, NB>, &cfg) == cudaSuccess && n >= 1) return sizes[q];
    cudaGetLastError();
  }
  return 0;
}

// largest cluster size (16, else 8) the device can co-schedule for the tail; 0: none
int tail_cluster_size(int kind, int nb) {
  if (nb == 27) return kind == STORE_F64 ? tail_size_t<STORE_F64, 27>() : kind == STORE_F32 ? tail_size_t<STORE_F32, 27>() : tail_size_t<STORE_F16, 27>();
  return kind == STORE_F64 ? tail_size_t<STORE_F64, 9>() : kind == STORE_F32 ? tail_size_t<STORE_F32, 9>() : tail_size_t<STORE_F16, 9>();
}

void fill_tail_masks(TailParams& P, int dim) {
  for (int c = 0; c < 8; ++c) P.zmask[c] = c < (1 << dim) ? zero_start_mask(dim, c) : 0u;
}

// Runs f(kernel) on the instantiation of k_vcycle_cl for a storage kind and stencil.
template <typename F>
static auto with_cl(int kind, int nb, F f) {
  if (nb == 27) return kind == STORE_F64 ? f(k_vcycle_cl<STORE_F64, 27>) : f(k_vcycle_cl<STORE_F32, 27>);
  return kind == STORE_F64 ? f(k_vcycle_cl<STORE_F64, 9>) : f(k_vcycle_cl<STORE_F32, 9>);
}

static cudaLaunchConfig_t tail_cl_config(int csize, int bytes, void* s, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(csize, 1, 1);
  cfg.blockDim = dim3(TAIL_THREADS, 1, 1);
  cfg.dynamicSmemBytes = (size_t)bytes;
  cfg.stream = (cudaStream_t)s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = csize;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_enabled() ? 2 : 1;
  return cfg;
}

// Lays out k_vcycle_cl's shared memory for a cluster of csize CTAs: every level's
// vectors first, then the matrices of as many levels as fit, the smallest first.
static bool tail_cl_layout(TailParams& P, int kind, int nb, int csize, int optin) {
  const int te = kind == STORE_F64 ? 8 : 4;
  long long at = 0;
  auto take = [&](long long bytes) {
    const long long o = at;
    at += (bytes + 15) / 16 * 16;
    return o;
  };
  for (int l = P.first; l < P.coarsest; ++l) {
    const Dims& d = P.L[l].op.d;
    const int nl = d.ny * (d.dim == 3 ? d.nz : 1);
    const long long halo = ((d.dim == 3 ? (long long)d.nx * d.ny : 0) + d.nx + d.E + 1) / 2 * 2;   // pairs, 16-byte multiple
    if (d.nv >= (1 << 20)) return false;   // (cl_div's range)
    P.cl_rows[l] = (nl + csize - 1) / csize * d.nx;
    P.cl_x[l] = (int)(take((d.nv + 2 * halo) * 2 * te) + halo * 2 * te);
    P.cl_t[l] = P.smoother == 1 ? P.cl_x[l] : (int)(take((d.nv + 2 * halo) * 2 * te) + halo * 2 * te);
    P.cl_b[l] = (int)take((long long)P.cl_rows[l] * 2 * te);
    P.cl_list[l] = (int)take((4 + 4LL * (P.cl_rows[l] / d.nx)) * sizeof(int));
    if (at > optin) return false;
  }
  P.cl_b[P.coarsest] = (int)take((long long)P.N * te);
  P.cl_x[P.coarsest] = P.cl_t[P.coarsest] = (int)take((long long)P.N * te);
  P.cl_vec_bytes = (int)at;
  for (int l = P.coarsest - 1; l >= P.first; --l) {
    const long long bytes = (long long)(nb + 1) * P.cl_rows[l] * 4 * te;
    P.cl_a[l] = at + bytes <= optin ? (int)take(bytes) : -1;
  }
  P.cl_bytes = (int)at;
  P.cl_cs = csize;
  return at <= optin;
}

// choose_cluster's view of a kernel on the current device; cfg(cs, smem, attr): its launch
template <typename Kernel, typename Cfg>
struct ClusterCalls {
  Kernel kernel;
  Cfg cfg;
  static bool ok(cudaError_t e) {
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess;
  }
  int device() {
    int dev = -1;
    return ok(cudaGetDevice(&dev)) ? dev : -1;
  }
  size_t smem_optin() {
    int v = 0;
    return ok(cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, device())) ? (size_t)v : 0;
  }
  bool allow(size_t cap) {
    return ok(cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) &&
           ok(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cap));
  }
  int clusters(int cs, size_t smem) {
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t c = cfg(cs, smem, attr);
    c.numAttrs = 1;   // the cluster's dimension
    int n = 0;
    return ok(cudaOccupancyMaxActiveClusters(&n, kernel, &c)) ? n : -1;
  }
};
template <typename Kernel, typename Cfg, typename Smem>
static int choose_cluster_of(Kernel kernel, int id, const std::vector<int>& sizes, Cfg cfg, Smem smem) {
  static ClusterAnswers known;   // (one per kernel type; id tells kernels of a type apart)
  return choose_cluster(ClusterCalls<Kernel, Cfg>{kernel, cfg}, known, id, sizes, smem);
}

// The kernel's dynamic shared-memory cap is set to the device's opt-in maximum,
// not to this plan's size: grids of different sizes share the kernel, and each
// launch passes its own size.
bool tail_cl_plan(TailParams& P, int kind, int nb) {
  int dev = 0, optin = 0;
  P.cl_bytes = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  const int cs = with_cl(kind, nb, [&](auto kernel) {
    return choose_cluster_of(
        kernel, kind * 64 + nb, {16, 8},
        [](int c, size_t smem, cudaLaunchAttribute* attr) { return tail_cl_config(c, (int)smem, nullptr, attr); },
        [&](int c) { return tail_cl_layout(P, kind, nb, c, optin) ? (size_t)P.cl_bytes : ~(size_t)0; });
  });
  if (cs == 0) P.cl_bytes = 0;   // (else the layout is that of cs, the last size asked for)
  return cs > 0;
}

cudaError_t launch_vcycle_cl(const TailParams& P, int kind, int nb, void* s) {
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = tail_cl_config(P.cl_cs, P.cl_bytes, s, attr);
  count_launch();
  return with_cl(kind, nb, [&](auto kernel) { return cudaLaunchKernelEx(&cfg, kernel, P); });
}

cudaError_t launch_vcycle_tail(const TailParams& P, int kind, int nb, int csize, void* s) {
  if (nb == 27) {
    if (kind == STORE_F64) return tail_launch<STORE_F64, 27>(P, csize, s);
    if (kind == STORE_F32) return tail_launch<STORE_F32, 27>(P, csize, s);
    return tail_launch<STORE_F16, 27>(P, csize, s);
  }
  if (kind == STORE_F64) return tail_launch<STORE_F64, 9>(P, csize, s);
  if (kind == STORE_F32) return tail_launch<STORE_F32, 9>(P, csize, s);
  return tail_launch<STORE_F16, 9>(P, csize, s);
}

// Galerkin product one axis at a time.  Trilinear P is the tensor product
// P_z P_y P_x of 1D linear interpolations and the Dirichlet masks are diagonal,
// so P_m^T A P_m = D_c P^T (D_f A D_f) P D_c is computed as three 1D
// coarsenings (x, then y, then z): the output grid halves one axis, every
// block offset along that axis becomes a coarse offset, the other offsets stay.
// With L, C, R the blocks of fine rows 2I - 1, 2I, 2I + 1 (missing rows are
// zero) at offsets -1, 0, 1 along the axis, the output blocks of row I are
//   D = -1: (L[-1] + L[0]/2 + C[-1]) / 2
//   D =  0: (L[0]/2 + L[1] + C[-1] + 2 C[0] + C[1] + R[-1] + R[0]/2) / 2
//   D = +1: (C[1] + R[0]/2 + R[1]) / 2,
// summed in this order (rows, then columns upwards).
// The fine masks D_f are applied while reading the first stage, the coarse
// masks D_c (and the identity of coarse Dirichlet rows) when writing the last.
//
// A thread makes the three blocks D of one row and one pair of other offsets:
// 9 block loads and 13 FP64 operations per entry (the set-up is FP64-pipe-bound
// on large grids).  M of the finest level is vertex-diagonal, so until the
// stages have spread it along an axis its blocks off that axis are zero and
// neither read nor written.  The stages run over windows of planes along the
// last axis, the intermediate operators of a window in a workspace that stays
// with the grid: the x stage's planes, and the y stage's planes in a ring, as
// the last plane of a window is also the first of the next (2D: the x stage's
// planes are the ring).  129^3 -> 65^3: one thread per output block over whole
// intermediate grids, its products and M's zeros unshared, took 3.63 ms (x 2.44,
// y 0.78, z 0.40) and 2 GB of temporaries; now 1.98 ms (1.02, 0.56, 0.40).
struct GalView {            // an operator, whole or a window of its planes
  const double* J;          // [block][plane slot][in-plane][4]
  const double* M;          // [block][plane slot][in-plane][2]; null: mdiag
  int64_t bs;               // vertices per block
  int f0, ring;             // plane q is slot q - f0, or q % ring where ring > 0
  __device__ __forceinline__ int64_t at(int pp, int plane, int q) const {
    return (int64_t)(ring > 0 ? (int)((uint32_t)plane % (uint32_t)ring) : plane - f0) * pp + q;
  }
};
struct GalStage {
  int nxi, nyi, nzi, nxo, nyo;   // in-plane extents before and after, planes before (2D: ny = 1, planes along y)
  int o0, o1;                    // output planes
  bool mfull;                    // the source's M is a full stencil (not the finest level's diagonal)
  const double2* mdiag;
  const uint8_t *dmf, *dmc;
  GalView in, out;
};

template <int DIM>
__device__ __forceinline__ int gal_blk(int dx, int dy, int dz) {
  return DIM == 3 ? (dx + 1) + 3 * (dy + 1) + 9 * (dz + 1) : (dx + 1) + 3 * (dz + 1);
}

__device__ __forceinline__ double2 gal_half(double2 a, double2 b) {   // a + b / 2
  return make_double2(fma(0.5, b.x, a.x), fma(0.5, b.y, a.y));
}
__device__ __forceinline__ double2 gal_add(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 gal_scale(double2 a) { return make_double2(0.5 * a.x, 0.5 * a.y); }

// AX: 0 = x, 1 = y (3D), 2 = the last axis
template <int DIM, int AX>
__global__ void __launch_bounds__(128) k_galerkin(const __grid_constant__ GalStage S) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int ppo = S.nxo * S.nyo, ppi = S.nxi * S.nyi;
  if (t >= (int64_t)(S.o1 - S.o0) * ppo) return;
  const uint32_t line = (uint32_t)t / (uint32_t)S.nxo, pl = line / (uint32_t)S.nyo;
  const int xt = (int)((uint32_t)t - line * (uint32_t)S.nxo), yo = (int)(line - pl * (uint32_t)S.nyo);
  const int zo = S.o0 + (int)pl;
  const int Eo = (S.nxo + 1) / 2, Ei = (S.nxi + 1) / 2;
  // x: threads in natural order (the fine rows they read are contiguous runs);
  // y, last: in parity-split order, unchanged by the stage
  const int xo = AX == 0 ? xt : (xt < Eo ? 2 * xt : 2 * (xt - Eo) + 1);
  const int xpo = AX == 0 ? ((xt & 1) ? Eo + (xt >> 1) : (xt >> 1)) : xt;
  // the two other offsets of this thread's blocks
  const int g0 = (int)blockIdx.y % 3 - 1, g1 = DIM == 3 ? (int)blockIdx.y / 3 - 1 : 0;
  const int dx = AX == 0 ? 0 : g0, dy = AX == 0 ? (DIM == 3 ? g0 : 0) : AX == 1 ? 0 : (DIM == 3 ? g1 : 0);
  const int dz = AX == 0 ? (DIM == 3 ? g1 : g0) : AX == 1 ? g1 : 0;
  const int c = AX == 0 ? xo : AX == 1 ? yo : zo;                  // I
  const int nin = AX == 0 ? S.nxi : AX == 1 ? S.nyi : S.nzi;
  const int bst = AX == 0 ? 1 : AX == 1 ? 3 : (DIM == 3 ? 9 : 3);  // block step along the axis
  const int b0 = gal_blk<DIM>(dx, dy, dz);                         // offset 0 along the axis
  int64_t pr[3];
  bool has[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int f = 2 * c + a - 1;
    has[a] = f >= 0 && f < nin;
    if (AX == 0) pr[a] = S.in.at(ppi, zo, yo * S.nxi + ((f & 1) ? Ei + (f >> 1) : (f >> 1)));
    else if (AX == 1) pr[a] = S.in.at(ppi, zo, f * S.nxi + xt);
    else pr[a] = has[a] ? S.in.at(ppi, f, yo * S.nxi + xt) : 0;
  }
  // first stage: row masks of the three rows, column masks of the five columns
  uint32_t mrow = 0, mcol = 0;
  if (AX == 0 && S.dmf) {
    const int yc = yo + dy, zc = zo + dz;
    const bool cin = yc >= 0 && yc < S.nyi && zc >= 0 && zc < S.nzi;
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      const int f = 2 * c + q - 2;
      if (f < 0 || f >= S.nxi) continue;
      const int xp = (f & 1) ? Ei + (f >> 1) : (f >> 1);
      if (cin && S.dmf[((int64_t)zc * S.nyi + yc) * S.nxi + xp]) mcol |= 1u << q;
      if (q >= 1 && q <= 3 && S.dmf[((int64_t)zo * S.nyi + yo) * S.nxi + xp]) mrow |= 1u << (q - 1);
    }
  }
  bool crow = false, ccol[3] = {false, false, false};
  if (AX == 2 && S.dmc) {
    const int nzo = (S.nzi - 1) / 2 + 1;
    crow = S.dmc[((int64_t)zo * S.nyo + yo) * S.nxo + xt] != 0;
    const int xc = xo + dx, yc = yo + dy;
    const bool cin = xc >= 0 && xc < S.nxo && yc >= 0 && yc < S.nyo;
    const int xp = (xc & 1) ? Eo + (xc >> 1) : (xc >> 1);
#pragma unroll
    for (int D = -1; D <= 1; ++D)
      if (cin && zo + D >= 0 && zo + D < nzo) ccol[D + 1] = S.dmc[((int64_t)(zo + D) * S.nyo + yc) * S.nxo + xp] != 0;
  }
  const int64_t po = S.out.at(ppo, zo, yo * S.nxo + xpo);
  const int h0 = gridDim.z == 2 ? (int)blockIdx.z : 0, h1 = gridDim.z == 2 ? h0 + 1 : 2;
  // M along the axes the stages have not reached yet: only the diagonal
  const bool has_m = S.mfull || (AX == 0 ? (dy == 0 && dz == 0) : AX == 1 ? dz == 0 : true);
  for (int h = h0; h < h1; ++h) {          // h = 0: the water row's entries, 1: the NAPL row's
    double2 A[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int e = 0; e < 3; ++e) {
        // row a - 1 reaches offset e - 1: L[-1], L[0], L[1], C[..], R[..]
        A[a][e] = make_double2(0.0, 0.0);
        if (has[a]) A[a][e] = reinterpret_cast<const double2*>(S.in.J)[((int64_t)(b0 + (e - 1) * bst) * S.in.bs + pr[a]) * 2 + h];
        if (AX == 0) {
          const bool mr = (mrow >> a) & 1, mc = (mcol >> (a + e)) & 1;
          if ((h == 0 && mr) || mc) A[a][e].x = 0.0;
          if (h == 0 && mr) A[a][e].y = 0.0;
        }
      }
    double2 o[3];
    o[0] = gal_scale(gal_add(gal_half(A[0][0], A[0][1]), A[1][0]));
    o[1] = gal_add(gal_half(A[0][2], A[0][1]), A[1][0]);
    o[1] = make_double2(fma(2.0, A[1][1].x, o[1].x), fma(2.0, A[1][1].y, o[1].y));
    o[1] = gal_scale(gal_half(gal_add(gal_add(o[1], A[1][2]), A[2][0]), A[2][1]));
    o[2] = gal_scale(gal_add(gal_half(A[1][2], A[2][1]), A[2][2]));
    double m[3] = {0.0, 0.0, 0.0};
    if (has_m) {
      double B[3][3];
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          B[a][e] = 0.0;
          if (!has[a] || (!S.mfull && e != 1)) continue;
          if (S.in.M) B[a][e] = S.in.M[((int64_t)(b0 + (e - 1) * bst) * S.in.bs + pr[a]) * 2 + h];
          else B[a][e] = h == 0 ? S.mdiag[pr[a]].x : S.mdiag[pr[a]].y;
          if (AX == 0 && h == 0 && ((mrow >> a) & 1)) B[a][e] = 0.0;
        }
      m[0] = 0.5 * (fma(0.5, B[0][1], B[0][0]) + B[1][0]);
      m[1] = 0.5 * fma(0.5, B[2][1], ((fma(2.0, B[1][1], fma(0.5, B[0][1], B[0][2]) + B[1][0])) + B[1][2]) + B[2][0]);
      m[2] = 0.5 * (fma(0.5, B[2][1], B[1][2]) + B[2][2]);
    }
#pragma unroll
    for (int D = 0; D < 3; ++D) {
      const int bo = b0 + (D - 1) * bst;
      if (AX == 2 && S.dmc) {
        if (h == 0 && crow) { o[D] = make_double2(0.0, 0.0); m[D] = 0.0; }
        if (ccol[D]) o[D].x = 0.0;
        if (h == 0 && crow && bo == (DIM == 3 ? 13 : 4)) o[D].x = -1.0;   // Dirichlet row: A = +identity
      }
      reinterpret_cast<double2*>(const_cast<double*>(S.out.J))[((int64_t)bo * S.out.bs + po) * 2 + h] = o[D];
      if (has_m) const_cast<double*>(S.out.M)[((int64_t)bo * S.out.bs + po) * 2 + h] = m[D];
    }
  }
}

// Doubles per plane of the x stage and of the ring, and the planes along the
// last axis that a window may hold in `bytes` (at least 4: two new fine planes,
// the kept one, and the last).
static int gal_window(const Dims& f, size_t bytes, int64_t& t1, int64_t& t2) {
  const int nxc = (f.nx - 1) / 2 + 1, nyc = (f.ny - 1) / 2 + 1;
  t1 = f.dim == 3 ? (int64_t)nxc * f.ny * f.nb * 6 : 0;
  t2 = (f.dim == 3 ? (int64_t)nxc * nyc : (int64_t)nxc) * f.nb * 6;
  const int nz = f.dim == 3 ? f.nz : f.ny;
  int64_t n = (int64_t)(bytes / sizeof(double)) / (t1 + t2);
  if (n < 4) n = 4;
  return (int)(n < nz ? n : nz);
}

size_t galerkin_workspace(const Dims& f) {
  int64_t t1, t2;
  const int planes = gal_window(f, GAL_WS_BYTES, t1, t2);
  return sizeof(double) * (size_t)(t1 + t2) * planes;
}

template <int DIM, int AX>
static void gal_launch(const GalStage& S, void* s) {
  const int64_t n = (int64_t)(S.o1 - S.o0) * S.nxo * S.nyo;
  if (n <= 0) return;
  // small windows take the two halves of a block in separate threads
  const dim3 g((unsigned)((n + 127) / 128), DIM == 3 ? 9 : 3, n <= 32768 ? 2 : 1);
  RF_LAUNCH((k_galerkin<DIM, AX>), g, 128, 0, s, S);
}

// Galerkin operators (Jc, Mc) of coarse level c from level f: J, M of level f
template <int DIM>
static void galerkin_t(const Dims& f, const uint8_t* dmf, const double* J, const double* M, const double* mdiag,
                       const Dims& c, const uint8_t* dmc, double* Jc, double* Mc, double* ws, size_t ws_bytes, void* s) {
  int64_t t1, t2;
  const int planes = gal_window(f, ws_bytes, t1, t2);
  const int nz = DIM == 3 ? f.nz : f.ny, nzc = DIM == 3 ? c.nz : c.ny;
  const int nyf = DIM == 3 ? f.ny : 1, nyc = DIM == 3 ? c.ny : 1;
  // workspace: x planes (J then M), ring planes (J then M)
  const int64_t v1 = (int64_t)c.nx * nyf, v2 = (int64_t)c.nx * nyc;   // vertices per plane
  double* w2 = ws + t1 * planes;
  GalStage S{};
  S.mfull = M != nullptr;
  S.mdiag = (const double2*)mdiag;
  S.nzi = nz;
  // windows: fine planes [f0, f1) join the ring, then coarse planes K with 2K + 1 < f1 (or at the end, all)
  int K0 = 0;
  for (int f0 = 0; f0 < nz;) {
    int f1 = f0 == 0 ? planes : f0 + planes - 1;
    if (f1 < nz && (f1 & 1)) --f1;      // an even count so far: the plane kept is 2K - 1
    if (f1 > nz) f1 = nz;
    const GalView src{J, M, f.nv, 0, 0};
    const GalView ring{w2, w2 + (int64_t)4 * f.nb * v2 * planes, v2 * planes, 0, planes};
    const GalView x1{ws, ws + (int64_t)4 * f.nb * v1 * (f1 - f0), v1 * (f1 - f0), f0, 0};
    S.nxi = f.nx; S.nyi = nyf; S.nxo = c.nx; S.nyo = nyf;
    S.o0 = f0; S.o1 = f1;
    S.dmf = dmf; S.dmc = nullptr;
    S.in = src;
    S.out = DIM == 3 ? x1 : ring;
    gal_launch<DIM, 0>(S, s);
    S.dmf = nullptr;
    if (DIM == 3) {
      S.nxi = c.nx; S.nyo = nyc;
      S.in = x1;
      S.out = ring;
      gal_launch<DIM, 1>(S, s);
    }
    S.nxi = c.nx; S.nyi = nyc; S.nxo = c.nx; S.nyo = nyc;
    S.dmc = dmc;
    S.in = ring;
    S.out = GalView{Jc, Mc, c.nv, 0, 0};
    const int K1 = f1 == nz ? nzc : f1 / 2;
    S.o0 = K0; S.o1 = K1;
    gal_launch<DIM, 2>(S, s);
    K0 = K1;
    f0 = f1;
  }
}

void launch_galerkin(const Dims& f, const uint8_t* dmf, const double* J, const double* M, const double* mdiag,
                     const Dims& c, const uint8_t* dmc, double* Jc, double* Mc, double* ws, size_t ws_bytes, void* s) {
  if (f.dim == 3) galerkin_t<3>(f, dmf, J, M, mdiag, c, dmc, Jc, Mc, ws, ws_bytes, s);
  else galerkin_t<2>(f, dmf, J, M, mdiag, c, dmc, Jc, Mc, ws, ws_bytes, s);
}

__global__ void k_coarse_mask(Dims df, const uint8_t* __restrict__ dmf, Dims dc, uint8_t* __restrict__ dmc) {
  int64_t pc = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (pc >= dc.nv) return;
  int I, J, K;
  pcoords(dc, pc, I, J, K);
  dmc[pc] = dmf[pidx(df, 2 * I, 2 * J, df.dim == 3 ? 2 * K : 0)];
}

// ----------------------------------------------------------------- packing
// Entries of A (coarse: shift*Mc - Jc for every shift; fine: J itself) in the
// storage kind, FP64 or FP32: a thread takes CH blocks of one vertex, J and M
// read once for all shifts.  Large levels take 9 (their loads in flight), small
// ones 1 (one thread per vertex walking 27 blocks took 24 us on the smallest
// levels, once per shift; now 8 us for all).
__device__ __forceinline__ void store_block(double a, double b, double c, double e, double* o) {
  reinterpret_cast<double2*>(o)[0] = make_double2(a, b);
  reinterpret_cast<double2*>(o)[1] = make_double2(c, e);
}
__device__ __forceinline__ void store_block(double a, double b, double c, double e, float* o) {
  *reinterpret_cast<float4*>(o) = make_float4((float)a, (float)b, (float)c, (float)e);
}

template <typename T, int CH>
__global__ void __launch_bounds__(256) k_pack(Dims d, bool fine, const double* __restrict__ J, const double* __restrict__ M,
                                              const __grid_constant__ PackOut out) {
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= d.nv) return;
  const int b0 = blockIdx.y * CH;
  double2 u[CH], w[CH], m[CH];
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    const double2* a = reinterpret_cast<const double2*>(J) + ((int64_t)(b0 + c) * d.nv + p) * 2;
    u[c] = __ldcs(a);
    w[c] = __ldcs(a + 1);
    if (!fine) m[c] = reinterpret_cast<const double2*>(M)[(int64_t)(b0 + c) * d.nv + p];
  }
  if (fine) {
#pragma unroll
    for (int c = 0; c < CH; ++c)
      store_block(u[c].x, u[c].y, w[c].x, w[c].y, reinterpret_cast<T*>(out.A[0]) + ((int64_t)(b0 + c) * d.nv + p) * 4);
    return;
  }
  for (int j = 0; j < out.n; ++j) {
    const double s = out.shift[j];
#pragma unroll
    for (int c = 0; c < CH; ++c)
      store_block(-u[c].x, s * m[c].x - u[c].y, -w[c].x, s * m[c].y - w[c].y,
                  reinterpret_cast<T*>(out.A[j]) + ((int64_t)(b0 + c) * d.nv + p) * 4);
  }
}

// The inverse of the 2x2 diagonal block of A = shift*M - J per shift, from its
// FP64 entries.
template <typename T>
__global__ void __launch_bounds__(256) k_pack_dinv(Dims d, bool fine, const double* __restrict__ J, const double* __restrict__ M,
                                                   const double2* __restrict__ md, const __grid_constant__ PackOut out) {
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= d.nv) return;
  const int C = d.dim == 3 ? 13 : 4;
  const double2* a = reinterpret_cast<const double2*>(J) + ((int64_t)C * d.nv + p) * 2;
  const double2 u = a[0], w = a[1];
  const double2 m = fine ? md[p] : reinterpret_cast<const double2*>(M)[(int64_t)C * d.nv + p];
  for (int j = 0; j < out.n; ++j) {
    const double a00 = -u.x, a01 = out.shift[j] * m.x - u.y, a10 = -w.x, a11 = out.shift[j] * m.y - w.y;
    // explicit, so that the inverse does not follow the compiler's choice of which product it fuses
    const double det = __fma_rn(a00, a11, -__dmul_rn(a01, a10)), r = recip(det);
    double q[4] = {a11, -a01, -a10, a00};
#pragma unroll
    for (int t = 0; t < 4; ++t) q[t] = div_by(q[t], det, r);
    store_block(q[0], q[1], q[2], q[3], reinterpret_cast<T*>(out.Dinv[j]) + p * 4);
  }
}

// The finest level in FP16: per vertex and entry position one FP32 scale (the
// largest magnitude over the block row), entries J / scale rounded to nearest,
// blocks in the paired layout of stencil_sum_f16.  The quotients are div_by's (108
// divisions per vertex took 2.9 ms at 129^3; the set-up there went from 11.6 to 6.2
// ms with this, k_galerkin and one pack for Dinv).
__global__ void __launch_bounds__(128) k_pack_f16(Dims d, const double* __restrict__ J, uint4* __restrict__ A,
                                                  float4* __restrict__ scale) {
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= d.nv) return;
  const int nb = d.nb;
  const double2* q = reinterpret_cast<const double2*>(J) + p * 2;
  const int64_t bs = d.nv * 2;
  long long mx[4] = {0, 0, 0, 0};       // bits of the largest magnitudes (as integers: off the FP64 pipe)
#pragma unroll 9
  for (int b = 0; b < nb; ++b) {
    const double2 u = q[b * bs], w = q[b * bs + 1];
    const double e[4] = {u.x, u.y, w.x, w.y};
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const long long k = __double_as_longlong(e[t]) & 0x7fffffffffffffffLL;
      if (k > mx[t] && k <= 0x7ff0000000000000LL) mx[t] = k;    // a NaN sets no scale
    }
  }
  // A position whose largest magnitude is below the smallest normal float
  // holds only entries that FP32 arithmetic flushes anyway: scale 1, entries 0.
  float sc[4];
  double r[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const double v = __longlong_as_double(mx[t]);
    sc[t] = v >= 1.17549435e-38 ? (float)v : 1.0f;
    r[t] = recip((double)sc[t]);
  }
  scale[p] = make_float4(sc[0], sc[1], sc[2], sc[3]);
  const int slots = (nb + 1) & ~1;
  for (int s2 = 0; s2 < slots; s2 += 2) {
    uint4 o;
    uint32_t hw[4];
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      const int b = nb == 27 ? f16_block_of_slot(27, s2 + hh) : f16_block_of_slot(9, s2 + hh);
      double e[4] = {0.0, 0.0, 0.0, 0.0};
      if (b >= 0) {                       // (the empty slot stays zero)
        const double2 u = q[b * bs], w = q[b * bs + 1];
        e[0] = u.x; e[1] = u.y; e[2] = w.x; e[3] = w.y;
      }
      __half v[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        v[t] = __double2half(div_by(e[t], (double)sc[t], r[t]));
      }
      hw[2 * hh] = (uint32_t)__half_as_ushort(v[0]) | (uint32_t)__half_as_ushort(v[1]) << 16;
      hw[2 * hh + 1] = (uint32_t)__half_as_ushort(v[2]) | (uint32_t)__half_as_ushort(v[3]) << 16;
    }
    o.x = hw[0]; o.y = hw[1]; o.z = hw[2]; o.w = hw[3];
    A[(int64_t)(s2 >> 1) * d.nv + p] = o;
  }
}

// dense coarsest matrix, rows/cols in parity-split unknown order 2p+alpha
__global__ void k_dense(Dims d, Nbr nb, const double* __restrict__ J, const double* __restrict__ M,
                        const double2* __restrict__ md, bool fine, double shift, double* __restrict__ D) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= d.nv * d.nb) return;
  const int b = (int)(t % d.nb);
  const int64_t p = t / d.nb;
  int i, j, k;
  pcoords(d, p, i, j, k);
  const int dx = b % 3 - 1, dy = (b / 3) % 3 - 1, dz = d.dim == 3 ? b / 9 - 1 : 0;
  const int ii = i + dx, jj = j + dy, kk = k + dz;
  if (ii < 0 || ii >= d.nx || jj < 0 || jj >= d.ny || kk < 0 || kk >= d.nz) return;
  const int64_t q = pidx(d, ii, jj, kk);
  const int64_t N = 2 * d.nv;
  const double* a = J + ((int64_t)b * d.nv + p) * 4;
  double e0 = -a[0], e1 = -a[1], e2 = -a[2], e3 = -a[3];
  const int C = d.dim == 3 ? 13 : 4;
  if (fine) {
    if (b == C) { e1 += shift * md[p].x; e3 += shift * md[p].y; }
  } else {
    const double* m = M + ((int64_t)b * d.nv + p) * 2;
    e1 += shift * m[0];
    e3 += shift * m[1];
  }
  D[(2 * p) * N + 2 * q] = e0;
  D[(2 * p) * N + 2 * q + 1] = e1;
  D[(2 * p + 1) * N + 2 * q] = e2;
  D[(2 * p + 1) * N + 2 * q + 1] = e3;
}

// LU factors with partial pivoting, one thread-block cluster per matrix: CTA r of
// the cluster keeps rows r, r + cs, ... in shared memory, and every step costs one
// cluster barrier.  Rows are not swapped; pos and at hold the order that swapping
// would give (the position of a row, the row at a position).  Step c:
//   - all take the largest of the CTAs' candidates (the earlier position on ties);
//     the first warp computes the multipliers l = A[row][c] / pivot of the CTA's
//     rows, a lane each, while the others copy the pivot row from column c on from its
//     owner through distributed shared memory;
//   - every unused row: A[row][t] -= l A[pivot][t] for t > c, and l in the place of
//     A[row][c]; one warp per row, but column c + 1 by the first warp, a lane per row,
//     before its share: the CTA's largest |A[row][c+1]| then goes to every CTA's table
//     while the other warps update the rest, and the barrier ends the step.
// The factors go to D in the order of the positions, the rows at them to piv.  A
// pivot that is zero or not finite, or a multiplier that is not finite (any NaN
// of A ends in one of these), sets status.
// Each operation is k_lu's, so are the factors, to the last bit.  (Gauss-Jordan
// elimination in the same place needs no substitution afterwards, but its sums run
// over whole columns one term after another: against a reference in 113 bits, on the
// coarsest operators of 129^3, 65^3 and 161 x 97 x 65 grids, the inverse's largest error
// was 1.1 to 5 times that of LU and substitution, whose sums are 32 lanes' partial
// sums.)
// The one-CTA k_lu does its N^3 / 3 multiply-adds on one SM's FP64 pipe (2 per
// clock) with four block barriers per column: 4.5 ms at N = 250 (5^3 vertices), 0.40
// ms at N = 50 (5^2).  Spread over a cluster: 0.51 ms and 0.085 ms, 2.0 and 1.7 us a
// step, most of it the chain of barrier, table, reciprocal and row copy (with the next
// candidates chosen after the whole update 0.68 and 0.09 ms).
constexpr int LU_THREADS = 512, LU_MAX_CS = 16;

struct LuShared {
  unsigned long long key[2][LU_MAX_CS];   // bits of |candidate| (as integers: no FP64-pipe comparisons)
  double val[2][LU_MAX_CS];
  int row[2][LU_MAX_CS];
};

__host__ __device__ inline size_t lu_smem(int N, int cs) {
  const int rows = (N + cs - 1) / cs;
  return sizeof(LuShared) + sizeof(double) * ((size_t)rows * N + N + rows) +
         sizeof(int) * (2 * (size_t)N + rows + 2);
}

__device__ __forceinline__ unsigned long long lu_key(double v) {
  const unsigned long long k = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffULL;
  return k > 0x7ff0000000000000ULL ? 0 : k;   // NaN: never a pivot
}

// Whether this lane of a warp holds the largest key, the lowest position among
// equals (positions differ)
__device__ __forceinline__ bool lu_largest(unsigned long long k, unsigned pos) {
  const unsigned hi = (unsigned)(k >> 32), lo = (unsigned)k;
  // (every lane takes part in all three reductions)
  const unsigned top = __reduce_max_sync(0xffffffffu, hi);
  const unsigned low = __reduce_max_sync(0xffffffffu, hi == top ? lo : 0u);
  const bool mine = hi == top && lo == low;
  const unsigned first = __reduce_min_sync(0xffffffffu, mine ? pos : ~0u);
  return mine && pos == first;
}

__global__ void __launch_bounds__(LU_THREADS) k_lu_cluster(int N, double* __restrict__ D, int* __restrict__ piv,
                                                           int* __restrict__ status) {
  cg::cluster_group cl = cg::this_cluster();
  const int cs = (int)cl.num_blocks(), rank = (int)cl.block_rank(), mat = blockIdx.x / cs;
  const int rows = (N + cs - 1) / cs, nloc = (N - rank + cs - 1) / cs;
  extern __shared__ __align__(16) unsigned char lu_raw[];
  LuShared& T = *reinterpret_cast<LuShared*>(lu_raw);
  double* A = reinterpret_cast<double*>(lu_raw + sizeof(LuShared));   // [rows][N]
  double* prow = A + (size_t)rows * N;
  double* mult = prow + N;                                            // [rows]
  int* pos = reinterpret_cast<int*>(mult + rows);                     // [N]
  int* at = pos + N;                                                  // [N]
  int* step = at + N;                                                 // [rows]: step a local row was pivot of, or -1
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = LU_THREADS >> 5;
  D += (int64_t)mat * N * N;
  for (int lr = warp; lr < nloc; lr += nw) {
    const double* src = D + (int64_t)(lr * cs + rank) * N;
    for (int t = lane; t < N; t += 32) {
      const double v = src[t];
      A[lr * N + t] = v;
      if (t == 0) step[lr] = -1;
    }
  }
  for (int t = tid; t < N; t += LU_THREADS) { pos[t] = t; at[t] = t; }
  cl.sync();   // every CTA of the cluster runs before a peer writes into its table
  bool bad = false, finite = true;
  // (first warp) this lane's candidate for the pivot of column c, then the warp's into
  // every CTA's table
  unsigned long long ck;
  unsigned cp;
  int crow;
  double cval;
  auto none = [&] { ck = 0; cp = N + lane; crow = 0; cval = 0.0; };   // (no candidate: key 0)
  auto consider = [&](int lr, double v) {
    const unsigned long long k = lu_key(v);
    const unsigned q = (unsigned)pos[lr * cs + rank];
    if (k > ck || (k == ck && k != 0 && q < cp)) { ck = k; cp = q; crow = lr; cval = v; }
  };
  auto publish = [&](int c) {
    const int src = __ffs(__ballot_sync(0xffffffffu, lu_largest(ck, cp))) - 1;
    const unsigned long long k = __shfl_sync(0xffffffffu, ck, src);
    const int r = __shfl_sync(0xffffffffu, crow, src);
    const double v = __shfl_sync(0xffffffffu, cval, src);
    if (lane < cs) {
      LuShared& O = *cl.map_shared_rank(&T, lane);
      O.key[c & 1][rank] = k;
      O.val[c & 1][rank] = v;
      O.row[c & 1][rank] = nloc > 0 ? r * cs + rank : 0;
    }
  };
  if (warp == 0) {
    none();
    for (int lr = lane; lr < nloc; lr += 32) consider(lr, A[lr * N]);
    publish(0);
  }
  for (int c = 0; c < N; ++c) {
    const int par = c & 1;
    cl.sync();
    const unsigned long long kq = lane < cs ? T.key[par][lane] : 0;
    const int rq = lane < cs ? T.row[par][lane] : 0;
    const unsigned pq = kq != 0 ? (unsigned)pos[rq] : (unsigned)(N + lane);
    const int best = __ffs(__ballot_sync(0xffffffffu, lu_largest(kq, pq))) - 1;
    const unsigned long long k = __shfl_sync(0xffffffffu, kq, best);
    if (k == 0 || k >= 0x7ff0000000000000ULL) { bad = true; break; }   // the same decision in every CTA
    const int pr = __shfl_sync(0xffffffffu, rq, best), p = (int)__shfl_sync(0xffffffffu, pq, best);
    const int owner = pr % cs, plr = rank == owner ? pr / cs : -1;
    if (warp == 0) {
      // (the general division leaves its fast path for a zero, of which there are many)
      const double pv = T.val[par][best], inv = recip(pv);
      for (int lr = lane; lr < nloc; lr += 32) {
        const double l = div_by(A[lr * N + c], pv, inv);
        mult[lr] = l;
        if (step[lr] < 0 && lr != plr) finite = finite && ((__double2hiint(l) & 0x7ff00000) != 0x7ff00000);
      }
    } else {
      const double* src = cl.map_shared_rank(A, owner) + (pr / cs) * N;
      for (int t = c + tid - 32; t < N; t += LU_THREADS - 32) prow[t] = src[t];
    }
    __syncthreads();
    if (warp == 0) {
      if (lane == 0) {                  // (the other warps read pos and at behind the next barrier)
        const int q = at[c];
        at[c] = pr;
        at[p] = q;
        pos[q] = p;
        pos[pr] = c;
      }
      __syncwarp();
      // column c + 1 of every row first: its candidates are on their way to the other
      // CTAs while the warps update the rest
      if (c + 1 < N) {
        none();
        for (int lr = lane; lr < nloc; lr += 32) {
          if (step[lr] >= 0 || lr == plr) continue;
          const double v = __fma_rn(-mult[lr], prow[c + 1], A[lr * N + c + 1]);
          A[lr * N + c + 1] = v;
          consider(lr, v);
        }
        __syncwarp();
        publish(c + 1);
      }
    }
    for (int lr = warp; lr < nloc; lr += nw) {
      if (lr == plr) {
        if (lane == 0) step[lr] = c;
        continue;
      }
      if (step[lr] >= 0) continue;
      double* a = A + lr * N;
      const double l = mult[lr];
      if (lane == 0) a[c] = l;
#pragma unroll 2
      for (int t = c + 2 + lane; t < N; t += 32) a[t] = __fma_rn(-l, prow[t], a[t]);
    }
  }
  cl.sync();   // no CTA leaves while its rows are read
  if (bad || !finite) status[mat] = 1;
  if (bad) return;
  for (int lr = warp; lr < nloc; lr += nw) {
    double* dst = D + (int64_t)step[lr] * N;
    for (int t = lane; t < N; t += 32) dst[t] = A[lr * N + t];
  }
  if (rank == 0)
    for (int t = tid; t < N; t += LU_THREADS) piv[(int64_t)mat * N + t] = at[t];
}

static cudaLaunchConfig_t lu_config(int nmat, int cs, size_t smem, void* s, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cs * nmat, 1, 1);
  cfg.blockDim = dim3(LU_THREADS, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = (cudaStream_t)s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

// Cluster size of k_lu_cluster for N unknowns (0: none).  A step's update takes
// N ceil(N / cs) multiply-adds of a CTA, its barrier and copies grow with cs.
// Measured for one inverse, cs = 4 / 8 / 16 (the call's 40 us of launch and
// read-back included): N = 50 166 / 166 / 169 us, N = 90 302 / 288 / 299, N = 126 437 /
// 401 / 416, N = 144 597 / 499 / 481, N = 250 1244 / 969 / 918.  A size that the
// device refuses is passed over: each gives the same factors, bit for bit.
static int lu_cluster(int N) {
  std::vector<int> sizes;
  const int first = N <= 50 ? 4 : N < 144 ? 8 : LU_MAX_CS;
  for (int cs = first; cs <= LU_MAX_CS; cs *= 2) sizes.push_back(cs);
  for (int cs = first / 2; cs >= 1; cs /= 2) sizes.push_back(cs);
  return choose_cluster_of(
      k_lu_cluster, 0, sizes,
      [](int cs, size_t smem, cudaLaunchAttribute* attr) { return lu_config(1, cs, smem, nullptr, attr); },
      [&](int cs) { return lu_smem(N, cs); });
}

static cudaError_t launch_lu_cluster(int N, int nmat, int cs, double* D, int* piv, int* status, void* s) {
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = lu_config(nmat, cs, lu_smem(N, cs), s, attr);
  count_launch();
  return cudaLaunchKernelEx(&cfg, k_lu_cluster, N, D, piv, status);
}

// LU with partial pivoting in one CTA (first maximal pivot on ties).  Per
// column: the pivot comes from candidates gathered while the previous column
// was applied; after the row swap the pivot row (from c on) and the column's
// multipliers go to shared memory, so the trailing update is a loop of
// independent loads and stores (warps over rows, lanes over columns) with no
// per-row dependency chain; the thread that updates column c+1 of a row
// records it as a candidate for the next pivot.  Four barriers per column.
// Dynamic shared memory: 2 N doubles.
__global__ void __launch_bounds__(1024) k_lu(int N, double* __restrict__ D, int* __restrict__ piv,
                                             int* __restrict__ status) {
  // one matrix per block: D, piv, status of matrix blockIdx.x
  D += (int64_t)blockIdx.x * N * N;
  piv += (int64_t)blockIdx.x * N;
  status += blockIdx.x;
  extern __shared__ double lu_sh[];
  double* prow = lu_sh;       // pivot row, columns c..N-1
  double* mult = lu_sh + N;   // multipliers of column c
  __shared__ double sval[32];
  __shared__ int sidx[32];
  __shared__ int sp;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  double best = -1.0;
  int bi = N;
  for (int r = tid; r < N; r += nt) {
    const double v = fabs(D[(int64_t)r * N]);
    if (v > best || (v == best && r < bi)) { best = v; bi = r; }
  }
  for (int c = 0; c < N; ++c) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double ov = __shfl_down_sync(0xffffffffu, best, o);
      const int oi = __shfl_down_sync(0xffffffffu, bi, o);
      if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
    }
    if (lane == 0) { sval[warp] = best; sidx[warp] = bi; }
    __syncthreads();
    if (tid == 0) {
      double bv = sval[0];
      int bidx = sidx[0];
      for (int w = 1; w < nw; ++w)
        if (sval[w] > bv || (sval[w] == bv && sidx[w] < bidx)) { bv = sval[w]; bidx = sidx[w]; }
      if (!(bv > 0.0) || !isfinite(bv)) { status[0] = 1; bidx = c; }
      sp = bidx;
      piv[c] = bidx;
    }
    __syncthreads();
    const int pr = sp;
    for (int t = tid; t < N; t += nt) {
      const double vc = D[(int64_t)c * N + t], vp = D[(int64_t)pr * N + t];
      if (pr != c) {
        D[(int64_t)c * N + t] = vp;
        D[(int64_t)pr * N + t] = vc;
      }
      if (t >= c) prow[t] = vp;
    }
    __syncthreads();
    const double dc = prow[c];
    for (int r = c + 1 + tid; r < N; r += nt) {
      const double l = (dc != 0.0) ? D[(int64_t)r * N + c] / dc : 0.0;
      // a NaN entry is never picked as pivot (fabs(NaN) > best is false) but
      // reaches the factors through its multiplier: report it
      if (!isfinite(l)) status[0] = 1;
      mult[r] = l;
      D[(int64_t)r * N + c] = l;
    }
    __syncthreads();
    best = -1.0;
    bi = N;
    for (int r = c + 1 + warp; r < N; r += nw) {
      double* Dr = D + (int64_t)r * N;
      const double l = mult[r];
      for (int t = c + 1 + lane; t < N; t += 32) {
        const double v = Dr[t] - l * prow[t];
        Dr[t] = v;
        if (t == c + 1) {
          const double av = fabs(v);
          if (av > best || (av == best && r < bi)) { best = av; bi = r; }
        }
      }
    }
    __syncthreads();
  }
}

// Columns of the inverse from the LU factors, one warp per column: x = P e_col,
// then L y = x and U z = y row by row, each row's dot product over the lanes
// with x kept in shared memory.
__global__ void __launch_bounds__(128) k_lu_inverse_cols(int N, const double* __restrict__ LU,
                                                         const int* __restrict__ piv, InvOut out) {
  // matrix blockIdx.y of the batch
  LU += (int64_t)blockIdx.y * N * N;
  piv += (int64_t)blockIdx.y * N;
  double* __restrict__ Ainv = out.Ainv[blockIdx.y];
  extern __shared__ double xs_all[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int col = blockIdx.x * (blockDim.x >> 5) + warp;
  if (col >= N) return;
  double* x = xs_all + (int64_t)warp * N;
  for (int r = lane; r < N; r += 32) x[r] = (r == col) ? 1.0 : 0.0;
  __syncwarp();
  if (lane == 0)
    for (int c = 0; c < N; ++c) {
      const int p = piv[c];
      if (p != c) { const double t = x[c]; x[c] = x[p]; x[p] = t; }
    }
  __syncwarp();
  for (int r = 1; r < N; ++r) {
    const double* Lr = LU + (int64_t)r * N;
    double s = 0.0;
    for (int c = lane; c < r; c += 32) s = __fma_rn(Lr[c], x[c], s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) x[r] -= s;
    __syncwarp();
  }
  for (int r = N - 1; r >= 0; --r) {
    const double* Ur = LU + (int64_t)r * N;
    double s = 0.0;
    for (int c = r + 1 + lane; c < N; c += 32) s = __fma_rn(Ur[c], x[c], s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) x[r] = (x[r] - s) / Ur[r];
    __syncwarp();
  }
  for (int r = lane; r < N; r += 32) Ainv[(int64_t)r * N + col] = x[r];
}

// The same, of the same operations, for the factors of k_lu_cluster (N <= ~650).  A
// row costs its chain of latencies, 2 N rows in turn with few warps in flight: the
// rows ahead are copied to shared memory (cp.async) while one is summed, and the
// division by a pivot is one Newton step on its reciprocal.  0.39 ms at N = 250 and
// 0.06 ms at N = 50, where k_lu_inverse_cols takes 0.78 and 0.11 ms.
constexpr int LU_AHEAD = 4;   // row buffers per warp

__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sa), "l"(gmem) : "memory");
}

__host__ __device__ inline size_t lu_ahead_smem(int N, int warps) {
  return sizeof(double) * ((size_t)warps * (LU_AHEAD + 1) + 2) * N;
}

__global__ void __launch_bounds__(128) k_lu_inverse_ahead(int N, const double* __restrict__ LU,
                                                          const int* __restrict__ piv, InvOut out) {
  LU += (int64_t)blockIdx.y * N * N;
  piv += (int64_t)blockIdx.y * N;
  double* __restrict__ Ainv = out.Ainv[blockIdx.y];
  extern __shared__ double la_raw[];
  double* diag = la_raw;                 // the pivots and their reciprocals
  double* rdiag = diag + N;
  for (int r = threadIdx.x; r < N; r += blockDim.x) {
    const double d = LU[(int64_t)r * N + r];
    diag[r] = d;
    rdiag[r] = recip(d);
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int col = blockIdx.x * (blockDim.x >> 5) + warp;
  if (col >= N) return;
  double* x = rdiag + N + (int64_t)warp * (LU_AHEAD + 1) * N;
  double* buf = x + N;                   // row r in buffer r % LU_AHEAD
  auto ahead = [&](int r, int c0, int c1) {   // columns [c0, c1) of row r (none: an empty group)
#pragma unroll 1
    for (int c = c0 + lane; c < c1; c += 32) cp_async8(buf + (r & (LU_AHEAD - 1)) * N + c, LU + (int64_t)r * N + c);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto dot = [&](int r, int c0, int c1) {
    asm volatile("cp.async.wait_group %0;" ::"n"(LU_AHEAD - 2) : "memory");   // row r has arrived
    __syncwarp();
    const double* row = buf + (r & (LU_AHEAD - 1)) * N;
    double s = 0.0;
#pragma unroll 1
    for (int c = c0 + lane; c < c1; c += 32) s = __fma_rn(row[c], x[c], s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
  };
  for (int r = lane; r < N; r += 32) x[r] = piv[r] == col ? 1.0 : 0.0;
#pragma unroll 1
  for (int r = 1; r < LU_AHEAD; ++r) ahead(r, 0, r < N ? r : 0);
#pragma unroll 1
  for (int r = 1; r < N; ++r) {
    const double s = dot(r, 0, r);
    if (lane == 0) x[r] -= s;
    __syncwarp();                        // (also: no lane reads this row's buffer any more)
    ahead(r + LU_AHEAD - 1, 0, r + LU_AHEAD - 1 < N ? r + LU_AHEAD - 1 : 0);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncwarp();
#pragma unroll 1
  for (int k = 0; k < LU_AHEAD - 1; ++k) ahead(N - 1 - k, N - k, N - 1 - k >= 0 ? N : N - k);
#pragma unroll 1
  for (int r = N - 1; r >= 0; --r) {
    const double s = dot(r, r + 1, N);
    if (lane == 0) x[r] = div_by(x[r] - s, diag[r], rdiag[r]);
    __syncwarp();
    ahead(r - LU_AHEAD + 1, r - LU_AHEAD + 2, r - LU_AHEAD + 1 >= 0 ? N : r - LU_AHEAD + 2);
  }
  for (int r = lane; r < N; r += 32) Ainv[(int64_t)r * N + col] = x[r];
}

// natural-order FP64 export of a level operator
__global__ void k_export(Dims d, bool fine, const double* __restrict__ J, const double* __restrict__ M,
                         const double2* __restrict__ md, double shift, double* __restrict__ out) {
  int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (v >= d.nv) return;
  const uint32_t line = (uint32_t)v / (uint32_t)d.nx;   // nv < 2^31
  const int i = (int)((uint32_t)v - line * (uint32_t)d.nx);
  const int64_t p = line * d.nx + ((i & 1) ? d.E + (i >> 1) : (i >> 1));
  const int C = d.dim == 3 ? 13 : 4;
  for (int b = 0; b < d.nb; ++b) {
    const double* a = J + ((int64_t)b * d.nv + p) * 4;
    double e[4] = {-a[0], -a[1], -a[2], -a[3]};
    if (fine) {
      if (b == C && md) { e[1] += shift * md[p].x; e[3] += shift * md[p].y; }
      if (!md) { e[0] = a[0]; e[1] = a[1]; e[2] = a[2]; e[3] = a[3]; }
    } else {
      const double* m = M + ((int64_t)b * d.nv + p) * 2;
      e[1] += shift * m[0];
      e[3] += shift * m[1];
    }
    double* o = out + (v * d.nb + b) * 4;
    o[0] = e[0]; o[1] = e[1]; o[2] = e[2]; o[3] = e[3];
  }
}

// gather the block rows and mass diagonals of listed natural vertices
__global__ void k_gather_rows(Dims d, const double* __restrict__ J, const double2* __restrict__ md,
                              const int64_t* __restrict__ verts, int count, double* __restrict__ Jout,
                              double2* __restrict__ mout) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= count * d.nb) return;
  const int r = t / d.nb, b = t % d.nb;
  const int64_t v = verts[r];
  const uint32_t line = (uint32_t)v / (uint32_t)d.nx;   // nv < 2^31
  const int i = (int)((uint32_t)v - line * (uint32_t)d.nx);
  const int64_t p = line * d.nx + ((i & 1) ? d.E + (i >> 1) : (i >> 1));
  const double* a = J + ((int64_t)b * d.nv + p) * 4;
  double* o = Jout + ((int64_t)r * d.nb + b) * 4;
  o[0] = a[0]; o[1] = a[1]; o[2] = a[2]; o[3] = a[3];
  if (b == 0) mout[r] = md[p];
}

void launch_gather_rows(const Dims& d, const double* J, const double* mdiag, const int64_t* verts, int count,
                        double* Jout, double* mout, void* s) {
  const int n = count * d.nb;
  RF_LAUNCH(k_gather_rows, (n + 127) / 128, 128, 0, s, d, J, (const double2*)mdiag, verts, count, Jout,
            (double2*)mout);
}

__global__ void k_cast_f64_f32(const double* __restrict__ in, float* __restrict__ out, int64_t n) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
    out[t] = (float)in[t];
}
__global__ void k_cast_f32_f64(const float* __restrict__ in, double* __restrict__ out, int64_t n) {
  rf_pdl_begin(in);
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
    out[t] = (double)in[t];
}

// ----------------------------------------------------------------- batched
// Several systems of one level shape per launch (see SysBatch): blockIdx.y
// selects the system, whose operator pointers replace those of L; the point
// functions are the single-system ones, so every value is computed exactly as
// there.
__device__ __forceinline__ bool sys_done(const SysLevel& P) {
  return P.scal != nullptr && P.scal[RF_SCAL_DONE] != 0.0;
}

__device__ __forceinline__ LevelOp sys_op(const LevelOp& L, const SysLevel& P) {
  LevelOp o = L;
  o.A = P.A;
  o.scale = P.scale;
  o.Dinv = P.Dinv;
  o.mdiag = P.mdiag;
  o.shift = P.shift;
  o.dmask = P.dmask;
  return o;
}

template <int KIND, bool FINE, int NB, int CH>
__global__ void __launch_bounds__(CH > 0 ? 256 : 512) k_residual_b(const __grid_constant__ LevelOp L,
                                                                   const __grid_constant__ SysBatch B) {
  typedef typename V2<typename Ty<KIND>::T>::t V;
  rf_pdl_begin();
  const SysLevel& P = B.s[blockIdx.y];
  if (sys_done(P)) return;
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= L.d.nv) return;
  residual_point<KIND, FINE, NB, CH>(sys_op(L, P), (const V*)P.in0, (const V*)P.in1, (V*)P.out, p);
}

template <int KIND, bool FINE, int NB, int CH>
__global__ void __launch_bounds__(CH > 0 ? 256 : 512) k_jacobi_b(const __grid_constant__ LevelOp L,
                                                                 const __grid_constant__ SysBatch B, double omega,
                                                                 int zero_x) {
  typedef typename V2<typename Ty<KIND>::T>::t V;
  rf_pdl_begin();
  const SysLevel& P = B.s[blockIdx.y];
  if (sys_done(P)) return;
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= L.d.nv) return;
  jacobi_point<KIND, FINE, NB, CH>(sys_op(L, P), (const V*)P.in0, (const V*)P.in1, (V*)P.out, omega, zero_x, p);
}

template <int KIND, bool FINE, int NB, int CH>
__global__ void __launch_bounds__(CH > 0 ? 256 : 512) k_gs_colour_b(const __grid_constant__ LevelOp L,
                                                                    const __grid_constant__ SysBatch B, int px,
                                                                    int py, int pz, int cnt_x, int lines_y,
                                                                    int64_t count, uint32_t skipmask, int reverse) {
  typedef typename V2<typename Ty<KIND>::T>::t V;
  rf_pdl_begin();
  const SysLevel& P = B.s[blockIdx.y];
  if (sys_done(P)) return;
  const int64_t bx = reverse ? (int64_t)(gridDim.x - 1 - blockIdx.x) : (int64_t)blockIdx.x;
  const int64_t t = bx * blockDim.x + threadIdx.x;
  if (t >= count) return;
  gs_point<KIND, FINE, NB, CH>(sys_op(L, P), (const V*)P.in0, (V*)P.out, px, py, pz, cnt_x, lines_y, t, skipmask);
}

// k_gs_pair for a batch of systems (blockIdx.y); a block of a converged
// system returns as a whole, before the barrier.
template <int KIND, bool FINE, int NB, int CH, int FPX>
__global__ void __launch_bounds__(GS_PAIR_MAX_THREADS) k_gs_pair_b(const __grid_constant__ LevelOp L,
                                                                    const __grid_constant__ SysBatch B, int py, int pz,
                                                                    int lines_y, int nlines, int lpb,
                                                                    uint32_t skip_first, uint32_t skip_second,
                                                                    int reverse) {
  typedef typename V2<typename Ty<KIND>::T>::t V;
  rf_pdl_begin();
  const SysLevel& P = B.s[blockIdx.y];
  if (sys_done(P)) return;
  const LevelOp Ls = sys_op(L, P);
  const V* b = (const V*)P.in0;
  V* x = (V*)P.out;
  const int bx = reverse ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x;
  const int l0 = bx * lpb;
  const int nl = min(lpb, nlines - l0);
  const int v = threadIdx.x;
  {
    const int cnt = FPX ? L.d.nx / 2 : (L.d.nx + 1) / 2;
    if (v < nl * cnt)
      gs_vertex<KIND, FINE, NB, CH, false>(Ls, b, x, FPX, pair_vertex(L.d, l0, v, cnt, FPX, py, pz, lines_y), skip_first);
  }
  __syncthreads();
  {
    const int cnt = FPX ? (L.d.nx + 1) / 2 : L.d.nx / 2;
    if (v < nl * cnt)
      gs_vertex<KIND, FINE, NB, CH, true>(Ls, b, x, 1 - FPX, pair_vertex(L.d, l0, v, cnt, 1 - FPX, py, pz, lines_y), skip_second);
  }
}

template <typename T>
__global__ void __launch_bounds__(256) k_restrict_planes_b(Dims df, Dims dc, const __grid_constant__ SysBatch B) {
  const SysLevel& P = B.s[blockIdx.z];
  // (the single-system kernel, with the system's masks and vectors)
  if (sys_done(P)) {
    rf_pdl_begin();
    return;
  }
  restrict_planes_body<T>(df, dc, P.dmask, P.dmask_c, (const typename V2<T>::t*)P.in0, (typename V2<T>::t*)P.out);
}

template <typename T>
__global__ void __launch_bounds__(256) k_prolong_planes_b(Dims df, Dims dc, const __grid_constant__ SysBatch B) {
  const SysLevel& P = B.s[blockIdx.z];
  if (sys_done(P)) {
    rf_pdl_begin();
    return;
  }
  prolong_pairs_body<T>(df, dc, P.dmask, P.dmask_c, (const typename V2<T>::t*)P.in0, (typename V2<T>::t*)P.out);
}

template <typename T>
__global__ void __launch_bounds__(256) k_coarse_solve_b(int N, const __grid_constant__ SysBatch B) {
  const SysLevel& P = B.s[blockIdx.y];
  if (sys_done(P)) {
    rf_pdl_begin();
    return;
  }
  coarse_solve_body<T>(N, (const double*)P.A, (const T*)P.in0, (T*)P.out);
}

__global__ void k_cast_f32_f64_b(int64_t n, const __grid_constant__ SysBatch B) {
  rf_pdl_begin();
  const SysLevel& P = B.s[blockIdx.y];
  if (sys_done(P)) return;
  const float* __restrict__ in = (const float*)P.in0;
  double* __restrict__ out = (double*)P.out;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
    out[t] = (double)in[t];
}

// Finest level of systems that share J (the LIMEX columns of one step): one
// thread per vertex loads each stencil block once and applies it to the NS
// systems' vectors, each with its own shift (and D^-1).  Per system the sums
// run block by block in the order of stencil_sum with the same expressions,
// so the values equal the single-system kernels' bit for bit.
template <int KIND, int NB, int NS, bool SAME = false>
__device__ __forceinline__ void shared_row(const LevelOp& L, const SysLevel* G, int64_t p, int par, bool skip_centre,
                                           uint32_t skipmask, const bool (&act)[NS],
                                           typename Ty<KIND>::T (&s0)[NS], typename Ty<KIND>::T (&s1)[NS]) {
  typedef typename Ty<KIND>::T T;
  typedef typename V2<T>::t V;
  constexpr int C = NB == 27 ? 13 : 4;
  float4 sc = make_float4(1.f, 1.f, 1.f, 1.f);
  if (KIND == STORE_F16) sc = reinterpret_cast<const float4*>(G[0].scale)[p];
  RowAcc<T> c0[NS], c1[NS];
  auto result = [&] {
#pragma unroll
    for (int q = 0; q < NS; ++q) {
      s0[q] = c0[q].value();
      s1[q] = c1[q].value();
    }
  };
  if constexpr (KIND == STORE_F16) {
    // pairs of slots, in the slot order of stencil_sum_f16
    const uint4* __restrict__ A = reinterpret_cast<const uint4*>(G[0].A);
#pragma unroll
    for (int qp = 0; qp < (NB + 1) / 2; ++qp) {
      bool use[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int b = f16_block_of_slot(NB, 2 * qp + h);
        use[h] = b >= 0 && !(skip_centre && b == C) && !((skipmask >> (b >= 0 ? b : 0)) & 1u);
      }
      if (!use[0] && !use[1]) continue;
      const uint4 raw = ld_stream_u4(A + (int64_t)qp * L.d.nv + p);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (!use[h]) continue;
        const int b = f16_block_of_slot(NB, 2 * qp + h);
        float a[4];
        f16_half(raw, h, sc, a);
        const int off = par ? L.nb.off[1][b] : L.nb.off[0][b];
#pragma unroll
        for (int q = 0; q < NS; ++q) {
          if (!act[q]) continue;
          const V xv = ld_xn_plain<SAME, NB>((const V*)G[q].in1 + p + off, b);
          c0[q].add(a[0], a[1], xv);
          c1[q].add(a[2], a[3], xv);
        }
      }
    }
    result();
    return;
  }
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    if (skip_centre && b == C) continue;
    if ((skipmask >> b) & 1u) continue;
    T a[4];
    load_block<KIND>(G[0].A, L.d.nv, b, p, sc, a);
    const int off = par ? L.nb.off[1][b] : L.nb.off[0][b];
#pragma unroll
    for (int q = 0; q < NS; ++q) {
      if (!act[q]) continue;
      const V xv = ld_xn_plain<SAME, NB>((const V*)G[q].in1 + p + off, b);
      c0[q].add(a[0], a[1], xv);
      c1[q].add(a[2], a[3], xv);
    }
  }
  result();
}

template <int KIND, int NB, int NS>
__global__ void __launch_bounds__(256) k_residual_shared(const __grid_constant__ LevelOp L,
                                                         const __grid_constant__ SysBatch B) {
  typedef typename Ty<KIND>::T T;
  typedef typename V2<T>::t V;
  rf_pdl_begin();
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= L.d.nv) return;
  const SysLevel* G = B.s + blockIdx.y * NS;   // this group's systems (one shared matrix)
  bool act[NS];
#pragma unroll
  for (int q = 0; q < NS; ++q) act[q] = !sys_done(G[q]);
  const int par = (int)((uint32_t)p % (uint32_t)L.d.nx) >= L.d.E;   // nv < 2^31
  T s0[NS], s1[NS];
  shared_row<KIND, NB, NS>(L, G, p, par, false, L.nomask, act, s0, s1);
  const double2 m = reinterpret_cast<const double2*>(G[0].mdiag)[p];
#pragma unroll
  for (int q = 0; q < NS; ++q) {
    if (!act[q]) continue;
    const V* x = (const V*)G[q].in1;
    const T xs = x[p].y, sh = (T)G[q].shift;
    const T a0 = (T)(sh * (T)m.x) * xs - s0[q];
    const T a1 = (T)(sh * (T)m.y) * xs - s1[q];
    const V bv = ((const V*)G[q].in0)[p];
    V o;
    o.x = bv.x - a0;
    o.y = bv.y - a1;
    ((V*)G[q].out)[p] = o;
  }
}

template <int KIND, int NB, int NS>
__global__ void __launch_bounds__(256) k_jacobi_shared(const __grid_constant__ LevelOp L,
                                                       const __grid_constant__ SysBatch B, double omega, int zero_x) {
  typedef typename Ty<KIND>::T T;
  typedef typename V2<T>::t V;
  rf_pdl_begin();
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= L.d.nv) return;
  const SysLevel* G = B.s + blockIdx.y * NS;   // this group's systems (one shared matrix)
  bool act[NS];
#pragma unroll
  for (int q = 0; q < NS; ++q) act[q] = !sys_done(G[q]);
  T s0[NS], s1[NS];
  if (!zero_x) {
    const int par = (int)((uint32_t)p % (uint32_t)L.d.nx) >= L.d.E;   // nv < 2^31
    shared_row<KIND, NB, NS>(L, G, p, par, false, L.nomask, act, s0, s1);
  }
  const double2 m = reinterpret_cast<const double2*>(G[0].mdiag)[p];
#pragma unroll
  for (int q = 0; q < NS; ++q) {
    if (!act[q]) continue;
    const V bv = ((const V*)G[q].in0)[p];
    T r0 = bv.x, r1 = bv.y, x0 = 0, x1 = 0;
    if (!zero_x) {
      const V* x = (const V*)G[q].in1;
      const T xs = x[p].y, sh = (T)G[q].shift;
      const T a0 = (T)(sh * (T)m.x) * xs - s0[q];
      const T a1 = (T)(sh * (T)m.y) * xs - s1[q];
      r0 -= a0;
      r1 -= a1;
      x0 = x[p].x;
      x1 = x[p].y;
    }
    T y0, y1;
    dinv_apply<T>(reinterpret_cast<const T*>(G[q].Dinv), p, r0, r1, y0, y1);
    V o;
    o.x = x0 + (T)omega * y0;
    o.y = x1 + (T)omega * y1;
    ((V*)G[q].out)[p] = o;
  }
}

// One vertex p (x parity px) of a GS colour for a group of systems that share
// the finest level's matrix.
template <int KIND, int NB, int NS, bool SAME = false>
__device__ __forceinline__ void gs_shared_vertex(const LevelOp& L, const SysLevel* G, int64_t p, int px,
                                                 uint32_t skipmask, const bool (&act)[NS]) {
  typedef typename Ty<KIND>::T T;
  typedef typename V2<T>::t V;
  T s0[NS], s1[NS];
  shared_row<KIND, NB, NS, SAME>(L, G, p, px, true, skipmask, act, s0, s1);
#pragma unroll
  for (int q = 0; q < NS; ++q) {
    if (!act[q]) continue;
    const V bv = ((const V*)G[q].in0)[p];
    const T r0 = bv.x + s0[q];   // fine level: A_pq = -J_pq off the diagonal
    const T r1 = bv.y + s1[q];
    T y0, y1;
    dinv_apply<T>(reinterpret_cast<const T*>(G[q].Dinv), p, r0, r1, y0, y1);
    V o;
    o.x = y0;
    o.y = y1;
    ((V*)G[q].out)[p] = o;
  }
}

template <int KIND, int NB, int NS>
__global__ void __launch_bounds__(256) k_gs_colour_shared(const __grid_constant__ LevelOp L,
                                                          const __grid_constant__ SysBatch B, int px, int py, int pz,
                                                          int cnt_x, int lines_y, int64_t count, uint32_t skipmask,
                                                          int reverse) {
  typedef typename Ty<KIND>::T T;
  typedef typename V2<T>::t V;
  rf_pdl_begin();
  const int64_t bx = reverse ? (int64_t)(gridDim.x - 1 - blockIdx.x) : (int64_t)blockIdx.x;
  const int64_t t = bx * blockDim.x + threadIdx.x;
  if (t >= count) return;
  const SysLevel* G = B.s + blockIdx.y * NS;   // this group's systems (one shared matrix)
  bool act[NS];
#pragma unroll
  for (int q = 0; q < NS; ++q) act[q] = !sys_done(G[q]);
  // 32-bit index arithmetic: a colour has fewer than 2^31 vertices
  const uint32_t tt = (uint32_t)t, line = tt / (uint32_t)cnt_x, kl = line / (uint32_t)lines_y;
  const int pos = (int)(tt - line * (uint32_t)cnt_x);
  const int jj = (int)(line - kl * (uint32_t)lines_y), kk = (int)kl;
  const int j = 2 * jj + py, k = 2 * kk + pz;
  const int64_t p = ((int64_t)j + (int64_t)L.d.ny * k) * L.d.nx + (px ? L.d.E : 0) + pos;
  gs_shared_vertex<KIND, NB, NS>(L, G, p, px, skipmask, act);
}

// k_gs_pair for groups of NS systems that share one matrix (blockIdx.y: group).
template <int KIND, int NB, int NS, int FPX>
__global__ void __launch_bounds__(GS_PAIR_MAX_THREADS) k_gs_pair_shared(const __grid_constant__ LevelOp L,
                                                                         const __grid_constant__ SysBatch B, int py,
                                                                         int pz, int lines_y, int nlines, int lpb,
                                                                         uint32_t skip_first, uint32_t skip_second,
                                                                         int reverse) {
  rf_pdl_begin();
  const SysLevel* G = B.s + blockIdx.y * NS;
  bool act[NS];
#pragma unroll
  for (int q = 0; q < NS; ++q) act[q] = !sys_done(G[q]);
  const int bx = reverse ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x;
  const int l0 = bx * lpb;
  const int nl = min(lpb, nlines - l0);
  const int v = threadIdx.x;
  {
    const int cnt = FPX ? L.d.nx / 2 : (L.d.nx + 1) / 2;
    if (v < nl * cnt)
      gs_shared_vertex<KIND, NB, NS, false>(L, G, pair_vertex(L.d, l0, v, cnt, FPX, py, pz, lines_y), FPX, skip_first, act);
  }
  __syncthreads();
  {
    const int cnt = FPX ? (L.d.nx + 1) / 2 : L.d.nx / 2;
    if (v < nl * cnt)
      gs_shared_vertex<KIND, NB, NS, true>(L, G, pair_vertex(L.d, l0, v, cnt, 1 - FPX, py, pz, lines_y), 1 - FPX,
                                           skip_second, act);
  }
}

// ----------------------------------------------------------------- launchers
// FP64 levels that are not small launch without programmatic dependence: their
// kernels are FP64-pipe-bound and few waves long, and blocks of the next launch
// that settle early on the SMs that finish first leave it unevenly spread
// (FP64 GS solves with and without: 97^3 21.3 and 16.0 ms, 129^3 32.1 and 29.5
// ms).  FP32 kernels gain from it (97^3 GS 8.5 and 8.1 ms).
static bool level_pdl(const LevelOp& L) { return L.kind != STORE_F64 || L.small; }

template <int KIND, bool FINE>
static void residual_t(const LevelOp& L, const void* b, const void* x, void* r, void* s) {
  typedef typename V2<typename Ty<KIND>::T>::t V;
  const int bs = L.block > 0 ? L.block : 256;
  const int g = (int)((L.d.nv + bs - 1) / bs);
  if (KIND == STORE_F32 && L.small) {
    const int gs = (int)((L.d.nv + 63) / 64);
    if (L.d.nb == 27) RF_LAUNCH_PDL((k_residual_small<27, FINE>), gs, 64, 0, s, L, (const float2*)b, (const float2*)x, (float2*)r);
    else RF_LAUNCH_PDL((k_residual_small<9, FINE>), gs, 64, 0, s, L, (const float2*)b, (const float2*)x, (float2*)r);
  } else if (KIND == STORE_F64 && L.small) {
    const int gs = (int)((2 * L.d.nv + 63) / 64);
    if (L.d.nb == 27) RF_LAUNCH_PDL((k_residual_small64<27, FINE>), gs, 64, 0, s, L, (const double2*)b, (const double2*)x, (double2*)r);
    else RF_LAUNCH_PDL((k_residual_small64<9, FINE>), gs, 64, 0, s, L, (const double2*)b, (const double2*)x, (double2*)r);
  } else if (L.batched) {
    if (L.d.nb == 27)
      RF_LAUNCH_PDL_IF(level_pdl(L), (k_residual<KIND, FINE, 27, chunk_of(KIND)>), g, bs, 0, s, L, (const V*)b, (const V*)x, (V*)r);
    else
      RF_LAUNCH_PDL_IF(level_pdl(L), (k_residual<KIND, FINE, 9, chunk_of(KIND)>), g, bs, 0, s, L, (const V*)b, (const V*)x, (V*)r);
  } else if (L.d.nb == 27)
    RF_LAUNCH_PDL_IF(level_pdl(L), (k_residual<KIND, FINE, 27, 0>), g, bs, 0, s, L, (const V*)b, (const V*)x, (V*)r);
  else
    RF_LAUNCH_PDL_IF(level_pdl(L), (k_residual<KIND, FINE, 9, 0>), g, bs, 0, s, L, (const V*)b, (const V*)x, (V*)r);
}

template <int KIND, bool FINE>
static void jacobi_t(const LevelOp& L, const void* b, const void* xin, void* xout, double omega, bool zero_x,
                     void* s) {
  typedef typename V2<typename Ty<KIND>::T>::t V;
  const int bs = L.block > 0 ? L.block : 256;
  const int g = (int)((L.d.nv + bs - 1) / bs);
  if (KIND == STORE_F32 && L.small && !zero_x) {
    const int gs = (int)((L.d.nv + 63) / 64);
    if (L.d.nb == 27)
      RF_LAUNCH_PDL((k_jacobi_small<27, FINE>), gs, 64, 0, s, L, (const float2*)b, (const float2*)xin, (float2*)xout, omega);
    else
      RF_LAUNCH_PDL((k_jacobi_small<9, FINE>), gs, 64, 0, s, L, (const float2*)b, (const float2*)xin, (float2*)xout, omega);
  } else if (KIND == STORE_F64 && L.small && !zero_x) {
    const int gs = (int)((2 * L.d.nv + 63) / 64);
    if (L.d.nb == 27)
      RF_LAUNCH_PDL((k_jacobi_small64<27, FINE>), gs, 64, 0, s, L, (const double2*)b, (const double2*)xin, (double2*)xout, omega);
    else
      RF_LAUNCH_PDL((k_jacobi_small64<9, FINE>), gs, 64, 0, s, L, (const double2*)b, (const double2*)xin, (double2*)xout, omega);
  } else if (L.batched) {
    if (L.d.nb == 27)
      RF_LAUNCH_PDL_IF(level_pdl(L), (k_jacobi<KIND, FINE, 27, chunk_of(KIND)>), g, bs, 0, s, L, (const V*)b, (const V*)xin, (V*)xout, omega, (int)zero_x);
    else
      RF_LAUNCH_PDL_IF(level_pdl(L), (k_jacobi<KIND, FINE, 9, chunk_of(KIND)>), g, bs, 0, s, L, (const V*)b, (const V*)xin, (V*)xout, omega, (int)zero_x);
  } else if (L.d.nb == 27)
    RF_LAUNCH_PDL_IF(level_pdl(L), (k_jacobi<KIND, FINE, 27, 0>), g, bs, 0, s, L, (const V*)b, (const V*)xin, (V*)xout, omega, (int)zero_x);
  else
    RF_LAUNCH_PDL_IF(level_pdl(L), (k_jacobi<KIND, FINE, 9, 0>), g, bs, 0, s, L, (const V*)b, (const V*)xin, (V*)xout, omega, (int)zero_x);
}

// First forward sweep from x = 0: the neighbours of colour c that have a
// higher colour are still zero, so their blocks are neither read nor applied.
static uint32_t zero_start_mask(int dim, int col) {
  uint32_t m = 0;
  const int nb = dim == 3 ? 27 : 9;
  for (int b = 0; b < nb; ++b) {
    const int dx = b % 3 - 1, dy = (b / 3) % 3 - 1, dz = dim == 3 ? b / 9 - 1 : 0;
    const int nc = ((col & 1) ^ (dx & 1)) | ((((col >> 1) & 1) ^ (dy & 1)) << 1) | ((((col >> 2) & 1) ^ (dz & 1)) << 2);
    if (nc > col) m |= 1u << b;
  }
  return m;
}

// Consecutive colour launches of a sweep walk the grid in alternating
// directions (blocks in order, then in reverse order): the vertices a launch
// starts with are the neighbours of those the previous launch ended with, whose
// x values are then still in L2.  The order within a colour changes nothing in
// the results.  `flip` starts a sweep reversed (after a launch that ended at
// the far end); RF_GS_ZIGZAG=0 keeps every launch in order.
static bool gs_zigzag() {
  const char* e = getenv("RF_GS_ZIGZAG");
  return !(e && atoi(e) == 0);
}

// The colour launches of one sweep: launch(px, py, pz, cnt_x, lines_y, count,
// skip, reverse) per colour, in sweep order.
template <typename F>
static void for_colours(const Dims& d, bool forward, bool zero_start, bool flip, F launch) {
  const int ncol = 1 << d.dim;
  const bool zigzag = gs_zigzag();
  int nl = 0;
  for (int cc = 0; cc < ncol; ++cc) {
    const int col = forward ? cc : ncol - 1 - cc;
    const uint32_t skip = (zero_start && forward) ? zero_start_mask(d.dim, col) : 0u;
    const int px = col & 1, py = (col >> 1) & 1, pz = (col >> 2) & 1;
    const int cnt_x = px ? d.nx / 2 : (d.nx + 1) / 2;
    const int lines_y = (d.ny - py + 1) / 2;
    const int lines_z = d.dim == 3 ? (d.nz - pz + 1) / 2 : 1;
    const int64_t count = (int64_t)cnt_x * lines_y * lines_z;
    if (count <= 0) continue;
    const int rev = zigzag ? ((nl + (flip ? 1 : 0)) & 1) : 0;
    ++nl;
    launch(px, py, pz, cnt_x, lines_y, count, skip, rev);
  }
}

// Colour pairs in one launch each (k_gs_pair) on FP32, FP16 and small FP64 levels;
// RF_GS_PAIRS=0 launches every colour on its own.  Both give bitwise the same
// sweep.
static bool gs_pairs() {
  const char* e = getenv("RF_GS_PAIRS");
  return !(e && atoi(e) == 0);
}

// Lines per block and threads of a pair launch: enough whole warps for the
// longer run of all the block's lines at once (a thread updates one vertex
// of each run), at most GS_PAIR_MAX_THREADS; of these shapes, the one with
// the fewest idle threads over both runs.  Lines longer than
// 2 GS_PAIR_MAX_THREADS - 1 vertices have no shape: their colours are
// launched one by one.
static bool pair_shape(int nx, int& lpb, int& threads) {
  const int e = (nx + 1) / 2, o = nx / 2;
  if (e > GS_PAIR_MAX_THREADS) return false;
  lpb = 1;
  threads = ((e + 31) / 32) * 32;
  double best = -1.0;
  for (int l = 1; l * e <= GS_PAIR_MAX_THREADS; ++l) {
    const int t = ((l * e + 31) / 32) * 32;
    const double eff = (double)l * (e + o) / (2.0 * t);
    if (eff > best + 1e-9) {
      best = eff;
      lpb = l;
      threads = t;
    }
  }
  return true;
}

// The pair launches of one sweep: launch(first_px, py, pz, lines_y, nlines,
// skip_first, skip_second, reverse) per pair, in sweep order.  Colour c =
// px + 2 py + 4 pz, so the pairs are (0,1), (2,3), ... forward and (7,6),
// (5,4), ... backward: the sweep's colour order is unchanged.
template <typename F>
static void for_colour_pairs(const Dims& d, bool forward, bool zero_start, bool flip, F launch) {
  const int ncol = 1 << d.dim;
  const bool zigzag = gs_zigzag();
  int nl = 0;
  for (int cc = 0; cc < ncol; cc += 2) {
    const int c1 = forward ? cc : ncol - 1 - cc;
    const int c2 = c1 ^ 1;
    const uint32_t s1 = (zero_start && forward) ? zero_start_mask(d.dim, c1) : 0u;
    const uint32_t s2 = (zero_start && forward) ? zero_start_mask(d.dim, c2) : 0u;
    const int py = (c1 >> 1) & 1, pz = (c1 >> 2) & 1;
    const int lines_y = (d.ny - py + 1) / 2;
    const int lines_z = d.dim == 3 ? (d.nz - pz + 1) / 2 : 1;
    const int nlines = lines_y * lines_z;
    if (nlines <= 0 || d.nx <= 0) continue;
    const int rev = zigzag ? ((nl + (flip ? 1 : 0)) & 1) : 0;
    ++nl;
    launch(c1 & 1, py, pz, lines_y, nlines, s1, s2, rev);
  }
}

template <int KIND, bool FINE>
static void gs_t(const LevelOp& L, const void* b, void* x, bool forward, bool zero_start, bool flip, void* s) {
  typedef typename V2<typename Ty<KIND>::T>::t V;
  // FP64 levels take one launch per colour unless they are small: with pairs
  // the all-FP64 257^3 solve measured 3% slower (its fine smoother 6%), as the
  // batched FP64 pair kernel needs 131 registers, one 288-thread block per SM
  int lpb = 1, threads = 32;
  if ((KIND != STORE_F64 || L.small) && gs_pairs() && pair_shape(L.d.nx, lpb, threads)) {
    if (L.small) {       // spread over the SMs
      lpb = 1;
      threads = ((L.d.nx + 1) / 2 + 31) / 32 * 32;
    }
    for_colour_pairs(L.d, forward, zero_start, flip,
                     [&](int fpx, int py, int pz, int lines_y, int nlines, uint32_t s1, uint32_t s2, int rev) {
      const int g = (nlines + lpb - 1) / lpb;
      if (KIND == STORE_F32 && L.small) {
#define RF_PAIR_SMALL(NBv, F)                                                                                      \
  RF_LAUNCH_PDL((k_gs_pair_small<NBv, FINE, F>), nlines, threads, 0, s, L, (const float2*)b, (float2*)x, py, pz, lines_y, \
                s1, s2)
        if (L.d.nb == 27) { if (fpx) RF_PAIR_SMALL(27, 1); else RF_PAIR_SMALL(27, 0); }
        else if (fpx) RF_PAIR_SMALL(9, 1);
        else RF_PAIR_SMALL(9, 0);
#undef RF_PAIR_SMALL
        return;
      }
      if (KIND == STORE_F64 && L.small) {
#define RF_PAIR_SMALL(NBv, F)                                                                                         \
  RF_LAUNCH_PDL((k_gs_pair_small64<NBv, FINE, F>), nlines, std::min(NBv == 27 ? 128 : 288, (L.d.nx + 32) / 32 * 32), 0, s, L, (const double2*)b, (double2*)x, py, pz, lines_y, \
                s1, s2)
        if (L.d.nb == 27) { if (fpx) RF_PAIR_SMALL(27, 1); else RF_PAIR_SMALL(27, 0); }
        else if (fpx) RF_PAIR_SMALL(9, 1);
        else RF_PAIR_SMALL(9, 0);
#undef RF_PAIR_SMALL
        return;
      }
#define RF_PAIR(NBv, CHv, F)                                                                                     \
  RF_LAUNCH_PDL_IF(level_pdl(L), (k_gs_pair<KIND, FINE, NBv, CHv, F>), g, threads, 0, s, L, (const V*)b, (V*)x, py, pz, lines_y, \
                nlines, lpb, s1, s2, rev)
#define RF_PAIR_PX(NBv, CHv) \
  if (fpx) RF_PAIR(NBv, CHv, 1); else RF_PAIR(NBv, CHv, 0)
      if (L.batched) {
        if (L.d.nb == 27) { RF_PAIR_PX(27, chunk_of(KIND)); } else { RF_PAIR_PX(9, chunk_of(KIND)); }
      } else if (L.d.nb == 27) {
        RF_PAIR_PX(27, 0);
      } else {
        RF_PAIR_PX(9, 0);
      }
#undef RF_PAIR_PX
#undef RF_PAIR
    });
    return;
  }
  const int bs = L.block > 0 ? L.block : 256;
  for_colours(L.d, forward, zero_start, flip,
              [&](int px, int py, int pz, int cnt_x, int lines_y, int64_t count, uint32_t skip, int rev) {
    const int g = (int)((count + bs - 1) / bs);
    if (L.batched) {
      if (L.d.nb == 27)
        RF_LAUNCH_PDL_IF(level_pdl(L), (k_gs_colour<KIND, FINE, 27, chunk_of(KIND)>), g, bs, 0, s, L, (const V*)b, (V*)x, px, py, pz, cnt_x, lines_y, count, skip, rev);
      else
        RF_LAUNCH_PDL_IF(level_pdl(L), (k_gs_colour<KIND, FINE, 9, chunk_of(KIND)>), g, bs, 0, s, L, (const V*)b, (V*)x, px, py, pz, cnt_x, lines_y, count, skip, rev);
    } else if (L.d.nb == 27) {
      RF_LAUNCH_PDL_IF(level_pdl(L), (k_gs_colour<KIND, FINE, 27, 0>), g, bs, 0, s, L, (const V*)b, (V*)x, px, py, pz, cnt_x, lines_y, count, skip, rev);
    } else {
      RF_LAUNCH_PDL_IF(level_pdl(L), (k_gs_colour<KIND, FINE, 9, 0>), g, bs, 0, s, L, (const V*)b, (V*)x, px, py, pz, cnt_x, lines_y, count, skip, rev);
    }
  });
}

bool level_shape_fixed(const LevelOp& L, bool gs) {
  int lpb = 1, threads = 32;
  return L.small && L.kind != STORE_F16 && (!gs || (gs_pairs() && pair_shape(L.d.nx, lpb, threads)));
}

void launch_residual(const LevelOp& L, const void* b, const void* x, void* r, void* s) {
  switch (L.kind) {
    case STORE_F64: L.fine ? residual_t<STORE_F64, true>(L, b, x, r, s) : residual_t<STORE_F64, false>(L, b, x, r, s); break;
    case STORE_F32: L.fine ? residual_t<STORE_F32, true>(L, b, x, r, s) : residual_t<STORE_F32, false>(L, b, x, r, s); break;
    default: L.fine ? residual_t<STORE_F16, true>(L, b, x, r, s) : residual_t<STORE_F16, false>(L, b, x, r, s); break;
  }
}

void launch_jacobi(const LevelOp& L, const void* b, const void* xin, void* xout, double omega, bool zero_x, void* s) {
  switch (L.kind) {
    case STORE_F64: L.fine ? jacobi_t<STORE_F64, true>(L, b, xin, xout, omega, zero_x, s) : jacobi_t<STORE_F64, false>(L, b, xin, xout, omega, zero_x, s); break;
    case STORE_F32: L.fine ? jacobi_t<STORE_F32, true>(L, b, xin, xout, omega, zero_x, s) : jacobi_t<STORE_F32, false>(L, b, xin, xout, omega, zero_x, s); break;
    default: L.fine ? jacobi_t<STORE_F16, true>(L, b, xin, xout, omega, zero_x, s) : jacobi_t<STORE_F16, false>(L, b, xin, xout, omega, zero_x, s); break;
  }
}

void launch_gs_sweep(const LevelOp& L, const void* b, void* x, bool forward, bool zero_start, void* s, bool flip) {
  switch (L.kind) {
    case STORE_F64: L.fine ? gs_t<STORE_F64, true>(L, b, x, forward, zero_start, flip, s) : gs_t<STORE_F64, false>(L, b, x, forward, zero_start, flip, s); break;
    case STORE_F32: L.fine ? gs_t<STORE_F32, true>(L, b, x, forward, zero_start, flip, s) : gs_t<STORE_F32, false>(L, b, x, forward, zero_start, flip, s); break;
    default: L.fine ? gs_t<STORE_F16, true>(L, b, x, forward, zero_start, flip, s) : gs_t<STORE_F16, false>(L, b, x, forward, zero_start, flip, s); break;
  }
}

// one thread per vertex of the written level: x = its planes' vertices in
// blocks of 256, y = its planes (RF_TRANSFER_POINT=1 selects the per-point
// kernels with a flat grid; read at every launch, so a graph keeps the choice
// made when it was captured)
static bool transfer_point() {
  const char* e = getenv("RF_TRANSFER_POINT");
  return e && atoi(e) == 1;
}

void launch_restrict(const LevelOp& F, const LevelOp& C, const void* rf, void* bc, void* s) {
  if (transfer_point()) {
    const int g = (int)((C.d.nv + 255) / 256);
    if (F.kind == STORE_F64)
      RF_LAUNCH_PDL(k_restrict<double>, g, 256, 0, s, F.d, C.d, F.dmask, C.dmask, (const double2*)rf, (double2*)bc);
    else
      RF_LAUNCH_PDL(k_restrict<float>, g, 256, 0, s, F.d, C.d, F.dmask, C.dmask, (const float2*)rf, (float2*)bc);
    return;
  }
  const dim3 g((unsigned)((C.d.nx * C.d.ny + 255) / 256), (unsigned)C.d.nz);
  if (F.kind == STORE_F64)
    RF_LAUNCH_PDL(k_restrict_planes<double>, g, 256, 0, s, F.d, C.d, F.dmask, C.dmask, (const double2*)rf, (double2*)bc);
  else
    RF_LAUNCH_PDL(k_restrict_planes<float>, g, 256, 0, s, F.d, C.d, F.dmask, C.dmask, (const float2*)rf, (float2*)bc);
}

void launch_prolong(const LevelOp& F, const LevelOp& C, const void* xc, void* xf, void* s) {
  if (transfer_point()) {
    const int g = (int)((F.d.nv + 255) / 256);
    if (F.kind == STORE_F64)
      RF_LAUNCH_PDL(k_prolong<double>, g, 256, 0, s, F.d, C.d, F.dmask, C.dmask, (const double2*)xc, (double2*)xf);
    else
      RF_LAUNCH_PDL(k_prolong<float>, g, 256, 0, s, F.d, C.d, F.dmask, C.dmask, (const float2*)xc, (float2*)xf);
    return;
  }
  const dim3 g((unsigned)((C.d.nx * F.d.ny + 255) / 256), (unsigned)F.d.nz);   // two fine vertices per thread
  if (F.kind == STORE_F64)
    RF_LAUNCH_PDL(k_prolong_planes<double>, g, 256, 0, s, F.d, C.d, F.dmask, C.dmask, (const double2*)xc, (double2*)xf);
  else
    RF_LAUNCH_PDL(k_prolong_planes<float>, g, 256, 0, s, F.d, C.d, F.dmask, C.dmask, (const float2*)xc, (float2*)xf);
}

void launch_coarse_solve(const LevelOp& C, const double* Ainv, const void* b, void* x, void* s) {
  const int N = (int)(2 * C.d.nv);
  const int g = (N + 7) / 8;   // 8 rows (warps) per 256-thread block
  const size_t smem = sizeof(double) * N;
  if (C.kind == STORE_F64)
    RF_LAUNCH_PDL(k_coarse_solve<double>, g, 256, smem, s, N, Ainv, (const double*)b, (double*)x);
  else
    RF_LAUNCH_PDL(k_coarse_solve<float>, g, 256, smem, s, N, Ainv, (const float*)b, (float*)x);
}


// ----------------------------------------------------------------- batched launchers
template <int KIND, bool FINE>
static void residual_bt(const LevelOp& L, const SysBatch& B, void* s) {
  const int bs = L.block > 0 ? L.block : 256;
  const dim3 g((unsigned)((L.d.nv + bs - 1) / bs), (unsigned)B.n);
  if (L.batched) {
    if (L.d.nb == 27) RF_LAUNCH_PDL_IF(level_pdl(L), (k_residual_b<KIND, FINE, 27, chunk_of(KIND)>), g, bs, 0, s, L, B);
    else RF_LAUNCH_PDL_IF(level_pdl(L), (k_residual_b<KIND, FINE, 9, chunk_of(KIND)>), g, bs, 0, s, L, B);
  } else if (L.d.nb == 27) {
    RF_LAUNCH_PDL_IF(level_pdl(L), (k_residual_b<KIND, FINE, 27, 0>), g, bs, 0, s, L, B);
  } else {
    RF_LAUNCH_PDL_IF(level_pdl(L), (k_residual_b<KIND, FINE, 9, 0>), g, bs, 0, s, L, B);
  }
}

template <int KIND, bool FINE>
static void jacobi_bt(const LevelOp& L, const SysBatch& B, double omega, bool zero_x, void* s) {
  const int bs = L.block > 0 ? L.block : 256;
  const dim3 g((unsigned)((L.d.nv + bs - 1) / bs), (unsigned)B.n);
  const int zx = zero_x ? 1 : 0;
  if (L.batched) {
    if (L.d.nb == 27) RF_LAUNCH_PDL_IF(level_pdl(L), (k_jacobi_b<KIND, FINE, 27, chunk_of(KIND)>), g, bs, 0, s, L, B, omega, zx);
    else RF_LAUNCH_PDL_IF(level_pdl(L), (k_jacobi_b<KIND, FINE, 9, chunk_of(KIND)>), g, bs, 0, s, L, B, omega, zx);
  } else if (L.d.nb == 27) {
    RF_LAUNCH_PDL_IF(level_pdl(L), (k_jacobi_b<KIND, FINE, 27, 0>), g, bs, 0, s, L, B, omega, zx);
  } else {
    RF_LAUNCH_PDL_IF(level_pdl(L), (k_jacobi_b<KIND, FINE, 9, 0>), g, bs, 0, s, L, B, omega, zx);
  }
}

template <int KIND, bool FINE>
static void gs_bt(const LevelOp& L, const SysBatch& B, bool forward, bool zero_start, bool flip, void* s) {
  int lpb = 1, threads = 32;
  if (KIND != STORE_F64 && gs_pairs() && pair_shape(L.d.nx, lpb, threads)) {   // as in gs_t
    for_colour_pairs(L.d, forward, zero_start, flip,
                     [&](int fpx, int py, int pz, int lines_y, int nlines, uint32_t s1, uint32_t s2, int rev) {
      const dim3 g((unsigned)((nlines + lpb - 1) / lpb), (unsigned)B.n);
#define RF_PAIR(NBv, CHv, F) \
  RF_LAUNCH_PDL_IF(level_pdl(L), (k_gs_pair_b<KIND, FINE, NBv, CHv, F>), g, threads, 0, s, L, B, py, pz, lines_y, nlines, lpb, s1, s2, rev)
#define RF_PAIR_PX(NBv, CHv) \
  if (fpx) RF_PAIR(NBv, CHv, 1); else RF_PAIR(NBv, CHv, 0)
      if (L.batched) {
        if (L.d.nb == 27) { RF_PAIR_PX(27, chunk_of(KIND)); } else { RF_PAIR_PX(9, chunk_of(KIND)); }
      } else if (L.d.nb == 27) {
        RF_PAIR_PX(27, 0);
      } else {
        RF_PAIR_PX(9, 0);
      }
#undef RF_PAIR_PX
#undef RF_PAIR
    });
    return;
  }
  const int bs = L.block > 0 ? L.block : 256;
  for_colours(L.d, forward, zero_start, flip,
              [&](int px, int py, int pz, int cnt_x, int lines_y, int64_t count, uint32_t skip, int rev) {
    const dim3 g((unsigned)((count + bs - 1) / bs), (unsigned)B.n);
    if (L.batched) {
      if (L.d.nb == 27)
        RF_LAUNCH_PDL_IF(level_pdl(L), (k_gs_colour_b<KIND, FINE, 27, chunk_of(KIND)>), g, bs, 0, s, L, B, px, py, pz, cnt_x, lines_y, count, skip, rev);
      else
        RF_LAUNCH_PDL_IF(level_pdl(L), (k_gs_colour_b<KIND, FINE, 9, chunk_of(KIND)>), g, bs, 0, s, L, B, px, py, pz, cnt_x, lines_y, count, skip, rev);
    } else if (L.d.nb == 27) {
      RF_LAUNCH_PDL_IF(level_pdl(L), (k_gs_colour_b<KIND, FINE, 27, 0>), g, bs, 0, s, L, B, px, py, pz, cnt_x, lines_y, count, skip, rev);
    } else {
      RF_LAUNCH_PDL_IF(level_pdl(L), (k_gs_colour_b<KIND, FINE, 9, 0>), g, bs, 0, s, L, B, px, py, pz, cnt_x, lines_y, count, skip, rev);
    }
  });
}

#define RF_KIND_FINE_SWITCH(L, CALL)                                                                  \
  switch ((L).kind) {                                                                                  \
    case STORE_F64: if ((L).fine) CALL(STORE_F64, true); else CALL(STORE_F64, false); break;         \
    case STORE_F32: if ((L).fine) CALL(STORE_F32, true); else CALL(STORE_F32, false); break;         \
    default: if ((L).fine) CALL(STORE_F16, true); else CALL(STORE_F16, false); break;                \
  }

void launch_residual_b(const LevelOp& L, const SysBatch& B, void* s) {
#define RF_CALL(K, F) residual_bt<K, F>(L, B, s)
  RF_KIND_FINE_SWITCH(L, RF_CALL)
#undef RF_CALL
}

void launch_jacobi_b(const LevelOp& L, const SysBatch& B, double omega, bool zero_x, void* s) {
#define RF_CALL(K, F) jacobi_bt<K, F>(L, B, omega, zero_x, s)
  RF_KIND_FINE_SWITCH(L, RF_CALL)
#undef RF_CALL
}

void launch_gs_sweep_b(const LevelOp& L, const SysBatch& B, bool forward, bool zero_start, void* s, bool flip) {
#define RF_CALL(K, F) gs_bt<K, F>(L, B, forward, zero_start, flip, s)
  RF_KIND_FINE_SWITCH(L, RF_CALL)
#undef RF_CALL
}

void launch_restrict_b(const LevelOp& F, const LevelOp& C, const SysBatch& B, void* s) {
  const dim3 g((unsigned)((C.d.nx * C.d.ny + 255) / 256), (unsigned)C.d.nz, (unsigned)B.n);
  if (F.kind == STORE_F64) RF_LAUNCH_PDL(k_restrict_planes_b<double>, g, 256, 0, s, F.d, C.d, B);
  else RF_LAUNCH_PDL(k_restrict_planes_b<float>, g, 256, 0, s, F.d, C.d, B);
}

void launch_prolong_b(const LevelOp& F, const LevelOp& C, const SysBatch& B, void* s) {
  const dim3 g((unsigned)((C.d.nx * F.d.ny + 255) / 256), (unsigned)F.d.nz, (unsigned)B.n);
  if (F.kind == STORE_F64) RF_LAUNCH_PDL(k_prolong_planes_b<double>, g, 256, 0, s, F.d, C.d, B);
  else RF_LAUNCH_PDL(k_prolong_planes_b<float>, g, 256, 0, s, F.d, C.d, B);
}

void launch_coarse_solve_b(const LevelOp& C, const SysBatch& B, void* s) {
  const int N = (int)(2 * C.d.nv);
  const dim3 g((unsigned)((N + 7) / 8), (unsigned)B.n);
  const size_t smem = sizeof(double) * N;
  if (C.kind == STORE_F64) RF_LAUNCH_PDL(k_coarse_solve_b<double>, g, 256, smem, s, N, B);
  else RF_LAUNCH_PDL(k_coarse_solve_b<float>, g, 256, smem, s, N, B);
}

void launch_cast_f32_to_f64_b(int64_t n, const SysBatch& B, void* s) {
  const dim3 g((unsigned)grid_for(n, 256), (unsigned)B.n);
  RF_LAUNCH_PDL(k_cast_f32_f64_b, g, 256, 0, s, n, B);
}

template <int KIND, int NS>
static void residual_sh(const LevelOp& L, const SysBatch& B, void* s) {
  const dim3 g((unsigned)((L.d.nv + 255) / 256), (unsigned)(B.n / NS));
  if (L.d.nb == 27) RF_LAUNCH_PDL((k_residual_shared<KIND, 27, NS>), g, 256, 0, s, L, B);
  else RF_LAUNCH_PDL((k_residual_shared<KIND, 9, NS>), g, 256, 0, s, L, B);
}
template <int KIND, int NS>
static void jacobi_sh(const LevelOp& L, const SysBatch& B, double omega, bool zero_x, void* s) {
  const dim3 g((unsigned)((L.d.nv + 255) / 256), (unsigned)(B.n / NS));
  if (L.d.nb == 27) RF_LAUNCH_PDL((k_jacobi_shared<KIND, 27, NS>), g, 256, 0, s, L, B, omega, zero_x ? 1 : 0);
  else RF_LAUNCH_PDL((k_jacobi_shared<KIND, 9, NS>), g, 256, 0, s, L, B, omega, zero_x ? 1 : 0);
}
template <int KIND, int NS>
static void gs_sh(const LevelOp& L, const SysBatch& B, bool forward, bool zero_start, bool flip, void* s) {
  int lpb = 1, threads = 32;
  if (KIND != STORE_F64 && gs_pairs() && pair_shape(L.d.nx, lpb, threads)) {   // as in gs_t
    for_colour_pairs(L.d, forward, zero_start, flip,
                     [&](int fpx, int py, int pz, int lines_y, int nlines, uint32_t s1, uint32_t s2, int rev) {
      const dim3 g((unsigned)((nlines + lpb - 1) / lpb), (unsigned)(B.n / NS));
#define RF_PAIR(NBv, F) \
  RF_LAUNCH_PDL((k_gs_pair_shared<KIND, NBv, NS, F>), g, threads, 0, s, L, B, py, pz, lines_y, nlines, lpb, s1, s2, rev)
      if (L.d.nb == 27) {
        if (fpx) RF_PAIR(27, 1); else RF_PAIR(27, 0);
      } else {
        if (fpx) RF_PAIR(9, 1); else RF_PAIR(9, 0);
      }
#undef RF_PAIR
    });
    return;
  }
  for_colours(L.d, forward, zero_start, flip,
              [&](int px, int py, int pz, int cnt_x, int lines_y, int64_t count, uint32_t skip, int rev) {
    const dim3 g((unsigned)((count + 255) / 256), (unsigned)(B.n / NS));
    if (L.d.nb == 27)
      RF_LAUNCH_PDL((k_gs_colour_shared<KIND, 27, NS>), g, 256, 0, s, L, B, px, py, pz, cnt_x, lines_y, count, skip, rev);
    else
      RF_LAUNCH_PDL((k_gs_colour_shared<KIND, 9, NS>), g, 256, 0, s, L, B, px, py, pz, cnt_x, lines_y, count, skip, rev);
  });
}

#define RF_KIND_NS_SWITCH(L, NSV, CALL)                                                                    \
  switch ((L).kind * 4 + (NSV) - 1) {                                                                      \
    case 0: CALL(STORE_F64, 1); break; case 1: CALL(STORE_F64, 2); break;                                  \
    case 2: CALL(STORE_F64, 3); break; case 3: CALL(STORE_F64, 4); break;                                  \
    case 4: CALL(STORE_F32, 1); break; case 5: CALL(STORE_F32, 2); break;                                  \
    case 6: CALL(STORE_F32, 3); break; case 7: CALL(STORE_F32, 4); break;                                  \
    case 8: CALL(STORE_F16, 1); break; case 9: CALL(STORE_F16, 2); break;                                  \
    case 10: CALL(STORE_F16, 3); break; default: CALL(STORE_F16, 4); break;                                \
  }

void launch_residual_shared(const LevelOp& L, const SysBatch& B, int share, void* s) {
#define RF_CALL(K, N) residual_sh<K, N>(L, B, s)
  RF_KIND_NS_SWITCH(L, share, RF_CALL)
#undef RF_CALL
}
void launch_jacobi_shared(const LevelOp& L, const SysBatch& B, int share, double omega, bool zero_x, void* s) {
#define RF_CALL(K, N) jacobi_sh<K, N>(L, B, omega, zero_x, s)
  RF_KIND_NS_SWITCH(L, share, RF_CALL)
#undef RF_CALL
}
void launch_gs_sweep_shared(const LevelOp& L, const SysBatch& B, int share, bool forward, bool zero_start, void* s,
                            bool flip) {
#define RF_CALL(K, N) gs_sh<K, N>(L, B, forward, zero_start, flip, s)
  RF_KIND_NS_SWITCH(L, share, RF_CALL)
#undef RF_CALL
}

void launch_coarse_mask(const Dims& df, const uint8_t* dmf, const Dims& dc, uint8_t* dmc, void* s) {
  RF_LAUNCH(k_coarse_mask, (int)((dc.nv + 255) / 256), 256, 0, s, df, dmf, dc, dmc);
}

void launch_pack_level(const Dims& d, bool fine, const double* J, const double* M, const double* mdiag, int kind,
                       PackOut out, float* scale, void* s) {
  const unsigned g = (unsigned)((d.nv + 255) / 256);
  const bool wide = d.nv >= 65536;
  const dim3 gb(g, wide ? d.nb / 9 : d.nb);
  if (!out.diag_only) {
    if (kind == STORE_F16) RF_LAUNCH(k_pack_f16, (unsigned)((d.nv + 127) / 128), 128, 0, s, d, J, (uint4*)out.A[0], (float4*)scale);
    else if (kind == STORE_F64 && wide) RF_LAUNCH((k_pack<double, 9>), gb, 256, 0, s, d, fine, J, M, out);
    else if (kind == STORE_F64) RF_LAUNCH((k_pack<double, 1>), gb, 256, 0, s, d, fine, J, M, out);
    else if (wide) RF_LAUNCH((k_pack<float, 9>), gb, 256, 0, s, d, fine, J, M, out);
    else RF_LAUNCH((k_pack<float, 1>), gb, 256, 0, s, d, fine, J, M, out);
  }
  if (kind == STORE_F64) RF_LAUNCH(k_pack_dinv<double>, g, 256, 0, s, d, fine, J, M, (const double2*)mdiag, out);
  else RF_LAUNCH(k_pack_dinv<float>, g, 256, 0, s, d, fine, J, M, (const double2*)mdiag, out);
}

void launch_dense_coarsest(const Dims& d, const Nbr& nb, const double* Jc, const double* Mc,
                           const double* mdiag, bool fine, double shift, double* D, void* s) {
  const int64_t n = d.nv * d.nb;
  RF_LAUNCH(k_dense, (int)((n + 127) / 128), 128, 0, s, d, nb, Jc, Mc, (const double2*)mdiag, fine, shift, D);
}

cudaError_t launch_dense_inverse_batched(int N, int nmat, double* D, double* const* Ainv, int* piv, int* status,
                                         void* s) {
  if (nmat < 1 || nmat > RF_MAXSHIFT) return cudaErrorInvalidValue;
  InvOut out;
  for (int j = 0; j < RF_MAXSHIFT; ++j) out.Ainv[j] = j < nmat ? Ainv[j] : nullptr;
  // k_lu in global memory serves N beyond a cluster's shared memory (N > ~650),
  // devices that run no such cluster, and comparisons (RF_LU_CLUSTER=0, read per call)
  const char* env = getenv("RF_LU_CLUSTER");
  const int cs = env && atoi(env) == 0 ? 0 : lu_cluster(N);
  if (cs > 0) {
    const cudaError_t e = launch_lu_cluster(N, nmat, cs, D, piv, status, s);
    if (e != cudaSuccess) return e;
  } else {
    const size_t lsm = sizeof(double) * 2 * (size_t)N;   // 64 KB at N = 4096
    cudaFuncSetAttribute(k_lu, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lsm);
    RF_LAUNCH(k_lu, nmat, 1024, lsm, s, N, D, piv, status);
  }
  const dim3 grid((N + 3) / 4, nmat);
  if (cs > 0) {
    const size_t bytes = lu_ahead_smem(N, 4);            // 114 KB at N = 650
    if (bytes > 48 * 1024)
      cudaFuncSetAttribute(k_lu_inverse_ahead, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    RF_LAUNCH(k_lu_inverse_ahead, grid, 128, bytes, s, N, D, piv, out);
    return cudaGetLastError();
  }
  const size_t smem = sizeof(double) * 4 * (size_t)N;   // 4 warps per block, one x each (128 KB at N = 4096)
  cudaFuncSetAttribute(k_lu_inverse_cols, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  RF_LAUNCH(k_lu_inverse_cols, grid, 128, smem, s, N, D, piv, out);
  return cudaGetLastError();
}

cudaError_t launch_dense_inverse(int N, double* D, double* Ainv, int* piv, double* work, int* status, void* s) {
  (void)work;
  return launch_dense_inverse_batched(N, 1, D, &Ainv, piv, status, s);
}

void launch_export_level(const Dims& d, bool fine, const double* J, const double* M, const double* mdiag,
                         double shift, double* A_nat, void* s) {
  RF_LAUNCH(k_export, (int)((d.nv + 127) / 128), 128, 0, s, d, fine, J, M, (const double2*)mdiag, shift, A_nat);
}

void launch_cast_f64_to_f32(const double* in, float* out, int64_t n, void* s) {
  RF_LAUNCH(k_cast_f64_f32, grid_for(n, 256), 256, 0, s, in, out, n);
}
void launch_cast_f32_to_f64(const float* in, double* out, int64_t n, void* s) {
  RF_LAUNCH_PDL(k_cast_f32_f64, grid_for(n, 256), 256, 0, s, in, out, n);
}

}  // namespace rf
