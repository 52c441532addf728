// AxLocal, fiber-per-thread design (templates over an arithmetic policy:
// native FP64, native FP32, or double-word FP32 pairs).
//
// The whole element (EPB elements per CTA) sits in padded shared memory.
// Every contraction of Algorithm 1 is done by a thread that owns a whole
// fiber of the tensor in the contraction's direction, so the differentiation
// matrix is read as a uniform constant-memory operand by all threads at once
// (the constant-memory idea of Sec. 4.3.1, applied to all three directions),
// and each fiber product uses the even-odd split of the centro-antisymmetric
// D (D[N-i][N-j] = -D[i][j]): outputs i and N-i come from two half-length
// dot products of the fiber's even and odd parts, nearly halving the
// multiply-adds.
//
//   r-fibers  x0 = D_r x -> B0;   s-fibers  x1 = D_s x -> B1
//   thread (i,j): t-fiber x2 = D_t x[i,j,:]; per node k the geometry
//           (stored / Algorithm 2 / Algorithm 3 / partial) and
//           (r,s,t) = G (x0,x1,x2); r -> B0, s -> B1; Y = D_t^T t
//   r-fibers  Y += D_r^T r;   s-fibers  Y += D_s^T s;   Y to HBM.
// Five barriers per element (two per k-layer in the layer-wise design).
// Phase 3 (own t-fiber) needs no barrier after the geometry: each thread
// reads and writes only its own fiber there.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "ax_internal.h"
#include "dw.cuh"
#include "dw2.cuh"
#include "reduce.cuh"
#include "tables.cuh"

namespace ax {
namespace fiber {

// 1-ulp reciprocal of a normal float whose reciprocal is normal too: the
// determinants of elements inside the extents that setup accepts (a general
// fast division also tests for divisors above 2^126, three more instructions)
__device__ __forceinline__ float rcp32(float b) {
  float v;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(v) : "f"(b));
  return v;
}

// ---------------------------------------------------------------------------
// arithmetic policies
// ---------------------------------------------------------------------------
template <typename T>
struct Native {
  using V = T;   // register value
  using S = T;   // shared-memory / geometry-record word
  using A = T;   // dot-product accumulator
  using C = T;   // constant-table word
  using IO = T;  // X, Y in HBM
  static constexpr bool kRoll = false;  // short code: unroll the phase and k loops
  static constexpr bool kScaleIO = false;  // native range: X and Y pass unscaled
  static constexpr int kTargetWarpsPerSM = 0;  // no cap
  static constexpr int kTiles = sizeof(T) == 4 ? 2 : 1;  // tile variants the autotuner may pick
  __device__ static __forceinline__ V ld(const S *p) { return *p; }
  __device__ static __forceinline__ S st(V v) { return v; }
  __device__ static __forceinline__ V cst(const C *p) { return *p; }
  __device__ static __forceinline__ V from_io(IO v) { return v; }
  __device__ static __forceinline__ V from_io_direct(IO v) { return v; }
  __device__ static __forceinline__ IO to_io(V v) { return v; }
  __device__ static __forceinline__ V lit(double v) { return (T)v; }
  __device__ static __forceinline__ A zero() { return T(0); }
  __device__ static __forceinline__ A mul0(V x, V y) { return x * y; }
  __device__ static __forceinline__ void mac(A &a, V x, V y) { a = fma(x, y, a); }
  __device__ static __forceinline__ V fin(A a) { return a; }
  __device__ static __forceinline__ V acc_sum(A a, A b) { return a + b; }
  __device__ static __forceinline__ V acc_dif(A a, A b) { return a - b; }
  __device__ static __forceinline__ V add(V a, V b) { return a + b; }
  __device__ static __forceinline__ V sub(V a, V b) { return a - b; }
  __device__ static __forceinline__ V add_lazy(V a, V b) { return a + b; }
  __device__ static __forceinline__ V sub_lazy(V a, V b) { return a - b; }
  __device__ static __forceinline__ V mul(V a, V b) { return a * b; }
  __device__ static __forceinline__ V fma3(V a, V b, V c) { return fma(a, b, c); }
  __device__ static __forceinline__ V twice(V a) { return a + a; }
  __device__ static __forceinline__ IO sum3_io(V a, V b, V c) { return (a + b) + c; }
  __device__ static __forceinline__ IO sum3_io_direct(V a, V b, V c) { return (a + b) + c; }
  __device__ static __forceinline__ V div(V a, V b) {
    if constexpr (sizeof(T) == 4)
      return a * rcp32(b);  // 2-ulp quotient: the FP32 path's tolerance is 2e-5
    else
      return a / b;
  }
  __device__ static __forceinline__ V neg(V a) { return -a; }
};

struct DW {
  using V = dw::dw;
  using S = float2;
  using A = dw::acc;
  using C = float2;
  using IO = double;
  static constexpr bool kRoll = true;  // long code: keep the phase and k loops rolled (instruction cache)
  // float64 X has float64's exponent range, the float pairs only float32's:
  // each element's X is scaled by a power of two that brings its largest
  // magnitude near 1 before the conversion, and Y is scaled back (both exact)
  static constexpr bool kScaleIO = true;
  static constexpr int kTiles = 1;
  // Resident warps per SM the launcher aims at for the trilinear kinds at
  // N1 = 8 (by padding the dynamic shared memory): more warps thrash the
  // instruction cache with this long code.  Measured on GB300: 5 CTAs of 4
  // warps 2% faster than 4, and fewer (3) or longer code per warp (unrolled
  // k or phase loops) slower; at other orders and for the stored kind a cap
  // measured slower, so it is not applied there.
  static constexpr int kTargetWarpsPerSM = 20;
  __device__ static __forceinline__ V ld(const S *p) { return dw::from_float2(*p); }
  __device__ static __forceinline__ S st(V v) { return make_float2(v.hi, v.lo); }
  __device__ static __forceinline__ V cst(const C *p) { return dw::from_float2(*p); }
  __device__ static __forceinline__ V from_io(IO v) { return dw::from_double(v); }
  // inside the direct range (the main kernel): no FP64-pipe instruction
  __device__ static __forceinline__ V from_io_direct(IO v) { return dw::from_double_direct(v); }
  __device__ static __forceinline__ IO to_io(V v) { return dw::to_double(v); }
  __device__ static __forceinline__ V lit(double v) { return dw::make((float)v, 0.0f); }  // exact small literals only
  __device__ static __forceinline__ A zero() { return dw::acc_zero(); }
  __device__ static __forceinline__ A mul0(V x, V y) { return dw::mul_acc(x, y); }
  __device__ static __forceinline__ void mac(A &a, V x, V y) { dw::mac(a, x, y); }
  __device__ static __forceinline__ V fin(A a) { return dw::fin(a); }
  // sums that feed only error-tolerant consumers skip the final Fast2Sum (dw.cuh)
  __device__ static __forceinline__ V acc_sum(A a, A b) { return dw::acc_sum(a, b); }
  __device__ static __forceinline__ V acc_dif(A a, A b) { return dw::acc_dif(a, b); }
  __device__ static __forceinline__ V add(V a, V b) { return dw::add(a, b); }
  __device__ static __forceinline__ V sub(V a, V b) { return dw::sub(a, b); }
  __device__ static __forceinline__ V add_lazy(V a, V b) { return dw::add_lazy(a, b); }
  __device__ static __forceinline__ V sub_lazy(V a, V b) { return dw::sub_lazy(a, b); }
  __device__ static __forceinline__ V mul(V a, V b) { return dw::mul(a, b); }
  __device__ static __forceinline__ V fma3(V a, V b, V c) { return dw::fma(a, b, c); }
  __device__ static __forceinline__ V twice(V a) { return dw::make(2.0f * a.hi, 2.0f * a.lo); }  // exact
  __device__ static __forceinline__ IO sum3_io(V a, V b, V c) { return dw::sum3_to_double(a, b, c); }
  __device__ static __forceinline__ IO sum3_io_direct(V a, V b, V c) { return dw::sum3_to_double_direct(a, b, c); }
  __device__ static __forceinline__ V div(V a, V b) { return dw::div(a, b); }
  __device__ static __forceinline__ V neg(V a) { return dw::neg(a); }
};


template <class P>
__device__ __forceinline__ typename P::V dot3(const typename P::V a[3], const typename P::V b[3]) {
  typename P::A s = P::mul0(a[0], b[0]);
  P::mac(s, a[1], b[1]);
  P::mac(s, a[2], b[2]);
  return P::fin(s);
}

// a*b - c*d
template <class P>
__device__ __forceinline__ typename P::V det2(typename P::V a, typename P::V b, typename P::V c, typename P::V d) {
  typename P::A s = P::mul0(a, b);
  P::mac(s, P::neg(c), d);
  return P::fin(s);
}

// ---------------------------------------------------------------------------
// even-odd fiber product: out = M in, M centro-antisymmetric (D or D^T).
// Table block of order N1 (N1*N1 words), c = N1/2:
//   rows i < c: [ A(i,0..c-1) | B(i,0..c-1) | M[i][c] if N1 odd ],
//     A = (M[i][m] + M[i][N-m]) / 2,  B = (M[i][m] - M[i][N-m]) / 2
//   row c (N1 odd): M[c][0..c-1]
// out[i] = P + Q, out[N-i] = Q - P with P = sum A e + M[i][c] f[c], Q = sum B o,
// e[m] = f[m] + f[N-m], o[m] = f[m] - f[N-m].
// ---------------------------------------------------------------------------
template <class P, int N1>
__device__ __forceinline__ void contract(const typename P::C *__restrict__ eo, const typename P::V *in,
                                         typename P::V *out) {
  using V = typename P::V;
  constexpr int c = N1 / 2;
  constexpr bool odd = (N1 & 1) != 0;
  V e[c], o[c];
#pragma unroll
  for (int m = 0; m < c; ++m) {
    e[m] = P::add_lazy(in[m], in[N1 - 1 - m]);
    o[m] = P::sub_lazy(in[m], in[N1 - 1 - m]);
  }
#pragma unroll
  for (int i = 0; i < c; ++i) {
    typename P::A p = P::mul0(P::cst(eo + i * N1), e[0]), q = P::mul0(P::cst(eo + i * N1 + c), o[0]);
#pragma unroll
    for (int m = 1; m < c; ++m) {
      P::mac(p, P::cst(eo + i * N1 + m), e[m]);
      P::mac(q, P::cst(eo + i * N1 + c + m), o[m]);
    }
    if constexpr (odd) P::mac(p, P::cst(eo + i * N1 + 2 * c), in[c]);
    if constexpr (N1 < 16) {
      out[i] = P::acc_sum(p, q);
      out[N1 - 1 - i] = P::acc_dif(q, p);
    } else {
      // N1 = 16: under the 128-register cap the sums straight from the
      // accumulators spill in double-word arithmetic; finalise them first
      const V Pv = P::fin(p), Qv = P::fin(q);
      out[i] = P::add(Pv, Qv);
      out[N1 - 1 - i] = P::sub(Qv, Pv);
    }
  }
  if constexpr (odd) {
    typename P::A q = P::mul0(P::cst(eo + c * N1), o[0]);
#pragma unroll
    for (int m = 1; m < c; ++m) P::mac(q, P::cst(eo + c * N1 + m), o[m]);
    out[c] = P::fin(q);
  }
}

// The double-word fiber product at even orders runs its two dot products per
// output pair in the lanes of packed FP32x2 instructions (dw2.cuh; the same
// roundings in the same order: bit-identical results, about half the issue
// slots for the products); eo2: the order's paired table.
template <class P, int N1>
constexpr bool kPairedDW = P::kRoll && (N1 % 2) == 0;
// FP32 likewise (the same products per lane, bit-identical).  Measured on
// GB300 against the scalar product: N = 7 trilinear 238 -> 255 GDOF/s,
// parallelepiped 314 -> 324, stored 180 -> 188, N = 3, 9 trilinear +5%,
// N = 15 trilinear 172 -> 178 (with the two-CTA register bound of
// shape_min_ctas; unbounded the kernel takes 161 registers and one CTA per
// SM: 131); the partial kind at N1 = 8 measured 6% slower and keeps the
// scalar product.
template <class P, int N1, int KIND>
constexpr bool kPairedF32 = !P::kRoll && sizeof(typename P::V) == 4 && (N1 % 2) == 0 &&
                            !(N1 == 8 && KIND == AX_GEOM_TRILINEAR_PARTIAL);
template <class P, int N1, int KIND>
__device__ __forceinline__ void contract_p(const typename P::C *__restrict__ eo, const float4 *__restrict__ eo2,
                                           const typename P::V *in, typename P::V *out) {
  if constexpr (kPairedDW<P, N1>)
    dw2::contract<N1>(eo2, in, out);
  else if constexpr (kPairedF32<P, N1, KIND>)
    dw2::contract_f32<N1>(eo2, in, out);
  else
    contract<P, N1>(eo, in, out);
}

// Elements per CTA for F threads per element: at least 128 threads, and
// among up to about four times that many elements (at most 512 threads) the
// count that leaves the fewest idle lanes in the last warp (N1 = 6: 7
// elements = 252 threads instead of 3 = 108 threads in four warps).
__host__ __device__ constexpr int idle_lanes_permille(int t) { return ((t + 31) / 32 * 32 - t) * 1000 / ((t + 31) / 32 * 32); }
__host__ __device__ constexpr int pick_epb(int F) {
  int base = F >= 128 ? 1 : 128 / F, best = base, bw = idle_lanes_permille(F * base);
  for (int e = base + 1; e <= 4 * base + 3 && F * e <= 512; ++e)
    if (idle_lanes_permille(F * e) < bw) {
      best = e;
      bw = idle_lanes_permille(F * e);
    }
  return best;
}

// Measured exceptions to the shape rules below, per policy (0: double-word,
// 1: FP32), order and kind: elements per CTA and the minimum resident CTAs
// that bound the registers (0: no override).
// Double-word recompute kernels at N1 = 6 and 10, whose register counts
// (96-127) let an SM hold only one or two filled CTAs (16-18 warps, stalled
// at their barriers), measured on GB300 against the filled shapes, with the
// register bounds' few spills included: N = 5 trilinear 7 elements, 3 CTAs
// (24.0 -> 32.1 GDOF/s), partial 6, 4 (27.1 -> 32.9); N = 9 trilinear 1, 5
// (21.9 -> 24.1), partial 3, 2 (21.8 -> 26.2).  Their stored and
// parallelepiped kinds (56-96 registers) and N1 = 12 measured no faster in
// any of the shapes tried.  With the packed fiber product (dw2.cuh) the
// trilinear kernel at N1 = 8 takes 127 registers unbounded (four CTAs per
// SM); bounded to five CTAs (96 registers, no spills) it runs 2.4% faster.
// FP32 (40-64 registers, mostly faster as they are): N = 5 partial 4
// elements (153 -> 163), N = 9 parallelepiped 2 (243 -> 251), N = 11 stored
// 1 element, 4 CTAs (156 -> 172); N = 7 trilinear eight CTAs (64 registers
// instead of 68: 298 -> 304); N1 = 16 two CTAs (the packed fiber
// product, kPairedF32, would otherwise take 161 registers).
__host__ __device__ constexpr int shape_epb(int pc, int N1, int KIND) {
  return pc == 0 ? (N1 == 6    ? (KIND == AX_GEOM_TRILINEAR ? 7 : KIND == AX_GEOM_TRILINEAR_PARTIAL ? 6 : 0)
                    : N1 == 10 ? (KIND == AX_GEOM_TRILINEAR ? 1 : KIND == AX_GEOM_TRILINEAR_PARTIAL ? 3 : 0)
                               : 0)
                 : (N1 == 6 && KIND == AX_GEOM_TRILINEAR_PARTIAL) ? 4
                 : (N1 == 10 && KIND == AX_GEOM_PARALLELEPIPED)   ? 2
                                                                  : 0;
}
__host__ __device__ constexpr int shape_min_ctas(int pc, int N1, int KIND) {
  return pc == 0 ? (N1 == 8    ? (KIND == AX_GEOM_TRILINEAR ? 5 : 0)
                    : N1 == 6  ? (KIND == AX_GEOM_TRILINEAR ? 3 : KIND == AX_GEOM_TRILINEAR_PARTIAL ? 4 : 0)
                    : N1 == 10 ? (KIND == AX_GEOM_TRILINEAR ? 5 : KIND == AX_GEOM_TRILINEAR_PARTIAL ? 2 : 0)
                               : 0)
                 : (N1 == 8 && KIND == AX_GEOM_TRILINEAR)  ? 8
                 : (N1 == 12 && KIND == AX_GEOM_STORED) ? 4
                 : N1 == 16                              ? 2
                                                        : 0;
}
// the policy class of shape_epb / shape_min_ctas (-1: none)
template <class P>
constexpr int kShapeClass = P::kRoll ? 0 : sizeof(typename P::S) == 4 ? 1 : -1;

// Elements per CTA of the per-order kernels (0: the plain 128-thread rule).
// Measured on GB300: filling the warps (pick_epb) pays for the trilinear
// kinds in 8-byte arithmetic (double-word, FP64) and for every recompute
// kind at N1 = 6; the stored and parallelepiped kinds elsewhere, and FP32
// at N1 = 10, 12, run faster with the smaller CTAs (more of them per SM).
// The exceptions of shape_epb come first; native FP64 at N1 = 5 keeps the
// plain shape, whose 125 threads fill four warps to 98% already (filled: 350
// threads, one CTA of 104 registers per SM, 262 against 246 us for 11781
// elements; at the other orders the filled shapes stay up to 20% faster).
template <class P, int N1, int KIND>
constexpr int kEpb =
    (kShapeClass<P> >= 0 && shape_epb(kShapeClass<P>, N1, KIND)) ? shape_epb(kShapeClass<P>, N1, KIND)
    : (!P::kRoll && sizeof(typename P::S) == 8 && N1 == 5) ? 0
    : (KIND != AX_GEOM_STORED && (N1 == 6 || (sizeof(typename P::S) == 8 && KIND != AX_GEOM_PARALLELEPIPED)))
        ? pick_epb(N1 * N1)
        : 0;

// Minimum resident CTAs for the register budget (0: no bound): the
// double-word kernels at N1 = 16 (256-thread CTAs) are held to 128 registers
// so that two CTAs fit per SM (unbounded they take about 147 and run one CTA
// per SM, 5-30% slower); the double-word trilinear kernel at N1 = 12
// (288-thread CTAs) likewise to two CTAs (96 registers and some spills
// instead of 119 registers and one CTA: 33% faster; the partial kind
// measured 5% slower so and keeps its allocation); native FP64's partial kind at
// N1 = 7 to two CTAs of 392 threads (72 registers; unbounded it takes 102 and runs
// one: 1181 -> 1149 us for 8.4e6 nodes, 197 -> 194.6 for 1e6); the exceptions of
// shape_min_ctas.  Elsewhere no bound is given: even an explicit 1 changes
// the register allocation for the worse.
template <class P, int N1, int KIND>
constexpr int kMinCtas =
    (kShapeClass<P> >= 0 && shape_min_ctas(kShapeClass<P>, N1, KIND)) ? shape_min_ctas(kShapeClass<P>, N1, KIND)
    : (!P::kRoll && sizeof(typename P::S) == 8 && N1 == 7 && KIND == AX_GEOM_TRILINEAR_PARTIAL)            ? 2
    : (P::kRoll && (N1 == 16 || (N1 == 12 && KIND == AX_GEOM_TRILINEAR)))  ? 2
                                                                           : 0;
// The tile of twice the elements (float32): half the CTAs where the base tile's
// bound would make its 512 threads spill (N1 = 8 at eight CTAs; N1 = 16 at two, 800
// bytes: stored 299 -> 117 us for 1.6e7 nodes, trilinear 202 -> 100), and two CTAs
// at N1 = 14, where the recompute kinds would otherwise take 82 to 86 registers
// and run one (trilinear 123 -> 86, partial 123 -> 92).  The stored kind at N1 =
// 12 keeps its four (90 against 100 us at two), at 14 the 108 registers it takes.
template <class P, int N1, int KIND, int EM>
constexpr int kMinCtasEm = EM == 1                                ? kMinCtas<P, N1, KIND>
                           : N1 == 8 || N1 == 16                  ? kMinCtas<P, N1, KIND> / EM
                           : N1 == 14 && KIND != AX_GEOM_STORED   ? 2
                                                                  : kMinCtas<P, N1, KIND>;

// Trilinear kinds: whether an element's first 2 N1 threads compute the axis
// terms of the geometry (Geometry::axis_terms) for all its threads.  Measured
// on GB300: native FP64 3% faster (N = 7), double-word 7% faster at N = 3 and
// 3% at N = 5 but 1-4% slower at N = 7 (where the prologue is amortised over
// more nodes), FP32 1-3% slower; so native FP64 at every order, double-word
// up to N1 = 6.
template <class P, int N1, int KIND>
constexpr bool kShareAxis = (KIND == AX_GEOM_TRILINEAR || KIND == AX_GEOM_TRILINEAR_PARTIAL) &&
                            (P::kRoll ? N1 <= 6 : sizeof(typename P::V) == 8);

// An element in shared memory: node (i, j, k) at i + P j + PK k, in words.
// 8-byte words (double-word, FP64: bound by their pipes): rows padded
// by one word.  4-byte words: the float32 kernels move about 15 words per node
// through shared memory and are bound by it next to issue, so their pitches
// come from a search over a model of the banks (32 of 4 bytes, vectors of 2
// and 4 words served in phases of 16 and 8 lanes) for the fewest wavefronts of
// a node's accesses: four by r-fiber owners (lane (j, k), a row each, in
// vectors of `vec` words where that costs no more), four by s-fiber owners
// (lane (i, k)), seven by t-fiber owners (lane (i, j)).  15 is the least;
// padded rows alone need 22 at N1 = 4, 8 and 16, 23 to 28 at 6, 9, 10 and 12
// to 14, 34 to 77 at 5, 7, 11 and 15.  Together with the loads below and the
// packed geometry (Geometry2), measured on GB300: order 7 trilinear 258 -> 221
// us for 131072 elements, order 5 stored 434 -> 366 us for 309808, 1.02 to 1.47
// times at every order and kind of 3.2e7 nodes but the stored kind at order 1
// (equal).
struct Pitches {
  int P, PK, ES, vec;  // row, plane and element pitch; words per row access
};
//                                    wavefronts per node: N1 = 3: 23, 4: 19, 5: 23, 6: 20.5, 7: 21, 8: 15, 9: 17.7,
constexpr Pitches kPitches32[17] = {  // 10: 17.5, 11: 19, 12: 15.8, 13: 18.3, 14: 18.1, 15: 22, 16: 15
    {}, {}, {2, 6, 12, 2}, {3, 11, 41, 1}, {4, 20, 80, 4}, {5, 25, 153, 1}, {6, 36, 228, 2}, {7, 52, 369, 1},
    {12, 104, 820, 4}, {9, 81, 729, 1}, {10, 106, 1054, 2}, {11, 121, 1331, 1}, {12, 172, 2036, 4}, {13, 169, 2197, 1},
    {14, 206, 2874, 2}, {15, 225, 3375, 1}, {20, 336, 5356, 4}};
// kinds of layout: padded rows, for words of any size, or the searched one
enum { kPaddedRows = 0, kSearched32 = 1 };
template <class P, int N1, int KIND>
constexpr int kLayout = sizeof(typename P::S) == 4 && !(N1 == 8 && KIND == AX_GEOM_STORED) ? kSearched32 : kPaddedRows;
template <int N1, int LK>
struct Layout {
  static constexpr Pitches pt =
      LK == kSearched32 ? kPitches32[N1] : Pitches{N1 + 1, N1 * (N1 + 1), N1 * N1 * (N1 + 1), 1};
  static constexpr int P = pt.P, PK = pt.PK, ES = pt.ES, vec = pt.vec;
  static_assert(P >= N1 && PK >= (N1 - 1) * P + N1 && ES >= (N1 - 1) * (PK + P) + N1, "nodes apart");
  static_assert(N1 % vec == 0 && P % vec == 0 && PK % vec == 0 && ES % vec == 0, "aligned rows");
  // row j of the t-fibers owned by threads N1 b .. N1 b + N1 - 1: where a row
  // fills whole banks (N1 = 8, 16) a warp takes rows that lie 8 or 16 banks
  // apart (not in the stored kind at N1 = 8, whose factors a warp then reads
  // in 32-byte pieces: it is bound by HBM, 180 against 168 GDOF/s)
  __host__ __device__ static constexpr int row_of(int b) {
    return LK == kSearched32 && N1 == 8    ? ((b & 3) << 1) | (b >> 2)                          // 0 2 4 6 | 1 3 5 7
           : LK == kSearched32 && N1 == 16 ? ((b >> 1) & 3) | ((b & 1) << 2) | ((b >> 3) << 3)  // 0 4 | 1 5 | 2 6 | ..
                                           : b;
  }
};

template <int N1, int EM = 1, int EPB0 = 0, int LK = kPaddedRows>
struct Shape {
  using L = Layout<N1, LK>;
  static constexpr int n3 = N1 * N1 * N1;
  static constexpr int F = N1 * N1;  // fibers (threads) per element
  static constexpr int EPB = EM * (EPB0 > 0 ? EPB0 : (F >= 128 ? 1 : 128 / F));  // elements per CTA (EM: tile variant)
  static constexpr int threads = F * EPB;
  static constexpr int P = L::P, PK = L::PK, ES = L::ES;  // row, plane and element pitch (words)
  __device__ static __forceinline__ int at(int i, int j, int k) {
    return LK == kPaddedRows ? i + P * (j + N1 * k) : i + P * j + PK * k;
  }
};

// a row of N values in vectors of VEC floats
template <int N, int VEC>
__device__ __forceinline__ void load_row(const float *p, float v[N]) {
#pragma unroll
  for (int c = 0; c < N; c += VEC) {
    if constexpr (VEC == 4) {
      const float4 t = *reinterpret_cast<const float4 *>(p + c);
      v[c] = t.x; v[c + 1] = t.y; v[c + 2] = t.z; v[c + 3] = t.w;
    } else {
      const float2 t = *reinterpret_cast<const float2 *>(p + c);
      v[c] = t.x; v[c + 1] = t.y;
    }
  }
}
template <int N, int VEC>
__device__ __forceinline__ void store_row(float *p, const float v[N]) {
#pragma unroll
  for (int c = 0; c < N; c += VEC) {
    if constexpr (VEC == 4)
      *reinterpret_cast<float4 *>(p + c) = make_float4(v[c], v[c + 1], v[c + 2], v[c + 3]);
    else
      *reinterpret_cast<float2 *>(p + c) = make_float2(v[c], v[c + 1]);
  }
}

// ---------------------------------------------------------------------------
// geometry (getFactors of Algorithm 4) in policy arithmetic
//
// Trilinear (Algorithm 2, true Jacobian): the element's record holds the
// map's monomial coefficients (A..G of x = x0 + Ar + Bs + Ct + Drs + Ert +
// Fst + Grst, Eq. 8), from which thread (i,j) forms the columns
//   J0(t) = E0 + t E1  (E0, E1 depend on s = xi_j),
//   J1(t) = F0 + t F1  (F0, F1 depend on r = xi_i),   J2 = Jc2(r, s),
// so along its k-fiber (t = xi_k) every entry of K = J^T J is a polynomial
// in t of degree <= 2 (K02, K12 affine, K22 constant) and so is
// det J = J2 . (J0 x J1).  The prologue computes their coefficients once;
// each node then costs 10 multiply-adds for K and det J, the adjugate
// (Eq. 12) and one division:  (r,s,t) = adj(K) (lambda x), lambda = w/det J.
// ---------------------------------------------------------------------------
template <class P, int N1, int KIND>
struct Geometry {
  using V = typename P::V;
  using S = typename P::S;
  V wij;
  V k00[3], k01[3], k11[3], k02[2], k12[2], k22, dt[3];  // polynomial coefficients in t
  V h[7];
  const S *gl = nullptr;

  // Terms of the trilinear geometry that depend on one reference coordinate
  // only, written to out[0..8]:  axis 0 (u = r = xi_idx): F0 = B + D r,
  // F1 = F + G r and the K11 coefficients (F0.F0, 2 F0.F1, F1.F1);  axis 1
  // (u = s = xi_idx): E0 = A + D s, E1 = E + G s and the K00 coefficients.
  // An element has N1 of each, which its first 2 N1 threads compute once and
  // share (kAxisWords words per set) instead of every thread recomputing them.
  static constexpr int kAxisWords = 9;
  __device__ __forceinline__ static void axis_terms(const S *sv, const typename P::C *xg, int axis, int idx,
                                                    S *out) {
    const V u = P::cst(xg + idx);
    V X0[3], X1[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      auto M = [&](int m) { return P::ld(sv + 3 * m + c); };  // A B C D E F G = 0..6
      X0[c] = P::fma3(M(3), u, M(axis ? 0 : 1));
      X1[c] = P::fma3(M(6), u, M(axis ? 4 : 5));
      out[c] = P::st(X0[c]);
      out[3 + c] = P::st(X1[c]);
    }
    out[6] = P::st(dot3<P>(X0, X0));
    out[7] = P::st(P::twice(dot3<P>(X0, X1)));
    out[8] = P::st(dot3<P>(X1, X1));
  }

  // AX: read the axis terms from ax, the element's shared table
  // ([2][N1][kAxisWords], see axis_terms), instead of computing them here.
  template <bool AX = false>
  __device__ __forceinline__ void prologue(const S *sv, const typename P::C *xg, const typename P::C *wg, int i,
                                           int j, const S *G_e, const S *lam_e, const S *ax = nullptr) {
    wij = P::mul(P::cst(wg + i), P::cst(wg + j));
    if constexpr (KIND == AX_GEOM_STORED) {
      gl = G_e;
    } else if constexpr (KIND == AX_GEOM_PARALLELEPIPED) {
#pragma unroll
      for (int q = 0; q < 7; ++q) h[q] = P::ld(sv + q);
    } else {
      // columns of J from the monomial coefficients of the map (Eq. 8):
      // J0 = E0 + t E1, E0 = A + D s, E1 = E + G s;  J1 = F0 + t F1, F0 = B + D r,
      // F1 = F + G r;  J2 = C + E r + F s + G rs   (r = xi_i, s = xi_j)
      V E0[3], E1[3], F0[3], F1[3], J2[3];
      const V r = P::cst(xg + i), s = P::cst(xg + j), rs = P::mul(r, s);
      if constexpr (AX) {
        const S *fi = ax + i * kAxisWords, *ej = ax + (N1 + j) * kAxisWords;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          F0[c] = P::ld(fi + c); F1[c] = P::ld(fi + 3 + c);
          E0[c] = P::ld(ej + c); E1[c] = P::ld(ej + 3 + c);
          k11[c] = P::ld(fi + 6 + c); k00[c] = P::ld(ej + 6 + c);
        }
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        auto M = [&](int m) { return P::ld(sv + 3 * m + c); };  // A B C D E F G = 0..6
        if constexpr (!AX) {
          E0[c] = P::fma3(M(3), s, M(0));
          E1[c] = P::fma3(M(6), s, M(4));
          F0[c] = P::fma3(M(3), r, M(1));
          F1[c] = P::fma3(M(6), r, M(5));
        }
        typename P::A q = P::mul0(M(4), r);
        P::mac(q, M(5), s);
        P::mac(q, M(6), rs);
        J2[c] = P::add(M(2), P::fin(q));
      }
      if constexpr (!AX) {
        k00[0] = dot3<P>(E0, E0); k00[1] = P::twice(dot3<P>(E0, E1)); k00[2] = dot3<P>(E1, E1);
        k11[0] = dot3<P>(F0, F0); k11[1] = P::twice(dot3<P>(F0, F1)); k11[2] = dot3<P>(F1, F1);
      }
      // K = J^T J as polynomials in t
      k01[0] = dot3<P>(E0, F0); k01[1] = P::add(dot3<P>(E0, F1), dot3<P>(E1, F0)); k01[2] = dot3<P>(E1, F1);
      k02[0] = dot3<P>(E0, J2); k02[1] = dot3<P>(E1, J2);
      k12[0] = dot3<P>(F0, J2); k12[1] = dot3<P>(F1, J2);
      k22 = dot3<P>(J2, J2);
      if constexpr (KIND == AX_GEOM_TRILINEAR) {
        // det J(t) = J2 . (J0 x J1) = J0 . (J1 x J2): with w_a = F_a x J2
        V w0[3], w1[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const int c1 = (c + 1) % 3, c2 = (c + 2) % 3;
          w0[c] = det2<P>(F0[c1], J2[c2], F0[c2], J2[c1]);
          w1[c] = det2<P>(F1[c1], J2[c2], F1[c2], J2[c1]);
        }
        dt[0] = dot3<P>(E0, w0);
        dt[1] = P::add(dot3<P>(E0, w1), dot3<P>(E1, w0));
        dt[2] = dot3<P>(E1, w1);
      }
      gl = lam_e;
    }
  }

  __device__ __forceinline__ static V quad(const V c[3], V t) { return P::fma3(t, P::fma3(t, c[2], c[1]), c[0]); }
  __device__ __forceinline__ static V lin(const V c[2], V t) { return P::fma3(t, c[1], c[0]); }

  // adjugate of K at t (symmetric: A00 A01 A02 A11 A12 A22)
  __device__ __forceinline__ void adjK(V t, V A[6]) const {
    const V K00 = quad(k00, t), K01 = quad(k01, t), K11 = quad(k11, t), K02 = lin(k02, t), K12 = lin(k12, t);
    A[0] = det2<P>(K11, k22, K12, K12);
    A[1] = det2<P>(K02, K12, K01, k22);
    A[2] = det2<P>(K01, K12, K02, K11);
    A[3] = det2<P>(K00, k22, K02, K02);
    A[4] = det2<P>(K01, K02, K00, K12);
    A[5] = det2<P>(K00, K11, K01, K01);
  }

  // (r, s, t) = G (x0, x1, x2) at local node l (t = xi_k, wk = w_k)
  __device__ __forceinline__ void apply(int l, V t, V wk, const V xv[3], V out[3]) const {
    constexpr int n3 = N1 * N1 * N1;
    V A[6];
    V y[3];
    if constexpr (KIND == AX_GEOM_STORED) {
#pragma unroll
      for (int q = 0; q < 6; ++q) A[q] = P::ld(gl + q * n3 + l);
      y[0] = xv[0]; y[1] = xv[1]; y[2] = xv[2];
    } else if constexpr (KIND == AX_GEOM_PARALLELEPIPED) {
#pragma unroll
      for (int q = 0; q < 6; ++q) A[q] = h[q];
      const V W = P::mul(wij, wk);
      y[0] = P::mul(W, xv[0]); y[1] = P::mul(W, xv[1]); y[2] = P::mul(W, xv[2]);
    } else {
      adjK(t, A);
      V lam;
      if constexpr (KIND == AX_GEOM_TRILINEAR)
        lam = P::div(P::mul(wij, wk), quad(dt, t));
      else
        lam = P::ld(gl + l);
      y[0] = P::mul(lam, xv[0]); y[1] = P::mul(lam, xv[1]); y[2] = P::mul(lam, xv[2]);
    }
    const V gr[3] = {A[0], A[1], A[2]}, gs[3] = {A[1], A[3], A[4]}, gt[3] = {A[2], A[4], A[5]};
    out[0] = dot3<P>(gr, y);
    out[1] = dot3<P>(gs, y);
    out[2] = dot3<P>(gt, y);
  }

  // g[0..5] = g00 g01 g02 g11 g12 g22 at local node l; returns the seventh factor w|J|.
  __device__ __forceinline__ V factors(int l, V t, V wk, V g[6]) const {
    constexpr int n3 = N1 * N1 * N1;
    if constexpr (KIND == AX_GEOM_STORED) {
#pragma unroll
      for (int q = 0; q < 6; ++q) g[q] = P::ld(gl + q * n3 + l);
      return P::ld(gl + 6 * n3 + l);
    } else if constexpr (KIND == AX_GEOM_PARALLELEPIPED) {
      const V W = P::mul(wij, wk);
#pragma unroll
      for (int q = 0; q < 6; ++q) g[q] = P::mul(W, h[q]);
      return P::mul(W, h[6]);
    } else {
      V A[6];
      adjK(t, A);
      const V W = P::mul(wij, wk);
      V lam, wdet;
      if constexpr (KIND == AX_GEOM_TRILINEAR) {
        const V det = quad(dt, t);
        lam = P::div(W, det);
        wdet = P::mul(W, det);
      } else {
        lam = P::ld(gl + l);
        wdet = P::div(P::mul(W, W), lam);
      }
#pragma unroll
      for (int q = 0; q < 6; ++q) g[q] = P::mul(lam, A[q]);
      return wdet;
    }
  }
};


// The float32 geometry at two nodes of a fiber at once, the nodes k and N - k
// in the lanes of packed FP32x2 instructions (dw2.cuh): the same operations in
// the same order per node as Geometry<Native<float>>, half the instructions.
// The coefficients along the fiber are held twice, once per lane: up to 17
// more registers (kPackedGeo says where that pays).
template <int N1, int KIND>
struct Geometry2 {
  using f2 = dw2::f2;
  using G = Geometry<Native<float>, N1, KIND>;
  f2 k00[3], k01[3], k11[3], k02[2], k12[2], k22, dt[3], h[6];
  const float *gl;
  float wij;
  __device__ __forceinline__ static f2 both(float v) { return make_float2(v, v); }
  __device__ __forceinline__ explicit Geometry2(const G &g) : gl(g.gl), wij(g.wij) {
    if constexpr (KIND == AX_GEOM_PARALLELEPIPED) {
#pragma unroll
      for (int q = 0; q < 6; ++q) h[q] = both(g.h[q]);
    } else if constexpr (KIND != AX_GEOM_STORED) {
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        k00[q] = both(g.k00[q]);
        k01[q] = both(g.k01[q]);
        k11[q] = both(g.k11[q]);
        if constexpr (KIND == AX_GEOM_TRILINEAR) dt[q] = both(g.dt[q]);
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        k02[q] = both(g.k02[q]);
        k12[q] = both(g.k12[q]);
      }
      k22 = both(g.k22);
    }
  }
  __device__ __forceinline__ static f2 quad(const f2 c[3], f2 t) { return dw2::fma(t, dw2::fma(t, c[2], c[1]), c[0]); }
  __device__ __forceinline__ static f2 lin(const f2 c[2], f2 t) { return dw2::fma(t, c[1], c[0]); }
  __device__ __forceinline__ static f2 neg(f2 a) { return make_float2(-a.x, -a.y); }
  // a b + d e  (nc: one factor of the subtracted product, negated)
  __device__ __forceinline__ static f2 det2n(f2 a, f2 b, f2 nc, f2 d) { return dw2::fma(nc, d, dw2::mul(a, b)); }
  __device__ __forceinline__ static f2 dot(f2 a, f2 b, f2 c, const f2 y[3]) {
    return dw2::fma(c, y[2], dw2::fma(b, y[1], dw2::mul(a, y[0])));
  }
  // (r, s, t) = G (x0, x1, x2) at local nodes l (lane 0, t = -tk... any pair) and l2 (lane 1)
  __device__ __forceinline__ void apply(int l, int l2, f2 t, float wk, const f2 xv[3], f2 out[3]) const {
    constexpr int n3 = N1 * N1 * N1;
    f2 A[6], y[3];
    if constexpr (KIND == AX_GEOM_STORED) {
#pragma unroll
      for (int q = 0; q < 6; ++q) A[q] = make_float2(gl[q * n3 + l], gl[q * n3 + l2]);
      y[0] = xv[0]; y[1] = xv[1]; y[2] = xv[2];
    } else if constexpr (KIND == AX_GEOM_PARALLELEPIPED) {
#pragma unroll
      for (int q = 0; q < 6; ++q) A[q] = h[q];
      const f2 W = both(wij * wk);  // the weights of nodes k and N - k are equal
      y[0] = dw2::mul(W, xv[0]); y[1] = dw2::mul(W, xv[1]); y[2] = dw2::mul(W, xv[2]);
    } else {
      const f2 K00 = quad(k00, t), K01 = quad(k01, t), K11 = quad(k11, t), K02 = lin(k02, t), K12 = lin(k12, t);
      const f2 n01 = neg(K01), n02 = neg(K02), n12 = neg(K12);
      A[0] = det2n(K11, k22, n12, K12);
      A[1] = det2n(K02, K12, n01, k22);
      A[2] = det2n(K01, K12, n02, K11);
      A[3] = det2n(K00, k22, n02, K02);
      A[4] = det2n(K01, K02, n12, K00);
      A[5] = det2n(K00, K11, n01, K01);
      f2 lam;
      if constexpr (KIND == AX_GEOM_TRILINEAR) {
        const f2 det = quad(dt, t);
        lam = dw2::mul(both(wij * wk), make_float2(rcp32(det.x), rcp32(det.y)));
      } else {
        lam = make_float2(gl[l], gl[l2]);
      }
      y[0] = dw2::mul(lam, xv[0]); y[1] = dw2::mul(lam, xv[1]); y[2] = dw2::mul(lam, xv[2]);
    }
    out[0] = dot(A[0], A[1], A[2], y);
    out[1] = dot(A[1], A[3], A[4], y);
    out[2] = dot(A[2], A[4], A[5], y);
  }
};
// Where the float32 kernels take it.  Measured on GB300 (3.2e7 nodes, GDOF/s,
// packed / one node at a time, same layouts): trilinear faster at every order
// but N = 5 (equal), N = 3 221 / 193, 7 272 / 264, 14 187 / 174; the partial
// kind at N = 7 242 / 202, 11 225 / 196, slower at N <= 5 (183 / 205 at 5) and
// at 8; the stored and parallelepiped kinds, whose node is short, within 4%
// from N = 5 on and slower below or where the registers cost CTAs (stored:
// 175 / 192 at N = 10), but for stored at N = 3 and 8 (183 / 167, 165 / 133).
template <class P, int N1, int KIND>
constexpr bool kPackedGeo = !P::kRoll && sizeof(typename P::V) == 4 &&
                            (KIND == AX_GEOM_TRILINEAR              ? true
                             : KIND == AX_GEOM_TRILINEAR_PARTIAL    ? N1 > 6 && N1 != 9
                             : KIND == AX_GEOM_PARALLELEPIPED       ? N1 > 5 && N1 != 12
                                                                    : N1 == 4 || N1 == 9);


// Power-of-two scaling of an element's float64 values (policies with
// kScaleIO).  emax is the largest biased exponent field among the element's
// values; the shift d brings the largest magnitude into [1, 2) (clamped so
// that 2^d and 2^-d are normal doubles).  Elements with an infinity or NaN
// (emax 0x7ff) are not scaled.
__device__ __forceinline__ int io_shift(int emax) {
  if (emax == 0x7ff) return 0;
  if (emax == 0) return 1022;  // zeros and float64 subnormals: brought up by 2^1022
  const int d = 1023 - emax;
  return d < -1022 ? -1022 : (d > 1022 ? 1022 : d);
}
__device__ __forceinline__ double pow2i(int d) { return __hiloint2double((1023 + d) << 20, 0); }
__device__ __forceinline__ int exp_field(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }
__device__ __forceinline__ int exp_field(float v) { return (__float_as_int(v) >> 23) & 0xff; }
// Direct range of the double-word kernels, tested per row of N1 values on
// the largest magnitude of the row, read from the upper 32 bits of the
// float64 values (sign cleared, integer order = magnitude order): a row is
// direct when it is all zero or its largest magnitude lies in
// [2^-60, 2^61), and no value of it is nonzero below 2^-74.  Within it the
// float pairs and every intermediate of the product stay normal floats for
// element extents in [2^-20, 2^24] (checked at setup), values far below their
// row's largest contribute below the accuracy, and X is converted by integer
// instructions (dw::from_double_direct, whose range ends at 2^-74); Y goes
// back the same way (dw::sum3_to_double_direct).  The other blocks are
// converted on the FP64 pipe.
__device__ __forceinline__ int mag_hi(double v) { return __double2hiint(v) & 0x7fffffff; }
__device__ __forceinline__ bool row_direct(int hmax) {
  return hmax == 0 || (hmax >= ((1023 - 60) << 20) && hmax < ((1023 + 61) << 20));
}

// Double-word blocks that load one i-row per thread instead of the thread's
// t-fiber.  Measured on GB300 (3.2e7 nodes): at N1 = 3, 12 and 14 the t-fibers
// cost registers that the arithmetic needs (9% slower for the trilinear kind at
// N1 = 3, 5 and 17% for the stored kind at 12 and 14); at the other orders they
// are equal to 3%, or faster (N1 = 4 stored 80 against 58 GDOF/s, N1 = 16 by 5
// to 9%).
template <class P, int N1>
constexpr bool kRowLoads = P::kRoll && (N1 == 3 || N1 == 12 || N1 == 14);

template <int KIND>
struct GeoWords {
  static constexpr int value = (KIND == AX_GEOM_STORED) ? 0 : (KIND == AX_GEOM_PARALLELEPIPED ? kParWords : kVertexWords);
};

// Sources of X: in place (element e's values at X[e n3 + m]), in place in host
// memory (XLink), or formed from the assembled vectors of a CG iteration (XCg).
template <typename IO>
struct XDirect {
  static constexpr bool kCg = false, kLink = false;
  const IO *__restrict__ p;
  __device__ __forceinline__ IO operator[](int64_t m) const { return p[m]; }
};
// X and Y in page-locked host memory, read and written over the host link
// (ax_local_host, float32): consecutive words by consecutive threads, both ways
// through shared memory.  The accesses that are best against HBM and shared
// memory are not against the link, which moves a line's pieces one by one and
// waits longer for each.  Measured on GB300 (3.2e7 nodes each way, us per call,
// with the plain kernel / with this one; the link alone takes about 750): order 7
// trilinear 950 / 789 (its warps touch four 32-byte pieces of four lines,
// Layout::row_of), parallelepiped 1010 / 793, partial 1120 / 787; stored order 1
// 980 / 760, order 3 853 / 777, order 5 1130 / 990; trilinear order 5 1110 / 778,
// order 15 838 / 804.
template <typename IO>
struct XLink {
  static constexpr bool kCg = false, kLink = true;
  const IO *__restrict__ p;
};
// The search direction of a CG iteration, formed at each local copy while it
// is loaded: p_new[g] = z[g] + beta p[g].  The thread that loads a node's
// first copy also stores p_new and brings x up to date, x += alpha p, with
// the last iteration's alpha and direction.  p_new goes to another vector
// than p, so every copy sees the same p.  Y is stored by rank (CgArgs).
template <typename IO>
struct XCg {
  static constexpr bool kCg = true, kLink = false;
  static constexpr int kBatch = 8;  // nodes whose loads are in flight together
  const gidx *__restrict__ own;
  const gidx *__restrict__ rank;
  const IO *__restrict__ z;
  const IO *__restrict__ p;
  IO *pn, *x, *U;
  IO alpha, beta;
  // local copies m, m + step, ... (n of them; all loads before the first store)
  template <int n>
  __device__ __forceinline__ void get(int64_t m, int step, IO *out) const {
    gidx g[n];
    IO zv[n], pv[n], xv[n];
#pragma unroll
    for (int u = 0; u < n; ++u) g[u] = own[m + u * step];
#pragma unroll
    for (int u = 0; u < n; ++u) {
      const gidx h = g[u] & 0x7fffffff;
      zv[u] = z[h];
      pv[u] = p[h];
      xv[u] = g[u] < 0 ? x[h] : IO(0);
    }
#pragma unroll
    for (int u = 0; u < n; ++u) {
      const gidx h = g[u] & 0x7fffffff;
      out[u] = zv[u] + beta * pv[u];
      if (g[u] < 0) {
        pn[h] = out[u];
        x[h] = xv[u] + alpha * pv[u];
      }
    }
  }
  __device__ __forceinline__ IO operator[](int64_t m) const { return U[m]; }  // after the block's loads (float64 IO)
};

// Shared-memory buffers of one block of EPB elements.
// EPB0: the block shape (kEpb for the per-order kernels).
template <class P, int N1, int KIND, int EM, int EPB0 = kEpb<P, N1, KIND>>
struct FiberSmem {
  using Sh = Shape<N1, EM, EPB0, kLayout<P, N1, KIND>>;
  using S = typename P::S;
  static constexpr int GW = GeoWords<KIND>::value, GWD = GW > 0 ? GW : 1;
  static constexpr bool AXS = kShareAxis<P, N1, KIND>;
  static constexpr int AXD = AXS ? 2 * N1 * Geometry<P, N1, KIND>::kAxisWords : 1;
  S *xs;        // [3][EPB][ES]: x, x0, x1; later t / Y_t, r / Y_r, s / Y_s
  S *sgeo;      // [EPB][GWD]: the elements' geometry records
  S *sax;       // [EPB][AXD]: per-element axis terms of the trilinear geometry (AXS)
  int *sexp;    // kScaleIO: [EPB] largest exponent field of each element's X, then the block's flag
  __host__ __device__ static constexpr size_t a16(size_t b) { return (b + 15) / 16 * 16; }
  // all four carved from one 16-byte aligned buffer of `bytes` bytes
  static constexpr size_t bytes = a16(sizeof(S) * 3 * Sh::EPB * Sh::ES) + a16(sizeof(S) * Sh::EPB * GWD) +
                                  a16(sizeof(S) * Sh::EPB * AXD) + a16(sizeof(int) * (Sh::EPB + 1));
  __device__ static __forceinline__ FiberSmem carve(unsigned char *raw) {
    FiberSmem m;
    m.xs = (S *)raw;
    raw += a16(sizeof(S) * 3 * Sh::EPB * Sh::ES);
    m.sgeo = (S *)raw;
    raw += a16(sizeof(S) * Sh::EPB * GWD);
    m.sax = (S *)raw;
    raw += a16(sizeof(S) * Sh::EPB * AXD);
    m.sexp = (int *)raw;
    return m;
  }
};

// ---------------------------------------------------------------------------
// AxLocal of one block of elements [e0, e0 + nel), nel <= EPB, by the CTA's
// threads (Algorithm 1 with the geometry of Algorithms 2 and 3).  Tables
// (per translation unit, constant memory): c_eoD / c_eoDT even-odd blocks of
// D and D^T, c_w, c_x weights and points.  IDLE: the CTA may have more
// threads than the order's shape (a CTA shaped for several orders); those
// threads only take part in the barriers.
// ---------------------------------------------------------------------------
// Returns, with X the direction of a CG iteration (XCg), this thread's share
// of X . Y (the dot product p . A p needs no assembled vector: p^T Q^T Y over
// the local copies), else 0.
template <class P, int N1, int KIND, int EM, bool IDLE, class XS, int EPB0 = kEpb<P, N1, KIND>>
__device__ __forceinline__ typename P::IO fiber_block(const FiberSmem<P, N1, KIND, EM, EPB0> &sm, const int tid, const int64_t e0,
                                            const int nel, const typename P::S *__restrict__ geo,
                                            const typename P::S *__restrict__ lam, const XS &X,
                                            typename P::IO *__restrict__ Y) {
  using Sh = Shape<N1, EM, EPB0, kLayout<P, N1, KIND>>;
  using Buf = FiberSmem<P, N1, KIND, EM, EPB0>;
  using V = typename P::V;
  using S = typename P::S;
  constexpr int n3 = Sh::n3, F = Sh::F, EPB = Sh::EPB, ES = Sh::ES;
  constexpr int GW = GeoWords<KIND>::value;
  static_assert(!IDLE || !P::kRoll, "idle threads are handled in the short (native) kernel body");
  S *const xs = sm.xs;          // [EPB][ES]: x, later Y
  S *const b0 = xs + EPB * ES;  // x0, later r
  S *const b1 = b0 + EPB * ES;  // x1, later s
  int *const sexp = sm.sexp;
  constexpr bool AXS = Buf::AXS;
  constexpr int AXW = Geometry<P, N1, KIND>::kAxisWords;
  const bool act = !IDLE || tid < Sh::threads;
  const int z = tid / Sh::F, q = tid % Sh::F;
  const int qa = q % N1, qb = q / N1;   // this thread's r-fiber (j, k), s-fiber (i, k) and t-fiber (i, jt)
  const int jt = Sh::L::row_of(qb);
  const typename P::C *eoD = c_eoD + tab_off_D(N1);
  const typename P::C *eoDT = c_eoDT + tab_off_D(N1);
  const float4 *eo2D = c_eo2D + tab_off_P(N1), *eo2DT = c_eo2DT + tab_off_P(N1);
  const typename P::C *cw = c_w + tab_off_v(N1);
  const typename P::C *cx = c_x + tab_off_v(N1);
  const S *const sgeo_z = sm.sgeo + (act ? z : 0) * Buf::GWD;
  S *const sax_z = sm.sax + (act && AXS ? z : 0) * Buf::AXD;
  const int64_t e = e0 + z;
  const bool live = act && z < nel;
  typename P::IO xy = 0;

  // pass 0: the elements into padded shared memory, each thread its own
  // t-fiber: for every k a warp reads consecutive (i, j), so the loads are
  // coalesced, and the shared-memory addresses need no division.  Against one
  // i-row per thread (64 contiguous bytes per lane at N1 = 8) this matters most
  // where a call is a fraction of a wave: order 7, 512 elements in double-word
  // pairs 14.3 -> 12.3 us.  In native arithmetic D_t x starts from the
  // registers that were just loaded.
  // Policies with kScaleIO (float64 data in float32 pairs): X is converted
  // directly, and the threads test whether their fiber's largest magnitude lies
  // outside the direct range (row_direct).  If any fiber of the block does, the
  // block reads X again: each element is scaled by the power of two that
  // brings its largest magnitude into [1, 2) before the conversion, and its Y
  // is scaled back on the way out.
  S *const x_e = xs + z * ES, *const r_e = b0 + z * ES, *const s_e = b1 + z * ES;
  const int fr = Sh::at(0, qa, qb), fs = Sh::at(qa, 0, qb), ft = Sh::at(qa, jt, 0);
  constexpr int str_r = 1, str_s = Sh::P, str_t = Sh::PK;
  const int64_t own = e * n3 + qa + N1 * jt;  // node (qa, jt, 0); k: + k F
  constexpr bool kRegX = !P::kRoll;  // native arithmetic: the fiber's x stays in registers for D_t x
  V xt[kRegX ? N1 : 1];
  // value m of the block in shared memory
  auto place = [](int m) {
    const int row = m / N1;  // row (j, k) of element row / F
    return row / F * ES + row / N1 % N1 * Sh::PK + row % N1 * Sh::P + m % N1;
  };
  bool wide = false;  // this thread's fiber (or row) lies outside the direct range
  constexpr bool kRows = kRowLoads<P, N1> && !XS::kCg;
  if constexpr (kRows) {
    static_assert(ES == N1 * N1 * Sh::P, "value m of the block at (m / N1) P + m % N1");
    for (int row = tid; row < nel * N1 * N1; row += Sh::threads) {
      const int64_t src = e0 * n3 + (int64_t)row * N1;
      S *dst = xs + row * Sh::P;
      int hmax = 0;
      bool tiny = false;
#pragma unroll
      for (int i = 0; i < N1; ++i) {
        const typename P::IO v = X[src + i];
        hmax = max(hmax, mag_hi(v));
        tiny |= dw::tiny_nonzero((unsigned)mag_hi(v));
        dst[i] = P::st(P::from_io_direct(v));
      }
      wide |= tiny || !row_direct(hmax);
    }
  } else if constexpr (XS::kLink) {
    static_assert(kRegX && !IDLE, "the float32 kernels");
#pragma unroll
    for (int s = 0; s < N1; ++s) {
      const int m = tid + s * Sh::threads;
      if (m < nel * n3) xs[place(m)] = P::st(P::from_io(X.p[e0 * n3 + m]));
    }
  } else if (live) {
    using IO = typename P::IO;
    int hmax = 0;       // the fiber's largest magnitude (upper 32 bits)
    bool tiny = false;  // a nonzero value below from_io_direct's range
    IO cgv[8];
#pragma unroll
    for (int k = 0; k < N1; ++k) {
      IO v;
      if constexpr (XS::kCg) {
        constexpr int B = XS::kBatch, R = N1 % B ? N1 % B : B;
        if (k % B == 0) {
          if (k + B <= N1)
            X.template get<B>(own + k * F, F, cgv);
          else
            X.template get<R>(own + k * F, F, cgv);
        }
        v = cgv[k % B];
        if constexpr (P::kScaleIO) X.U[own + k * F] = v;  // read back for the dot product and the scaled reload
      } else {
        v = X[own + k * F];
      }
      if constexpr (P::kScaleIO) {
        hmax = max(hmax, mag_hi(v));
        tiny |= dw::tiny_nonzero((unsigned)mag_hi(v));
      }
      const V xv = P::from_io_direct(v);
      x_e[ft + k * str_t] = P::st(xv);
      if constexpr (kRegX) xt[k] = xv;
    }
    if constexpr (P::kScaleIO) wide = tiny || !row_direct(hmax);
  } else if constexpr (kRegX) {
#pragma unroll
    for (int k = 0; k < N1; ++k) xt[k] = P::lit(0.0);
  }
  if constexpr (GW > 0) {
    if (act) {
      for (int m = tid; m < nel * GW; m += Sh::threads) sm.sgeo[(m / GW) * Buf::GWD + m % GW] = geo[e0 * GW + m];
    }
  }
  if constexpr (P::kScaleIO) {
    const bool any_wide = __syncthreads_or(wide);
    if (tid == 0) sexp[EPB] = any_wide;  // read again when Y is stored (a register less meanwhile)
    if (any_wide) {
      if (tid < EPB) sexp[tid] = 0;
      __syncthreads();
      if (live) {
        int mx = 0;
#pragma unroll 1
        for (int k = 0; k < N1; ++k) mx = max(mx, exp_field(X[kRows ? e * n3 + q * N1 + k : own + k * F]));
        atomicMax(&sexp[z], mx);
      }
      __syncthreads();
      if (live) {
        const typename P::IO sc = pow2i(io_shift(sexp[z]));
#pragma unroll 1
        for (int k = 0; k < N1; ++k)
          x_e[kRows ? fr + k : ft + k * str_t] = P::st(P::from_io(X[kRows ? e * n3 + q * N1 + k : own + k * F] * sc));
      }
      __syncthreads();
    }
  } else {
    __syncthreads();
  }
  if constexpr (XS::kLink) {
#pragma unroll
    for (int k = 0; k < N1; ++k) xt[k] = live ? P::ld(x_e + ft + k * str_t) : P::lit(0.0);
  }
  if constexpr (AXS) {
    // threads q < 2 N1 of each element: the N1 r-axis and N1 s-axis terms,
    // read by every thread's geometry prologue after the next barriers
    if (live && q < 2 * N1) Geometry<P, N1, KIND>::axis_terms(sgeo_z, cx, q / N1, q % N1, sax_z + q * AXW);
  }

  // Six fiber products in two rolled phase loops (one code copy of the fiber
  // product per matrix, D or D^T, so the constants stay immediate operands
  // and the instruction footprint fits the instruction cache):
  //   ph 0: r-fibers  D x -> B0 (x0)     ph 1: s-fibers  D x -> B1 (x1)
  //   ph 2: t-fiber   D x -> X  (x2);  then per node the geometry and
  //         (r,s,t) = G (x0,x1,x2): r -> B0, s -> B1, t -> X
  //   ph 3: t-fiber   D^T t -> registers (Y_t)
  //   ph 4: r-fibers  D^T r -> B0 (Y_r)  ph 5: s-fibers  D^T s -> B1 (Y_s)
  //   then the t-fiber owner stores Y = Y_t + Y_r + Y_s to HBM
  auto forward = [&](int ph) {
    if (ph == 2) __syncthreads();  // every r/s-fiber read of x is done before x is overwritten
    S *dst = ph == 0 ? r_e : (ph == 1 ? s_e : x_e);
    const int base = ph == 0 ? fr : (ph == 1 ? fs : ft);
    const int stride = ph == 0 ? str_r : (ph == 1 ? str_s : str_t);
    V fin_[N1], fout[N1];
#pragma unroll
    for (int n = 0; n < N1; ++n) fin_[n] = P::ld(x_e + base + n * stride);
    contract_p<P, N1, KIND>(eoD, eo2D, fin_, fout);
#pragma unroll
    for (int n = 0; n < N1; ++n) dst[base + n * stride] = P::st(fout[n]);
  };
  if constexpr (P::kRoll) {
#pragma unroll 1
    for (int ph = 0; ph < 3; ++ph) forward(ph);
  __syncthreads();
  {
    // thread (i, j) = (qa, jt): geometry and G x along its own t-fiber
    const int i = qa, j = jt;
    Geometry<P, N1, KIND> gm;
    gm.template prologue<AXS>(sgeo_z, cx, cw, i, j, (KIND == AX_GEOM_STORED && live) ? geo + e * 7 * n3 : nullptr,
                              (KIND == AX_GEOM_TRILINEAR_PARTIAL && live) ? lam + e * n3 : nullptr, sax_z);
    auto node = [&](int k) {
      const int sidx = ft + k * str_t;
      const V xv[3] = {P::ld(r_e + sidx), P::ld(s_e + sidx), P::ld(x_e + sidx)};
      V o3[3];
      if (live) {
        gm.apply(i + j * N1 + k * N1 * N1, P::cst(cx + k), P::cst(cw + k), xv, o3);
      } else {
        o3[0] = o3[1] = o3[2] = P::lit(0.0);
      }
      r_e[sidx] = P::st(o3[0]);
      s_e[sidx] = P::st(o3[1]);
      x_e[sidx] = P::st(o3[2]);
    };
#pragma unroll 1
    for (int k = 0; k < N1; ++k) node(k);
  }
    // transposed products: D_t^T t of the own t-fiber, then the r- and
    // s-fibers in place in B0, B1 (one rolled loop: one code copy of the D^T
    // product); the t-fiber owner sums and stores Y.  Y_t stays in registers
    // up to N1 = 10; above, the 2 N1 extra registers would cost resident
    // warps, so it goes back in place into X (read only by its owner).
    constexpr bool kYtRegs = N1 <= 10;
    V yt[kYtRegs ? N1 : 1];
#pragma unroll 1
    for (int ph = 3; ph < 6; ++ph) {
      if (ph == 4) __syncthreads();  // every thread's r, s values are in B0, B1
      S *buf = ph == 3 ? x_e : (ph == 4 ? r_e : s_e);
      const int base = ph == 3 ? ft : (ph == 4 ? fr : fs);
      const int stride = ph == 3 ? str_t : (ph == 4 ? str_r : str_s);
      V fin_[N1], fout[N1];
#pragma unroll
      for (int n = 0; n < N1; ++n) fin_[n] = P::ld(buf + base + n * stride);
      contract_p<P, N1, KIND>(eoDT, eo2DT, fin_, fout);
      if (kYtRegs && ph == 3) {
#pragma unroll
        for (int n = 0; n < N1; ++n) yt[kYtRegs ? n : 0] = fout[n];
      } else {
#pragma unroll
        for (int n = 0; n < N1; ++n) buf[base + n * stride] = P::st(fout[n]);
      }
    }
    __syncthreads();  // every Y_r, Y_s value is in B0, B1
    if (live) {
      auto yt_of = [&](int k) { return kYtRegs ? yt[kYtRegs ? k : 0] : P::ld(x_e + ft + k * str_t); };
      auto store = [&](auto y_of) {
        if constexpr (XS::kCg) {
          constexpr int B = 4;  // places and x of B nodes are loaded before the first of them is stored
#pragma unroll
          for (int k0 = 0; k0 < N1; k0 += B) {
            gidx at[B];
            typename P::IO xv[B];
#pragma unroll
            for (int k = k0; k < N1 && k < k0 + B; ++k) {
              at[k - k0] = X.rank[own + k * F];
              xv[k - k0] = X[own + k * F];
            }
#pragma unroll
            for (int k = k0; k < N1 && k < k0 + B; ++k) {
              const typename P::IO y = y_of(k);
              Y[at[k - k0]] = y;
              xy += xv[k - k0] * y;
            }
          }
        } else {
#pragma unroll
          for (int k = 0; k < N1; ++k) Y[own + k * F] = y_of(k);
        }
      };
      if (!sexp[EPB]) {
        store([&](int k) {
          const int sidx = ft + k * str_t;
          return P::sum3_io_direct(yt_of(k), P::ld(r_e + sidx), P::ld(s_e + sidx));
        });
      } else {
        // the element entered as X 2^d: undo it (exact)
        const typename P::IO ysc = pow2i(-io_shift(sexp[z]));
        store([&](int k) {
          const int sidx = ft + k * str_t;
          return P::sum3_io(yt_of(k), P::ld(r_e + sidx), P::ld(s_e + sidx)) * ysc;
        });
      }
    }
  } else {
    // Short code (native arithmetic): the thread's own t-fiber stays in
    // registers from D_t x through the geometry to D_t^T t (no shared-memory
    // round trips, x never overwritten); the r- and s-fiber transposed
    // products overwrite B0 and B1 in place (no read-modify-write of Y, no
    // barrier between them); the t-fiber owner sums Y = Y_t + Y_r + Y_s at
    // its nodes and stores it to HBM (for each k the warp writes consecutive
    // i, j: coalesced).  (IDLE threads skip every step but the barriers.)
    V tf[N1];
    if (act) {
      contract_p<P, N1, KIND>(eoD, eo2D, xt, tf);
      if constexpr (Sh::L::vec > 1) {
        V fin_[N1], fout[N1];
        load_row<N1, Sh::L::vec>(x_e + fr, fin_);
        contract_p<P, N1, KIND>(eoD, eo2D, fin_, fout);
        store_row<N1, Sh::L::vec>(r_e + fr, fout);
      } else {
        forward(0);
      }
      forward(1);
    }
    __syncthreads();  // every r/s fiber product is in B0, B1
    V yt[N1];
    if (act) {
      const int i = qa, j = jt;
      Geometry<P, N1, KIND> gm;
      const int64_t eg = live ? e : e0;
      gm.template prologue<AXS>(sgeo_z, cx, cw, i, j, KIND == AX_GEOM_STORED ? geo + eg * 7 * n3 : nullptr,
                                KIND == AX_GEOM_TRILINEAR_PARTIAL ? lam + eg * n3 : nullptr, sax_z);
      // (threads beyond the last element work on the block's first one's
      // geometry: no branch per node, their results are not stored; but for the
      // stored kind at order 1, where the loads are scheduled better with one:
      // 162 -> 164.5 GDOF/s on 3.2e7 nodes)
      constexpr bool kNodeBranch = N1 == 2 && KIND == AX_GEOM_STORED;
      auto node = [&](int k) {
        const int sidx = ft + k * str_t;
        const V xv[3] = {P::ld(r_e + sidx), P::ld(s_e + sidx), tf[k]};
        V o3[3];
        if (!kNodeBranch || live)
          gm.apply(i + j * N1 + k * N1 * N1, P::cst(cx + k), P::cst(cw + k), xv, o3);
        else
          o3[0] = o3[1] = o3[2] = P::lit(0.0);
        r_e[sidx] = P::st(o3[0]);
        s_e[sidx] = P::st(o3[1]);
        tf[k] = o3[2];
      };
      if constexpr (kPackedGeo<P, N1, KIND>) {
        const Geometry2<N1, KIND> g2(gm);
#pragma unroll
        for (int k = 0; k < N1 / 2; ++k) {
          const int k2 = N1 - 1 - k, s1 = ft + k * str_t, s2 = ft + k2 * str_t;
          const float2 xv[3] = {make_float2(r_e[s1], r_e[s2]), make_float2(s_e[s1], s_e[s2]),
                                make_float2(tf[k], tf[k2])};
          float2 o3[3];
          g2.apply(i + j * N1 + k * N1 * N1, i + j * N1 + k2 * N1 * N1, make_float2(cx[k], cx[k2]), cw[k], xv, o3);
          r_e[s1] = o3[0].x;
          r_e[s2] = o3[0].y;
          s_e[s1] = o3[1].x;
          s_e[s2] = o3[1].y;
          tf[k] = o3[2].x;
          tf[k2] = o3[2].y;
        }
        if constexpr (N1 & 1) node(N1 / 2);
      } else {
#pragma unroll
        for (int k = 0; k < N1; ++k) node(k);
      }
      contract_p<P, N1, KIND>(eoDT, eo2DT, tf, yt);
    }
    __syncthreads();  // every r, s value is in B0, B1
#pragma unroll
    for (int d = 0; d < 2; ++d) {
      if (!act) break;
      S *buf = d == 0 ? r_e : s_e;
      const int base = d == 0 ? fr : fs, stride = d == 0 ? str_r : str_s;
      V fin_[N1], fout[N1];
      if constexpr (Sh::L::vec > 1) {
        if (d == 0) {
          load_row<N1, Sh::L::vec>(buf + base, fin_);
          contract_p<P, N1, KIND>(eoDT, eo2DT, fin_, fout);
          store_row<N1, Sh::L::vec>(buf + base, fout);
          continue;
        }
      }
#pragma unroll
      for (int n = 0; n < N1; ++n) fin_[n] = P::ld(buf + base + n * stride);
      contract_p<P, N1, KIND>(eoDT, eo2DT, fin_, fout);
#pragma unroll
      for (int n = 0; n < N1; ++n) buf[base + n * stride] = P::st(fout[n]);
    }
    __syncthreads();  // every Y_r, Y_s value is in B0, B1
    if (live) {
      gidx at[XS::kCg ? N1 : 1];
      if constexpr (XS::kCg) {
#pragma unroll
        for (int k = 0; k < N1; ++k) at[k] = X.rank[own + k * F];
      }
#pragma unroll
      for (int k = 0; k < N1; ++k) {
        const int sidx = ft + k * str_t;
        const V y = P::sum3_io(yt[k], P::ld(r_e + sidx), P::ld(s_e + sidx));
        if constexpr (XS::kCg) {
          Y[at[k]] = y;
          xy += P::ld(x_e + sidx) * y;  // X still lies where it was loaded
        } else if constexpr (XS::kLink) {
          x_e[sidx] = P::st(y);  // x is no longer read
        } else {
          Y[own + k * F] = y;
        }
      }
    }
  }

  if constexpr (XS::kLink) {
    __syncthreads();
#pragma unroll
    for (int s = 0; s < N1; ++s) {
      const int m = tid + s * Sh::threads;
      if (m < nel * n3) Y[e0 * n3 + m] = P::ld(xs + place(m));
    }
  }

  __syncthreads();  // the next block reuses the shared buffers
  return xy;
}

// ---------------------------------------------------------------------------
// the per-order kernel: blocks of EPB elements, persistent over blocks when
// the grid is capped (autotuner)
// ---------------------------------------------------------------------------
template <class P, int N1, int KIND, int EM>
__global__ void __launch_bounds__(Shape<N1, EM, kEpb<P, N1, KIND>>::threads, kMinCtasEm<P, N1, KIND, EM>)
    ax_fiber_kernel(int64_t E, const typename P::S *__restrict__ geo, const typename P::S *__restrict__ lam,
                    const typename P::IO *__restrict__ X, typename P::IO *__restrict__ Y) {
  using Sh = Shape<N1, EM, kEpb<P, N1, KIND>>;
  using Buf = FiberSmem<P, N1, KIND, EM>;
  using S = typename P::S;
  constexpr int EPB = Sh::EPB;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ S sgeo[EPB][Buf::GWD];
  __shared__ S sax[Buf::AXS ? EPB : 1][Buf::AXD];
  __shared__ int sexp[P::kScaleIO ? EPB + 1 : 1];
  Buf sm;
  sm.xs = (S *)smem_raw;
  sm.sgeo = &sgeo[0][0];
  sm.sax = &sax[0][0];
  sm.sexp = sexp;
  const int tid = threadIdx.x;
  const int64_t nblk = (E + EPB - 1) / EPB;
  for (int64_t blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
    const int64_t e0 = blk * EPB;
    const int nel = (int)((E - e0) < EPB ? (E - e0) : EPB);
    fiber_block<P, N1, KIND, EM, false>(sm, tid, e0, nel, geo, lam, XDirect<typename P::IO>{X}, Y);
  }
}

// Where ax_local_host runs this kernel on host memory: float32 (with float64
// values the copies by chunks are faster), but for the recompute kinds of order
// 2, whose blocks of 14 elements end in the middle of a line whatever the order
// of the accesses (trilinear: the plain kernel 932 us, this one 968).
template <class P, int N1, int KIND>
constexpr bool kHasLink = sizeof(typename P::IO) == 4 && !(N1 == 3 && KIND != AX_GEOM_STORED);

// The same with X and Y in host memory (XLink).
template <class P, int N1, int KIND>
__global__ void __launch_bounds__(Shape<N1, 1, kEpb<P, N1, KIND>>::threads, kMinCtas<P, N1, KIND>)
    ax_fiber_link_kernel(int64_t E, const typename P::S *__restrict__ geo, const typename P::S *__restrict__ lam,
                         const typename P::IO *__restrict__ X, typename P::IO *__restrict__ Y) {
  using Sh = Shape<N1, 1, kEpb<P, N1, KIND>>;
  using Buf = FiberSmem<P, N1, KIND, 1>;
  using S = typename P::S;
  constexpr int EPB = Sh::EPB;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ S sgeo[EPB][Buf::GWD];
  __shared__ S sax[Buf::AXS ? EPB : 1][Buf::AXD];
  Buf sm;
  sm.xs = (S *)smem_raw;
  sm.sgeo = &sgeo[0][0];
  sm.sax = &sax[0][0];
  sm.sexp = nullptr;
  const int64_t nblk = (E + EPB - 1) / EPB;
  for (int64_t blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
    const int64_t e0 = blk * EPB;
    const int nel = (int)((E - e0) < EPB ? (E - e0) : EPB);
    fiber_block<P, N1, KIND, 1, false>(sm, threadIdx.x, e0, nel, geo, lam, XLink<typename P::IO>{X}, Y);
  }
}

// The policies with a CG form of the kernel: those that solvers run on by
// default (native FP64 and the tensor-core kernels take the general iteration).
template <class P>
constexpr bool kHasCg = P::kRoll || sizeof(typename P::IO) == 4;

// First half of a CG iteration (ax_gs.cu): p_new = z + beta p formed in the
// loads, x += alpha p, W = A_e p_new, and alpha = r.z / p.w by the CTA that
// arrives last.  It takes the place of a direction-and-scatter kernel, the
// plain AxLocal and a dot product; the vectors' loads overlap the arithmetic
// that bounds the operator: order 7, 4096 elements, double-word 75 us (AxLocal
// alone 60), float32 20 (10); the kernels whose place it takes took 38 and 25.
// (A resident CTA per slot that loops over the blocks keeps the CTAs' phases
// in step: 86 us instead of 78.)
template <class P, int N1, int KIND>
__global__ void __launch_bounds__(Shape<N1, 1, kEpb<P, N1, KIND>>::threads, kMinCtas<P, N1, KIND>)
    ax_fiber_cg_kernel(int64_t E, const typename P::S *__restrict__ geo, const typename P::S *__restrict__ lam,
                       const CgArgs c, typename P::IO *__restrict__ Y) {
  using Sh = Shape<N1, 1, kEpb<P, N1, KIND>>;
  using Buf = FiberSmem<P, N1, KIND, 1>;
  using S = typename P::S;
  using IO = typename P::IO;
  constexpr int EPB = Sh::EPB;
  const double stop = c.S[6], alpha = c.S[10], beta = c.S[11];
  if (stop != 0.0) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ S sgeo[EPB][Buf::GWD];
  __shared__ S sax[Buf::AXS ? EPB : 1][Buf::AXD];
  __shared__ int sexp[P::kScaleIO ? EPB + 1 : 1];
  Buf sm;
  sm.xs = (S *)smem_raw;
  sm.sgeo = &sgeo[0][0];
  sm.sax = &sax[0][0];
  sm.sexp = sexp;
  const int tid = threadIdx.x;
  const XCg<IO> X{c.own, c.rank, (const IO *)c.z, (const IO *)c.p, (IO *)c.pn, (IO *)c.x, (IO *)c.U, (IO)alpha, (IO)beta};
  const int64_t nblk = (E + EPB - 1) / EPB;
  IO dot = 0;
  for (int64_t blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
    const int64_t e0 = blk * EPB;
    const int nel = (int)((E - e0) < EPB ? (E - e0) : EPB);
    dot += fiber_block<P, N1, KIND, 1, false>(sm, tid, e0, nel, geo, lam, X, Y);
  }
  // sums in a fixed order: over the CTA's threads in the vectors' type, then
  // over the CTAs in double (the shared buffers are free: fiber_block ends
  // with a barrier); results in thread 0
  auto sum_cta = [&](auto v) {
    using T = decltype(v);
    T *sums = (T *)smem_raw;
    sums[tid] = v;
    __syncthreads();
    T s = 0;
    if (tid < 32) {
      for (int q = tid; q < Sh::threads; q += 32) s += sums[q];
      for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    }
    return s;
  };
  const IO mine = sum_cta(dot);
  if (tid == 0) c.part[blockIdx.x] = (double)mine;
  if (!red::arrive_last(c.cnt)) return;
  double s = 0.0;
  for (int q = tid; q < (int)gridDim.x; q += Sh::threads) s += __ldcg(c.part + q);
  const double pw = sum_cta(s);
  if (tid == 0) {
    c.S[1] = pw;
    c.S[10] = pw != 0.0 ? c.S[0] / pw : 0.0;
  }
}

// Factor export through the same geometry code: G_out [E][7][n3] float64.
template <class P, int N1, int KIND>
__global__ void __launch_bounds__(Shape<N1, 1, kEpb<P, N1, KIND>>::threads)
    factors_fiber_kernel(int64_t E, const typename P::S *__restrict__ geo, const typename P::S *__restrict__ lam,
                         double *__restrict__ G) {
  using Sh = Shape<N1, 1, kEpb<P, N1, KIND>>;
  using V = typename P::V;
  using S = typename P::S;
  constexpr int n3 = Sh::n3, EPB = Sh::EPB;
  constexpr int GW = GeoWords<KIND>::value;
  __shared__ S sgeo[EPB][GW > 0 ? GW : 1];
  const int tid = threadIdx.x;
  const int z = tid / Sh::F, q = tid % Sh::F;
  const int i = q % N1, j = q / N1;
  const int64_t e0 = (int64_t)blockIdx.x * EPB;
  const int nel = (int)((E - e0) < EPB ? (E - e0) : EPB);
  const int64_t e = e0 + z;
  const typename P::C *cw = c_w + tab_off_v(N1);
  const typename P::C *cx = c_x + tab_off_v(N1);
  if constexpr (GW > 0) {
    for (int m = tid; m < nel * GW; m += Sh::threads) sgeo[m / GW][m % GW] = geo[e0 * GW + m];
  }
  __syncthreads();
  if (z >= nel) return;
  Geometry<P, N1, KIND> gm;
  gm.prologue(sgeo[z], cx, cw, i, j, KIND == AX_GEOM_STORED ? geo + e * 7 * n3 : nullptr,
              KIND == AX_GEOM_TRILINEAR_PARTIAL ? lam + e * n3 : nullptr);
  for (int k = 0; k < N1; ++k) {
    const int l = i + j * N1 + k * N1 * N1;
    V g[6];
    const V gwj = gm.factors(l, P::cst(cx + k), P::cst(cw + k), g);
    for (int w = 0; w < 6; ++w) G[(e * 7 + w) * n3 + l] = (double)P::to_io(g[w]);
    G[(e * 7 + 6) * n3 + l] = (double)P::to_io(gwj);
  }
}

// Dynamic shared memory of a kernel of this shape.
template <class P, int N1, int KIND, int EM>
size_t launch_smem(const void *kernel) {
  using Sh = Shape<N1, EM, kEpb<P, N1, KIND>, kLayout<P, N1, KIND>>;
  const size_t smem = (size_t)3 * Sh::EPB * Sh::ES * sizeof(typename P::S);
  if constexpr (P::kTargetWarpsPerSM > 0 && N1 == 8 &&
                (KIND == AX_GEOM_TRILINEAR || KIND == AX_GEOM_TRILINEAR_PARTIAL)) {
    // cap the resident CTAs by their shared memory (the kernel uses only its share)
    int dev = 0, sm_smem = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    cudaFuncAttributes fa;
    const int static_smem = cudaFuncGetAttributes(&fa, kernel) == cudaSuccess ? (int)fa.sharedSizeBytes : 4096;
    const int warps = (Sh::threads + 31) / 32;
    int ctas = (P::kTargetWarpsPerSM + warps / 2) / warps;
    if (ctas < 1) ctas = 1;
    // per CTA: dynamic + static shared memory + the 1 KB the hardware
    // reserves, with 1 KB to spare (with none the driver chose a smaller
    // shared-memory carveout and only ctas - 1 CTAs fitted: measured)
    const size_t cap = sm_smem > 0 ? (size_t)sm_smem / ctas - (size_t)static_smem - 2048 : 0;
    if (cap > smem && cap <= 200 * 1024) return cap;
  }
  return smem;
}

template <class P, int N1, int KIND, int EM, bool LINK = false>
cudaError_t launch_ax_em(const AxArgs &a) {
  using Sh = Shape<N1, EM, kEpb<P, N1, KIND>>;
  constexpr auto kernel = [] {
    if constexpr (LINK)
      return ax_fiber_link_kernel<P, N1, KIND>;
    else
      return ax_fiber_kernel<P, N1, KIND, EM>;
  }();
  const int64_t nblk = (a.E + Sh::EPB - 1) / Sh::EPB;
  if (nblk <= 0) return cudaSuccess;
  const int64_t grid = a.grid > 0 && a.grid < nblk ? a.grid : nblk;
  if (grid > 0x7fffffffLL) return cudaErrorInvalidValue;
  static const size_t smem = launch_smem<P, N1, KIND, EM>((const void *)kernel);
  // per instantiation; static shared memory counts against the same 48 KB
  // default, so the attribute is set whatever the dynamic size
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  kernel<<<(unsigned)grid, Sh::threads, smem, a.stream>>>(
      a.E, (const typename P::S *)a.geo, (const typename P::S *)a.lam, (const typename P::IO *)a.X,
      (typename P::IO *)a.Y);
  return cudaGetLastError();
}

// The CG form (a.cg); with E = 0 the kernel is only prepared (before a
// capture).  A partial sum per CTA: at most E of them.
template <class P, int N1, int KIND>
cudaError_t launch_ax_cg(const AxArgs &a) {
  using Sh = Shape<N1, 1, kEpb<P, N1, KIND>, kLayout<P, N1, KIND>>;
  static_assert(Sh::threads >= 32 && (size_t)3 * Sh::EPB * Sh::ES * sizeof(typename P::S) >= Sh::threads * sizeof(double),
                "a whole warp and a double per thread for the sums");
  // (no cap on the resident CTAs as in launch_smem: their registers keep them
  // to five at N1 = 8, and what shared memory leaves of L1 serves the gathers:
  // double-word iterations at order 7, 4096 elements 104 -> 100 us)
  constexpr size_t smem = (size_t)3 * Sh::EPB * Sh::ES * sizeof(typename P::S);
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(ax_fiber_cg_kernel<P, N1, KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  const int64_t nblk = (a.E + Sh::EPB - 1) / Sh::EPB;
  if (nblk <= 0) return cudaSuccess;
  if (nblk > 0x7fffffffLL) return cudaErrorInvalidValue;
  ax_fiber_cg_kernel<P, N1, KIND><<<(unsigned)nblk, Sh::threads, smem, a.stream>>>(
      a.E, (const typename P::S *)a.geo, (const typename P::S *)a.lam, *a.cg, (typename P::IO *)a.Y);
  return cudaGetLastError();
}

template <class P, int N1, int KIND>
cudaError_t launch_fiber_n(const AxArgs &a, double *G_out) {
  using Sh = Shape<N1, 1, kEpb<P, N1, KIND>>;
  if (G_out) {
    const int64_t blocks = (a.E + Sh::EPB - 1) / Sh::EPB;
    if (blocks <= 0) return cudaSuccess;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    factors_fiber_kernel<P, N1, KIND><<<(unsigned)blocks, Sh::threads, 0, a.stream>>>(
        a.E, (const typename P::S *)a.geo, (const typename P::S *)a.lam, G_out);
    return cudaGetLastError();
  }
  if (a.cg) {
    if constexpr (kHasCg<P>)
      return launch_ax_cg<P, N1, KIND>(a);
    else
      return cudaErrorNotSupported;
  }
  if constexpr (kHasLink<P, N1, KIND>) {
    if (a.link) return launch_ax_em<P, N1, KIND, 1, true>(a);
  }
  if constexpr (P::kTiles > 1) {
    if (a.tile == 1) return launch_ax_em<P, N1, KIND, 2>(a);
  }
  return launch_ax_em<P, N1, KIND, 1>(a);
}

template <class P, int N1>
cudaError_t launch_fiber_kinds(const AxArgs &a, double *G_out) {
  switch (a.kind) {
    case AX_GEOM_STORED: return launch_fiber_n<P, N1, AX_GEOM_STORED>(a, G_out);
    case AX_GEOM_TRILINEAR: return launch_fiber_n<P, N1, AX_GEOM_TRILINEAR>(a, G_out);
    case AX_GEOM_PARALLELEPIPED: return launch_fiber_n<P, N1, AX_GEOM_PARALLELEPIPED>(a, G_out);
    case AX_GEOM_TRILINEAR_PARTIAL: return launch_fiber_n<P, N1, AX_GEOM_TRILINEAR_PARTIAL>(a, G_out);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace fiber
}  // namespace ax
