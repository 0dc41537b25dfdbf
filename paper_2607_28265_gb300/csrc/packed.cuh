// FP32 arithmetic on one value (float) or a pair (f2, one 64-bit register): the
// packed forms of the Blackwell FP32 pipe do two operations per instruction.
#pragma once

#include <cuda_runtime.h>

namespace swig {

using f2 = unsigned long long;
__device__ __forceinline__ f2 f2_make(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f2_split(f2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// The same operations by element type: PkOps<1> on float, PkOps<2> on f2.
template <int N>
struct PkOps;
template <>
struct PkOps<1> {
  using T = float;
  __device__ static __forceinline__ T all(float a) { return a; }
  __device__ static __forceinline__ T load(const float* p) { return *p; }
  __device__ static __forceinline__ T add(T a, T b) { return __fadd_rn(a, b); }
  __device__ static __forceinline__ T mul(T a, T b) { return __fmul_rn(a, b); }
  __device__ static __forceinline__ T fma(T a, T b, T c) { return __fmaf_rn(a, b, c); }
  __device__ static __forceinline__ void get(T v, float* o) { o[0] = v; }
  __device__ static __forceinline__ T set(const float* o) { return o[0]; }
};
template <>
struct PkOps<2> {
  using T = f2;
  __device__ static __forceinline__ T all(float a) { return f2_make(a, a); }
  __device__ static __forceinline__ T load(const float* p) { return *reinterpret_cast<const f2*>(p); }
  __device__ static __forceinline__ T add(T a, T b) { return f2_add(a, b); }
  __device__ static __forceinline__ T mul(T a, T b) { return f2_mul(a, b); }
  __device__ static __forceinline__ T fma(T a, T b, T c) { return f2_fma(a, b, c); }
  __device__ static __forceinline__ void get(T v, float* o) { f2_split(v, o[0], o[1]); }
  __device__ static __forceinline__ T set(const float* o) { return f2_make(o[0], o[1]); }
};

// Double-float arithmetic (device_common.cuh two_sum, df_mul, df_add) on N
// values at once; the subtractions are multiply-adds by -1, which round alike.
template <int N>
struct DflN {
  typename PkOps<N>::T hi, lo;
};
template <int N>
__device__ __forceinline__ typename PkOps<N>::T pk_sub(typename PkOps<N>::T a, typename PkOps<N>::T b) {
  return PkOps<N>::fma(b, PkOps<N>::all(-1.0f), a);
}
template <int N>
__device__ __forceinline__ DflN<N> dfn_fast_two_sum(typename PkOps<N>::T a, typename PkOps<N>::T b) {
  using O = PkOps<N>;
  const auto s = O::add(a, b);
  return {s, pk_sub<N>(b, pk_sub<N>(s, a))};
}
template <int N>
__device__ __forceinline__ DflN<N> dfn_mul(DflN<N> a, DflN<N> b) {
  using O = PkOps<N>;
  const auto p = O::mul(a.hi, b.hi);
  auto e = O::fma(a.hi, b.hi, O::mul(p, O::all(-1.0f)));
  e = O::fma(a.hi, b.lo, e);
  e = O::fma(a.lo, b.hi, e);
  return dfn_fast_two_sum<N>(p, e);
}
template <int N>
__device__ __forceinline__ DflN<N> dfn_add(DflN<N> a, DflN<N> b) {
  using O = PkOps<N>;
  const auto s = O::add(a.hi, b.hi);
  const auto bb = pk_sub<N>(s, a.hi);
  const auto t = O::add(pk_sub<N>(a.hi, pk_sub<N>(s, bb)), pk_sub<N>(b.hi, bb));
  return dfn_fast_two_sum<N>(s, O::add(t, O::add(a.lo, b.lo)));
}
// The fractional part (nearest integer removed) of each value; |hi| < 2^22.
template <int N>
__device__ __forceinline__ typename PkOps<N>::T dfn_frac(DflN<N> a) {
  using O = PkOps<N>;
  const auto n = O::add(O::add(a.hi, O::all(12582912.0f)), O::all(-12582912.0f));
  return O::add(pk_sub<N>(a.hi, n), a.lo);
}

// One level of the halving reduction of 2 O per-lane values: lanes with bit O
// set keep the upper O values, the others the lower O, each adding its
// partner's copy of them.
template <int O>
__device__ __forceinline__ void warp_halve(float* a, int lane) {
  const bool up = (lane & O) != 0;
#pragma unroll
  for (int k = 0; k < O; ++k) {
    const float s = up ? a[k] : a[k + O], m = up ? a[k + O] : a[k];
    a[k] = m + __shfl_xor_sync(0xffffffffu, s, O);
  }
}
// 32 values per lane -> lane l returns the warp sum of value l (31 shuffles).
__device__ __forceinline__ float warp_transpose_sum(float* a, int lane) {
  warp_halve<16>(a, lane);
  warp_halve<8>(a, lane);
  warp_halve<4>(a, lane);
  warp_halve<2>(a, lane);
  warp_halve<1>(a, lane);
  return a[0];
}

}  // namespace swig
