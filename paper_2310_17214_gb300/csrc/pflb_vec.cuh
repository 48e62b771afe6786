// pflb_vec.cuh -- the arithmetic of the per-cell update over one cell (float
// or double) or over two cells that are neighbours in x (float2, the packed
// f32x2 instructions of sm_100 and later: one issue slot for two cells).
//
// Every operation is written out (add, mul, fma with one rounding each), so
// that the compiler has no multiply-add contraction to choose and all kernels
// that share the update round alike: a cell's result is the same bits whether
// it is updated alone, as either half of a pair, or under any tile shape.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace pflb {

// FP32 uses the fast hardware approximations (a few ulp); FP64 stays IEEE.
__device__ __forceinline__ float fdiv(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double fdiv(double a, double b) { return a / b; }
__device__ __forceinline__ float fexp(float x) { return __expf(x); }
__device__ __forceinline__ double fexp(double x) { return exp(x); }
__device__ __forceinline__ float fpow(float x, float y) { return __powf(x, y); }
__device__ __forceinline__ double fpow(double x, double y) { return pow(x, y); }
__device__ __forceinline__ float fsqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double fsqrt(double x) { return sqrt(x); }

__device__ __forceinline__ uint64_t f2_bits(float2 v) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(v.x), "f"(v.y));
  return r;
}
__device__ __forceinline__ float2 f2_of(uint64_t r) {
  float2 v;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(r));
  return v;
}

// Lanes: number of cells, scalar type, mask type (one truth value per cell).
template <class V> struct Lanes;
template <> struct Lanes<float> { using S = float; using M = bool; static constexpr int n = 1; };
template <> struct Lanes<double> { using S = double; using M = bool; static constexpr int n = 1; };
struct bool2x { bool x, y; };
template <> struct Lanes<float2> { using S = float; using M = bool2x; static constexpr int n = 2; };

template <class V> __device__ __forceinline__ V splat(typename Lanes<V>::S a);
template <> __device__ __forceinline__ float splat<float>(float a) { return a; }
template <> __device__ __forceinline__ double splat<double>(double a) { return a; }
template <> __device__ __forceinline__ float2 splat<float2>(float a) { return make_float2(a, a); }

__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double vadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double vsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double vmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) {
  uint64_t d;
  asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2_bits(a)), "l"(f2_bits(b)));
  return f2_of(d);
}
__device__ __forceinline__ float2 vsub(float2 a, float2 b) {
  uint64_t d;
  asm("sub.rn.ftz.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2_bits(a)), "l"(f2_bits(b)));
  return f2_of(d);
}
__device__ __forceinline__ float2 vmul(float2 a, float2 b) {
  uint64_t d;
  asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2_bits(a)), "l"(f2_bits(b)));
  return f2_of(d);
}
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) {
  uint64_t d;
  asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(f2_bits(a)), "l"(f2_bits(b)),
      "l"(f2_bits(c)));
  return f2_of(d);
}
__device__ __forceinline__ float vneg(float a) { return -a; }
__device__ __forceinline__ double vneg(double a) { return -a; }
__device__ __forceinline__ float2 vneg(float2 a) { return make_float2(-a.x, -a.y); }

// with a scalar of the compute type
template <class V> __device__ __forceinline__ V vmuls(typename Lanes<V>::S s, V a) {
  return vmul(splat<V>(s), a);
}
template <class V> __device__ __forceinline__ V vfmas(typename Lanes<V>::S s, V a, V c) {
  return vfma(splat<V>(s), a, c);
}
template <class V> __device__ __forceinline__ V vadds(typename Lanes<V>::S s, V a) {
  return vadd(splat<V>(s), a);
}

__device__ __forceinline__ float2 fdiv(float2 a, float2 b) {
  return make_float2(fdiv(a.x, b.x), fdiv(a.y, b.y));
}
__device__ __forceinline__ float2 fexp(float2 a) { return make_float2(fexp(a.x), fexp(a.y)); }
__device__ __forceinline__ float2 fpow(float2 a, float b) {
  return make_float2(fpow(a.x, b), fpow(a.y, b));
}
__device__ __forceinline__ float2 fsqrt(float2 a) { return make_float2(fsqrt(a.x), fsqrt(a.y)); }
template <class V> __device__ __forceinline__ V vrcp(V a) {
  return fdiv(splat<V>(typename Lanes<V>::S(1)), a);
}

__device__ __forceinline__ bool vgt(float a, float b) { return a > b; }
__device__ __forceinline__ bool vgt(double a, double b) { return a > b; }
__device__ __forceinline__ bool2x vgt(float2 a, float2 b) { return {a.x > b.x, a.y > b.y}; }
__device__ __forceinline__ bool vge(float a, float b) { return a >= b; }
__device__ __forceinline__ bool vge(double a, double b) { return a >= b; }
__device__ __forceinline__ bool2x vge(float2 a, float2 b) { return {a.x >= b.x, a.y >= b.y}; }
__device__ __forceinline__ bool vany(bool a) { return a; }
__device__ __forceinline__ bool vany(bool2x a) { return a.x || a.y; }
__device__ __forceinline__ float vsel(bool m, float a, float b) { return m ? a : b; }
__device__ __forceinline__ double vsel(bool m, double a, double b) { return m ? a : b; }
__device__ __forceinline__ float2 vsel(bool2x m, float2 a, float2 b) {
  return make_float2(m.x ? a.x : b.x, m.y ? a.y : b.y);
}

// lane access (l is a compile-time constant where the caller unrolls)
__device__ __forceinline__ float get_lane(float a, int) { return a; }
__device__ __forceinline__ double get_lane(double a, int) { return a; }
__device__ __forceinline__ float get_lane(float2 a, int l) { return l == 0 ? a.x : a.y; }
__device__ __forceinline__ void set_lane(float& a, int, float v) { a = v; }
__device__ __forceinline__ void set_lane(double& a, int, double v) { a = v; }
__device__ __forceinline__ void set_lane(float2& a, int l, float v) {
  if (l == 0) a.x = v;
  else a.y = v;
}

}  // namespace pflb
