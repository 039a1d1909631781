// FP32 pairs: the f32x2 instructions (two lanes per issue slot; each lane
// rounds exactly like the scalar instruction) as functions on float2, and as
// the arithmetic type F2, which the lattice's collision templates take in
// the place of float, so that a pair of nodes is collided by the same
// sequence of operations as one node.
#pragma once

#include <stdint.h>

#include <type_traits>

namespace mdf {

__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }

#define MDF_F32X2_BINARY(name, op)                                                              \
  __device__ __forceinline__ float2 name(float2 a, float2 b) {                                  \
    float2 r;                                                                                   \
    asm("{\n .reg .b64 a, b, d;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n " op           \
        " d, a, b;\n mov.b64 {%0, %1}, d;\n}\n"                                                 \
        : "=f"(r.x), "=f"(r.y)                                                                  \
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));                                              \
    return r;                                                                                   \
  }
MDF_F32X2_BINARY(vadd, "add.rn.f32x2")
MDF_F32X2_BINARY(vsub, "sub.rn.f32x2")
MDF_F32X2_BINARY(vmul, "mul.rn.f32x2")
#undef MDF_F32X2_BINARY
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) {
  float2 r;
  asm("{\n .reg .b64 a, b, c, d;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n"
      " mov.b64 c, {%6, %7};\n fma.rn.f32x2 d, a, b, c;\n mov.b64 {%0, %1}, d;\n}\n"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return r;
}


// Two FP32 lanes (two x-adjacent nodes).
struct F2 {
  float x, y;
  F2() = default;
  __device__ __forceinline__ F2(float a, float b) : x(a), y(b) {}
  explicit __device__ __forceinline__ F2(float2 v) : x(v.x), y(v.y) {}
  explicit __device__ __forceinline__ F2(double c) : x((float)c), y((float)c) {}
  __device__ __forceinline__ float2 f2() const { return make_float2(x, y); }
};
__device__ __forceinline__ F2 operator+(F2 a, F2 b) { return F2(vadd(a.f2(), b.f2())); }
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return F2(vsub(a.f2(), b.f2())); }
// Constants of the collision.
enum Lit { LIT_2_3, LIT_3_4, LIT_M4, LIT_M6, LIT_1_20, LIT_1_5, LIT_1_42, LIT_1_7, LIT_1_6, LIT_1_2,
           LIT_1, LIT_1_4, LIT_1_3, LIT_1_12, LITS };
constexpr double kLit[LITS] = {2.0 / 3.0,  0.75,      -4.0, -6.0, 0.05, 0.2, 1.0 / 42.0, 1.0 / 7.0, 1.0 / 6.0,
                               0.5,        1.0,       0.25, 1.0 / 3.0, 1.0 / 12.0};
template <class T, Lit K> __device__ __forceinline__ T lit() {
  constexpr double v = kLit[K];
  return T(v);
}
// A product is two scalar ones.  A sum of a mul.rn.f32x2 and another value was
// compiled into one fused f32x2 operation (measured: other bits than mul and
// add, also with -fmad=false), and the scalar kernels, whose bits these must
// be, round the product.  The f32x2 forms take two slots of the FP32 pipe, so
// a pair of scalar products costs it nothing more, and most of them multiply
// by an immediate.  (As a f32x2 fma with -0 and with the constants, both read
// from constant memory: 158 us per update at 4096^2 against 152; the dither's
// FMAs as scalar ones too: 148.)
__device__ __forceinline__ F2 operator*(F2 a, F2 b) { return F2(__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y)); }
// b + c a for a power of two c: the product is exact, so one rounding either way
template <Lit K, class T> __device__ __forceinline__ T add_scaled(T b, T a) {
  constexpr float c = (float)kLit[K];
  if constexpr (std::is_same<T, F2>::value) return F2(vfma(a.f2(), make_float2(c, c), b.f2()));
  else return b + lit<T, K>() * a;
}
__device__ __forceinline__ F2 operator-(F2 a) { return F2(-a.x, -a.y); }
__device__ __forceinline__ F2 &operator+=(F2 &a, F2 b) { a = a + b; return a; }

// The absent body force: the terms it enters drop out at compile time.
struct NoForce {};
template <class T> __device__ __forceinline__ NoForce operator*(NoForce, T) { return {}; }
template <class T> __device__ __forceinline__ T operator+(T a, NoForce) { return a; }
template <class T> __device__ __forceinline__ T operator+(NoForce, T a) { return a; }
// 0 - a, not yet formed: (0 - a) + b is b - a in one operation
template <class T> struct Negated { T a; };
template <class T> __device__ __forceinline__ Negated<T> operator-(NoForce, T a) { return {a}; }
template <class T> __device__ __forceinline__ T operator+(Negated<T> n, T b) { return b - n.a; }
template <class T> __device__ __forceinline__ T operator-(Negated<T> n, T b) { return (T(0) - n.a) - b; }

}  // namespace mdf
