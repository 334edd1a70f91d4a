// One or two FP32 values per thread with the same source: Vf<2> uses the
// packed instructions of sm_100+ (one issue slot for two lanes' worth of work;
// each half is the IEEE operation, so values are those of the scalar forms).
// Every operation is rounded as written: none is contracted by the compiler.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace srw {

__device__ __forceinline__ uint64_t pk(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpk(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

template <int N>
struct Vf;
template <>
struct Vf<1> {
  float v;
  __device__ __forceinline__ static Vf dup(float x) { return {x}; }
  __device__ __forceinline__ static Vf of(const float* x) { return {x[0]}; }
  __device__ __forceinline__ void to(float* x) const { x[0] = v; }
};
template <>
struct Vf<2> {
  uint64_t v;
  __device__ __forceinline__ static Vf dup(float x) { return {pk(x, x)}; }
  __device__ __forceinline__ static Vf of(const float* x) { return {pk(x[0], x[1])}; }
  __device__ __forceinline__ void to(float* x) const {
    const float2 t = unpk(v);
    x[0] = t.x;
    x[1] = t.y;
  }
};

__device__ __forceinline__ Vf<1> vfma(Vf<1> a, Vf<1> b, Vf<1> c) { return {__fmaf_rn(a.v, b.v, c.v)}; }
__device__ __forceinline__ Vf<1> vmul(Vf<1> a, Vf<1> b) { return {__fmul_rn(a.v, b.v)}; }
__device__ __forceinline__ Vf<1> vadd(Vf<1> a, Vf<1> b) { return {__fadd_rn(a.v, b.v)}; }
__device__ __forceinline__ Vf<1> vsub(Vf<1> a, Vf<1> b) { return {__fsub_rn(a.v, b.v)}; }
__device__ __forceinline__ Vf<2> vfma(Vf<2> a, Vf<2> b, Vf<2> c) { return {fma2(a.v, b.v, c.v)}; }
__device__ __forceinline__ Vf<2> vmul(Vf<2> a, Vf<2> b) { return {mul2(a.v, b.v)}; }
__device__ __forceinline__ Vf<2> vadd(Vf<2> a, Vf<2> b) { return {add2(a.v, b.v)}; }
__device__ __forceinline__ Vf<2> vsub(Vf<2> a, Vf<2> b) { return {sub2(a.v, b.v)}; }

}  // namespace srw
