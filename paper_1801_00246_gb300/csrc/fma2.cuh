// Products of one operator entry with several elements' values, two FP32
// multiply-adds to an instruction (fma.f32x2: each lane rounds as fmaf does).
#pragma once
#include <cstdint>

namespace dgx {

__device__ __forceinline__ uint64_t twice(float a) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
  return r;
}
// (x0, x1) += a (w0, w1), a from twice()
__device__ __forceinline__ void fma2(float& x0, float& x1, uint64_t a, float w0, float w1) {
  uint64_t x, w;
  asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(x0), "f"(x1));
  asm("mov.b64 %0, {%1, %2};" : "=l"(w) : "f"(w0), "f"(w1));
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(x) : "l"(a), "l"(w));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x0), "=f"(x1) : "l"(x));
}
// x[e] += a w[e]
template <int G>
__device__ __forceinline__ void fma_vec(float (&x)[G], float a, const float (&w)[G]) {
  const uint64_t aa = twice(a);
#pragma unroll
  for (int e = 0; e < G; e += 2) fma2(x[e], x[e + 1], aa, w[e], w[e + 1]);
}
// G values at a 16-byte aligned address
template <int G>
__device__ __forceinline__ void load_vec(float (&w)[G], const float* p) {
#pragma unroll
  for (int q = 0; q < G; q += 4) {
    const float4 v = *reinterpret_cast<const float4*>(p + q);
    w[q] = v.x, w[q + 1] = v.y, w[q + 2] = v.z, w[q + 3] = v.w;
  }
}
template <int G>
__device__ __forceinline__ void store_vec(float* p, const float (&x)[G]) {
#pragma unroll
  for (int q = 0; q < G; q += 4) *reinterpret_cast<float4*>(p + q) = make_float4(x[q], x[q + 1], x[q + 2], x[q + 3]);
}

}  // namespace dgx
