// mqo_x16.cuh -- pairs of 16-bit x in one 32-bit word, for the step kernels that
// work on whole words (mqo_step_dense.cu, mqo_step_rows.cu).
#pragma once

#include "mqo_dev.cuh"

namespace mqo {

template <typename TX>
struct X16;
template <>
struct X16<__nv_bfloat16> {
  using T2 = __nv_bfloat162;
  static constexpr uint32_t kType = 1u;  // operand type in the instruction descriptor
  static constexpr bool kScaled = true;
  static constexpr uint32_t kHalf = 0x3F00u, kTwo9 = 0x4400u, kTwo13 = 0x4600u;
  __device__ __forceinline__ static T2 splat(float f) { return __float2bfloat162_rn(f); }
  __device__ __forceinline__ static void add(float& a, float& b, uint32_t w) { add_bf16x2_word(a, b, w); }
  __device__ __forceinline__ static void unpack(uint32_t w, float& a, float& b) {
    a = __uint_as_float(w << 16);
    b = __uint_as_float(w & 0xffff0000u);
  }
  __device__ __forceinline__ static uint32_t pack(float a, float b) {
    const T2 r = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&r);
  }
};
template <>
struct X16<__half> {
  using T2 = __half2;
  static constexpr uint32_t kType = 0u;
  static constexpr bool kScaled = false;
  static constexpr uint32_t kHalf = 0x3800u, kTwo9 = 0x6000u, kTwo13 = 0x7000u;
  __device__ __forceinline__ static T2 splat(float f) { return __float2half2_rn(f); }
  __device__ __forceinline__ static void add(float& a, float& b, uint32_t w) {
    float x, y;
    unpack(w, x, y);
    a = a + x;
    b = b + y;
  }
  __device__ __forceinline__ static void unpack(uint32_t w, float& a, float& b) {
    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w));
    a = f.x;
    b = f.y;
  }
  __device__ __forceinline__ static uint32_t pack(float a, float b) {
    const T2 r = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&r);
  }
};
template <typename T2>
__device__ __forceinline__ T2 as2(uint32_t w) {
  return *reinterpret_cast<const T2*>(&w);
}
// (a, b) *= (x, y).  Sums of such products are taken with scalar adds: ptxas
// contracts a packed multiply and a packed add into a packed multiply-add
__device__ __forceinline__ void mul2(float& a, float& b, float x, float y) {
  asm("{\n\t.reg .b64 p, q;\n\t"
      "mov.b64 p, {%0, %1};\n\t"
      "mov.b64 q, {%2, %3};\n\t"
      "mul.rn.f32x2 p, p, q;\n\t"
      "mov.b64 {%0, %1}, p;\n\t}"
      : "+f"(a), "+f"(b)
      : "f"(x), "f"(y));
}

}  // namespace mqo
