// Eq. 2 on pairs of entries, shared by the kernels that hold a group in registers or shared memory.
#pragma once
#include <cuda_fp16.h>

namespace gear {

// pairs of binary32 operations, each rounded like the scalar one
struct F32x2 { unsigned long long v; };
__device__ __forceinline__ F32x2 pack2(float x, float y) {
  F32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float2 unpack2(F32x2 a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
  return r;
}
__device__ __forceinline__ F32x2 add2(F32x2 a, F32x2 b) { F32x2 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r; }
__device__ __forceinline__ F32x2 mul2(F32x2 a, F32x2 b) { F32x2 r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r; }
__device__ __forceinline__ F32x2 fma2(F32x2 a, F32x2 b, F32x2 c) {
  F32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ void store8(float* dst, const float2 (&r)[4]) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "f"(r[0].x), "f"(r[0].y), "f"(r[1].x),
               "f"(r[1].y), "f"(r[2].x), "f"(r[2].y), "f"(r[3].x), "f"(r[3].y) : "memory");
}

// Eq. 2 for a pair of entries of one group: t = (x - min) * inv, code = round-to-nearest-even of t by adding 1.5 * 2^23 (the
// low byte of the sum), residual x - (code * step + min).  Kept entries have t >= 0; t can exceed the top level where the
// step is subnormal in fp16.  The filtered entries come out as anything and are cleared by the caller.
struct PairQuant {
  F32x2 neg_min, inv, neg_step;
  float levels;
  __device__ __forceinline__ PairQuant(float mn, float invs, float d, float levels_)
      : neg_min(pack2(-mn, -mn)), inv(pack2(invs, invs)), neg_step(pack2(-d, -d)), levels(levels_) {}
  __device__ __forceinline__ float2 operator()(float2 x, unsigned int& c0, unsigned int& c1) const {
    const F32x2 round = pack2(12582912.0f, 12582912.0f), unround = pack2(-12582912.0f, -12582912.0f);
    const F32x2 x2 = pack2(x.x, x.y);
    // The bound between the product and the sum also keeps the compiler from contracting the two packed operations into one
    // fused one, which would not round the product: the two results differ where a value lies half way between two codes.
    float2 t = unpack2(mul2(add2(x2, neg_min), inv));
    t.x = fminf(t.x, levels); t.y = fminf(t.y, levels);
    const F32x2 y2 = add2(pack2(t.x, t.y), round);
    const float2 y = unpack2(y2);
    c0 = __float_as_uint(y.x); c1 = __float_as_uint(y.y);            // the code is the low byte
    return unpack2(add2(x2, fma2(add2(y2, unround), neg_step, neg_min)));
  }
};

}  // namespace gear
