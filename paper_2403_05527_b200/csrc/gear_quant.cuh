// Eq. 2 on pairs of entries, shared by the kernels that hold a group in registers or shared memory.
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

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

// Bound on the residuals of a group's kept entries; it picks the powers of two that residuals are scaled by.  Half a step, or, where the
// step is subnormal in fp16 and its rounding leaves the top entries beyond the last code (up to fourteen times that; a step of
// zero: the whole range), what they lie beyond it; and the rounding of the dequantised value.
__device__ __forceinline__ float residual_bound(float mn, float mx, float range, float d, float levels) {
  return fmaxf(0.50390625f * d, fmaf(-levels, d, range)) + 2.4e-7f * (fabsf(mn) + fabsf(mx));
}

// Entry of the first set bit of L mask bits: bit t of the low / high half of word w stands for entry 2 (16 w + t) / that + 1 of
// a group whose pairs are rotated by `turn` (a multiple of four).  An entry of the group also if no bit is set (all NaN).
template <int L>
__device__ __forceinline__ int first_set(const unsigned int (&m)[4], int turn) {
  auto first = [&](unsigned int sel) {
    const unsigned int lo = __byte_perm(m[0], m[L == 32 ? 0 : 1], sel);            // 32 entries: their 16 bits twice
    if (L <= 64) return __ffs((int)__funnelshift_l(lo, lo, turn)) - 1;
    const unsigned int hi = __byte_perm(m[2], m[3], sel);
    const unsigned int l = __funnelshift_l(hi, lo, turn), h = __funnelshift_l(lo, hi, turn);
    return l ? __ffs((int)l) - 1 : h ? 32 + __ffs((int)h) - 1 : -1;
  };
  const int even = first(0x5410), odd = first(0x7632);
  return min(L - 1, min(even < 0 ? L : 2 * even, odd < 0 ? L : 2 * odd + 1));
}

// Filter_s (Eq. 4) of a group of packed pairs, at most one entry per side: the largest and the smallest entry leave the group (imax,
// imin), the second largest and second smallest instances bound what is kept (no outliers: the largest and the smallest).
// Comparisons of fp16 values are exact in fp16, so the search runs on the packed pairs: even and odd entries keep their own
// two largest / smallest and are merged at the end.  `turn`: see first_set.
// TREE: the extremes of four pairs at a time from a small sorting network, merged by twos (4.5 instead of 6 operations per
// pair); an entry that is NaN then counts as its neighbour again, which only a caller may take whose result it spoils anyway.
struct Extremes { __half2 M1, M2, m1, m2; };     // largest, second largest, smallest, second smallest of the low and of the high halves
__device__ __forceinline__ Extremes extremes_of4(__half2 a, __half2 b, __half2 c, __half2 d) {
  const __half2 t0 = __hmax2(a, b), u0 = __hmin2(a, b), t1 = __hmax2(c, d), u1 = __hmin2(c, d);
  const __half2 low = __hmin2(t0, t1), high = __hmax2(u0, u1);      // the two in the middle
  return {__hmax2(t0, t1), __hmax2(low, high), __hmin2(u0, u1), __hmin2(low, high)};
}
__device__ __forceinline__ Extremes merge(const Extremes& a, const Extremes& b) {
  return {__hmax2(a.M1, b.M1), __hmax2(__hmin2(a.M1, b.M1), __hmax2(a.M2, b.M2)),
          __hmin2(a.m1, b.m1), __hmin2(__hmax2(a.m1, b.m1), __hmin2(a.m2, b.m2))};
}
template <int L, int K, bool TREE = false>
__device__ __forceinline__ void filter_one(const __half2 (&xp)[L / 2], int turn, float& mn, float& mx, int& imax, int& imin) {
  imax = 0; imin = 1;
  const __half2 ninf = __float2half2_rn(-INFINITY), pinf = __float2half2_rn(INFINITY);
  __half2 M1 = ninf, M2 = ninf, m1 = pinf, m2 = pinf;
  if (K == 1 && TREE) {
    Extremes x = extremes_of4(xp[0], xp[1], xp[2], xp[3]);
#pragma unroll
    for (int q = 4; q < L / 2; q += 4) x = merge(x, extremes_of4(xp[q], xp[q + 1], xp[q + 2], xp[q + 3]));
    M1 = x.M1; M2 = x.M2; m1 = x.m1; m2 = x.m2;
  }
#pragma unroll
  for (int q = 0; q < (K == 1 && TREE ? 0 : L / 2); ++q) {
    if (K == 1) {
      M2 = __hmax2(M2, __hmin2(xp[q], M1));
      m2 = __hmin2(m2, __hmax2(xp[q], m1));
    }
    M1 = __hmax2(M1, xp[q]);
    m1 = __hmin2(m1, xp[q]);
  }
  const float2 fM1 = __half22float2(M1), fM2 = __half22float2(M2), fm1 = __half22float2(m1), fm2 = __half22float2(m2);
  const float max1 = fmaxf(fM1.x, fM1.y), min1 = fminf(fm1.x, fm1.y);
  mx = K == 0 ? max1 : fmaxf(fminf(fM1.x, fM1.y), fmaxf(fM2.x, fM2.y));
  mn = K == 0 ? min1 : fminf(fmaxf(fm1.x, fm1.y), fminf(fm2.x, fm2.y));
  // first index of the maximum and of the minimum (ties go to the lower index): one mask bit per entry
  if (K == 1) {
    const __half2 vM = __float2half2_rn(max1), vm = __float2half2_rn(min1);
    unsigned int a[4] = {0u, 0u, 0u, 0u}, b[4] = {0u, 0u, 0u, 0u};   // bit t of a half of word w: pair 16 w + t
#pragma unroll
    for (int q = 0; q < L / 2; ++q) {
      const unsigned int bit = 0x00010001u << (q & 15);
      a[q >> 4] |= __heq2_mask(xp[q], vM) & bit;
      b[q >> 4] |= __heq2_mask(xp[q], vm) & bit;
    }
    imax = first_set<L>(a, turn);
    imin = first_set<L>(b, turn);
    if (imin == imax) imin = 1;               // all entries equal: the bottom entry is the next index
  }
}

// PairQuant for a residual that goes on in fp16: codes as there, the residual times a power of two as an fp16 head and TWICE the
// rest as a second fp16 number.
struct PairQuantSplit {
  F32x2 neg_min, inv, scale, neg_step, neg_zero;   // the last two scaled
  float levels;
  __device__ __forceinline__ PairQuantSplit(float mn, float invs, float d, float levels_, float sr)
      : neg_min(pack2(-mn, -mn)), inv(pack2(invs, invs)), scale(pack2(sr, sr)), neg_step(pack2(-d * sr, -d * sr)),
        neg_zero(pack2(-mn * sr, -mn * sr)), levels(levels_) {}
  __device__ __forceinline__ void operator()(__half2 x, unsigned int& c0, unsigned int& c1, uint32_t& head, uint32_t& rest) const {
    const F32x2 round = pack2(12582912.0f, 12582912.0f), unround = pack2(-12582912.0f, -12582912.0f);
    const float2 xf = __half22float2(x);
    const F32x2 x2 = pack2(xf.x, xf.y);
    float2 t = unpack2(mul2(add2(x2, neg_min), inv));                // see PairQuant
    t.x = fminf(t.x, levels); t.y = fminf(t.y, levels);
    const F32x2 y2 = add2(pack2(t.x, t.y), round);
    const float2 y = unpack2(y2);
    c0 = __float_as_uint(y.x); c1 = __float_as_uint(y.y);
    const F32x2 s = fma2(x2, scale, fma2(add2(y2, unround), neg_step, neg_zero));
    const float2 sv = unpack2(s), s2 = unpack2(add2(s, s));
    const __half2 h = __floats2half2_rn(sv.x, sv.y);
    head = *reinterpret_cast<const uint32_t*>(&h);
    const __half2 l = __floats2half2_rn(minus_twice(__low2half(h), s2.x), minus_twice(__high2half(h), s2.y));
    rest = *reinterpret_cast<const uint32_t*>(&l);
  }
  // c - 2 h in one instruction
  static __device__ __forceinline__ float minus_twice(__half h, float c) {
    float r;
    asm("fma.rn.f32.f16 %0, %1, %2, %3;" : "=f"(r) : "h"(__half_as_ushort(h)), "h"((unsigned short)0xC000), "f"(c));
    return r;
  }
};

// mask of the lowest field of every byte
template <int BITS>
__device__ __forceinline__ constexpr unsigned int field_of_bytes() { return BITS == 2 ? 0x03030303u : 0x0F0F0F0Fu; }

}  // namespace gear
