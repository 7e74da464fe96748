// Device helpers shared by the kernels of Algorithm 2.
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

#include "gear_internal.cuh"

namespace gear {

// ------------------------------------------------------------------ bulk copies and barriers
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(uint64_t* b, int count = 1) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(b)) : "memory");
}
// bounded: false when the phase did not complete within the limit
__device__ __forceinline__ bool bar_wait(uint64_t* b, uint32_t parity, int limit = kDecodeSpinLimit) {
  uint32_t ok = 0;
#pragma unroll 1
  for (int i = 0; i < limit && !ok; ++i)
    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\nselp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok) : "r"(smem_addr(b)), "r"(parity), "r"(kWaitHintNs) : "memory");
  return ok != 0;
}
__device__ __forceinline__ void bar_expect(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, uint32_t bytes, uint64_t* b) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(b)) : "memory");
}

// ------------------------------------------------------------------ numbers

// floor(log2 |x|) for a finite x > 0 (0 for x == 0): the power of two that brings x into [1, 2)
__device__ __forceinline__ int pow2_exponent(float x) { return x > 0.f ? ilogbf(x) : 0; }
__device__ __forceinline__ float exp2_int(int e) { return scalbnf(1.0f, e); }
// (x0, x1) -> packed fp16 heads and packed fp16 remainders (x - head, exact in fp32 before its own rounding)
__device__ __forceinline__ void split_pair(float x0, float x1, uint32_t& hi, uint32_t& lo) {
  const __half2 h = __floats2half2_rn(x0, x1);
  const float2 hf = __half22float2(h);
  const __half2 l = __floats2half2_rn(x0 - hf.x, x1 - hf.y);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Counter-based Gaussian for library-drawn start vectors (splitmix64 + Box-Muller).
__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
// entry (channel ch, column rho) of the start matrix of tile gtile = 2 (batch, head) + side
__device__ __forceinline__ float start_value(unsigned long long seed, int segment, size_t gtile, int ch, int rho) {
  const unsigned long long h = mix64(seed ^ mix64(((unsigned long long)segment << 40) ^ (gtile * 4096ull + ch * 16 + rho)));
  const float u1 = ((float)(unsigned int)(h >> 40) + 1.0f) * (1.0f / 16777217.0f);
  const float u2 = (float)(unsigned int)((h >> 8) & 0xFFFFFFu) * (1.0f / 16777216.0f);
  return sqrtf(-2.0f * logf(u1)) * cospif(2.0f * u2);
}

// W = U^-1 of the Cholesky factor G = U^T U of the r x r Gram matrix G, by one warp: lane c holds column c of U, then of
// U^-1 (a chain of r steps with shuffles; one lane alone takes r^3 / 3).  G and W in shared memory, rows `pitch` apart.
// FLOOR = true (scaling a factor that has not been computed yet): a pivot below 1e-6 of the trace is rounding of G as much
// as it is the column, so the column is scaled by that floor and nothing is eliminated with it; FLOOR = false (columns of
// norm about one, or shorter where the floor was used): a column below 1e-6, i.e. below 1e-12 of the trace of the
// unscaled factor, is zeroed.  Returns whether a pivot lies below a thousandth of the largest diagonal entry.
template <int RP, bool FLOOR>
__device__ __forceinline__ bool warp_chol_inverse(const float* G, float* W, int pitch, int r, int lane) {
  float u[RP], x[RP];
  const int c = lane < RP ? lane : 0;
#pragma unroll
  for (int k = 0; k < RP; ++k) u[k] = lane < r && k < r ? G[k * pitch + c] : 0.f;
  float low = 1e-6f, diag = 0.f;
#pragma unroll
  for (int k = 0; k < RP; ++k) diag = lane == k ? u[k] : diag;
  const float dmax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(diag, 0.f))));
  bool small = false;
  if (FLOOR) {
    low = 1e-6f * warp_sum(diag);
    if (!(low > 0.f)) low = 1.f;                   // a residual of zeros: no scaling
  }
#pragma unroll
  for (int j = 0; j < RP; ++j) {
    const float d = __shfl_sync(0xffffffffu, u[j], j);
    const bool good = d > low;
    small = small || (j < r && d < 1e-3f * dmax);
    const float ujj = j >= r ? 0.f : (good ? sqrtf(d) : (FLOOR ? sqrtf(low) : 0.f));
    const float ujc = lane == j ? ujj : (lane > j && good ? u[j] / ujj : 0.f);
    u[j] = ujc;
#pragma unroll
    for (int k = j + 1; k < RP; ++k) u[k] = fmaf(-__shfl_sync(0xffffffffu, ujc, k), ujc, u[k]);
  }
#pragma unroll
  for (int i = RP - 1; i >= 0; --i) {
    float s = i == lane ? 1.f : 0.f;
#pragma unroll
    for (int k = i + 1; k < RP; ++k) s = fmaf(-__shfl_sync(0xffffffffu, u[i], k), x[k], s);
    const float uii = __shfl_sync(0xffffffffu, u[i], i);
    x[i] = i <= lane && uii != 0.f ? s / uii : 0.f;
  }
  if (lane < RP) {
#pragma unroll
    for (int k = 0; k < RP; ++k) W[k * pitch + lane] = x[k];
  }
  __syncwarp();
  return small;
}

}  // namespace gear
