// Device helpers and block shapes shared by the decode kernels (one query head per warp: gear_decode.cu; grouped query
// rows: gear_decode_rows.cu).
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "gear_internal.cuh"

namespace gear {

constexpr int kBufPitch = 272;                  // bytes per fp16 row of a buffer slab in shared memory
constexpr int kFragKRow = 40;                   // 32-bit words per (head, limb) row of the key B-operand staging area
constexpr int kTokLimit = 16384;                // tokens a value accumulator takes before it is folded (int32 headroom)
// Bits of the value fixed point kept free for a lagging running maximum: the one that its unsigned digits have more than the
// signed ones of the keys, so that a probability of one keeps 22 bits.  (With two, 20 bits are left, and a value is up to
// 9e-5 off where a block holds one large score and many that are 2^-18 to 2^-22 of it; without the lag batch 8 x 32 heads
// x 4096, 2 bits, takes 157.3 instead of 155.5 us for four layers.)
constexpr int kLag = 1;
constexpr float kMagic = 12582912.0f;           // 1.5 * 2^23: x + kMagic carries rint(x) in its low mantissa bits, |x| < 2^22
constexpr uint32_t kMagicBits = 0x4B400000u;
constexpr float kMagicV = 8388608.0f;           // 2^23: the same for 0 <= x < 2^23; the low three bytes of the sum are the digits of rint(x)


// ------------------------------------------------------------------ PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* b, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* b) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(b))
               : "memory");
}
// The hardware may suspend the warp for up to kWaitHintNs instead of coming back empty-handed at once: a poll costs eight
// instructions, and warps that wait for a copy took a quarter of the issue slots with them.
__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\nselp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(b)), "r"(parity), "r"(kWaitHintNs)
      : "memory");
  return ok != 0;
}
// Bounded wait: gives up after `limit` polls and reports through `status`.
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, int limit, int* status) {
#pragma unroll 1
  for (int i = 0; i < limit; ++i)
    if (mbar_try(b, parity)) return true;
  atomicExch(status, -7 /* GEAR_ERR_TIMEOUT */);
  return false;
}
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// d = a * b (no accumulator input)
__device__ __forceinline__ void mma16816_z(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  const float z = 0.f;
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(z));
}
// integer products: A unsigned bytes (codes in place), B signed (imma16832, keys) or unsigned bytes (imma16832_u, values),
// 32-bit sums
__device__ __forceinline__ void imma16832(int (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void imma16832_u(int (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k32.row.col.s32.u8.u8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_u32(p)));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_u32(p)));
}
__device__ __forceinline__ uint32_t h2_as_u32(__half2 h) { return *reinterpret_cast<uint32_t*>(&h); }
__device__ __forceinline__ __half2 u32_as_h2(uint32_t u) { return *reinterpret_cast<__half2*>(&u); }

// mask of field j of every byte of a word of packed codes
template <int BITS>
__host__ __device__ constexpr uint32_t field_mask(int j) {
  return BITS == 2 ? (0x03030303u << (2 * j)) : (0x0F0F0F0Fu << (4 * j));
}
// fp32 pair -> half2 of the high parts and half2 of the rounding remainders
__device__ __forceinline__ void split_hi_lo(float x0, float x1, uint32_t& hi, uint32_t& lo) {
  const __half2 h = __floats2half2_rn(x0, x1);
  hi = h2_as_u32(h);
  lo = h2_as_u32(__floats2half2_rn(x0 - __low2float(h), x1 - __high2float(h)));
}

// maximum over the warp in one instruction (by five shuffles: one head of 256 tokens 6.46 us instead of 6.34, 32 layers of one sequence
// 347.4 instead of 343.3, 200 steps of a request of two layers 4438 instead of 4390)
__device__ __forceinline__ float warp_max(float x) {
  float r;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ uint32_t warp_max_u32(uint32_t x) { return __reduce_max_sync(0xffffffffu, x); }
__device__ __forceinline__ int float_exponent(float x) { return (int)((__float_as_uint(x) >> 23) & 0xFFu) - 127; }
// 2^x for x <= 0 (scores minus a maximum): one instruction, relative error about 2^-22, flushes tiny results to zero
__device__ __forceinline__ float exp2_fast(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// 2^e for |e| <= 120
__device__ __forceinline__ float pow2i(int e) { return __uint_as_float((uint32_t)(127 + e) << 23); }
__device__ __forceinline__ int clamp60(int e) { return max(-60, min(60, e)); }

// ------------------------------------------------------------------ block shapes
// The work on a block depends on its shape: tokens T, outliers per key group, padded rank, outliers per value
// group.  The shapes of the usual configurations are compile-time constants (every offset inside the record becomes
// an immediate and the loops unroll); any other segment runs through the same code with run-time values.
struct DynShape {                      // values read from the segment descriptor
  static constexpr bool kDyn = true, kCsr = true;     // kCsr: the segment may keep its key outliers in a list
  static constexpr int T = 0, k2k = 0, r_pad = 0, k2v = 0, unroll = 1;
  static constexpr int off_kscale = 0, off_koval = 0, off_koidx = 0, off_kcodes = 0, off_ak = 0, off_av = 0, off_vscale = 0,
                       off_voval = 0, off_voidx = 0;
};
template <int BITS, int NGV, int T_, int KK, int RP, int KV, bool CSR = false>
struct StaticShape {                   // mirrors layout_segment(); checked against it on the host (static_shape_id)
  static constexpr bool kDyn = false, kCsr = CSR;
  static constexpr int T = T_, k2k = 2 * KK, r_pad = RP, k2v = 2 * KV, unroll = 2;
  static constexpr int nslab = T_ / kSlab, slab_codes = kSlab * kHeadDim * BITS / 8, nchunk = (T_ + 31) / 32;
  static constexpr int off_kscale = kRecHeader;
  static constexpr int off_koval = off_kscale + kHeadDim * 4;
  static constexpr int off_koidx = off_koval + kHeadDim * 2 * KK * 2;
  static constexpr int off_kcodes = off_koidx + (kHeadDim * 2 * KK + 15) / 16 * 16;
  static constexpr int off_ak = off_kcodes + nslab * slab_codes;
  static constexpr int off_vpart = off_ak + (nslab * kSlab * RP * 2 + 15) / 16 * 16;
  // value part, relative to its start
  static constexpr int off_av = nchunk * 2 * slab_codes;
  static constexpr int off_vscale = off_av + (nslab * kSlab * RP * 2 + 15) / 16 * 16;
  static constexpr int off_voval = off_vscale + T_ * NGV * 4;
  static constexpr int off_voidx = off_voval + (T_ * NGV * 2 * KV * 2 + 15) / 16 * 16;
  static constexpr int rec_bytes = off_vpart + off_voidx + (T_ * NGV * 2 * KV + 15) / 16 * 16;
  static bool matches(const SegDesc& s, const CacheConst& c) {
    return c.bits == BITS && c.ngv == NGV && c.k_v == KV && s.T == T_ && s.k_k == KK && s.r_pad == RP &&
           (s.csr_base16 != 0) == CSR &&
           s.off_kscale == off_kscale && s.off_koval == off_koval && s.off_koidx == off_koidx &&
           s.off_kcodes == off_kcodes && s.off_ak == off_ak && s.off_vpart == off_vpart &&
           s.off_vcodes == off_vpart && s.off_av == off_vpart + off_av && s.off_vscale == off_vpart + off_vscale &&
           s.off_voval == off_vpart + off_voval && s.off_voidx == off_vpart + off_voidx && s.rec_bytes == rec_bytes;
  }
};
// static shapes by id (0 = none).  Two value groups per token (g = 64): ids 1, 2; one group (g = 128): ids 3, 4.
template <int BITS> using ShapeA1 = StaticShape<BITS, 2, 64, 1, 4, 1>;     // g 64, s <= 3 %, rank 3..4
template <int BITS> using ShapeA2 = StaticShape<BITS, 2, 64, 1, 8, 1>;     // g 64, rank 5..8
template <int BITS> using ShapeB1 = StaticShape<BITS, 1, 128, 2, 4, 2>;    // g 128 prefill blocks
template <int BITS> using ShapeB2 = StaticShape<BITS, 1, 64, 1, 4, 2>;     // g 128, flushed 64-token buffers
template <int BITS> using ShapeP1 = StaticShape<BITS, 1, 64, 0, 4, 2, true>;   // per-vector keys (outlier list), rank 3..4

// Whether the first copies of a ring of `stages` items may be requested before the wait for the kernel in front: none of
// them may read what that kernel can have written.
__device__ __forceinline__ bool early_start(const DecodeArgs& a, int stages, int blk_lo, int n_left) {
  return a.early_reads && (a.early_buf || blk_lo + min(n_left, (stages + 1) / 2) <= a.n_blocks_c);
}

}  // namespace gear
