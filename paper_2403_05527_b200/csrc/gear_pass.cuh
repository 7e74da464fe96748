// The last product of Algorithm 2, A0 = R b, on the tensor cores (mma.sync.m16n8k16, fp16 operands, fp32 accumulation; n is the rank,
// too narrow for a tile of its own in tensor memory): what the kernels share that read the residual (gear_compress.cu) or compute
// it again from the codes (gear_pass_codes.cu).  Every fp32 operand is cut into an fp16 head and an fp16 remainder, the four
// cross products summed in fp32: 22 bits of each operand survive.  Powers of two bring the operands into fp16's range first (R
// by the tile's largest magnitude, each column of b by its own) and are divided out of the results, so the scaling itself is exact.
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

#include "gear_pi.cuh"

namespace gear {

__device__ __forceinline__ void mma16816_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
constexpr int kChunkRows = 512;                  // rows per CTA at most (PiArgs::chunk_rows)
constexpr int kPassWarps = 4;

// NT = 8-column tiles of n: four rank columns (head and remainder each) per tile.
template <int NT>
struct PassFactor {
  static constexpr int RP = 4 * NT;              // rank columns: each gives a (head, remainder) column pair of n
  static constexpr bool kGram = NT <= 2;         // A0^T A0 here (in registers), else by pi_gram2_kernel
  struct Shared {
    __align__(16) __half bsplit[2 * RP][kHeadDim];   // [2 rho + (0: head, 1: remainder)][channel]
    float colmax[kPassWarps][RP];
    float gred[kGram ? kPassWarps : 1][RP][RP];
  };
  float inv_a[NT];                               // back to a for column rho = 4 nt + t
  float gram[kGram ? NT : 1][kGram ? RP : 1];    // gram[nt][v]: row rho = 4 nt + t of A0^T A0, column v

  // the scaled, split factor columns into shared memory; one channel per thread (kPassWarps * 32 == kHeadDim)
  __device__ __forceinline__ void load(const PiArgs& p, int tile, int er, Shared& sh) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, t = lane & 3, j = threadIdx.x;
    float bj[RP];
    int eb[RP];
#pragma unroll
    for (int r = 0; r < RP; ++r) {
      bj[r] = p.Bcur[((size_t)tile * kHeadDim + j) * kMaxRank + r];
      const float m = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(bj[r]))));
      if (lane == 0) sh.colmax[warp][r] = m;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RP; ++r) {
      float m = 0.f;
#pragma unroll
      for (int w = 0; w < kPassWarps; ++w) m = fmaxf(m, sh.colmax[w][r]);
      eb[r] = pow2_exponent(m);
      const float v = bj[r] * exp2_int(-eb[r]);
      const __half h = __float2half_rn(v);
      sh.bsplit[2 * r][j] = h;
      sh.bsplit[2 * r + 1][j] = __float2half_rn(v - __half2float(h));
    }
    __syncthreads();
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      int ebt = eb[4 * nt];
#pragma unroll
      for (int q = 1; q < 4; ++q) ebt = t == q ? eb[4 * nt + q] : ebt;
      inv_a[nt] = exp2_int(er + ebt);
    }
#pragma unroll
    for (int nt = 0; nt < (kGram ? NT : 1); ++nt)
#pragma unroll
      for (int v = 0; v < (kGram ? RP : 1); ++v) gram[nt][v] = 0.f;
  }

  // d[nt]: the products of 16 rows; this lane's are rows ra and rc (of the tile, valid where va / vc), the others come as zero
  __device__ __forceinline__ void store(float (&d)[NT][4], float* A0, int ra, int rc, bool va, bool vc) {
    const int t = threadIdx.x & 3;
    mine_rows(d);
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      if (va) A0[(size_t)ra * RP + 4 * nt + t] = mine[0][nt];
      if (vc) A0[(size_t)rc * RP + 4 * nt + t] = mine[1][nt];
    }
  }
  __device__ __forceinline__ void add_gram() {
    const int lane = threadIdx.x & 31;
    if (kGram) {
#pragma unroll
      for (int half = 0; half < 2; ++half)
#pragma unroll
        for (int nv = 0; nv < NT; ++nv)
#pragma unroll
          for (int tv = 0; tv < 4; ++tv) {
            const float other = __shfl_sync(0xffffffffu, mine[half][nv], (lane & ~3) | tv);   // a[row][4 nv + tv]
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
              gram[kGram ? nt : 0][kGram ? 4 * nv + tv : 0] = fmaf(mine[half][nt], other, gram[kGram ? nt : 0][kGram ? 4 * nv + tv : 0]);
          }
    }
  }
  // this chunk's part of A0^T A0: rows of the warp (over gid), then the warps, in a fixed order
  __device__ __forceinline__ void leave_gram(const PiArgs& p, int tile, int chunk, Shared& sh) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, t = lane & 3;
    if (kGram) {
#pragma unroll
      for (int nt = 0; nt < (kGram ? NT : 1); ++nt)
#pragma unroll
        for (int v = 0; v < (kGram ? RP : 1); ++v) {
          float g = gram[nt][v];
#pragma unroll
          for (int o = 4; o < 32; o <<= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
          if (gid == 0) sh.gred[kGram ? warp : 0][4 * nt + t][v] = g;
        }
      __syncthreads();
      for (int i = threadIdx.x; i < RP * RP; i += blockDim.x) {
        const int u = i / RP, v = i % RP;
        float g = 0.f;
        for (int w = 0; w < kPassWarps; ++w) g += sh.gred[kGram ? w : 0][u][v];
        p.Gp[((size_t)tile * p.nchunk + chunk) * 256 + u * kMaxRank + v] = g;
      }
    }
  }

 private:
  float mine[2][NT];                             // a[row ra | rc][rho 4 nt + t]
  __device__ __forceinline__ void mine_rows(float (&d)[NT][4]) {
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      mine[0][nt] = (d[nt][0] + d[nt][1]) * inv_a[nt];
      mine[1][nt] = (d[nt][2] + d[nt][3]) * inv_a[nt];
    }
  }
};

}  // namespace gear
