// Algorithm 2 of a long segment, the loops: every loop of the power iteration multiplies by R^T R, a 128 x 128 matrix
// whatever the length of the segment.  pi_gram_kernel sums that matrix once per tile on the tensor cores (one pass over
// the residual instead of one per loop), pi_iterate_kernel runs the loops, the QR of B and the scaling of the last
// factor on it, on chip.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "gear_internal.cuh"
#include "gear_pi.cuh"
#include "gear_umma.cuh"

namespace gear {

// ------------------------------------------------------------------ G = R^T R
// Work: the 32-row blocks of all tiles, one after the other, cut into equal contiguous ranges, one per CTA (two CTAs per
// SM); a CTA leaves one partial G per tile it touches.  Partial number = CTA + tile, which is different for all of them.
constexpr int kGramRows = 32;
constexpr int kGramStages = 4;                                      // blocks in flight or being converted
constexpr int kGramStage = kGramRows * kHeadDim * 4;                // fp32 rows as they lie in memory
constexpr int kGramOperand = kGramRows * kHeadDim * 2;              // fp16 heads or remainders of a block
constexpr int kGramSmem = 1024 + 4 * kGramOperand + kGramStages * kGramStage;   // heads and remainders, two buffers
constexpr int kGramMinBlocks = 8;                                   // a partial is 128 KB, a block 16 KB: at least 256 rows per CTA
constexpr int kGramPartial = 2 * kHeadDim * kHeadDim;               // floats: two planes

struct GramSplit { int nb; long long blocks; int ctas; };
static __host__ __device__ inline GramSplit gram_split(int ntiles, int n_c, int sms) {
  GramSplit s;
  s.nb = (n_c + kGramRows - 1) / kGramRows;
  s.blocks = (long long)ntiles * s.nb;
  const long long most = (s.blocks + kGramMinBlocks - 1) / kGramMinBlocks;
  s.ctas = (int)(most < 2LL * sms ? most : 2LL * sms);
  return s;
}
size_t pi_gram_workspace_bytes(int ntiles, int n_c, int sms) {
  return (size_t)(gram_split(ntiles, n_c, sms).ctas + ntiles) * kGramPartial * 4 + (size_t)ntiles * kHeadDim * kHeadDim * 4;
}

// Bound: the fp32 residual from HBM, once, with the shared memory close behind (a block crosses it as fp32 twice, as fp16
// operands once, and the products read their operands from there).  Every fp32 entry becomes an fp16 head h and an fp16
// remainder l after exact power-of-two scaling by the tile's largest magnitude; h h, h l and l h are summed in fp32, so 22
// bits of each operand count.  One tcgen05.mma of 128 x 256 x 16 takes h^T [h | l]: 12 KB of operands per step instead of
// the 24 KB of three 128 x 128 products, l h being the transpose of h l.  The rows of a block lie in shared memory as they
// come ([token][channel]), which is the MN-major layout for both operands.  Blocks of 32 rows keep four of them in flight
// per CTA and the operands double, so that the conversion of a block runs beside the products of the one before.
// Eight warps convert, a ninth requests the copies and issues the products; they meet at mbarriers only, so a warp that is
// done with its part of a block goes on to the next one.
constexpr int kGramWarps = 8;
__global__ void __launch_bounds__(kGramWarps * 32 + 32, 2) pi_gram_kernel(PiArgs p, int sms) {
  extern __shared__ unsigned char smem_raw[];
  // full: the copy of a stage has landed; ready: every converting warp is done with a block (its operands are written, its
  // stage is read); mma_done: the products of a block are complete (its operand buffer is free, the accumulator current)
  __shared__ uint64_t full[kGramStages], ready[2], mma_done[2];
  __shared__ uint32_t tmem_slot;
  unsigned char* smem = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
  // operand buffer b: heads at 2 b, remainders at 2 b + 1 (in units of kGramOperand); each [2 halves of the channels]
  // [8-token groups][8][128 B], 128B swizzle
  unsigned char* stage = smem + 4 * kGramOperand;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const GramSplit sp = gram_split(p.ntiles, p.n_c, sms);
  const long long f0 = blockIdx.x * sp.blocks / gridDim.x, f1 = (blockIdx.x + 1LL) * sp.blocks / gridDim.x;
  if (tid == 0) {
    for (uint64_t& b : full) bar_init(&b);
    for (uint64_t& b : mma_done) bar_init(&b);
    for (uint64_t& b : ready) bar_init(&b, kGramWarps);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kGramWarps) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(smem_addr(&tmem_slot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  after_previous();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  const int count = (int)(f1 - f0);
  int tile = (int)(f0 / sp.nb), blk = (int)(f0 - (long long)tile * sp.nb);    // 64-bit divisions only here
  bool ok = true;                                                   // a wait gave up: go on without waiting, every loop still ends

  if (warp == kGramWarps) {
    if (lane == 0) {
      // descriptors: 128B swizzle, 64-channel halves 4 KB apart (leading), 8-token groups 1 KB apart (stride); the remainders
      // follow the heads, so the N = 256 operand has the same strides; fp32 accumulator, fp16 operands, both MN-major
      constexpr uint64_t kDesc = ((uint64_t)(kGramOperand / 2 >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
      constexpr uint32_t kIdesc = (1u << 4) | (1u << 15) | (1u << 16) | ((256u >> 3) << 17) | ((128u >> 4) << 24);
      int q_it = 0, q_tile = tile, q_blk = blk;
      auto request_next = [&]() {
        const int s = q_it % kGramStages;
        const float* src = p.R + ((size_t)q_tile * p.n_c + (size_t)q_blk * kGramRows) * kHeadDim;
        const uint32_t bytes = (uint32_t)min(kGramRows, p.n_c - q_blk * kGramRows) * kHeadDim * 4;
        bar_expect(&full[s], bytes);
        bulk_copy(stage + s * kGramStage, src, bytes, &full[s]);
        ++q_it;
        if (++q_blk == sp.nb) { q_blk = 0; ++q_tile; }
      };
      for (int s = 0; s < kGramStages && s < count; ++s) request_next();
      for (int it = 0; it < count; ++it) {
        ok = ok && bar_wait(&ready[it & 1], (uint32_t)(it >> 1) & 1u);
        if (ok) {
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint64_t op = kDesc | (smem_addr(smem + (it & 1) * 2 * kGramOperand) >> 4);
#pragma unroll
          for (int k = 0; k < kGramRows / 16; ++k)
            umma_f16(tmem, op + k * (2048 >> 4), op + k * (2048 >> 4), kIdesc, ((it == 0 || blk == 0) && k == 0) ? 0u : 1u);
          umma_commit(&mma_done[it & 1]);
          if (q_it < count) request_next();
        }
        if (++blk == sp.nb) blk = 0;
      }
      if (!ok) {
        atomicExch(p.status, -7 /* GEAR_ERR_TIMEOUT */);
        for (int it = max(0, q_it - kGramStages); it < q_it; ++it)  // let the copies in flight land (bounded)
          bar_wait(&full[it % kGramStages], (uint32_t)(it / kGramStages) & 1u);
      }
    }
  } else {
    float sr = 0.f;
    for (int it = 0; it < count; ++it) {
      const int s = it % kGramStages, rows = min(kGramRows, p.n_c - blk * kGramRows);
      unsigned char* op_hi = smem + (it & 1) * 2 * kGramOperand;
      unsigned char* op_lo = op_hi + kGramOperand;
      if (it == 0 || blk == 0) sr = exp2_int(-pow2_exponent(__uint_as_float(p.Rmax[tile])));
      ok = ok && bar_wait(&full[s], (uint32_t)(it / kGramStages) & 1u);
      if (it >= 2) ok = ok && bar_wait(&mma_done[it & 1], (uint32_t)((it - 2) >> 1) & 1u);    // this operand buffer is free again
      const float4* src = reinterpret_cast<const float4*>(stage + s * kGramStage);
#pragma unroll
      for (int j = 0; j < kGramRows / kGramWarps; ++j) {
        const int row = warp + kGramWarps * j, q = lane;            // a row per warp, four channels per lane
        const float4 v = row < rows ? src[row * 32 + q] : make_float4(0.f, 0.f, 0.f, 0.f);
        uint32_t h0, l0, h1, l1;
        split_pair(v.x * sr, v.y * sr, h0, l0);
        split_pair(v.z * sr, v.w * sr, h1, l1);
        const int at = (q >> 4) * (kGramOperand / 2) + (row >> 3) * 1024 + (row & 7) * 128 + ((((q & 15) >> 1) ^ (row & 7)) << 4) + (q & 1) * 8;
        *reinterpret_cast<uint2*>(op_hi + at) = make_uint2(h0, h1);
        *reinterpret_cast<uint2*>(op_lo + at) = make_uint2(l0, l1);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) bar_arrive(&ready[it & 1]);
      if (it + 1 == count || blk + 1 == sp.nb) {                    // last block of the tile in this range: leave the partial
        ok = ok && bar_wait(&mma_done[it & 1], (uint32_t)(it >> 1) & 1u);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        __syncwarp();
        // columns 0..127 of accumulator row i are h h, 128..255 h l; plane 0 of the partial gets (h h + h l)[i][c] in row c
        // (h h is symmetric), plane 1 h l[i][c] in row c: a warp writes 128 consecutive bytes.  The transpose of h l is
        // taken where the partials are summed (adding it here costs a second trip to L2: 41 us of 220 at 512 tiles)
        float* part = p.Gpart + (size_t)(blockIdx.x + tile) * kGramPartial + (warp & 3) * 32 + lane;
        const uint32_t lanes = tmem + ((uint32_t)((warp & 3) * 32) << 16);
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
          const int c0 = (warp >> 2) * 64 + h * 32;
          uint32_t v[32], w[32];
          tmem_ld32(v, lanes + c0);
          tmem_ld32(w, lanes + 128 + c0);
#pragma unroll
          for (int c = 0; c < 32; ++c) {
            part[(size_t)(c0 + c) * kHeadDim] = __uint_as_float(v[c]) + __uint_as_float(w[c]);
            part[(size_t)(kHeadDim + c0 + c) * kHeadDim] = __uint_as_float(w[c]);
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      }
      if (++blk == sp.nb) { blk = 0; ++tile; }
    }
    if (!ok && lane == 0) atomicExch(p.status, -7 /* GEAR_ERR_TIMEOUT */);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == kGramWarps) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tmem) : "memory");
}

// G of every tile from its partials (fixed order): 8 rows per CTA, thread i sums column i.  Plane 0 is read by rows, of plane
// 1 (the transpose is wanted) the thread takes one 32-byte sector of row i.  Few tiles have many partials each (one
// per CTA of the Gram kernel); 16 CTAs per tile keep their sum short.  Bound: the partials, from L2.
constexpr int kSumRows = 8;
__global__ void __launch_bounds__(kHeadDim) pi_gram_sum_kernel(PiArgs p, int gram_ctas, int sms) {
  const int tile = blockIdx.y, k0 = blockIdx.x * kSumRows, i = threadIdx.x;
  const GramSplit sp = gram_split(p.ntiles, p.n_c, sms);
  const long long NW = gram_ctas, b0 = (long long)tile * sp.nb, b1 = b0 + sp.nb;
  const int w0 = (int)(((b0 + 1) * NW + sp.blocks - 1) / sp.blocks - 1), w1 = (int)((b1 * NW + sp.blocks - 1) / sp.blocks - 1);
  float g[kSumRows];
  after_previous();
#pragma unroll
  for (int k = 0; k < kSumRows; ++k) g[k] = 0.f;
  const float* src = p.Gpart + (size_t)(w0 + tile) * kGramPartial;
#pragma unroll 2
  for (int w = w0; w <= w1; ++w, src += kGramPartial) {
    const float4* hl = reinterpret_cast<const float4*>(src + (size_t)(kHeadDim + i) * kHeadDim + k0);
    const float4 a = __ldcg(hl), b = __ldcg(hl + 1);
#pragma unroll
    for (int k = 0; k < kSumRows; ++k) g[k] += __ldcg(src + (size_t)(k0 + k) * kHeadDim + i);
    g[0] += a.x; g[1] += a.y; g[2] += a.z; g[3] += a.w;
    g[4] += b.x; g[5] += b.y; g[6] += b.z; g[7] += b.w;
  }
#pragma unroll
  for (int k = 0; k < kSumRows; ++k) p.G[((size_t)tile * kHeadDim + k0 + k) * kHeadDim + i] = g[k];
}

// ------------------------------------------------------------------ the loops on G
template <int RP>
__device__ __forceinline__ void load_row(const float* src, float (&v)[RP]) {
#pragma unroll
  for (int q = 0; q < RP / 4; ++q) {
    const float4 f = reinterpret_cast<const float4*>(src)[q];
    v[4 * q] = f.x; v[4 * q + 1] = f.y; v[4 * q + 2] = f.z; v[4 * q + 3] = f.w;
  }
}
// Sums of N numbers over the lanes of a warp, N - 1 + log2(32 / N) shuffles: a[0] of lane l becomes the sum of number l N / 32.
template <int N>
__device__ __forceinline__ void warp_sums(float (&a)[N], int lane) {
#pragma unroll
  for (int o = 16, n = N; o > 0; o >>= 1) {
    const bool upper = (lane & o) != 0;
    if (n > 1) {
      n >>= 1;
#pragma unroll
      for (int i = 0; i < N / 2; ++i)
        if (i < n) a[i] = (upper ? a[i + n] : a[i]) + __shfl_xor_sync(0xffffffffu, upper ? a[i] : a[i + n], o);
    } else {
      a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
    }
  }
}

// One CTA per tile.  Thread (i, half) holds 64 entries of row i of G in registers; B (128 x r) is in shared memory.
//   B <- G B, iters - 1 times (each time brought back to magnitude one by a power of two, which the QR drops again);
//   B <- Q(B), classical Gram-Schmidt with each projection taken twice, one warp;
//   G0 = B^T G B is the Gram matrix of A0 = R B up to rounding: U^-1 of its Cholesky factor, folded into B, makes the
//   columns of R B nearly orthonormal before they are computed, so one explicit round of CholeskyQR is enough after.
// Bound: latency of the chain (G from L2, products, Gram-Schmidt, Cholesky); r^2 and 128 r work per step.  Two CTAs per SM, for
// which sixteen columns give up G during the QR and read it again (512 tiles, rank 16: 232 -> 145 us); G0 from rows read as
// 128 bits and sums of all its entries in one exchange (rank 16: 311 -> 232, rank 8: 63 -> 54).
template <int RP>
__global__ void __launch_bounds__(256, 2) pi_iterate_kernel(PiArgs p, const float* B0, unsigned long long seed, int segment,
                                                         int iters) {
  __shared__ __align__(16) float Bs[kHeadDim][RP];
  __shared__ __align__(16) float Cs[kHeadDim][RP];
  __shared__ float Gm[RP][RP + 1], Wm[RP][RP + 1];
  __shared__ float wmax[4];
  const int tile = blockIdx.x, tid = threadIdx.x, i = tid & 127, half = tid >> 7, warp = tid >> 5, lane = tid & 31;
  const int r = p.rank;
  float g[64];
  auto load_g = [&]() {
    const float* src = p.G + ((size_t)tile * kHeadDim + half * 64) * kHeadDim + i;
#pragma unroll
    for (int k = 0; k < 64; ++k) g[k] = __ldcg(src + (size_t)k * kHeadDim);
  };
  after_previous();
  load_g();
  if (half == 0) {
    const size_t gtile = (size_t)p.bh0 * 2 + tile;
#pragma unroll
    for (int rho = 0; rho < RP; ++rho)
      Bs[i][rho] = rho < r ? (B0 ? B0[(gtile * kHeadDim + i) * r + rho] : start_value(seed, segment, gtile, i, rho)) : 0.f;
  }
  __syncthreads();
  float c[RP];
  auto times_g = [&]() {                          // c = (G B) row i: half 0 holds the sum of both halves
#pragma unroll
    for (int rho = 0; rho < RP; ++rho) c[rho] = 0.f;
#pragma unroll
    for (int k = 0; k < 64; ++k)
#pragma unroll
      for (int q = 0; q < RP / 4; ++q) {
        const float4 b = *reinterpret_cast<const float4*>(&Bs[half * 64 + k][4 * q]);
        c[4 * q] = fmaf(g[k], b.x, c[4 * q]);
        c[4 * q + 1] = fmaf(g[k], b.y, c[4 * q + 1]);
        c[4 * q + 2] = fmaf(g[k], b.z, c[4 * q + 2]);
        c[4 * q + 3] = fmaf(g[k], b.w, c[4 * q + 3]);
      }
    if (half == 1) {
#pragma unroll
      for (int rho = 0; rho < RP; ++rho) Cs[i][rho] = c[rho];
    }
    __syncthreads();
    if (half == 0) {
#pragma unroll
      for (int rho = 0; rho < RP; ++rho) c[rho] += Cs[i][rho];
    }
  };
  for (int l = 0; l + 1 < iters; ++l) {
    times_g();
    float m = 0.f;
    if (half == 0) {
#pragma unroll
      for (int rho = 0; rho < RP; ++rho) m = fmaxf(m, fabsf(c[rho]));
      m = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m)));
      if (lane == 0) wmax[warp] = m;
    }
    __syncthreads();
    if (half == 0) {
      const float sc = exp2_int(-pow2_exponent(fmaxf(fmaxf(wmax[0], wmax[1]), fmaxf(wmax[2], wmax[3]))));
#pragma unroll
      for (int rho = 0; rho < RP; ++rho) Bs[i][rho] = c[rho] * sc;
    }
    __syncthreads();
  }
  if (warp == 0) {                                // B <- Q(B)
    float b[4][RP];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int rho = 0; rho < RP; ++rho) b[j][rho] = Bs[lane + 32 * j][rho];
#pragma unroll
    for (int cc = 0; cc < RP; ++cc) {
      if (cc < r) {
#pragma unroll
        for (int sweep = 0; sweep < 2; ++sweep) {
          float d[RP];
#pragma unroll
          for (int q = 0; q < cc; ++q) {
            d[q] = 0.f;
#pragma unroll
            for (int j = 0; j < 4; ++j) d[q] = fmaf(b[j][q], b[j][cc], d[q]);
          }
#pragma unroll
          for (int q = 0; q < cc; ++q) d[q] = warp_sum(d[q]);
#pragma unroll
          for (int q = 0; q < cc; ++q)
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j][cc] = fmaf(-d[q], b[j][q], b[j][cc]);
        }
        auto norm2 = [&]() {
          float s = 0.f;
#pragma unroll
          for (int j = 0; j < 4; ++j) s = fmaf(b[j][cc], b[j][cc], s);
          return warp_sum(s);
        };
        const float nrm2 = norm2();
        const float inv = nrm2 > 0.f ? rsqrtf(nrm2) : 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) b[j][cc] *= inv;
        const float n2 = norm2();                 // one Newton step keeps the column norm at 1 to rounding
        const float fix = n2 > 0.f ? 1.5f - 0.5f * n2 : 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) b[j][cc] *= fix;
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int rho = 0; rho < RP; ++rho) Bs[lane + 32 * j][rho] = b[j][rho];
  }
  __syncthreads();
  if (RP == 16) load_g();                         // sixteen columns leave no registers for G beside the QR
  times_g();
  __syncthreads();
  if (half == 0) {
#pragma unroll
    for (int rho = 0; rho < RP; ++rho) Cs[i][rho] = c[rho];
  }
  __syncthreads();
  constexpr int U = RP / 8 > 0 ? RP / 8 : 1;      // rows of Q^T G Q per warp
  if (warp * U < RP) {
    float e[U * RP];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float cv[RP];
      load_row<RP>(Cs[lane + 32 * j], cv);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const float bu = Bs[lane + 32 * j][warp * U + u];
#pragma unroll
        for (int v = 0; v < RP; ++v) e[u * RP + v] = j == 0 ? bu * cv[v] : fmaf(bu, cv[v], e[u * RP + v]);
      }
    }
    warp_sums<U * RP>(e, lane);                   // lane l: number l U RP / 32
    const int at = lane * U * RP / 32;
    Gm[warp * U + at / RP][at % RP] = e[0];
  }
  __syncthreads();
  if (warp == 0) {
    const bool small = warp_chol_inverse<RP, true>(&Gm[0][0], &Wm[0][0], RP + 1, r, lane);
    if (lane == 0) p.ill[tile] = small;
  }
  __syncthreads();
  {
    // half 0: b = Q(B) W; half 1: (R^T R) b = G Q(B) W.  G was summed over R 2^-er, so the columns of R b would have norm 2^er
    const float (*m)[RP] = half == 0 ? Bs : Cs;
    const int er = pow2_exponent(__uint_as_float(p.Rmax[tile]));
    const float sc = exp2_int(half == 0 ? -er : er);
    float* out = (half == 0 ? p.Bcur : p.Bg) + ((size_t)tile * kHeadDim + i) * kMaxRank;
    float row[RP];
    load_row<RP>(m[i], row);
#pragma unroll
    for (int rho = 0; rho < kMaxRank; ++rho) {
      float v = 0.f;
      if (rho < RP && rho < r) {
#pragma unroll
        for (int q = 0; q < RP; ++q)
          if (q <= rho && q < r) v = fmaf(row[q], Wm[q][rho < RP ? rho : 0], v);
      }
      out[rho] = v * sc;
    }
  }
}

cudaError_t launch_pi_gram(const PiArgs& p, const float* B0, unsigned long long seed, int segment, int iters, int sms,
                           bool overlap, cudaStream_t st) {
  const GramSplit sp = gram_split(p.ntiles, p.n_c, sms);
  cudaError_t e = cudaFuncSetAttribute(pi_gram_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kGramSmem);
  if (e == cudaSuccess) e = launch_after(overlap, pi_gram_kernel, dim3(sp.ctas), kGramWarps * 32 + 32, kGramSmem, st, p, sms);
  if (e == cudaSuccess) e = launch_after(overlap, pi_gram_sum_kernel, dim3(kHeadDim / kSumRows, p.ntiles), kHeadDim, 0, st, p, sp.ctas, sms);
  if (e != cudaSuccess) return e;
  count_launches(2);
  return launch_pi_iterate(p, B0, seed, segment, iters, st);
}

cudaError_t launch_pi_iterate(const PiArgs& p, const float* B0, unsigned long long seed, int segment, int iters, cudaStream_t st) {
  auto iterate = p.rank <= 4 ? pi_iterate_kernel<4> : p.rank <= 8 ? pi_iterate_kernel<8> : pi_iterate_kernel<16>;
  const cudaError_t e = launch_dependent(iterate, dim3(p.ntiles), 256, 0, st, p, B0, seed, segment, iters);
  if (e != cudaSuccess) return e;
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace gear
