// Filter (Eq. 4), Quant (Eq. 2, Eq. 5) and packing of a long segment whose residual R = X - D^ - S is not kept: the sum
// R^T R, all that the loops of Algorithm 2 need of it (gear_gram.cu), is taken on the tensor cores while a block is on chip,
// and the one product R B that is left afterwards computes the residual again from X and the codes (gear_pass_codes.cu).
// Segments in blocks of 64 or 128 tokens whose key and value groups are both as long, with up to one (64) or two (128)
// outliers per side; the others keep the fp32 residual in a workspace (gear_compress.cu).
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "gear_internal.cuh"
#include "gear_pi.cuh"
#include "gear_quant.cuh"
#include "gear_tma.cuh"
#include "gear_umma.cuh"

namespace gear {

constexpr int kQgPart = 64;                        // entries of a thread: a group of 64, or half a group of 128
__host__ __device__ constexpr int qg_threads(int len) { return 2 * len; }                     // 128 channels times `len` tokens a block
__host__ __device__ constexpr int qg_operand(int len) { return len * kHeadDim * 2; }          // fp16 heads, or remainders, of a block
constexpr int kQgCodeKey = kHeadDim + 4;           // bytes per row of packed key codes
// Tokens per CTA at least, a partial sum being 64 KB; where there are fewer blocks than SMs a block each.
constexpr int kQgMinRows = 128;
// Bits a tile's residuals may grow by before the sums are scaled again: the first block's largest is brought to 2^4 .. 2^5,
// fp16 ends at 2^16.
constexpr int kQgStart = 4, kQgGrow = 14;

__host__ __device__ constexpr int qg_ctas_per_sm(int len) { return len == 64 ? 4 : 2; }
__host__ __device__ constexpr int qg_code_bytes(int bits, int side, int len) {
  return side == 0 ? len * bits / 8 * kQgCodeKey : kHeadDim * bits / 8 * (len + 4);
}
__host__ __device__ constexpr int qg_smem(int bits, int side, int len) {
  return 1024 + 2 * qg_operand(len) + len * kHeadDim * 2 + qg_code_bytes(bits, side, len);
}

QgSplit qg_split(int nbh, const SegDesc& sd, int sms) {
  QgSplit s;
  s.blocks = (long long)nbh * sd.nblk;
  const long long per = s.blocks <= sms ? 1 : kQgMinRows / sd.T, most = (s.blocks + per - 1) / per, room = (long long)qg_ctas_per_sm(sd.T) * sms;
  s.ctas = (int)(most < room ? most : room);
  return s;
}
bool qg_fits(const SegDesc& sd, const CacheConst& cc) {
  if (sd.rank == 0 || sd.csr_base16 != 0 || sd.T != cc.g_v) return false;
  return sd.k_k == cc.k_v && (sd.T == 64 ? sd.k_k <= 1 : sd.T == 128 && sd.k_k <= 2);
}
size_t qg_partials(int nbh, const SegDesc& sd, int sms) { return 2 * (size_t)(qg_split(nbh, sd, sms).ctas + nbh); }

// Largest and smallest instances of a thread's entries and of its partner's (K = 0: one of each, 1: two, 2: three), as pairs (i-th largest,
// minus the i-th smallest), so that one comparison serves both sides.  An entry that is NaN makes
// the first of them NaN.
template <int K> struct Ends { __half2 v[K + 1]; };
// the first K + 1 of the union: the k-th largest is the maximum over i + j = k of min(a_i, b_j), a_0 = b_0 = infinity
template <int K>
__device__ __forceinline__ Ends<K> merge_ends(const Ends<K>& a, const Ends<K>& b) {
  Ends<K> r;
  r.v[0] = __hmax2_nan(a.v[0], b.v[0]);
  if constexpr (K > 0) r.v[1] = __hmax2_nan(__hmin2_nan(a.v[0], b.v[0]), __hmax2_nan(a.v[1], b.v[1]));
  if constexpr (K > 1)
    r.v[2] = __hmax2_nan(__hmax2_nan(__hmin2_nan(a.v[0], b.v[1]), __hmin2_nan(a.v[1], b.v[0])), __hmax2_nan(a.v[2], b.v[2]));
  return r;
}
// of 64 entries in packed pairs.  Sorting networks of four pairs, merged one after the other per half of the pairs (largest and smallest
// apart), the halves at the end: 7 instructions per pair for K = 2, where a chain that keeps three of each takes 10.
template <int K>
__device__ __forceinline__ Ends<K> ends_of(const __half2 (&xp)[kQgPart / 2]) {
  Ends<K> top, bot;                                // bot: negated
#pragma unroll
  for (int q = 0; q < kQgPart / 2; q += 4) {
    __half2 a = xp[q], b = xp[q + 1], c = xp[q + 2], d = xp[q + 3];
    auto order = [](__half2& hi, __half2& lo) { const __half2 h = __hmax2_nan(hi, lo); lo = __hmin2_nan(hi, lo); hi = h; };
    order(a, b); order(c, d); order(a, c); order(b, d);
    if (K > 0) order(b, c);
    Ends<K> t, u;
    t.v[0] = a; u.v[0] = __hneg2(d);
    if constexpr (K > 0) { t.v[1] = b; u.v[1] = __hneg2(c); }
    if constexpr (K > 1) { t.v[2] = c; u.v[2] = __hneg2(b); }
    top = q == 0 ? t : merge_ends(top, t);
    bot = q == 0 ? u : merge_ends(bot, u);
  }
  Ends<K> even, odd;
#pragma unroll
  for (int i = 0; i <= K; ++i) { even.v[i] = __lows2half2(top.v[i], bot.v[i]); odd.v[i] = __highs2half2(top.v[i], bot.v[i]); }
  return merge_ends(even, odd);
}
// first set entry of 64 mask bits (even entries, odd entries), removed from them; 64 if none
__device__ __forceinline__ int take_entry(unsigned int& even, unsigned int& odd) {
  const int fe = even ? 2 * (__ffs((int)even) - 1) : 64, fo = odd ? 2 * (__ffs((int)odd) - 1) + 1 : 64;
  if (fe < fo) { even &= even - 1; return fe; }
  if (fo < 64) odd &= odd - 1;
  return fo;
}

// Bound: instruction issue, with the 2 bytes per entry of X behind it.  A thread owns 64 entries of a group (keys: tokens of a
// channel, values: channels of a token), which it keeps in registers as packed pairs; groups of 128 belong to two threads, which
// exchange what the filter has to know of the other half.  See quant_fast_kernel for the order of the arithmetic.  The residual of
// an entry, scaled by a power of two, leaves as an fp16 head and an
// fp16 remainder (22 bits) for the products h^T h and h^T 2l: with l h the transpose of h l, the mean of the accumulator
// and its transpose is h h + h l + l h, in 128 columns of tensor memory instead of 256, so that four CTAs fit on an SM.
// Keys are stored [channel][token] (K-major), as the thread of a channel has them, values [token][channel] (MN-major);
// both with 128-byte swizzle, eight entries per store.  A CTA works through a contiguous range of blocks of one side; what it
// summed over a tile leaves as a partial with the exponent it was scaled by.  The exponent comes from the bound on the first
// block's residuals; a block that exceeds it by more than fp16's range has the sums scaled down in place.
// Codes: the F entries that share a byte of the fragments are added up as the rounded sums hold them in their low bytes, each
// times its field's weight; what the filtered entries left there is taken out again afterwards (modulo 256).
// 2 bits, 8 x 32 heads x 4096: keys 157, values 155 us (quant_fast_kernel 154 and 168, and 182 for R^T R from the fp32
// residual); 22 to 24 instructions per entry, 60 % of the issue slots, tensor cores 22 %.  The whole call 851 -> 575 us; 4 bits, 16 x
// 40 heads x 8192 4162 -> 2854 us, one head of 192 to 2048 tokens 70 -> 45 to 68 us (half of that from launches that overlap).
// Groups of 128 with two outliers per side, 2 bits, 2 x 8 heads x 16384: keys 64, values 58 us (one thread per group 74 and 82: three
// CTAs of four warps, and more code than the instruction cache holds); the call for two such layers 603 -> 455 us.
template <int BITS, int SIDE, int L, int K>
__global__ void __launch_bounds__(qg_threads(L), qg_ctas_per_sm(L))
quant_gram_kernel(CompressArgs p, int nbh, const __grid_constant__ CUtensorMap value_rows) {
  constexpr int F = 8 / BITS, kPartRows = kQgPart / F;              // rows of packed codes of a thread's entries
  constexpr int kThreads = qg_threads(L), kOperand = qg_operand(L);
  constexpr int kCodePitch = SIDE == 0 ? kQgCodeKey : L + 4;
  constexpr bool kShared = L > kQgPart;            // two threads per group
  extern __shared__ unsigned char smem_raw[];
  __shared__ uint64_t full, mma_done;
  __shared__ uint32_t tmem_slot;
  __shared__ unsigned int dmax_bits[2], smax_bits[2], rmax_bits[2];    // of even and odd blocks
  __shared__ __half2 ends_s[kShared ? K + 1 : 1][kShared ? kThreads : 1];
  unsigned char* op_hi = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
  unsigned char* op_lo = op_hi + kOperand;
  unsigned char* tile = op_lo + kOperand;          // keys: [token][channel]; values: boxes, [64-channel half][token]
  unsigned char* codes = tile + L * kHeadDim * 2;
  const SegDesc& sd = p.seg;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // keys: channel and which 64 tokens; values: token and which 64 channels.  A warp's lanes are neighbours.
  const int line = SIDE == 0 ? tid % kHeadDim : tid % L, part = SIDE == 0 ? tid / kHeadDim : tid / L;
  const int gi = SIDE == 1 && !kShared ? 2 * line + part : line;    // the group's number in the record
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) { dmax_bits[i] = 0u; smax_bits[i] = 0u; rmax_bits[i] = 0u; }
    bar_init(&full);
    bar_init(&mma_done);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc<kHeadDim>(&tmem_slot);
  // The two sides do not touch each other's results: the values' CTAs start as SMs come free and wait for the keys only at their end, so
  // that whoever waits for them waits for both.
  if (SIDE == 0) after_previous();
  else asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  tmem_fence_before();
  __syncthreads();
  tmem_fence_after();
  const uint32_t tmem = tmem_slot;

  const long long blocks = (long long)nbh * sd.nblk;
  const long long f0 = blockIdx.x * blocks / gridDim.x, f1 = (blockIdx.x + 1LL) * blocks / gridDim.x;
  const int count = (int)(f1 - f0);
  int bhl = (int)(f0 / sd.nblk), blk = (int)(f0 - (long long)bhl * sd.nblk);
  auto request = [&](int it) {                     // by thread 0; blocks of consecutive (batch, head) pairs are adjacent
    bar_expect(&full, L * kHeadDim * 2);
    if (SIDE == 0) {
      bulk_copy(tile, p.K + (size_t)(f0 + it) * L * kHeadDim, L * kHeadDim * 2, &full);
    } else {
#pragma unroll
      for (int b = 0; b < 2 * (L / kBoxRows); ++b)
        load_box(tile + b * kBoxBytes, &value_rows, b / (L / kBoxRows) * kBoxChannels, (int)(f0 + it) * L + b % (L / kBoxRows) * kBoxRows, &full);
    }
  };
  if (tid == 0 && count > 0) request(0);

  // entry e of part q of the thread's line
  auto entry_of = [&](int q, int e) -> __half {
    if (SIDE == 0) return reinterpret_cast<const __half*>(tile)[(q * kQgPart + e) * kHeadDim + line];
    return *reinterpret_cast<const __half*>(tile + q * (L * 128) + box_at(line, e));
  };
  // where the thread's entries e .. e + 7 go as operands (e a multiple of eight)
  unsigned char* const op_line = op_hi + (SIDE == 0 ? part * (kHeadDim * 128) + line * 128 : part * (L * 128) + line * 128);
  auto op_at = [&](int e) { return ((e / 8) ^ (line & 7)) << 4; };
  // row of the packed codes and field of entry e
  auto code_row = [&](int e) { return SIDE == 0 ? e % kPartRows : e / (16 * F) * 16 + e % 16; };
  auto code_field = [&](int e) { return SIDE == 0 ? e / kPartRows : e % (16 * F) / 16; };
  unsigned char* mine = codes + part * kPartRows * kCodePitch + line;

  int exp_cur = 0;
  bool exp_set = false;
  uint32_t parity = 0, mma_parity = 0;
  bool mma_pending = false, fresh = true;          // fresh: the accumulator starts with the next product
  bool ok = true;
  for (int it = 0; it < count; ++it) {
    ok = ok && bar_wait(&full, parity);
    parity ^= 1u;
    unsigned char* rec = p.arena + sd.seg_base + (size_t)(p.bh0 + bhl) * sd.bh_stride + sd.bfac_bytes + (size_t)blk * sd.rec_bytes;
    __half2 xp[kQgPart / 2];                       // entries 2q, 2q + 1
    if (SIDE == 0) {
      const __half* col = reinterpret_cast<const __half*>(tile) + part * kQgPart * kHeadDim + line;
#pragma unroll
      for (int q = 0; q < kQgPart / 2; ++q) xp[q] = __halves2half2(col[(2 * q) * kHeadDim], col[(2 * q + 1) * kHeadDim]);
    } else {
      const unsigned char* row = tile + part * (L * 128) + line * 128;
#pragma unroll
      for (int q = 0; q < kQgPart / 8; ++q) {
        const uint4 v = *reinterpret_cast<const uint4*>(row + ((q ^ (line & 7)) << 4));
        xp[4 * q] = *reinterpret_cast<const __half2*>(&v.x);
        xp[4 * q + 1] = *reinterpret_cast<const __half2*>(&v.y);
        xp[4 * q + 2] = *reinterpret_cast<const __half2*>(&v.z);
        xp[4 * q + 3] = *reinterpret_cast<const __half2*>(&v.w);
      }
    }
    float mn, mx;
    int oi[2 * K + 1];                             // the thread's filtered entries, ascending; kQgPart and more: none
    oi[2 * K] = kQgPart;
    int before = 0;                                // filtered entries of the group in the part ahead
    if constexpr (!kShared) {
      static_assert(K <= 1, "");
      int imax, imin;
      filter_one<L, K, true>(xp, 0, mn, mx, imax, imin);
      if (K == 1) { oi[0] = min(imax, imin); oi[2 * K - 1] = max(imax, imin); }
    } else {
      Ends<K> ends = ends_of<K>(xp), other;
#pragma unroll
      for (int i = 0; i <= K; ++i) ends_s[i][tid] = ends.v[i];
      __syncthreads();
#pragma unroll
      for (int i = 0; i <= K; ++i) other.v[i] = ends_s[i][tid ^ (kThreads / 2)];
      ends = merge_ends(ends, other);
      float top[K + 1], bot[K + 1];
#pragma unroll
      for (int i = 0; i <= K; ++i) { top[i] = __low2float(ends.v[i]); bot[i] = -__high2float(ends.v[i]); }
      mx = top[K]; mn = bot[K];
      if constexpr (K > 0) {
        if (bot[K - 1] < top[K - 1]) {
          // The K entries above or at the K-th largest instance, of equal ones the first; the smallest likewise
          const __half2 vT = __float2half2_rn(top[K - 1]), vB = __float2half2_rn(bot[K - 1]);
          unsigned int t[2] = {0u, 0u}, b[2] = {0u, 0u};            // bit i of a half of word w: pair 16 w + i
#pragma unroll
          for (int q = 0; q < kQgPart / 2; ++q) {
            const unsigned int bit = 0x00010001u << (q & 15);
            t[q >> 4] |= __hge2_mask(xp[q], vT) & bit;
            b[q >> 4] |= __hle2_mask(xp[q], vB) & bit;
          }
          unsigned int even = 0u, odd = 0u;
          auto collect = [&](const unsigned int (&m)[2], const float (&end)[K + 1], auto of_other) {
            unsigned int me = __byte_perm(m[0], m[1], 0x5410), mo = __byte_perm(m[0], m[1], 0x7632);
            if (end[K] == end[K - 1]) {              // more than K entries reach the bound: one group in fifty of ordinary data
              int take = K, ahead = 0;
#pragma unroll
              for (int i = 0; i < K; ++i) take -= end[i] != end[K - 1];
#pragma unroll
              for (int i = 0; i <= K; ++i) ahead += of_other(i) == end[K - 1];
              if (part > 0) take -= min(take, ahead);
              unsigned int ke = 0u, ko = 0u;
#pragma unroll 1
              while (me | mo) {
                const int e = take_entry(me, mo);
                if (__half2float(entry_of(part, e)) == end[K - 1] && --take < 0) continue;
                if (e & 1) ko |= 1u << (e >> 1); else ke |= 1u << (e >> 1);
              }
              me = ke; mo = ko;
            }
            even |= me; odd |= mo;
          };
          collect(t, top, [&](int i) { return __low2float(other.v[i]); });
          collect(b, bot, [&](int i) { return -__high2float(other.v[i]); });
#pragma unroll
          for (int a = 0; a < 2 * K; ++a) oi[a] = take_entry(even, odd);
          int own = 0;
#pragma unroll
          for (int a = 0; a < 2 * K; ++a) own += oi[a] < kQgPart;
          before = part == 0 ? 0 : 2 * K - own;
        } else {
          // The sides share entries (or NaN): one after the other, ties to the lower index, the largest K, then the smallest K of what
          // is left, then the bounds of the rest
          int pick[2 * K];
          mn = INFINITY; mx = -INFINITY;
#pragma unroll 1
          for (int n = 0; n <= 2 * K; ++n) {
            int best = -1;
            float v = 0.f;
#pragma unroll 1
            for (int e = 0; e < L; ++e) {
              bool gone = false;
#pragma unroll
              for (int a = 0; a < 2 * K; ++a) gone = gone || (a < n && pick[a] == e);
              if (gone) continue;
              const float x = __half2float(entry_of(e / kQgPart, e % kQgPart));
              if (n == 2 * K) { mn = fminf(mn, x); mx = fmaxf(mx, x); }
              else if (best < 0 || (n < K ? x > v : x < v)) { best = e; v = x; }
            }
#pragma unroll
            for (int a = 0; a < 2 * K; ++a) pick[a] = a == n ? best : pick[a];
          }
#pragma unroll
          for (int a = 0; a < 2 * K; ++a)
#pragma unroll
            for (int b = a + 1; b < 2 * K; ++b) { const int lo = min(pick[a], pick[b]), hi = max(pick[a], pick[b]); pick[a] = lo; pick[b] = hi; }
          int n = 0;
#pragma unroll
          for (int a = 0; a < 2 * K; ++a) oi[a] = kQgPart;
#pragma unroll
          for (int a = 0; a < 2 * K; ++a) {
            if (pick[a] / kQgPart < part) ++before;
            if (pick[a] / kQgPart == part) {
#pragma unroll
              for (int b = 0; b < 2 * K; ++b) oi[b] = b == n ? pick[a] % kQgPart : oi[b];
              ++n;
            }
          }
        }
      }
    }
    auto filtered = [&](int a) { return !kShared || oi[a] < kQgPart; };
    // Eq. 2 on the kept entries: binary32, one rounding per operation
    const float levels = (float)((1 << BITS) - 1);
    const float range = __fsub_rn(mx, mn);
    const float d32 = __fdiv_rn(range, levels);
    const __half d16 = __float2half_rn(d32);
    const float d = __half2float(d16);
    const float inv = d != 0.f ? __fdiv_rn(1.0f, d) : 0.f;
    float dm = 0.f;
    __half ov[2 * K + 1];
    // Stored ahead of the barrier: the next block's copy is requested behind it and does not wait for loads that are still on
    // their way, so everything loaded from the block has to be used before it.
    if constexpr (K > 0) {
#pragma unroll
      for (int a = 0; a < 2 * K; ++a) ov[a] = entry_of(part, kShared ? min(oi[a], kQgPart - 1) : oi[a]);
      __half* dv = reinterpret_cast<__half*>(rec + (SIDE == 0 ? sd.off_koval : sd.off_voval)) + gi * 2 * K + before;
      unsigned char* di = rec + (SIDE == 0 ? sd.off_koidx : sd.off_voidx) + gi * 2 * K + before;
#pragma unroll
      for (int a = 0; a < 2 * K; ++a)
        if (filtered(a)) dm = fmaxf(dm, fabsf(__half2float(ov[a]) - mn));
      if constexpr (!kShared) {
        *reinterpret_cast<__half2*>(dv) = __halves2half2(ov[0], ov[1]);
        *reinterpret_cast<uchar2*>(di) = make_uchar2((unsigned char)oi[0], (unsigned char)oi[1]);
      } else {
#pragma unroll
        for (int a = 0; a < 2 * K; ++a)
          if (filtered(a)) { dv[a] = ov[a]; di[a] = (unsigned char)(part * kQgPart + oi[a]); }
      }
    }
    if (!kShared || part == 0)
      reinterpret_cast<__half2*>(rec + (SIDE == 0 ? sd.off_kscale : sd.off_vscale))[gi] = __halves2half2(d16, __float2half_rn(mn));
    {
      // Non-negative floats order like their bit patterns.
      const float rm = residual_bound(mn, mx, range, d, levels);
      const unsigned int wr = __reduce_max_sync(0xffffffffu, __float_as_uint(rm)), ws = __reduce_max_sync(0xffffffffu, __float_as_uint(d)),
                         wd = __reduce_max_sync(0xffffffffu, __float_as_uint(dm));
      if (lane == 0) {
        atomicMax(&rmax_bits[it & 1], wr);
        atomicMax(&smax_bits[it & 1], ws);
        atomicMax(&dmax_bits[it & 1], wd);
      }
    }
    if (__syncthreads_or(!ok)) {                   // every thread has read the block
      bar_wait(&full, parity ^ 1u);                // gave up, reported below: the copy lands before its memory goes (bounded)
      break;
    }
    if (tid == 0 && it + 1 < count) request(it + 1);
    const float rmax = __uint_as_float(rmax_bits[it & 1]);
    const int er = max(-150, min(130, pow2_exponent(rmax)));
    if (mma_pending) ok = ok && bar_wait(&mma_done, mma_parity);    // the operands may be written, the sums are current
    // accumulator row 32 (warp % 4) + lane, and the columns from c0 on that the warp takes
    const uint32_t sums = tmem + ((uint32_t)(warp % 4 * 32) << 16);
    const int c0 = warp / 4 * (kHeadDim / (kThreads / 128)), c1 = c0 + kHeadDim / (kThreads / 128);
    if (rmax > 0.f) {
      if (!exp_set) {
        exp_cur = er - kQgStart;
        exp_set = true;
      } else if (er > exp_cur + kQgGrow) {         // the same for all threads
        const int e_new = er - kQgStart;
        if (!fresh) {
          tmem_fence_after();
          const float f = exp2_int(2 * (exp_cur - e_new));
#pragma unroll 1
          for (int c = c0; c < c1; c += 32) {
            uint32_t v[32];
            tmem_ld32(v, sums + c);
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) * f);
            tmem_st32(sums + c, v);
          }
          tmem_fence_before();
        }
        exp_cur = e_new;
      }
    }
    // Codes and residuals are computed for every entry as if it were kept.
    const PairQuantSplit quantize(mn, inv, d, levels, exp2_int(-exp_cur));
#pragma unroll
    for (int r8 = 0; r8 < kPartRows / 8; ++r8) {
      unsigned int acc[8];
#pragma unroll
      for (int f = 0; f < F; ++f) {
        const int e = SIDE == 0 ? f * kPartRows + r8 * 8 : r8 / 2 * 16 * F + f * 16 + r8 % 2 * 8;
        uint32_t h[4], l[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          unsigned int k0, k1;
          quantize(xp[e / 2 + k], k0, k1, h[k], l[k]);
          acc[2 * k] = f == 0 ? k0 : k0 * (1u << (BITS * f)) + acc[2 * k];
          acc[2 * k + 1] = f == 0 ? k1 : k1 * (1u << (BITS * f)) + acc[2 * k + 1];
        }
        *reinterpret_cast<uint4*>(op_line + op_at(e)) = make_uint4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<uint4*>(op_line + kOperand + op_at(e)) = make_uint4(l[0], l[1], l[2], l[3]);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) mine[(r8 * 8 + i) * kCodePitch] = (unsigned char)acc[i];
    }
    // the filtered entries: no residual, code zero
#pragma unroll
    for (int a = 0; a < K; ++a) {
      unsigned int c[2];
      uint32_t h, l;
      quantize(__halves2half2(ov[2 * a], ov[2 * a + 1]), c[0], c[1], h, l);
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        if (!filtered(2 * a + b)) continue;
        const int e = oi[2 * a + b], at = op_at(e) + (e & 7) * 2;
        *reinterpret_cast<unsigned short*>(op_line + at) = 0;
        *reinterpret_cast<unsigned short*>(op_line + kOperand + at) = 0;
        unsigned char* byte = mine + code_row(e) * kCodePitch;
        *byte = (unsigned char)(*byte - (c[b] << (BITS * code_field(e))));
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tmem_fence_before();
    __syncthreads();
    if (tid == 0) {
      tmem_fence_after();
      // 128B swizzle, 8-row groups 1 KB apart (stride).  Keys K-major, 64 tokens a row; values MN-major, their 64-channel halves
      // L rows apart (leading).  fp32 accumulator, fp16 operands, M = N = 128.
      constexpr uint64_t kDesc = (SIDE == 0 ? 1ull << 16 : (uint64_t)(L * 128 >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
                                 (1ull << 46) | (2ull << 61);
      constexpr uint32_t kIdesc = (1u << 4) | (SIDE == 0 ? 0u : (1u << 15) | (1u << 16)) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
      const uint64_t dh = kDesc | (smem_addr(op_hi) >> 4), dl = kDesc | (smem_addr(op_lo) >> 4);
#pragma unroll
      for (int k = 0; k < L / 16; ++k) {           // 16 tokens further
        const uint32_t at = (SIDE == 0 ? k / 4 * (kHeadDim * 128) + k % 4 * 32 : k * 2048) >> 4;
        umma_f16(tmem, dh + at, dh + at, kIdesc, fresh && k == 0 ? 0u : 1u);
        umma_f16(tmem, dh + at, dl + at, kIdesc, 1u);
      }
      umma_commit(&mma_done);
      const int s = it & 1;
      reinterpret_cast<float*>(rec)[SIDE] = __uint_as_float(dmax_bits[s]);
      reinterpret_cast<float*>(rec)[2 + SIDE] = __uint_as_float(smax_bits[s]);
      atomicMax(p.Rmax + bhl * 2 + SIDE, rmax_bits[s]);
      dmax_bits[s] = 0u; smax_bits[s] = 0u; rmax_bits[s] = 0u;      // used again two blocks on, behind the next block's first barrier
    }
    if (mma_pending) mma_parity ^= 1u;
    mma_pending = true;
    fresh = false;
    // the codes in fragment order (code_coord_k / code_coord_v)
    unsigned int* dst = reinterpret_cast<unsigned int*>(rec + (SIDE == 0 ? sd.off_kcodes : sd.off_vcodes));
    if (SIDE == 0) {
      // word (w, lane, tau) of a slab: four neighbouring channels of a token in each of its fields; a row of packed bytes holds the
      // channels' codes of F tokens, 64 / F apart
      constexpr int kWords = kSlab * kHeadDim * BITS / 32, kPartSlabs = kPartRows / kSlab;    // words per slab
#pragma unroll
      for (int li = tid; li < L / F / kSlab * kWords; li += kThreads) {
        const int slab = li / kWords, wl = li % kWords;            // slab of rows
        const int w = wl & 3, ln = (wl >> 2) & 31, tau = wl >> 7;
        const int row = slab * kSlab + (ln >> 2) + 8 * (w & 1), ch = 32 * F * tau + 16 * (w >> 1) + 4 * (ln & 3);
        unsigned int v[F];
#pragma unroll
        for (int j = 0; j < F; ++j) v[j] = *reinterpret_cast<const unsigned int*>(codes + row * kCodePitch + ch + 32 * j);
        unsigned int* out = dst + (slab / kPartSlabs * (kQgPart / kSlab) + slab % kPartSlabs) * kWords + wl;
#pragma unroll
        for (int f = 0; f < F; ++f) {
          unsigned int word = 0;
#pragma unroll
          for (int j = 0; j < F; ++j) {
            const unsigned int m = field_of_bytes<BITS>() << (BITS * j);
            word |= (j >= f ? v[j] << (BITS * (j - f)) : v[j] >> (BITS * (f - j))) & m;
          }
          out[f * kPartSlabs * kWords] = word;
        }
      }
    } else {
      // a row of packed bytes is the byte rows of one channel of a tuple: four tokens are a word
      constexpr int kWords = 32 * kHeadDim * BITS / 32;               // words per 32-token chunk
#pragma unroll
      for (int li = tid; li < L / 32 * kWords; li += kThreads) {
        const int chunk = li / kWords, wl = li % kWords;
        const int w = wl & 3, ln = (wl >> 2) & 31, tau = wl >> 7;
        dst[li] = *reinterpret_cast<const unsigned int*>(codes + (tau * 16 + (ln >> 2) + 8 * (w & 1)) * kCodePitch + chunk * 32 +
                                                         16 * (w >> 1) + 4 * (ln & 3));
      }
    }
    if (it + 1 == count || blk + 1 == sd.nblk) {   // the tile's last block in this range: leave the partial
      ok = ok && bar_wait(&mma_done, mma_parity);
      if (p.test_dead_wait && it + 1 == count) ok = bar_wait(&full, parity, 64) && ok;
      tmem_fence_after();
      __syncwarp();
      const size_t at = (size_t)blockIdx.x + bhl + (SIDE == 0 ? 0 : gridDim.x + nbh);
      float* part_sum = p.Gpart + at * (kHeadDim * kHeadDim) + warp % 4 * 32 + lane;
#pragma unroll 1
      for (int c = c0; c < c1; c += 32) {          // row c of the partial gets the accumulator's column c
        uint32_t v[32];
        tmem_ld32(v, sums + c);
#pragma unroll
        for (int i = 0; i < 32; ++i) part_sum[(size_t)(c + i) * kHeadDim] = __uint_as_float(v[i]);
      }
      tmem_fence_before();
      if (tid == 0) p.Gexp[at] = exp_cur;
      fresh = true; exp_set = false; exp_cur = 0;
    }
    if (++blk == sd.nblk) { blk = 0; ++bhl; }
  }
  if (mma_pending) ok = bar_wait(&mma_done, mma_parity) && ok;      // also when a wait gave up: the products end before their operands' memory does
  if (!ok) atomicExch(p.status, -7 /* GEAR_ERR_TIMEOUT */);
  tmem_fence_before();
  __syncthreads();
  if (warp == 0) tmem_free<kHeadDim>(tmem);
  if (SIDE == 1) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// G of every tile from its partials (fixed order), each brought to the tile's power of two; entry (k, i) of a partial counts as the mean
// of (k, i) and (i, k).  A CTA takes a 32 x 32 piece and the one across the diagonal, so that every entry is read once; each
// of its GROUPS times 256 threads takes every GROUPS-th partial: one group where a tile has a few, four where few tiles have up to
// a hundred (one head of 8192 tokens: the whole call 101 -> 67 us).  Bound: the partials' bytes.
constexpr int kQgPieces = kHeadDim / 32, kQgPairs = kQgPieces * (kQgPieces + 1) / 2;
template <int GROUPS>
__global__ void __launch_bounds__(256 * GROUPS) quant_gram_sum_kernel(PiArgs p, int ctas) {
  __shared__ float a_s[GROUPS][32][33], b_s[GROUPS][32][33];
  const int tile = blockIdx.y, bhl = tile >> 1, side = tile & 1, nbh = p.ntiles >> 1;
  int I = 0, J = blockIdx.x;
  while (J >= kQgPieces - I) { J -= kQgPieces - I; ++I; }
  J += I;
  const int x = threadIdx.x & 31, y = (threadIdx.x >> 5) & 7, g = threadIdx.x >> 8;       // column, first row (then every eighth), group
  const long long nblk = p.seg.nblk, blocks = nbh * nblk, b0 = bhl * nblk, b1 = b0 + nblk;
  const int w0 = (int)(((b0 + 1) * ctas + blocks - 1) / blocks - 1), w1 = (int)((b1 * ctas + blocks - 1) / blocks - 1);
  after_previous();
  const int er = pow2_exponent(__uint_as_float(p.Rmax[tile]));
  const size_t at = (size_t)w0 + bhl + (side == 0 ? 0 : ctas + nbh);
  const int aoff = (I * 32 + y) * kHeadDim + J * 32 + x, boff = (J * 32 + y) * kHeadDim + I * 32 + x;
  float a[4] = {0.f, 0.f, 0.f, 0.f}, b[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
  for (int w = g; w <= w1 - w0; w += GROUPS) {
    const float* src = p.Gpart + (at + w) * (kHeadDim * kHeadDim);
    const float s = 0.5f * exp2_int(2 * (p.Gexp[at + w] - er));
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      a[q] = fmaf(__ldcg(src + aoff + q * 8 * kHeadDim), s, a[q]);
      if (I != J) b[q] = fmaf(__ldcg(src + boff + q * 8 * kHeadDim), s, b[q]);
    }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    a_s[g][y + 8 * q][x] = a[q];
    b_s[g][y + 8 * q][x] = I != J ? b[q] : a[q];
  }
  __syncthreads();
  float* G = p.G + (size_t)tile * kHeadDim * kHeadDim;
#pragma unroll
  for (int row = threadIdx.x >> 5; row < 32; row += 8 * GROUPS) {
    float ga = 0.f, gb = 0.f;
#pragma unroll
    for (int q = 0; q < GROUPS; ++q) {
      ga += a_s[q][row][x] + b_s[q][x][row];
      gb += b_s[q][row][x] + a_s[q][x][row];
    }
    G[(I * 32 + row) * kHeadDim + J * 32 + x] = ga;
    if (I != J) G[(J * 32 + row) * kHeadDim + I * 32 + x] = gb;
  }
}

template <int BITS, int SIDE, int L, int K>
static cudaError_t launch_side(const CompressArgs& a, int nbh, int ctas, const CUtensorMap& value_rows, cudaStream_t st) {
  const int smem = qg_smem(BITS, SIDE, L);
  const cudaError_t e = cudaFuncSetAttribute(quant_gram_kernel<BITS, SIDE, L, K>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  return e == cudaSuccess ? launch_dependent(quant_gram_kernel<BITS, SIDE, L, K>, dim3(ctas), qg_threads(L), smem, st, a, nbh, value_rows) : e;
}
template <int BITS, int L, int K>
static cudaError_t launch_sides(const CompressArgs& a, int nbh, int ctas, const CUtensorMap& value_rows, cudaStream_t st) {
  const cudaError_t e = launch_side<BITS, 0, L, K>(a, nbh, ctas, value_rows, st);
  return e == cudaSuccess ? launch_side<BITS, 1, L, K>(a, nbh, ctas, value_rows, st) : e;
}
cudaError_t launch_quant_gram(const CompressArgs& a, const PiArgs& p, int nbh, int sms, cudaStream_t st) {
  const int ctas = qg_split(nbh, a.seg, sms).ctas, k = a.seg.k_k;
  CUtensorMap rows;
  cudaError_t e = make_row_map(&rows, a.V, (long long)nbh * a.seg.n_c);
  if (e != cudaSuccess) return e;
  auto run = [&](auto bits) {
    constexpr int B = decltype(bits)::value;
    if (a.seg.T == 64) return k == 0 ? launch_sides<B, 64, 0>(a, nbh, ctas, rows, st) : launch_sides<B, 64, 1>(a, nbh, ctas, rows, st);
    return k == 0 ? launch_sides<B, 128, 0>(a, nbh, ctas, rows, st) : k == 1 ? launch_sides<B, 128, 1>(a, nbh, ctas, rows, st)
                                                                              : launch_sides<B, 128, 2>(a, nbh, ctas, rows, st);
  };
  e = a.cc.bits == 2 ? run(std::integral_constant<int, 2>()) : run(std::integral_constant<int, 4>());
  if (e != cudaSuccess) return e;
  e = ctas < 8 * nbh ? launch_dependent(quant_gram_sum_kernel<1>, dim3(kQgPairs, p.ntiles), 256, 0, st, p, ctas)
                     : launch_dependent(quant_gram_sum_kernel<4>, dim3(kQgPairs, p.ntiles), 1024, 0, st, p, ctas);
  if (e != cudaSuccess) return e;
  count_launches(3);
  return cudaSuccess;
}

}  // namespace gear
