// GEAR compression of one segment (Algorithm 1, prefill body / buffer flush):
//   quant_pack_kernel : Filter_s (Eq. 4), Quant_b(X - S) (Eq. 2, Eq. 5), packing, residual R = X - D^ - S
//   pi_* kernels      : SVDSolver (Algorithm 2) on every head's residual R_h, batch-wise and head-wise
// All arithmetic that decides a code is a fixed sequence of binary32 operations
// (round-to-nearest-even, no fused multiply-add, no fast-math).
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include "gear_internal.cuh"
#include "gear_pass.cuh"
#include "gear_pi.cuh"
#include "gear_quant.cuh"

namespace gear {

// ---------------------------------------------------------------------------
// Filter + Quant + pack for one block (T tokens x 128 channels) of K or V.
// ---------------------------------------------------------------------------
constexpr int kXPitch = 130;   // halves per row of the fp16 tile in shared memory
constexpr int kRPitch = 129;   // floats per row of the residual tile

struct TopList {
  float v[kMaxOutliers];
  int i[kMaxOutliers];
};

// (value, index) order used by Filter_s: larger value first (smaller for the
// bottom list), then lower index.
template <bool TOP>
__device__ __forceinline__ bool goes_before(float va, int ia, float vb, int ib) {
  if (ib < 0) return ia >= 0;
  if (ia < 0) return false;
  if (TOP ? (va > vb) : (va < vb)) return true;
  return va == vb && ia < ib;
}

template <int KMAX, bool TOP>
__device__ __forceinline__ void list_insert(TopList& l, int k, float v, int idx) {
#pragma unroll
  for (int s = 0; s < KMAX; ++s) {
    if (s < k && goes_before<TOP>(v, idx, l.v[s], l.i[s])) {
      float tv = l.v[s]; int ti = l.i[s];
      l.v[s] = v; l.i[s] = idx;
      v = tv; idx = ti;
    }
  }
}

template <int KMAX>
__device__ __forceinline__ bool list_has(const TopList& l, int k, int idx) {
  bool h = false;
#pragma unroll
  for (int s = 0; s < KMAX; ++s) h |= (s < k && l.i[s] == idx);
  return h;
}

struct GroupResult {
  __half scale, zero;
  float dmax;   // max |x - zero| over the group's outliers
};

// One quantization group of `len` entries reached through x_at(e); writes the
// code and residual of every entry through put(e, code, resid) and the sorted
// outlier list (in-group index ascending) through put_out(slot, idx, value).
template <int BITS, int KMAX, class XAt, class Put, class PutOut>
__device__ __forceinline__ GroupResult process_group(int len, int k, XAt x_at, Put put, PutOut put_out) {
  TopList top, bot;
#pragma unroll
  for (int s = 0; s < KMAX; ++s) { top.v[s] = 0.f; top.i[s] = -1; bot.v[s] = 0.f; bot.i[s] = -1; }
  float mn = INFINITY, mx = -INFINITY;
  if (KMAX == 1 && k == 1) {
    // One outlier per side: a single pass finds the first maximum, the first minimum and the second largest /
    // second smallest instances, which bound the kept entries.  (The first maximum is also the first minimum
    // only when all entries are equal; the bottom entry is then the next index.)
    float max1 = -INFINITY, max2 = -INFINITY, min1 = INFINITY, min2 = INFINITY;
    int imax = 0, imin = 0;
    for (int e = 0; e < len; ++e) {
      const float x = x_at(e);
      if (x > max1) { max2 = max1; max1 = x; imax = e; } else if (x > max2) { max2 = x; }
      if (x < min1) { min2 = min1; min1 = x; imin = e; } else if (x < min2) { min2 = x; }
    }
    if (imin == imax) imin = 1;
    top.v[0] = max1; top.i[0] = imax;
    bot.v[0] = min1; bot.i[0] = imin;
    mn = min2; mx = max2;
  } else {
    if (k > 0) {
      for (int e = 0; e < len; ++e) list_insert<KMAX, true>(top, k, x_at(e), e);
      for (int e = 0; e < len; ++e)
        if (!list_has<KMAX>(top, k, e)) list_insert<KMAX, false>(bot, k, x_at(e), e);
    }
    for (int e = 0; e < len; ++e) {
      if (k > 0 && (list_has<KMAX>(top, k, e) || list_has<KMAX>(bot, k, e))) continue;
      const float x = x_at(e);
      mn = fminf(mn, x);
      mx = fmaxf(mx, x);
    }
  }
  // Eq. 2 on the kept entries: binary32, one rounding per operation.
  const float levels = (float)((1 << BITS) - 1);
  const float range = __fsub_rn(mx, mn);
  const float d32 = __fdiv_rn(range, levels);
  const __half d16 = __float2half_rn(d32);
  const float d = __half2float(d16);
  const float inv = d != 0.f ? __fdiv_rn(1.0f, d) : 0.f;
  for (int e = 0; e < len; ++e) {
    const float x = x_at(e);
    const bool out = k > 0 && (list_has<KMAX>(top, k, e) || list_has<KMAX>(bot, k, e));
    int code = 0;
    float resid = 0.f;
    if (!out) {
      if (d != 0.f) {
        const float t = __fmul_rn(__fsub_rn(x, mn), inv);
        code = (int)fminf(fmaxf(rintf(t), 0.f), levels);
      }
      resid = x - fmaf((float)code, d, mn);
    }
    put(e, code, resid);
  }
  GroupResult r;
  r.scale = d16;
  r.zero = __float2half_rn(mn);
  r.dmax = 0.f;
  if (k > 0) {
    // merge the two lists by index: rank of each entry among the 2k
#pragma unroll
    for (int a = 0; a < 2 * KMAX; ++a) {
      const bool from_top = a < KMAX;
      const int s = from_top ? a : a - KMAX;
      if (s >= k) continue;
      const int ia = from_top ? top.i[s] : bot.i[s];
      const float va = from_top ? top.v[s] : bot.v[s];
      int rank = 0;
#pragma unroll
      for (int b = 0; b < KMAX; ++b) {
        rank += (b < k && top.i[b] < ia);
        rank += (b < k && bot.i[b] < ia);
      }
      put_out(rank, ia, va);
      r.dmax = fmaxf(r.dmax, fabsf(va - mn));
    }
  }
  return r;
}

// Pack the codes of one block (T tokens x 128 channels, xs[token * kXPitch + channel]) into the fragment order of
// the integer tensor-core product (gear_layout.cuh); one 32-bit word per thread and step, stores coalesced.
template <int BITS>
__device__ __forceinline__ void pack_block_codes(const unsigned short* xs, int T, int side, unsigned int* dst, int tid,
                                                 int nthreads) {
  constexpr int F = 8 / BITS;
  if (side == 0) {
    constexpr int kWords = kSlab * kHeadDim * BITS / 32;            // words per slab
    for (int li = tid; li < ((T + kSlab - 1) / kSlab) * kWords; li += nthreads) {
      const int slab = li / kWords, wl = li % kWords;
      const int w = wl & 3, lane = (wl >> 2) & 31, tau = wl >> 7;
      unsigned int word = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < F; ++j) {
          int tok, ch;
          code_coord_k(BITS, lane, tau, w, i, j, tok, ch);
          tok += slab * kSlab;
          if (tok < T) word |= (unsigned int)xs[tok * kXPitch + ch] << (8 * i + BITS * j);
        }
      dst[li] = word;
    }
  } else {
    constexpr int kWords = 32 * kHeadDim * BITS / 32;               // words per 32-token chunk
    const int nchunk = (T + 31) / 32;
    for (int li = tid; li < nchunk * kWords; li += nthreads) {
      const int chunk = li / kWords, wl = li % kWords;
      const int w = wl & 3, lane = (wl >> 2) & 31, tau = wl >> 7;
      unsigned int word = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < F; ++j) {
          int tok, ch;
          code_coord_v(BITS, lane, tau, w, i, j, tok, ch);
          tok += chunk * 32;
          if (tok < T) word |= (unsigned int)xs[tok * kXPitch + ch] << (8 * i + BITS * j);
        }
      dst[li] = word;
    }
  }
}

template <int BITS, int KMAX>
__global__ void __launch_bounds__(128) quant_pack_kernel(CompressArgs p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const SegDesc& sd = p.seg;
  const int T = sd.T;
  const int side = blockIdx.z + p.side0, bhl = blockIdx.y, blk = blockIdx.x, tid = threadIdx.x;
  unsigned short* xs = reinterpret_cast<unsigned short*>(smem_raw);   // fp16 bits of the block; each entry is replaced by its code
  float* rs = reinterpret_cast<float*>(smem_raw + round_up(T * kXPitch * 2, 16));
  auto x_of = [&](int idx) { return __half2float(__ushort_as_half(xs[idx])); };
  __shared__ unsigned int dmax_bits, smax_bits;
  if (tid == 0) { dmax_bits = 0u; smax_bits = 0u; }
  after_previous();

  const __half* X = (side == 0 ? p.K : p.V) + ((size_t)bhl * sd.n_c + (size_t)blk * T) * kHeadDim;
  for (int i = tid; i < T * 16; i += 128) {
    const int row = i >> 4, c = i & 15;
    const uint4 v = *reinterpret_cast<const uint4*>(X + row * kHeadDim + c * 8);
    unsigned int* dst = reinterpret_cast<unsigned int*>(xs + row * kXPitch + c * 8);
    dst[0] = v.x; dst[1] = v.y; dst[2] = v.z; dst[3] = v.w;
  }
  __syncthreads();

  unsigned char* rec = p.arena + sd.seg_base + (size_t)(p.bh0 + bhl) * sd.bh_stride + sd.bfac_bytes +
                       (size_t)blk * sd.rec_bytes;
  float my_dmax = 0.f, my_smax = 0.f;
  if (side == 0) {
    // keys: one group per channel over the T tokens of the block (per-channel grouping)
    const int j = tid;
    const int k = sd.k_k;
    __half* oval = reinterpret_cast<__half*>(rec + sd.off_koval) + j * 2 * k;
    unsigned char* oidx = rec + sd.off_koidx + j * 2 * k;
    GroupResult g = process_group<BITS, KMAX>(
        T, k, [&](int e) { return x_of(e * kXPitch + j); },
        [&](int e, int code, float r) { xs[e * kXPitch + j] = (unsigned short)code; rs[e * kRPitch + j] = r; },
        [&](int slot, int idx, float v) { oval[slot] = __float2half_rn(v); oidx[slot] = (unsigned char)idx; });
    reinterpret_cast<__half2*>(rec + sd.off_kscale)[j] = __halves2half2(g.scale, g.zero);
    my_dmax = g.dmax;
    my_smax = __half2float(g.scale);
  } else {
    // values: one group per token over g_V consecutive channels (per-token grouping)
    const int k = p.cc.k_v, gv = p.cc.g_v, ngv = p.cc.ngv;
    for (int gi = tid; gi < T * ngv; gi += 128) {
      const int tok = gi / ngv, c = gi % ngv;
      __half* oval = reinterpret_cast<__half*>(rec + sd.off_voval) + gi * 2 * k;
      unsigned char* oidx = rec + sd.off_voidx + gi * 2 * k;
      GroupResult g = process_group<BITS, KMAX>(
          gv, k, [&](int e) { return x_of(tok * kXPitch + c * gv + e); },
          [&](int e, int code, float r) {
            xs[tok * kXPitch + c * gv + e] = (unsigned short)code;
            rs[tok * kRPitch + c * gv + e] = r;
          },
          [&](int slot, int idx, float v) { oval[slot] = __float2half_rn(v); oidx[slot] = (unsigned char)idx; });
      reinterpret_cast<__half2*>(rec + sd.off_vscale)[gi] = __halves2half2(g.scale, g.zero);
      my_dmax = fmaxf(my_dmax, g.dmax);
      my_smax = fmaxf(my_smax, __half2float(g.scale));
    }
  }
  atomicMax(&dmax_bits, __float_as_uint(my_dmax));   // non-negative floats order like their bit patterns
  atomicMax(&smax_bits, __float_as_uint(my_smax));
  __syncthreads();
  if (tid == 0) {
    reinterpret_cast<float*>(rec)[side] = __uint_as_float(dmax_bits);
    reinterpret_cast<float*>(rec)[2 + side] = __uint_as_float(smax_bits);
  }

  // pack the codes into mma-fragment order
  pack_block_codes<BITS>(xs, T, side, reinterpret_cast<unsigned int*>(rec + (side == 0 ? sd.off_kcodes : sd.off_vcodes)),
                         tid, 128);
  // residual tile -> workspace (only needed when a low-rank part is fitted)
  if (p.R != nullptr) {
    float* R = p.R + (((size_t)bhl * 2 + side) * sd.n_c + (size_t)blk * T) * kHeadDim;
    float rmax = 0.f;
    for (int i = tid; i < T * kHeadDim; i += 128) {
      const float v = rs[(i >> 7) * kRPitch + (i & 127)];
      R[i] = v;
      rmax = fmaxf(rmax, fabsf(v));
    }
    // the largest residual magnitude of the (batch, head, side) tile: the power iteration scales by it
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rmax = fmaxf(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
    if ((tid & 31) == 0) atomicMax(p.Rmax + bhl * 2 + side, __float_as_uint(rmax));
  }
}

// ---------------------------------------------------------------------------
// The same step for groups of L = 32, 64 or 128 entries with at most one outlier per side (64 at s <= 3.1 %, 128 at s <= 1.5 %)
// with the group in registers: a thread owns one group (keys: a channel's L tokens, read as a column of a block of L tokens;
// values: L consecutive channels of a token; a block has 128 groups), walks it in fully unrolled loops, stores the residual itself and
// leaves only the codes in shared memory, one byte each, transposed so that the packing step fetches the four codes
// of an output byte row with one 32-bit load.  Every code, scale, outlier and residual is bit-identical to
// quant_pack_kernel: the operations on a group are the same binary32 sequence.
//
// Bound: instruction issue (about thirty instructions per pair of entries), with the residual's bytes not far behind.  CTAs
// are persistent and the block after the one being worked on comes into shared memory by a bulk copy, so that no warp
// waits for a load it has just issued; the entries' arithmetic runs on pairs (f32x2); a value group reads and writes its
// own 32-byte sectors (256-bit stores), so the residual takes no way through shared memory.  Against one CTA per block,
// scalar arithmetic and a residual staged through shared memory (2 bits, 8 x 32 heads x 4096): keys 181 -> 153 us, values
// 261 -> 168 us; 4 bits, 16 x 40 heads x 8192: 469 -> 415 and 652 -> 434 us.  Against quant_pack_kernel (8 x 32 heads x 4096,
// keys / values): groups of 32 283 / 298 -> 165 / 175 us, of 64 without outliers 266 / 299 -> 150 / 159, of 128 with one
// outlier 581 / 604 -> 172 / 169, without 441 / 480 -> 146 / 162, values of per-vector keys 517 -> 209.  All with the residual
// stored; key blocks of 64 and 128 tokens with value groups as long come here without a low-rank part only (quant_gram_kernel
// takes the others), where it is not.
// ---------------------------------------------------------------------------
constexpr int kCodePitchK = kHeadDim + 4;   // bytes per token row of the key codes  [token][channel]
// CTAs per SM.  L = 64 (128 registers): five or six are slower, keys 153 -> 166 -> 196 us, values 168 -> 169 -> 171 (8 x 32 heads
// x 4096).  Columns of 128 tokens spill at four (240 us against 204 with two outliers, 4 x 8 heads x 32768).  L = 32: five,
// six and eight are alike.
__host__ __device__ constexpr int fast_ctas_per_sm(int side, int len) {
  return len == 32 ? 6 : len == kHeadDim && side == 0 ? 3 : 4;
}

// The blocks that a persistent CTA works on, one after the other through one buffer in shared memory: the copy of the next
// block is requested as soon as every thread is done with the present one.
struct BlockFeed {
  unsigned char* tile; uint64_t* full;
  const __half* X; int n_c, nblk, T, total;
  uint32_t parity;
  __device__ __forceinline__ void request(int item) const {
    const int bhl = item / nblk, blk = item - bhl * nblk;
    bar_expect(full, T * kHeadDim * 2);
    bulk_copy(tile, X + ((size_t)bhl * n_c + (size_t)blk * T) * kHeadDim, T * kHeadDim * 2, full);
  }
};

template <int BITS, int SIDE, int L, int K>
__global__ void __launch_bounds__(128, fast_ctas_per_sm(SIDE, L)) quant_fast_kernel(CompressArgs p, int nbh) {
  constexpr int F = 8 / BITS, side = SIDE, kGroups = kHeadDim / L, kPieces = L / 8;
  constexpr int kCodePitchV = L + 4;               // bytes per channel row of the value codes [channel][token]
  extern __shared__ __align__(128) unsigned char tile[];            // the block's T x 128 fp16 entries
  __shared__ __align__(16) unsigned char codes[SIDE == 0 ? L * kCodePitchK : kHeadDim * kCodePitchV];
  __shared__ uint64_t full;
  __shared__ unsigned int dmax_bits, smax_bits, rmax_bits;
  const SegDesc& sd = p.seg;
  const int tid = threadIdx.x;
  const int T = SIDE == 1 && L == kHeadDim ? sd.T : L;              // tokens of a block; values: 128 / L groups each
  const bool active = L < kHeadDim || SIDE == 0 || tid < T;         // a thread per group
  BlockFeed feed{tile, &full, side == 0 ? p.K : p.V, sd.n_c, sd.nblk, T, sd.nblk * nbh, 0u};
  // The values' CTAs run beside the keys' and wait at their end (see quant_gram_kernel); without keys in front of them (per-vector
  // key groups) the kernel in front may be the one that writes V, and the keys' kernel starts at their end (launch_kcvt_keys).
  if (SIDE == 0) after_previous();
  else if (p.side0 == 1) asm volatile("griddepcontrol.wait;" ::: "memory");
  else asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (tid == 0) {
    dmax_bits = 0u; smax_bits = 0u; rmax_bits = 0u;
    bar_init(&full);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if ((int)blockIdx.x < feed.total) feed.request(blockIdx.x);
  }
  __syncthreads();
  const __half* group = reinterpret_cast<const __half*>(tile) + (side == 0 ? tid : tid * L);   // entry e: group[e * step]
  constexpr int step = SIDE == 0 ? kHeadDim : 1;
  // values: a thread starts with another 16-byte piece than the neighbours whose groups lie in the same banks
  const int rot = SIDE == 0 ? 0 : L == 32 ? (tid >> 1) & 3 : tid & 7;

  for (int item = blockIdx.x; item < feed.total; item += gridDim.x) {
    const int bhl = item / sd.nblk, blk = item - bhl * sd.nblk;
    const bool ok = bar_wait(&full, feed.parity);
    feed.parity ^= 1u;
    float* R = p.R ? p.R + (((size_t)bhl * 2 + side) * sd.n_c + (size_t)blk * T) * kHeadDim : nullptr;
    unsigned char* rec = p.arena + sd.seg_base + (size_t)(p.bh0 + bhl) * sd.bh_stride + sd.bfac_bytes +
                         (size_t)blk * sd.rec_bytes;

    // the group as packed pairs: keys entries 2q, 2q + 1; values the same, in pieces of eight entries from piece `rot` on
    __half2 xp[L / 2];
    if (side == 0) {
#pragma unroll
      for (int q = 0; q < L / 2; ++q) xp[q] = __halves2half2(group[(2 * q) * step], group[(2 * q + 1) * step]);
    } else {
      const uint4* src = reinterpret_cast<const uint4*>(group);
#pragma unroll
      for (int q = 0; q < kPieces; ++q) {
        const uint4 v = active ? src[(q + rot) & (kPieces - 1)] : make_uint4(0u, 0u, 0u, 0u);
        xp[4 * q] = *reinterpret_cast<const __half2*>(&v.x);
        xp[4 * q + 1] = *reinterpret_cast<const __half2*>(&v.y);
        xp[4 * q + 2] = *reinterpret_cast<const __half2*>(&v.z);
        xp[4 * q + 3] = *reinterpret_cast<const __half2*>(&v.w);
      }
    }
    float mx, mn;
    int imax, imin;
    filter_one<L, K>(xp, 4 * rot, mn, mx, imax, imin);
    // Eq. 2 on the kept entries: binary32, one rounding per operation
    const float levels = (float)((1 << BITS) - 1);
    const float range = __fsub_rn(mx, mn);
    const float d32 = __fdiv_rn(range, levels);
    const __half d16 = __float2half_rn(d32);
    const float d = __half2float(d16);
    const float inv = d != 0.f ? __fdiv_rn(1.0f, d) : 0.f;
    // The group's scale, zero point and its two outliers (in-group index ascending), ahead of the barrier: the next block's copy is
    // requested behind it and does not wait for loads from this one that are still on their way, so everything loaded has to
    // be used before it.  The two stores depend on all of it.
    __half vmax = __ushort_as_half(0), vmin = vmax;
    if (active) {
      if (K == 1) {
        vmax = group[imax * step];
        vmin = group[imin * step];
        const bool max_first = imax < imin;
        const __half2 ov = max_first ? __halves2half2(vmax, vmin) : __halves2half2(vmin, vmax);
        const uchar2 oi = max_first ? make_uchar2((unsigned char)imax, (unsigned char)imin)
                                    : make_uchar2((unsigned char)imin, (unsigned char)imax);
        reinterpret_cast<__half2*>(rec + (side == 0 ? sd.off_koval : sd.off_voval))[tid] = ov;
        reinterpret_cast<uchar2*>(rec + (side == 0 ? sd.off_koidx : sd.off_voidx))[tid] = oi;
      }
      reinterpret_cast<__half2*>(rec + (side == 0 ? sd.off_kscale : sd.off_vscale))[tid] = __halves2half2(d16, __float2half_rn(mn));
    }
    if (__syncthreads_or(!ok)) {              // every thread has read the block
      if (tid == 0) atomicExch(p.status, -7 /* GEAR_ERR_TIMEOUT */);
      bar_wait(&full, feed.parity ^ 1u);       // the copy lands before its memory goes (bounded)
      break;
    }
    if (tid == 0 && item + (int)gridDim.x < feed.total) feed.request(item + gridDim.x);
    // Codes and residuals are computed for every entry as if it were kept; the two filtered entries are cleared afterwards.
    const PairQuant quantize(mn, inv, d, levels);
    if (side == 0) {
#pragma unroll
      for (int q = 0; q < L / 2; ++q) {
        unsigned int c0, c1;
        const float2 r = quantize(__half22float2(xp[q]), c0, c1);
        codes[(2 * q) * kCodePitchK + tid] = (unsigned char)c0;
        codes[(2 * q + 1) * kCodePitchK + tid] = (unsigned char)c1;
        if (R != nullptr) {
          R[(2 * q) * kHeadDim + tid] = r.x;
          R[(2 * q + 1) * kHeadDim + tid] = r.y;
        }
      }
      if (K == 1) {
        codes[imax * kCodePitchK + tid] = 0;
        codes[imin * kCodePitchK + tid] = 0;
        if (R != nullptr) {
          R[imax * kHeadDim + tid] = 0.f;
          R[imin * kHeadDim + tid] = 0.f;
        }
      }
    } else if (active) {
      const int tok = tid / kGroups;
      unsigned char* mine = codes + (tid % kGroups) * L * kCodePitchV + tok;
#pragma unroll
      for (int q = 0; q < kPieces; ++q) {
        const int piece = (q + rot) & (kPieces - 1);
        unsigned char* cp = mine + piece * 8 * kCodePitchV;
        float2 r[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          unsigned int c0, c1;
          r[k] = quantize(__half22float2(xp[4 * q + k]), c0, c1);
          cp[(2 * k) * kCodePitchV] = (unsigned char)c0;
          cp[(2 * k + 1) * kCodePitchV] = (unsigned char)c1;
        }
        if (R != nullptr) store8(R + tid * L + piece * 8, r);
      }
      if (K == 1) {
        mine[imax * kCodePitchV] = 0;
        mine[imin * kCodePitchV] = 0;
        if (R != nullptr) {
          R[tid * L + imax] = 0.f;
          R[tid * L + imin] = 0.f;
        }
      }
    }
    // a bound on the group's residuals instead of their maximum (it only picks the power of two the power iteration scales by)
    float rmax = active ? residual_bound(mn, mx, range, d, levels) : 0.f;
    {
      float dm = K == 1 && active ? fmaxf(fabsf(__half2float(vmax) - mn), fabsf(__half2float(vmin) - mn)) : 0.f;
      float sm = active ? d : 0.f;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        dm = fmaxf(dm, __shfl_xor_sync(0xffffffffu, dm, o));
        sm = fmaxf(sm, __shfl_xor_sync(0xffffffffu, sm, o));
        rmax = fmaxf(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
      }
      if ((tid & 31) == 0) {                   // non-negative floats order like their bit patterns
        atomicMax(&dmax_bits, __float_as_uint(dm));
        atomicMax(&smax_bits, __float_as_uint(sm));
        atomicMax(&rmax_bits, __float_as_uint(rmax));
      }
    }
    __syncthreads();
    if (tid == 0) {
      reinterpret_cast<float*>(rec)[side] = __uint_as_float(dmax_bits);
      reinterpret_cast<float*>(rec)[2 + side] = __uint_as_float(smax_bits);
      if (R != nullptr) atomicMax(p.Rmax + bhl * 2 + side, rmax_bits);
      dmax_bits = 0u; smax_bits = 0u; rmax_bits = 0u;       // the next updates come behind the next block's first barrier
    }
    // pack the codes into mma-fragment order (code_coord_k / code_coord_v): the four codes of a byte row are neighbours
    // in shared memory, a field of the word is one 32-bit load shifted into place
    unsigned int* dst = reinterpret_cast<unsigned int*>(rec + (side == 0 ? sd.off_kcodes : sd.off_vcodes));
    if (side == 0) {
      constexpr int kWords = kSlab * kHeadDim * BITS / 32;            // words per slab
      for (int li = tid; li < (L / kSlab) * kWords; li += 128) {
        const int slab = li / kWords, wl = li % kWords;
        const int w = wl & 3, lane = (wl >> 2) & 31, tau = wl >> 7;
        const int tok = slab * kSlab + (lane >> 2) + 8 * (w & 1);
        const int ch = 32 * F * tau + 16 * (w >> 1) + 4 * (lane & 3);
        unsigned int word = 0;
#pragma unroll
        for (int j = 0; j < F; ++j)
          word |= *reinterpret_cast<const unsigned int*>(&codes[tok * kCodePitchK + ch + 32 * j]) << (BITS * j);
        dst[li] = word;
      }
    } else {
      constexpr int kWords = 32 * kHeadDim * BITS / 32;               // words per 32-token chunk
      for (int li = tid; li < (T / 32) * kWords; li += 128) {
        const int chunk = li / kWords, wl = li % kWords;
        const int w = wl & 3, lane = (wl >> 2) & 31, tau = wl >> 7;
        const int ch = 16 * F * tau + (lane >> 2) + 8 * (w & 1);
        const int tok = chunk * 32 + 16 * (w >> 1) + 4 * (lane & 3);
        unsigned int word = 0;
#pragma unroll
        for (int j = 0; j < F; ++j)
          word |= *reinterpret_cast<const unsigned int*>(&codes[(ch + 16 * j) * kCodePitchV + tok]) << (BITS * j);
        dst[li] = word;
      }
    }
  }
  if (SIDE == 1) after_previous();
}

// ---------------------------------------------------------------------------
// Groups of 128 entries with two outliers per side (g = 128 at s = 2 %: keys in blocks of 128 tokens, values one
// group per token), again with the group in registers.  Per half of the packed pairs a chain keeps the three largest
// and three smallest instances; the halves are merged; the entries above / equal to the second largest instance (and
// below / equal to the second smallest) are found as bit masks, which give the two filtered entries per side in
// (value, index) order.  A group in which the two sides would share an entry (nearly constant groups) takes the
// general routine instead.  Same binary32 sequence per entry as everywhere else.  Bound and layout as above (2 bits, 4 x 8
// heads x 32768 with the residual stored: keys 279 -> 204 us, values 290 -> 184 us; today that is the values of per-vector keys alone).
// ---------------------------------------------------------------------------
constexpr int kFast2Len = 128;
constexpr int kCodePitch2 = kFast2Len + 4;

// first set entry of the pair of 64-bit masks (even entries, odd entries), removed from them; 2 * 64 if none
__device__ __forceinline__ int take_first(unsigned long long& even, unsigned long long& odd) {
  const int fe = even ? 2 * (__ffsll((long long)even) - 1) : 2 * 64;
  const int fo = odd ? 2 * (__ffsll((long long)odd) - 1) + 1 : 2 * 64;
  if (fe < fo) { even &= even - 1; return fe; }
  if (fo < 2 * 64) odd &= odd - 1;
  return fo;
}
// four accumulators (bit q of the low / high half word: even / odd entry of pair 16 w + q) -> the two 64-bit masks
__device__ __forceinline__ void masks_of(const unsigned int (&a)[4], unsigned long long& even, unsigned long long& odd) {
  const unsigned int e0 = __byte_perm(a[0], a[1], 0x5410), e1 = __byte_perm(a[2], a[3], 0x5410);
  const unsigned int o0 = __byte_perm(a[0], a[1], 0x7632), o1 = __byte_perm(a[2], a[3], 0x7632);
  even = ((unsigned long long)e1 << 32) | e0;
  odd = ((unsigned long long)o1 << 32) | o0;
}
// the three largest of six values (with multiplicity), in order
__device__ __forceinline__ void top3_of6(float (&v)[6], float (&out)[3]) {
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    float m = v[0];
#pragma unroll
    for (int i = 1; i < 6; ++i) m = fmaxf(m, v[i]);
    out[r] = m;
    bool gone = false;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      const bool hit = !gone && v[i] == m;
      v[i] = hit ? -INFINITY : v[i];
      gone = gone || hit;
    }
  }
}

template <int BITS, int SIDE>
__global__ void __launch_bounds__(128, fast_ctas_per_sm(SIDE, kFast2Len)) quant_fast2_kernel(CompressArgs p, int nbh) {
  constexpr int L = kFast2Len, F = 8 / BITS;
  extern __shared__ __align__(128) unsigned char tile[];            // the block's T x 128 fp16 entries
  __shared__ __align__(16) unsigned char codes[L * kCodePitch2];    // keys [token][channel], values [channel][token]
  __shared__ uint64_t full;
  __shared__ unsigned int dmax_bits, smax_bits, rmax_bits;
  const SegDesc& sd = p.seg;
  const int T = sd.T;                               // keys: 128; values: tokens (= groups) of the block
  const int tid = threadIdx.x;
  BlockFeed feed{tile, &full, SIDE == 0 ? p.K : p.V, sd.n_c, sd.nblk, T, sd.nblk * nbh, 0u};
  // The values' CTAs run beside the keys' and wait at their end (see quant_gram_kernel); without keys in front of them (per-vector
  // key groups) the kernel in front may be the one that writes V, and the keys' kernel starts at their end (launch_kcvt_keys).
  if (SIDE == 0) after_previous();
  else if (p.side0 == 1) asm volatile("griddepcontrol.wait;" ::: "memory");
  else asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (tid == 0) {
    dmax_bits = 0u; smax_bits = 0u; rmax_bits = 0u;
    bar_init(&full);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if ((int)blockIdx.x < feed.total) feed.request(blockIdx.x);
  }
  __syncthreads();
  const int first = SIDE == 0 ? tid : tid * kHeadDim;      // element e of the group: X[first + e * step]
  constexpr int step = SIDE == 0 ? kHeadDim : 1;
  const __half* group = reinterpret_cast<const __half*>(tile) + first;
  const int rot = SIDE == 0 ? 0 : tid & 7;        // values: a thread starts with another 16-byte piece than its neighbours
  // where code / residual of element e go
  auto code_at = [&](int e) -> unsigned char& { return codes[e * kCodePitch2 + tid]; };   // row: token (keys) / channel (values)
  const bool active = SIDE == 0 || tid < T;

  for (int item = blockIdx.x; item < feed.total; item += gridDim.x) {
    const int bhl = item / sd.nblk, blk = item - bhl * sd.nblk;
    const bool ok = bar_wait(&full, feed.parity);
    feed.parity ^= 1u;
    const __half* X = (SIDE == 0 ? p.K : p.V) + ((size_t)bhl * sd.n_c + (size_t)blk * T) * kHeadDim;
    float* R = p.R ? p.R + (((size_t)bhl * 2 + SIDE) * sd.n_c + (size_t)blk * T) * kHeadDim : nullptr;
    unsigned char* rec = p.arena + sd.seg_base + (size_t)(p.bh0 + bhl) * sd.bh_stride + sd.bfac_bytes +
                         (size_t)blk * sd.rec_bytes;
    unsigned char* orec_v = rec + (SIDE == 0 ? sd.off_koval : sd.off_voval) + tid * 8;
    unsigned char* orec_i = rec + (SIDE == 0 ? sd.off_koidx : sd.off_voidx) + tid * 4;
    __half2 xp[L / 2];
    int it[2] = {0, 0}, ib[2] = {0, 0};
    float top[3], bot[3];
    unsigned short ov[4];
    int oi[4] = {0, 0, 0, 0};
    if (active) {
      if (SIDE == 0) {
#pragma unroll
        for (int q = 0; q < L / 2; ++q) xp[q] = __halves2half2(group[(2 * q) * step], group[(2 * q + 1) * step]);
      } else {
        const uint4* src = reinterpret_cast<const uint4*>(group);
#pragma unroll
        for (int q = 0; q < L / 8; ++q) {
          const uint4 v = src[(q + rot) & 15];
          xp[4 * q] = *reinterpret_cast<const __half2*>(&v.x);
          xp[4 * q + 1] = *reinterpret_cast<const __half2*>(&v.y);
          xp[4 * q + 2] = *reinterpret_cast<const __half2*>(&v.z);
          xp[4 * q + 3] = *reinterpret_cast<const __half2*>(&v.w);
        }
      }
      // the three largest / smallest instances of the even and of the odd entries, then of all
      {
        const __half2 ninf = __float2half2_rn(-INFINITY), pinf = __float2half2_rn(INFINITY);
        __half2 M1 = ninf, M2 = ninf, M3 = ninf, m1 = pinf, m2 = pinf, m3 = pinf;
#pragma unroll
        for (int q = 0; q < L / 2; ++q) {
          const __half2 t = __hmin2(xp[q], M1);
          M1 = __hmax2(M1, xp[q]);
          const __half2 u = __hmin2(t, M2);
          M2 = __hmax2(M2, t);
          M3 = __hmax2(M3, u);
          const __half2 tb = __hmax2(xp[q], m1);
          m1 = __hmin2(m1, xp[q]);
          const __half2 ub = __hmax2(tb, m2);
          m2 = __hmin2(m2, tb);
          m3 = __hmin2(m3, ub);
        }
        float v[6] = {__low2float(M1), __low2float(M2), __low2float(M3), __high2float(M1), __high2float(M2), __high2float(M3)};
        top3_of6(v, top);
        float w[6] = {-__low2float(m1), -__low2float(m2), -__low2float(m3), -__high2float(m1), -__high2float(m2), -__high2float(m3)};
        top3_of6(w, bot);
        bot[0] = -bot[0]; bot[1] = -bot[1]; bot[2] = -bot[2];
      }
      // entries above / equal to the second largest instance, below / equal to the second smallest
      {
        const __half2 vT = __float2half2_rn(top[1]), vB = __float2half2_rn(bot[1]);
        unsigned int gt[4] = {0u, 0u, 0u, 0u}, et[4] = {0u, 0u, 0u, 0u}, lt[4] = {0u, 0u, 0u, 0u}, eb[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int q = 0; q < L / 2; ++q) {
          const unsigned int bit = 0x00010001u << (q & 15);
          gt[q >> 4] |= __hgt2_mask(xp[q], vT) & bit;
          et[q >> 4] |= __heq2_mask(xp[q], vT) & bit;
          lt[q >> 4] |= __hlt2_mask(xp[q], vB) & bit;
          eb[q >> 4] |= __heq2_mask(xp[q], vB) & bit;
        }
        unsigned long long ge, go, ee, eo;
        auto in_order = [&](unsigned long long m) {            // values: the pieces back in order
          return SIDE == 0 || rot == 0 ? m : (m << (4 * rot)) | (m >> (64 - 4 * rot));
        };
        auto masks = [&](const unsigned int (&acc)[4], unsigned long long& even, unsigned long long& odd) {
          masks_of(acc, even, odd);
          even = in_order(even); odd = in_order(odd);
        };
        masks(gt, ge, go); masks(et, ee, eo);
        it[0] = take_first(ge, go);                      // the one entry above the second largest instance, if any
        if (it[0] >= L) it[0] = take_first(ee, eo);
        it[1] = take_first(ee, eo);
        masks(lt, ge, go); masks(eb, ee, eo);
        ib[0] = take_first(ge, go);
        if (ib[0] >= L) ib[0] = take_first(ee, eo);
        ib[1] = take_first(ee, eo);
      }
      // the four filtered entries, in-group index ascending
      oi[0] = it[0]; oi[1] = it[1]; oi[2] = ib[0]; oi[3] = ib[1];
      auto order = [&](int a, int b) { if (oi[a] > oi[b]) { const int t = oi[a]; oi[a] = oi[b]; oi[b] = t; } };
      order(0, 1); order(2, 3); order(0, 2); order(1, 3); order(1, 2);
#pragma unroll
      for (int a = 0; a < 4; ++a) ov[a] = __half_as_ushort(group[min(oi[a], L - 1) * step]);
      // stored ahead of the barrier, so that all loads from the block have returned (see quant_fast_kernel); a group that takes
      // the general routine below overwrites them
      *reinterpret_cast<uint2*>(orec_v) = make_uint2(ov[0] | ((unsigned int)ov[1] << 16), ov[2] | ((unsigned int)ov[3] << 16));
      *reinterpret_cast<unsigned int*>(orec_i) = (unsigned int)oi[0] | ((unsigned int)oi[1] << 8) |
                                                 ((unsigned int)oi[2] << 16) | ((unsigned int)oi[3] << 24);
    }
    if (__syncthreads_or(!ok)) {                    // every thread has read the block
      if (tid == 0) atomicExch(p.status, -7 /* GEAR_ERR_TIMEOUT */);
      bar_wait(&full, feed.parity ^ 1u);       // the copy lands before its memory goes (bounded)
      break;
    }
    if (tid == 0 && item + (int)gridDim.x < feed.total) feed.request(item + gridDim.x);
    if (active) {
      const bool shared_entry = it[0] == ib[0] || it[0] == ib[1] || it[1] == ib[0] || it[1] == ib[1];
      const float levels = (float)((1 << BITS) - 1);
      float d, mn, dm, rmax;
      __half d16;
      if (!shared_entry) {
        mn = bot[2];
        const float mx = top[2];
        // Eq. 2 on the kept entries: binary32, one rounding per operation
        const float range = __fsub_rn(mx, mn);
        const float d32 = __fdiv_rn(range, levels);
        d16 = __float2half_rn(d32);
        d = __half2float(d16);
        const float inv = d != 0.f ? __fdiv_rn(1.0f, d) : 0.f;
        const PairQuant quantize(mn, inv, d, levels);
        if (SIDE == 0) {
#pragma unroll
          for (int q = 0; q < L / 2; ++q) {
            unsigned int c0, c1;
            const float2 r = quantize(__half22float2(xp[q]), c0, c1);
            code_at(2 * q) = (unsigned char)c0;
            code_at(2 * q + 1) = (unsigned char)c1;
            if (R != nullptr) {
              R[(2 * q) * kHeadDim + tid] = r.x;
              R[(2 * q + 1) * kHeadDim + tid] = r.y;
            }
          }
        } else {
#pragma unroll
          for (int q = 0; q < L / 8; ++q) {
            const int piece = (q + rot) & 15;
            float2 r[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              unsigned int c0, c1;
              r[k] = quantize(__half22float2(xp[4 * q + k]), c0, c1);
              code_at(8 * piece + 2 * k) = (unsigned char)c0;
              code_at(8 * piece + 2 * k + 1) = (unsigned char)c1;
            }
            if (R != nullptr) store8(R + first + 8 * piece, r);
          }
        }
        // the filtered entries: cleared
        dm = 0.f;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          code_at(oi[a]) = 0;
          if (R != nullptr) R[SIDE == 0 ? oi[a] * kHeadDim + tid : first + oi[a]] = 0.f;
          dm = fmaxf(dm, fabsf(__half2float(__ushort_as_half(ov[a])) - mn));
        }
        rmax = residual_bound(mn, mx, range, d, levels);
      } else {
        rmax = 0.f;
        GroupResult g = process_group<BITS, 2>(
            L, 2, [&](int e) { return __half2float(X[first + e * step]); },
            [&](int e, int code, float r) {
              code_at(e) = (unsigned char)code;
              if (R != nullptr) R[SIDE == 0 ? e * kHeadDim + tid : first + e] = r;
              rmax = fmaxf(rmax, fabsf(r));
            },
            [&](int slot, int idx, float v) {
              reinterpret_cast<__half*>(orec_v)[slot] = __float2half_rn(v);
              orec_i[slot] = (unsigned char)idx;
            });
        d16 = g.scale;
        d = __half2float(d16);
        mn = __half2float(g.zero);
        dm = g.dmax;
      }
      reinterpret_cast<__half2*>(rec + (SIDE == 0 ? sd.off_kscale : sd.off_vscale))[tid] = __halves2half2(d16, __float2half_rn(mn));
      atomicMax(&dmax_bits, __float_as_uint(dm));       // non-negative floats order like their bit patterns
      atomicMax(&smax_bits, __float_as_uint(d));
      atomicMax(&rmax_bits, __float_as_uint(rmax));
    }
    __syncthreads();
    if (tid == 0) {
      reinterpret_cast<float*>(rec)[SIDE] = __uint_as_float(dmax_bits);
      reinterpret_cast<float*>(rec)[2 + SIDE] = __uint_as_float(smax_bits);
      if (R != nullptr) atomicMax(p.Rmax + bhl * 2 + SIDE, rmax_bits);
      dmax_bits = 0u; smax_bits = 0u; rmax_bits = 0u;       // the next updates come behind the next block's first barrier
    }
    // pack the codes into mma-fragment order (code_coord_k / code_coord_v), one 32-bit load per field
    unsigned int* dst = reinterpret_cast<unsigned int*>(rec + (SIDE == 0 ? sd.off_kcodes : sd.off_vcodes));
    if (SIDE == 0) {
      constexpr int kWords = kSlab * kHeadDim * BITS / 32;            // words per slab
      for (int li = tid; li < (L / kSlab) * kWords; li += 128) {
        const int slab = li / kWords, wl = li % kWords;
        const int w = wl & 3, lane = (wl >> 2) & 31, tau = wl >> 7;
        const int tok = slab * kSlab + (lane >> 2) + 8 * (w & 1);
        const int ch = 32 * F * tau + 16 * (w >> 1) + 4 * (lane & 3);
        unsigned int word = 0;
#pragma unroll
        for (int j = 0; j < F; ++j)
          word |= *reinterpret_cast<const unsigned int*>(&codes[tok * kCodePitch2 + ch + 32 * j]) << (BITS * j);
        dst[li] = word;
      }
    } else {
      constexpr int kWords = 32 * kHeadDim * BITS / 32;               // words per 32-token chunk
      for (int li = tid; li < (T / 32) * kWords; li += 128) {
        const int chunk = li / kWords, wl = li % kWords;
        const int w = wl & 3, lane = (wl >> 2) & 31, tau = wl >> 7;
        const int ch = 16 * F * tau + (lane >> 2) + 8 * (w & 1);
        const int tok = chunk * 32 + 16 * (w >> 1) + 4 * (lane & 3);
        unsigned int word = 0;
#pragma unroll
        for (int j = 0; j < F; ++j)
          word |= *reinterpret_cast<const unsigned int*>(&codes[(ch + 16 * j) * kCodePitch2 + tok]) << (BITS * j);
        dst[li] = word;
      }
    }
  }
  if (SIDE == 1) after_previous();
}

// ---------------------------------------------------------------------------
// Power iteration (Algorithm 2).  A "tile" is one (batch, head, K|V) residual
// R_h [n_c, 128] in the workspace.  Factor buffers are [128][16] fp32, zero
// beyond the rank.
// ---------------------------------------------------------------------------
constexpr int kPassPitch = kHeadDim * 4 + 16;    // bytes per residual row in shared memory (the lanes' 128-bit reads of two rows hit different banks)
constexpr int kPassStage = 16 * kPassPitch;      // the 16 rows a warp takes at a time
constexpr int kPassStages = 2;
constexpr int kPassSmem = kPassWarps * kPassStages * kPassStage;

// The last loop's pass over the residual: the rows A0 = R b, stored, and this chunk's part of A0^T A0.  The loops before it
// run on R^T R alone (gear_gram.cu), which also gives R^T A0 = (R^T R) b, so this is the only product of the residual
// itself.  The orthonormalising factor W comes from pi_finish_kernel, and R^T (A0 W) = (R^T A0) W.
//
// Bound: the fp32 residual from HBM.  The product runs on the tensor cores (mma.sync.m16n8k16, fp16 operands, fp32
// accumulation; n is the rank, too narrow for a tile of its own in tensor memory) with every fp32 operand cut into an
// fp16 head and an fp16 remainder, the four cross products summed in fp32: 22 bits of each operand survive.  Powers of two
// bring the operands into fp16's range first (R by the tile's largest magnitude, each column of b by its own) and are
// divided out of the results, so the scaling itself is exact.  A warp owns 16 rows at a time; they come through a ring of
// its own in shared memory (bulk copies of a row each), because rows loaded into registers leave nothing in flight
// during the products.  A lane reads, for rows gid and gid + 8, the four channels 16c + 4t .. + 3 of each 16-channel step c
// as one 128-bit load; since a contraction does not care about the order of its index, these four channels serve as the
// step's k indices 2t, 2t+1, 2t+8, 2t+9 of the A fragment.  NT = 8-column tiles of n: four rank columns (head and
// remainder each) per tile.
template <int NT>
__global__ void __launch_bounds__(kPassWarps * 32, 3) pi_pass_kernel(PiArgs p) {
  constexpr int RP = 4 * NT;
  __shared__ typename PassFactor<NT>::Shared sh;
  __shared__ uint64_t full[kPassWarps][kPassStages];
  extern __shared__ __align__(128) unsigned char ring_all[];
  const int tile = blockIdx.y, chunk = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, t = lane & 3;
  const int row0 = chunk * kChunkRows;
  const int row1 = min(p.n_c, row0 + kChunkRows);
  const float* R = p.R + (size_t)tile * p.n_c * kHeadDim;
  float* A0 = p.A0 + (size_t)tile * p.n_c * RP;
  after_previous();

  // ---- the warp's ring: rows [rb, rb + 16) of its it-th group go to stage it % kPassStages
  unsigned char* ring = ring_all + warp * kPassStages * kPassStage;
  if (lane == 0) {
#pragma unroll
    for (int s = 0; s < kPassStages; ++s) bar_init(&full[warp][s]);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  auto request = [&](int rb, int s) {
    const int rows = min(16, row1 - rb);
    if (rows <= 0) return;
    __syncwarp();                                  // every lane is done with the stage
    if (lane == 0) bar_expect(&full[warp][s], rows * kHeadDim * 4);
    __syncwarp();
    if (lane < rows) bulk_copy(ring + s * kPassStage + lane * kPassPitch, R + (size_t)(rb + lane) * kHeadDim, kHeadDim * 4, &full[warp][s]);
  };
#pragma unroll
  for (int s = 0; s < kPassStages; ++s) request(row0 + (s * kPassWarps + warp) * 16, s);

  const int er = pow2_exponent(__uint_as_float(p.Rmax[tile]));
  const float sr = exp2_int(-er);
  PassFactor<NT> factor;
  factor.load(p, tile, er, sh);
  // B fragments of a = R b: column n = gid of tile nt is (rho = 4 nt + gid / 2, head | remainder), k as described above
  uint32_t bf[8][NT][2];
#pragma unroll
  for (int c = 0; c < 8; ++c)
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      const uint2 v = *reinterpret_cast<const uint2*>(&sh.bsplit[8 * nt + gid][16 * c + 4 * t]);
      bf[c][nt][0] = v.x; bf[c][nt][1] = v.y;
    }
  int stage = 0;
  uint32_t parity = 0;
  for (int rb = row0 + warp * 16; rb < row1; rb += kPassWarps * 16) {
    const int ra = rb + gid, rc = rb + gid + 8;
    const bool va = ra < row1, vc = rc < row1;
    if (!bar_wait(&full[warp][stage], parity)) {   // gave up: report, let the later copies land (bounded), leave the loop
      if (lane == 0) atomicExch(p.status, -7 /* GEAR_ERR_TIMEOUT */);
      for (int s = 0; s < kPassStages - 1; ++s) {
        rb += kPassWarps * 16;
        if (++stage == kPassStages) { stage = 0; parity ^= 1; }
        if (rb < row1) bar_wait(&full[warp][stage], parity);
      }
      break;
    }
    const float4* xa = reinterpret_cast<const float4*>(ring + stage * kPassStage + gid * kPassPitch) + t;
    const float4* xc = reinterpret_cast<const float4*>(ring + stage * kPassStage + (gid + 8) * kPassPitch) + t;
    float d[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) d[nt][0] = d[nt][1] = d[nt][2] = d[nt][3] = 0.f;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const float4 a = va ? xa[4 * c] : make_float4(0.f, 0.f, 0.f, 0.f), b = vc ? xc[4 * c] : make_float4(0.f, 0.f, 0.f, 0.f);
      uint32_t fh[4], fl[4];
      split_pair(a.x * sr, a.y * sr, fh[0], fl[0]);
      split_pair(b.x * sr, b.y * sr, fh[1], fl[1]);
      split_pair(a.z * sr, a.w * sr, fh[2], fl[2]);
      split_pair(b.z * sr, b.w * sr, fh[3], fl[3]);
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        mma16816_f16(d[nt], fh, bf[c][nt][0], bf[c][nt][1]);
        mma16816_f16(d[nt], fl, bf[c][nt][0], bf[c][nt][1]);
      }
    }
    const int used = stage;
    if (++stage == kPassStages) { stage = 0; parity ^= 1; }
    factor.store(d, A0, ra, rc, va, vc);           // rows past the chunk are zero
    request(rb + kPassStages * kPassWarps * 16, used);             // behind stores that need every load from the stage
    factor.add_gram();
  }
  factor.leave_gram(p, tile, chunk, sh);
}

// R^T A0 from the residual itself, for tiles whose factor columns differ so much in norm that (R^T R) b would lose digits
// of the small ones (pi_iterate_kernel sets the flag; most residuals have no such tile, and the CTAs leave at once).  One
// channel per thread; kRtaParts CTAs per tile, each with a contiguous share of the rows.
__global__ void __launch_bounds__(kHeadDim) pi_rta_kernel(PiArgs p) {
  constexpr int kRows = 32;
  __shared__ float a[kRows * kMaxRank];
  const int tile = blockIdx.y, part = blockIdx.x, j = threadIdx.x;
  after_previous();
  if (!p.ill[tile]) return;
  const int RP = p.a0_pitch;
  const int row0 = (int)((long long)part * p.n_c / kRtaParts), row1 = (int)((long long)(part + 1) * p.n_c / kRtaParts);
  const float* R = p.R + (size_t)tile * p.n_c * kHeadDim + j;
  const float* A0 = p.A0 + (size_t)tile * p.n_c * RP;
  float b[kMaxRank];
#pragma unroll
  for (int q = 0; q < kMaxRank; ++q) b[q] = 0.f;
  for (int r0 = row0; r0 < row1; r0 += kRows) {
    const int rows = min(kRows, row1 - r0);
    __syncthreads();
    for (int i = j; i < rows * RP; i += kHeadDim) a[(i / RP) * kMaxRank + i % RP] = A0[(size_t)r0 * RP + i];
    __syncthreads();
    for (int i = 0; i < rows; ++i) {
      const float x = R[(size_t)(r0 + i) * kHeadDim];
#pragma unroll
      for (int q = 0; q < kMaxRank; ++q)
        if (q < RP) b[q] = fmaf(x, a[i * kMaxRank + q], b[q]);
    }
  }
  float* out = p.Bp + (((size_t)tile * kRtaParts + part) * kHeadDim + j) * kMaxRank;
#pragma unroll
  for (int q = 0; q < kMaxRank; ++q) out[q] = q < RP ? b[q] : 0.f;
}

// The stored A = A0 W (W = U^-1 of A0's Cholesky factor): one thread per row.  Keys: a row is r_pad
// consecutive fp16 of its slab; values: the slab is transposed ([r_pad][16 tokens]), so the threads of a slab fill
// 32 contiguous bytes per rank index.  fp32 copy on request.
template <int RP>
__global__ void __launch_bounds__(256) pi_store_a_kernel(PiArgs p) {
  __shared__ __align__(16) float Wm[RP][RP];
  const int tile = blockIdx.y;
  after_previous();
  for (int i = threadIdx.x; i < RP * RP; i += blockDim.x) Wm[i / RP][i % RP] = p.W[(size_t)tile * 256 + (i / RP) * kMaxRank + i % RP];
  __syncthreads();
  const int row = blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= p.n_c) return;
  const SegDesc& sd = p.seg;
  const int r = sd.rank;
  const float4* a0p = reinterpret_cast<const float4*>(p.A0 + ((size_t)tile * p.n_c + row) * RP);
  float a0[RP], a[kMaxRank];
#pragma unroll
  for (int q = 0; q < RP / 4; ++q) {               // columns past the rank are zero (the factor's are)
    const float4 v = a0p[q];
    a0[4 * q] = v.x; a0[4 * q + 1] = v.y; a0[4 * q + 2] = v.z; a0[4 * q + 3] = v.w;
  }
#pragma unroll
  for (int c = 0; c < kMaxRank; ++c) {
    float v = 0.f;
    if (c < RP) {
#pragma unroll
      for (int q = 0; q < RP; ++q)
        if (q <= c) v = fmaf(a0[q], Wm[q][c < RP ? c : 0], v);         // W is upper triangular
    }
    a[c] = v;
  }
  const int bhl = tile >> 1, side = tile & 1;
  const int blk = row / sd.T, tib = row % sd.T, slab = tib / kSlab, ts = tib % kSlab;
  unsigned char* rec = p.arena + sd.seg_base + (size_t)(p.bh0 + bhl) * sd.bh_stride + sd.bfac_bytes +
                       (size_t)blk * sd.rec_bytes;
  if (side == 0) {
    __half2* dst = reinterpret_cast<__half2*>(rec + sd.off_ak + slab * sd.slab_a) + ts * (sd.r_pad / 2);
#pragma unroll
    for (int c = 0; c < kMaxRank; c += 2)
      if (c < sd.r_pad) dst[c / 2] = __floats2half2_rn(a[c], a[c + 1]);
  } else {
    __half* dst = reinterpret_cast<__half*>(rec + sd.off_av + slab * sd.slab_a) + ts;
#pragma unroll
    for (int c = 0; c < kMaxRank; ++c)
      if (c < sd.r_pad) dst[c * kSlab] = __float2half_rn(a[c]);
  }
  if (p.dbgA != nullptr) {
    float* dd = p.dbgA + (((size_t)(p.bh0 + bhl) * 2 + side) * sd.n_c + row) * r;
#pragma unroll
    for (int c = 0; c < kMaxRank; ++c)
      if (c < r) dd[c] = a[c];
  }
}

// One CTA per tile: the chunk partials of A0^T A0 are summed (fixed order), W = U^-1 of the Gram matrix's
// Cholesky factor orthonormalises A0 (its columns are nearly orthonormal already, see pi_iterate_kernel) and the final
// factor B = (R^T A0) W is stored as fp16 ([r_pad][128] for keys, [128][r_pad] for values).
template <int RP>
__global__ void __launch_bounds__(kHeadDim) pi_finish_kernel(PiArgs p) {
  __shared__ float Gm[RP][RP + 1], Wm[RP][RP + 1];
  const int tile = blockIdx.x, j = threadIdx.x, lane = j & 31, warp = j >> 5, r = p.rank;
  after_previous();
  for (int e = j; e < r * r; e += kHeadDim) {
    const float* src = p.Gp + (size_t)tile * p.nchunk * 256 + (e / r) * kMaxRank + e % r;
    float s = 0.f;
#pragma unroll 4
    for (int c = 0; c < p.nchunk; ++c) s += src[(size_t)c * 256];
    Gm[e / r][e % r] = s;
  }
  float b[RP];
#pragma unroll
  for (int q = 0; q < RP; ++q) b[q] = 0.f;
  const bool ill = p.ill[tile] != 0;               // R^T A0: from pi_rta_kernel's partials, else (R^T R) b
  const float4* bp = reinterpret_cast<const float4*>(ill ? p.Bp + ((size_t)tile * kRtaParts * kHeadDim + j) * kMaxRank
                                                         : p.Bg + ((size_t)tile * kHeadDim + j) * kMaxRank);
  for (int c = 0; c < (ill ? kRtaParts : 1); ++c)
#pragma unroll
    for (int q = 0; q < RP / 4; ++q) {
      const float4 v = bp[(size_t)c * (kHeadDim * kMaxRank / 4) + q];
      b[4 * q] += v.x; b[4 * q + 1] += v.y; b[4 * q + 2] += v.z; b[4 * q + 3] += v.w;
    }
  __syncthreads();
  if (warp == 0) warp_chol_inverse<RP, false>(&Gm[0][0], &Wm[0][0], RP + 1, r, lane);
  __syncthreads();
  for (int e = j; e < kMaxRank * kMaxRank; e += kHeadDim) {
    const int u = e / kMaxRank, v = e % kMaxRank;
    p.W[(size_t)tile * 256 + e] = u < r && v < r ? Wm[u < RP ? u : 0][v < RP ? v : 0] : 0.f;
  }
  const SegDesc& sd = p.seg;
  const int bhl = tile >> 1, side = tile & 1;
  __half* bf = reinterpret_cast<__half*>(p.arena + sd.seg_base + (size_t)(p.bh0 + bhl) * sd.bh_stride);
#pragma unroll
  for (int c = 0; c < RP; ++c) {
    if (c < sd.r_pad) {
      float v = 0.f;
#pragma unroll
      for (int q = 0; q <= c; ++q) v = q < r && c < r ? fmaf(b[q], Wm[q][c], v) : v;
      const __half h = __float2half_rn(v);
      if (side == 0) bf[c * kHeadDim + j] = h;
      else bf[sd.r_pad * kHeadDim + j * sd.r_pad + c] = h;
      if (p.dbgB != nullptr && c < r) p.dbgB[(((size_t)(p.bh0 + bhl) * 2 + side) * kHeadDim + j) * r + c] = v;
    }
  }
}

// Gram partials of A0 for ranks above 8 (the pass has no registers left for them).  A warp takes 32 rows at a time through shared
// memory, a lane a 2 x 4 block of the matrix: two loads for eight products instead of sixteen (512 tiles of 4096 rows
// 208 -> 64 us; the bytes take 21).
__global__ void __launch_bounds__(256) pi_gram2_kernel(PiArgs p) {
  __shared__ __align__(16) float rows[8][32][kMaxRank + 4];
  __shared__ float red[8][256];
  const int tile = blockIdx.y, chunk = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = p.rank, u0 = (lane >> 2) * 2, v0 = (lane & 3) * 4;
  const int row0 = chunk * p.chunk_rows, row1 = min(p.n_c, row0 + p.chunk_rows);
  const float4* A0 = reinterpret_cast<const float4*>(p.A0 + (size_t)tile * p.n_c * kMaxRank);
  float g[2][4] = {};
  after_previous();
  for (int base = row0 + warp * 32; base < row1; base += 8 * 32) {
    const int row = base + lane;
#pragma unroll
    for (int q = 0; q < kMaxRank / 4; ++q)
      *reinterpret_cast<float4*>(&rows[warp][lane][4 * q]) =
          row < row1 ? A0[(size_t)row * (kMaxRank / 4) + q] : make_float4(0.f, 0.f, 0.f, 0.f);
    __syncwarp();
#pragma unroll 8
    for (int t = 0; t < 32; ++t) {
      const float2 u = *reinterpret_cast<const float2*>(&rows[warp][t][u0]);
      const float4 v = *reinterpret_cast<const float4*>(&rows[warp][t][v0]);
      g[0][0] = fmaf(u.x, v.x, g[0][0]); g[0][1] = fmaf(u.x, v.y, g[0][1]);
      g[0][2] = fmaf(u.x, v.z, g[0][2]); g[0][3] = fmaf(u.x, v.w, g[0][3]);
      g[1][0] = fmaf(u.y, v.x, g[1][0]); g[1][1] = fmaf(u.y, v.y, g[1][1]);
      g[1][2] = fmaf(u.y, v.z, g[1][2]); g[1][3] = fmaf(u.y, v.w, g[1][3]);
    }
    __syncwarp();
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) red[warp][(u0 + i) * kMaxRank + v0 + j] = u0 + i < r && v0 + j < r ? g[i][j] : 0.f;
  __syncthreads();
  {
    const int i = threadIdx.x;
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) s += red[w][i];
    p.Gp[((size_t)tile * p.nchunk + chunk) * 256 + i] = s;
  }
}

// ---------------------------------------------------------------------------
// Whole-tile compression for short segments (a flushed buffer, Algorithm 1's
// decoding phase): one CTA takes one (batch, head, K|V) tile of n_c <= 128
// tokens through Filter, Quant, residual and all of Algorithm 2 with the
// residual held in shared memory, so that a flush is one launch instead of a
// chain of a dozen latency-bound ones.
// ---------------------------------------------------------------------------
constexpr int kTileMaxTokens = 128;
constexpr int kFPitch = kMaxRank + 1;      // floats per row of the factor matrices in shared memory

struct TileArgs {
  SegDesc seg;
  CacheConst cc;
  unsigned char* arena;
  const __half* K;      // [BH][n_c][128]
  const __half* V;
  const float* B0;      // [BH][2][128][rank] or nullptr
  float* dbgA;
  float* dbgB;
  unsigned long long seed;
  int segment_index;
  int iters;
};

__device__ __forceinline__ float block_sum128(float v, float* wsum, int lane, int warp) {
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) wsum[warp] = v;
  __syncthreads();
  return (wsum[0] + wsum[1]) + (wsum[2] + wsum[3]);
}

// G = U^T U (upper Cholesky factor) and U^-1 for the r x r Gram matrix G; first: W <- U^-1, else W <- W U^-1.
// A column whose pivot vanishes is zeroed.  Run by one warp; matrices have pitch kFPitch.
__device__ void chol_update(const float* G, float* U, float* Ui, float* W, int r, int first, int lane) {
  for (int i = lane; i < kMaxRank * kFPitch; i += 32) { U[i] = 0.f; Ui[i] = 0.f; }
  __syncwarp();
  if (lane == 0) {
    float tr = 0.f;
    for (int i = 0; i < r; ++i) tr += G[i * kFPitch + i];
    const float tiny = tr * 1e-12f;
    for (int j = 0; j < r; ++j) {
      float d = G[j * kFPitch + j];
      for (int k = 0; k < j; ++k) d -= U[k * kFPitch + j] * U[k * kFPitch + j];
      const bool ok = d > tiny && d > 0.f;
      const float ujj = ok ? sqrtf(d) : 0.f;
      U[j * kFPitch + j] = ujj;
      for (int i = j + 1; i < r; ++i) {
        float sacc = G[j * kFPitch + i];
        for (int k = 0; k < j; ++k) sacc -= U[k * kFPitch + j] * U[k * kFPitch + i];
        U[j * kFPitch + i] = ok ? sacc / ujj : 0.f;
      }
    }
    for (int c = 0; c < r; ++c) {
      for (int i = c; i >= 0; --i) {
        if (U[i * kFPitch + i] == 0.f) { Ui[i * kFPitch + c] = 0.f; continue; }
        float sacc = (i == c) ? 1.f : 0.f;
        for (int k = i + 1; k <= c; ++k) sacc -= U[i * kFPitch + k] * Ui[k * kFPitch + c];
        Ui[i * kFPitch + c] = sacc / U[i * kFPitch + i];
      }
      if (U[c * kFPitch + c] == 0.f) for (int i = 0; i <= c; ++i) Ui[i * kFPitch + c] = 0.f;
    }
  }
  __syncwarp();
  // W (r x r): each lane owns entries lane, lane + 32, ...; the product needs the old W, so read it all first
  float wn[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const int i = lane + 32 * e, a = i / kMaxRank, b = i % kMaxRank;
    float v = 0.f;
    if (a < r && b < r) {
      if (first) v = Ui[a * kFPitch + b];
      else for (int k = 0; k < r; ++k) v = fmaf(W[a * kFPitch + k], Ui[k * kFPitch + b], v);
    }
    wn[e] = v;
  }
  __syncwarp();
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const int i = lane + 32 * e;
    W[(i / kMaxRank) * kFPitch + i % kMaxRank] = wn[e];
  }
  __syncwarp();
}

// Shared memory: [ region 0 | residual rs[n_c][kRPitch] ].  Region 0 first holds the fp16 tile of the block being
// quantized (each entry is replaced by its code once it is known), later the factor matrices of Algorithm 2.
template <int RP>
__host__ __device__ constexpr int tile_factor_bytes(int n_c) {
  return ((kHeadDim + n_c) * (RP + 1) + 4 * kMaxRank * kFPitch + 8) * 4;
}

template <int BITS, int KMAX, int RP>
__global__ void __launch_bounds__(128) compress_tile_kernel(TileArgs p) {
  constexpr int FP = RP + 1;                 // floats per row of B and A in shared memory
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const SegDesc& sd = p.seg;
  const int T = sd.T, n_c = sd.n_c, r = sd.rank;
  const int side = blockIdx.y, bh = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int reg0 = max(round_up(T * kXPitch * 2, 16), tile_factor_bytes<RP>(n_c));
  unsigned short* xs = reinterpret_cast<unsigned short*>(smem_raw);      // [T][kXPitch] fp16 bits, then codes
  float* rs = reinterpret_cast<float*>(smem_raw + reg0);                 // [n_c][kRPitch] residual of the whole tile
  float* Bm = reinterpret_cast<float*>(smem_raw);                        // [128][FP]
  float* Am = Bm + kHeadDim * FP;                                        // [n_c][FP]
  float* Gm = Am + n_c * FP;                                             // [16][kFPitch]
  float* Um = Gm + kMaxRank * kFPitch;
  float* Uim = Um + kMaxRank * kFPitch;
  float* Wm = Uim + kMaxRank * kFPitch;
  float* wsum = Wm + kMaxRank * kFPitch;                                 // [4]
  __shared__ unsigned int dmax_bits, smax_bits;

  const __half* Xt = (side == 0 ? p.K : p.V) + (size_t)bh * n_c * kHeadDim;
  unsigned char* seg_bh = p.arena + sd.seg_base + (size_t)bh * sd.bh_stride;
  auto x_of = [&](int idx) { return __half2float(__ushort_as_half(xs[idx])); };
  after_previous();

  // ---- Filter, Quant, pack, residual: block by block (one key group per channel spans one block)
  for (int blk = 0; blk < sd.nblk; ++blk) {
    if (tid == 0) { dmax_bits = 0u; smax_bits = 0u; }
    const __half* X = Xt + (size_t)blk * T * kHeadDim;
    for (int i = tid; i < T * 16; i += 128) {
      const int row = i >> 4, c = i & 15;
      const uint4 v = *reinterpret_cast<const uint4*>(X + row * kHeadDim + c * 8);
      unsigned int* dst = reinterpret_cast<unsigned int*>(xs + row * kXPitch + c * 8);
      dst[0] = v.x; dst[1] = v.y; dst[2] = v.z; dst[3] = v.w;
    }
    __syncthreads();
    unsigned char* rec = seg_bh + sd.bfac_bytes + (size_t)blk * sd.rec_bytes;
    float* rb = rs + (size_t)blk * T * kRPitch;
    float my_dmax = 0.f, my_smax = 0.f;
    if (side == 0) {
      const int j = tid, k = sd.k_k;
      __half* oval = reinterpret_cast<__half*>(rec + sd.off_koval) + j * 2 * k;
      unsigned char* oidx = rec + sd.off_koidx + j * 2 * k;
      GroupResult g = process_group<BITS, KMAX>(
          T, k, [&](int e) { return x_of(e * kXPitch + j); },
          [&](int e, int code, float res) { xs[e * kXPitch + j] = (unsigned short)code; rb[e * kRPitch + j] = res; },
          [&](int slot, int idx, float v) { oval[slot] = __float2half_rn(v); oidx[slot] = (unsigned char)idx; });
      reinterpret_cast<__half2*>(rec + sd.off_kscale)[j] = __halves2half2(g.scale, g.zero);
      my_dmax = g.dmax;
      my_smax = __half2float(g.scale);
    } else {
      const int k = p.cc.k_v, gv = p.cc.g_v, ngv = p.cc.ngv;
      for (int gi = tid; gi < T * ngv; gi += 128) {
        const int tok = gi / ngv, c = gi % ngv;
        __half* oval = reinterpret_cast<__half*>(rec + sd.off_voval) + gi * 2 * k;
        unsigned char* oidx = rec + sd.off_voidx + gi * 2 * k;
        GroupResult g = process_group<BITS, KMAX>(
            gv, k, [&](int e) { return x_of(tok * kXPitch + c * gv + e); },
            [&](int e, int code, float res) {
              xs[tok * kXPitch + c * gv + e] = (unsigned short)code;
              rb[tok * kRPitch + c * gv + e] = res;
            },
            [&](int slot, int idx, float v) { oval[slot] = __float2half_rn(v); oidx[slot] = (unsigned char)idx; });
        reinterpret_cast<__half2*>(rec + sd.off_vscale)[gi] = __halves2half2(g.scale, g.zero);
        my_dmax = fmaxf(my_dmax, g.dmax);
        my_smax = fmaxf(my_smax, __half2float(g.scale));
      }
    }
    atomicMax(&dmax_bits, __float_as_uint(my_dmax));
    atomicMax(&smax_bits, __float_as_uint(my_smax));
    __syncthreads();
    if (tid == 0) {
      reinterpret_cast<float*>(rec)[side] = __uint_as_float(dmax_bits);
      reinterpret_cast<float*>(rec)[2 + side] = __uint_as_float(smax_bits);
    }
    pack_block_codes<BITS>(xs, T, side, reinterpret_cast<unsigned int*>(rec + (side == 0 ? sd.off_kcodes : sd.off_vcodes)),
                           tid, 128);
    __syncthreads();
  }
  if (r == 0) return;

  // ---- Algorithm 2 on the residual in shared memory.  Thread `tid` owns channel tid of B.
  const size_t gtile = (size_t)bh * 2 + side;
  float b[RP];
#pragma unroll
  for (int rho = 0; rho < RP; ++rho) {
    float v = 0.f;
    if (rho < r) {
      if (p.B0 != nullptr) {
        v = p.B0[(gtile * kHeadDim + tid) * r + rho];
      } else {
        v = start_value(p.seed, p.segment_index, gtile, tid, rho);
      }
    }
    b[rho] = v;
  }
  for (int l = 0; l < p.iters; ++l) {
    const bool last = l == p.iters - 1;
    if (last) {
      // B <- Q(B): modified Gram-Schmidt, two sweeps per column, then a Newton step on the norm
#pragma unroll
      for (int c = 0; c < RP; ++c) {
        if (c < r) {
#pragma unroll
          for (int sweep = 0; sweep < 2; ++sweep) {
#pragma unroll
            for (int q = 0; q < RP; ++q) {
              if (q < c) {
                const float d = block_sum128(b[q] * b[c], wsum, lane, warp);
                b[c] = fmaf(-d, b[q], b[c]);
              }
            }
          }
          const float nrm2 = block_sum128(b[c] * b[c], wsum, lane, warp);
          b[c] = nrm2 > 0.f ? b[c] * rsqrtf(nrm2) : 0.f;
          const float n2 = block_sum128(b[c] * b[c], wsum, lane, warp);
          if (n2 > 0.f) b[c] *= (1.5f - 0.5f * n2);
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int rho = 0; rho < RP; ++rho) Bm[tid * FP + rho] = b[rho];
    __syncthreads();
    // A = R B: one row of A per thread and round (all columns at once)
    for (int i = tid; i < n_c; i += 128) {
      const float* rr = rs + i * kRPitch;
      float acc[RP];
#pragma unroll
      for (int rho = 0; rho < RP; ++rho) acc[rho] = 0.f;
#pragma unroll 4
      for (int c = 0; c < kHeadDim; ++c) {
        const float x = rr[c];
#pragma unroll
        for (int rho = 0; rho < RP; ++rho) acc[rho] = fmaf(x, Bm[c * FP + rho], acc[rho]);
      }
#pragma unroll
      for (int rho = 0; rho < RP; ++rho) Am[i * FP + rho] = acc[rho];
    }
    __syncthreads();
    if (last) {
      // A <- Q(A) by Cholesky QR, twice: Gram matrix, U^-1 of its Cholesky factor, A <- A U^-1
      for (int round = 0; round < 2; ++round) {
        for (int o = tid; o < r * r; o += 128) {
          const int u = o / r, v = o % r;
          float acc = 0.f;
          for (int i = 0; i < n_c; ++i) acc = fmaf(Am[i * FP + u], Am[i * FP + v], acc);
          Gm[u * kFPitch + v] = acc;
        }
        __syncthreads();
        if (warp == 0) chol_update(Gm, Um, Uim, Wm, r, 1, lane);
        __syncthreads();
        for (int i = tid; i < n_c; i += 128) {           // one row per thread
          float a0[RP], an[RP];
#pragma unroll
          for (int k = 0; k < RP; ++k) a0[k] = Am[i * FP + k];
#pragma unroll
          for (int c = 0; c < RP; ++c) {
            float acc = 0.f;
#pragma unroll
            for (int k = 0; k < RP; ++k) acc = fmaf(a0[k], Wm[k * kFPitch + c], acc);
            an[c] = acc;
          }
#pragma unroll
          for (int c = 0; c < RP; ++c) Am[i * FP + c] = an[c];
          if (round == 1) {
            // the final A: fp16 in the records (fragment order), fp32 copy on request
            const int blk = i / T, tib = i % T, slab = tib / kSlab, ts = tib % kSlab;
            unsigned char* rec = seg_bh + sd.bfac_bytes + (size_t)blk * sd.rec_bytes;
#pragma unroll
            for (int c = 0; c < RP; ++c) {
              if (c < sd.r_pad) {
                const float val = c < r ? an[c] : 0.f;
                if (side == 0)
                  reinterpret_cast<__half*>(rec + sd.off_ak + slab * sd.slab_a)[ts * sd.r_pad + c] = __float2half_rn(val);
                else
                  reinterpret_cast<__half*>(rec + sd.off_av + slab * sd.slab_a)[c * kSlab + ts] = __float2half_rn(val);
                if (p.dbgA != nullptr && c < r) p.dbgA[(gtile * n_c + i) * r + c] = val;
              }
            }
          }
        }
        __syncthreads();
      }
    }
    // B = R^T A: channel tid
#pragma unroll
    for (int rho = 0; rho < RP; ++rho) b[rho] = 0.f;
#pragma unroll 4
    for (int i = 0; i < n_c; ++i) {
      const float x = rs[i * kRPitch + tid];
#pragma unroll
      for (int rho = 0; rho < RP; ++rho) b[rho] = fmaf(x, Am[i * FP + rho], b[rho]);
    }
  }
  // ---- store B: fp16 [r_pad][128] for keys, [128][r_pad] for values
  __half* bf = reinterpret_cast<__half*>(seg_bh);
#pragma unroll
  for (int rho = 0; rho < RP; ++rho) {
    if (rho < sd.r_pad) {
      const __half v = __float2half_rn(rho < r ? b[rho] : 0.f);
      if (side == 0) bf[rho * kHeadDim + tid] = v;
      else bf[sd.r_pad * kHeadDim + tid * sd.r_pad + rho] = v;
      if (p.dbgB != nullptr && rho < r) p.dbgB[(gtile * kHeadDim + tid) * r + rho] = b[rho];
    }
  }
}

static int tile_rp(int rank) { return rank <= 4 ? 4 : (rank <= 8 ? 8 : 16); }

static size_t tile_smem_bytes(int T, int n_c, int rank) {
  const int rp = tile_rp(rank);
  const int fb = rp == 4 ? tile_factor_bytes<4>(n_c) : (rp == 8 ? tile_factor_bytes<8>(n_c) : tile_factor_bytes<16>(n_c));
  const int x = round_up(T * kXPitch * 2, 16);
  return (size_t)(x > fb ? x : fb) + (size_t)n_c * kRPitch * 4;
}

bool compress_tile_fits(int T, int n_c, int rank) {
  return n_c <= kTileMaxTokens && tile_smem_bytes(T, n_c, rank) <= 200 * 1024;
}

cudaError_t compress_tile(const CompressJob& job, int BH, cudaStream_t st) {
  TileArgs a;
  a.seg = job.seg; a.cc = job.cc; a.arena = job.arena; a.K = job.K; a.V = job.V; a.B0 = job.B0;
  a.dbgA = job.dbgA; a.dbgB = job.dbgB; a.seed = job.seed; a.segment_index = job.segment_index; a.iters = job.iters;
  const size_t smem = tile_smem_bytes(job.seg.T, job.seg.n_c, job.seg.rank);
  const int kneed = job.seg.k_k > job.cc.k_v ? job.seg.k_k : job.cc.k_v;
  const int rp = tile_rp(job.seg.rank);
  dim3 grid(BH, 2);
  cudaError_t e = cudaSuccess;
#define GEAR_TILE(B, KM, R)                                                                                          \
  {                                                                                                                  \
    e = cudaFuncSetAttribute(compress_tile_kernel<B, KM, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem); \
    if (e != cudaSuccess) return e;                                                                                  \
    e = launch_dependent(compress_tile_kernel<B, KM, R>, grid, 128, smem, st, a);                                    \
  }
#define GEAR_TILE_R(B, KM) \
  { if (rp == 4) GEAR_TILE(B, KM, 4) else if (rp == 8) GEAR_TILE(B, KM, 8) else GEAR_TILE(B, KM, 16) }
  if (job.cc.bits == 2) {
    if (kneed <= 1) GEAR_TILE_R(2, 1) else if (kneed <= 2) GEAR_TILE_R(2, 2) else GEAR_TILE_R(2, 8)
  } else {
    if (kneed <= 1) GEAR_TILE_R(4, 1) else if (kneed <= 2) GEAR_TILE_R(4, 2) else GEAR_TILE_R(4, 8)
  }
#undef GEAR_TILE_R
#undef GEAR_TILE
  count_launches(1);
  return cudaGetLastError();
}

// Segment with rank 0: nothing to fit, but the A sections of the records do not exist either.
// Segment descriptor table entry, written by the device so that no host copy is needed.
__global__ void write_desc_kernel(SegDesc* table, int* blk2seg, int index, SegDesc d) {
  after_previous();
  if (threadIdx.x == 0) table[index] = d;
  for (int b = threadIdx.x; b < d.nblk; b += blockDim.x) blk2seg[d.blk_start + b] = index;
}

// One decoding step's rows into the streaming buffer (and, for the host-buffer calls, the query into its device copy):
// one 16-byte piece per thread.  With `host_src` the sources are pinned host memory that the caller filled before the
// launch: they are read across the bus before the wait for the kernel in front, so that the round trip (2 us) runs
// while that kernel drains; a device source may be that kernel's output and is read after the wait.  The launch is a
// programmatic dependent of the kernel before it and keeps the rule of the decode kernel: dependents start only after
// the own wait.
__global__ void __launch_bounds__(256) push_kernel(PushArgs p) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int rows = p.k_new ? p.BH * 16 : 0;                // pieces per side
  const bool mine = i < 2 * rows + p.q_pieces;
  const uint4* src = nullptr;
  uint4* dst = nullptr;
  if (i < 2 * rows) {
    const int side = i >= rows, r = side ? i - rows : i, bh = r >> 4, c = r & 15;
    src = reinterpret_cast<const uint4*>(side == 0 ? p.k_new : p.v_new) + r;
    dst = reinterpret_cast<uint4*>(side == 0 ? p.buf_k : p.buf_v) + ((size_t)bh * p.n_b + p.slot) * 16 + c;
  } else if (mine) {
    src = reinterpret_cast<const uint4*>(p.q_src) + (i - 2 * rows);
    dst = reinterpret_cast<uint4*>(p.q_dst) + (i - 2 * rows);
  }
  uint4 v = make_uint4(0u, 0u, 0u, 0u);
  if (p.host_src && mine) v = __ldcv(src);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (!mine) return;
  if (!p.host_src) v = *src;
  *dst = v;
}

// ---------------------------------------------------------------------------
// host side: launch sequence for a range of (batch, head) pairs
// ---------------------------------------------------------------------------
// Filter / Quant / pack / residual of a long segment: per side, the register-resident kernel that fits the group
// shape, else the general one.  side0 = 1: the value side only.  Returns the number of launches through *launches.
template <int BITS>
static cudaError_t launch_quant(CompressArgs a, int nbh, int kmax_needed, int sms, bool overlap, cudaStream_t st, int* launches) {
  const int T = a.seg.T;
  const size_t smem = round_up(T * kXPitch * 2, 16) + (size_t)T * kRPitch * 4;
  const dim3 grid(a.seg.nblk, nbh, 1);
  const int first_side = a.side0;
  *launches = 0;
  for (int side = first_side; side < 2; ++side) {
    const int len = side == 0 ? T : a.cc.g_v, k = side == 0 ? a.seg.k_k : a.cc.k_v;
    cudaError_t e = cudaSuccess;
    const long long items = (long long)a.seg.nblk * nbh;
    // a thread per group of 32, 64 or 128 entries (values of 128: one per token, whole 32-token chunks of codes)
    const bool shape = len == kHeadDim && side == 1 ? T % 32 == 0 && T <= kHeadDim : T == len;
    const long long room = (long long)fast_ctas_per_sm(side, len) * sms;
    const int ctas = (int)(items < room ? items : room);
    auto launch = [&](auto kern) {
      const int tile = T * kHeadDim * 2;
      if (len == kHeadDim) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kHeadDim * kHeadDim * 2);
      if (e == cudaSuccess) e = launch_after(overlap, kern, dim3(ctas), 128, tile, st, a, nbh);
    };
#define GEAR_LAUNCH_FAST(LEN, K) \
  if (side == 0) launch(quant_fast_kernel<BITS, 0, LEN, K>); else launch(quant_fast_kernel<BITS, 1, LEN, K>);
    if (shape && len == 32 && k == 0) { GEAR_LAUNCH_FAST(32, 0) }
    else if (shape && len == 32 && k == 1) { GEAR_LAUNCH_FAST(32, 1) }
    else if (shape && len == 64 && k == 0) { GEAR_LAUNCH_FAST(64, 0) }
    else if (shape && len == 64 && k == 1) { GEAR_LAUNCH_FAST(64, 1) }
    else if (shape && len == 128 && k == 0) { GEAR_LAUNCH_FAST(128, 0) }
    else if (shape && len == 128 && k == 1) { GEAR_LAUNCH_FAST(128, 1) }
    else if (shape && len == 128 && k == 2) {
      if (side == 0) launch(quant_fast2_kernel<BITS, 0>); else launch(quant_fast2_kernel<BITS, 1>);
#undef GEAR_LAUNCH_FAST
    } else {
      a.side0 = side;
#define GEAR_LAUNCH_Q(KM)                                                                                   \
  {                                                                                                         \
    e = cudaFuncSetAttribute(quant_pack_kernel<BITS, KM>, cudaFuncAttributeMaxDynamicSharedMemorySize,      \
                             (int)smem);                                                                   \
    if (e != cudaSuccess) return e;                                                                         \
    e = launch_after(overlap, quant_pack_kernel<BITS, KM>, grid, 128, smem, st, a);                                              \
  }
      if (kmax_needed <= 1) GEAR_LAUNCH_Q(1)
      else if (kmax_needed <= 2) GEAR_LAUNCH_Q(2)
      else if (kmax_needed <= 4) GEAR_LAUNCH_Q(4)
      else GEAR_LAUNCH_Q(8)
#undef GEAR_LAUNCH_Q
    }
    if (e != cudaSuccess) return e;
    *launches += 1;
  }
  return cudaGetLastError();
}

static cudaError_t launch_pass(const PiArgs& p, bool overlap, cudaStream_t st) {
  auto launch = [&](auto kern) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kPassSmem);
    return e == cudaSuccess ? launch_after(overlap, kern, dim3(p.nchunk, p.ntiles), kPassWarps * 32, kPassSmem, st, p) : e;
  };
  return p.rank <= 4 ? launch(pi_pass_kernel<1>) : p.rank <= 8 ? launch(pi_pass_kernel<2>) : launch(pi_pass_kernel<4>);
}

static int a0_columns(int rank) { return rank <= 4 ? 4 : (rank <= 8 ? 8 : kMaxRank); }   // of the A0 rows in the workspace

// bytes of the power iteration's part of the workspace (a multiple of 256)
static size_t pi_workspace_bytes(int nbh, const SegDesc& sd, const CacheConst& cc, int sms) {
  const int rank = sd.rank, n_c = sd.n_c;
  if (rank == 0) return 256;
  const size_t ntiles = (size_t)nbh * 2;
  const size_t chunk_rows = pass_chunk_rows(nbh, sd, cc, sms), nchunk = (n_c + chunk_rows - 1) / chunk_rows;
  size_t b = 0;
  if (qg_fits(sd, cc)) {
    b += ntiles * kHeadDim * kHeadDim * 4;        // G
    b += qg_partials(nbh, sd, sms) * (kHeadDim * kHeadDim + 1) * 4;    // Gpart, Gexp
  } else {
    b += ntiles * n_c * kHeadDim * 4;             // R
    b += pi_gram_workspace_bytes((int)ntiles, n_c, sms);   // G, Gpart
  }
  b += ntiles * kHeadDim * kMaxRank * 4;          // Bcur
  b += ntiles * kHeadDim * kMaxRank * 4;          // Bg
  b += ntiles * kRtaParts * kHeadDim * kMaxRank * 4;   // Bp
  b += ntiles * n_c * a0_columns(rank) * 4;       // A0
  b += ntiles * nchunk * 256 * 4;                 // Gp
  b += ntiles * 256 * 4;                          // W
  b += ntiles * 8;                                // Rmax, ill
  return (b + 1024 + 255) / 256 * 256;
}

size_t compress_workspace_bytes(int nbh, const SegDesc& sd, const CacheConst& cc, int sms) {
  return pi_workspace_bytes(nbh, sd, cc, sms) + (sd.csr_base16 != 0 ? kcvt_workspace_bytes(nbh, sd.n_c, sd.csr_k) : 0);
}

cudaError_t compress_range(const CompressJob& job, int bh0, int nbh, unsigned char* ws, cudaStream_t st) {
  const SegDesc& sd = job.seg;
  const size_t ntiles = (size_t)nbh * 2;
  const int chunk_rows = pass_chunk_rows(nbh, sd, job.cc, job.sms), nchunk = (sd.n_c + chunk_rows - 1) / chunk_rows;
  float* wsf = reinterpret_cast<float*>(ws);
  PiArgs pa;
  pa.seg = sd; pa.arena = job.arena; pa.bh0 = bh0; pa.ntiles = (int)ntiles; pa.n_c = sd.n_c; pa.rank = sd.rank;
  pa.nchunk = nchunk; pa.chunk_rows = chunk_rows;
  pa.status = job.status; pa.a0_pitch = a0_columns(sd.rank);
  pa.K = job.K + (size_t)bh0 * sd.n_c * kHeadDim; pa.V = job.V + (size_t)bh0 * sd.n_c * kHeadDim; pa.cc = job.cc;
  pa.R = nullptr; pa.Rmax = nullptr; pa.Gpart = nullptr; pa.Gexp = nullptr; pa.G = nullptr; pa.Bcur = nullptr; pa.Bp = nullptr; pa.Bg = nullptr; pa.ill = nullptr; pa.A0 = nullptr; pa.Gp = nullptr; pa.W = nullptr;
  pa.dbgA = job.dbgA; pa.dbgB = job.dbgB;
  const bool from_codes = qg_fits(sd, job.cc);         // the residual is not kept
  if (sd.rank > 0) {
    if (from_codes) {
      const size_t parts = qg_partials(nbh, sd, job.sms);
      pa.G = wsf;     wsf += ntiles * kHeadDim * kHeadDim;
      pa.Gpart = wsf; wsf += parts * kHeadDim * kHeadDim;
    } else {
      pa.R = wsf;     wsf += ntiles * sd.n_c * kHeadDim;
      pa.G = wsf;     pa.Gpart = wsf + ntiles * kHeadDim * kHeadDim;
      wsf += pi_gram_workspace_bytes((int)ntiles, sd.n_c, job.sms) / 4;
    }
    pa.Bcur = wsf;    wsf += ntiles * kHeadDim * kMaxRank;
    pa.Bg = wsf;      wsf += ntiles * kHeadDim * kMaxRank;
    pa.Bp = wsf;      wsf += ntiles * kRtaParts * kHeadDim * kMaxRank;
    pa.A0 = wsf;      wsf += ntiles * sd.n_c * a0_columns(sd.rank);
    pa.Gp = wsf;      wsf += ntiles * nchunk * 256;
    pa.W = wsf;       wsf += ntiles * 256;
    pa.Rmax = reinterpret_cast<unsigned int*>(wsf);
    pa.ill = reinterpret_cast<int*>(wsf) + ntiles;
    pa.Gexp = pa.ill + ntiles;
    if (cudaMemsetAsync(pa.Rmax, 0, ntiles * 4, st) != cudaSuccess) return cudaGetLastError();
  }
  CompressArgs ca;
  ca.seg = sd; ca.cc = job.cc; ca.arena = job.arena; ca.bh0 = bh0;
  ca.K = pa.K; ca.V = pa.V;
  ca.R = pa.R; ca.Rmax = pa.Rmax; ca.status = job.status; ca.Gpart = pa.Gpart; ca.Gexp = pa.Gexp;
  ca.test_dead_wait = job.test_dead_wait;
  const int kneed = sd.k_k > job.cc.k_v ? sd.k_k : job.cc.k_v;
  const bool per_vector = sd.csr_base16 != 0;          // keys: one group per channel over the whole segment
  ca.side0 = per_vector ? 1 : 0;
  cudaError_t e = cudaSuccess;
  if (from_codes) {
    e = launch_quant_gram(ca, pa, nbh, job.sms, st);                 // R^T R too
    if (e == cudaSuccess) e = launch_pi_iterate(pa, job.B0, job.seed, job.segment_index, job.iters, st);
    if (e == cudaSuccess) e = launch_pass_codes(pa, st);             // A0 = R B; for ranks up to 8 also A0^T A0
    if (e != cudaSuccess) return e;
  } else {
    // Launches that overlap pay where they are short (256 tokens x 32 heads, us without and with: groups of 16 66.3 / 59.2, of 32 61.9 / 53.8,
    // per-vector keys 91.1 / 86.0; one head of 4096 77.6 / 68.9, 72.5 / 67.4, 125.8 / 112.4) and without a low-rank part (128 heads x 4096
    // 120 / 110).  Over a kept residual the two cross between 12288 rows (384 tokens x 32 heads 76.7 / 68.5, 70.5 / 61.4, 101.8 / 97.1) and
    // 32768 (1024 x 32 100.9 / 103.7, 86.8 / 86.6; four heads of 8192 121.8 / 131.7, 107.6 / 116.8), at 16384 by shape and group
    // (512 x 32 78.1 / 81.7, 69.9 / 64.8, 102.3 / 101.6; 1024 x 16 77.5 / 77.7, 69.9 / 63.6, 96.6 / 91.7; 4096 x 4 82.2 / 84.9, 73.9 /
    // 75.8, 125.0 / 124.5), and long chains run 4 to 9 % longer (4096 x 32 215 / 227, 167 / 175): all of it the early start of the kernel
    // that sums the partials of R^T R.  What follows that kernel overlaps always.
    const bool overlap = sd.rank == 0 || (long long)nbh * sd.n_c <= 16384;
    int n_quant = 0;
    e = job.cc.bits == 2 ? launch_quant<2>(ca, nbh, kneed, job.sms, overlap, st, &n_quant)
                           : launch_quant<4>(ca, nbh, kneed, job.sms, overlap, st, &n_quant);
    if (e != cudaSuccess) return e;
    count_launches(n_quant);
    if (per_vector) {
      KcvtArgs ka;
      ka.seg = sd; ka.arena = job.arena; ka.K = ca.K; ka.R = pa.R; ka.Rmax = pa.Rmax; ka.bh0 = bh0;
      e = launch_kcvt_keys(ka, nbh, job.cc.bits, ws + pi_workspace_bytes(nbh, sd, job.cc, job.sms), overlap, st);
      if (e != cudaSuccess) return e;
    }
    if (sd.rank == 0) return cudaSuccess;
    e = launch_pi_gram(pa, job.B0, job.seed, job.segment_index, job.iters, job.sms, overlap, st);   // the loops, B <- Q(B), its scaling
    if (e != cudaSuccess) return e;
    e = launch_pass(pa, overlap, st);                                          // A0 = R B; for ranks up to 8 also A0^T A0
    if (e != cudaSuccess) return e;
    e = launch_after(overlap, pi_rta_kernel, dim3(kRtaParts, (int)ntiles), kHeadDim, 0, st, pa);   // R^T A0 of ill-conditioned tiles
    if (e != cudaSuccess) return e;
    count_launches(2);
  }
  if (sd.rank > 8) e = launch_dependent(pi_gram2_kernel, dim3(nchunk, (int)ntiles), 256, 0, st, pa);
  if (e != cudaSuccess) return e;
  auto finish = sd.rank <= 4 ? pi_finish_kernel<4> : sd.rank <= 8 ? pi_finish_kernel<8> : pi_finish_kernel<16>;
  e = launch_dependent(finish, dim3((int)ntiles), kHeadDim, 0, st, pa);                  // W, B
  if (e != cudaSuccess) return e;
  auto store = sd.rank <= 4 ? pi_store_a_kernel<4> : sd.rank <= 8 ? pi_store_a_kernel<8> : pi_store_a_kernel<16>;
  e = launch_dependent(store, dim3((sd.n_c + 255) / 256, (int)ntiles), 256, 0, st, pa);  // A = A0 W
  if (e != cudaSuccess) return e;
  count_launches(sd.rank > 8 ? 3 : 2);
  return cudaGetLastError();
}

cudaError_t launch_write_desc(SegDesc* table, int* blk2seg, int index, const SegDesc& d, cudaStream_t st) {
  const cudaError_t e = launch_dependent(write_desc_kernel, dim3(1), 256, 0, st, table, blk2seg, index, d);
  if (e == cudaSuccess) count_launches(1);
  return e;
}

cudaError_t launch_push(const PushArgs& a, cudaStream_t st) {
  const int n = (a.k_new ? a.BH * 32 : 0) + a.q_pieces;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3((unsigned)((n + 255) / 256)); cfg.blockDim = dim3(256); cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, push_kernel, a);
  if (e == cudaSuccess) count_launches(1);
  return e;
}

}  // namespace gear
