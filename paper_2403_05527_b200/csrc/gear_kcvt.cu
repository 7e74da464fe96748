// Keys of a segment under per-vector grouping (Section 2, "Group-wise Quantization": per-channel key vectors; the
// KCVT backbone of Section 4): one quantization group per channel over all n_c tokens of the segment, Filter_s
// (Eq. 4) on that whole vector.
//   kcvt_select_kernel : per channel, the k largest and k smallest entries in the fp16 order (ties to the lower token),
//                        Eq. 2 on the rest, codes (one byte each, token-major) and the fp32 residual
//   kcvt_list_kernel   : the outliers of a (batch, head), sorted into per-block lists; block headers, scales
//   kcvt_pack_kernel   : codes of a 64-token block into the fragment order of the decode kernel
// The arithmetic that decides a code is the same binary32 sequence as in the per-group kernels.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>

#include "gear_internal.cuh"
#include "gear_quant.cuh"

namespace gear {

constexpr int kSelChannels = 8;     // channels per CTA of the select kernel, one per warp
constexpr int kBlockTok = 64;       // tokens per record block of such a segment
constexpr int kListAhead = 16;      // list entries that a thread of the list kernel loads at once

// Two fp16 values <-> two 16-bit keys with the order of the values; -0 and +0 share a key.
__device__ __forceinline__ unsigned int order_keys(unsigned int h2) {
  const __half2 z = __hadd2(*reinterpret_cast<const __half2*>(&h2), __float2half2_rn(0.f));     // -0 + 0 = +0
  const unsigned int h = *reinterpret_cast<const unsigned int*>(&z);
  return h ^ (0x80008000u | ((h >> 15) & 0x00010001u) * 0x7FFFu);
}
__device__ __forceinline__ unsigned int key_halves(unsigned int k) { return k ^ (0x80008000u | ((~k >> 15) & 0x00010001u) * 0x7FFFu); }
__device__ __forceinline__ float key_value(unsigned int key) { return __half2float(__ushort_as_half((unsigned short)key_halves(key))); }
__device__ __forceinline__ unsigned int max2(unsigned int a, unsigned int b) { unsigned int r; asm("max.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b)); return r; }
__device__ __forceinline__ unsigned int min2(unsigned int a, unsigned int b) { unsigned int r; asm("min.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b)); return r; }

// Of a 256-bin histogram, the highest bin b with (count of the bins above b) < want <= (count of the bins >= b);
// over = the count of the bins above it.  One warp; lane l owns bins 8 l .. 8 l + 7.
__device__ __forceinline__ int pick_bin(const unsigned int* hist, int want, int lane, int& over) {
  unsigned int mine = 0u;
#pragma unroll
  for (int b = 0; b < 8; ++b) mine += hist[8 * lane + b];
  unsigned int incl = mine;                      // sum over lanes >= this one
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int v = __shfl_down_sync(0xffffffffu, incl, o);
    if (lane + o < 32) incl += v;
  }
  const unsigned int above = incl - mine;
  const bool here = above < (unsigned int)want && (unsigned int)want <= incl;
  const int src = __ffs((int)__ballot_sync(0xffffffffu, here)) - 1;
  int bin = 0, ov = 0;
  if (here) {
    unsigned int acc = above;
    for (int b = 7; b >= 0; --b) {
      const unsigned int c = hist[8 * lane + b];
      if (acc + c >= (unsigned int)want) { bin = 8 * lane + b; ov = (int)acc; break; }
      acc += c;
    }
  }
  over = __shfl_sync(0xffffffffu, ov, src);
  return __shfl_sync(0xffffffffu, bin, src);
}

// The k-th largest key of keys[0 .. n) and the k-th smallest, by two 8-bit histogram levels; beyond_t / beyond_b: how
// many keys lie strictly beyond them.  The smallest is the largest of the complemented keys: its first-level histogram
// is the mirror image of the other one, its second level is counted in the same pass.  One warp, hist = 512 words.
__device__ __forceinline__ void warp_select(const unsigned short* keys, int n, int k, unsigned int* hist, int lane,
                                            unsigned int& key_t, int& beyond_t, unsigned int& key_b, int& beyond_b) {
  unsigned int* hist_b = hist + 256;
  for (int i = lane; i < 256; i += 32) hist[i] = 0u;
  __syncwarp();
  for (int i = lane; i < n; i += 32) atomicAdd(&hist[keys[i] >> 8], 1u);
  __syncwarp();
  for (int i = lane; i < 256; i += 32) hist_b[i] = hist[255 - i];
  __syncwarp();
  int over_t, over_b;
  const unsigned int pre_t = (unsigned int)pick_bin(hist, k, lane, over_t);
  const unsigned int pre_b = (unsigned int)pick_bin(hist_b, k, lane, over_b);
  __syncwarp();
  for (int i = lane; i < 512; i += 32) hist[i] = 0u;
  __syncwarp();
  for (int i = lane; i < n; i += 32) {
    const unsigned int key = keys[i], kf = key ^ 0xFFFFu;
    if ((key >> 8) == pre_t) atomicAdd(&hist[key & 0xFFu], 1u);
    if ((kf >> 8) == pre_b) atomicAdd(&hist_b[kf & 0xFFu], 1u);
  }
  __syncwarp();
  int over2_t, over2_b;
  const unsigned int lo_t = (unsigned int)pick_bin(hist, k - over_t, lane, over2_t);
  const unsigned int lo_b = (unsigned int)pick_bin(hist_b, k - over_b, lane, over2_b);
  __syncwarp();
  key_t = (pre_t << 8) | lo_t;
  key_b = ((pre_b << 8) | lo_b) ^ 0xFFFFu;
  beyond_t = over_t + over2_t;
  beyond_b = over_b + over2_b;
}

// ---------------------------------------------------------------------------
// Filter_s of one channel by one warp without a pass over the histogram of all entries.  Each lane keeps the largest (or the two
// largest) entries of the even and of the odd positions that it reads: of these 64 (128) entries the (k + 1)-th largest is a
// bound that at least k + 1 and few more entries of the channel reach (k + 1 of 4096 normal entries: 60 % more at k = 41).
// Those are listed, and the k-th largest, the largest entry that stays and the ties are found among them; the smallest entries
// are the largest of the complemented keys.  Needs bounds that leave room between them and lists that fit; false leaves everything to the
// general routine.
// ---------------------------------------------------------------------------
constexpr int kListCap = 256;                 // entries of a list, 8 per lane

// the largest v for which `count(v)` (non-increasing) is at least `want`; lo: a v that is reached, hi: an upper limit
template <class Count>
__device__ __forceinline__ unsigned int bisect(unsigned int lo, unsigned int hi, int want, Count count) {
  const int nb = 32 - __clz((int)(lo ^ hi));
  unsigned int v = lo & ~((1u << nb) - 1u);
  for (int b = nb - 1; b >= 0; --b)
    if ((int)__reduce_add_sync(0xffffffffu, count(v | (1u << b))) >= want) v |= 1u << b;
  return v;
}

// One side among its list (key << 16 | token; the entries from the bound on): marks the k that leave in `omask`, returns the
// key next to them.
__device__ __forceinline__ unsigned int select_listed(const unsigned int* list, int cnt, int k, unsigned int bound, unsigned int top,
                                                      unsigned int* omask, int lane) {
  unsigned int c[kListCap / 32];
#pragma unroll
  for (int j = 0; j < kListCap / 32; ++j) c[j] = 32 * j + lane < cnt ? list[32 * j + lane] : 0u;
  const unsigned int kth = bisect(bound, top, k, [&](unsigned int v) {
    unsigned int n = 0u;
#pragma unroll
    for (int j = 0; j < kListCap / 32; ++j)
      if (32 * j < cnt) n += (c[j] >> 16) >= v;
    return n;
  });
  unsigned int n = 0u, next = 0u;              // beyond | equal << 16
#pragma unroll
  for (int j = 0; j < kListCap / 32; ++j) {
    const unsigned int key = c[j] >> 16;
    const bool there = 32 * j + lane < cnt;
    n += there && key > kth ? 1u : there && key == kth ? 0x10000u : 0u;
    if (key < kth) next = max(next, key);
  }
  n = __reduce_add_sync(0xffffffffu, n);
  next = __reduce_max_sync(0xffffffffu, next);
  const int need = k - (int)(n & 0xFFFFu);      // entries equal to the k-th that leave, lowest tokens first
  const bool tie = (int)(n >> 16) > need;
  int rank[kListCap / 32] = {};
  if (tie) {
    for (int i = 0; i < cnt; ++i) {
      const unsigned int w = list[i];
      if ((w >> 16) != kth) continue;
#pragma unroll
      for (int j = 0; j < kListCap / 32; ++j) rank[j] += w < c[j];            // equal keys order by token
    }
  }
#pragma unroll
  for (int j = 0; j < kListCap / 32; ++j) {
    if (32 * j + lane >= cnt) continue;
    const unsigned int key = c[j] >> 16, tok = c[j] & 0xFFFFu;
    if (key > kth || (key == kth && rank[j] < need)) atomicOr(&omask[tok >> 5], 1u << (tok & 31));
  }
  return tie ? kth : next;
}

template <bool TWO>
__device__ __forceinline__ bool select_channel(unsigned short* keys, int n, int k, unsigned int* lists, unsigned int* omask, int lane,
                                               unsigned int& kmin, unsigned int& kmax) {
  const uint4* kv = reinterpret_cast<const uint4*>(keys);
  unsigned int t1 = 0u, t2 = 0u, b1 = ~0u, b2 = ~0u;
  for (int v = lane; v < n / 8; v += 32) {
    const uint4 q = kv[v];
    const unsigned int w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (TWO) { t2 = max2(t2, min2(t1, w[i])); b2 = min2(b2, max2(b1, w[i])); }
      t1 = max2(t1, w[i]);
      b1 = min2(b1, w[i]);
    }
  }
  b1 = ~b1; b2 = ~b2;
  const unsigned int top = __reduce_max_sync(0xffffffffu, max(t1 >> 16, t1 & 0xFFFFu));
  const unsigned int bottom = __reduce_max_sync(0xffffffffu, max(b1 >> 16, b1 & 0xFFFFu));
  if (k == 0) { kmax = top; kmin = bottom ^ 0xFFFFu; return true; }
  auto bound = [&](unsigned int a, unsigned int b, unsigned int hi) {
    return bisect(0u, hi, k + 1, [&](unsigned int v) {
      unsigned int c = ((a >> 16) >= v) + ((a & 0xFFFFu) >= v);
      if (TWO) c += ((b >> 16) >= v) + ((b & 0xFFFFu) >= v);
      return c;
    });
  };
  const unsigned int lt = bound(t1, t2, top), lbc = bound(b1, b2, bottom), lb = lbc ^ 0xFFFFu;
  if (lt <= lb + 1u) return false;              // also where lanes have nothing (short channels)
  // entries >= lt or <= lb into their lists
  const unsigned int in_hi = (lt - 1u) * 0x10001u, in_lo = (lb + 1u) * 0x10001u;
  int ct = 0, cb = 0;
  for (int v0 = 0; v0 < n / 8; v0 += 128) {
    unsigned int m = 0u;                        // bit 4 j + i: low half of word i of vector j; + 16: high half
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int v = v0 + 32 * j + lane;
      if (v >= n / 8) break;
      const uint4 q = kv[v];
      const unsigned int w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) m |= min2(w[i] ^ min2(max2(w[i], in_lo), in_hi), 0x00010001u) << (4 * j + i);
    }
    while (__any_sync(0xffffffffu, m != 0u)) {
      const bool mine = m != 0u;
      const int bit = mine ? __ffs((int)m) - 1 : 0;
      m &= m - 1u;
      const unsigned int tok = (unsigned int)((v0 + 32 * ((bit >> 2) & 3) + lane) * 8 + 2 * (bit & 3) + (bit >> 4));
      const unsigned int key = mine ? keys[tok] : 0u;
      const bool is_t = mine && key >= lt;
      const unsigned int mt = __ballot_sync(0xffffffffu, is_t), mb = __ballot_sync(0xffffffffu, mine && !is_t);
      const unsigned int below = (1u << lane) - 1u;
      const int pos = is_t ? ct + __popc(mt & below) : cb + __popc(mb & below);
      if (mine && pos < kListCap) lists[(is_t ? 0 : kListCap) + pos] = ((is_t ? key : key ^ 0xFFFFu) << 16) | tok;
      ct += __popc(mt); cb += __popc(mb);
    }
  }
  if (ct > kListCap || cb > kListCap) return false;
  for (int i = lane; i < n / 32; i += 32) omask[i] = 0u;
  __syncwarp();
  kmax = select_listed(lists, ct, k, lt, top, omask, lane);
  kmin = select_listed(lists + kListCap, cb, k, lbc, bottom, omask, lane) ^ 0xFFFFu;
  __syncwarp();
  return true;
}

// Bound: shared-memory and load / store pipes (rows of the CTA's eight channels are 16 to 32 bytes of a line each), with the
// residual's bytes behind them; two histogram levels over all entries and residuals staged in shared memory made it 1145 us at 8 x 32
// heads x 4096, 4 bits, s = 2 %, now 517 (2 x 32 x 8192: 911 -> 309).  Two warps per channel, one for either side, come to the same
// (523 and 275 us, but 83 -> 99 at 4 x 32 x 1024).
template <int BITS>
__global__ void __launch_bounds__(kSelChannels * 32, 2) kcvt_select_kernel(KcvtArgs p) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const SegDesc& sd = p.seg;
  const int n_c = sd.n_c, k = sd.csr_k / 2;
  const int cg = blockIdx.x, bhl = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ch = cg * kSelChannels + warp;
  // shared memory: keys [8][n_c] u16 | outlier bitmask [8][n_c / 32] | histograms or lists [8][512]
  unsigned short* keys_all = reinterpret_cast<unsigned short*>(sm_raw);
  unsigned int* mask_all = reinterpret_cast<unsigned int*>(sm_raw + (size_t)kSelChannels * n_c * 2);
  unsigned int* hist_all = mask_all + kSelChannels * (n_c / 32);
  __shared__ float4 quant[kSelChannels];        // minimum, 1 / step, step of a channel
  unsigned short* keys = keys_all + (size_t)warp * n_c;
  unsigned int* omask = mask_all + warp * (n_c / 32);
  unsigned int* hist = hist_all + warp * 512;

  const __half* X = p.K + (size_t)bhl * n_c * kHeadDim;
  after_previous();
#pragma unroll 4
  for (int t2 = tid; t2 < n_c / 2; t2 += kSelChannels * 32) {  // 16 bytes (this CTA's 8 channels) of two token rows
    const uint4 a = *reinterpret_cast<const uint4*>(X + (size_t)(2 * t2) * kHeadDim + cg * kSelChannels);
    const uint4 b = *reinterpret_cast<const uint4*>(X + (size_t)(2 * t2 + 1) * kHeadDim + cg * kSelChannels);
    const unsigned int wa[4] = {a.x, a.y, a.z, a.w}, wb[4] = {b.x, b.y, b.z, b.w};
    unsigned int* dst = reinterpret_cast<unsigned int*>(keys_all) + t2;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      dst[(size_t)(2 * i) * (n_c / 2)] = order_keys(__byte_perm(wa[i], wb[i], 0x5410));
      dst[(size_t)(2 * i + 1) * (n_c / 2)] = order_keys(__byte_perm(wa[i], wb[i], 0x7632));
    }
  }
  __syncthreads();

  // ---- Filter_s (Eq. 4) on the channel's whole vector
  unsigned int kmin = 0xFFFFu, kmax = 0u;
  const bool few = k + 1 <= 48;                 // of 64 lane maxima; up to 112 of 128, beyond that the bound lets too many pass
  if (!(few ? select_channel<false>(keys, n_c, k, hist, omask, lane, kmin, kmax)
            : k + 1 <= 112 && select_channel<true>(keys, n_c, k, hist, omask, lane, kmin, kmax))) {
    kmin = 0xFFFFu; kmax = 0u;
    unsigned int key_t = 0xFFFFu, key_b = 0u;
    int need_t = 0, need_b = 0;                   // entries equal to the threshold key that still leave, lowest tokens first
    int beyond_t, beyond_b;
    warp_select(keys, n_c, k, hist, lane, key_t, beyond_t, key_b, beyond_b);
    need_t = k - beyond_t;
    need_b = k - beyond_b;
    const bool same = key_t == key_b;             // the thresholds meet only when all kept entries would be equal
    int eq_t = 0, eq_b = 0;
    for (int base = 0; base < n_c; base += 32) {
      const unsigned int key = keys[base + lane];
      bool out = false;
      {
        const bool is_t = key == key_t, is_b = key == key_b;
        out = key > key_t || key < key_b;
        if (__any_sync(0xffffffffu, is_t || is_b)) {        // an entry on a threshold: ties go to the lower token
          const unsigned int bt = __ballot_sync(0xffffffffu, is_t), bb = __ballot_sync(0xffffffffu, is_b);
          const unsigned int below = (1u << lane) - 1u;
          const int rt = eq_t + __popc(bt & below), rb = eq_b + __popc(bb & below);
          out = out || (is_t && rt < need_t) ||
                (is_b && (same ? (rt >= need_t && rt < need_t + need_b) : rb < need_b));
          eq_t += __popc(bt); eq_b += __popc(bb);
        }
      }
      const unsigned int bo = __ballot_sync(0xffffffffu, out);
      if (lane == 0) omask[base >> 5] = bo;
      if (!out) { kmin = min(kmin, key); kmax = max(kmax, key); }
    }
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    __syncwarp();
  }
  if (k > 0) {
    // the list of the outliers, token ascending: a lane has a run of mask words.  An outlier's key becomes the smallest kept one,
    // whose code and residual are zero.
    const int words = (n_c / 32 + 31) / 32, w0 = lane * words, w1 = min(w0 + words, n_c / 32);
    int mine = 0;
    for (int w = w0; w < w1; ++w) mine += __popc(omask[w]);
    int pos = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, pos, o);
      if (lane >= o) pos += v;
    }
    pos -= mine;
    unsigned int* olist = p.olist + ((size_t)bhl * kHeadDim + ch) * sd.csr_k;
    for (int w = w0; w < w1; ++w) {
      for (unsigned int m = omask[w]; m != 0u; m &= m - 1u) {
        const int tok = 32 * w + __ffs((int)m) - 1;
        unsigned int bits = key_halves(keys[tok]) & 0xFFFFu;
        if (bits == 0u || (bits & 0x7FFFu) > 0x7C00u)                 // the key has lost the sign of a zero and what kind of NaN
          bits = __half_as_ushort(X[(size_t)tok * kHeadDim + ch]);
        olist[pos++] = (unsigned int)tok | (bits << 16);
        keys[tok] = (unsigned short)kmin;
      }
    }
  }
  // ---- Eq. 2 on the kept entries: binary32, one rounding per operation
  const float mn = key_value(kmin), mx = key_value(kmax);
  const float levels = (float)((1 << BITS) - 1);
  const float range = __fsub_rn(mx, mn);
  const float d32 = __fdiv_rn(range, levels);
  const __half d16 = __float2half_rn(d32);
  const float d = __half2float(d16);
  const float inv = d != 0.f ? __fdiv_rn(1.0f, d) : 0.f;
  if (lane == 0) {
    quant[warp] = make_float4(mn, inv, d, 0.f);
    p.sz[(size_t)bhl * kHeadDim + ch] = __halves2half2(d16, __float2half_rn(mn));
    if (p.Rmax != nullptr) {        // a bound on the residuals of the channel
      atomicMax(p.Rmax + bhl * 2, __float_as_uint(residual_bound(mn, mx, range, d, levels)));
    }
  }
  // ---- codes and residuals: a thread takes four tokens of all eight channels, so that it has whole 32-byte sectors to store
  __syncthreads();
  float* R = p.R ? p.R + ((size_t)bhl * 2) * n_c * kHeadDim : nullptr;
  unsigned char* C8 = p.codes8 + (size_t)bhl * n_c * kHeadDim;
  for (int t4 = tid; t4 < n_c / 4; t4 += kSelChannels * 32) {
    float2 r[4][4];                             // [token][channel pair]
    unsigned int code[4][2] = {};
#pragma unroll
    for (int c = 0; c < kSelChannels; ++c) {
      const float4 qp = quant[c];
      const PairQuant quantize(qp.x, qp.y, qp.z, levels);
      const uint2 kk = *reinterpret_cast<const uint2*>(keys_all + (size_t)c * n_c + 4 * t4);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const unsigned int w = key_halves(h == 0 ? kk.x : kk.y);
        unsigned int c0, c1;
        const float2 e = quantize(__half22float2(*reinterpret_cast<const __half2*>(&w)), c0, c1);
        if (c & 1) { r[2 * h][c >> 1].y = e.x; r[2 * h + 1][c >> 1].y = e.y; }
        else { r[2 * h][c >> 1].x = e.x; r[2 * h + 1][c >> 1].x = e.y; }
        constexpr unsigned int kPut[4] = {0x3214u, 0x3240u, 0x3410u, 0x4210u};
        code[2 * h][c >> 2] = __byte_perm(code[2 * h][c >> 2], c0, kPut[c & 3]);
        code[2 * h + 1][c >> 2] = __byte_perm(code[2 * h + 1][c >> 2], c1, kPut[c & 3]);
      }
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const size_t row = (size_t)(4 * t4 + t) * kHeadDim + cg * kSelChannels;
      *reinterpret_cast<uint2*>(C8 + row) = make_uint2(code[t][0], code[t][1]);
      if (R != nullptr) store8(R + row, r[t]);
    }
  }
}

// One CTA per (batch, head): the per-channel outlier lists (token ascending) become per-block lists, and every
// block record gets its header fields of the key side and the channels' (scale, zero).
// Bound: latency; a channel's list is walked by one thread, so its entries are loaded sixteen at a time (8 x 32 heads x 4096
// 57 -> 36 us).
__global__ void __launch_bounds__(256) kcvt_list_kernel(KcvtArgs p) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const SegDesc& sd = p.seg;
  const int nblk = sd.nblk, k2 = sd.csr_k, bhl = blockIdx.x, tid = threadIdx.x;
  unsigned int* cnt = reinterpret_cast<unsigned int*>(sm_raw);          // [nblk][128], then exclusive offsets
  unsigned int* off = cnt + (size_t)nblk * kHeadDim;                   // [nblk + 1]
  unsigned int* dmax = off + nblk + 1;                                  // [nblk] bit patterns
  __shared__ unsigned int smax_bits;
  for (int i = tid; i < nblk * kHeadDim; i += blockDim.x) cnt[i] = 0u;
  for (int i = tid; i < nblk; i += blockDim.x) dmax[i] = 0u;
  if (tid == 0) smax_bits = 0u;
  after_previous();
  __syncthreads();
  const unsigned int* olist = p.olist + (size_t)bhl * kHeadDim * k2;
  const __half2* sz = p.sz + (size_t)bhl * kHeadDim;
  if (tid < kHeadDim) {
    for (int e0 = 0; e0 < k2; e0 += kListAhead) {
      unsigned int w[kListAhead];
#pragma unroll
      for (int i = 0; i < kListAhead; ++i) w[i] = e0 + i < k2 ? olist[tid * k2 + e0 + i] : 0u;
#pragma unroll
      for (int i = 0; i < kListAhead; ++i)
        if (e0 + i < k2) cnt[((w[i] & 0xFFFFu) / kBlockTok) * kHeadDim + tid] += 1u;
    }
    atomicMax(&smax_bits, __float_as_uint(__low2float(sz[tid])));      // scales are non-negative
  }
  __syncthreads();
  for (int b = tid; b < nblk; b += blockDim.x) {          // exclusive scan over the channels of a block
    unsigned int acc = 0u;
    for (int c = 0; c < kHeadDim; ++c) { const unsigned int v = cnt[b * kHeadDim + c]; cnt[b * kHeadDim + c] = acc; acc += v; }
    off[b + 1] = acc;
  }
  __syncthreads();
  if (tid == 0) {
    off[0] = 0u;
    for (int b = 0; b < nblk; ++b) off[b + 1] += off[b];
  }
  __syncthreads();
  unsigned char* seg0 = p.arena + sd.seg_base;
  unsigned char* csr = seg0 + (size_t)sd.csr_base16 * 16 + (size_t)(p.bh0 + bhl) * csr_stride_bytes(nblk, k2);
  unsigned int* g_off = reinterpret_cast<unsigned int*>(csr);
  unsigned int* g_ent = reinterpret_cast<unsigned int*>(csr + csr_offsets_bytes(nblk));
  for (int i = tid; i <= nblk; i += blockDim.x) g_off[i] = off[i];
  if (tid < kHeadDim) {
    const float zero = __high2float(sz[tid]);
    int prev_blk = -1, run = 0;
    for (int e0 = 0; e0 < k2; e0 += kListAhead) {
      unsigned int ws[kListAhead];
#pragma unroll
      for (int i = 0; i < kListAhead; ++i) ws[i] = e0 + i < k2 ? olist[tid * k2 + e0 + i] : 0u;
#pragma unroll
      for (int i = 0; i < kListAhead; ++i) {
        if (e0 + i >= k2) break;
        const unsigned int w = ws[i];
        const int tok = (int)(w & 0xFFFFu), blk = tok / kBlockTok;
        run = blk == prev_blk ? run + 1 : 0;
        prev_blk = blk;
        g_ent[off[blk] + cnt[blk * kHeadDim + tid] + run] =
            (unsigned int)(tok - blk * kBlockTok) | ((unsigned int)tid << 8) | (w & 0xFFFF0000u);
        const float v = __half2float(__ushort_as_half((unsigned short)(w >> 16)));
        atomicMax(&dmax[blk], __float_as_uint(fabsf(v - zero)));
      }
    }
  }
  __syncthreads();
  unsigned char* recs = seg0 + (size_t)(p.bh0 + bhl) * sd.bh_stride + sd.bfac_bytes;
  for (int i = tid; i < nblk * kHeadDim; i += blockDim.x) {
    const int b = i / kHeadDim, c = i % kHeadDim;
    reinterpret_cast<__half2*>(recs + (size_t)b * sd.rec_bytes + sd.off_kscale)[c] = sz[c];
  }
  for (int b = tid; b < nblk; b += blockDim.x) {
    float* hdr = reinterpret_cast<float*>(recs + (size_t)b * sd.rec_bytes);
    hdr[0] = __uint_as_float(dmax[b]);
    hdr[2] = __uint_as_float(smax_bits);
  }
}

template <int BITS>
__global__ void __launch_bounds__(128) kcvt_pack_kernel(KcvtArgs p) {
  constexpr int F = 8 / BITS, kPitch = kHeadDim + 4;
  __shared__ __align__(16) unsigned char codes[kBlockTok * kPitch];
  const SegDesc& sd = p.seg;
  const int blk = blockIdx.x, bhl = blockIdx.y, tid = threadIdx.x;
  after_previous();
  const unsigned char* C8 = p.codes8 + ((size_t)bhl * sd.n_c + (size_t)blk * kBlockTok) * kHeadDim;
  for (int i = tid; i < kBlockTok * 8; i += 128) {          // 16-byte pieces
    const int tok = i >> 3, q = i & 7;
    const uint4 v = reinterpret_cast<const uint4*>(C8)[i];
    unsigned int* dst = reinterpret_cast<unsigned int*>(codes + tok * kPitch + 16 * q);
    dst[0] = v.x; dst[1] = v.y; dst[2] = v.z; dst[3] = v.w;
  }
  __syncthreads();
  unsigned char* rec = p.arena + sd.seg_base + (size_t)(p.bh0 + bhl) * sd.bh_stride + sd.bfac_bytes +
                       (size_t)blk * sd.rec_bytes;
  unsigned int* dst = reinterpret_cast<unsigned int*>(rec + sd.off_kcodes);
  constexpr int kWords = kSlab * kHeadDim * BITS / 32;            // words per slab
  for (int li = tid; li < (kBlockTok / kSlab) * kWords; li += 128) {
    const int slab = li / kWords, wl = li % kWords;
    const int w = wl & 3, lane = (wl >> 2) & 31, tau = wl >> 7;
    const int tok = slab * kSlab + (lane >> 2) + 8 * (w & 1);
    const int ch = 32 * F * tau + 16 * (w >> 1) + 4 * (lane & 3);
    unsigned int word = 0;
#pragma unroll
    for (int j = 0; j < F; ++j)
      word |= *reinterpret_cast<const unsigned int*>(&codes[tok * kPitch + ch + 32 * j]) << (BITS * j);
    dst[li] = word;
  }
}

size_t kcvt_select_smem(int n_c) {
  return (size_t)kSelChannels * n_c * 2 + (size_t)kSelChannels * (n_c / 32) * 4 + kSelChannels * 512 * 4;
}
size_t kcvt_list_smem(int nblk) { return ((size_t)nblk * kHeadDim + 2 * (size_t)nblk + 1) * 4; }

bool kcvt_fits(int n_c) {
  return n_c % kBlockTok == 0 && n_c <= 65535 && kcvt_select_smem(n_c) <= 200 * 1024 &&
         kcvt_list_smem(n_c / kBlockTok) <= 200 * 1024;
}

size_t kcvt_workspace_bytes(int nbh, int n_c, int csr_k) {
  return (size_t)nbh * n_c * kHeadDim + (size_t)nbh * kHeadDim * csr_k * 4 + (size_t)nbh * kHeadDim * 4 + 256;
}

// Key side of a per-vector segment for the (batch, head) range of `a`; three launches.  Where they overlap, the select kernel may start
// when the values' CTAs end: those that came beside running ones shared SMs two by two while others fell idle (us, from the start / from
// the end, 4 bits without a low-rank part: three heads of 3072 tokens 62.4 / 47.2, four of 2560 56.7 / 45.2, eight of 4096 66.8 / 58.4;
// rank 4: three heads of 3072 128.2 / 107.4; nine heads of 4096 67.4 / 69.5; at 1024 tokens and less, or one head, as before).
cudaError_t launch_kcvt_keys(KcvtArgs a, int nbh, int bits, unsigned char* ws, bool overlap, cudaStream_t st) {
  const SegDesc& sd = a.seg;
  a.codes8 = ws;
  a.olist = reinterpret_cast<unsigned int*>(ws + (size_t)nbh * sd.n_c * kHeadDim);
  a.sz = reinterpret_cast<__half2*>(a.olist + (size_t)nbh * kHeadDim * sd.csr_k);
  const size_t sm_sel = kcvt_select_smem(sd.n_c), sm_list = kcvt_list_smem(sd.nblk);
  cudaError_t e;
  if (bits == 2) {
    e = cudaFuncSetAttribute(kcvt_select_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm_sel);
    if (e != cudaSuccess) return e;
    e = launch_after(overlap, kcvt_select_kernel<2>, dim3(kHeadDim / kSelChannels, nbh), kSelChannels * 32, sm_sel, st, a);
  } else {
    e = cudaFuncSetAttribute(kcvt_select_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm_sel);
    if (e != cudaSuccess) return e;
    e = launch_after(overlap, kcvt_select_kernel<4>, dim3(kHeadDim / kSelChannels, nbh), kSelChannels * 32, sm_sel, st, a);
  }
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(kcvt_list_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm_list);
  if (e == cudaSuccess) e = launch_after(overlap, kcvt_list_kernel, dim3(nbh), 256, sm_list, st, a);
  if (e == cudaSuccess) e = launch_after(overlap, bits == 2 ? kcvt_pack_kernel<2> : kcvt_pack_kernel<4>, dim3(sd.nblk, nbh), 128, 0, st, a);
  if (e == cudaSuccess) count_launches(3);
  return e;
}

}  // namespace gear
