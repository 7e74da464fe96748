// Decode attention (Eq. 1, one query per sequence) over the compressed cache:
//   scores = q . dequant(codes_K)^T + (q B_K) A_K^T + q . S_K^T      (+ q . K_buffer^T)
//   out    = softmax(scores) . [dequant(codes_V) + A_V B_V^T + S_V]  (+ . V_buffer)
// fp16 K / V are never materialised.
//
// Every warp is its own CTA and an independent stream processor.  The
// (batch, kv head, head pass, block) space is cut into contiguous ranges, one per
// warp.  A block travels as two items -- its key part and its value part --
// through a private shared-memory ring filled by bulk asynchronous copies
// (cp.async.bulk + mbarrier), so that the copies of the next items run while the
// warp works on the current one.
//
// Codes meet the query on the integer tensor cores (mma.sync.m16n8k32, u8 x s8
// for keys, u8 x u8 for values, s32 accumulation).  A packed word becomes fragment registers of the A operand
// with one AND per register: a b-bit field left where it sits in its byte is the
// code times a power of two, which the B operand (keys) or the output row
// (values) absorbs.  The B operand is a block-wide fixed-point image of
// q * scale (keys, per channel) or p * scale (values, per token and group), cut
// into base-256 digits ("limbs"; signed for keys), one column per limb: integer products
// are exact, so the result does not depend on any order of summation.  Key
// scores leave the integers once per 16-token slab; value sums stay in 32-bit
// integers across blocks and are folded into an fp32 copy in shared memory only
// when the running maximum, the fixed-point scale or the integer range demands
// it.  Zero-points go into one constant per block (keys) or an fp32 side sum
// (values); outlier corrections are scattered with 32-bit fixed-point
// shared-memory adds; the low-rank terms and the fp16 rows of the streaming
// buffer use the fp16 tensor-core path with an exact high / low split of the
// query-side operand.  A warp writes one partial (m, l, o) per (batch, head) it
// touched; the last warp to arrive for a (batch, head) merges them.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <type_traits>

#include "gear_decode.cuh"

namespace gear {

constexpr int kBufItem = kSlab * kBufPitch;     // one slab of key rows or of value rows
constexpr int kCsrAhead = 6;                    // outlier-list entries per lane requested one block ahead (per-vector keys)
// 32-bit words per fp16 B-fragment row set.  A row set holds, for every column that carries a query head (hi, lo) and
// every lane column t, two registers; with one head only two of the eight columns exist and the lanes of the other
// columns read those (their results are never used).  Padded against bank conflicts.
__host__ __device__ constexpr int frag_row_words(int hp) { return hp == 1 ? 24 : 72; }

static_assert(sizeof(SegDesc) <= 128 && sizeof(SegDesc) % 4 == 0, "descriptor copy assumes <= 32 words");

// ------------------------------------------------------------------ shared memory plan (per warp)
bool decode_plan(int bits, int heads, int ngv, int max_kpart, int max_vpart, int max_bfac, int max_T, size_t smem_budget,
                 int warps_cap, DecodeArgs* a) {
  (void)bits;
  const int HP = fp16_heads_per_pass(heads);
  const int frs = frag_row_words(HP);
  const int bregion = round_up(max_bfac / 2, 16);
  int part = max_kpart > max_vpart ? max_kpart : max_vpart;
  int stage = bregion + part;
  if (stage < kBufItem) stage = kBufItem;
  stage = round_up(stage, 16);
  if (max_T < kSlab) max_T = kSlab;
  const int nslab = max_T / kSlab, nchunk = (max_T + 31) / 32;
  // one region serves, in turn, the key B operand (limb rows), the value B operand (limb rows) with the fp16
  // probability fragments behind it, and the fp16 query / probability fragments of buffer slabs
  const int fragk = HP * 4 * kFragKRow * 4;
  const int fv_stride = nchunk * 8 + 8;
  const int fragv = round_up(ngv * HP * 4 * fv_stride * 4, 16);
  const int fragp = nslab * frs * 4;
  const int fragf = 9 * frs * 4;
  int xr = fragk > fragv + fragp ? fragk : fragv + fragp;
  if (fragf > xr) xr = fragf;
  WarpSmem w;
  int o = 0;
  w.sdc = o;     o += 128;
  w.qs = o;      o += HP * kHeadDim * 2;
  w.xr = o;      o += round_up(xr, 16);
  w.ps = o;      o += HP * max_T * 4;
  w.corr_k = o;  o += HP * max_T * 4;
  w.corr_v = o;  o += HP * kHeadDim * 4;
  w.ocorr = o;   o += HP * kHeadDim * 4;
  w.wl = o;      o += kMaxRank * 4 + 16;
  w.misc = o;    o += 32 + (kMaxStages + 1) * 8 + 8;   // exponents of max |q| per head, the ring's mbarriers, one test barrier
  w.ring = round_up(o, 16);
  w.fragv_stride = fv_stride;
  w.fragp = fragv;
  // most resident warps (in steps of four: one per scheduler) whose ring still holds two stages; then as many
  // stages as fit
  int reg_limit = HP == 1 ? 16 : 8;
  const bool capped = warps_cap > 0 && warps_cap < reg_limit;
  if (capped) reg_limit = warps_cap;
  for (int warps = reg_limit; warps >= 1; warps -= (warps > 12 ? 4 : 1)) {
    const long long per = (long long)smem_budget / warps - 1024;     // the system reserves 1 KB per CTA
    long long ns = (per - w.ring) / stage;
    if (ns < 2) continue;
    if (ns > kMaxStages) ns = kMaxStages;
    w.total = round_up(w.ring + (int)ns * stage, 16);
    // a cap below what the registers allow is enforced through the shared-memory request
    if (capped && warps == warps_cap) w.total = (int)(per & ~15LL);
    a->aligned = 0;
    a->nstage = (int)ns; a->stage_bytes = stage; a->bregion = bregion; a->max_T = max_T; a->hpa = HP; a->ws = w;
    a->spin_limit = kDecodeSpinLimit; a->test_dead_wait = 0; a->early_reads = 0; a->early_buf = 0; a->cta_warps = 1; a->unit_ctas = 0;
    a->wide = (HP == 1 && warps <= 12) ? 1 : 0;          // twelve warps or fewer: the 168-register build
    return true;
  }
  return false;
}

// ------------------------------------------------------------------ block shapes
int static_shape_id(const SegDesc& s, const CacheConst& c) {
  if (ShapeA1<2>::matches(s, c) || ShapeA1<4>::matches(s, c)) return 1;
  if (ShapeA2<2>::matches(s, c) || ShapeA2<4>::matches(s, c)) return 2;
  if (ShapeB1<2>::matches(s, c) || ShapeB1<4>::matches(s, c)) return 3;
  if (ShapeB2<2>::matches(s, c) || ShapeB2<4>::matches(s, c)) return 4;
  if (ShapeP1<2>::matches(s, c) || ShapeP1<4>::matches(s, c)) return 5;
  return 0;
}

// ------------------------------------------------------------------ the kernel
// HEADS = query heads handled per pass: 1, or 4 for grouped queries over an fp16 cache (a pass may hold fewer); compressed
// caches with several query rows per kv head take gear_decode_rows_kernel.
// MINB = resident warps per SM the registers are budgeted for: 16 (128 registers) or 12 (168 registers: about a tenth
// fewer instructions, for long streams where twelve warps are enough) with one head per pass, 8 with four.
// JOIN: up to sixteen warps of one unit per CTA, joined in shared memory at the end (short ranges of few units).
template <int BITS, int HEADS, int NGV, int MINB, bool JOIN>
__global__ void __launch_bounds__(JOIN ? 512 : 32, JOIN ? 1 : MINB) gear_decode_kernel(const __grid_constant__ DecodeArgs a) {
  constexpr int HP = HEADS;
  constexpr int F = 8 / BITS;                     // code fields per byte
  constexpr int kTop = BITS * (F - 1);            // the shift of the highest field
  constexpr int GV = kHeadDim / NGV;              // channels per value group
  constexpr int KT = 4 / F;                       // key tuples per slab
  constexpr int VT = 8 / F;                       // value tuples per 32-token chunk
  constexpr int kFragStride = frag_row_words(HP);
  constexpr int CMASK = HP == 1 ? 1 : 7;          // fp16 fragment columns that exist, as a mask on the lane's column
  extern __shared__ __align__(128) unsigned char smem_all[];

  const int lane = JOIN ? threadIdx.x & 31 : threadIdx.x, gid = lane >> 2, t = lane & 3, wrp = JOIN ? threadIdx.x >> 5 : 0;
  unsigned char* smem = smem_all + wrp * a.ws.total;
  const int G = a.group_heads;
  const int passes = (G + HP - 1) / HP;
  const int maxT = a.max_T;
  const int NS = a.nstage;
  const int RS = a.ws.fragv_stride;
  unsigned char* ring = smem + a.ws.ring;
  SegDesc* sdc = reinterpret_cast<SegDesc*>(smem + a.ws.sdc);
  __half* qs = reinterpret_cast<__half*>(smem + a.ws.qs);        // [HP][128] q
  uint32_t* xr = reinterpret_cast<uint32_t*>(smem + a.ws.xr);    // B-operand staging, see decode_plan
  uint32_t* fragPc = reinterpret_cast<uint32_t*>(smem + a.ws.xr + a.ws.fragp);   // fp16 probability fragments (compressed blocks)
  uint32_t* fragPb = xr + 8 * kFragStride;                       // the same for buffer slabs
  int* corr_k = reinterpret_cast<int*>(smem + a.ws.corr_k);      // [HP][maxT]
  float* ps = reinterpret_cast<float*>(smem + a.ws.ps);          // [HP][maxT] scores, then probabilities
  int* corr_v = reinterpret_cast<int*>(smem + a.ws.corr_v);      // [HP][128]
  float* ocorr = reinterpret_cast<float*>(smem + a.ws.ocorr);    // [HP][128] fp32 copy of the output accumulators
  float* wl = reinterpret_cast<float*>(smem + a.ws.wl);          // [16]
  int* qexp_s = reinterpret_cast<int*>(smem + a.ws.misc);        // [HP]
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + a.ws.misc + 32);   // [kMaxStages] ring, [kMaxStages] test barrier

  // lane roles in the integer products (one head): B / D column n is limb n % 4.  As owner of B column gid the lane fetches
  // limb gid % 4; as owner of D columns 2t, 2t + 1 it holds the limb pair t % 2.
  const int limb_b = gid & 3;
  const bool pair_hi = (t & 1) != 0;
  const bool writer = t == 0;                           // lanes that hold the low limb pair finish the sums

  if (lane == 0)
    for (int s = 0; s <= kMaxStages; ++s) mbar_init(&bar[s], 1);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  for (int i = lane; i < (a.ws.ps - a.ws.xr) / 4; i += 32) xr[i] = 0u;
  for (int i = lane; i < HP * maxT; i += 32) corr_k[i] = 0;
  for (int i = lane; i < HP * kHeadDim; i += 32) corr_v[i] = 0;
  __syncwarp();

  // ---- this warp's range of the flat (unit, block) space; unit = (batch, kv head, head pass)
  const int nbuf_blocks = (a.buf_len + kSlab - 1) / kSlab;
  const int NB = a.n_blocks_c + nbuf_blocks;
  int n_left, u, blk_lo;                        // blocks left for this warp, current unit, first block in it
  int part = 0, parts_u = 0;                    // unit-aligned split: this warp's range inside its unit, ranges of the unit
  if (JOIN) {
    const int W = blockDim.x >> 5;
    u = blockIdx.x / a.unit_ctas;
    part = (blockIdx.x % a.unit_ctas) * W + wrp;
    parts_u = a.unit_ctas * W;                                      // may exceed NB: the last warps have no block
    const int base = NB / parts_u, rem = NB - base * parts_u;
    blk_lo = part * base + min(part, rem);
    n_left = base + (part < rem ? 1 : 0);
  } else if (a.aligned) {
    int k = 0;
    while (k < 3 && (int)blockIdx.x >= a.cls_start[k + 1]) ++k;
    const int idx = blockIdx.x - a.cls_start[k];
    u = a.cls_u0[k] + idx / a.cls_n[k];
    part = a.cls_p0[k] + idx % a.cls_n[k];
    parts_u = u < a.units_a ? a.parts_a : a.parts_b;
    const int base = NB / parts_u, rem = NB - base * parts_u;       // base > 0: the host keeps parts <= NB
    blk_lo = part * base + min(part, rem);                          // the first `rem` ranges are one block longer
    n_left = base + (part < rem ? 1 : 0);
  } else {
    const long long Fl = (long long)a.cc.BH * passes * NB;
    const long long NW = gridDim.x, gw = blockIdx.x;
    const long long f0 = gw * Fl / NW, f1 = (gw + 1) * Fl / NW;
    if (f0 >= f1) return;                       // the host launches no more warps than blocks
    n_left = (int)(f1 - f0);
    u = (int)(f0 / NB);
    blk_lo = (int)(f0 - (long long)u * NB);
  }

  // Everything above used kernel parameters and shared memory only.  The launch is a programmatic dependent of the
  // kernel before it on the stream: it waits (griddepcontrol.wait) until that kernel has completed and its writes
  // are visible.  Only after its own wait does a decode kernel let its dependents start, so whoever starts early
  // knows that everything two launches back is complete.  When the host has seen another launch of the library on
  // this stream since the records (early_reads) and the buffer rows (early_buf: the kernel in front is the push of a
  // decoding step) were last written, the first copies of the ring -- descriptors, records, buffer rows -- are requested
  // before the wait, so that they travel while that kernel drains; the query and everything else is read after it.
  const bool early = early_start(a, NS, blk_lo, n_left);
  if (!early) asm volatile("griddepcontrol.wait;" ::: "memory");

  auto load_desc = [&](SegDesc* dst, int blk) {
    const int* src = reinterpret_cast<const int*>(a.table + a.blk2seg[blk]);
    __syncwarp();
    if (lane < (int)(sizeof(SegDesc) / 4)) reinterpret_cast<int*>(dst)[lane] = src[lane];
    __syncwarp();
  };

  // ---- producer: two items per block (key part, value part), issued in order into the ring
  int p_left = n_left, p_blk = blk_lo, p_share_lo = blk_lo, p_half = 0, p_stage = 0;
  int p_bh = u / passes, p_pass = u - p_bh * passes;
  int p_seg_lo = 0, p_seg_hi = 0, p_kbytes = 0, p_vbytes = 0, p_hb = 0;
  const unsigned char* p_segb = nullptr;        // B factors of the producer's (segment, batch, head)
  const unsigned char* p_rec = nullptr;         // record of block p_blk
  int n_inflight = 0;
  auto issue = [&]() {
    if (p_left == 0) return;
    unsigned char* dst = ring + p_stage * a.stage_bytes;
    uint64_t* b = &bar[p_stage];
    if (p_blk < a.n_blocks_c) {
      if (p_blk >= p_seg_hi) {                  // new segment (or new unit): read its descriptor
        const SegDesc* sd = a.table + a.blk2seg[p_blk];
        p_seg_lo = sd->blk_start;
        p_seg_hi = p_seg_lo + sd->nblk;
        p_kbytes = sd->off_vpart;
        p_vbytes = sd->rec_bytes - p_kbytes;
        p_hb = sd->bfac_bytes >> 1;
        p_segb = a.arena + sd->seg_base + (size_t)p_bh * sd->bh_stride;
        p_rec = p_segb + 2 * p_hb + (size_t)(p_blk - p_seg_lo) * (p_kbytes + p_vbytes);
      }
      if (lane == 0) {
        if (p_half == 0) {
          const bool wb = p_hb > 0 && (p_blk == p_seg_lo || p_blk == p_share_lo);
          mbar_expect_tx(b, p_kbytes + (wb ? p_hb : 0));
          if (wb) bulk_g2s(dst, p_segb, p_hb, b);
          bulk_g2s(dst + a.bregion, p_rec, p_kbytes, b);
        } else {
          const bool wb = p_hb > 0 && (p_blk == p_seg_hi - 1 || p_left == 1);
          mbar_expect_tx(b, p_vbytes + (wb ? p_hb : 0));
          if (wb) bulk_g2s(dst, p_segb + p_hb, p_hb, b);
          bulk_g2s(dst + a.bregion, p_rec + p_kbytes, p_vbytes, b);
        }
      }
    } else if (lane == 0) {
      const int j = p_blk - a.n_blocks_c;
      const int rows = min(kSlab, a.buf_len - j * kSlab);
      const __half* src = (p_half == 0 ? a.buf_k : a.buf_v) + ((size_t)p_bh * a.cc.n_b + (size_t)j * kSlab) * kHeadDim;
      mbar_expect_tx(b, rows * 256);
      for (int r = 0; r < rows; ++r) bulk_g2s(dst + r * kBufPitch, src + r * kHeadDim, 256, b);
    }
    ++n_inflight;
    if (++p_stage == NS) p_stage = 0;
    if (p_half == 0) {
      p_half = 1;
    } else {
      p_half = 0; --p_left; ++p_blk;
      p_rec += p_kbytes + p_vbytes;
      if (p_blk == NB) {
        p_blk = 0; p_share_lo = 0; p_seg_hi = 0;
        if (++p_pass == passes) { p_pass = 0; ++p_bh; }
      }
    }
  };
  for (int s = 0; s < NS; ++s) issue();
  int c_stage = 0, c_par = 0, c_seg_lo = 0, c_seg_hi = 0, c_shape = 0;
  if (early) {
    // The first block's descriptor, too (us without and with: one head of 256 tokens 6.73 / 6.34, 32 layers of one sequence 354 / 343,
    // four layers of 8 x 32 heads x 4096 155.2 / 152.6).
    if (n_left > 0 && blk_lo < a.n_blocks_c) {
      load_desc(sdc, blk_lo);
      c_seg_lo = sdc->blk_start;
      c_seg_hi = c_seg_lo + sdc->nblk;
      c_shape = sdc->shape_id;
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
  }
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  bool alive = true;
  // test only: a wait that nothing ends, so that the give-up path runs; the copies in flight are drained below
  if (a.test_dead_wait && !mbar_wait(&bar[kMaxStages], 0u, 64, a.status)) alive = false;
  // wait for the next item (items are consumed in order); returns its stage
  auto acquire = [&]() -> unsigned char* {
    unsigned char* st = ring + c_stage * a.stage_bytes;
    if (!mbar_wait(&bar[c_stage], (uint32_t)c_par, a.spin_limit, a.status)) alive = false;
    if (++c_stage == NS) { c_stage = 0; c_par ^= 1; }
    --n_inflight;
    return st;
  };
  auto release = [&]() {       // the oldest item is consumed: refill its stage
    __syncwarp();
    issue();
  };

  // the partials of a unit, all written and visible -> its output rows
  auto merge = [&](int unit, int row0, int rows, int n_parts) {
      const float* pb = a.partial + (size_t)unit * a.max_parts * (HP * kPartRow);
      const size_t pstride = (size_t)HP * kPartRow;
      for (int h = 0; h < rows; ++h) {
        // Chunks of up to 16 partials: every load of a chunk (lane i: max and denominator of partial i; all lanes: their
        // four channels of every partial) is issued before anything is used, so a chunk costs one round trip to L2.
        float M = -INFINITY, den = 0.f, n0 = 0.f, n1 = 0.f, n2 = 0.f, n3 = 0.f;
        for (int base = 0; base < n_parts; base += 16) {
          const int cnt = min(16, n_parts - base);
          const float* ph = pb + (size_t)base * pstride + h * kPartRow;
          float mi = -INFINITY, li = 0.f;
          if (lane < cnt) { mi = __ldcg(ph + lane * pstride + 128); li = __ldcg(ph + lane * pstride + 129); }
          float4 v[16];
#pragma unroll
          for (int j = 0; j < 16; ++j)
            v[j] = j < cnt ? __ldcg(reinterpret_cast<const float4*>(ph + j * pstride) + lane) : make_float4(0.f, 0.f, 0.f, 0.f);
          const float Mn = fmaxf(M, warp_max(mi));
          const float resc = M == -INFINITY ? 0.f : exp2f(M - Mn);
          const float wgt = mi == -INFINITY ? 0.f : exp2f(mi - Mn);
          float dsum = wgt * li;
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) dsum += __shfl_xor_sync(0xffffffffu, dsum, o);
          den = fmaf(den, resc, dsum);
          n0 *= resc; n1 *= resc; n2 *= resc; n3 *= resc;
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const float wj = __shfl_sync(0xffffffffu, wgt, j);
            n0 = fmaf(wj, v[j].x, n0); n1 = fmaf(wj, v[j].y, n1); n2 = fmaf(wj, v[j].z, n2); n3 = fmaf(wj, v[j].w, n3);
          }
          M = Mn;
        }
        const float inv = 1.0f / den;
        *reinterpret_cast<float4*>(a.out + (size_t)(row0 + h) * kHeadDim + lane * 4) =
            make_float4(n0 * inv, n1 * inv, n2 * inv, n3 * inv);
      }
  };

  // ---- loop over the units this warp touches
  const int unit0 = u;
  float* ml_s = reinterpret_cast<float*>(qexp_s + HP);          // [2] maximum and denominator of the warp's range (JOIN)
  if (JOIN && lane == 0) { ml_s[0] = -INFINITY; ml_s[1] = 0.f; }
  while (n_left > 0 && alive) {
    const int blk_hi = min(NB, blk_lo + n_left);
    const int c_hi = min(blk_hi, a.n_blocks_c);          // end of the compressed blocks of this range
    const int bh = u / passes, pass = u - bh * passes;
    const int HPu = HEADS == 1 ? 1 : min(HP, G - pass * HP);   // query heads this pass holds
    constexpr int HC = HP;          // heads computed: a pass with fewer heads carries zero queries in the others, so that
                                    // nothing in the block loop depends on the count; only the stores to global memory do
    const int hq0 = bh * G + pass * HP;                 // first query head of this pass

    // unit state
    float m_run[HP], l_run[HP];
#pragma unroll
    for (int h = 0; h < HP; ++h) { m_run[h] = -INFINITY; l_run[h] = 0.f; }

    // query rows of this pass -> shared (fp16 as given); exponent of max |q * scale|; the fp32 output copy starts at 0
    float qreg[4] = {0.f, 0.f, 0.f, 0.f};               // one head per pass: this lane's four channels of q * scale * log2 e
    __syncwarp();
#pragma unroll
    for (int h = 0; h < HP; ++h) {
      {
        const uint2 v = h < HPu ? *reinterpret_cast<const uint2*>(a.q + (size_t)(hq0 + h) * kHeadDim + lane * 4)
                                : make_uint2(0u, 0u);
        *reinterpret_cast<uint2*>(qs + h * kHeadDim + lane * 4) = v;
        const __half2 q01 = u32_as_h2(v.x), q23 = u32_as_h2(v.y);
        const float4 qv = make_float4(__low2float(q01) * a.scale_log2, __high2float(q01) * a.scale_log2,
                                      __low2float(q23) * a.scale_log2, __high2float(q23) * a.scale_log2);
        if (HP == 1) { qreg[0] = qv.x; qreg[1] = qv.y; qreg[2] = qv.z; qreg[3] = qv.w; }
        const float mx = warp_max(fmaxf(fmaxf(fabsf(qv.x), fabsf(qv.y)), fmaxf(fabsf(qv.z), fabsf(qv.w))));
        if (lane == 0) qexp_s[h] = float_exponent(mx);
      }
      *reinterpret_cast<float4*>(ocorr + h * kHeadDim + lane * 4) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncwarp();

    // scale everything accumulated in fp32 for head h by alpha[h] (the running maximum grew)
    auto scale_ocorr = [&](const float (&alpha)[HP]) {
#pragma unroll
      for (int h = 0; h < HP; ++h) {
        if (h < HC) {
          float4* oc = reinterpret_cast<float4*>(ocorr + h * kHeadDim + lane * 4);
          float4 v = *oc;
          v.x *= alpha[h]; v.y *= alpha[h]; v.z *= alpha[h]; v.w *= alpha[h];
          *oc = v;
        }
      }
    };

    // ==================================================================== compressed blocks
    if constexpr (HEADS == 1) if (blk_lo < c_hi) {
      int O[8][4];                                       // value sums: a tile of 16 channels each, 32-bit integers
      float U[4], cm[NGV];
      uint32_t bw[2] = {0u, 0u};                         // low-rank key term: B operand (q B_K) of the current segment
#pragma unroll
      for (int mt = 0; mt < 8; ++mt)
#pragma unroll
        for (int k = 0; k < 4; ++k) O[mt][k] = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k) U[k] = 0.f;
#pragma unroll
      for (int g = 0; g < NGV; ++g) cm[g] = 0.f;
      bool u_pending = false;
      int eV_cur = 1000;                                 // exponent of the value fixed-point scale the integer sums carry
      int tok_acc = 0;                                   // tokens in the integer sums since they were last folded

      // integer sums -> fp32 copy in shared memory, times alpha; the integers start again from zero
      auto fold_O = [&](float alpha) {
        const float fs = pow2i(-eV_cur);
        __syncwarp();
        const float w1 = pair_hi ? 0.f : 256.f;              // the high pair's second column is no limb: dropped
        const float w0 = pair_hi ? 65536.f * fs : fs;
#pragma unroll
        for (int mt = 0; mt < 8; ++mt) {
          const float rs = w0 * (1.0f / (float)(1 << (BITS * (mt % F))));
          float v0 = fmaf((float)O[mt][1], w1, (float)O[mt][0]) * rs;
          float v1 = fmaf((float)O[mt][3], w1, (float)O[mt][2]) * rs;
          v0 += __shfl_xor_sync(0xffffffffu, v0, 1);
          v1 += __shfl_xor_sync(0xffffffffu, v1, 1);
          if (writer) {
            float* oc = ocorr + 16 * mt + gid;
            oc[0] = (oc[0] + v0) * alpha;
            oc[8] = (oc[8] + v1) * alpha;
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) O[mt][i] = 0;
        }
        __syncwarp();
      };

      // outlier lists of per-vector key segments: this lane's offset, the entries requested ahead for block cs_blk
      // (such segments have one value group per token: the state exists in the NGV = 1 kernels only)
      constexpr int kAhead = NGV == 1 ? kCsrAhead : 1;
      unsigned int cs_off = 0u, cs_e[kAhead];
      int cs_seg = -1, cs_unit = -1, cs_base = 0, cs_blk = -1;
#pragma unroll
      for (int j = 0; j < kAhead; ++j) cs_e[j] = 0u;
#pragma unroll 1
      for (int blk = blk_lo; blk < c_hi; ++blk) {
        if (blk >= c_seg_hi || blk < c_seg_lo) {
          load_desc(sdc, blk);
          c_seg_lo = sdc->blk_start;
          c_seg_hi = c_seg_lo + sdc->nblk;
          c_shape = sdc->shape_id;
        }
        auto body = [&](auto shape_tag) {
          using S = decltype(shape_tag);
          // ---------------- block geometry
          const int T = S::kDyn ? sdc->T : S::T;
          const int r_pad = S::kDyn ? sdc->r_pad : S::r_pad;
          const int k2k = S::kDyn ? 2 * sdc->k_k : S::k2k;
          const int k2v = S::kDyn ? 2 * a.cc.k_v : S::k2v;
          const int off_kscale = S::kDyn ? sdc->off_kscale : S::off_kscale;
          const int off_koval = S::kDyn ? sdc->off_koval : S::off_koval;
          const int off_koidx = S::kDyn ? sdc->off_koidx : S::off_koidx;
          const int off_kcodes = S::kDyn ? sdc->off_kcodes : S::off_kcodes;
          const int off_ak = S::kDyn ? sdc->off_ak : S::off_ak;
          const int o_av = S::kDyn ? sdc->off_av - sdc->off_vpart : S::off_av;
          const int o_vsz = S::kDyn ? sdc->off_vscale - sdc->off_vpart : S::off_vscale;
          const int o_voval = S::kDyn ? sdc->off_voval - sdc->off_vpart : S::off_voval;
          const int o_voidx = S::kDyn ? sdc->off_voidx - sdc->off_vpart : S::off_voidx;
          const bool with_bk = r_pad > 0 && (blk == c_seg_lo || blk == blk_lo);
          const bool with_bv = r_pad > 0 && (blk == c_seg_hi - 1 || blk == blk_hi - 1);
          const int nslab = (T + kSlab - 1) / kSlab;        // a block may end inside a slab (tokens past T: no score)
          const int nchunk = (T + 31) / 32;

          // ================================================================ key item
          unsigned char* stK = acquire();
          if (!alive) return;
          const unsigned char* kp = stK + a.bregion;
          const float dmax_k = reinterpret_cast<const float*>(kp)[0];
          const float dmax_v = reinterpret_cast<const float*>(kp)[1];
          const float smax_v = reinterpret_cast<const float*>(kp)[3];
          int sexp_k;                                     // exponent of the sparse key term's fixed-point scale
          float c_zero;                                   // sum over channels of q * zero-point
          float kscl;                                     // what turns this lane's integer sums into scores

          if (with_bk) {
            // w = q B_K through the fp16 tensor cores, kept as the B operand of the low-rank key term
            const __half* bk = reinterpret_cast<const __half*>(stK);     // [r_pad][128]
            float wacc[4] = {0.f, 0.f, 0.f, 0.f}, wodd[4] = {0.f, 0.f, 0.f, 0.f};     // two chains where latency counts (344.4 / 343.3)
#pragma unroll (JOIN ? 4 : 2)
            for (int kc = 0; kc < 8; ++kc) {
              uint32_t af[4] = {0u, 0u, 0u, 0u};
              if (gid < r_pad) {
                af[0] = *reinterpret_cast<const uint32_t*>(bk + gid * kHeadDim + 16 * kc + 2 * t);
                af[2] = *reinterpret_cast<const uint32_t*>(bk + gid * kHeadDim + 16 * kc + 2 * t + 8);
              }
              if (gid + 8 < r_pad) {
                af[1] = *reinterpret_cast<const uint32_t*>(bk + (gid + 8) * kHeadDim + 16 * kc + 2 * t);
                af[3] = *reinterpret_cast<const uint32_t*>(bk + (gid + 8) * kHeadDim + 16 * kc + 2 * t + 8);
              }
              uint32_t b0 = 0u, b1 = 0u;
              if ((gid & 1) == 0 && gid < 2) {      // column 0 (written as gid == 0, a launch of one block per warp takes 0.2 us more)
                const __half* qrow = qs + 16 * kc + 2 * t;
                b0 = *reinterpret_cast<const uint32_t*>(qrow);
                b1 = *reinterpret_cast<const uint32_t*>(qrow + 8);
              }
              if (JOIN && (kc & 1)) mma16816(wodd, af, b0, b1);
              else mma16816(wacc, af, b0, b1);
            }
            __syncwarp();
            if (t == 0) {                           // D[rho][column 0] = w[rho]
              wl[gid] = (wacc[0] + wodd[0]) * a.scale_log2;
              wl[gid + 8] = (wacc[2] + wodd[2]) * a.scale_log2;
            }
            __syncwarp();
            // B operand of the low-rank key product: columns 0, 4 hold the high parts, 1, 5 the remainders, the others are
            // zero -- so that the lane that finishes the integer sum also receives the low-rank term
            uint32_t hi0, lo0, hi1, lo1;
            split_hi_lo(wl[2 * t], wl[2 * t + 1], hi0, lo0);
            split_hi_lo(wl[2 * t + 8], wl[2 * t + 9], hi1, lo1);
            bw[0] = limb_b == 0 ? hi0 : (limb_b == 1 ? lo0 : 0u);
            bw[1] = limb_b == 0 ? hi1 : (limb_b == 1 ? lo1 : 0u);
            __syncwarp();
          }

          // ---------------- B operand of the key scores: the block-wide fixed-point image of q * scale per channel,
          //                  as four signed base-256 digits; sum of q * zero; sparse key term scattered to its token
          {
            const uint4 kz = reinterpret_cast<const uint4*>(kp + off_kscale)[lane];
            const uint32_t w4[4] = {kz.x, kz.y, kz.z, kz.w};
            float sc4[4], zr4[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              sc4[j] = __low2float(u32_as_h2(w4[j]));
              zr4[j] = __high2float(u32_as_h2(w4[j]));
            }
            // this lane's four channels sit in 32-channel chunk lane / 8, i.e. in code field (lane / 8) % F: the digits
            // carry the power of two that brings every field to the weight of the highest one
            const int sh = BITS * (F - 1 - ((lane >> 3) % F));
            const uint32_t mulc = 1u << sh, addc = 0x80808080u - (kMagicBits << sh);
            const int ed = float_exponent(dmax_k);
            float qd[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) qd[j] = qreg[j] * sc4[j];
            const float am = fmaxf(fmaxf(fabsf(qd[0]), fabsf(qd[1])), fmaxf(fabsf(qd[2]), fabsf(qd[3])));
            const uint32_t mb = warp_max_u32(__float_as_uint(am));         // non-negative floats order like their bits
            const int e = clamp60(21 - ((int)(mb >> 23) - 127));            // |q * scale| * 2^e < 2^22
            const float Sk = pow2i(e);
            uint32_t z[4];
#pragma unroll
            for (int j = 0; j < 4; ++j)
              z[j] = (__float_as_uint(fmaf(qd[j], Sk, kMagic)) * mulc + addc) ^ 0x80808080u;    // balanced digits
            // digits of four channels -> one register per limb (bytes = the lane's four channels in order)
            const uint32_t p01l = __byte_perm(z[0], z[1], 0x5140), p23l = __byte_perm(z[2], z[3], 0x5140);
            const uint32_t p01h = __byte_perm(z[0], z[1], 0x7362), p23h = __byte_perm(z[2], z[3], 0x7362);
            uint32_t* row = xr + (lane >> 3) * 8 + (lane & 3) * 2 + ((lane >> 2) & 1);
            row[0] = __byte_perm(p01l, p23l, 0x5410);
            row[kFragKRow] = __byte_perm(p01l, p23l, 0x7632);
            row[2 * kFragKRow] = __byte_perm(p01h, p23h, 0x5410);
            row[3 * kFragKRow] = __byte_perm(p01h, p23h, 0x7632);

            float c = fmaf(qreg[0], zr4[0], fmaf(qreg[1], zr4[1], fmaf(qreg[2], zr4[2], qreg[3] * zr4[3])));   // this lane's part
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
            c_zero = c;
            sexp_k = clamp60(21 - qexp_s[0] - ed);
            const float Sx = pow2i(sexp_k);
            const float qS[4] = {qreg[0] * Sx, qreg[1] * Sx, qreg[2] * Sx, qreg[3] * Sx};
            // the inverse fixed-point scale, the weight of the highest field, and 2^16 for the high limb pair
            kscl = pow2i(-e - kTop + (pair_hi ? 16 : 0));
            if (k2k > 0) {
              auto k_entry = [&](int j, float val, int idx) {
                const float d = val - zr4[j];
                atomicAdd(&corr_k[idx], __float2int_rn(qS[j] * d));
              };
              if (k2k == 2) {
                const uint4 ov = reinterpret_cast<const uint4*>(kp + off_koval)[lane];
                const uint2 oi = reinterpret_cast<const uint2*>(kp + off_koidx)[lane];
                const uint32_t o4[4] = {ov.x, ov.y, ov.z, ov.w};
                const uint32_t i2[2] = {oi.x, oi.y};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                  k_entry(j, __low2float(u32_as_h2(o4[j])), (i2[j >> 1] >> (16 * (j & 1))) & 0xFFu);
                  k_entry(j, __high2float(u32_as_h2(o4[j])), (i2[j >> 1] >> (16 * (j & 1) + 8)) & 0xFFu);
                }
              } else if (k2k == 4) {
                // this lane's 4 channels x 4 entries: 32 bytes of values, 16 bytes of token indices
                const uint4 ova = reinterpret_cast<const uint4*>(kp + off_koval)[2 * lane];
                const uint4 ovb = reinterpret_cast<const uint4*>(kp + off_koval)[2 * lane + 1];
                const uint4 oi = reinterpret_cast<const uint4*>(kp + off_koidx)[lane];
                const uint32_t o8[8] = {ova.x, ova.y, ova.z, ova.w, ovb.x, ovb.y, ovb.z, ovb.w};
                const uint32_t i4[4] = {oi.x, oi.y, oi.z, oi.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                  k_entry(j, __low2float(u32_as_h2(o8[2 * j])), i4[j] & 0xFFu);
                  k_entry(j, __high2float(u32_as_h2(o8[2 * j])), (i4[j] >> 8) & 0xFFu);
                  k_entry(j, __low2float(u32_as_h2(o8[2 * j + 1])), (i4[j] >> 16) & 0xFFu);
                  k_entry(j, __high2float(u32_as_h2(o8[2 * j + 1])), i4[j] >> 24);
                }
              } else {
                const __half* ov = reinterpret_cast<const __half*>(kp + off_koval) + lane * 4 * k2k;
                const unsigned char* oi = kp + off_koidx + lane * 4 * k2k;
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll 1
                  for (int e = 0; e < k2k; ++e) k_entry(j, __half2float(ov[j * k2k + e]), oi[j * k2k + e]);
              }
            }
            if (NGV == 1 && S::kCsr && sdc->csr_base16 != 0) {
              // per-vector keys: the block's outliers come from the list of the (batch, head), any channel to any lane.
              // A lane keeps one offset of the list (31 blocks per load), and the entries of the next block are
              // requested as soon as this block's are used, so that they arrive during the rest of the block.
              const unsigned char* csr = a.arena + sdc->seg_base + (size_t)sdc->csr_base16 * 16 +
                                         (size_t)bh * csr_stride_bytes(sdc->nblk, sdc->csr_k);
              const unsigned int* offs = reinterpret_cast<const unsigned int*>(csr);
              const unsigned int* ent = reinterpret_cast<const unsigned int*>(csr + csr_offsets_bytes(sdc->nblk));
              const int bi = blk - c_seg_lo;
              if (cs_seg != c_seg_lo || cs_unit != u || bi < cs_base || bi + 1 > cs_base + 31) {
                cs_seg = c_seg_lo; cs_unit = u; cs_base = bi; cs_blk = -1;
                cs_off = bi + lane <= sdc->nblk ? offs[bi + lane] : 0u;
              }
              const unsigned int e_lo = __shfl_sync(0xffffffffu, cs_off, bi - cs_base);
              const unsigned int e_hi = __shfl_sync(0xffffffffu, cs_off, bi - cs_base + 1);
              const __half2* szp = reinterpret_cast<const __half2*>(kp + off_kscale);
              auto apply = [&](unsigned int w) {
                const int tok = (int)(w & 0xFFu), ch = (int)((w >> 8) & 0xFFu);
                const float d = __half2float(__ushort_as_half((unsigned short)(w >> 16))) - __high2float(szp[ch]);
                const float qv = __half2float(qs[ch]) * a.scale_log2;
                atomicAdd(&corr_k[tok], __float2int_rn(qv * pow2i(sexp_k) * d));
              };
              const bool have = cs_blk == blk;
#pragma unroll
              for (int j = 0; j < kAhead; ++j) {
                const unsigned int e = e_lo + lane + 32 * j;
                if (e < e_hi) apply(have ? cs_e[j] : ent[e]);
              }
              for (unsigned int e = e_lo + lane + 32 * kAhead; e < e_hi; e += 32) apply(ent[e]);
              if (blk + 1 < min(c_hi, c_seg_hi) && bi + 2 <= cs_base + 31) {
                const unsigned int n_lo = __shfl_sync(0xffffffffu, cs_off, bi + 1 - cs_base);
                const unsigned int n_hi = __shfl_sync(0xffffffffu, cs_off, bi + 2 - cs_base);
#pragma unroll
                for (int j = 0; j < kAhead; ++j) {
                  const unsigned int e = n_lo + lane + 32 * j;
                  cs_e[j] = e < n_hi ? ent[e] : 0u;
                }
                cs_blk = blk + 1;
              }
            }
          }
          __syncwarp();
          // this lane's B registers: limb gid % 4 for the four 32-channel chunks
          uint32_t bK[4][2];
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const uint2 v = *reinterpret_cast<const uint2*>(xr + limb_b * kFragKRow + 2 * t + c * 8);
            bK[c][0] = v.x; bK[c][1] = v.y;
          }

          // ---------------- key scores, slab by slab; scores go to shared memory
          {
            const bool pa0 = 2 * t < r_pad, pa1 = 2 * t + 8 < r_pad;
            const uint4* cwp = reinterpret_cast<const uint4*>(kp + off_kcodes) + lane;
            const __half* akp = reinterpret_cast<const __half*>(kp + off_ak) + gid * r_pad + 2 * t;
            const int ak8 = 8 * r_pad, ak_step = kSlab * r_pad;
            int tok0 = gid;
#pragma unroll (S::unroll)
            for (int slab = 0; slab < nslab; ++slab) {
              int acc[4] = {0, 0, 0, 0};
#pragma unroll
              for (int tau = 0; tau < KT; ++tau) {
                const uint4 w = cwp[tau * 32];
#pragma unroll
                for (int j = 0; j < F; ++j) {
                  constexpr uint32_t m0 = field_mask<BITS>(0);
                  const uint32_t m = m0 << (BITS * j);
                  const uint32_t af[4] = {w.x & m, w.y & m, w.z & m, w.w & m};
                  imma16832(acc, af, bK[F * tau + j][0], bK[F * tau + j][1]);
                }
              }
              cwp += KT * 32;
              // low-rank key term: A_K rows times w (zero rows when r = 0)
              uint32_t aa[4] = {0u, 0u, 0u, 0u};
              if (pa0) {
                aa[0] = *reinterpret_cast<const uint32_t*>(akp);
                aa[1] = *reinterpret_cast<const uint32_t*>(akp + ak8);
              }
              if (pa1) {
                aa[2] = *reinterpret_cast<const uint32_t*>(akp + 8);
                aa[3] = *reinterpret_cast<const uint32_t*>(akp + ak8 + 8);
              }
              akp += ak_step;
              // low limb pair + 2^16 high limb pair, each lane converting its own pair; the partner adds the other
              float f0 = (float)(acc[0] + acc[1] * 256) * kscl;
              float f1 = (float)(acc[2] + acc[3] * 256) * kscl;
              f0 += __shfl_xor_sync(0xffffffffu, f0, 1);
              f1 += __shfl_xor_sync(0xffffffffu, f1, 1);
              if (r_pad > 0) {
                float d[4];
                mma16816_z(d, aa, bw[0], bw[1]);
                f0 += d[0] + d[1];
                f1 += d[2] + d[3];
              }
              if (writer) {
                // raw sums only: the zero-point constant and the sparse term are added in the softmax pass
                ps[tok0] = f0; ps[tok0 + 8] = f1;
              }
              tok0 += kSlab;
            }
          }
          release();                                      // the key item is consumed

          // ================================================================ value item
          unsigned char* stV = acquire();
          if (!alive) return;
          const unsigned char* vp = stV + a.bregion;          // value part of the record

          // ---------------- softmax over the block, the B operands of the value products and the sparse value term in
          //                  one pass over this lane's token pairs (pairs lane, lane + 32), probabilities in registers
          constexpr int NPR = S::kDyn ? 2 : (S::T > 64 ? S::T / 64 : 1);
          // The integer value sums carry the scale 2^eV_cur, which a block keeps when p * scale * 2^eV_cur stays below 2^23 at
          // p = 1 and is no more than three bits short of it (precision).  What is left of those bits is room for the
          // running maximum to lag behind: it is moved, and everything summed so far scaled, only when a score exceeds it
          // by more than that, because the integers have to be folded into the fp32 copy then.  (Every second or third
          // block of a short range raises the maximum by a little.)
          const int need = clamp60(22 - float_exponent(smax_v));
          const bool exp_bad = eV_cur > need || eV_cur < need - 3;
          const int eV_new = exp_bad ? need - kLag : eV_cur;
          const float room = (float)(need - eV_new);
          float2 sc[NPR];
          const float Sik = pow2i(-sexp_k);
          float mx = -INFINITY;
#pragma unroll
          for (int i = 0; i < NPR; ++i) {
            const int tp = 2 * (lane + 32 * i);
            float2 v = make_float2(-INFINITY, -INFINITY);
            if (tp < T) {
              v = *reinterpret_cast<const float2*>(ps + tp);
              v.x += c_zero; v.y += c_zero;
              if (k2k > 0 || (NGV == 1 && S::kCsr && sdc->csr_base16 != 0)) {
                const int2 c = *reinterpret_cast<const int2*>(corr_k + tp);
                v.x = fmaf((float)c.x, Sik, v.x);
                v.y = fmaf((float)c.y, Sik, v.y);
                *reinterpret_cast<int2*>(corr_k + tp) = make_int2(0, 0);
              }
            }
            sc[i] = v;
            mx = fmaxf(mx, fmaxf(v.x, v.y));
          }
          mx = warp_max(mx);
          const bool grew = mx > m_run[0] + room;         // warp-uniform
          float alpha = 1.f;
          if (grew) {
            alpha = exp2f(m_run[0] - mx);
            m_run[0] = mx;
          }
          const float m_new = m_run[0];
          // the sparse value term's fixed point is set for probabilities of one at most: the block's own maximum
          const float lag = pow2i(-max(0, (int)ceilf(mx - m_new)));
          // The integers are folded into the fp32 copy when the maximum moved (everything so far shrinks by alpha), when this
          // block's scales do not fit their exponent, or when the 32-bit range nears its end.
          {
            const bool conv = tok_acc > 0 && (grew || exp_bad || tok_acc + T > kTokLimit);
            if (conv) {
              fold_O(alpha);
              tok_acc = 0;
            } else if (grew) {
              const float of_head[HP] = {alpha};
              scale_ocorr(of_head);
            }
            if (grew) {
#pragma unroll
              for (int i = 0; i < 4; ++i) U[i] *= alpha;
#pragma unroll
              for (int g = 0; g < NGV; ++g) cm[g] *= alpha;
            }
            eV_cur = eV_new;                    // a change comes with a fold (or with empty sums)
            tok_acc += T;
          }
          const float Sv = pow2i(eV_cur);
          const float Sx = pow2i(clamp60(21 - float_exponent(dmax_v)));     // fixed-point scale of the sparse value term
          const __half2* vsz = reinterpret_cast<const __half2*>(vp + o_vsz);
          unsigned char* fragVb = reinterpret_cast<unsigned char*>(xr);
          float l = 0.f;
#pragma unroll
          for (int i = 0; i < NPR; ++i) {
            const int pr = lane + 32 * i, tp = 2 * pr;
            const int s = pr >> 3, pi = pr & 7, tw = pi & 3, rg = pi >> 2;
            if (S::kDyn && tp >= T) {
              // a block that ends inside a slab: the absent tokens of that slab get probability zero in the fp16
              // fragments (the region held other operands before; their A_V rows are zero, but 0 x NaN is not)
              if (r_pad > 0 && tp < nslab * kSlab) {
                uint32_t* bp = fragPc + s * kFragStride + rg;
                bp[tw * 2] = 0u;
                bp[(4 + tw) * 2] = 0u;
              }
              break;
            }
            if (!S::kDyn && S::T < 64 && tp >= T) break;
            // where this pair's two bytes go in a row of the value B operand: chunk, register (tokens 4t.. / 16+4t..),
            // lane column, half word
            const int vboff = (((pr >> 4) * 8 + ((pr & 7) >> 1) * 2 + ((pr & 15) >> 3)) << 2) + ((pr & 1) << 1);
            __half2 z[2][NGV];
#pragma unroll
            for (int g = 0; g < NGV; ++g) { z[0][g] = vsz[tp * NGV + g]; z[1][g] = vsz[(tp + 1) * NGV + g]; }
            const float p[2] = {exp2_fast(sc[i].x - m_new), exp2_fast(sc[i].y - m_new)};
            l += p[0] + p[1];
            if (r_pad > 0) {                                // fp16 fragments of p for the low-rank value term
              uint32_t hi, lo;
              split_hi_lo(p[0], p[1], hi, lo);
              uint32_t* bp = fragPc + s * kFragStride + rg;
              bp[tw * 2] = hi;
              bp[(4 + tw) * 2] = lo;
            }
#pragma unroll
            for (int g = 0; g < NGV; ++g) {
              const uint32_t y0 = __float_as_uint(fmaf(p[0] * __low2float(z[0][g]), Sv, kMagicV));
              const uint32_t y1 = __float_as_uint(fmaf(p[1] * __low2float(z[1][g]), Sv, kMagicV));
              unsigned char* rowb = fragVb + g * 4 * RS * 4 + vboff;
              *reinterpret_cast<unsigned short*>(rowb) = (unsigned short)__byte_perm(y0, y1, 0x0040);
              *reinterpret_cast<unsigned short*>(rowb + RS * 4) = (unsigned short)__byte_perm(y0, y1, 0x0051);
              *reinterpret_cast<unsigned short*>(rowb + 2 * RS * 4) = (unsigned short)__byte_perm(y0, y1, 0x0062);
              cm[g] = fmaf(p[0], __high2float(z[0][g]), fmaf(p[1], __high2float(z[1][g]), cm[g]));
            }
            if (k2v > 0) {                                  // sparse value term of the two tokens, scattered in fixed point
#pragma unroll
              for (int e2 = 0; e2 < 2; ++e2) {
                const int tk = tp + e2;
                auto v_entry = [&](int g, float val, int idx) {
                  const float d = (val - __high2float(z[e2][g])) * Sx;
                  atomicAdd(&corr_v[g * GV + idx], __float2int_rn(p[e2] * lag * d));
                };
                if (NGV * k2v == 4) {
                  const uint2 ov = reinterpret_cast<const uint2*>(vp + o_voval)[tk];
                  const uint32_t oi = reinterpret_cast<const uint32_t*>(vp + o_voidx)[tk];
                  v_entry(0, __low2float(u32_as_h2(ov.x)), oi & 0xFFu);
                  v_entry(0, __high2float(u32_as_h2(ov.x)), (oi >> 8) & 0xFFu);
                  v_entry(NGV == 2 ? 1 : 0, __low2float(u32_as_h2(ov.y)), (oi >> 16) & 0xFFu);
                  v_entry(NGV == 2 ? 1 : 0, __high2float(u32_as_h2(ov.y)), oi >> 24);
                } else {
                  const __half* ov = reinterpret_cast<const __half*>(vp + o_voval) + (size_t)tk * NGV * k2v;
                  const unsigned char* oi = vp + o_voidx + (size_t)tk * NGV * k2v;
#pragma unroll
                  for (int g = 0; g < NGV; ++g)
#pragma unroll 1
                    for (int e = 0; e < k2v; ++e) v_entry(g, __half2float(ov[g * k2v + e]), oi[g * k2v + e]);
                }
              }
            }
          }
          l_run[0] = fmaf(l_run[0], alpha, l);
          __syncwarp();

          // ---------------- values: out += sum_tok (p * scale) * code on the integer tensor cores, low rank on the side
          {
            const bool pv0 = gid < r_pad, pv1 = gid + 8 < r_pad;
            const uint4* cwp = reinterpret_cast<const uint4*>(vp) + lane;
            const __half* avp = reinterpret_cast<const __half*>(vp + o_av) + gid * kSlab + 2 * t;
            const uint32_t* fpp = fragPc + ((gid & CMASK) * 4 + t) * 2;
            const int av_step = kSlab * r_pad;
#pragma unroll (S::unroll)
            for (int ck = 0; ck < nchunk; ++ck) {
              uint32_t bV[NGV][2];
#pragma unroll
              for (int g = 0; g < NGV; ++g) {
                const uint2 v = *reinterpret_cast<const uint2*>(xr + (g * 4 + limb_b) * RS + ck * 8 + 2 * t);
                bV[g][0] = v.x; bV[g][1] = v.y;
              }
#pragma unroll
              for (int tau = 0; tau < VT; ++tau) {
                const uint4 w = cwp[tau * 32];
#pragma unroll
                for (int j = 0; j < F; ++j) {
                  constexpr uint32_t m0 = field_mask<BITS>(0);
                  const uint32_t m = m0 << (BITS * j);
                  const int mt = F * tau + j, g = (mt * 16) / GV;
                  const uint32_t af[4] = {w.x & m, w.y & m, w.z & m, w.w & m};
                  imma16832_u(O[mt], af, bV[g][0], bV[g][1]);
                }
              }
              cwp += VT * 32;
              if (r_pad > 0) {
                // low-rank value term, first product: U = A_V^T p, slab by slab
#pragma unroll
                for (int s2 = 0; s2 < 2; ++s2) {
                  if (2 * ck + s2 < nslab) {
                    const uint2 bpv = *reinterpret_cast<const uint2*>(fpp);
                    fpp += kFragStride;
                    uint32_t aa[4] = {0u, 0u, 0u, 0u};
                    if (pv0) {
                      aa[0] = *reinterpret_cast<const uint32_t*>(avp);
                      aa[2] = *reinterpret_cast<const uint32_t*>(avp + 8);
                    }
                    if (pv1) {
                      aa[1] = *reinterpret_cast<const uint32_t*>(avp + 8 * kSlab);
                      aa[3] = *reinterpret_cast<const uint32_t*>(avp + 8 * kSlab + 8);
                    }
                    avp += av_step;
                    mma16816(U, aa, bpv.x, bpv.y);
                  }
                }
              }
            }
            if (r_pad > 0) u_pending = true;
          }

          // ---------------- sparse value term: the fixed-point sums of this block join the fp32 copy
          if (k2v > 0) {
            const float Si = 1.0f / (Sx * lag);
            int4* cv = reinterpret_cast<int4*>(corr_v) + lane;
            float4* oc = reinterpret_cast<float4*>(ocorr) + lane;
            const int4 v = *cv;
            *cv = make_int4(0, 0, 0, 0);
            float4 o = *oc;
            o.x = fmaf((float)v.x, Si, o.x);
            o.y = fmaf((float)v.y, Si, o.y);
            o.z = fmaf((float)v.z, Si, o.z);
            o.w = fmaf((float)v.w, Si, o.w);
            *oc = o;
            __syncwarp();
          }

          // ---------------- end of a segment (or of this warp's share of it): out += B_V U, into the fp32 copy
          if (with_bv && u_pending) {
            __syncwarp();
            if (t == 0) {
              wl[gid] = U[0] + U[1];
              wl[gid + 8] = U[2] + U[3];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) U[i] = 0.f;
            __syncwarp();
            uint32_t bu[2];
            {
              uint32_t hi0, lo0, hi1, lo1;
              split_hi_lo(wl[2 * t], wl[2 * t + 1], hi0, lo0);
              split_hi_lo(wl[2 * t + 8], wl[2 * t + 9], hi1, lo1);
              bu[0] = (gid & 1) ? lo0 : hi0;
              bu[1] = (gid & 1) ? lo1 : hi1;
            }
            const __half* bvf = reinterpret_cast<const __half*>(stV);      // B_V [128][r_pad]
#pragma unroll
            for (int mt = 0; mt < 8; ++mt) {
              uint32_t aa[4] = {0u, 0u, 0u, 0u};
              const __half* r0 = bvf + (16 * mt + gid) * r_pad, *r1 = bvf + (16 * mt + gid + 8) * r_pad;
              if (2 * t < r_pad) {
                aa[0] = *reinterpret_cast<const uint32_t*>(r0 + 2 * t);
                aa[1] = *reinterpret_cast<const uint32_t*>(r1 + 2 * t);
              }
              if (2 * t + 8 < r_pad) {
                aa[2] = *reinterpret_cast<const uint32_t*>(r0 + 2 * t + 8);
                aa[3] = *reinterpret_cast<const uint32_t*>(r1 + 2 * t + 8);
              }
              float d[4];
              mma16816_z(d, aa, bu[0], bu[1]);
              if (t == 0) {                              // columns 0, 1: high and low part
                float* oc = ocorr + 16 * mt + gid;
                oc[0] += d[0] + d[1];
                oc[8] += d[2] + d[3];
              }
            }
            __syncwarp();
            u_pending = false;
          }
          release();                                      // the value item is consumed
        };
        if (NGV == 2 && c_shape == 1) body(ShapeA1<BITS>{});
        else if (NGV == 2 && c_shape == 2) body(ShapeA2<BITS>{});
        else if (NGV == 1 && c_shape == 3) body(ShapeB1<BITS>{});
        else if (NGV == 1 && c_shape == 4) body(ShapeB2<BITS>{});
        else if (NGV == 1 && c_shape == 5) body(ShapeP1<BITS>{});
        else body(DynShape{});
        if (!alive) break;
      }
      if (!alive) break;
      // the integer sums and the zero-point side sums join the fp32 copy
      {
        if (tok_acc > 0) fold_O(1.f);
        __syncwarp();
        float add = 0.f;
#pragma unroll
        for (int g = 0; g < NGV; ++g) {
          float c = cm[g];
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
          if ((lane * 4) / GV == g) add = c;
        }
        float4* oc = reinterpret_cast<float4*>(ocorr) + lane;
        float4 v = *oc;
        v.x += add; v.y += add; v.z += add; v.w += add;
        *oc = v;
        __syncwarp();
      }
    }

    // ==================================================================== fp16 rows of the streaming buffer
    if (blk_hi > a.n_blocks_c && alive) {
      float Ob[8][4];
#pragma unroll
      for (int mt = 0; mt < 8; ++mt)
#pragma unroll
        for (int i = 0; i < 4; ++i) Ob[mt][i] = 0.f;
      // B operand of the scores: q * scale * log2 e per channel, split into fp16 high and low parts (columns 2h, 2h + 1)
      __syncwarp();
      {
        const int kc = lane >> 2, reg = (lane >> 1) & 1, tA = 2 * (lane & 1);
#pragma unroll
        for (int h = 0; h < HP; ++h) {
          if (h < HC) {
            const uint2 qh = *reinterpret_cast<const uint2*>(qs + h * kHeadDim + lane * 4);
            const __half2 q01 = u32_as_h2(qh.x), q23 = u32_as_h2(qh.y);
            uint32_t hiA, loA, hiB, loB;
            split_hi_lo(__low2float(q01) * a.scale_log2, __high2float(q01) * a.scale_log2, hiA, loA);
            split_hi_lo(__low2float(q23) * a.scale_log2, __high2float(q23) * a.scale_log2, hiB, loB);
            uint32_t* base = xr + kc * kFragStride + reg;
            const int cl = 2 * (h & 3);
            base[(4 * cl + tA) * 2] = hiA;
            base[(4 * (cl + 1) + tA) * 2] = loA;
            base[(4 * cl + tA + 1) * 2] = hiB;
            base[(4 * (cl + 1) + tA + 1) * 2] = loB;
          }
        }
      }
      __syncwarp();
      uint32_t bq[8][2];
#pragma unroll
      for (int kc = 0; kc < 8; ++kc) {
        const uint2 v = *reinterpret_cast<const uint2*>(xr + kc * kFragStride + ((gid & CMASK) * 4 + t) * 2);
        bq[kc][0] = v.x; bq[kc][1] = v.y;
      }
#pragma unroll 1
      for (int blk = max(blk_lo, a.n_blocks_c); blk < blk_hi; ++blk) {
        const int valid_tokens = min(kSlab, a.buf_len - (blk - a.n_blocks_c) * kSlab);
        // ---- key rows
        unsigned char* stK = acquire();
        if (!alive) break;
        {
          float acc[2][4];
#pragma unroll
          for (int hf = 0; hf < 2; ++hf)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[hf][i] = 0.f;
#pragma unroll
          for (int kc = 0; kc < 8; ++kc) {
            uint32_t af[4];
            ldmatrix_x4(af, stK + ((lane & 7) + 8 * ((lane >> 3) & 1)) * kBufPitch + (16 * kc + 8 * (lane >> 4)) * 2);
            mma16816(acc[kc & 1], af, bq[kc][0], bq[kc][1]);
          }
          if (t < HC) {
            float* pr = ps + t * maxT + gid;
            pr[0] = (acc[0][0] + acc[0][1]) + (acc[1][0] + acc[1][1]);
            pr[8] = (acc[0][2] + acc[0][3]) + (acc[1][2] + acc[1][3]);
          }
        }
        release();
        __syncwarp();
        // ---- online softmax over the slab: one rescale at most
        {
          float alpha[HP];
          bool grew = false;
#pragma unroll
          for (int h = 0; h < HP; ++h) {
            alpha[h] = 1.f;
            if (h < HC) {
              float* row = ps + h * maxT;
              const float v = lane < valid_tokens ? row[lane & 15] : -INFINITY;
              const float mx = warp_max(v);
              const float m_new = fmaxf(m_run[h], mx);       // finite: every slab holds a valid token
              if (m_new > m_run[h]) {
                alpha[h] = exp2f(m_run[h] - m_new);
                grew = true;
                m_run[h] = m_new;
              }
              const float p = lane < valid_tokens ? exp2f(v - m_new) : 0.f;   // tokens past the end of the buffer
              l_run[h] = fmaf(l_run[h], alpha[h], lane < kSlab ? p : 0.f);
              __syncwarp();
              if (lane < kSlab) row[lane] = p;
            }
          }
          if (grew) {
            float al = alpha[0];
#pragma unroll
            for (int hh = 1; hh < HP; ++hh)
              if (t == hh) al = alpha[hh];
#pragma unroll
            for (int mt = 0; mt < 8; ++mt)
#pragma unroll
              for (int i = 0; i < 4; ++i) Ob[mt][i] *= al;
            scale_ocorr(alpha);
          }
        }
        __syncwarp();
        // ---- value rows
        unsigned char* stV = acquire();
        if (!alive) break;
        if (valid_tokens < kSlab) {
          // rows past the end of the buffer hold stale bytes: clear them (0 * garbage must stay 0)
          for (int i = lane; i < (kSlab - valid_tokens) * (kBufPitch / 16); i += 32) {
            const int r = valid_tokens + i / (kBufPitch / 16), cc = i % (kBufPitch / 16);
            reinterpret_cast<uint4*>(stV + r * kBufPitch)[cc] = make_uint4(0u, 0u, 0u, 0u);
          }
          fence_async_smem();
        }
        // probabilities -> fp16 high / low fragments
        if (lane < kSlab / 2) {
          const int pr = lane, pi = pr & 7, tw = pi & 3, rg = pi >> 2;
#pragma unroll
          for (int h = 0; h < HP; ++h) {
            if (h < HC) {
              const float2 pp = *reinterpret_cast<const float2*>(ps + h * maxT + 2 * pr);
              const int col = 2 * (h & 3);
              uint32_t hi, lo;
              split_hi_lo(pp.x, pp.y, hi, lo);
              uint32_t* bp = fragPb + rg;
              bp[(col * 4 + tw) * 2] = hi;
              bp[((col + 1) * 4 + tw) * 2] = lo;
            }
          }
        }
        __syncwarp();
        {
          const uint2 bpv = *reinterpret_cast<const uint2*>(fragPb + ((gid & CMASK) * 4 + t) * 2);
#pragma unroll
          for (int mt = 0; mt < 8; ++mt) {
            uint32_t av[4];
            ldmatrix_x4_trans(av, stV + ((lane & 7) + 8 * (lane >> 4)) * kBufPitch + (16 * mt + 8 * ((lane >> 3) & 1)) * 2);
            mma16816(Ob[mt], av, bpv.x, bpv.y);
          }
        }
        release();
      }
      if (!alive) break;
      // the tensor-core part of the buffer rows joins the fp32 copy
      __syncwarp();
      if (t < HC) {
#pragma unroll
        for (int mt = 0; mt < 8; ++mt) {
          float* oc = ocorr + t * kHeadDim + 16 * mt + gid;
          oc[0] += Ob[mt][0] + Ob[mt][1];
          oc[8] += Ob[mt][2] + Ob[mt][3];
        }
      }
      __syncwarp();
    }
    if (!alive) break;

    if (JOIN) {                                // the whole range lies in one unit: joined with the other warps' below
      float l = l_run[0];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
      if (lane == 0) { ml_s[0] = m_run[0]; ml_s[1] = l; }
      break;
    }
    // ---------------- partial result of this unit: (m, l, o) per head
    int n_parts, slot;
    if (a.aligned) {
      n_parts = parts_u;
      slot = part;
    } else {
      const long long Fl = (long long)a.cc.BH * passes * NB, NW = gridDim.x;
      const long long bflat = (long long)u * NB, eflat = bflat + NB;
      const long long w_first = ((bflat + 1) * NW + Fl - 1) / Fl - 1;
      const long long w_last = (eflat * NW + Fl - 1) / Fl - 1;
      n_parts = (int)(w_last - w_first + 1);
      slot = (int)(blockIdx.x - w_first);
    }
    float* part_base = a.partial + ((size_t)u * a.max_parts + slot) * (HP * kPartRow);
    __syncwarp();
#pragma unroll
    for (int h = 0; h < HP; ++h) {
      if (h < HPu) {
        float l = l_run[h];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (lane == 0) { part_base[h * kPartRow + 128] = m_run[h]; part_base[h * kPartRow + 129] = l; }
        reinterpret_cast<float4*>(part_base + h * kPartRow)[lane] = reinterpret_cast<const float4*>(ocorr + h * kHeadDim)[lane];
      }
    }
    // The ticket is one acquire-release atomic at device scope: it publishes this warp's partial (the warp barrier
    // before it orders the other lanes' stores) and, for the warp that takes the last ticket, makes the others' visible.
    __syncwarp();
    int last = 0;
    if (lane == 0) {
      int old;
      asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(old) : "l"(a.tickets + u) : "memory");
      last = old == n_parts - 1;
    }
    last = __shfl_sync(0xffffffffu, last, 0);
    __syncwarp();
    if (last) {
      merge(u, hq0, HPu, n_parts);
      if (lane == 0) a.tickets[u] = 0;
    }
    n_left -= blk_hi - blk_lo;
    blk_lo = 0;
    ++u;
  }
  if (JOIN) {
    // Join the warps of the CTA: thread i takes channel i.  The result is the unit's output, or one partial of it for the
    // CTA that takes the last ticket.
    __syncthreads();
    const int W = blockDim.x >> 5, hq0 = unit0 * G;              // one head per pass: the unit is its query head
    const int off_ml = a.ws.misc + HP * 4;
    float* part_base = a.partial + ((size_t)unit0 * a.max_parts + blockIdx.x % a.unit_ctas) * kPartRow;
    // Every warp weighs the ranges, a lane each, instead of every thread one after the other (32 layers of one sequence 344.3 -> 343.3 us).
    const float* ml = reinterpret_cast<const float*>(smem_all + min(lane, W - 1) * a.ws.total + off_ml);
    const float mw = lane < W ? ml[0] : -INFINITY;
    const float M = warp_max(mw);
    const float wgt = mw == -INFINITY ? 0.f : exp2f(mw - M);     // no block: its output row was never set
    float den = wgt * (lane < W ? ml[1] : 0.f);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) den += __shfl_xor_sync(0xffffffffu, den, o);
    for (int ch = threadIdx.x; ch < kHeadDim; ch += blockDim.x) {
      float acc = 0.f;
#pragma unroll 4
      for (int w = 0; w < W; ++w) {
        const float wj = __shfl_sync(0xffffffffu, wgt, w);
        const float o = reinterpret_cast<const float*>(smem_all + w * a.ws.total + a.ws.ocorr)[ch];
        if (wj != 0.f) acc = fmaf(wj, o, acc);
      }
      if (a.unit_ctas == 1) {
        a.out[(size_t)hq0 * kHeadDim + ch] = acc * (1.0f / den);
      } else {
        part_base[ch] = acc;
        if (ch == 0) { part_base[128] = M; part_base[129] = den; }
      }
    }
    if (a.unit_ctas > 1) {
      __syncthreads();
      if (wrp == 0) {
        int last = 0;
        if (lane == 0) {
          int old;
          asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(old) : "l"(a.tickets + unit0) : "memory");
          last = old == a.unit_ctas - 1;
        }
        last = __shfl_sync(0xffffffffu, last, 0);
        __syncwarp();
        if (last) {
          merge(unit0, hq0, 1, a.unit_ctas);
          if (lane == 0) a.tickets[unit0] = 0;
        }
      }
    }
  }
  // a warp that gave up still has copies in flight: let them land (bounded) before leaving
  if (!alive) {
    for (int i = 0; i < n_inflight; ++i) {
      for (int k = 0; k < kDecodeSpinLimit && !mbar_try(&bar[c_stage], (uint32_t)c_par); ++k) {}
      if (++c_stage == NS) { c_stage = 0; c_par ^= 1; }
    }
  }
}

// ------------------------------------------------------------------ host side
template <class Fn>
static bool with_decode_kernel(int bits, int heads, int ngv, int wide, bool join, Fn fn) {
  const int hp = fp16_heads_per_pass(heads);
  const int minb = hp == 1 ? (wide ? 12 : 16) : 8;
#define GEAR_DEC_CASE(B, N, V, M, J) \
  if (bits == B && hp == N && ngv == V && minb == M && join == J) { fn(gear_decode_kernel<B, N, V, M, J>); return true; }
#define GEAR_DEC_HEADS(B, V) GEAR_DEC_CASE(B, 1, V, 16, false) GEAR_DEC_CASE(B, 1, V, 16, true) GEAR_DEC_CASE(B, 1, V, 12, false)
  GEAR_DEC_CASE(2, 4, 1, 8, false)   // four heads: fp16 caches only (compressed ones take gear_decode_rows_kernel)
  GEAR_DEC_HEADS(2, 1) GEAR_DEC_HEADS(2, 2) GEAR_DEC_HEADS(2, 4) GEAR_DEC_HEADS(2, 8)
  GEAR_DEC_HEADS(4, 1) GEAR_DEC_HEADS(4, 2) GEAR_DEC_HEADS(4, 4) GEAR_DEC_HEADS(4, 8)
#undef GEAR_DEC_HEADS
#undef GEAR_DEC_CASE
  return false;
}

cudaError_t launch_decode(const DecodeArgs& a, int grid, cudaStream_t st) {
  cudaError_t e = cudaSuccess;
  const size_t smem = (size_t)a.ws.total;
  const bool ok = with_decode_kernel(a.cc.bits, a.hpa, a.cc.ngv, a.wide, a.unit_ctas > 0, [&](auto kern) {
    // Programmatic dependent launch: the CTAs of this launch may become resident while the kernel before it on the
    // stream drains (the kernel below announces that at once, and waits for its predecessor before its first read of
    // global memory), so that back-to-back decode calls do not pay the launch ramp one after the other.
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)grid); cfg.blockDim = dim3(32 * a.cta_warps); cfg.dynamicSmemBytes = smem * a.cta_warps; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kern, a);
  });
  if (!ok) return cudaErrorInvalidValue;
  if (e == cudaSuccess) count_launches(1);
  return e;
}

int decode_occupancy(int bits, int heads, int ngv, int wide, size_t smem) {
  int occ = 0;
  cudaError_t e = cudaErrorInvalidValue;
  if (!wide && fp16_heads_per_pass(heads) == 1)       // the joining form may follow from the same plan
    with_decode_kernel(bits, heads, ngv, wide, true, [&](auto kern) {
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kDecodeSmemBudget);
    });
  with_decode_kernel(bits, heads, ngv, wide, false, [&](auto kern) {
    // every launch is planned first, through here: the kernel may then ask for any amount (the plans of different caches
    // differ), and the launches themselves need no attribute call
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kDecodeSmemBudget);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, 32, smem);
  });
  if (e != cudaSuccess) { cudaGetLastError(); return 0; }
  return occ;
}

}  // namespace gear
