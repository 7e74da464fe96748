// Decode attention over the compressed cache for several query rows per kv head (grouped queries, several positions):
// the same streaming of records and the same arithmetic as gear_decode.cu, with a CTA of NW warps on one block.
//
// Bound: instruction issue.  What a block costs once -- the codes' unpacking, the scales, the outlier entries -- is shared by
// HP query rows and cut over the warps; what it costs per row (query-side operands, softmax) is cut over the warps by row:
//   A  key operand     rows by warp; outlier entries by thread, for all rows
//   B  key scores      16-token slabs by warp, all rows
//   C  softmax, value operand   rows by warp
//   D  values          16-channel tiles by warp, all rows; outlier entries by thread; low-rank sums by slab
// with a CTA barrier after A, B and C (D runs on into A of the next block).  One warp per CTA doing all of it for four rows
// (the kernel this one replaced) needs 248 registers and 31 KB per warp: seven warps per SM, which issue on 39 % of the
// cycles; sixteen warps here issue on 55 %.  Grouped queries over 32k tokens (four rows, 118 MB): 75 -> 63 us.
// Sixteen rows over 8k tokens (22 MB): four passes of four rows 48 us (58 in the kernel before), two of eight 54, one pass of
// sixteen rows with eight warps per CTA 72 us (spills, two CTAs per SM); eight rows pay over longer caches (rows_per_pass in
// gear_api.cu).  Rows cost about 260 instructions per warp and
// block each, half of them for the outlier entries (a product, a conversion and a shared-memory add per entry and row).
//
// Columns of the integer B operands: a pair of 8-column tiles carries four rows, limbs 0 and 1 of row 4 u + t in columns
// 2t, 2t + 1 of the first, limbs 2 and 3 in the same columns of the second, so that lane t holds everything of row t and no
// partner lane is asked.  Value operands have three limbs; for eight rows the third limbs share a tile.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "gear_decode.cuh"

namespace gear {

constexpr int kRowsBufTok = kRowsBufBlock;              // buffer tokens per item
constexpr int kRowsBufItem = kRowsBufTok * kBufPitch;
constexpr int kPFrag = 72;                              // 32-bit words per fp16 B-fragment set (eight columns, four lanes, two registers, padding)

__host__ __device__ constexpr int rows_value_tiles(int hp) { return hp / 4 + (hp / 8 > 1 ? hp / 8 : 1); }
// A block has at most min(128, group) tokens and a token 128 / group value groups, so the group fixes how long a row of
// scores can be (one slab-pair at least) and how many words a row of the value operand has.
__host__ __device__ constexpr int rows_pitch(int ngv) { return kHeadDim / ngv > kRowsBufTok ? kHeadDim / ngv : kRowsBufTok; }
__host__ __device__ constexpr int rows_fragv_words(int ngv) { return rows_pitch(ngv) / 32 * 8 + 8; }

// ------------------------------------------------------------------ the kernel
template <int BITS, int HP, int NGV>
__global__ void __launch_bounds__(kRowsWarps * 32, kRowsCtasPerSm) gear_decode_rows_kernel(const __grid_constant__ DecodeArgs a) {
  constexpr int NW = kRowsWarps, NTH = NW * 32;
  constexpr int F = 8 / BITS, kTop = BITS * (F - 1), GV = kHeadDim / NGV, KT = 4 / F, VT = 8 / F;
  constexpr int NU = HP / 4;                      // groups of four rows
  constexpr int NTV = rows_value_tiles(HP);       // 8-column tiles of the value B operand
  constexpr int HW = HP / NW;                     // rows a warp owns in A and C
  constexpr int TPW = 8 / NW;                     // channel tiles a warp owns in D
  constexpr int CW = 16 * TPW;                    // channels of a warp
  constexpr int HS = 32 / CW, NO = HP / HS;       // output accumulators: thread (channel lane % CW, rows (lane / CW) * NO ..)
  static_assert(HP % NW == 0 && 8 % NW == 0, "");
  extern __shared__ __align__(128) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gid = lane >> 2, t = lane & 3;
  const int G = a.group_heads;
  const int passes = (G + HP - 1) / HP;
  constexpr int PT = rows_pitch(NGV), RS = rows_fragv_words(NGV);
  const int NS = a.nstage;
  unsigned char* ring = smem + a.rows.ring;
  SegDesc* sdc = reinterpret_cast<SegDesc*>(smem + a.rows.sdc);
  __half* qs = reinterpret_cast<__half*>(smem + a.rows.qs);              // [HP][128] q as given
  float* qf = reinterpret_cast<float*>(smem + a.rows.qf);                // [HP][128] q * softmax scale * log2 e
  uint32_t* xk = reinterpret_cast<uint32_t*>(smem + a.rows.xk);          // [HP * 4 rows][kFragKRow] key digits
  uint32_t* fragv = reinterpret_cast<uint32_t*>(smem + a.rows.fragv);    // [NGV][NTV * 8 rows][RS] value digits
  uint32_t* fragp = reinterpret_cast<uint32_t*>(smem + a.rows.fragp);    // [slab][NU][kPFrag] fp16 probabilities
  float* ps = reinterpret_cast<float*>(smem + a.rows.ps);                // [HP][PT] scores, then probabilities
  int* corr_k = reinterpret_cast<int*>(smem + a.rows.corr_k);            // [HP][PT]
  int* corr_v = reinterpret_cast<int*>(smem + a.rows.corr_v);            // [HP][128]
  float* fold = reinterpret_cast<float*>(smem + a.rows.fold) + warp * HP * CW;   // the warp's [HP][CW]
  float* usum = reinterpret_cast<float*>(smem + a.rows.usum);            // [NW][16][HP]
  float* wl = reinterpret_cast<float*>(smem + a.rows.wl);                // [16][HP]
  float* alpha_s = reinterpret_cast<float*>(smem + a.rows.scal);         // [HP]
  float* ks_s = alpha_s + HP;                                            // [HP] integer key sums -> scores
  float* cz_s = alpha_s + 2 * HP;                                        // [HP]
  float* qn_s = alpha_s + 3 * HP;                                        // [HP]
  float* lag_s = alpha_s + 4 * HP;                                       // [HP] 2^-(bits a block's scores exceed the maximum by)
  float* side_s = alpha_s + 5 * HP;                                      // [HP][NGV]
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + a.rows.bars);       // [kMaxStages] ring, one test barrier
  int* last_s = reinterpret_cast<int*>(bar + kMaxStages + 1);

  if (tid == 0) {
    for (int s = 0; s <= kMaxStages; ++s) mbar_init(&bar[s], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = tid; i < (a.rows.ps - a.rows.xk) / 4; i += NTH) xk[i] = 0u;
  for (int i = tid; i < HP * PT; i += NTH) corr_k[i] = 0;
  for (int i = tid; i < HP * kHeadDim; i += NTH) corr_v[i] = 0;
  __syncthreads();

  // ---- this CTA's range of the flat (unit, block) space; unit = (batch, kv head, pass over the rows)
  const int nbuf_blocks = (a.buf_len + kRowsBufTok - 1) / kRowsBufTok;
  const int NB = a.n_blocks_c + nbuf_blocks;
  int n_left, u, blk_lo, part = 0, parts_u = 0;
  if (a.aligned) {
    int k = 0;
    while (k < 3 && (int)blockIdx.x >= a.cls_start[k + 1]) ++k;
    const int idx = blockIdx.x - a.cls_start[k];
    u = a.cls_u0[k] + idx / a.cls_n[k];
    part = a.cls_p0[k] + idx % a.cls_n[k];
    parts_u = u < a.units_a ? a.parts_a : a.parts_b;
    const int base = NB / parts_u, rem = NB - base * parts_u;
    blk_lo = part * base + min(part, rem);
    n_left = base + (part < rem ? 1 : 0);
  } else {
    const long long Fl = (long long)a.cc.BH * passes * NB, NWG = gridDim.x, gw = blockIdx.x;
    const long long f0 = gw * Fl / NWG, f1 = (gw + 1) * Fl / NWG;
    if (f0 >= f1) return;                         // the host launches no more CTAs than blocks
    n_left = (int)(f1 - f0);
    u = (int)(f0 / NB);
    blk_lo = (int)(f0 - (long long)u * NB);
  }
  // programmatic dependent launch: see gear_decode_kernel
  const bool early = early_start(a, NS, blk_lo, n_left);
  if (!early) asm volatile("griddepcontrol.wait;" ::: "memory");

  // ---- producer (warp 0): two items per block, issued in order into the ring
  int p_left = n_left, p_blk = blk_lo, p_share_lo = blk_lo, p_half = 0, p_stage = 0;
  int p_bh = u / passes, p_pass = u - p_bh * passes;
  int p_seg_lo = 0, p_seg_hi = 0, p_kbytes = 0, p_vbytes = 0, p_hb = 0, n_issued = 0;
  const unsigned char* p_segb = nullptr;
  const unsigned char* p_rec = nullptr;
  auto issue = [&]() {
    if (warp != 0 || p_left == 0) return;
    unsigned char* dst = ring + p_stage * a.stage_bytes;
    uint64_t* b = &bar[p_stage];
    if (p_blk < a.n_blocks_c) {
      if (p_blk >= p_seg_hi) {                    // new segment (or new unit): read its descriptor
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
    } else {
      const int j = p_blk - a.n_blocks_c;
      const int rows = min(kRowsBufTok, a.buf_len - j * kRowsBufTok);
      const __half* src = (p_half == 0 ? a.buf_k : a.buf_v) + ((size_t)p_bh * a.cc.n_b + (size_t)j * kRowsBufTok) * kHeadDim;
      if (lane == 0) mbar_expect_tx(b, rows * 256);
      __syncwarp();
      if (lane < rows) bulk_g2s(dst + lane * kBufPitch, src + lane * kHeadDim, 256, b);
    }
    ++n_issued;
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
  if (early) asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  int c_stage = 0, c_par = 0, n_used = 0, c_seg_lo = 0, c_seg_hi = 0, c_shape = 0;
  bool ok = true, alive = true;                   // ok: this thread's waits; alive: all threads', agreed at the barriers
  if (a.test_dead_wait && !mbar_wait(&bar[kMaxStages], 0u, 64, a.status)) ok = false;
  auto acquire = [&]() -> unsigned char* {        // the next item, in order; its stage
    unsigned char* st = ring + c_stage * a.stage_bytes;
    if (ok && !mbar_wait(&bar[c_stage], (uint32_t)c_par, a.spin_limit, a.status)) ok = false;
    if (++c_stage == NS) { c_stage = 0; c_par ^= 1; }
    ++n_used;
    return st;
  };
  bool v_free = false;                            // the value item of the block before is consumed: refill after the next barrier
  if (__syncthreads_or(!ok)) alive = false;

  // ---- loop over the units this CTA touches
  while (n_left > 0 && alive) {
    const int blk_hi = min(NB, blk_lo + n_left);
    const int c_hi = min(blk_hi, a.n_blocks_c);
    const int bh = u / passes, pass = u - bh * passes;
    const int HPu = min(HP, G - pass * HP);       // rows this pass holds; absent rows carry zero queries
    const int hq0 = bh * G + pass * HP;

    // ---- the rows' queries: own rows in registers (four channels per lane), all rows in shared memory
    float m_run[HW], l_run[HW];
#pragma unroll
    for (int i = 0; i < HW; ++i) {
      const int h = warp * HW + i;
      m_run[i] = -INFINITY; l_run[i] = 0.f;
      const uint2 v = h < HPu ? *reinterpret_cast<const uint2*>(a.q + (size_t)(hq0 + h) * kHeadDim + lane * 4) : make_uint2(0u, 0u);
      *reinterpret_cast<uint2*>(qs + h * kHeadDim + lane * 4) = v;
      const __half2 q01 = u32_as_h2(v.x), q23 = u32_as_h2(v.y);
      const float4 qv = make_float4(__low2float(q01) * a.scale_log2, __high2float(q01) * a.scale_log2,
                                    __low2float(q23) * a.scale_log2, __high2float(q23) * a.scale_log2);
      *reinterpret_cast<float4*>(qf + h * kHeadDim + lane * 4) = qv;
      const float mx = fmaxf(fmaxf(fabsf(qv.x), fabsf(qv.y)), fmaxf(fabsf(qv.z), fabsf(qv.w)));
      const uint32_t mb = warp_max_u32(__float_as_uint(mx));
      // 2^-(exponent of the row's largest entry): the fixed point of the sparse key term
      if (lane == 0) qn_s[h] = pow2i(-clamp60((int)(mb >> 23) - 127));
    }
    __syncthreads();
    float oc[NO];                                 // fp32 part of the output: channel warp * CW + lane % CW, rows (lane / CW) * NO + i
#pragma unroll
    for (int i = 0; i < NO; ++i) oc[i] = 0.f;
    const int oc_ch = lane % CW, oc_h0 = (lane / CW) * NO;
    // what the warp has put into its fold buffer ([row][channel]) joins the fp32 part
    auto take_fold = [&]() {
      __syncwarp();
#pragma unroll
      for (int i = 0; i < NO; ++i) oc[i] += fold[(oc_h0 + i) * CW + oc_ch];
      __syncwarp();
    };
    auto scale_oc = [&]() {
#pragma unroll
      for (int i = 0; i < NO; ++i) oc[i] *= alpha_s[oc_h0 + i];
    };
    auto any_grew = [&]() {
      bool g = false;
#pragma unroll
      for (int h = 0; h < HP; h += 4) {
        const float4 al = *reinterpret_cast<const float4*>(alpha_s + h);
        g = g || al.x != 1.f || al.y != 1.f || al.z != 1.f || al.w != 1.f;
      }
      return g;
    };

    // ==================================================================== compressed blocks
    if (blk_lo < c_hi) {
      int O[TPW][NTV][4];
      float U[NU][4], cm[HW][NGV];
      uint32_t bw[NU][2];
#pragma unroll
      for (int i = 0; i < TPW; ++i)
#pragma unroll
        for (int n = 0; n < NTV; ++n)
#pragma unroll
          for (int k = 0; k < 4; ++k) O[i][n][k] = 0;
#pragma unroll
      for (int n = 0; n < NU; ++n) {
        bw[n][0] = bw[n][1] = 0u;
#pragma unroll
        for (int k = 0; k < 4; ++k) U[n][k] = 0.f;
      }
#pragma unroll
      for (int i = 0; i < HW; ++i)
#pragma unroll
        for (int g = 0; g < NGV; ++g) cm[i][g] = 0.f;
      int eV_cur = 1000, tok_acc = 0;
      // integer sums -> the fp32 part; the integers start again from zero
      auto fold_O = [&]() {
        const float fs = pow2i(-eV_cur);
#pragma unroll
        for (int i = 0; i < TPW; ++i) {
          const int j = (TPW * warp + i) % F;
          const float rs = fs * pow2i(-BITS * j);
#pragma unroll
          for (int n = 0; n < NU; ++n) {
            const int third = NU + n / 2;                            // the tile and column of limb 2
            const int c = HP == 4 ? 0 : (n & 1);
            const float v0 = fmaf((float)O[i][third][c], 65536.f, fmaf((float)O[i][n][1], 256.f, (float)O[i][n][0])) * rs;
            const float v1 = fmaf((float)O[i][third][2 + c], 65536.f, fmaf((float)O[i][n][3], 256.f, (float)O[i][n][2])) * rs;
            fold[(4 * n + t) * CW + 16 * i + gid] = v0;
            fold[(4 * n + t) * CW + 16 * i + gid + 8] = v1;
          }
#pragma unroll
          for (int n = 0; n < NTV; ++n)
#pragma unroll
            for (int k = 0; k < 4; ++k) O[i][n][k] = 0;
        }
        take_fold();
      };
      // the fixed-point sums of a block's value outliers join the fp32 part behind a barrier that all adds precede: in B of
      // the next block (whose own adds come in D), or after the last one
      float corr_scale = 0.f;
      auto take_corr = [&]() {
        if (corr_scale == 0.f) return;
#pragma unroll
        for (int i = 0; i < NO; ++i) {
          int* cv = corr_v + (oc_h0 + i) * kHeadDim + warp * CW + oc_ch;
          oc[i] = fmaf((float)*cv, corr_scale * __uint_as_float((254u << 23) - __float_as_uint(lag_s[oc_h0 + i])), oc[i]);
          *cv = 0;
        }
        corr_scale = 0.f;
      };
      // outlier lists of per-vector key segments: entries of the next block requested ahead, two per thread
      constexpr int kAhead = NGV == 1 ? 2 : 1;
      unsigned int cs_lo = 0u, cs_hi = 0u, cs_e[kAhead];
      int cs_blk = -1;
#pragma unroll
      for (int j = 0; j < kAhead; ++j) cs_e[j] = 0u;

#pragma unroll 1
      for (int blk = blk_lo; blk < c_hi; ++blk) {
        if (blk >= c_seg_hi || blk < c_seg_lo) {  // uniform over the CTA
          const int* src = reinterpret_cast<const int*>(a.table + a.blk2seg[blk]);
          __syncthreads();
          if (tid < (int)(sizeof(SegDesc) / 4)) reinterpret_cast<int*>(sdc)[tid] = src[tid];
          __syncthreads();
          c_seg_lo = sdc->blk_start;
          c_seg_hi = c_seg_lo + sdc->nblk;
          c_shape = sdc->shape_id;
        }
        auto body = [&](auto shape_tag) {
          using S = decltype(shape_tag);
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
          const bool csr = NGV == 1 && S::kCsr && sdc->csr_base16 != 0;
          const int nslab = (T + kSlab - 1) / kSlab, nchunk = (T + 31) / 32;

          // ================================================================ A: key operand
          unsigned char* stK = acquire();
          const unsigned char* kp = stK + a.bregion;
          const float dmax_k = reinterpret_cast<const float*>(kp)[0];
          const float dmax_v = reinterpret_cast<const float*>(kp)[1];
          const float smax_v = reinterpret_cast<const float*>(kp)[3];
          // fixed-point exponent of the sparse key term for a row whose query has exponent 0
          const int ekx = clamp60(21 - float_exponent(dmax_k));
          if (with_bk && warp == NW - 1) {
            // w = q B_K through the fp16 tensor cores, [rank][row], scaled
            const __half* bk = reinterpret_cast<const __half*>(stK);     // [r_pad][128]
#pragma unroll
            for (int n = 0; n < (HP + 7) / 8; ++n) {
              float wacc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
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
                if (8 * n + gid < HP) {
                  const __half* qrow = qs + (8 * n + gid) * kHeadDim + 16 * kc + 2 * t;
                  b0 = *reinterpret_cast<const uint32_t*>(qrow);
                  b1 = *reinterpret_cast<const uint32_t*>(qrow + 8);
                }
                mma16816(wacc, af, b0, b1);
              }
              if (8 * n + 2 * t < HP) {           // D[rho][col 2t, 2t + 1]
                *reinterpret_cast<float2*>(&wl[gid * HP + 8 * n + 2 * t]) = make_float2(wacc[0] * a.scale_log2, wacc[1] * a.scale_log2);
                *reinterpret_cast<float2*>(&wl[(gid + 8) * HP + 8 * n + 2 * t]) = make_float2(wacc[2] * a.scale_log2, wacc[3] * a.scale_log2);
              }
            }
          }
          {
            // the block-wide fixed-point image of q * scale per channel, as four signed base-256 digits; sum q * zero
            const uint4 kz = reinterpret_cast<const uint4*>(kp + off_kscale)[lane];
            const uint32_t w4[4] = {kz.x, kz.y, kz.z, kz.w};
            const int sh = BITS * (F - 1 - ((lane >> 3) % F));
            const uint32_t mulc = 1u << sh, addc = 0x80808080u - (kMagicBits << sh);
            uint32_t* wcol = xk + (lane >> 3) * 8 + (lane & 3) * 2 + ((lane >> 2) & 1);
#pragma unroll
            for (int i = 0; i < HW; ++i) {
              const int h = warp * HW + i;
              const float4 q4 = *reinterpret_cast<const float4*>(qf + h * kHeadDim + lane * 4);
              const float qv[4] = {q4.x, q4.y, q4.z, q4.w};
              float qd[4], c = 0.f;
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const __half2 sz = u32_as_h2(w4[j]);
                qd[j] = qv[j] * __low2float(sz);
                c = fmaf(qv[j], __high2float(sz), c);
              }
              const float am = fmaxf(fmaxf(fabsf(qd[0]), fabsf(qd[1])), fmaxf(fabsf(qd[2]), fabsf(qd[3])));
              const uint32_t mb = warp_max_u32(__float_as_uint(am));
              const int e = clamp60(21 - ((int)(mb >> 23) - 127));        // |q * scale| * 2^e < 2^22
              const float Sk = pow2i(e);
              uint32_t z[4];
#pragma unroll
              for (int j = 0; j < 4; ++j)
                z[j] = (__float_as_uint(fmaf(qd[j], Sk, kMagic)) * mulc + addc) ^ 0x80808080u;
              const uint32_t p01l = __byte_perm(z[0], z[1], 0x5140), p23l = __byte_perm(z[2], z[3], 0x5140);
              const uint32_t p01h = __byte_perm(z[0], z[1], 0x7362), p23h = __byte_perm(z[2], z[3], 0x7362);
              uint32_t* row = wcol + ((h >> 2) * 16 + 2 * (h & 3)) * kFragKRow;      // limbs 0, 1; the second tile is 8 rows on
              row[0] = __byte_perm(p01l, p23l, 0x5410);
              row[kFragKRow] = __byte_perm(p01l, p23l, 0x7632);
              row[8 * kFragKRow] = __byte_perm(p01h, p23h, 0x5410);
              row[9 * kFragKRow] = __byte_perm(p01h, p23h, 0x7632);
              c += __shfl_xor_sync(0xffffffffu, c, 16);
              c += __shfl_xor_sync(0xffffffffu, c, 8);
              c += __shfl_xor_sync(0xffffffffu, c, 4);
              c += __shfl_xor_sync(0xffffffffu, c, 2);
              c += __shfl_xor_sync(0xffffffffu, c, 1);
              if (lane == 0) { ks_s[h] = pow2i(-e - kTop); cz_s[h] = c; }
            }
          }
          if (k2k > 0) {                          // sparse key term: entries of this thread's channel, scattered to their tokens
            constexpr int PARTS = NTH / 128;      // threads per channel
            const int ch = tid & 127;
            const float zero = __high2float(reinterpret_cast<const __half2*>(kp + off_kscale)[ch]);
            const float Sx = pow2i(ekx);
            auto k_entry = [&](__half v, int tok) {
              const float d = (__half2float(v) - zero) * Sx;
              int* dst = corr_k + tok;
#pragma unroll
              for (int h = 0; h < HP; ++h) atomicAdd(dst + h * PT, __float2int_rn(qf[h * kHeadDim + ch] * qn_s[h] * d));
            };
            if (S::kDyn) {
              const __half* ov = reinterpret_cast<const __half*>(kp + off_koval) + ch * k2k;
              const unsigned char* oi = kp + off_koidx + ch * k2k;
              for (int e = tid >> 7; e < k2k; e += PARTS) k_entry(ov[e], oi[e]);
            } else {
              // consecutive entries in one load
              constexpr int N = S::k2k / PARTS > 0 ? S::k2k / PARTS : 1;
              struct __align__(2 * N) Vals { __half v[N]; };
              struct __align__(N) Toks { unsigned char i[N]; };
              const Vals ov = reinterpret_cast<const Vals*>(kp + off_koval)[ch * PARTS + (tid >> 7)];
              const Toks oi = reinterpret_cast<const Toks*>(kp + off_koidx)[ch * PARTS + (tid >> 7)];
              float qx[HP];
#pragma unroll
              for (int h = 0; h < HP; ++h) qx[h] = qf[h * kHeadDim + ch] * (qn_s[h] * Sx);
#pragma unroll
              for (int e = 0; e < N; ++e) {
                const float d = __half2float(ov.v[e]) - zero;
                int* dst = corr_k + oi.i[e];
#pragma unroll
                for (int h = 0; h < HP; ++h) atomicAdd(dst + h * PT, __float2int_rn(qx[h] * d));
              }
            }
          }
          if (csr) {
            const unsigned char* list = a.arena + sdc->seg_base + (size_t)sdc->csr_base16 * 16 + (size_t)bh * csr_stride_bytes(sdc->nblk, sdc->csr_k);
            const unsigned int* offs = reinterpret_cast<const unsigned int*>(list);
            const unsigned int* ent = reinterpret_cast<const unsigned int*>(list + csr_offsets_bytes(sdc->nblk));
            const int bi = blk - c_seg_lo;
            const bool have = cs_blk == blk;
            if (!have) { cs_lo = offs[bi]; cs_hi = offs[bi + 1]; }
            const float Sx = pow2i(ekx);
            const __half2* szp = reinterpret_cast<const __half2*>(kp + off_kscale);
            auto apply = [&](unsigned int w) {
              const int tok = (int)(w & 0xFFu), ch = (int)((w >> 8) & 0xFFu);
              const float d = (__half2float(__ushort_as_half((unsigned short)(w >> 16))) - __high2float(szp[ch])) * Sx;
#pragma unroll
              for (int h = 0; h < HP; ++h) {
                atomicAdd(&corr_k[h * PT + tok], __float2int_rn(qf[h * kHeadDim + ch] * qn_s[h] * d));
              }
            };
#pragma unroll
            for (int j = 0; j < kAhead; ++j) {
              const unsigned int e = cs_lo + tid + NTH * j;
              if (e < cs_hi) apply(have ? cs_e[j] : ent[e]);
            }
            for (unsigned int e = cs_lo + tid + NTH * kAhead; e < cs_hi; e += NTH) apply(ent[e]);
            if (blk + 1 < min(c_hi, c_seg_hi)) {
              cs_lo = cs_hi;
              cs_hi = offs[bi + 2];
#pragma unroll
              for (int j = 0; j < kAhead; ++j) {
                const unsigned int e = cs_lo + tid + NTH * j;
                cs_e[j] = e < cs_hi ? ent[e] : 0u;
              }
              cs_blk = blk + 1;
            }
          }
          if (__syncthreads_or(!ok)) { alive = false; return; }
          if (v_free) issue();                    // every warp is past D of the block before

          // ================================================================ B: key scores, a slab per warp at a time
          if (with_bk) {                          // B operand of the low-rank key product: head and remainder of w per row
#pragma unroll
            for (int n = 0; n < NU; ++n) {
              const int h = 4 * n + (gid >> 1);
              uint32_t hi0, lo0, hi1, lo1;
              split_hi_lo(wl[(2 * t) * HP + h], wl[(2 * t + 1) * HP + h], hi0, lo0);
              split_hi_lo(wl[(2 * t + 8) * HP + h], wl[(2 * t + 9) * HP + h], hi1, lo1);
              bw[n][0] = (gid & 1) ? lo0 : hi0;
              bw[n][1] = (gid & 1) ? lo1 : hi1;
            }
          }
          {
            const bool pa0 = 2 * t < r_pad, pa1 = 2 * t + 8 < r_pad;
#pragma unroll
            for (int si = 0; si < 8 / NW; ++si) {
              const int slab = warp + NW * si;
              if (slab < nslab) {
                const uint4* cwp = reinterpret_cast<const uint4*>(kp + off_kcodes) + slab * KT * 32 + lane;
                uint32_t af[4][4];
#pragma unroll
                for (int tau = 0; tau < KT; ++tau) {
                  const uint4 w = cwp[tau * 32];
#pragma unroll
                  for (int j = 0; j < F; ++j) {
                    constexpr uint32_t m0 = field_mask<BITS>(0);
                    const uint32_t m = m0 << (BITS * j);
                    af[F * tau + j][0] = w.x & m; af[F * tau + j][1] = w.y & m;
                    af[F * tau + j][2] = w.z & m; af[F * tau + j][3] = w.w & m;
                  }
                }
                uint32_t aa[4] = {0u, 0u, 0u, 0u};
                const __half* akp = reinterpret_cast<const __half*>(kp + off_ak) + (slab * kSlab + gid) * r_pad + 2 * t;
                if (pa0) {
                  aa[0] = *reinterpret_cast<const uint32_t*>(akp);
                  aa[1] = *reinterpret_cast<const uint32_t*>(akp + 8 * r_pad);
                }
                if (pa1) {
                  aa[2] = *reinterpret_cast<const uint32_t*>(akp + 8);
                  aa[3] = *reinterpret_cast<const uint32_t*>(akp + 8 * r_pad + 8);
                }
#pragma unroll
                for (int n = 0; n < NU; ++n) {
                  int lo[4] = {0, 0, 0, 0}, hi[4] = {0, 0, 0, 0};
                  const uint32_t* row = xk + (n * 16 + gid) * kFragKRow + 2 * t;
#pragma unroll
                  for (int c = 0; c < 4; ++c) {
                    const uint2 b0 = *reinterpret_cast<const uint2*>(row + c * 8);
                    const uint2 b1 = *reinterpret_cast<const uint2*>(row + 8 * kFragKRow + c * 8);
                    imma16832(lo, af[c], b0.x, b0.y);
                    imma16832(hi, af[c], b1.x, b1.y);
                  }
                  const float s0 = ks_s[4 * n + t], s1 = s0 * 65536.f;
                  float f0 = fmaf((float)(hi[0] + hi[1] * 256), s1, (float)(lo[0] + lo[1] * 256) * s0);
                  float f1 = fmaf((float)(hi[2] + hi[3] * 256), s1, (float)(lo[2] + lo[3] * 256) * s0);
                  if (r_pad > 0) {
                    float d[4];
                    mma16816_z(d, aa, bw[n][0], bw[n][1]);
                    f0 += d[0] + d[1];
                    f1 += d[2] + d[3];
                  }
                  float* pr = ps + (4 * n + t) * PT + slab * kSlab + gid;
                  pr[0] = f0; pr[8] = f1;
                }
              }
            }
          }
          take_corr();
          __syncthreads();
          issue();                                // the key item is consumed

          // ================================================================ C: softmax and value operand of the warp's rows
          unsigned char* stV = acquire();
          const unsigned char* vp = stV + a.bregion;
          // The integer value sums carry the scale 2^eV_cur, which this block keeps when p * scale * 2^eV_cur stays below
          // 2^23 at p = 1 and is no more than three bits short of it.  What is left of those bits is room for the
          // running maximum to lag behind: a row's maximum is moved (and everything summed so far scaled) only when
          // a score exceeds it by more than that, because the integers have to be folded then (a row's maximum grows in
          // every other block of a range otherwise, and a block has several rows).
          const int need = clamp60(22 - float_exponent(smax_v));
          const bool exp_bad = eV_cur > need || eV_cur < need - 3;
          const int eV_new = exp_bad ? need - kLag : eV_cur;
          const float room = (float)(need - eV_new);                      // p <= 2^room
          {
            constexpr int NPR = S::kDyn ? 2 : (S::T > 64 ? S::T / 64 : 1);
            const float Sv = pow2i(eV_new);
            const __half2* vsz = reinterpret_cast<const __half2*>(vp + o_vsz);
            unsigned char* fragVb = reinterpret_cast<unsigned char*>(fragv);
#pragma unroll
            for (int i = 0; i < HW; ++i) {
              const int h = warp * HW + i;
              const float cz = cz_s[h];
              const float Sik = pow2i(-ekx) * __uint_as_float((254u << 23) - __float_as_uint(qn_s[h]));   // powers of two
              float2 sc[NPR];
              float mx = -INFINITY;
#pragma unroll
              for (int k = 0; k < NPR; ++k) {
                const int tp = 2 * (lane + 32 * k);
                float2 v = make_float2(-INFINITY, -INFINITY);
                if (tp < T) {
                  v = *reinterpret_cast<const float2*>(ps + h * PT + tp);
                  v.x += cz; v.y += cz;
                  if (k2k > 0 || csr) {
                    int2* cp = reinterpret_cast<int2*>(corr_k + h * PT + tp);
                    const int2 c = *cp;
                    v.x = fmaf((float)c.x, Sik, v.x);
                    v.y = fmaf((float)c.y, Sik, v.y);
                    *cp = make_int2(0, 0);
                  }
                }
                sc[k] = v;
                mx = fmaxf(mx, fmaxf(v.x, v.y));
              }
              mx = warp_max(mx);
              const bool move = mx > m_run[i] + room;
              const float m_new = move ? mx : m_run[i];
              const float alpha = move ? exp2f(m_run[i] - m_new) : 1.f;
              m_run[i] = m_new;
              // the sparse value term's fixed point is set for probabilities of one at most: the block's own maximum
              if (lane == 0) { alpha_s[h] = alpha; lag_s[h] = pow2i(-max(0, (int)ceilf(mx - m_new))); }
              if (alpha != 1.f) {
#pragma unroll
                for (int g = 0; g < NGV; ++g) cm[i][g] *= alpha;
              }
              float l = 0.f;
              // rows of the value operand: limbs 0, 1 in tile h / 4, limb 2 in the shared tile
              unsigned char* rows01 = fragVb + ((h >> 2) * 8 + 2 * (h & 3)) * RS * 4;
              unsigned char* row2 = fragVb + ((NU + (h >> 3)) * 8 + 2 * (h & 3) + (HP == 4 ? 0 : ((h >> 2) & 1))) * RS * 4;
              uint32_t* bp0 = fragp + (h >> 2) * kPFrag + 2 * (h & 3) * 8;
#pragma unroll
              for (int k = 0; k < NPR; ++k) {
                const int pr = lane + 32 * k, tp = 2 * pr;
                const int s = pr >> 3, pi = pr & 7, tw = pi & 3, rg = pi >> 2;
                if (S::kDyn && tp >= T) {
                  if (r_pad > 0 && tp < nslab * kSlab) {          // absent tokens of the last slab: probability zero
                    uint32_t* bp = bp0 + s * NU * kPFrag + tw * 2 + rg;
                    bp[0] = 0u; bp[8] = 0u;
                  }
                  break;
                }
                if (!S::kDyn && S::T < 64 && tp >= T) break;
                const int vboff = (((pr >> 4) * 8 + ((pr & 7) >> 1) * 2 + ((pr & 15) >> 3)) << 2) + ((pr & 1) << 1);
                const float p0 = exp2_fast(sc[k].x - m_new), p1 = exp2_fast(sc[k].y - m_new);
                l += p0 + p1;
                *reinterpret_cast<float2*>(ps + h * PT + tp) = make_float2(p0, p1);
                if (r_pad > 0) {
                  uint32_t hi, lo;
                  split_hi_lo(p0, p1, hi, lo);
                  uint32_t* bp = bp0 + s * NU * kPFrag + tw * 2 + rg;
                  bp[0] = hi; bp[8] = lo;
                }
#pragma unroll
                for (int g = 0; g < NGV; ++g) {
                  const __half2 z0 = vsz[tp * NGV + g], z1 = vsz[(tp + 1) * NGV + g];
                  const uint32_t y0 = __float_as_uint(fmaf(p0 * __low2float(z0), Sv, kMagicV));
                  const uint32_t y1 = __float_as_uint(fmaf(p1 * __low2float(z1), Sv, kMagicV));
                  const int go = g * NTV * 8 * RS * 4 + vboff;
                  *reinterpret_cast<unsigned short*>(rows01 + go) = (unsigned short)__byte_perm(y0, y1, 0x0040);
                  *reinterpret_cast<unsigned short*>(rows01 + RS * 4 + go) = (unsigned short)__byte_perm(y0, y1, 0x0051);
                  *reinterpret_cast<unsigned short*>(row2 + go) = (unsigned short)__byte_perm(y0, y1, 0x0062);
                  cm[i][g] = fmaf(p0, __high2float(z0), fmaf(p1, __high2float(z1), cm[i][g]));
                }
              }
              l_run[i] = fmaf(l_run[i], alpha, l);
            }
          }
          if (__syncthreads_or(!ok)) { alive = false; return; }

          // ================================================================ D: values
          const bool grew = any_grew();
          if (tok_acc > 0 && (grew || exp_bad || tok_acc + T > kTokLimit)) { fold_O(); tok_acc = 0; }
          if (grew) {
            scale_oc();
#pragma unroll
            for (int n = 0; n < NU; ++n) {
              const float al = alpha_s[4 * n + t];
#pragma unroll
              for (int k = 0; k < 4; ++k) U[n][k] *= al;
            }
          }
          eV_cur = eV_new;
          tok_acc += T;
          if (k2v > 0) {                          // sparse value term: entries by thread, scattered in fixed point
            const float Sx = pow2i(clamp60(21 - float_exponent(dmax_v)));
            const __half2* vsz = reinterpret_cast<const __half2*>(vp + o_vsz);
            if (S::kDyn || NGV * S::k2v != 4 || S::T * 4 < NTH) {
              const int per = NGV * k2v;          // entries per token
              for (int x = tid; x < T * per; x += NTH) {
                const int tk = x / per, g = (x - tk * per) / k2v;
                const float d = (__half2float(reinterpret_cast<const __half*>(vp + o_voval)[x]) - __high2float(vsz[tk * NGV + g])) * Sx;
                int* dst = corr_v + g * GV + (vp + o_voidx)[x];
#pragma unroll
                for (int h = 0; h < HP; ++h) atomicAdd(dst + h * kHeadDim, __float2int_rn(ps[h * PT + tk] * lag_s[h] * d));
              }
            } else {
              // four entries per token: 4 T / threads consecutive ones of a token each, in one load
              constexpr int N = S::T * 4 / NTH > 0 ? (S::T * 4 / NTH < 4 ? S::T * 4 / NTH : 4) : 1, PER = 4 / N;
              struct __align__(2 * N) Vals { __half v[N]; };
              struct __align__(N) Chs { unsigned char i[N]; };
              const int tk = tid / PER, e0 = (tid % PER) * N;
              const Vals ov = reinterpret_cast<const Vals*>(vp + o_voval)[tid];
              const Chs oi = reinterpret_cast<const Chs*>(vp + o_voidx)[tid];
              float px[HP];
#pragma unroll
              for (int h = 0; h < HP; ++h) px[h] = ps[h * PT + tk] * (lag_s[h] * Sx);
#pragma unroll
              for (int e = 0; e < N; ++e) {
                const int g = NGV == 2 ? (e0 + e) >> 1 : 0;
                const float d = __half2float(ov.v[e]) - __high2float(vsz[tk * NGV + g]);
                int* dst = corr_v + g * GV + oi.i[e];
#pragma unroll
                for (int h = 0; h < HP; ++h) atomicAdd(dst + h * kHeadDim, __float2int_rn(px[h] * d));
              }
            }
          }
          {
            // the warp's channel tiles: code fields j of tuple tau
            const int mt0 = TPW * warp, tau = mt0 / F;
            const uint4* cwp = reinterpret_cast<const uint4*>(vp) + tau * 32 + lane;
            constexpr uint32_t m0 = field_mask<BITS>(0);
#pragma unroll (S::kDyn ? 1 : 4)
            for (int ck = 0; ck < nchunk; ++ck) {
              const uint4 w = cwp[ck * VT * 32];
              uint2 bV[NTV];
#pragma unroll
              for (int i = 0; i < TPW; ++i) {
                const int g = ((mt0 + i) * 16) / GV;
                if (i == 0 || GV < 32) {
                  const uint32_t* row = fragv + (g * NTV * 8 + gid) * RS + ck * 8 + 2 * t;
#pragma unroll
                  for (int n = 0; n < NTV; ++n) bV[n] = *reinterpret_cast<const uint2*>(row + n * 8 * RS);
                }
                const uint32_t m = m0 << (BITS * ((mt0 + i) % F));
                const uint32_t af[4] = {w.x & m, w.y & m, w.z & m, w.w & m};
#pragma unroll
                for (int n = 0; n < NTV; ++n) imma16832_u(O[i][n], af, bV[n].x, bV[n].y);
              }
            }
            if (r_pad > 0) {                      // low-rank value term, first product: U = A_V^T p, the warp's slabs
              const bool pv0 = gid < r_pad, pv1 = gid + 8 < r_pad;
#pragma unroll
              for (int si = 0; si < 8 / NW; ++si) {
                const int slab = warp + NW * si;
                if (slab < nslab) {
                  const __half* avp = reinterpret_cast<const __half*>(vp + o_av) + (slab * r_pad + gid) * kSlab + 2 * t;
                  uint32_t aa[4] = {0u, 0u, 0u, 0u};
                  if (pv0) {
                    aa[0] = *reinterpret_cast<const uint32_t*>(avp);
                    aa[2] = *reinterpret_cast<const uint32_t*>(avp + 8);
                  }
                  if (pv1) {
                    aa[1] = *reinterpret_cast<const uint32_t*>(avp + 8 * kSlab);
                    aa[3] = *reinterpret_cast<const uint32_t*>(avp + 8 * kSlab + 8);
                  }
#pragma unroll
                  for (int n = 0; n < NU; ++n) {
                    const uint2 b = *reinterpret_cast<const uint2*>(fragp + (slab * NU + n) * kPFrag + (gid * 4 + t) * 2);
                    mma16816(U[n], aa, b.x, b.y);
                  }
                }
              }
            }
          }
          if (with_bv) {
            // end of a segment (or of this CTA's share of it): out += B_V U with U summed over the warps
#pragma unroll
            for (int n = 0; n < NU; ++n) {
              usum[(warp * kMaxRank + gid) * HP + 4 * n + t] = U[n][0] + U[n][1];
              usum[(warp * kMaxRank + gid + 8) * HP + 4 * n + t] = U[n][2] + U[n][3];
#pragma unroll
              for (int k = 0; k < 4; ++k) U[n][k] = 0.f;
            }
            __syncthreads();
            const __half* bvf = reinterpret_cast<const __half*>(stV);      // B_V [128][r_pad]
#pragma unroll
            for (int n = 0; n < NU; ++n) {
              const int h = 4 * n + (gid >> 1);
              float x0 = 0.f, x1 = 0.f, x2 = 0.f, x3 = 0.f;
#pragma unroll
              for (int w = 0; w < NW; ++w) {
                const float* us = usum + (w * kMaxRank + 2 * t) * HP + h;
                x0 += us[0]; x1 += us[HP]; x2 += us[8 * HP]; x3 += us[9 * HP];
              }
              uint32_t hi0, lo0, hi1, lo1;
              split_hi_lo(x0, x1, hi0, lo0);
              split_hi_lo(x2, x3, hi1, lo1);
              const uint32_t b0 = (gid & 1) ? lo0 : hi0, b1 = (gid & 1) ? lo1 : hi1;
#pragma unroll
              for (int i = 0; i < TPW; ++i) {
                uint32_t aa[4] = {0u, 0u, 0u, 0u};
                const __half* r0 = bvf + (16 * (TPW * warp + i) + gid) * r_pad, *r1 = r0 + 8 * r_pad;
                if (2 * t < r_pad) {
                  aa[0] = *reinterpret_cast<const uint32_t*>(r0 + 2 * t);
                  aa[1] = *reinterpret_cast<const uint32_t*>(r1 + 2 * t);
                }
                if (2 * t + 8 < r_pad) {
                  aa[2] = *reinterpret_cast<const uint32_t*>(r0 + 2 * t + 8);
                  aa[3] = *reinterpret_cast<const uint32_t*>(r1 + 2 * t + 8);
                }
                float d[4];
                mma16816_z(d, aa, b0, b1);
                fold[(4 * n + t) * CW + 16 * i + gid] = d[0] + d[1];
                fold[(4 * n + t) * CW + 16 * i + gid + 8] = d[2] + d[3];
              }
            }
            take_fold();
          }
          corr_scale = k2v > 0 ? pow2i(-clamp60(21 - float_exponent(dmax_v))) : 0.f;
          v_free = true;
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
      if (tok_acc > 0) fold_O();
      // the zero-point side sums: per row and value group, over the lanes of the owner warp
#pragma unroll
      for (int i = 0; i < HW; ++i)
#pragma unroll
        for (int g = 0; g < NGV; ++g) {
          float c = cm[i][g];
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
          if (lane == 0) side_s[(warp * HW + i) * NGV + g] = c;
        }
      __syncthreads();
      if (v_free) { issue(); v_free = false; }
      take_corr();
#pragma unroll
      for (int i = 0; i < NO; ++i) oc[i] += side_s[(oc_h0 + i) * NGV + (warp * CW + oc_ch) / GV];
    }

    // ==================================================================== fp16 rows of the streaming buffer
    if (blk_hi > a.n_blocks_c) {
      float Ob[TPW][NU][4];
#pragma unroll
      for (int i = 0; i < TPW; ++i)
#pragma unroll
        for (int n = 0; n < NU; ++n)
#pragma unroll
          for (int k = 0; k < 4; ++k) Ob[i][n][k] = 0.f;
      // B operand of the scores: q * scale * log2 e, fp16 head and remainder per row
      uint32_t* xq = xk;                          // [8 steps][NU][kPFrag]
      __syncthreads();
      {
        const int kc = lane >> 2, reg = (lane >> 1) & 1, tA = 2 * (lane & 1);
#pragma unroll
        for (int i = 0; i < HW; ++i) {
          const int h = warp * HW + i;
          const float4 qv = *reinterpret_cast<const float4*>(qf + h * kHeadDim + lane * 4);
          uint32_t hiA, loA, hiB, loB;
          split_hi_lo(qv.x, qv.y, hiA, loA);
          split_hi_lo(qv.z, qv.w, hiB, loB);
          uint32_t* base = xq + (kc * NU + (h >> 2)) * kPFrag + 2 * (h & 3) * 8 + reg;
          base[tA * 2] = hiA; base[8 + tA * 2] = loA;
          base[(tA + 1) * 2] = hiB; base[8 + (tA + 1) * 2] = loB;
        }
      }
      __syncthreads();
#pragma unroll 1
      for (int blk = max(blk_lo, a.n_blocks_c); blk < blk_hi; ++blk) {
        const int valid = min(kRowsBufTok, a.buf_len - (blk - a.n_blocks_c) * kRowsBufTok);
        const int nslab = (valid + kSlab - 1) / kSlab;
        unsigned char* stK = acquire();
        if (warp < nslab) {
          float acc[NU][4];
#pragma unroll
          for (int n = 0; n < NU; ++n)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[n][k] = 0.f;
#pragma unroll
          for (int kc = 0; kc < 8; ++kc) {
            uint32_t af[4];
            ldmatrix_x4(af, stK + (warp * kSlab + (lane & 7) + 8 * ((lane >> 3) & 1)) * kBufPitch + (16 * kc + 8 * (lane >> 4)) * 2);
#pragma unroll
            for (int n = 0; n < NU; ++n) {
              const uint2 b = *reinterpret_cast<const uint2*>(xq + (kc * NU + n) * kPFrag + (gid * 4 + t) * 2);
              mma16816(acc[n], af, b.x, b.y);
            }
          }
#pragma unroll
          for (int n = 0; n < NU; ++n) {
            float* pr = ps + (4 * n + t) * PT + warp * kSlab + gid;
            pr[0] = acc[n][0] + acc[n][1];
            pr[8] = acc[n][2] + acc[n][3];
          }
        }
        unsigned char* stV = acquire();
        if (__syncthreads_or(!ok)) { alive = false; break; }
        issue();                                  // the key item is consumed
        if (valid < nslab * kSlab) {
          // rows of the last slab past the end of the buffer hold stale bytes: clear them (0 * garbage must stay 0)
          for (int i = tid; i < (nslab * kSlab - valid) * (kBufPitch / 16); i += NTH)
            reinterpret_cast<uint4*>(stV + (valid + i / (kBufPitch / 16)) * kBufPitch)[i % (kBufPitch / 16)] = make_uint4(0u, 0u, 0u, 0u);
          fence_async_smem();
        }
#pragma unroll
        for (int i = 0; i < HW; ++i) {
          const int h = warp * HW + i;
          const int tp = 2 * lane;                // lanes 0 .. 15: a pair of tokens each
          float2 v = make_float2(-INFINITY, -INFINITY);
          if (tp < valid) v.x = ps[h * PT + tp];
          if (tp + 1 < valid) v.y = ps[h * PT + tp + 1];
          const float m_new = fmaxf(m_run[i], warp_max(fmaxf(v.x, v.y)));
          const float alpha = m_new > m_run[i] ? exp2f(m_run[i] - m_new) : 1.f;
          m_run[i] = m_new;
          if (lane == 0) alpha_s[h] = alpha;
          const float p0 = exp2f(v.x - m_new), p1 = exp2f(v.y - m_new);     // tokens past the end: zero
          l_run[i] = fmaf(l_run[i], alpha, p0 + p1);
          if (lane < 16) {
            uint32_t hi, lo;
            split_hi_lo(p0, p1, hi, lo);
            uint32_t* bp = fragp + ((lane >> 3) * NU + (h >> 2)) * kPFrag + 2 * (h & 3) * 8 + (lane & 3) * 2 + ((lane & 7) >> 2);
            bp[0] = hi; bp[8] = lo;
          }
        }
        __syncthreads();
        if (any_grew()) {
          scale_oc();
#pragma unroll
          for (int n = 0; n < NU; ++n) {
            const float al = alpha_s[4 * n + t];
#pragma unroll
            for (int i = 0; i < TPW; ++i)
#pragma unroll
              for (int k = 0; k < 4; ++k) Ob[i][n][k] *= al;
          }
        }
        for (int slab = 0; slab < nslab; ++slab) {
          uint2 b[NU];
#pragma unroll
          for (int n = 0; n < NU; ++n) b[n] = *reinterpret_cast<const uint2*>(fragp + (slab * NU + n) * kPFrag + (gid * 4 + t) * 2);
#pragma unroll
          for (int i = 0; i < TPW; ++i) {
            uint32_t av[4];
            ldmatrix_x4_trans(av, stV + (slab * kSlab + (lane & 7) + 8 * (lane >> 4)) * kBufPitch + (16 * (TPW * warp + i) + 8 * ((lane >> 3) & 1)) * 2);
#pragma unroll
            for (int n = 0; n < NU; ++n) mma16816(Ob[i][n], av, b[n].x, b[n].y);
          }
        }
        __syncthreads();
        issue();                                  // the value item is consumed
      }
      if (!alive) break;
#pragma unroll
      for (int i = 0; i < TPW; ++i)
#pragma unroll
        for (int n = 0; n < NU; ++n) {
          fold[(4 * n + t) * CW + 16 * i + gid] = Ob[i][n][0] + Ob[i][n][1];
          fold[(4 * n + t) * CW + 16 * i + gid + 8] = Ob[i][n][2] + Ob[i][n][3];
        }
      take_fold();
    }

    // ---------------- partial result of this unit: (m, l, o) per row
    int n_parts, slot;
    if (a.aligned) {
      n_parts = parts_u;
      slot = part;
    } else {
      const long long Fl = (long long)a.cc.BH * passes * NB, NWG = gridDim.x;
      const long long bflat = (long long)u * NB, eflat = bflat + NB;
      const long long w_first = ((bflat + 1) * NWG + Fl - 1) / Fl - 1;
      const long long w_last = (eflat * NWG + Fl - 1) / Fl - 1;
      n_parts = (int)(w_last - w_first + 1);
      slot = (int)(blockIdx.x - w_first);
    }
    float* part_base = a.partial + ((size_t)u * a.max_parts + slot) * (HP * kPartRow);
#pragma unroll
    for (int i = 0; i < NO; ++i)
      if (oc_h0 + i < HPu) part_base[(oc_h0 + i) * kPartRow + warp * CW + oc_ch] = oc[i];
#pragma unroll
    for (int i = 0; i < HW; ++i) {
      const int h = warp * HW + i;
      float l = l_run[i];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
      if (lane == 0 && h < HPu) { part_base[h * kPartRow + 128] = m_run[i]; part_base[h * kPartRow + 129] = l; }
    }
    // the ticket: one acquire-release atomic at device scope behind a CTA barrier (see gear_decode_kernel)
    __syncthreads();
    if (tid == 0) {
      int old;
      asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(old) : "l"(a.tickets + u) : "memory");
      *last_s = old == n_parts - 1;
    }
    __syncthreads();
    if (*last_s) {
      const float* pb = a.partial + (size_t)u * a.max_parts * (HP * kPartRow);
      const size_t pstride = (size_t)HP * kPartRow;
      for (int h = warp; h < HPu; h += NW) {
        float M = -INFINITY, den = 0.f, n0 = 0.f, n1 = 0.f, n2 = 0.f, n3 = 0.f;
        for (int base = 0; base < n_parts; base += 16) {         // every load of a chunk before anything is used
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
        *reinterpret_cast<float4*>(a.out + (size_t)(hq0 + h) * kHeadDim + lane * 4) =
            make_float4(n0 * inv, n1 * inv, n2 * inv, n3 * inv);
      }
      if (tid == 0) a.tickets[u] = 0;
    }
    n_left -= blk_hi - blk_lo;
    blk_lo = 0;
    ++u;
  }
  // gave up: the copies in flight land (bounded) before the CTA leaves
  if (!alive && warp == 0) {
    for (; n_used < n_issued; ++n_used) {
      for (int k = 0; k < kDecodeSpinLimit && !mbar_try(&bar[c_stage], (uint32_t)c_par); ++k) {}
      if (++c_stage == NS) { c_stage = 0; c_par ^= 1; }
    }
  }
}

}  // namespace gear
