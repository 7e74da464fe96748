// A0 = R b (Algorithm 2, the last product) of segments whose residual is not kept (gear_quant_gram.cu): R = X - D^ - S is computed again
// from X and the stored codes, with the operations that gave it there, so that it has the same bits.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "gear_internal.cuh"
#include "gear_pass.cuh"
#include "gear_pi.cuh"
#include "gear_quant.cuh"
#include "gear_tma.cuh"

namespace gear {

constexpr int kCpRows = 64;                        // tokens that a CTA works on at a time, 16 per warp
static_assert(kCpRows == kBoxRows, "a stage is a box per 64 channels");

// What a stage of the ring holds behind the two boxes of X: the pieces of the block's record that these 64 tokens need.
struct CpStage { int scales, scale_bytes, codes, code_bytes, idx, idx_bytes, total; };
__host__ __device__ inline CpStage cp_stage(const SegDesc& sd, const CacheConst& cc, int side) {
  CpStage s;
  s.scales = 2 * kBoxBytes;
  if (side == 0) {                                 // (scale, zero), outlier values and indices of all channels: one piece
    s.scale_bytes = sd.off_kcodes - sd.off_kscale;
    s.idx = s.scales + sd.off_koidx - sd.off_kscale; s.idx_bytes = 0;
    s.codes = s.scales + s.scale_bytes;
  } else {
    s.scale_bytes = kCpRows * cc.ngv * 4;
    s.idx = s.scales + s.scale_bytes; s.idx_bytes = kCpRows * cc.ngv * 2 * cc.k_v;
    s.codes = s.idx + s.idx_bytes;
  }
  s.code_bytes = kCpRows / kSlab * sd.slab_codes;
  s.total = (s.codes + s.code_bytes + 1023) / 1024 * 1024;
  return s;
}
constexpr int kCpStages = 2;

// the codes in byte `sel & 3` and the next one of a word as a pair of floats
__device__ __forceinline__ F32x2 code_pair(unsigned int w, unsigned int sel0, unsigned int sel1) {
  return add2(pack2(__uint_as_float(__byte_perm(w, 0x4B000000u, sel0)), __uint_as_float(__byte_perm(w, 0x4B000000u, sel1))),
              pack2(-8388608.0f, -8388608.0f));
}
// c - h in one instruction
__device__ __forceinline__ float minus(__half h, float c) {
  float r;
  asm("fma.rn.f32.f16 %0, %1, %2, %3;" : "=f"(r) : "h"(__half_as_ushort(h)), "h"((unsigned short)0xBC00), "f"(c));
  return r;
}
// two residuals scaled by a power of two: x sr - (code d + m) sr, as fp16 heads and remainders
__device__ __forceinline__ void residual_pair(uint32_t x, F32x2 c, F32x2 neg_d, F32x2 neg_m, F32x2 sr, uint32_t& hi, uint32_t& lo) {
  const float2 xf = __half22float2(*reinterpret_cast<const __half2*>(&x));
  const float2 s = unpack2(fma2(pack2(xf.x, xf.y), sr, fma2(c, neg_d, neg_m)));
  const __half2 h = __floats2half2_rn(s.x, s.y);
  const __half2 l = __floats2half2_rn(minus(__low2half(h), s.x), minus(__high2half(h), s.y));
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}
__device__ __forceinline__ uint32_t transpose8(uint32_t v) {
  uint32_t r;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(v));
  return r;
}

// Bound: instruction issue (about eight instructions per entry), with the 2 bytes of X and the codes behind it.  64 tokens at a
// time come through a ring in shared memory; where an outlier was filtered, X is overwritten by the group's zero point there, which
// makes the residual zero (its code is zero).  The lanes of a warp take the codes as the decode kernel's fragments have them.
//   keys    a word is four channels of one token: the lane's fragment of R has rows gid, gid + 8 and, for a step of 16 channels,
//           channels 4t .. 4t + 3 as k indices 2t, 2t + 1, 2t + 8, 2t + 9 (a contraction does not care about their order)
//   values  a word is four tokens 4t .. 4t + 3 of channel gid: X comes transposed (ldmatrix), the residuals of two tokens
//           are transposed back as heads and remainders (movmatrix).  Which two of the four go first differs between the lanes, so
//           that the eight rows of an ldmatrix hit different banks.
// 2 bits, rank 4, 8 x 32 heads x 4096: keys 78, values 82 us (both from the fp32 residual 169 us); 131 and 138 with a bulk copy per
// row into padded rows instead of boxes with swizzle: one warp issued 64 copies while the others waited for it.
template <int BITS, int SIDE, int NGV, int NT>
__global__ void __launch_bounds__(kPassWarps * 32, NT == 4 ? 3 : 4) pi_codes_pass_kernel(PiArgs p, const __grid_constant__ CUtensorMap rows) {
  constexpr int F = 8 / BITS, RP = 4 * NT;
  __shared__ typename PassFactor<NT>::Shared sh;
  __shared__ uint64_t full[kCpStages];
  __shared__ __align__(16) float neg_d[kHeadDim], neg_m[kHeadDim];   // keys: -scale, -zero of the channels, scaled as X is
  extern __shared__ unsigned char smem_raw[];
  unsigned char* ring = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
  const SegDesc& sd = p.seg;
  const int bhl = blockIdx.y, tile = 2 * bhl + SIDE, chunk = blockIdx.x;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gid = lane >> 2, t = lane & 3;
  const int row0 = chunk * p.chunk_rows, items = min(p.chunk_rows, p.n_c - row0) / kCpRows;
  const CpStage cs = cp_stage(sd, p.cc, SIDE);
  float* A0 = p.A0 + (size_t)tile * p.n_c * RP;
  const unsigned char* recs = p.arena + sd.seg_base + (size_t)(p.bh0 + bhl) * sd.bh_stride + sd.bfac_bytes;

  if (tid == 0) {
    for (uint64_t& b : full) bar_init(&b);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  auto request = [&](int item) {                   // by thread 0
    unsigned char* st = ring + item % kCpStages * cs.total;
    uint64_t* b = &full[item % kCpStages];
    const int row = row0 + item * kCpRows, blk = row / sd.T, part = (row - blk * sd.T) / kCpRows;
    const unsigned char* rec = recs + (size_t)blk * sd.rec_bytes;
    bar_expect(b, 2 * kBoxBytes + cs.scale_bytes + cs.code_bytes + cs.idx_bytes);
    load_box(st, &rows, 0, bhl * p.n_c + row, b);
    load_box(st + kBoxBytes, &rows, kBoxChannels, bhl * p.n_c + row, b);
    bulk_copy(st + cs.scales, rec + (SIDE == 0 ? sd.off_kscale : sd.off_vscale + part * cs.scale_bytes), cs.scale_bytes, b);
    bulk_copy(st + cs.codes, rec + (SIDE == 0 ? sd.off_kcodes : sd.off_vcodes) + part * cs.code_bytes, cs.code_bytes, b);
    if (SIDE == 1 && cs.idx_bytes > 0) bulk_copy(st + cs.idx, rec + sd.off_voidx + part * cs.idx_bytes, cs.idx_bytes, b);
  };
  if (tid == 0)
    for (int i = 0; i < kCpStages && i < items; ++i) request(i);    // complete two launches back: X, and the codes
  // as in quant_gram_kernel, the values wait for the keys' pass at their end only; what both read was there when the keys' started
  if (SIDE == 0) after_previous();
  else asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  const int er = pow2_exponent(__uint_as_float(p.Rmax[tile]));
  const float sr = exp2_int(-er);
  const F32x2 sr2 = pack2(sr, sr);
  PassFactor<NT> factor;
  factor.load(p, tile, er, sh);
  // B fragments of a = R b: column n = gid of tile nt is (rho = 4 nt + gid / 2, head | remainder), k as described above
  uint32_t bf[8][NT][2];
#pragma unroll
  for (int c = 0; c < 8; ++c)
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      if (SIDE == 0) {
        const uint2 v = *reinterpret_cast<const uint2*>(&sh.bsplit[8 * nt + gid][16 * c + 4 * t]);
        bf[c][nt][0] = v.x; bf[c][nt][1] = v.y;
      } else {
        bf[c][nt][0] = *reinterpret_cast<const uint32_t*>(&sh.bsplit[8 * nt + gid][16 * c + 2 * t]);
        bf[c][nt][1] = *reinterpret_cast<const uint32_t*>(&sh.bsplit[8 * nt + gid][16 * c + 2 * t + 8]);
      }
    }
  const int first = SIDE == 0 ? 0 : 2 * (t >> 1);  // values: of the tokens 4t .. 4t + 3, the pair that goes first
  bool ok = true;
  for (int item = 0; item < items; ++item) {
    unsigned char* st = ring + item % kCpStages * cs.total;
    ok = bar_wait(&full[item % kCpStages], (uint32_t)(item / kCpStages) & 1u);
    if (ok) {
      const __half2* sz = reinterpret_cast<const __half2*>(st + cs.scales);
      if (SIDE == 0) {
        const __half2 v = sz[tid];
        neg_d[tid] = -__low2float(v) * sr;
        neg_m[tid] = -__high2float(v) * sr;
        const int row = row0 + item * kCpRows, part = row % sd.T / kCpRows;
        for (int e = 0; e < 2 * sd.k_k; ++e) {
          const int tk = st[cs.idx + tid * 2 * sd.k_k + e];
          if (tk / kCpRows == part) *reinterpret_cast<__half*>(st + tid / kBoxChannels * kBoxBytes + box_at(tk % kCpRows, tid % kBoxChannels)) = __high2half(v);
        }
      } else if (tid < kCpRows * NGV) {
        const __half zero = __high2half(sz[tid]);
        for (int e = 0; e < 2 * p.cc.k_v; ++e) {
          const int ch = (tid % NGV) * (kHeadDim / NGV) + st[cs.idx + tid * 2 * p.cc.k_v + e];
          *reinterpret_cast<__half*>(st + ch / kBoxChannels * kBoxBytes + box_at(tid / NGV, ch % kBoxChannels)) = zero;
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (__syncthreads_or(!ok)) {                   // gave up: report, let the copies of both stages land (bounded)
      if (tid == 0) atomicExch(p.status, -7 /* GEAR_ERR_TIMEOUT */);
      for (int i = item; i < items && i < item + kCpStages; ++i) bar_wait(&full[i % kCpStages], (uint32_t)(i / kCpStages) & 1u);
      break;
    }
    float d[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) d[nt][0] = d[nt][1] = d[nt][2] = d[nt][3] = 0.f;
    auto product = [&](int c, const uint32_t (&fh)[4], const uint32_t (&fl)[4]) {
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        mma16816_f16(d[nt], fh, bf[c][nt][0], bf[c][nt][1]);
        mma16816_f16(d[nt], fl, bf[c][nt][0], bf[c][nt][1]);
      }
    };
    constexpr unsigned int mask = field_of_bytes<BITS>();
    int ra = row0 + item * kCpRows + warp * kSlab, rc;
    if (SIDE == 0) {
      const unsigned char* xa = st + (warp * kSlab + gid) * 128 + 8 * (t & 1);     // piece 2 c + t / 2 of row gid, box c / 4
      const int swz = ((t >> 1) ^ gid) << 4;
      const uint4* cw = reinterpret_cast<const uint4*>(st + cs.codes) + warp * (256 * BITS / 16) + lane;
      uint4 w = make_uint4(0u, 0u, 0u, 0u);        // the codes of 2 F steps
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        if (c % (2 * F) == 0) w = cw[c / (2 * F) * 32];
        const unsigned int wa = (((c & 1) ? w.z : w.x) >> (BITS * (c / 2 % F))) & mask, wc = (((c & 1) ? w.w : w.y) >> (BITS * (c / 2 % F))) & mask;
        const unsigned char* xc = xa + c / 4 * kBoxBytes + (swz ^ (c % 4 << 5));
        const uint2 va = *reinterpret_cast<const uint2*>(xc), vc = *reinterpret_cast<const uint2*>(xc + 8 * 128);
        const float4 nd = *reinterpret_cast<const float4*>(&neg_d[16 * c + 4 * t]), nm = *reinterpret_cast<const float4*>(&neg_m[16 * c + 4 * t]);
        const F32x2 d0 = pack2(nd.x, nd.y), d1 = pack2(nd.z, nd.w), m0 = pack2(nm.x, nm.y), m1 = pack2(nm.z, nm.w);
        uint32_t fh[4], fl[4];
        residual_pair(va.x, code_pair(wa, 0x7440u, 0x7441u), d0, m0, sr2, fh[0], fl[0]);
        residual_pair(vc.x, code_pair(wc, 0x7440u, 0x7441u), d0, m0, sr2, fh[1], fl[1]);
        residual_pair(va.y, code_pair(wa, 0x7442u, 0x7443u), d1, m1, sr2, fh[2], fl[2]);
        residual_pair(vc.y, code_pair(wc, 0x7442u, 0x7443u), d1, m1, sr2, fh[3], fl[3]);
        product(c, fh, fl);
      }
      rc = ra + gid + 8;
      ra += gid;
    } else {
      F32x2 vd[2][NGV], vm[2][NGV];                // pair, value group
      const __half2* sz = reinterpret_cast<const __half2*>(st + cs.scales) + (warp * kSlab + 4 * t) * NGV;
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int g = 0; g < NGV; ++g) {
          const int o = first ^ (2 * q);
          const float2 a = __half22float2(sz[o * NGV + g]), b = __half22float2(sz[(o + 1) * NGV + g]);
          vd[q][g] = pack2(-a.x * sr, -b.x * sr);
          vm[q][g] = pack2(-a.y * sr, -b.y * sr);
        }
      const unsigned int s0 = 0x7440u + first, s1 = s0 + 1, s2 = 0x7440u + (first ^ 2), s3 = s2 + 1;
      const int mi = lane >> 3, kp = lane & 7;
      const int xrow = 4 * (kp >> 1) + (kp & 1) + 2 * ((mi & 1) ^ (kp >> 2));      // piece 2 c + mi / 2 of this row, box c / 4
      const uint32_t xaddr = smem_addr(st) + (warp * kSlab + xrow) * 128, swz = ((mi >> 1) ^ (xrow & 7)) << 4;
      const unsigned char* cw = st + cs.codes + (warp >> 1) * (512 * BITS) + lane * 16 + 8 * (warp & 1);
      uint2 w = make_uint2(0u, 0u);                // the codes of F steps
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        if (c % F == 0) w = *reinterpret_cast<const uint2*>(cw + c / F * 512);
        const unsigned int w0 = (w.x >> (BITS * (c % F))) & mask, w1 = (w.y >> (BITS * (c % F))) & mask;
        const int g = c * 16 / (kHeadDim / NGV);
        uint32_t x[4], fh[4], fl[4];
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]) : "r"(xaddr + c / 4 * kBoxBytes + (swz ^ (c % 4 << 5))) : "memory");
        residual_pair(x[0], code_pair(w0, s0, s1), vd[0][g], vm[0][g], sr2, fh[0], fl[0]);
        residual_pair(x[1], code_pair(w0, s2, s3), vd[1][g], vm[1][g], sr2, fh[1], fl[1]);
        residual_pair(x[2], code_pair(w1, s0, s1), vd[0][g], vm[0][g], sr2, fh[2], fl[2]);
        residual_pair(x[3], code_pair(w1, s2, s3), vd[1][g], vm[1][g], sr2, fh[3], fl[3]);
#pragma unroll
        for (int i = 0; i < 4; ++i) { fh[i] = transpose8(fh[i]); fl[i] = transpose8(fl[i]); }
        product(c, fh, fl);
      }
      const int at = ra + 4 * (gid >> 1) + (gid & 1);
      rc = at + 2 * ((gid >> 2) ^ 1);
      ra = at + 2 * (gid >> 2);
    }
    factor.store(d, A0, ra, rc, true, true);
    __syncthreads();                               // behind stores that need every load from the stage
    if (tid == 0 && item + kCpStages < items) request(item + kCpStages);
    factor.add_gram();
  }
  __syncthreads();
  factor.leave_gram(p, tile, chunk, sh);
  if (SIDE == 1) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// R^T A0 from the residual itself for tiles with `ill` set (see pi_rta_kernel): one channel per thread, kRtaParts CTAs per tile.
__global__ void __launch_bounds__(kHeadDim) pi_codes_rta_kernel(PiArgs p) {
  constexpr int kRows = 32;
  __shared__ float a[kRows * kMaxRank];
  const int tile = blockIdx.y, part = blockIdx.x, j = threadIdx.x, bhl = tile >> 1, side = tile & 1;
  after_previous();
  if (!p.ill[tile]) return;
  const SegDesc& sd = p.seg;
  const int RP = p.a0_pitch, bits = p.cc.bits, gv = p.cc.g_v, ngv = p.cc.ngv;
  const int row0 = (int)((long long)part * p.n_c / kRtaParts), row1 = (int)((long long)(part + 1) * p.n_c / kRtaParts);
  const __half* X = (side == 0 ? p.K : p.V) + (size_t)bhl * p.n_c * kHeadDim + j;
  const float* A0 = p.A0 + (size_t)tile * p.n_c * RP;
  const unsigned char* recs = p.arena + sd.seg_base + (size_t)(p.bh0 + bhl) * sd.bh_stride + sd.bfac_bytes;
  auto residual = [&](int row) {
    const int blk = row / sd.T, tk = row - blk * sd.T;
    const unsigned char* rec = recs + (size_t)blk * sd.rec_bytes;
    const int grp = side == 0 ? j : tk * ngv + j / gv, e = side == 0 ? tk : j % gv, k2 = 2 * (side == 0 ? sd.k_k : p.cc.k_v);
    const unsigned char* idx = rec + (side == 0 ? sd.off_koidx : sd.off_voidx) + grp * k2;
    for (int i = 0; i < k2; ++i)
      if (idx[i] == e) return 0.f;
    int word, shift;
    const unsigned int* codes;
    if (side == 0) {
      code_slot_k(bits, tk % kSlab, j, word, shift);
      codes = reinterpret_cast<const unsigned int*>(rec + sd.off_kcodes + tk / kSlab * sd.slab_codes);
    } else {
      code_slot_v(bits, tk % 32, j, word, shift);
      codes = reinterpret_cast<const unsigned int*>(rec + sd.off_vcodes + tk / 32 * 2 * sd.slab_codes);
    }
    const float code = (float)((codes[word] >> shift) & ((1u << bits) - 1u));
    const float2 sz = __half22float2(reinterpret_cast<const __half2*>(rec + (side == 0 ? sd.off_kscale : sd.off_vscale))[grp]);
    return __half2float(X[(size_t)row * kHeadDim]) - fmaf(code, sz.x, sz.y);
  };
  float b[kMaxRank];
#pragma unroll
  for (int q = 0; q < kMaxRank; ++q) b[q] = 0.f;
  for (int r0 = row0; r0 < row1; r0 += kRows) {
    const int rows = min(kRows, row1 - r0);
    __syncthreads();
    for (int i = j; i < rows * RP; i += kHeadDim) a[(i / RP) * kMaxRank + i % RP] = A0[(size_t)r0 * RP + i];
    __syncthreads();
    for (int i = 0; i < rows; ++i) {
      const float x = residual(r0 + i);
#pragma unroll
      for (int q = 0; q < kMaxRank; ++q)
        if (q < RP) b[q] = fmaf(x, a[i * kMaxRank + q], b[q]);
    }
  }
  float* out = p.Bp + (((size_t)tile * kRtaParts + part) * kHeadDim + j) * kMaxRank;
#pragma unroll
  for (int q = 0; q < kMaxRank; ++q) out[q] = q < RP ? b[q] : 0.f;
}

// Rows per CTA of the pass: fewer where that fills the SMs sooner (the residual kept: always the most).
int pass_chunk_rows(int nbh, const SegDesc& sd, const CacheConst& cc, int sms) {
  int rows = kChunkRows;
  if (qg_fits(sd, cc))
    while (rows > 128 && (long long)nbh * ((sd.n_c + rows - 1) / rows) < 2LL * sms) rows /= 2;
  return rows;
}

template <int BITS, int SIDE, int NGV, int NT>
static cudaError_t launch_one(const PiArgs& p, cudaStream_t st) {
  const int smem = 1024 + kCpStages * cp_stage(p.seg, p.cc, SIDE).total;
  CUtensorMap rows;
  cudaError_t e = make_row_map(&rows, SIDE == 0 ? p.K : p.V, (long long)p.ntiles / 2 * p.n_c);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(pi_codes_pass_kernel<BITS, SIDE, NGV, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  return e == cudaSuccess ? launch_dependent(pi_codes_pass_kernel<BITS, SIDE, NGV, NT>, dim3(p.nchunk, p.ntiles / 2), kPassWarps * 32, smem, st, p, rows) : e;
}
template <int BITS, int NT>
static cudaError_t launch_both(const PiArgs& p, cudaStream_t st) {
  const cudaError_t e = launch_one<BITS, 0, 1, NT>(p, st);
  if (e != cudaSuccess) return e;
  return p.cc.ngv == 2 ? launch_one<BITS, 1, 2, NT>(p, st) : launch_one<BITS, 1, 1, NT>(p, st);
}
cudaError_t launch_pass_codes(const PiArgs& p, cudaStream_t st) {
  cudaError_t e;
  if (p.cc.bits == 2) e = p.rank <= 4 ? launch_both<2, 1>(p, st) : p.rank <= 8 ? launch_both<2, 2>(p, st) : launch_both<2, 4>(p, st);
  else e = p.rank <= 4 ? launch_both<4, 1>(p, st) : p.rank <= 8 ? launch_both<4, 2>(p, st) : launch_both<4, 4>(p, st);
  if (e != cudaSuccess) return e;
  e = launch_dependent(pi_codes_rta_kernel, dim3(kRtaParts, p.ntiles), kHeadDim, 0, st, p);
  if (e != cudaSuccess) return e;
  count_launches(3);
  return cudaSuccess;
}

}  // namespace gear
