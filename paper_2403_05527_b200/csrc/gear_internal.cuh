// Internal declarations shared by the library's translation units.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "gear_layout.cuh"

namespace gear {

// process-wide count of kernels this library launched (read through gear_kernel_launches)
void count_launches(int n);

// A launch that may start while the kernel in front of it on the stream drains (programmatic dependent launch); that kernel's results
// are there behind after_previous().
template <class... P, class... A>
inline cudaError_t launch_after(bool overlap, void (*kern)(P...), dim3 grid, int block, size_t smem, cudaStream_t st, const A&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = dim3((unsigned)block); cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = overlap ? 1 : 0;
  cfg.attrs = attr; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}
template <class... P, class... A>
inline cudaError_t launch_dependent(void (*kern)(P...), dim3 grid, int block, size_t smem, cudaStream_t st, const A&... args) {
  return launch_after(true, kern, grid, block, smem, st, args...);
}
#ifdef __CUDACC__
// Waits for the kernel in front, and only then lets the next one start: whoever starts early knows that everything two launches back
// is complete.
__device__ __forceinline__ void after_previous() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
#endif

struct CompressArgs {
  SegDesc seg;
  CacheConst cc;
  unsigned char* arena;
  const __half* K;      // [nbh][n_c][128], already offset to the first (batch, head) of the range
  const __half* V;
  float* R;             // residual workspace [nbh][2][n_c][128] or nullptr (rank 0)
  unsigned int* Rmax;   // [nbh][2] bit patterns of max |R| per tile (zeroed before the launch), with R
  int bh0;              // first (batch, head) of the range, for addressing the records
  int side0;            // first side the launch covers (blockIdx.z + side0: 0 keys, 1 values)
  int* status;          // the cache's status word
  float* Gpart;         // quant_gram_kernel: see PiArgs
  int* Gexp;
  int test_dead_wait;   // test only: quant_gram_kernel waits behind a CTA's last block for a copy that nothing requests, with a short limit
};

// Key side of a segment with per-vector grouping (gear_kcvt.cu)
struct KcvtArgs {
  SegDesc seg;
  unsigned char* arena;
  const __half* K;      // [nbh][n_c][128], already offset to the first (batch, head) of the range
  float* R;             // residual workspace [nbh][2][n_c][128] or nullptr (rank 0)
  unsigned int* Rmax;   // [nbh][2] (see CompressArgs) or nullptr
  int bh0;
  unsigned char* codes8;   // workspace: [nbh][n_c][128] one code per byte
  unsigned int* olist;     // workspace: [nbh][128][csr_k] token | fp16 value << 16, token ascending
  __half2* sz;             // workspace: [nbh][128] (scale, zero)
};
bool kcvt_fits(int n_c);
size_t kcvt_workspace_bytes(int nbh, int n_c, int csr_k);
cudaError_t launch_kcvt_keys(KcvtArgs a, int nbh, int bits, unsigned char* ws, bool overlap, cudaStream_t st);

struct PiArgs {
  SegDesc seg;
  unsigned char* arena;
  float* R;             // [ntiles][n_c][128]
  unsigned int* Rmax;   // [ntiles] bit pattern of the tile's largest |R|
  const __half* K;      // [nbh][n_c][128]: the range's rows, and the constants of its codes (residual not kept)
  const __half* V;
  CacheConst cc;
  float* Gpart;         // partials of R^T R: [CTA + tile][2][128][128] (gear_gram.cu), or, where the residual is not kept,
                        // [side][CTA + (batch, head)][128][128] (gear_quant_gram.cu)
  int* Gexp;            // and the power of two that each of these was scaled by
  float* G;             // [ntiles][128][128]: R^T R (of R scaled by the tile's power of two)
  int* status;          // the cache's status word
  float* Bcur;          // [ntiles][128][16]
  float* Bg;            // [ntiles][128][16]: (R^T R) Bcur = R^T A0
  float* Bp;            // [ntiles][parts][128][16]: R^T A0 summed from the residual (tiles with `ill` set)
  int* ill;             // [ntiles]
  float* A0;            // [ntiles][n_c][a0_pitch]
  float* Gp;            // [ntiles][nchunk][256]
  float* W;             // [ntiles][256]
  float* dbgA;          // fp32 copies for export, whole segment: [BH][2][n_c][rank] / [BH][2][128][rank]
  float* dbgB;
  int bh0, ntiles, n_c, rank, nchunk;
  int chunk_rows;       // rows per CTA of the pass, and per partial of A0^T A0
  int a0_pitch;         // 4, 8 or 16 columns, zero past the rank
};

struct CompressJob {
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
  int sms;
  int* status;
  int test_dead_wait;   // see CompressArgs
};

size_t compress_workspace_bytes(int nbh, const SegDesc& sd, const CacheConst& cc, int sms);
// R^T R of every tile, then everything of Algorithm 2 that runs on it: leaves the last loop's factor in p.Bcur
size_t pi_gram_workspace_bytes(int ntiles, int n_c, int sms);
cudaError_t launch_pi_gram(const PiArgs& p, const float* B0, unsigned long long seed, int segment, int iters, int sms,
                           bool overlap, cudaStream_t st);
// Filter, Quant, packing and R^T R of segments whose residual is not kept (gear_quant_gram.cu), A0 = R b of them (gear_pass_codes.cu)
constexpr int kRtaParts = 4;      // CTAs per tile that sum R^T A0 where it is asked for
struct QgSplit { long long blocks; int ctas; };
QgSplit qg_split(int nbh, const SegDesc& sd, int sms);
int pass_chunk_rows(int nbh, const SegDesc& sd, const CacheConst& cc, int sms);
bool qg_fits(const SegDesc& sd, const CacheConst& cc);
size_t qg_partials(int nbh, const SegDesc& sd, int sms);
cudaError_t launch_quant_gram(const CompressArgs& a, const PiArgs& p, int nbh, int sms, cudaStream_t st);
cudaError_t launch_pass_codes(const PiArgs& p, cudaStream_t st);
cudaError_t launch_pi_iterate(const PiArgs& p, const float* B0, unsigned long long seed, int segment, int iters, cudaStream_t st);
// whole-tile path for short segments (one launch): usable when compress_tile_fits()
bool compress_tile_fits(int T, int n_c, int rank);
cudaError_t compress_tile(const CompressJob& job, int BH, cudaStream_t st);
cudaError_t compress_range(const CompressJob& job, int bh0, int nbh, unsigned char* ws, cudaStream_t st);
cudaError_t launch_write_desc(SegDesc* table, int* blk2seg, int index, const SegDesc& d, cudaStream_t st);
// Rows of one decoding step into the streaming buffer and / or a query into its device copy
struct PushArgs {
  __half* buf_k;        // [BH][n_b][128]
  __half* buf_v;
  const __half* k_new;  // [BH][128], or nullptr: no rows
  const __half* v_new;
  const __half* q_src;  // q_pieces x 16 bytes
  __half* q_dst;
  int BH, n_b, slot, q_pieces;
  int host_src;         // the sources are pinned host memory, complete before the launch
};
cudaError_t launch_push(const PushArgs& a, cudaStream_t st);

// decode attention over the compressed cache
constexpr int kMaxStages = 4;
constexpr int kPartRow = 132;     // floats per head of a partial result: 128 outputs, running max, denominator, padding to 16 bytes
struct WarpSmem {      // byte offsets of a warp's (= a CTA's) shared-memory regions
  int ring, sdc, qs, xr, ps, corr_k, corr_v, ocorr, wl, misc, total;
  int fragv_stride;    // words per row of the value B-operand staging area
  int fragp;           // byte offset of the fp16 probability fragments inside the xr region
};
struct RowsSmem {      // the same of a CTA of gear_decode_rows_kernel
  int sdc, qs, qf, xk, fragv, fragp, ps, corr_k, corr_v, fold, usum, wl, scal, bars, ring, total;
};
struct DecodeArgs {
  const unsigned char* arena;
  const SegDesc* table;
  const int* blk2seg;         // [n_blocks_c] segment index of every compressed block
  const __half* buf_k;        // [BH][n_b][128]
  const __half* buf_v;
  const __half* q;            // [B][Hq][128]
  float* out;                 // [B][Hq][128]
  float* partial;             // [units][max_parts][HP][kPartRow]
  int* tickets;               // [units]
  int* status;
  CacheConst cc;
  int n_blocks_c;             // compressed blocks per (batch, head)
  int buf_len;                // tokens in the fp16 buffer
  int n_kv_heads, group_heads;   // H, G = Hq / H
  int max_parts;
  // Unit-aligned split (aligned != 0): no warp crosses from one unit into the next.  Units [0, units_a) are cut into
  // parts_a ranges, the others into parts_b = parts_a - 1; the CTAs are ordered by the length of their range,
  // longest first, in up to four classes (unit type x one-block-longer or not): class k holds the CTAs
  // [cls_start[k], cls_start[k + 1]), cls_n[k] consecutive parts from cls_p0[k] on per unit, units from cls_u0[k] on.
  // aligned == 0: the flat (unit, block) space is cut into gridDim.x equal ranges.
  int aligned, units_a, parts_a, parts_b;
  int cls_start[5], cls_u0[4], cls_n[4], cls_p0[4];
  // Short ranges of few units (unit_ctas > 0): cta_warps warps per CTA, unit_ctas CTAs per unit, joined in shared memory.
  int cta_warps, unit_ctas;
  int nstage;                 // ring stages (<= kMaxStages)
  int stage_bytes;            // bytes of one ring stage
  int bregion;                // bytes at the front of a stage reserved for one B factor
  int max_T;                  // largest block length over the segments
  int hpa;                    // query rows per pass
  int spin_limit;             // polls a consumer spends on one ring stage before it gives up
  int test_dead_wait;         // test only: wait once on a barrier that nothing completes, with a short limit
  int wide;                   // one head per pass: use the kernel built for twelve resident warps (more registers)
  int early_reads;            // the segments were last written at least two launches back on this stream (see the kernel)
  int early_buf;              // so were the buffer rows
  WarpSmem ws;
  RowsSmem rows;
  float scale_log2;           // softmax scale * log2(e)
};
cudaError_t launch_decode(const DecodeArgs& a, int grid, cudaStream_t st);
// Shared-memory plan of one warp; returns false if no stage count fits.  heads = G (query heads per kv head).
// warps_cap > 0 limits the resident warps per SM below what registers and shared memory allow.
bool decode_plan(int bits, int heads, int ngv, int max_kpart, int max_vpart, int max_bfac, int max_T, size_t smem_budget,
                 int warps_cap, DecodeArgs* a);
int decode_occupancy(int bits, int heads, int ngv, int wide, size_t smem);
int static_shape_id(const SegDesc& s, const CacheConst& c);
// passes over the cache that G query rows per kv head take, hp rows (1, 4 or 8) at a time
inline int decode_passes(int G, int hp) { return (G + hp - 1) / hp; }
// several rows per pass (gear_decode_rows.cuh): warps of a CTA, CTAs per SM that registers and shared memory are planned for
constexpr int kRowsWarps = 4;
constexpr int kRowsCtasPerSm = 4;
constexpr int kRowsBufBlock = 32;      // buffer tokens per block of work there (one row per pass: a slab)
bool rows_plan(int hp, int ngv, int max_kpart, int max_vpart, int max_bfac, int max_T, DecodeArgs* a);
int rows_occupancy(const DecodeArgs& a, int bits, int ngv);
cudaError_t launch_rows(const DecodeArgs& a, int grid, cudaStream_t st);
// the fp16-cache kernel takes one or four query heads per pass
inline int fp16_heads_per_pass(int G) { return G == 1 ? 1 : 4; }
inline int fp16_passes(int G) { return (G + fp16_heads_per_pass(G) - 1) / fp16_heads_per_pass(G); }
constexpr int kDecodeSmemBudget = 227 * 1024;    // shared memory of an SM that a launch may spread over its warps
constexpr unsigned int kWaitHintNs = 20000;       // longest suspension of one poll of a barrier
constexpr int kDecodeSpinLimit = 200000;          // polls before a wait gives up: four seconds at most

// fp16-cache attention
cudaError_t launch_fp16_attn(const void* K, const void* V, const void* q, float* out, int batch, int n_q_heads,
                             int n_kv_heads, long long n, long long n_alloc, float scale, void* scratch,
                             size_t scratch_bytes, cudaStream_t st);
size_t fp16_attn_scratch(int batch, int n_q_heads);

// canonical export
cudaError_t launch_export(const unsigned char* arena, const SegDesc& sd, const CacheConst& cc, int what, void* dst,
                          size_t n_elems, cudaStream_t st);

}  // namespace gear
