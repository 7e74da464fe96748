// Shared-memory plan and launch of gear_decode_rows_kernel.
#include <string.h>

#include "gear_decode_rows.cuh"

namespace gear {

// ------------------------------------------------------------------ shared memory plan (per CTA)
bool rows_plan(int hp, int ngv, int max_kpart, int max_vpart, int max_bfac, int max_T, DecodeArgs* a) {
  const int nw = kRowsWarps;
  const int bregion = round_up(max_bfac / 2, 16);
  int stage = bregion + (max_kpart > max_vpart ? max_kpart : max_vpart);
  if (stage < kRowsBufItem) stage = kRowsBufItem;
  stage = round_up(stage, 16);
  if (max_T > rows_pitch(ngv)) return false;
  max_T = rows_pitch(ngv);
  const int nslab = max_T / kSlab;
  RowsSmem w;
  int o = 0;
  w.sdc = o;     o += 128;
  w.qs = o;      o += hp * kHeadDim * 2;
  w.qf = o;      o += hp * kHeadDim * 4;
  w.xk = o;      o += hp * 4 * kFragKRow * 4;           // also the fp16 query fragments of the buffer part
  w.fragv = o;   o += ngv * rows_value_tiles(hp) * 8 * rows_fragv_words(ngv) * 4;
  w.fragp = o;   o += nslab * (hp / 4) * kPFrag * 4;
  w.ps = o;      o += hp * max_T * 4;
  w.corr_k = o;  o += hp * max_T * 4;
  w.corr_v = o;  o += hp * kHeadDim * 4;
  w.fold = o;    o += hp * kHeadDim * 4;
  w.usum = o;    o += nw * kMaxRank * hp * 4;
  w.wl = o;      o += kMaxRank * hp * 4;
  w.scal = o;    o += 5 * hp * 4 + hp * ngv * 4;        // alpha, key scales, zero-point constants, query powers of two, lags; side sums
  w.bars = round_up(o, 8); o = w.bars + (kMaxStages + 1) * 8 + 16;
  w.ring = round_up(o, 128);
  for (int ctas = kRowsCtasPerSm; ctas >= 1; --ctas) {
    const long long per = (long long)kDecodeSmemBudget / ctas - 1024;
    long long ns = (per - w.ring) / stage;
    if (ns < 2) continue;
    if (ns > kMaxStages) ns = kMaxStages;
    w.total = w.ring + (int)ns * stage;
    a->aligned = 0;
    a->nstage = (int)ns; a->stage_bytes = stage; a->bregion = bregion; a->max_T = max_T; a->hpa = hp; a->rows = w;
    a->spin_limit = kDecodeSpinLimit; a->test_dead_wait = 0; a->early_reads = 0; a->early_buf = 0; a->wide = 0;
    return true;
  }
  return false;
}

// the kernel for (bits, rows per pass, value groups per token), instantiated in gear_decode_rows_b2.cu / _b4.cu
const void* rows_kernel_b2(int hp, int ngv);
const void* rows_kernel_b4(int hp, int ngv);
static const void* rows_kernel(int bits, int hp, int ngv) { return bits == 2 ? rows_kernel_b2(hp, ngv) : rows_kernel_b4(hp, ngv); }

int rows_occupancy(const DecodeArgs& a, int bits, int ngv) {
  const void* fn = rows_kernel(bits, a.hpa, ngv);
  int occ = 0;
  if (!fn || cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kDecodeSmemBudget) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, kRowsWarps * 32, (size_t)a.rows.total) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return occ;
}

cudaError_t launch_rows(const DecodeArgs& a, int grid, cudaStream_t st) {
  const void* fn = rows_kernel(a.cc.bits, a.hpa, a.cc.ngv);
  if (!fn) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3((unsigned)grid); cfg.blockDim = dim3(kRowsWarps * 32); cfg.dynamicSmemBytes = (size_t)a.rows.total;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;       // see launch_decode
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  void* args[1] = {const_cast<DecodeArgs*>(&a)};
  const cudaError_t e = cudaLaunchKernelExC(&cfg, fn, args);
  if (e == cudaSuccess) count_launches(1);
  return e;
}

}  // namespace gear
