// 2-bit instantiations of gear_decode_rows_kernel.
#include "gear_decode_rows.cuh"

namespace gear {

const void* rows_kernel_b2(int hp, int ngv) {
#define GEAR_ROWS(N, V) \
  if (hp == N && ngv == V) return reinterpret_cast<const void*>(&gear_decode_rows_kernel<2, N, V>);
#define GEAR_ROWS_V(V) GEAR_ROWS(4, V) GEAR_ROWS(8, V)
  GEAR_ROWS_V(1) GEAR_ROWS_V(2) GEAR_ROWS_V(4) GEAR_ROWS_V(8)
#undef GEAR_ROWS_V
#undef GEAR_ROWS
  return nullptr;
}

}  // namespace gear
