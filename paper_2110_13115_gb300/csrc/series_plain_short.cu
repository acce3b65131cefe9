// Instances of the fused transforms (series.cuh): template method, 2^14..2^16 points.
#include "series.cuh"

namespace rbseries {

int launch_plain_short(int log2n, const Args& a, int rows_ws, cudaStream_t st) {
  switch (log2n) {
    case 14: return launch<14, 4, KIND_PLAIN>(a, rows_ws, st);
    case 15: return launch<15, 4, KIND_PLAIN>(a, rows_ws, st);
    case 16: return launch<16, 4, KIND_PLAIN>(a, rows_ws, st);
  }
  rb::set_detail("fused transform of 2^%d points", log2n);
  return RB_ERR_UNSUPPORTED;
}

}  // namespace rbseries
