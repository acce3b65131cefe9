// Instances of the fused transforms (series.cuh): template method, 2^17..2^20 points.
#include "series.cuh"

namespace rbseries {

int launch_plain_long(int log2n, const Args& a, int rows_ws, cudaStream_t st) {
  switch (log2n) {
    case 17: return launch<17, 4, KIND_PLAIN>(a, rows_ws, st);
    case 18: return launch<18, 4, KIND_PLAIN>(a, rows_ws, st);
    case 19: return launch<19, 4, KIND_PLAIN>(a, rows_ws, st);
    case 20:  // items of 8 columns; a bin of 16 needs items of 16 (one CTA of eight warps per SM)
      return a.w > 8 ? launch<20, 8, KIND_PLAIN>(a, rows_ws, st) : launch<20, 4, KIND_PLAIN>(a, rows_ws, st);
  }
  rb::set_detail("fused transform of 2^%d points", log2n);
  return RB_ERR_UNSUPPORTED;
}

}  // namespace rbseries
