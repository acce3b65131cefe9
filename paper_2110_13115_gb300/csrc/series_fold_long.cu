// Instances of the fused transforms (series.cuh): folded first stage, 2^17..2^19 points.
#include "series.cuh"

namespace rbseries {

int launch_fold_long(int log2n, const Args& a, int rows_ws, cudaStream_t st) {
  switch (log2n) {
    case 17: return launch<17, 4, KIND_FOLD>(a, rows_ws, st);
    case 18: return launch<18, 4, KIND_FOLD>(a, rows_ws, st);
    case 19: return launch<19, 4, KIND_FOLD>(a, rows_ws, st);
  }
  rb::set_detail("fused transform of 2^%d points", log2n);
  return RB_ERR_UNSUPPORTED;
}

}  // namespace rbseries
