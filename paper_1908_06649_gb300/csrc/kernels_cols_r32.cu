// kernels_cols_r32.cu -- radix-32 column passes of 2-D transforms (role kCols:
// the array's shape is a runtime value), every precision mode.
#include "launch_impl.cuh"

namespace tcu {

// (stages, with an inter-pass twiddle)
cudaError_t launch_cols_r32(int prec, int s, int twid, const GArgs &a, int num_sms,
                           cudaStream_t st) {
  constexpr int R = 32;
  TCU_COLS_CASE(1, 0, launch_pass_t)
  TCU_COLS_CASE(2, 0, launch_pass_t)
  TCU_COLS_CASE(1, 1, launch_pass_t)
  TCU_COLS_CASE(2, 1, launch_pass_t)
  return cudaErrorInvalidValue;
}

}  // namespace tcu
