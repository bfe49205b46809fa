// kernels_cols_r32.cu -- radix-32 column passes of 2-D transforms (role kCols:
// the array's shape is a runtime value), every precision mode.
#include "launch_impl.cuh"

namespace tcu {

// (stages, ColMode)
cudaError_t launch_cols_r32(int prec, int s, int mode, const GArgs &a, int num_sms,
                           cudaStream_t st) {
  constexpr int R = 32;
  TCU_COLS_CASE(1, kColPlain)
  TCU_COLS_CASE(2, kColPlain)
  TCU_COLS_CASE(1, kColTwiddle)
  TCU_COLS_CASE(2, kColTwiddle)
  TCU_COLS_CASE(1, kColSpectrum)
  TCU_COLS_CASE(2, kColSpectrum)
  if (prec != 3) return cudaErrorInvalidValue;
  // real tiles: 1024 points a side
  if (s == 2 && mode == kColGather) return launch_pass_t<R, 3, 2, 0, kCols, kColGather>(a, num_sms, st);
  if (s == 2 && mode == kColScatter) return launch_pass_t<R, 3, 2, 0, kCols, kColScatter>(a, num_sms, st);
  return cudaErrorInvalidValue;
}

}  // namespace tcu
