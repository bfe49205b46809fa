// kernels_mixed_r16.cu -- radix-16 passes of mixed-radix transforms
// n = q 16^k: the pass that takes the q-point sums on its way in (kSecondQF: the
// only pass, any q = 2 .. 16; kFirstQ: the strided pass of two, q a power of
// two), the last pass with n1 = q 16^s points before it, and, where q does
// not fit an item, the strided pass after a q-point pass.
#include "launch_impl.cuh"

namespace tcu {

// (stages, log2 other size, role, log2 prefix)
cudaError_t launch_pass_mixed_r16(int prec, int s, int lo, int role, int lp, int tw,
                                  const GArgs &a, int num_sms, cudaStream_t st) {
  constexpr int R = 16;
  TCU_PASS_CASE_L(2, 5, kSecond, 0)
  TCU_PASS_CASE_L(2, 9, kSecond, 0)
  TCU_PASS_CASE_L(2, 6, kSecond, 0)
  TCU_PASS_CASE_L(2, 10, kSecond, 0)
  TCU_PASS_CASE_L(2, 7, kSecond, 0)
  TCU_PASS_CASE_L(2, 8, kFirst, 3)
  TCU_PASS_CASE_L(2, 11, kSecond, 0)
  TCU_PASS_CASE_L(1, 8, kFirstQ, 0)
  TCU_TEAM_CASE_L(2, 8, kFirstQ, 0, 2)
  TCU_PASS_CASE_L(1, 0, kSecondQF, 0)
  if (tw == 2) {
    TCU_TEAM_CASE_L(2, 0, kSecondQF, 0, 2)
  }
  TCU_PASS_CASE_L(2, 0, kSecondQF, 0)
  return cudaErrorInvalidValue;
}

}  // namespace tcu
