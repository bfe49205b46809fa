// kernels_mixed_r32.cu -- radix-32 passes of mixed-radix transforms
// n = q 32^k: the pass that takes the q-point sums on its way in (kSecondQF: the
// only pass; kFirstQ: the strided pass of two, q a power of two), the last pass
// with n1 = q 32^s points before it, and, where q does not fit an item, the
// pass after a q-point pass.
#include "launch_impl.cuh"

namespace tcu {

// (stages, log2 other size, role, log2 prefix)
cudaError_t launch_pass_mixed_r32(int prec, int s, int lo, int role, int lp, int,
                                  const GArgs &a, int num_sms, cudaStream_t st) {
  constexpr int R = 32;
  TCU_PASS_CASE_L(2, 6, kSecond, 0)
  TCU_PASS_CASE_L(2, 7, kSecond, 0)
  TCU_PASS_CASE_L(2, 3, kSecond, 0)
  TCU_PASS_CASE_L(2, 8, kSecond, 0)
  TCU_PASS_CASE_L(2, 4, kSecond, 0)
  TCU_PASS_CASE_L(2, 9, kSecond, 0)
  TCU_PASS_CASE_L(1, 10, kFirstQ, 0)
  TCU_PASS_CASE_L(1, 0, kSecondQF, 0)
  TCU_PASS_CASE_L(2, 0, kSecondQF, 0)
  TCU_PASS_CASE_L(2, 0, kSecondQ, 0)
  return cudaErrorInvalidValue;
}

}  // namespace tcu
