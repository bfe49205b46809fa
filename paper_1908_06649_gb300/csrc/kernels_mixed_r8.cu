// kernels_mixed_r8.cu -- radix-8 passes of mixed-radix transforms n = q 8^k: the
// pass that takes the q-point sums on its way in (kSecondQF: the only pass,
// any q = 2 .. 16; kFirstQ: the strided pass of two, q a power of two), the last
// pass with n1 = q 8^s points before it, and, where q does not fit an item, the
// pass after a q-point pass.
#include "launch_impl.cuh"

namespace tcu {

// (stages, log2 other size, role, log2 prefix)
cudaError_t launch_pass_mixed_r8(int prec, int s, int lo, int role, int lp, int,
                                  const GArgs &a, int num_sms, cudaStream_t st) {
  constexpr int R = 8;
  TCU_PASS_CASE_L(2, 7, kSecond, 0)
  TCU_PASS_CASE_L(2, 8, kSecond, 0)
  TCU_PASS_CASE_L(2, 6, kFirstQ, 0)
  TCU_PASS_CASE_L(1, 0, kSecondQF, 0)
  TCU_PASS_CASE_L(2, 0, kSecondQF, 0)
  TCU_TEAM_CASE_L(3, 0, kSecondQF, 0, 4)
  TCU_PASS_CASE_L(1, 0, kSecondQ, 0)
  TCU_PASS_CASE_L(2, 0, kSecondQ, 0)
  TCU_TEAM_CASE_L(3, 0, kSecondQ, 0, 4)
  return cudaErrorInvalidValue;
}

}  // namespace tcu
