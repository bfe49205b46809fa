// launch_impl.cuh -- launch wrappers for one radix; included once per radix
// by kernels_r8.cu / kernels_r16.cu / kernels_r32.cu.
#pragma once
#include <string.h>

#include "launch.h"

namespace tcu {

// The status of a launch.  A failure is read from the runtime, which would return
// it again to the next launch that asks for the last error (the element-wise
// kernels do), and so to a call whose kernels ran.
inline cudaError_t launch_status(cudaError_t e) {
  if (e != cudaSuccess) cudaGetLastError();
  return e;
}

// A pass kernel's launch: `sm` bytes of shared memory and, with `beside`, set up
// beside the stream's previous kernel (programmatic serialization; the kernel
// waits for it before it touches data), which takes 2-3 us off every launch:
// n = 65536 x 64 30.8 -> 26.0 us a call, 4096^2 stencils 136 -> 128.
inline cudaError_t launch_serial(void (*kernel)(const GArgs), long long grid, int threads,
                                 size_t sm, bool beside, const GArgs &a, cudaStream_t st) {
  cudaError_t e =
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return launch_status(e);
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = beside ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return launch_status(cudaLaunchKernelEx(&cfg, kernel, a));
}

// Long passes are launched after the kernel before them: CTAs that take the SMs in
// the order they fall free no longer walk the arrays side by side, which costs more
// than the 3 us a launch gained (n = 65536 x 512 168 us beside, 172 after; x 1024
// 331, 332; x 2048 660, 655; 2^24 x 4 508, 511; x 8 1022, 1011; 2-D 1024^2 x 128
// 790, 715).  The line lies between 67 and 84 million points; at radix 8 and with
// one product in BF16, the lightest passes, between 49 and 64 (32768 x 1500, radix
// 8: 289, 293; x 4096 796, 780; 2^20 x 45, radix 32 in BF16: 346, 346; x 61 464,
// 459).  Whole transforms in one pass at radix 16 and 32 gain at any size (256 x
// 400000 264, 268; 4096 x 32768 410, 413).
template <class G, int PREC>
bool launch_beside(bool whole, long long nitems) {
  if (whole && G::LOG2R > 3) return true;
  return nitems * G::GPTS <= (G::LOG2R == 3 || PREC == 4 ? 56 : 72) * 1000000ll;
}

template <int R, int PREC, int S, int LO, int ROLE, int LP>
cudaError_t launch_pass_t(const GArgs &a, int num_sms, cudaStream_t st) {
  using G = Geo<R, S, LO, ROLE, LP, pass_nwg(R, ROLE, S, PREC)>;
  const size_t sm =
      SmemLayout<R, G::NWG, G::TW_ENTRIES, G::MIX_ENTRIES, G::TW_SMEM, G::TWB, 1, G::KS>::BYTES;
  // one CTA per SM, each item on its own SM while there are fewer items
  // than SMs (latency), several per SM otherwise
  const long long nitems = pass_items<G>(a.p[0]);
  long long grid = nitems < num_sms ? nitems : num_sms;
  const bool whole = ROLE == kSingle || ROLE == kSecondQF;
  return launch_serial(dft_pass_kernel<R, PREC, S, LO, ROLE, LP>, grid, G::THREADS, sm,
                       launch_beside<G, PREC>(whole, nitems), a, st);
}

// A team pass: items of TW warpgroups (128 TW rows), team_nwg(R) warpgroups
// a CTA.
template <int R, int PREC, int S, int LO, int ROLE, int LP, int TW>
cudaError_t launch_team_t(const GArgs &a, int num_sms, cudaStream_t st) {
  using G = Geo<R, S, LO, ROLE, LP, team_nwg(R), TW>;
  const size_t sm = SmemLayout<R, G::NWG, G::TW_ENTRIES, G::MIX_ENTRIES, G::TW_SMEM, G::TWB, TW>::BYTES;
  const long long nitems = pass_items<G>(a.p[0]);
  long long grid = nitems < num_sms ? nitems : num_sms;
  const bool whole = ROLE == kSingle || ROLE == kSecondQF;
  return launch_serial(dft_pass_kernel<R, PREC, S, LO, ROLE, LP, kNoConv, TW>, grid, G::THREADS,
                       sm, launch_beside<G, PREC>(whole, nitems), a, st);
}

#define TCU_TEAM_CASE_L(S, LO, ROLE, LP, TW)                                             \
  if (s == S && lo == LO && role == ROLE && lp == LP)                                     \
    return prec == 3 ? launch_team_t<R, 3, S, LO, ROLE, LP, TW>(a, num_sms, st)           \
                     : launch_team_t<R, 1, S, LO, ROLE, LP, TW>(a, num_sms, st);
#define TCU_TEAM_CASE(S, SO, ROLE, SP, TW) \
  TCU_TEAM_CASE_L(S, log2_radix(R) * (SO), ROLE, log2_radix(R) * (SP), TW)

// The convolution row pass (forward rows, spectrum product, inverse rows).
template <int R, int PREC, int S, int CONV>
cudaError_t launch_rowconv_t(const GArgs &a, int num_sms, cudaStream_t st) {
  using G = Geo<R, S, 0, kSingle, 0, whole_k_nwg(R, S)>;
  const size_t sm = SmemLayout<R, G::NWG, G::TW_ENTRIES, G::TW_ENTRIES, false, 0>::BYTES;
  const long long nitems = pass_items<G>(a.p[0]);
  long long grid = nitems < num_sms ? nitems : num_sms;
  return launch_serial(dft_pass_kernel<R, PREC, S, 0, kSingle, 0, CONV>, grid, G::THREADS, sm,
                       launch_beside<G, PREC>(false, nitems), a, st);
}

#define TCU_ROWCONV_CASE(S)                                                         \
  if (s == S && !real)                                                              \
    return prec == 3 ? launch_rowconv_t<R, 3, S, kConv>(a, num_sms, st)             \
                     : launch_rowconv_t<R, 1, S, kConv>(a, num_sms, st);
// ... of real tiles (3xTF32)
#define TCU_REAL_ROWCONV_CASE(S) \
  if (s == S && real && prec == 3) return launch_rowconv_t<R, 3, S, kRealConv>(a, num_sms, st);

template <int R, int PREC, int S1, int S2>
cudaError_t launch_fused_t(const GArgs &a, int num_sms, cudaStream_t st) {
  using G1 = Geo<R, S1, log2_radix(R) * S2, kFirst, 0, whole_k_nwg(R)>;
  using G2 = Geo<R, S2, log2_radix(R) * S1, kSecond, 0, G1::NWG>;
  const size_t sm =
      SmemLayout<R, G1::NWG, G1::TW_ENTRIES, G2::TW_ENTRIES, G1::TW_SMEM, G1::TWB>::BYTES;
  cudaError_t e = cudaFuncSetAttribute(dft_fused_kernel<R, PREC, S1, S2>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sm);
  if (e != cudaSuccess) return launch_status(e);
  dft_fused_kernel<R, PREC, S1, S2><<<(unsigned)num_sms, G1::THREADS, sm, st>>>(a);
  return cudaGetLastError();
}

// Both passes of a two-pass transform in one launch on clusters of two CTAs
// (dft_pair_kernel): grid = 2 x clusters, one CTA per SM.
template <int R, int PREC, int S1, int S2>
cudaError_t launch_pair_t(const GArgs &a, int clusters, cudaStream_t st) {
  using PL = PairLayout<R, S1, S2>;
  const size_t sm = PL::BYTES;
  cudaError_t e = cudaFuncSetAttribute(dft_pair_kernel<R, PREC, S1, S2>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return launch_status(e);
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3((unsigned)(2 * clusters), 1, 1);
  cfg.blockDim = dim3(PL::G1::THREADS, 1, 1);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return launch_status(cudaLaunchKernelEx(&cfg, dft_pair_kernel<R, PREC, S1, S2>, a));
}

#define TCU_PAIR_CASE(S1, S2)                                                       \
  if (s1 == S1 && s2 == S2)                                                         \
    return prec == 3 ? launch_pair_t<R, 3, S1, S2>(a, clusters, st)                 \
                     : launch_pair_t<R, 1, S1, S2>(a, clusters, st);

// Supported combinations of the warpgroup pass kernel for radix R, listed as
// a compile-time table; the plan only asks for these.  The dispatcher gets
// (s, lo, role, lp): stages, log2 of the other size (columns of a strided
// pass, points before the last pass) and log2 of the prefix count.
// TCU_PASS_CASE names sizes in stages of R, TCU_PASS_CASE_L in log2 units
// (mixed radix, where a factor q < R enters).
#define TCU_PASS_CASE_L(S, LO, ROLE, LP)                                            \
  if (s == S && lo == LO && role == ROLE && lp == LP)                               \
    return prec == 3 ? launch_pass_t<R, 3, S, LO, ROLE, LP>(a, num_sms, st)         \
                     : launch_pass_t<R, 1, S, LO, ROLE, LP>(a, num_sms, st);
#define TCU_PASS_CASE(S, SO, ROLE, SP) \
  TCU_PASS_CASE_L(S, log2_radix(R) * (SO), ROLE, log2_radix(R) * (SP))
// The BF16 modes (precision 4: BF16, 5: 3xBF16; tcgen05 kind::f16) of a
// pass or a team pass (items of TW warpgroups).
#define TCU_BF16_CASE(S, SO, ROLE, SP)                                                  \
  if (s == S && lo == log2_radix(R) * (SO) && role == ROLE &&                           \
      lp == log2_radix(R) * (SP))                                                       \
    return prec == 5 ? launch_pass_t<R, 5, S, log2_radix(R) * (SO), ROLE,               \
                                     log2_radix(R) * (SP)>(a, num_sms, st)              \
                     : launch_pass_t<R, 4, S, log2_radix(R) * (SO), ROLE,               \
                                     log2_radix(R) * (SP)>(a, num_sms, st);
#define TCU_BF16_TEAM_CASE(S, SO, ROLE, SP, TW)                                         \
  if (s == S && lo == log2_radix(R) * (SO) && role == ROLE &&                           \
      lp == log2_radix(R) * (SP))                                                       \
    return prec == 5 ? launch_team_t<R, 5, S, log2_radix(R) * (SO), ROLE,               \
                                     log2_radix(R) * (SP), TW>(a, num_sms, st)          \
                     : launch_team_t<R, 4, S, log2_radix(R) * (SO), ROLE,               \
                                     log2_radix(R) * (SP), TW>(a, num_sms, st);
// A column pass of a 2-D transform (kCols) of S stages in ColMode MODE, items
// of one warpgroup (or, TCU_COLS_TEAM_CASE, of TW); every precision.
#define TCU_COLS_CASE(S, MODE)                                                            \
  if (s == S && mode == MODE) {                                                           \
    if (prec == 3) return launch_pass_t<R, 3, S, 0, kCols, MODE>(a, num_sms, st);         \
    if (prec == 1) return launch_pass_t<R, 1, S, 0, kCols, MODE>(a, num_sms, st);         \
    if (prec == 5) return launch_pass_t<R, 5, S, 0, kCols, MODE>(a, num_sms, st);         \
    return launch_pass_t<R, 4, S, 0, kCols, MODE>(a, num_sms, st);                        \
  }
#define TCU_COLS_TEAM_CASE(S, MODE, TW)                                                   \
  if (s == S && mode == MODE) {                                                           \
    if (prec == 3) return launch_team_t<R, 3, S, 0, kCols, MODE, TW>(a, num_sms, st);     \
    if (prec == 1) return launch_team_t<R, 1, S, 0, kCols, MODE, TW>(a, num_sms, st);     \
    if (prec == 5) return launch_team_t<R, 5, S, 0, kCols, MODE, TW>(a, num_sms, st);     \
    return launch_team_t<R, 4, S, 0, kCols, MODE, TW>(a, num_sms, st);                    \
  }
#define TCU_FUSED_CASE(S1, S2)                                                      \
  if (s1 == S1 && s2 == S2)                                                         \
    return prec == 3 ? launch_fused_t<R, 3, S1, S2>(a, num_sms, st)                 \
                     : launch_fused_t<R, 1, S1, S2>(a, num_sms, st);

}  // namespace tcu
