// grid_plan.cu -- the 2-D rows of the library (Sec. 4.6): 2-D DFT plans,
// circular 2-D convolution and the linear stencil of Lemmas 1 and 2.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <cmath>
#include <mutex>
#include <vector>

#include "host_plan.h"

using namespace tcu;
using namespace tcu::host;

// =========================================================== 2-D transforms
// A 2-D DFT of batch row-major n1 x n2 arrays (Sec. 4.6: the 1-D DFT of
// every column, then of every row) is two warpgroup passes: the column pass
// (kCols: the strided geometry without a twiddle, T[b][k1][v]) and the
// row pass (kSingle over batch * n1 rows, natural order).  A circular
// convolution with a fixed array whose spectrum S is given is three:
// columns, rows (forward, times S, inverse -- on chip, one item at a time),
// inverse columns (1/(n1 n2) folded into the last stage's F images).


// Axes beyond one warpgroup pass, and the BF16 modes (the general path): the
// rows by a 1-D plan of length n2, then the columns in up to three strided
// passes of role kCols (the four-step split of the column length; the digit
// reversal is in their output rows, so nothing is transposed).  HBM-bound: one
// round trip per pass, two fewer than with a transpose each way (4096 x 4096 x 4
// 917 -> 534 us, 256 x 256 x 1000 in BF16 780 -> 321, 65536 x 16 x 64
// 1504 -> 619).  A convolution multiplies by the spectrum as the last forward
// column pass stores, then runs the inverse columns and rows.
// Arrays smaller than one column item (n1 n2 < 128 r) transpose instead:
// rows, transpose, the columns as rows, transpose back.
struct tcu_dft2_plan_s {
  long long n1, n2, batch;
  int r, precision, num_sms;
  PassPlan rows;
  float *bimg[2];     // [dir index]; scaled copies by 2^-log2(n1 n2), by 1/n1 (general path)
  float *cimg;        // convolution rows: forward hi, lo | inverse hi, lo
  float2 *scratch;    // batch * n1 * n2
  int *err;
  int ncol;  // column passes (0: transpose instead)
  PassPlan colp[kMaxPasses];
  bool general;
  tcu_dft_plan_t rows1d, cols1d;  // length n2 / n1 plans (cols1d: ncol = 0)
  float2 *spec_t;                 // ncol = 0: the spectrum transposed
};

// A stencil plan.  In 3xTF32 with tiles of one warpgroup pass per axis the
// tiles stay real (`real`): the column pass gathers them from the grid, two
// real columns as one complex one (N / 2 columns a tile); the row pass
// untangles the rows 0 .. N / 2 of the column spectra (the others are their
// conjugates), convolves them and packs them again; the inverse column pass
// scatters the output blocks to the grid.  Half the transforms and a third of
// the traffic of complex tiles (4096^2, 85 steps: 1666 -> 771 us; 512^2 radix-8
// tiles, 100 steps: 1022 -> 400; with the spectrum below too, 16 steps 365 -> 128).
// The other modes keep complex tiles: with single products every rounding of the
// operands would move.
struct tcu_stencil_plan_s {
  long long side, N, Nw, tiles;
  int B;  // output block side: N - 2k (Lemma 1's tiles are blocks of k)
  int k, r, precision, num_sms;
  bool real;              // real tiles
  bool closed;            // the spectrum by stencil_spectrum_kernel
  tcu_dft2_plan_t conv;   // N x N (real: N x N / 2), batch = tiles
  tcu_dft2_plan_t wconv;  // N x N, batch 1 (spectrum of the kernel; not closed)
  tcu_dft2_plan_t wpow;   // Nw x Nw, batch 1 (Lemma 2)
  float2 *tile_buf;       // tiles * N * N (not real)
  float2 *wgrid;          // Nw * Nw
  float2 *wker;           // N * N: the kernel W', then its spectrum
  double2 *roots;         // closed: w_N^{-f}, f < N
};

// Steps up to which a real-tile plan evaluates the kernel's spectrum directly:
// one launch instead of nine (a grid of 1000^2: 25 us with 20 steps, 50 with 21),
// and more exact (error of the output with 16 steps 7.9e-6 -> 1.3e-6).  Neither
// speed nor exactness sets the line: beyond it the spectrum comes, as before, from
// the transforms of Lemma 2, as tcu_stencil_weights' weights do, whose error grows
// with k (about 5e-7 k of the output), so that results stay within 2e-5 of what
// those weights give on either side of the line.
constexpr int kClosedSteps = 20;

namespace {

bool is_power_of(long long n, int r, int &k) {
  k = 0;
  long long m = 1;
  while (m < n) {
    m *= r;
    ++k;
  }
  return m == n && k >= 1;
}

// A single-pass stage count for radix r (the largest sub-transform of one
// warpgroup item).
int single_pass_stages(int r) { return r == 8 ? 3 : 2; }

void free_dft2(tcu_dft2_plan_s *p) {
  if (!p) return;
  tcu_dft_destroy(p->rows1d);
  tcu_dft_destroy(p->cols1d);
  cudaFree(p->spec_t);
  for (int d = 0; d < 2; ++d) {
    for (int i = 0; i < p->ncol; ++i) {
      cudaFree(p->colp[i].tw_stage[d]);
      cudaFree(p->colp[i].tw_a[d]);
      cudaFree(p->colp[i].tw_b[d]);
    }
    cudaFree(p->bimg[d]);
    cudaFree(p->rows.tw_stage[d]);
  }
  cudaFree(p->cimg);
  cudaFree(p->scratch);
  cudaFree(p->err);
  delete p;
}

PRun dft2_pass(const tcu_dft2_plan_s *p, const PassPlan &pp, int di, const float2 *in,
               float2 *out, bool scaled, const float2 *spec, int reverse = 0) {
  PRun g;
  memset(&g, 0, sizeof(g));
  g.in = in;
  g.out = out;
  g.in_bmask = g.out_bmask = -1;
  g.U = pp.U;
  g.tw_stage = pp.tw_stage[di];
  g.swz_tab = pp.swz_tab;
  g.last_img = scaled ? 2 * (prec_bf16(p->precision) ? 8 : 16) * p->r * p->r : 0;
  g.spec = spec;
  g.spec_mask = p->n1 - 1;
  g.reverse = reverse;
  return g;
}

// The row pass of the two-pass path; it follows the column pass: items last to
// first (L2 reuse).
int run_rows(const tcu_dft2_plan_s *p, int di, const float2 *in, float2 *out, bool scaled,
             cudaStream_t st) {
  GArgs g;
  memset(&g, 0, sizeof(g));
  g.p[0] = dft2_pass(p, p->rows, di, in, out, scaled, nullptr, 1);
  g.bimg = p->bimg[di];
  g.err = p->err;
  return pass_dispatch(p->r, p->precision, p->rows, g, p->num_sms, st) == cudaSuccess
             ? TCU_DFT_OK
             : TCU_DFT_ERR_CUDA;
}

// Column pass i; scaled: with the scaled F images; spec: its output times this
// spectrum (last pass); reverse: items last to first.
int run_col_pass(const tcu_dft2_plan_s *p, int i, int di, const float2 *in, float2 *out,
                 bool scaled, const float2 *spec, bool reverse, cudaStream_t st) {
  const PassPlan &c = p->colp[i];
  GArgs g;
  memset(&g, 0, sizeof(g));
  g.p[0] = dft2_pass(p, c, di, in, out, scaled, spec, reverse && c.tw == 1);
  g.p[0].lo = c.lo;
  g.p[0].lp = c.lp;
  g.p[0].lc = ilog2(p->n2);
  g.p[0].tw_out = c.tw_a[di];
  g.p[0].tw_b = c.tw_b[di];
  const long long L = 1ll << c.log2L;
  const int gg = (int)((128ll * c.tw * p->r) >> c.log2L);
  if (!encode_map(&g.tm_in, in, 1ll << c.lo, L, p->batch << c.lp, L << c.lo, gg,
                  L < 256 ? (int)L : 256))
    return TCU_DFT_ERR_CUDA;
  g.bimg = p->bimg[di];
  g.err = p->err;
  const int mode = !c.last ? kColTwiddle : (spec ? kColSpectrum : kColPlain);
  return launch_cols(p->r, p->precision, c.s, mode, g, p->num_sms, st) == cudaSuccess
             ? TCU_DFT_OK
             : TCU_DFT_ERR_CUDA;
}

int check_buffers(const void *in, const void *out, size_t bytes) {
  if (!in || !out || ((uintptr_t)in & 15) || ((uintptr_t)out & 15)) return TCU_DFT_ERR_INVALID;
  if (in != out && overlaps(in, out, bytes)) return TCU_DFT_ERR_INVALID;
  return TCU_DFT_OK;
}

// Stages of the strided passes of columns of length r^k beside n2 columns, as
// plan_stages but with at most two radix-16 stages each.  Every item's columns
// must exist: GG <= rest n2.  0: no such split (transpose instead).
int col_stages(int r, int k, long long n2, int precision, int st[kMaxPasses]) {
  int P;
  if (k <= single_pass_stages(r)) {
    st[0] = k;
    P = 1;
  } else if (r == 16 && k == 3) {
    st[0] = 1;
    st[1] = 2;
    P = 2;
  } else if (r == 8 && k == 4 && n2 < 16) {
    // a 2-stage item spans 16 columns, a 3-stage team item 8; the other split
    // rounds the operands of the single-product modes elsewhere
    if (precision != TCU_DFT_3XTF32) return 0;
    st[0] = 1;
    st[1] = 3;
    P = 2;
  } else {
    P = plan_stages(r, k, st);
  }
  long long rest = n2;
  for (int i = P - 1; i >= 0; --i) {
    const long long L = 1ll << (ilog2(r) * st[i]);
    const int tw = r == 8 && st[i] == 3 ? 4 : 1;
    if (rest * L < 128ll * tw * r) return 0;
    rest *= L;
  }
  return P;
}

// The columns' tables: the F images scaled by 1/n (unscaled ones also to
// *conv_img, a convolution row pass's), and per column pass
// its geometry, stage twiddles and inter-pass twiddles [row of rest][k].
int make_cols(tcu_dft2_plan_s *p, const int *st, long long n,
              std::vector<float> *conv_img = nullptr) {
  const int log2r = ilog2(p->r);
  int rc = TCU_DFT_OK;
  long long pre = 1;
  for (int i = 0; i < p->ncol; ++i) {
    PassPlan &c = p->colp[i];
    const long long L = 1ll << (log2r * st[i]), rest = p->n1 / (pre * L);
    c.s = st[i];
    c.role = kCols;
    c.log2L = log2r * c.s;
    c.lo = ilog2(rest * p->n2);
    c.lp = ilog2(pre);
    c.last = i == p->ncol - 1;
    c.U = p->batch * pre * rest * p->n2;
    c.modes[0] = c.modes[1] = c.modes[2] = kUF;
    c.tw = team_size(p->r, c);
    c.swz_tab = choose_swizzle(p->r, c.s, c.modes, c.tw);
    for (int d = 0; d < 2 && rc == TCU_DFT_OK; ++d) {
      const int sign = d == 0 ? -1 : 1;
      rc = upload(&c.tw_stage[d], stage_twiddles(p->r, c.s, sign));
      if (c.last || rc != TCU_DFT_OK) continue;
      // [row of rest][k], in two levels beyond kColRows rows
      const long long low = rest >> kLog2ColRows ? 1ll << kLog2ColRows : rest;
      std::vector<float2> t((size_t)(low * L));
      for (long long a = 0; a < low; ++a)
        for (long long k = 0; k < L; ++k) t[(size_t)(a * L + k)] = root(a * k, L * rest, sign);
      rc = upload(&c.tw_a[d], t);
      if (low == rest || rc != TCU_DFT_OK) continue;
      t.resize((size_t)(rest / low * L));
      for (long long a = 0; a < rest / low; ++a)
        for (long long k = 0; k < L; ++k)
          t[(size_t)(a * L + k)] = root(a * low * k, L * rest, sign);
      rc = upload(&c.tw_b[d], t);
    }
    pre *= L;
  }
  for (int d = 0; d < 2 && rc == TCU_DFT_OK; ++d) {
    std::vector<float> img;
    build_images(p->r, d == 0 ? -1 : 1, n, p->precision, img);
    rc = upload(&p->bimg[d], img);
    // hi and lo of each direction (the first two images)
    if (conv_img) conv_img->insert(conv_img->end(), img.begin(), img.begin() + img.size() / 2);
  }
  return rc;
}

// The general path: the rows by a 1-D plan (n2, batch n1 of them), the columns
// by strided passes, or (small arrays) by a 1-D plan between transposes.
// UNSUPPORTED if either length has no 1-D plan.
tcu_dft2_plan_s *make_dft2_general(int64_t n1, int64_t n2, int64_t batch, int32_t r, int k1,
                                   int32_t precision, int &rc) {
  // both lengths must have a 1-D plan (a host-side question: no CUDA call)
  int32_t st[kMaxPasses];
  if (tcu_dft_plan_passes(n1, r, st) == 0 || tcu_dft_plan_passes(n2, r, st) == 0) {
    rc = TCU_DFT_ERR_UNSUPPORTED;
    return nullptr;
  }
  tcu_dft2_plan_s *p = new tcu_dft2_plan_s();
  memset(p, 0, sizeof(*p));
  p->n1 = n1;
  p->n2 = n2;
  p->batch = batch;
  p->r = r;
  p->precision = precision;
  p->general = true;
  int cst[kMaxPasses];
  p->ncol = col_stages(r, k1, n2, precision, cst);
  p->rows1d = tcu_dft_plan(n2, batch * n1, r, precision);
  rc = p->rows1d ? TCU_DFT_OK : tcu_dft_last_error();
  if (rc == TCU_DFT_OK && p->ncol) rc = make_cols(p, cst, n1);
  if (rc == TCU_DFT_OK && !p->ncol) {
    p->cols1d = tcu_dft_plan(n1, batch * n2, r, precision);
    rc = p->cols1d ? TCU_DFT_OK : tcu_dft_last_error();
  }
  if (rc == TCU_DFT_OK) {
    p->num_sms = p->rows1d->num_sms;
    if (dev_malloc((void **)&p->scratch, (size_t)(batch * n1 * n2) * sizeof(float2)) !=
            cudaSuccess ||
        (!p->ncol &&
         dev_malloc((void **)&p->spec_t, (size_t)(n1 * n2) * sizeof(float2)) != cudaSuccess) ||
        dev_malloc((void **)&p->err, sizeof(int)) != cudaSuccess ||
        cudaMemset(p->err, 0, sizeof(int)) != cudaSuccess) {
      cudaGetLastError();
      rc = TCU_DFT_ERR_OOM;
    }
  }
  if (rc != TCU_DFT_OK) {
    free_dft2(p);
    return nullptr;
  }
  return p;
}

// The column passes of one direction on `at`, one of the scratch and `out`,
// alternating between the two; returns a status and leaves `at` at the result.
int run_cols(const tcu_dft2_plan_s *p, int di, float2 *&at, float2 *out, const float2 *spec,
             cudaStream_t st) {
  for (int i = 0; i < p->ncol; ++i) {
    float2 *dst = at == p->scratch ? out : p->scratch;
    const bool last = p->colp[i].last;
    // every second pass last to first, from the rows' pass on (L2 reuse)
    const int rc = run_col_pass(p, i, di, at, dst, di == 1 && last, last ? spec : nullptr,
                                !(i & 1), st);
    if (rc != TCU_DFT_OK) return rc;
    at = dst;
  }
  return TCU_DFT_OK;
}

// General path: the 2-D transform of `in` into `out`.
int general_dft2(const tcu_dft2_plan_s *p, const void *in, void *out, int dir,
                 cudaStream_t st) {
  if (p->ncol) {
    // the column passes alternate and end in out
    float2 *at = p->ncol & 1 ? p->scratch : (float2 *)out;
    const int rc = tcu_dft_exec_dir(p->rows1d, in, at, dir, st);
    return rc != TCU_DFT_OK ? rc
                            : run_cols(p, dir_index(dir), at, (float2 *)out, nullptr, st);
  }
  int rc = tcu_dft_exec_dir(p->rows1d, in, out, dir, st);
  if (rc != TCU_DFT_OK) return rc;
  if (launch_transpose(p->scratch, (const float2 *)out, p->batch, p->n1, p->n2, p->num_sms,
                       st) != cudaSuccess)
    return TCU_DFT_ERR_CUDA;
  rc = tcu_dft_exec_dir(p->cols1d, p->scratch, p->scratch, dir, st);
  if (rc != TCU_DFT_OK) return rc;
  return launch_transpose((float2 *)out, p->scratch, p->batch, p->n2, p->n1, p->num_sms, st) ==
                 cudaSuccess
             ? TCU_DFT_OK
             : TCU_DFT_ERR_CUDA;
}

// General path: the convolution of `in` with the array of the given spectrum.
int general_conv2(const tcu_dft2_plan_s *p, const void *in, const float2 *spectrum, void *out,
                  cudaStream_t st) {
  if (p->ncol) {
    // rows and columns forward, times the spectrum, columns and rows back
    float2 *at = (float2 *)out;
    int rc = tcu_dft_exec_dir(p->rows1d, in, out, TCU_DFT_FORWARD, st);
    if (rc == TCU_DFT_OK) rc = run_cols(p, 0, at, (float2 *)out, spectrum, st);
    if (rc == TCU_DFT_OK) rc = run_cols(p, 1, at, (float2 *)out, nullptr, st);
    return rc != TCU_DFT_OK ? rc : tcu_dft_exec_dir(p->rows1d, out, out, TCU_DFT_INVERSE, st);
  }
  // rows and columns forward (left transposed in the scratch), times the
  // spectrum transposed, columns back, transpose back, rows back
  int rc = tcu_dft_exec_dir(p->rows1d, in, out, TCU_DFT_FORWARD, st);
  if (rc != TCU_DFT_OK) return rc;
  if (launch_transpose(p->scratch, (const float2 *)out, p->batch, p->n1, p->n2, p->num_sms,
                       st) != cudaSuccess)
    return TCU_DFT_ERR_CUDA;
  rc = tcu_dft_exec_dir(p->cols1d, p->scratch, p->scratch, TCU_DFT_FORWARD, st);
  if (rc != TCU_DFT_OK) return rc;
  if (launch_transpose(p->spec_t, spectrum, 1, p->n1, p->n2, p->num_sms, st) != cudaSuccess ||
      launch_spectrum_product(p->scratch, p->spec_t, p->batch, p->n1 * p->n2, p->num_sms, st) !=
          cudaSuccess)
    return TCU_DFT_ERR_CUDA;
  rc = tcu_dft_exec_dir(p->cols1d, p->scratch, p->scratch, TCU_DFT_INVERSE, st);
  if (rc != TCU_DFT_OK) return rc;
  if (launch_transpose((float2 *)out, p->scratch, p->batch, p->n2, p->n1, p->num_sms, st) !=
      cudaSuccess)
    return TCU_DFT_ERR_CUDA;
  return tcu_dft_exec_dir(p->rows1d, out, out, TCU_DFT_INVERSE, st);
}

// Plans run on sm_103 only; the number of its SMs.
int device_sms(int &rc) {
  int dev = 0;
  cudaDeviceProp prop;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaGetDeviceProperties(&prop, dev) != cudaSuccess ||
      prop.major != 10 || prop.minor != 3) {
    cudaGetLastError();
    rc = TCU_DFT_ERR_CUDA;
    return 0;
  }
  rc = TCU_DFT_OK;
  return prop.multiProcessorCount;
}

// Tables and buffers of the two-pass path: rows of row_len points (U of them) in
// one pass, the columns of n1 x n2 arrays in another; images scaled by
// 1 / (n1 row_len).
int make_two_pass(tcu_dft2_plan_s *p, int k1, int k2, long long row_len, long long U) {
  const int r = p->r;
  PassPlan &w = p->rows;
  w.s = k2;
  w.role = kSingle;
  w.so = w.sp = w.lo = w.lp = 0;
  w.log2L = ilog2(r) * k2;
  w.U = U;
  w.modes[0] = kQF;
  w.modes[1] = kUF;
  w.modes[2] = kRQF;
  w.tw = team_size(r, w);
  w.swz_tab = choose_swizzle(r, w.s, w.modes, w.tw);
  std::vector<float> conv_img;
  p->ncol = 1;
  int rc = make_cols(p, &k1, p->n1 * row_len, &conv_img);
  for (int d = 0; d < 2 && rc == TCU_DFT_OK; ++d)
    rc = upload(&w.tw_stage[d], stage_twiddles(r, w.s, d == 0 ? -1 : 1));
  if (rc == TCU_DFT_OK) rc = upload(&p->cimg, conv_img);
  if (rc == TCU_DFT_OK &&
      (dev_malloc((void **)&p->scratch, (size_t)(p->batch * p->n1 * p->n2) * sizeof(float2)) !=
           cudaSuccess ||
       dev_malloc((void **)&p->err, sizeof(int)) != cudaSuccess ||
       cudaMemset(p->err, 0, sizeof(int)) != cudaSuccess)) {
    cudaGetLastError();
    rc = TCU_DFT_ERR_OOM;
  }
  return rc;
}

// The passes of `tiles` real N x N tiles (N = r^k, 3xTF32): packed arrays of
// N x N / 2.
tcu_dft2_plan_s *make_real_tiles(int64_t N, int k, int64_t tiles, int32_t r, int &rc) {
  const int sms = device_sms(rc);
  if (rc != TCU_DFT_OK) return nullptr;
  tcu_dft2_plan_s *p = new tcu_dft2_plan_s();
  memset(p, 0, sizeof(*p));
  p->n1 = N;
  p->n2 = N / 2;
  p->batch = tiles;
  p->r = r;
  p->precision = TCU_DFT_3XTF32;
  p->num_sms = sms;
  rc = make_two_pass(p, k, k, N, tiles * (N / 2 + 1));
  if (rc != TCU_DFT_OK) {
    free_dft2(p);
    return nullptr;
  }
  return p;
}

cudaError_t launch_rowconv(const tcu_dft2_plan_s *p, bool real, const GArgs &g,
                           cudaStream_t st) {
  if (p->r == 8) return launch_rowconv_r8(p->precision, p->rows.s, real, g, p->num_sms, st);
  if (p->r == 16) return launch_rowconv_r16(p->precision, p->rows.s, real, g, p->num_sms, st);
  return launch_rowconv_r32(p->precision, p->rows.s, real, g, p->num_sms, st);
}

// Convolve every tile of the grid A with the kernel of the given spectrum (rows
// 0 .. N / 2 of it) into the output blocks of Ak: three launches.
int run_real_tiles(const tcu_stencil_plan_s *sp, const float *A, float *Ak,
                   const float2 *spectrum, cudaStream_t st) {
  const tcu_dft2_plan_s *p = sp->conv;
  const PassPlan &c = p->colp[0];
  GArgs g;
  memset(&g, 0, sizeof(g));
  g.err = p->err;
  for (int pass = 0; pass < 3; ++pass) {
    const int di = pass == 2 ? 1 : 0;
    // the row pass runs last to first, so each pass starts on what the one
    // before wrote last
    g.p[0] = pass == 1 ? dft2_pass(p, p->rows, 0, p->scratch, p->scratch, false, spectrum, 1)
                       : dft2_pass(p, c, di, p->scratch, p->scratch, pass == 2, nullptr);
    PRun &q = g.p[0];
    q.lo = q.lc = c.lo;
    q.grid_in = A;
    q.grid_out = Ak;
    q.side = sp->side;
    q.tpr = (int)((sp->side + sp->B - 1) / sp->B);
    q.block = sp->B;
    q.halo = sp->k;
    q.half = (int)(sp->N / 2 + 1);
    g.bimg = pass == 1 ? p->cimg : p->bimg[di];
    g.p[1].tw_stage = p->rows.tw_stage[1];
    cudaError_t e;
    if (pass == 1) {
      e = launch_rowconv(p, true, g, st);
    } else {
      const int gg = (int)((128ll * c.tw * p->r) >> c.log2L);
      if (pass == 2 && !encode_map(&g.tm_in, p->scratch, p->n2, p->n1, p->batch, p->n1 * p->n2,
                                   gg, p->n1 < 256 ? (int)p->n1 : 256))
        return TCU_DFT_ERR_CUDA;
      e = launch_cols(p->r, p->precision, c.s, pass == 0 ? kColGather : kColScatter, g,
                      p->num_sms, st);
    }
    if (e != cudaSuccess) return TCU_DFT_ERR_CUDA;
  }
  return TCU_DFT_OK;
}

tcu_dft2_plan_s *make_dft2(int64_t n1, int64_t n2, int64_t batch, int32_t r,
                           int32_t precision, int &rc) {
  rc = TCU_DFT_OK;
  if (n1 < 1 || n2 < 1 || batch < 1 ||
      (precision != TCU_DFT_TF32 && precision != TCU_DFT_3XTF32 && !prec_bf16(precision))) {
    rc = TCU_DFT_ERR_INVALID;
    return nullptr;
  }
  int k1 = 0, k2 = 0;
  if ((r != 8 && r != 16 && r != 32) || !is_power_of(n1, r, k1) || !is_power_of(n2, r, k2) ||
      batch * n1 * n2 > (1ll << 40)) {
    rc = TCU_DFT_ERR_UNSUPPORTED;
    return nullptr;
  }
  // each axis one warpgroup pass (a column item spans 128 r / n1 columns),
  // TF32 modes: the two-pass path; otherwise the general path
  if (prec_bf16(precision) || k1 > single_pass_stages(r) || k2 > single_pass_stages(r) ||
      n1 * n2 < 128ll * r)
    return make_dft2_general(n1, n2, batch, r, k1, precision, rc);
  const int sms = device_sms(rc);
  if (rc != TCU_DFT_OK) return nullptr;
  tcu_dft2_plan_s *p = new tcu_dft2_plan_s();
  memset(p, 0, sizeof(*p));
  p->n1 = n1;
  p->n2 = n2;
  p->batch = batch;
  p->r = r;
  p->precision = precision;
  p->num_sms = sms;
  rc = make_two_pass(p, k1, k2, n2, batch * n1);
  if (rc != TCU_DFT_OK) {
    free_dft2(p);
    return nullptr;
  }
  return p;
}

void free_stencil(tcu_stencil_plan_s *p) {
  if (!p) return;
  free_dft2(p->conv);
  free_dft2(p->wconv);
  free_dft2(p->wpow);
  cudaFree(p->tile_buf);
  cudaFree(p->wgrid);
  cudaFree(p->wker);
  cudaFree(p->roots);
  delete p;
}

// Smallest power of r, at least `need`, whose square holds a column item
// (128 r points): one warpgroup pass per axis where that suffices, else the
// general path up to 2^26 points per grid (8192^2); 0 if none.
long long grid_side(int r, long long need) {
  for (long long N = r; N * N <= (1ll << 26); N *= r)
    if (N >= need && N * N >= 128ll * r) return N;
  return 0;
}

// Tile side of a stencil plan: the smallest N = r^s with N >= 3k and
// N^2 >= 128 r (one warpgroup pass per axis); 0 if none.  Larger tiles give
// larger output blocks (fewer tile points) but were measured slower per
// point where they take three radix-8 stages per axis or radix-32 rows
// (4096^2 x 16 steps, complex tiles: 512^2 1.31 ms against 0.856 ms for 64^2).
long long stencil_tile(int r, long long k, long long side) {
  (void)side;
  return grid_side(r, 3 * k);
}

}  // namespace

extern "C" {

int64_t tcu_stencil_tiles(int64_t side, int32_t steps, int32_t sqrt_m, int64_t *tile,
                          int64_t *block) {
  if (side < 1 || steps < 1 || (sqrt_m != 8 && sqrt_m != 16 && sqrt_m != 32)) return 0;
  const long long N = stencil_tile(sqrt_m, steps, side);
  if (!N) return 0;
  const long long B = N - 2ll * steps, tpr = (side + B - 1) / B;
  if (tile) *tile = N;
  if (block) *block = B;
  return tpr * tpr;
}

tcu_dft2_plan_t tcu_dft2_plan(int64_t n1, int64_t n2, int64_t batch, int32_t sqrt_m,
                              int32_t precision) {
  int rc;
  arm_alloc_faults();
  tcu_dft2_plan_s *p = make_dft2(n1, n2, batch, sqrt_m, precision, rc);
  g_last_error = rc;
  return p;
}

int tcu_dft2_exec(tcu_dft2_plan_t p, const void *in, void *out, int dir, void *stream) {
  if (!p || (dir != TCU_DFT_FORWARD && dir != TCU_DFT_INVERSE)) return TCU_DFT_ERR_INVALID;
  const size_t bytes = (size_t)(p->batch * p->n1 * p->n2) * sizeof(float2);
  int rc = check_buffers(in, out, bytes);
  if (rc != TCU_DFT_OK) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  const int di = dir_index(dir);
  if (p->general) {
    const NvtxRange range("tcu_dft2 (general)");
    rc = general_dft2(p, in, out, dir, st);
    return rc == TCU_DFT_OK && debug_exec() ? tcu_dft2_check(p, stream) : rc;
  }
  {
    const NvtxRange range("tcu_dft2");
    rc = run_col_pass(p, 0, di, (const float2 *)in, p->scratch, false, nullptr, false, st);
    if (rc == TCU_DFT_OK)
      rc = run_rows(p, di, p->scratch, (float2 *)out, dir == TCU_DFT_INVERSE, st);
  }
  return rc == TCU_DFT_OK && debug_exec() ? tcu_dft2_check(p, stream) : rc;
}

int tcu_conv2_exec(tcu_dft2_plan_t p, const void *in, const void *spectrum, void *out,
                   void *stream) {
  if (!p || !spectrum || ((uintptr_t)spectrum & 15)) return TCU_DFT_ERR_INVALID;
  const size_t bytes = (size_t)(p->batch * p->n1 * p->n2) * sizeof(float2);
  int rc = check_buffers(in, out, bytes);
  if (rc != TCU_DFT_OK) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  const NvtxRange range("tcu_conv2");
  if (p->general) {
    rc = general_conv2(p, in, (const float2 *)spectrum, out, st);
    return rc == TCU_DFT_OK && debug_exec() ? tcu_dft2_check(p, stream) : rc;
  }
  // columns: in -> scratch; rows forward, times the spectrum and inverse on
  // chip: scratch -> scratch (an item reads its rows before writing them);
  // inverse columns with 1/(n1 n2): scratch -> out
  rc = run_col_pass(p, 0, 0, (const float2 *)in, p->scratch, false, nullptr, false, st);
  if (rc != TCU_DFT_OK) return rc;
  GArgs g;
  memset(&g, 0, sizeof(g));
  g.p[0] = dft2_pass(p, p->rows, 0, p->scratch, p->scratch, false, (const float2 *)spectrum, 1);
  g.p[1].tw_stage = p->rows.tw_stage[1];
  g.bimg = p->cimg;
  g.err = p->err;
  const cudaError_t e = launch_rowconv(p, false, g, st);
  if (e != cudaSuccess) return TCU_DFT_ERR_CUDA;
  rc = run_col_pass(p, 0, 1, p->scratch, (float2 *)out, true, nullptr, false, st);
  return rc == TCU_DFT_OK && debug_exec() ? tcu_dft2_check(p, stream) : rc;
}

int tcu_dft2_check(tcu_dft2_plan_t p, void *stream) {
  if (!p) return TCU_DFT_ERR_INVALID;
  if (p->general) {
    int rc = tcu_dft_check(p->rows1d, stream);
    if (rc == TCU_DFT_OK && p->cols1d) rc = tcu_dft_check(p->cols1d, stream);
    if (rc != TCU_DFT_OK) return rc;
  }
  if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return TCU_DFT_ERR_CUDA;
  int flag = 0;
  if (cudaMemcpy(&flag, p->err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
    return TCU_DFT_ERR_CUDA;
  if (flag) cudaMemset(p->err, 0, sizeof(int));
  return word_status(flag);
}

int tcu_dft2_destroy(tcu_dft2_plan_t p) {
  free_dft2(p);
  return TCU_DFT_OK;
}

tcu_stencil_plan_t tcu_stencil_plan(int64_t side, int32_t steps, int32_t sqrt_m,
                                    int32_t precision) {
  g_last_error = TCU_DFT_OK;
  arm_alloc_faults();
  if (side < 1 || steps < 1 ||
      (precision != TCU_DFT_TF32 && precision != TCU_DFT_3XTF32 && !prec_bf16(precision))) {
    g_last_error = TCU_DFT_ERR_INVALID;
    return nullptr;
  }
  const long long N =
      (sqrt_m == 8 || sqrt_m == 16 || sqrt_m == 32) ? stencil_tile(sqrt_m, steps, side) : 0;
  const long long Nw = N ? grid_side(sqrt_m, 2ll * steps + 1) : 0;
  if (!N || !Nw) {
    g_last_error = TCU_DFT_ERR_UNSUPPORTED;
    return nullptr;
  }
  // output blocks of B = N - 2k >= k points a side: the (B + 2k)^2 input
  // window of a block fits the N x N tile without wrapping (Lemma 1 is
  // B = k); the last blocks of a row may be cut; N from stencil_tile
  const int B = (int)(N - 2ll * steps);
  const long long tpr = (side + B - 1) / B;
  tcu_stencil_plan_s *p = new tcu_stencil_plan_s();
  memset(p, 0, sizeof(*p));
  p->side = side;
  p->k = steps;
  p->r = sqrt_m;
  p->precision = precision;
  p->N = N;
  p->Nw = Nw;
  p->B = B;
  p->tiles = tpr * tpr;
  int rc = TCU_DFT_OK;
  int kt = 0;
  is_power_of(N, sqrt_m, kt);
  p->real = precision == TCU_DFT_3XTF32 && kt <= single_pass_stages(sqrt_m);
  p->closed = p->real && steps <= kClosedSteps;
  p->conv = p->real ? make_real_tiles(N, kt, p->tiles, sqrt_m, rc)
                    : make_dft2(N, N, p->tiles, sqrt_m, precision, rc);
  if (rc == TCU_DFT_OK && p->closed) {
    std::vector<double2> roots((size_t)N);
    for (long long f = 0; f < N; ++f)
      roots[f] = make_double2(cos(2.0 * M_PI * f / N), sin(2.0 * M_PI * f / N));
    rc = upload(&p->roots, roots);
  } else if (rc == TCU_DFT_OK) {
    p->wconv = make_dft2(N, N, 1, sqrt_m, precision, rc);
  }
  if (rc == TCU_DFT_OK) p->wpow = make_dft2(Nw, Nw, 1, sqrt_m, precision, rc);
  if (rc == TCU_DFT_OK) {
    p->num_sms = p->conv->num_sms;
    if ((!p->real && dev_malloc((void **)&p->tile_buf,
                                (size_t)(p->tiles * N * N) * sizeof(float2)) != cudaSuccess) ||
        dev_malloc((void **)&p->wgrid, (size_t)(Nw * Nw) * sizeof(float2)) != cudaSuccess ||
        dev_malloc((void **)&p->wker, (size_t)(N * N) * sizeof(float2)) != cudaSuccess) {
      cudaGetLastError();
      rc = TCU_DFT_ERR_OOM;
    }
  }
  if (rc != TCU_DFT_OK) {
    free_stencil(p);
    g_last_error = rc;
    return nullptr;
  }
  return p;
}

// Lemma 2 on the device: P placed on the Nw x Nw grid, its 2-D DFT, the
// pointwise k-th power, the inverse 2-D DFT; W = the centred real part.
static int stencil_weight_grid(tcu_stencil_plan_t p, const float *w3x3, cudaStream_t st) {
  Stencil3 w;
  for (int i = 0; i < 9; ++i) w.w[i] = w3x3[i];
  const long long cnt = p->Nw * p->Nw;
  if (launch_place_poly(p->wgrid, p->Nw, w, p->num_sms, st) != cudaSuccess)
    return TCU_DFT_ERR_CUDA;
  int rc = tcu_dft2_exec(p->wpow, p->wgrid, p->wgrid, TCU_DFT_FORWARD, st);
  if (rc != TCU_DFT_OK) return rc;
  if (launch_cpow(p->wgrid, cnt, p->k, p->num_sms, st) != cudaSuccess) return TCU_DFT_ERR_CUDA;
  return tcu_dft2_exec(p->wpow, p->wgrid, p->wgrid, TCU_DFT_INVERSE, st);
}

int tcu_stencil_weights(tcu_stencil_plan_t p, const float *w3x3, float *W, void *stream) {
  if (!p || !w3x3 || !W) return TCU_DFT_ERR_INVALID;
  cudaStream_t st = (cudaStream_t)stream;
  int rc = stencil_weight_grid(p, w3x3, st);
  if (rc != TCU_DFT_OK) return rc;
  return launch_extract_weights(W, p->wgrid, p->Nw, p->k, p->num_sms, st) == cudaSuccess
             ? TCU_DFT_OK
             : TCU_DFT_ERR_CUDA;
}

int tcu_stencil_exec(tcu_stencil_plan_t p, const float *w3x3, const float *A, float *Ak,
                     void *stream) {
  if (!p || !w3x3 || !A || !Ak) return TCU_DFT_ERR_INVALID;
  const size_t bytes = (size_t)(p->side * p->side) * sizeof(float);
  if (A != Ak && overlaps(A, Ak, bytes)) return TCU_DFT_ERR_INVALID;
  cudaStream_t st = (cudaStream_t)stream;
  const NvtxRange range("tcu_stencil");
  // the spectrum of W': directly, or W (Lemma 2), the kernel and its transform
  int rc = TCU_DFT_OK;
  if (p->closed) {
    Stencil3 w;
    for (int i = 0; i < 9; ++i) w.w[i] = w3x3[i];
    if (launch_stencil_spectrum(p->wker, p->roots, p->N, w, p->k, p->num_sms, st) != cudaSuccess)
      return TCU_DFT_ERR_CUDA;
  } else {
    rc = stencil_weight_grid(p, w3x3, st);
    if (rc != TCU_DFT_OK) return rc;
    if (launch_place_kernel(p->wker, p->N, p->wgrid, p->Nw, p->k, p->num_sms, st) !=
        cudaSuccess)
      return TCU_DFT_ERR_CUDA;
    rc = tcu_dft2_exec(p->wconv, p->wker, p->wker, TCU_DFT_FORWARD, st);
    if (rc != TCU_DFT_OK) return rc;
  }
  if (p->real) {
    rc = run_real_tiles(p, A, Ak, p->wker, st);
    return rc == TCU_DFT_OK && debug_exec() ? tcu_stencil_check(p, stream) : rc;
  }
  // Lemma 1: every block's input window as one batch of tiles, circular
  // convolution, the B x B centres
  if (launch_gather_tiles(p->tile_buf, A, p->side, p->k, p->N, p->B, p->num_sms, st) !=
      cudaSuccess)
    return TCU_DFT_ERR_CUDA;
  rc = tcu_conv2_exec(p->conv, p->tile_buf, p->wker, p->tile_buf, st);
  if (rc != TCU_DFT_OK) return rc;
  if (launch_extract_tiles(Ak, p->tile_buf, p->side, p->k, p->N, p->B, p->num_sms, st) !=
      cudaSuccess)
    return TCU_DFT_ERR_CUDA;
  return debug_exec() ? tcu_stencil_check(p, stream) : TCU_DFT_OK;
}

int tcu_stencil_check(tcu_stencil_plan_t p, void *stream) {
  if (!p) return TCU_DFT_ERR_INVALID;
  int rc = tcu_dft2_check(p->wpow, stream);
  if (rc == TCU_DFT_OK && p->wconv) rc = tcu_dft2_check(p->wconv, stream);
  if (rc == TCU_DFT_OK) rc = tcu_dft2_check(p->conv, stream);
  return rc;
}

int tcu_stencil_destroy(tcu_stencil_plan_t p) {
  free_stencil(p);
  return TCU_DFT_OK;
}

}  // extern "C"
