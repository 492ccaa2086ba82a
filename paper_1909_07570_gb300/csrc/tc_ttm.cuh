// Tensor-core passes over X (tc_ttm.cu): BF16, and FP32-accurate as FP16 pairs or TF32x3.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "common.cuh"

namespace nnc {
namespace tc {

constexpr int kKindBf16 = 0;
constexpr int kKindTf32x3 = 1;
constexpr int kKindF16x3 = 2;

// The device words of a plan (TcPlan::err): a pipeline wait timed out; F16x3 only: an entry of X
// lies outside the range of a pair; rounds that CTAs of passes took beyond the first (tc_ttm.cu).
constexpr int kFlagWideX = 1, kFlagRounds = 2, kFlags = 3;

// Where and how the epilogue writes one pass's FP32 result.
struct TcEpilogue {
  float* out;
  int q;                  // output columns written (m_n)
  // pass X x_3 F3^T: out is rows x q, row r scaled by row_scale[r / rows_per_slice]
  // (row_scale NULL: no scaling)
  int64_t rows;
  int64_t rows_per_slice;
  const float* row_scale;
  // p1_layout 0: out is rows x q, tile row = output row (as above)
  // p1_layout 1 (pass X x_1 F1^T): tile row c = (j, k) of the N2 x kp layout
  //   (kp = padded row length of the operand view); out is q x n2 x n3
  //   (slab = n2 n3)
  // p1_layout 2 (pass X x_1 F1^T): tile row c = (j, k) of the N2 x kp layout;
  //   out has rows (k, j): out[(k n2 + j) q + col]
  int p1_layout;
  int64_t kp, n2, n3, slab;
  // Optional contraction of each tile with the matching rows of a factor F
  // (N2 % 128 == 0, q <= 32, yf_m <= 32). Both passes see tiles of 128 rows
  // (s, j) with j = j0 .. j0 + 127, j0 = 128 (tile % y_nh), y_nh = N2 / 128,
  // s = i (pass X x_3 F3^T) or k (pass X x_1 F1^T with rows (k, j)). The tile
  // writes its share of Y[s] = F^T P[s] (yf_m x q), or of its transpose when
  // y_tr (q x yf_m):
  //   ysh[tile yf_m q + b q + c] = sum_r yf[(j0 + r) yf_m + b] P[(s, j0 + r), c]
  float* ysh;
  const float* yf;
  int yf_m;
  int y_tr;
  int64_t y_nh;
  // FP16 pairs: tile row = (a, b) = (row / kp, row % kp), written when a < ra_n
  // and b < rb_n, times ra_scale[a] rb_scale[b]. x_resident: the pair stays in
  // L2 from pass to pass (no evict-first hint).
  const float *ra_scale, *rb_scale;
  int64_t ra_n, rb_n;
  int x_resident;
};

// Operands and TMA descriptors of the two passes over a 3-way FP32 X.
//   BF16:   a BF16 copy Xb of X (per-slice power-of-two scales, rows padded to a
//           multiple of 64) and BF16 operands Bt1, Bt3 of F^(1), F^(3).
//   TF32x3: X itself for pass 1, a transposed copy Xt (N2 N3 x N1p, i
//           contiguous; rows (j, k), or (k, j) with p1_kj) so that pass 2 is
//           K-major too, and hi / lo TF32 operands B1hi/B1lo, B3hi/B3lo.
//   F16x3:  X as a pair of FP16 copies Xh, Xl (rows padded to a multiple of 8,
//           power-of-two scales s, t, u per slice of modes 1, 2, 3) that both
//           passes read; they form their B operand themselves (tc_ttm.cu).
// B operands are [np x k] row-major, zero outside the factor.
struct TcPlan {
  int kind = kKindBf16;
  // Layout of the pass-2 result: false: m1 x N2 x N3; true: rows (k, j),
  // (N3 N2) x m1 (the nnTD sweep's layout).
  bool p1_kj = false;
  int64_t N1 = 0, N2 = 0, N3 = 0;
  int m1 = 0, m3 = 0, kp1 = 0, kp3 = 0, kb3 = 0, np1 = 0, np3 = 0;
  __nv_bfloat16 *Xb = nullptr, *Bt1 = nullptr, *Bt3 = nullptr;
  float *B1hi = nullptr, *B1lo = nullptr, *B3hi = nullptr, *B3lo = nullptr, *Xt = nullptr;
  float *scale = nullptr, *inv_scale = nullptr;
  __half *Xh = nullptr, *Xl = nullptr;
  float *sc_t = nullptr, *sc_u = nullptr;  // F16x3: t and u (s is in `scale`)
  // Bits of the largest magnitude of every row (i, j); another plan's for the same X
  // may be handed in before init.
  unsigned* rmax = nullptr;
  int x_resident = 0;
  CUtensorMap mapL3, mapL1;  // F16x3: Xl as operand A of pass 1 and pass 2
  int* err = nullptr;  // F16x3: kFlags entries, else one
  // SMs a pass of at least 8 tiles per SM (F16x3: of any number) leaves to
  // kernels that run beside it (the nnTD sweep's small kernels); 0: every SM.
  int reserve_sms = 0;
  CUtensorMap mapA3, mapB3, mapB3lo, mapA1, mapB1, mapB1lo;

  // Builds the operand buffers (BF16: Xb and the scales) from X, stream-ordered.
  // UNSUPPORTED when the shape is outside the path (m_n > 64; TF32x3 also
  // needs N3 % 4 == 0 for its TMA row strides).
  // need_p1 = false: pass1 will not be called (TF32x3 then makes no copy of X).
  int init(int kind, const float* X, int64_t N1, int64_t N2, int64_t N3, int m1, int m3,
           Scratch& sc, cudaStream_t s, bool p1_kj = false, bool need_p1 = true);
  // FP32-accurate passes that a fit runs again and again: F16x3 where the shape
  // allows it, else TF32x3. Whether the values of X allow it the device knows after init
  // (PairGuard::wide, check: an entry outside the range of a pair, whose results are then
  // not FP32-accurate): the caller then turns the plan into the TF32x3 one.
  int init_fp32(const float* X, int64_t N1, int64_t N2, int64_t N3, int m1, int m3, Scratch& sc,
                cudaStream_t s, bool p1_kj = false);
  // An F16x3 plan becomes the TF32x3 plan of the same tensor; no work that reads the pair
  // is in flight but on `s`.
  int to_tf32(const float* X, Scratch& sc, cudaStream_t s);
  int init_f16(const float* X, Scratch& sc, cudaStream_t s);  // parts of init
  int row_maxima(const float* X, Scratch& sc, cudaStream_t s);
  // B operands from the current factor (BF16: F^(1) scaled by s).
  int convert_b3(const float* F3, cudaStream_t s) const;
  int convert_b1(const float* F1, cudaStream_t s) const;
  // P3 = X x_3 F3^T ((N1 N2) x m3, FP32); convert first builds the B operand.
  // With Y1 (y1_fusable(m2) only) the pass also writes the per-tile shares of
  // Y1[i] = F2^T P3[i, :, :] (m2 x m3 each; see TcEpilogue::ysh).
  int pass3(const float* F3, float* P3, cudaStream_t s, bool convert = true,
            const float* F2 = nullptr, int m2 = 0, float* Y1 = nullptr) const;
  bool y1_fusable(int m2) const;
  // P1 = X x_1 F1^T (FP32; m1 x N2 x N3, or rows (k, j) with p1_kj).
  // With Y3 (y3_fusable(m2) only: TF32x3 with p1_kj) the pass also writes the
  // per-tile shares of Y3[k] = P1[k, :, :]^T F2 (m1 x m2 each).
  int pass1(const float* F1, float* P1, cudaStream_t s, bool convert = true,
            const float* F2 = nullptr, int m2 = 0, float* Y3 = nullptr) const;
  bool y3_fusable(int m2) const;
  // Synchronises s and turns a device-side pipeline time-out into NNC_ERR_TIMEOUT.
  // *wide (F16x3): X has an entry outside the pairs' range.
  int check(cudaStream_t s, bool* wide = nullptr) const;
};

// Watches a fit whose passes read FP16 pairs: once some CTA took another round for wide factors
// in every fourth pass (as far as the sum of rounds says) since the last look, the fit does
// better with TF32x3 passes (at 512^3 a round takes 100-120 us, a TF32x3 pass 140). A look is of
// the first sweeps, then of 20 more, then of a quarter of those done; it comes once the next sweeps
// are queued, so that the device does not wait; what it sees is as of its mark, so it depends
// on the data alone.
struct PairGuard {
  bool slow = false;  // at the last look
  PairGuard() = default;
  PairGuard(const PairGuard&) = delete;
  PairGuard& operator=(const PairGuard&) = delete;
  ~PairGuard();
  // Right after the plan's init on `s`; the first look is of `first` sweeps.
  int start(const TcPlan* p, int first, cudaStream_t s);
  // Whether X has an entry outside the pairs' range (waits for the init alone).
  int wide(cudaStream_t s, bool* w);
  // After every launch on `cs`, with `t` sweeps queued: marks, or looks, when that is due
  // (NNC_ERR_TIMEOUT as TcPlan::check).
  int step(cudaStream_t cs, int t);

 private:
  const TcPlan* plan = nullptr;
  int next = 0, marked = 0, looked = 0, rounds = 0;
  bool pending = false;
  int* slot = nullptr;
  cudaEvent_t at = nullptr;
};

// Runs the pass kernel's bounded mbarrier wait once, with a limit of `cycles`,
// on a barrier that never completes: NNC_ERR_TIMEOUT when it gives up (the
// expected outcome), NNC_OK if it did not.
int wait_selftest(long long cycles, cudaStream_t s);

}  // namespace tc
}  // namespace nnc
