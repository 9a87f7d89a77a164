// Tensor-core smoother-gain solve (mixed mode with float32 solve).
#pragma once

#include "ozaki.cuh"
#include "tc_gemm.cuh"

namespace kfm {

// In place: L (n x n, lower triangle used) <- chol(L); W <- L^{-1} (lower, the
// strict upper triangle of W must be zero on entry and stays zero).  T is
// scratch of at least n x n.  A non-positive pivot sets KF_ERR_NOT_PD (step).
kf_status chol_inverse_tc(cudaStream_t s, TcScratch& sc, int n, float* L, int64_t ldl, float* W, int64_t ldw,
                          float* T, int64_t ldt, int* status, int step);

// J = (Bm W^T) W for W = L^{-1} from chol_inverse_tc, i.e. J = Bm (L L^T)^{-1};
// Z is n x n scratch.
kf_status gain_from_inverse_tc(cudaStream_t s, TcScratch& sc, int n, const float* Bm, int64_t ldb, const float* W,
                               int64_t ldw, float* Z, int64_t ldz, float* J, int64_t ldj, int* status);

// F = I with Q = q I or diagonal: J = P_{t|t} (P_{t|t} + Q)^{-1} = I - Q P_{t+1|t}^{-1},
// with P_{t+1|t}^{-1} = W^T W formed on the lower triangle (n^3 / 3 instead of
// the 2 n^3 of the two triangular products); J is written by that product's
// epilogue, so P_{t+1|t}^{-1} itself is never stored.
kf_status gain_identity_tc(cudaStream_t s, TcScratch& sc, int n, const float* W, int64_t ldw, int q_kind,
                           const double* q, float* J, int64_t ldj, int* status);

// Buffers of refine_inverse_tc: three n x ld float64 matrices (the first holds the float32 Y_0 and C), the
// slices of P (7) and of the iterate (3, then 2), and the balancing exponents.
struct RefineBufs {
  double *X0 = nullptr, *R = nullptr, *X1 = nullptr;
  int64_t ld = 0;
  OzSlices Ps, Xs;
  int* scale = nullptr;
};
uint64_t refine_bytes(int64_t n, int64_t ld);
void refine_layout(RefineBufs& rb, void* mem, int64_t n, int64_t ld);

// Inverse of the symmetric positive definite P (float32, or float64 when p_f64; n x n) to float64
// accuracy, from W = L^{-1} of its float32-class factor (chol_inverse_tc): Newton's iteration, each residual
// I - X_k P exact to 2^-51 of the row maxima,
//   Y_0 = W^T W rounded to 24 bits below its row maxima;   E_0 = I - Y_0 P;
//   X_1 = Y_0 + C_s, C_s = E_0 Y_0 rounded to 16 bits;     E_1 = I - X_1 P = E_0 - C_s P;
//   X_2 = X_1 + E_1 X_1.
// The iterates are rounded so that few slices hold them exactly, and the second residual updates the
// first: 18 slice products (3 slices of Y_0 against 7 of P, levels below 7) and 9 (2 of C_s against 5,
// levels below 5), where separate residuals of unrounded iterates took 15 + 28 (N = 8196: 19.6 + 27.9 ms;
// now 15.8 + 9.4 ms).  Row maxima are those of the balanced matrices D P D and D^{-1} X D^{-1} (D_i a power of
// two near P_ii^(-1/2)): without that, small rows lose to the rounding of large ones (variances spread over
// 1e6 and 1e10: errors of 2e-11 and 1e-6 relative to sqrt(X_ii X_jj), as accurate as without the spread now).
// The corrections are split-bf16 products (symmetric: lower triangle + mirror).
// The last correction is fused into its consumer:
//  - gain_q != NULL (F = I, Q = q I or diagonal): J = I - Q X_2 into J64
//    (float64) and Jf (float32), X_2 itself never stored;
//  - gain_q == NULL: X_2 into X2 (float64, n x ldx; may be rb.X0).
kf_status refine_inverse_tc(cudaStream_t s, TcScratch& sc, int n, const void* P, int p_f64, int64_t ldp, const float* W,
                            int64_t ldw, RefineBufs& rb, int q_kind, const double* gain_q, double* J64, float* Jf,
                            int64_t ldj, double* X2, int64_t ldx, int* status, int step);

}  // namespace kfm
