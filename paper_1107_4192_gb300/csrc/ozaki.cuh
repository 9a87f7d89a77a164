// Exact-slice products on the tensor cores: float64-accurate C = A B^T from
// bf16 tcgen05 MMAs (the splitting scheme of Ozaki et al. 2012, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication and its applications", with the exponent-aligned integer
// slices of Mukunoki, Ozaki, Ogita and Imamura 2020, "DGEMM using Tensor Cores,
// and Its Accurate and Reproducible Versions").
//
// Row r of an operand X (rows x K) is written as
//     X[r][k] ~= 2^(e_r - 7) * sum_{p < S} 2^(-8p) q_p[r][k]
// with e_r the exponent of the row's largest magnitude (max |X[r][:]| < 2^e_r)
// and integer slices q_p in [-128, 128], each exact in bf16: the signed
// base-256 digits (each rounded to nearest, ties to even) of X[r][k] rounded
// to the grid 2^(e_r - 7 - 8(S-1)).  A product of two
// slices is an integer below 2^14, so the sum over k of the products of one
// slice level l = p_A + p_B is an exact integer as long as it stays below 2^24:
// the tensor cores' float32 accumulation (which truncates) then loses nothing.
// The products with l < L are kept (L(L+1)/2 slice pairs); the dropped levels
// and the slices' own truncation leave an error in element (i, j) of about
// 2^(-8L+3) K 2^(e_i + e_j) (per term, 2^(-8L+3) of the row maxima's product):
// 2^-37 for L = 5, 2^-53 for L = 7.
#pragma once

#include "tc_gemm.cuh"

namespace kfm {

// Slices of a rows x cols operand: S planes of rows_pad x ldk bf16 (plane p at
// planes + p * rows_pad * ldk; rows >= rows and columns >= cols are zero) and
// the per-row exponents e_r (rows_pad ints, 0 for zero rows).
struct OzSlices {
  __nv_bfloat16* planes = nullptr;
  int* exps = nullptr;
  int64_t rows = 0, rows_pad = 0, ldk = 0;
  int S = 0;       // planes the memory holds
  int filled = 0;  // planes the last oz_slice wrote
};

// Bytes of the planes and exponents for rows x cols with S slices.
uint64_t oz_slice_bytes(int64_t rows, int64_t cols, int S);
// Points `out` at memory of oz_slice_bytes(rows, cols, S) bytes.
void oz_slice_layout(OzSlices& out, void* mem, int64_t rows, int64_t cols, int S);

// Fills `out` (laid out by oz_slice_layout for at least these rows, cols and
// S slices) from X (float64 when f64, else float32; rows x cols, leading
// dimension ld, row-major).  A row that holds an infinity or NaN gets zero slices and a
// marked exponent, from which the product's row or column becomes NaN.
kf_status oz_slice(cudaStream_t s, const void* X, int64_t ld, int f64, int64_t rows, int64_t cols, int S,
                   OzSlices& out);

// The refined inverse's slices, balanced by s_i = -round(log2(P_ii) / 2) per row and column of P (scale[i], from
// oz_balance, zero from n to the slices' ldk; 16-byte aligned; P float32 or float64).
kf_status oz_balance(cudaStream_t s, const void* P, int64_t ld, int f64, int64_t n, int64_t ldk, int* scale);

// S slices of the rows of the n x n X[r][k] 2^(sign scale[k]).  Their products with slices weighed by the opposite sign
// are X's own.
kf_status oz_slice_weighed(cudaStream_t s, const void* X, int64_t ld, int f64, int64_t n, const int* scale, int sign, int S,
                           OzSlices& out);

// A symmetric n x n float32 X (16-byte aligned, ld a multiple of 4) rounded in place so that it stays symmetric and
// three slices of its rows weighed by 2^(-scale[k]) hold it exactly (each element of the balanced matrix to 2^-24 of
// the larger of its two row maxima), and those slices.
kf_status oz_slice_symmetric(cudaStream_t s, float* X, int64_t ld, int64_t n, const int* scale, OzSlices& out);

// Two slices of the rows of a float32 C weighed by 2^(-scale[k]) (2^-16 of the row maxima), and X = Y + Cs in float64
// (Y float32, both n x n with leading dimension ld as above) for the Cs that they hold.
kf_status oz_slice_correction(cudaStream_t s, const float* C, const float* Y, int64_t ld, int64_t n, const int* scale,
                              double* X, int64_t ldx, OzSlices& out);

// Epilogue of the exact-slice product, float64.  With acc = (A B^T)[i][j]:
//   v = alpha acc + beta cin[i][j] + (i == j ? delta : 0) + Radd[i][j]
//   out[i][j] = v,  outf[i][j] = (float) v,  outT[j][i] = v,
//   out2[i][j] = v + Q[i][j],  diag_out[i] = v at i == j
// (each optional; Radd per radd_kind and Q per q_kind as kf_cov_kind, < 0 =
// none).  check_diag: a diagonal v that is not finite and > 0 raises
// KF_ERR_NUMERIC at `step`.  sym (M == N): only i >= j is computed and out,
// outf and out2 are mirrored to (j, i), so they come out exactly symmetric.
struct OzEpilogue {
  double alpha = 1.0, beta = 0.0, delta = 0.0;
  const double* cin = nullptr;
  int64_t ldcin = 0;
  double* out = nullptr;
  int64_t ldo = 0;
  float* outf = nullptr;
  int64_t ldof = 0;
  double* outT = nullptr;
  int64_t ldoT = 0;
  double* out2 = nullptr;
  int64_t ldo2 = 0;
  int q_kind = -1;
  const double* q = nullptr;
  int64_t ldq = 0;
  int radd_kind = -1;
  const double* radd = nullptr;
  int64_t ldradd = 0;
  double* diag_out = nullptr;
  int check_diag = 0;
  int sym = 0;
  int* status = nullptr;  // KF_ERR_TIMEOUT on an expired wait; kernels skip when already failed
  int step = 0;
  // set by oz_gemm: alpha is 1 or -1 (else 0), beta is 1; the epilogue's usual forms (1: away from the diagonal)
  int alpha_unit = 0, beta_unit = 0, simple = 0;
};

// Optional event timing of the exact-slice kernel launches alone (installed by a plan while it
// profiles the smoother-gain refinement).
extern thread_local TcLaunchTimer* g_oz_timer;

// C = A B^T for A (M x K) and B (N x K) given by their slices, keeping the
// slice levels l < levels (4 to 7; B needs at least `levels` slices, A as
// many or a_slices).  K <= 2^20.  splits > 1 divides K among that many CTAs per output
// tile, whose float64 partial sums (splits x M x N doubles at `partials`) are
// added in a fixed order by a second kernel that applies the epilogue.
//
// work (five levels, splits == 1, plain out / outT / cin epilogues): products with too few tiles for the GPU
// and a long K are split too, into 64-bit integer sums (M x N rounded up to 64 per split) that a second kernel
// adds; integers, so the result is bit for bit the unsplit one.
// a_slices > 0: A has only that many slices (its other slices are zero by construction), and only their
// products are formed.
struct OzSums {
  long long* p = nullptr;
  int64_t count = 0;
};
constexpr int kOzSumsMaxK = 1 << 15;
int64_t oz_sums_splits(int64_t M, int64_t N, int64_t K);  // the splits such a product gets (1: none)
kf_status oz_gemm(cudaStream_t s, const OzSlices& A, const OzSlices& B, int M, int N, int K, int levels,
                  const OzEpilogue& e, int splits = 1, double* partials = nullptr, const OzSums& work = OzSums{},
                  int a_slices = 0);

}  // namespace kfm
