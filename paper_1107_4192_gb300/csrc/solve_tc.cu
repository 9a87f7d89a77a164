// Smoother-gain solve on the tensor cores (mixed mode, float32-class solve).
//
// J_t = P_{t|t} F^T P_{t+1|t}^{-1} (eqn 11) is formed as
//   P_{t+1|t} = L L^T,   W = L^{-1},   J_t = ((P_{t|t} F^T) W^T) W,
// so that, apart from the diagonal blocks, all O(N^3) work is large
// products that run as three-way split-bf16 GEMMs (six bf16 products with
// float32 accumulation, float32-class accuracy) on the tensor cores:
//  - Cholesky, recursive on halves:  L11 = chol(A11);  L21 = A21 W11^T;
//    A22 <- A22 - L21 L21^T;  L22 = chol(A22);
//  - triangular inverse on the same halves: W21 = -W22 (L21 W11);
//  - the diagonal blocks (up to kDirectMax rows) are factored and inverted by one launch each (chol_direct.cu).
// Products with a triangular operand skip the k-tiles outside its band.
// This replaces the two triangular solves with N right-hand sides by a
// triangular inverse and two triangular products (2.67 N^3 instead of
// 2.33 N^3 flops), in exchange for large, fully parallel products only.
// With F = I and a scalar or diagonal Q the gain needs no product with
// P_{t|t} at all: J_t = P_{t|t} (P_{t|t} + Q)^{-1} = I - Q P_{t+1|t}^{-1}, and
// P_{t+1|t}^{-1} = W^T W costs N^3 / 3 and the gain is formed in the product's
// epilogue (gain_identity_tc).
#include <set>
#include <utility>

#include "solve_tc.cuh"

namespace kfm {

namespace {

struct Ctx {
  cudaStream_t s;
  TcScratch* sc;
  int* status;
  int step;
  float* L;
  int64_t ldl;
  float* W;
  int64_t ldw;
  float* T;
  int64_t ldt;
  int nb;
  std::set<std::pair<int, int>> done;
};

int split_point(int n, int nb) { return (int)round_up((n + 1) / 2, nb); }

kf_status gemm(Ctx& c, const GemmParams<float>& g, bool transB) {
  // both operands are split into scratch first, so in place is safe
  return tc_gemm_split(c.s, *c.sc, g, 3, transB);
}

// Matrices up to this size are factored and inverted by one launch (chol_direct.cu); above it the products
// between the halves are large enough for the tensor cores.  Whole smoothing calls with the line at 1024 / 1536 /
// 2048: N = 1501 8.71 / 8.38 / 8.38 ms, N = 2048 12.17 / 12.12 / 13.54 ms, N = 5124 (leaves of 1281) 22.7 / 21.6 /
// 21.6 ms, N = 8196 (leaves of 1025) 134.8 / 134.4 / 136.2 ms.
constexpr int kDirectMax = 1536;
static_assert(kDirectMax <= kCholDirectMaxN, "leaf size");

kf_status trtri_rec(Ctx& c, int off, int n) {
  if (c.done.count({off, n})) return KF_OK;
  if (n <= kDirectMax) return KF_ERR_ARG;  // leaves come from potrf_rec
  const int n1 = split_point(n, c.nb), n2 = n - n1;
  KF_TRY(trtri_rec(c, off, n1));
  KF_TRY(trtri_rec(c, off + n1, n2));
  // T = L21 W11   (n2 x n1; op(B) = W11^T has row j zero for k < j)
  GemmParams<float> a;
  a.M = n2; a.N = n1; a.K = n1;
  a.A = c.L + (int64_t)(off + n1) * c.ldl + off; a.lda = c.ldl;
  a.B = c.W + (int64_t)off * c.ldw + off; a.ldb = c.ldw;
  a.tri_b = -1;
  a.out = c.T; a.ldo = c.ldt;
  a.status = c.status;
  KF_TRY(gemm(c, a, false));
  // W21 = -W22 T   (W22 lower triangular)
  GemmParams<float> b;
  b.M = n2; b.N = n1; b.K = n2;
  b.A = c.W + (int64_t)(off + n1) * c.ldw + off + n1; b.lda = c.ldw;
  b.tri_a = 1;
  b.B = c.T; b.ldb = c.ldt;
  b.alpha = -1.0f;
  b.out = c.W + (int64_t)(off + n1) * c.ldw + off; b.ldo = c.ldw;
  b.status = c.status;
  KF_TRY(gemm(c, b, false));
  c.done.insert({off, n});
  return KF_OK;
}

kf_status potrf_rec(Ctx& c, int off, int n) {
  if (n <= kDirectMax) {
    KF_TRY(chol_inverse_direct(c.s, n, c.L + (int64_t)off * c.ldl + off, c.ldl, c.W + (int64_t)off * c.ldw + off,
                               c.ldw, c.sc->a[0], c.status, c.step, off));
    c.done.insert({off, n});
    return KF_OK;
  }
  const int n1 = split_point(n, c.nb), n2 = n - n1;
  KF_TRY(potrf_rec(c, off, n1));
  KF_TRY(trtri_rec(c, off, n1));
  float* A21 = c.L + (int64_t)(off + n1) * c.ldl + off;
  // L21 = A21 W11^T  (row j of W11 is zero for k > j)
  GemmParams<float> p;
  p.M = n2; p.N = n1; p.K = n1;
  p.A = A21; p.lda = c.ldl;
  p.B = c.W + (int64_t)off * c.ldw + off; p.ldb = c.ldw;
  p.tri_b = 1;
  p.out = A21; p.ldo = c.ldl;
  p.status = c.status;
  KF_TRY(gemm(c, p, true));
  // A22 <- A22 - L21 L21^T on the lower triangle
  GemmParams<float> u;
  u.M = n2; u.N = n2; u.K = n1;
  u.A = A21; u.lda = c.ldl;
  u.B = A21; u.ldb = c.ldl;
  u.alpha = -1.0f;
  u.cin = c.L + (int64_t)(off + n1) * c.ldl + off + n1; u.ldcin = c.ldl; u.beta = 1.0f;
  u.out = c.L + (int64_t)(off + n1) * c.ldl + off + n1; u.ldo = c.ldl;
  u.sym = 2;
  u.status = c.status;
  KF_TRY(gemm(c, u, true));
  return potrf_rec(c, off + n1, n2);
}

}  // namespace

kf_status chol_inverse_tc(cudaStream_t s, TcScratch& sc, int n, float* L, int64_t ldl, float* W, int64_t ldw,
                          float* T, int64_t ldt, int* status, int step) {
  Ctx c{s, &sc, status, step, L, ldl, W, ldw, T, ldt, 128, {}};
  KF_TRY(potrf_rec(c, 0, n));
  if (n > c.nb) KF_TRY(trtri_rec(c, 0, n));
  return KF_OK;
}

kf_status gain_from_inverse_tc(cudaStream_t s, TcScratch& sc, int n, const float* Bm, int64_t ldb, const float* W,
                               int64_t ldw, float* Z, int64_t ldz, float* J, int64_t ldj, int* status) {
  GemmParams<float> a;  // Z = Bm W^T  (row j of W zero for k > j)
  a.M = n; a.N = n; a.K = n;
  a.A = Bm; a.lda = ldb;
  a.B = W; a.ldb = ldw;
  a.tri_b = 1;
  a.out = Z; a.ldo = ldz;
  a.status = status;
  KF_TRY(tc_gemm_split(s, sc, a, 3, true));
  GemmParams<float> b;  // J = Z W   (op(B) = W^T, row j zero for k < j)
  b.M = n; b.N = n; b.K = n;
  b.A = Z; b.lda = ldz;
  b.B = W; b.ldb = ldw;
  b.tri_b = -1;
  b.out = J; b.ldo = ldj;
  b.status = status;
  return tc_gemm_split(s, sc, b, 3, false);
}

kf_status gain_identity_tc(cudaStream_t s, TcScratch& sc, int n, const float* W, int64_t ldw, int q_kind,
                           const double* q, float* J, int64_t ldj, int* status) {
  if (q_kind != 0 && q_kind != 1) return KF_ERR_ARG;
  GemmParams<float> g;  // J = I - Q (W^T W): lower triangle computed, the upper one mirrored with q_j
  g.M = n; g.N = n; g.K = n;
  g.out = J; g.ldo = ldj;
  g.gain_q = q;
  g.gain_q_kind = q_kind;
  g.sym = 1;
  g.tri_a = -1;  // row r of W^T is zero for k < r
  g.tri_b = -1;
  g.status = status;
  return tc_gemm_ops(s, sc, TcOperand{W, ldw, 0, 1}, TcOperand{W, ldw, 0, 1}, g, 3);
}

uint64_t refine_bytes(int64_t n, int64_t ld) {
  const uint64_t mat = round_up((int64_t)(n * ld * 8), 256);
  return 3 * mat + 2 * round_up((int64_t)oz_slice_bytes(n, n, 7), 256);
}

void refine_layout(RefineBufs& rb, void* mem, int64_t n, int64_t ld) {
  const uint64_t mat = round_up((int64_t)(n * ld * 8), 256);
  char* p = static_cast<char*>(mem);
  rb.X0 = reinterpret_cast<double*>(p);
  rb.R = reinterpret_cast<double*>(p + mat);
  rb.X1 = reinterpret_cast<double*>(p + 2 * mat);
  rb.ld = ld;
  oz_slice_layout(rb.Ps, p + 3 * mat, n, n, 7);
  // room for seven slices, of which three are used; the balancing exponents lie behind them
  char* xs = p + 3 * mat + round_up((int64_t)oz_slice_bytes(n, n, 7), 256);
  oz_slice_layout(rb.Xs, xs, n, n, 3);
  rb.scale = reinterpret_cast<int*>(xs + round_up((int64_t)oz_slice_bytes(n, n, 3), 256));
}

kf_status refine_inverse_tc(cudaStream_t s, TcScratch& sc, int n, const void* P, int p_f64, int64_t ldp, const float* W,
                            int64_t ldw, RefineBufs& rb, int q_kind, const double* gain_q, double* J64, float* Jf,
                            int64_t ldj, double* X2, int64_t ldx, int* status, int step) {
  if (gain_q && q_kind != 0 && q_kind != 1) return KF_ERR_ARG;
  const int64_t ld = rb.ld;
  float* Y = reinterpret_cast<float*>(rb.X0);  // X_0, then its rounding Y_0
  float* C = Y + n * ld;
  double *E = rb.R, *X1 = rb.X1;
  {
    GemmParams<float> g;  // X_0 = W^T W (lower triangle + mirror; row r of W^T is zero for k < r)
    g.M = n; g.N = n; g.K = n;
    g.out = Y; g.ldo = ld;
    g.sym = 1;
    g.tri_a = -1;
    g.tri_b = -1;
    g.status = status;
    KF_TRY(tc_gemm_ops(s, sc, TcOperand{W, ldw, 0, 1}, TcOperand{W, ldw, 0, 1}, g, 3));
  }
  KF_TRY(oz_balance(s, P, ldp, p_f64, n, rb.Ps.ldk, rb.scale));
  KF_TRY(oz_slice_weighed(s, P, ldp, p_f64, n, rb.scale, 1, 7, rb.Ps));
  KF_TRY(oz_slice_symmetric(s, Y, ld, n, rb.scale, rb.Xs));
  {
    OzEpilogue e;  // E_0 = I - Y_0 P (P symmetric: its rows are the product's columns)
    e.alpha = -1.0;
    e.delta = 1.0;
    e.out = E; e.ldo = ld;
    e.status = status;
    e.step = step;
    KF_TRY(oz_gemm(s, rb.Xs, rb.Ps, n, n, n, 7, e, 1, nullptr, OzSums{}, 3));
  }
  {
    GemmParams<float> g;  // C = E_0 Y_0, symmetric
    g.M = n; g.N = n; g.K = n;
    g.out = C; g.ldo = ld;
    g.sym = 1;
    g.status = status;
    g.step = step;
    KF_TRY(tc_gemm_ops(s, sc, TcOperand{E, ld, 1, 0}, TcOperand{Y, ld, 0, 0}, g, 2));
  }
  KF_TRY(oz_slice_correction(s, C, Y, ld, n, rb.scale, X1, ld, rb.Xs));
  {
    OzEpilogue e;  // E_1 = I - X_1 P = E_0 - C_s P
    e.alpha = -1.0;
    e.cin = E; e.ldcin = ld; e.beta = 1.0;
    e.out = E; e.ldo = ld;
    e.status = status;
    e.step = step;
    KF_TRY(oz_gemm(s, rb.Xs, rb.Ps, n, n, n, 5, e, 1, nullptr, OzSums{}, 2));
  }
  // X_2 = X_1 + E_1 X_1: the correction is ~1e-9 of X, so two bf16 slices (16 bits) leave it accurate to
  // ~1e-14 of X, and the asymmetry of X_1 (~1e-10) does not matter in it
  GemmParams<double> g;
  g.M = n; g.N = n; g.K = n;
  g.cin = X1; g.ldcin = ld; g.beta = 1.0;
  g.sym = 1;
  g.status = status;
  g.step = step;
  if (gain_q) {
    g.gain_q = gain_q; g.gain_q_kind = q_kind;
    g.out = J64; g.ldo = ldj;
    g.outf = Jf; g.ldof = ldj;
  } else {
    g.out = X2; g.ldo = ldx;
  }
  return tc_gemm_ops(s, sc, TcOperand{E, ld, 1, 0}, TcOperand{X1, ld, 1, 0}, g, 2);
}

}  // namespace kfm
