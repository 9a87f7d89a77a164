// Minimum-norm estimate, eqn 5:  X[t] = lambda C H^T (lambda H C H^T + R)^{-1} y_t
// for all T rows of Y at once, at float64 accuracy.  G = lambda H C H^T + R is
// factored like S_t; W = Y G^{-1} is two triangular products with the factor's
// inverse; X = lambda W H C is one product (plus a column scaling when C is
// diagonal).
//
// mne_init: the paper's initialisation from these estimates (Sec. 2.4):
// x0 = X[0] and Q = the sample covariance of the differences X[k+1] - X[k].
#include "ops.cuh"
#include "ozaki.cuh"

using namespace kfm;

namespace {

__global__ void scale_cols_kernel(int64_t rows, int64_t cols, double* X, int64_t ldx, int c_kind, const double* c,
                                  double lam) {
  for (int64_t i = blockIdx.y; i < rows; i += gridDim.y)
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < cols; j += (int64_t)gridDim.x * blockDim.x) {
      double w = c_kind == 0 ? c[0] : c[j];
      X[i * ldx + j] *= lam * w;
    }
}

// A = H |C|^(1/2) and B = H sign(C) |C|^(1/2) for scalar or diagonal C, so that H C H^T = A B^T with each
// row's largest term bounded by its diagonal element: slices relative to the row maxima then lose nothing
// that matters, however differently the columns (sources) are scaled.
__global__ void weigh_cols_kernel(int64_t rows, int64_t cols, const double* H, int c_kind, const double* c, double* A,
                                  double* B) {
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < cols; j += (int64_t)gridDim.x * blockDim.x) {
    const double w = c_kind == 0 ? c[0] : c[j];
    const double r = sqrt(fabs(w));  // once per column: a float64 square root takes as long as ten products
    const long long flip = w < 0.0 ? 1ll << 63 : 0ll;
    for (int64_t i = blockIdx.y; i < rows; i += gridDim.y) {
      const double a = H[i * cols + j] * r;
      A[i * cols + j] = a;
      B[i * cols + j] = __longlong_as_double(__double_as_longlong(a) ^ flip);
    }
  }
}

// scale[k] = 2^e, the power of two at the largest magnitude of row k of X (1 for a zero or non-finite row).
__global__ void __launch_bounds__(256) row_scale_kernel(int64_t cols, const double* X, double* scale) {
  __shared__ unsigned long long red[8];
  const double* row = X + blockIdx.x * cols;
  unsigned long long mx = 0;
  for (int64_t j = threadIdx.x; j < cols; j += 256)
    mx = max(mx, (unsigned long long)__double_as_longlong(row[j]) & 0x7fffffffffffffffull);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) mx = max(mx, red[w]);
    const unsigned long long E = mx >> 52;
    scale[blockIdx.x] = E >= 1 && E <= 2044 ? __longlong_as_double((long long)(E << 52)) : 1.0;
  }
}

// dst[j][k] = src[k][j] / scale[k] for an m x N src (powers of two: exact).
__global__ void transpose_balanced_kernel(int64_t m, int64_t N, const double* src, const double* scale, double* dst) {
  __shared__ double tile[32][33];
  const int64_t k0 = blockIdx.y * 32, j0 = blockIdx.x * 32;
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int64_t k = k0 + i, j = j0 + threadIdx.x;
    tile[i][threadIdx.x] = k < m && j < N ? src[k * N + j] * (1.0 / scale[k]) : 0.0;
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int64_t j = j0 + i, k = k0 + threadIdx.x;
    if (j < N && k < m) dst[j * m + k] = tile[threadIdx.x][i];
  }
}

// X[t][j] again in float64 where the slices may hold it badly.  Their error is absolute, about 2^-52 of the product
// of the two row maxima (2^exw[t] and 2^exh[j]); an element far below that product (a source that only weakly
// weighted sensors see, a sample that is large in other sensors) would lose its digits.  Elements below 2^-6 of it are
// summed again from the same operands, so each is good to 2^-46 or float64's own rounding.  With Gaussian data these are
// one in a hundred (N = 5124, m = 306, T = 200: 24 us; eight loads ahead of the sum's chain changed nothing).
__global__ void __launch_bounds__(256) small_elements_kernel(int64_t T, int64_t N, int64_t m, const double* W,
                                                             const double* HCt, const int* exw, const int* exh, double lambda,
                                                             double* X, const int* status) {
  if (status_failed(status)) return;
  const int lane = threadIdx.x % 32;
  const int64_t j0 = blockIdx.x * 256 + threadIdx.x / 32 * 32, j = j0 + lane;
  const int limit = (j < N ? exh[j] : 0) + (((__double2hiint(lambda) >> 20) & 0x7ff) - 1022) - 6;
  for (int64_t t = blockIdx.y; t < T; t += gridDim.y) {
    bool again = false;
    if (j < N) {
      const int E = (__double2hiint(X[t * N + j]) >> 20) & 0x7ff;  // the exponent is E - 1022
      again = E == 0x7ff || E - 1022 < exw[t] + limit;
    }
    for (unsigned mask = __ballot_sync(0xffffffffu, again); mask; mask &= mask - 1) {
      const int64_t jj = j0 + __ffs(mask) - 1;
      double acc = 0.0;
      for (int64_t k = lane; k < m; k += 32) acc = fma(W[t * m + k], HCt[jj * m + k], acc);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane == 0) X[t * N + jj] = lambda * acc;
    }
  }
}

// One device allocation per call, handed out in 256-byte aligned pieces (cudaMalloc and cudaFree, which
// synchronises, cost more than most of the kernels here).
struct Tmp {
  char* base = nullptr;
  size_t used = 0, size = 0;
  ~Tmp() { cudaFree(base); }
  static size_t pad(size_t bytes) { return (bytes + 255) / 256 * 256; }
  kf_status reserve(size_t bytes) {
    size = bytes;
    if (cudaMalloc((void**)&base, bytes) != cudaSuccess) {
      cudaGetLastError();
      base = nullptr;
      return KF_ERR_CUDA;
    }
    return KF_OK;
  }
  void* take(size_t bytes) {
    char* p = base + used;
    used += pad(bytes);
    return used <= size ? p : nullptr;
  }
  double* doubles(size_t n) { return static_cast<double*>(take(n * sizeof(double))); }
};

// K splits of the m x m product that fill the GPU (tiles of 128 x 64 on and below the diagonal).
int gram_splits(int64_t m, int64_t K) {
  const int64_t tm = ceil_div(m, 128), tn = ceil_div(m, 64), tiles = tm * tn - tm * (tm - 1);
  return (int)std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(152 / tiles, K / 256), 16));
}

}  // namespace

// The two products with N in them run as exact-slice products (7 levels, about 2^-53 of the row maxima's product
// per term) on the tensor cores, G's with rows weighted so that their maxima are bounded by its diagonal, as the factor's
// own rounding errors are, X's with its small elements summed again in float64: at N = 5124,
// m = 306, T = 200 the m x m one took 0.74 ms and the T x N one 1.0 ms on the float64 units; 0.06 ms each now.
// G's factor and inverse come from the one-launch factorisation (block kernels 1.3 ms, now 0.30 ms).
extern "C" kf_status mne_solve(const double* H, const double* C, int32_t c_kind, const double* R, int32_t r_kind,
                               const double* Y, int64_t N, int64_t m, int64_t T, double lambda, double* X_out,
                               void* stream) {
  if (!H || !C || !R || !Y || !X_out || N < 1 || m < 1 || T < 1) return KF_ERR_ARG;
  if (c_kind < 0 || c_kind > 2 || r_kind < 0 || r_kind > 2 || !(lambda > 0)) return KF_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  constexpr int LV = 7;
  bool slices = tc_available() && N <= (1 << 20) && m <= (1 << 20) && N <= INT32_MAX - 128 && T <= INT32_MAX - 128;
  const bool direct = m <= kInnovFactorMaxM;
  const int nb = direct ? 32 : potrf_block<double>();
  const int splits = gram_splits(m, N);
  // G's product and X's use the same memory one after the other: about 44 bytes per element of H beside H C's 8
  const size_t gram = c_kind == KF_COV_DENSE ? 0
                                             : 2 * oz_slice_bytes(m, N, LV) + (size_t)((splits > 1 ? splits : 0) * m + 2 * N) * m * 8;
  const size_t outp = oz_slice_bytes(T, m, LV) + oz_slice_bytes(N, m, LV) + (size_t)(N + 1) * m * 8;
  const size_t factor = direct ? (2 * (m + 32) * round_up(m, 32) + (T + m) * m) * 8 + innovation_factor_flags(m) * 4 : 0;
  const size_t plain = ((size_t)m * N + m * m + round_up(m, nb) * nb + T * m) * 8 + factor + 32 * 256;
  Tmp tmp;
  if (slices && tmp.reserve(plain + std::max(gram, outp)) != KF_OK) slices = false;  // the float64 products need less
  if (!slices) KF_TRY(tmp.reserve(plain));
  const bool gram_slices = slices && c_kind != KF_COV_DENSE;
  double* HC = tmp.doubles(m * N);
  double* G = tmp.doubles(m * m);
  double* dinv = tmp.doubles(round_up(m, nb) * nb);
  double* W = tmp.doubles(T * m);
  int* st = (int*)tmp.take(ST_WORDS * sizeof(int));
  double *Linv = nullptr, *V = nullptr, *work = nullptr;
  int* flags = nullptr;
  if (direct) {
    Linv = tmp.doubles(m * m);
    V = tmp.doubles(T * m);
    work = tmp.doubles((m + 32) * round_up(m, 32));
    flags = (int*)tmp.take(innovation_factor_flags(m) * sizeof(int));
  }
  const size_t shared = tmp.used;
  KF_CUDA_TRY(cudaMemsetAsync(st, 0, ST_WORDS * sizeof(int), s));
  // HC = H C  (m x N)
  if (c_kind == KF_COV_DENSE) {
    GemmParams<double> g;
    g.M = (int)m; g.N = (int)N; g.K = (int)N;
    g.A = H; g.lda = N;
    g.B = C; g.ldb = N;
    g.out = HC; g.ldo = N;
    KF_TRY(gemm_simt<double>(s, false, g));
  } else {
    KF_CUDA_TRY(cudaMemcpyAsync(HC, H, (size_t)m * N * 8, cudaMemcpyDeviceToDevice, s));
    dim3 grid((unsigned)std::min<int64_t>(ceil_div(N, 256), 64), (unsigned)std::min<int64_t>(m, 65535));
    scale_cols_kernel<<<grid, 256, 0, s>>>(m, N, HC, N, c_kind, C, 1.0);
    note_launch();
    KF_TRY(launch_check("scale_cols"));
  }
  // G = lambda (H C) H^T + R, symmetric by construction
  if (gram_slices) {
    OzSlices a, b;
    oz_slice_layout(a, tmp.take(oz_slice_bytes(m, N, LV)), m, N, LV);
    oz_slice_layout(b, tmp.take(oz_slice_bytes(m, N, LV)), m, N, LV);
    double* partials = splits > 1 ? tmp.doubles((size_t)splits * m * m) : nullptr;
    double *wa = tmp.doubles(m * N), *wb = tmp.doubles(m * N);
    const dim3 grid((unsigned)std::min<int64_t>(ceil_div(N, 256), 64), (unsigned)std::min<int64_t>(m, 32));
    weigh_cols_kernel<<<grid, 256, 0, s>>>(m, N, H, c_kind, C, wa, wb);
    note_launch();
    KF_TRY(launch_check("weigh_cols"));
    KF_TRY(oz_slice(s, wa, N, 1, m, N, LV, a));
    KF_TRY(oz_slice(s, wb, N, 1, m, N, LV, b));
    OzEpilogue e;
    e.alpha = lambda;
    e.out = G; e.ldo = m;
    e.radd_kind = r_kind; e.radd = R; e.ldradd = m;
    e.sym = 1;
    e.status = st;
    KF_TRY(oz_gemm(s, a, b, (int)m, (int)m, (int)N, LV, e, splits, partials));
  } else {
    GemmParams<double> g;
    g.M = (int)m; g.N = (int)m; g.K = (int)N;
    g.A = HC; g.lda = N;
    g.B = H; g.ldb = N;
    g.alpha = lambda;
    g.out2 = G; g.ldo2 = m;
    g.q_kind = r_kind; g.q = R; g.ldq = m;
    g.sym = 1;
    KF_TRY(gemm_simt<double>(s, true, g));
  }
  // W = Y G^{-1}
  if (direct) {
    KF_CUDA_TRY(cudaMemsetAsync(flags, 0, innovation_factor_flags(m) * sizeof(int), s));
    KF_TRY(innovation_factor(s, (int)m, G, m, dinv, Linv, nullptr, work, work + m * round_up(m, 32), flags, st, 0));
    GemmParams<double> g;  // (Y L^{-T}) L^{-1}
    g.M = (int)T; g.N = (int)m; g.K = (int)m;
    g.A = Y; g.lda = m;
    g.B = Linv; g.ldb = m;
    g.tri_b = 1;
    g.out = V; g.ldo = m;
    g.status = st;
    KF_TRY(gemm_simt<double>(s, true, g));
    g.A = V;
    g.tri_b = -1;
    g.out = W;
    KF_TRY(gemm_simt<double>(s, false, g));
  } else {
    KF_TRY(potrf<double>(s, G, m, (int)m, dinv, nb, st, 0));
    KF_CUDA_TRY(cudaMemcpyAsync(W, Y, (size_t)T * m * 8, cudaMemcpyDeviceToDevice, s));
    KF_TRY(trsm_right<double>(s, true, (int)T, (int)m, G, m, dinv, nb, W, m, st));
    KF_TRY(trsm_right<double>(s, false, (int)T, (int)m, G, m, dinv, nb, W, m, st));
  }
  // X = lambda W (H C)
  if (slices) {
    tmp.used = shared;
    OzSlices a, b;
    oz_slice_layout(a, tmp.take(oz_slice_bytes(T, m, LV)), T, m, LV);
    oz_slice_layout(b, tmp.take(oz_slice_bytes(N, m, LV)), N, m, LV);
    // the sensors balanced by powers of two, so that no sensor's unit dominates the row maxima:
    // sum_k W_k HC_k = sum_k (W_k scale_k) (HC_k / scale_k)
    double *HCt = tmp.doubles(N * m), *scale = tmp.doubles(m);
    row_scale_kernel<<<(unsigned)m, 256, 0, s>>>(N, HC, scale);
    note_launch();
    transpose_balanced_kernel<<<dim3((unsigned)ceil_div(N, 32), (unsigned)ceil_div(m, 32)), dim3(32, 8), 0, s>>>(
        m, N, HC, scale, HCt);
    note_launch();
    dim3 grid((unsigned)std::min<int64_t>(ceil_div(m, 256), 64), (unsigned)std::min<int64_t>(T, 65535));
    scale_cols_kernel<<<grid, 256, 0, s>>>(T, m, W, m, 1, scale, 1.0);
    note_launch();
    KF_TRY(launch_check("balance"));
    KF_TRY(oz_slice(s, W, m, 1, T, m, LV, a));
    KF_TRY(oz_slice(s, HCt, m, 1, N, m, LV, b));
    OzEpilogue e;
    e.alpha = lambda;
    e.out = X_out; e.ldo = N;
    e.status = st;
    KF_TRY(oz_gemm(s, a, b, (int)T, (int)N, (int)m, LV, e));
    small_elements_kernel<<<dim3((unsigned)ceil_div(N, 256), (unsigned)std::min<int64_t>(T, 65535)), 256, 0, s>>>(
        T, N, m, W, HCt, a.exps, b.exps, lambda, X_out, st);
    note_launch();
    KF_TRY(launch_check("small_elements"));
  } else {
    GemmParams<double> g;
    g.M = (int)T; g.N = (int)N; g.K = (int)m;
    g.A = W; g.lda = m;
    g.B = HC; g.ldb = N;
    g.alpha = lambda;
    g.out = X_out; g.ldo = N;
    KF_TRY(gemm_simt<double>(s, false, g));
  }
  int h[ST_WORDS];
  KF_CUDA_TRY(cudaMemcpyAsync(h, st, sizeof(h), cudaMemcpyDeviceToHost, s));
  KF_CUDA_TRY(cudaStreamSynchronize(s));
  return (kf_status)h[ST_CODE];
}

namespace {

// Dt[i][k] = (X[k+1][i] - X[k][i]) - dbar_i for k < T - 1, where the mean of the
// differences telescopes to dbar_i = (X[T-1][i] - X[0][i]) / (T - 1).
__global__ void centred_differences_kernel(int64_t N, int64_t T, const double* X, double* Dt) {
  const int64_t K = T - 1;
  for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < N * K; u += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k = u / N, i = u % N;  // consecutive threads read consecutive sources of one row
    const double dbar = (X[(T - 1) * N + i] - X[i]) / (double)K;
    Dt[i * K + k] = (X[(k + 1) * N + i] - X[k * N + i]) - dbar;
  }
}

}  // namespace

extern "C" kf_status mne_init(const double* H, const double* C, int32_t c_kind, const double* R, int32_t r_kind,
                              const double* Y, int64_t N, int64_t m, int64_t T, double lambda, double* X_out,
                              double* x0_out, double* Q_out, void* stream) {
  if (!x0_out || !Q_out || T < 3 || N < 1 || N > INT32_MAX) return KF_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  const int64_t K = T - 1;
  auto estimates = [&](double* X) -> kf_status {  // X and x0
    KF_TRY(mne_solve(H, C, c_kind, R, r_kind, Y, N, m, T, lambda, X, stream));
    KF_CUDA_TRY(cudaMemcpyAsync(x0_out, X, (size_t)N * 8, cudaMemcpyDeviceToDevice, s));
    return KF_OK;
  };
  auto differences = [&](const double* X, double* Dt) -> kf_status {
    const unsigned blocks = (unsigned)std::min<int64_t>(ceil_div(N * K, 256), 152 * 16);
    centred_differences_kernel<<<blocks, 256, 0, s>>>(N, T, X, Dt);
    note_launch();
    return launch_check("centred_differences");
  };
  const size_t x_bytes = X_out ? 0 : (size_t)T * N * 8;
  if (tc_available() && K <= (1 << 20) && N <= INT32_MAX - 128) {
    // Q = Dt Dt^T / (T - 2) as an exact-slice product like those of mne_solve (N = 8196, T = 300: 17.8 ms on the
    // float64 units, at their rate), all memory in one piece
    constexpr int LV = 7;
    Tmp tmp;
    if (tmp.reserve(x_bytes + (size_t)N * K * 8 + oz_slice_bytes(N, K, LV) + 8 * 256) == KF_OK) {
      double* X = X_out ? X_out : tmp.doubles(T * N);
      double* Dt = tmp.doubles(N * K);
      int* st = (int*)tmp.take(ST_WORDS * sizeof(int));
      const kf_status r = estimates(X);
      if (r == KF_OK) {
        KF_TRY(differences(X, Dt));
        KF_CUDA_TRY(cudaMemsetAsync(st, 0, ST_WORDS * sizeof(int), s));
        OzSlices a;
        oz_slice_layout(a, tmp.take(oz_slice_bytes(N, K, LV)), N, K, LV);
        KF_TRY(oz_slice(s, Dt, K, 1, N, K, LV, a));
        OzEpilogue e;
        e.alpha = 1.0 / (double)(T - 2);
        e.out = Q_out; e.ldo = N;
        e.sym = 1;
        e.status = st;
        KF_TRY(oz_gemm(s, a, a, (int)N, (int)N, (int)K, LV, e));
        int h[ST_WORDS];
        KF_CUDA_TRY(cudaMemcpyAsync(h, st, sizeof(h), cudaMemcpyDeviceToHost, s));
        KF_CUDA_TRY(cudaStreamSynchronize(s));
        return (kf_status)h[ST_CODE];
      }
      if (r != KF_ERR_CUDA) return r;  // else no memory left for the estimates
    }
  }
  // float64 product, memory taken when it is needed
  Tmp tx, td;
  if (!X_out) KF_TRY(tx.reserve(x_bytes));
  double* X = X_out ? X_out : (double*)tx.base;
  KF_TRY(estimates(X));
  KF_TRY(td.reserve((size_t)N * K * 8));
  double* Dt = (double*)td.base;
  KF_TRY(differences(X, Dt));
  GemmParams<double> g;  // lower triangle computed and mirrored
  g.M = (int)N; g.N = (int)N; g.K = (int)K;
  g.A = Dt; g.lda = K;
  g.B = Dt; g.ldb = K;
  g.alpha = 1.0 / (double)(T - 2);
  g.out = Q_out; g.ldo = N;
  g.sym = 1;
  KF_TRY(gemm_simt<double>(s, true, g));
  KF_CUDA_TRY(cudaStreamSynchronize(s));
  return KF_OK;
}
