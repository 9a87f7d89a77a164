// Mesh-coupled prediction (eqn 2 generalised to eqn 3): F P F^T + Q with the
// sparse neighbourhood matrix F in compressed-row form (<= 7 entries per row
// for the six-neighbour mesh).  Both passes stream whole rows of an N x N
// matrix, so they are HBM-bound: W = F P combines rows of P, and
// out = W F^T gathers, for each output column j, the entries of one row of W
// at the column indices of row j of F.
#include "ops.cuh"

namespace kfm {

template <typename T>
__global__ void spmm_fp_kernel(int64_t N, const int64_t* rowptr, const int64_t* col, const double* val,
                               const T* P, int64_t ldp, T* W, int64_t ldw) {
  for (int64_t i = blockIdx.x; i < N; i += gridDim.x) {
    const int64_t k0 = rowptr[i], k1 = rowptr[i + 1];
    for (int64_t j = threadIdx.x; j < N; j += blockDim.x) {
      double acc = 0.0;
      for (int64_t k = k0; k < k1; ++k) acc = fma(val[k], (double)P[col[k] * ldp + j], acc);
      W[i * ldw + j] = (T)acc;
    }
  }
}

template <typename T>
__global__ void spmm_wft_kernel(int64_t N, const int64_t* rowptr, const int64_t* col, const double* val,
                                const T* W, int64_t ldw, T* out, int64_t ldo, int q_kind, const double* q) {
  for (int64_t i = blockIdx.x; i < N; i += gridDim.x) {
    const T* wrow = W + i * ldw;
    for (int64_t j = threadIdx.x; j < N; j += blockDim.x) {
      double acc = 0.0;
      for (int64_t k = rowptr[j]; k < rowptr[j + 1]; ++k) acc = fma(val[k], (double)__ldg(wrow + col[k]), acc);
      if (q_kind == 0 && i == j) acc += q[0];
      else if (q_kind == 1 && i == j) acc += q[i];
      else if (q_kind == 2) acc += q[i * N + j];
      out[i * ldo + j] = (T)acc;
    }
  }
}

template <typename T>
kf_status spmm_fpft(cudaStream_t s, int64_t N, const int64_t* rowptr, const int64_t* col, const double* val,
                    const T* P, int64_t ldp, T* W, int64_t ldw, T* out, int64_t ldo, int q_kind,
                    const double* q) {
  if (N <= 0) return KF_OK;
  unsigned blocks = (unsigned)std::min<int64_t>(N, 1 << 20);
  spmm_fp_kernel<T><<<blocks, 256, 0, s>>>(N, rowptr, col, val, P, ldp, W, ldw);
  note_launch();
  KF_TRY(launch_check("spmm_fp"));
  spmm_wft_kernel<T><<<blocks, 256, 0, s>>>(N, rowptr, col, val, W, ldw, out, ldo, q_kind, q);
  note_launch();
  return launch_check("spmm_wft");
}

template <typename T>
kf_status spmm_pft(cudaStream_t s, int64_t N, const int64_t* rowptr, const int64_t* col, const double* val,
                   const T* P, int64_t ldp, T* out, int64_t ldo) {
  if (N <= 0) return KF_OK;
  unsigned blocks = (unsigned)std::min<int64_t>(N, 1 << 20);
  spmm_wft_kernel<T><<<blocks, 256, 0, s>>>(N, rowptr, col, val, P, ldp, out, ldo, -1, nullptr);
  note_launch();
  return launch_check("spmm_pft");
}

// ---------------------------------------------------------------- float32 matrices, packed F
//
// The sums of a float32 matrix in float64 took 14 float64 operations per element (a conversion and a
// multiply-add per entry of F): 0.73 ms per pass at N = 5124, on the float64 units, where the matrix passes HBM
// in 0.03 ms.  Here a sum is a pair of float32 (its rounded value and what the rounding lost, Knuth's two-sum;
// products exact by fused multiply-add, F as value + remainder), 46 bits of the largest partial sum, rounded once at
// the end.  Where that leaves fewer than 30 bits of the sum (cancellation), or a term leaves float32's range
// (small or large covariances, entries of F, infinities), the element is summed again in float64; so the result
// is the float64 sum's rounding but for ties to 2^-6 of a unit (N = 5124: 0.13 ms for F P and 0.17 ms for W F^T).

// A sum's range in which its low half keeps its bits and no product overflows; of F's entries too.
constexpr float kPairMin = 0x1p-100f, kPairMax = 0x1p+120f;

struct Pair {
  float h = 0.0f, l = 0.0f, mag = 0.0f;  // mag: sum of the terms' magnitudes
  __device__ __forceinline__ void add(float x) {  // exact sum of h and x, the error into l
    const float s = h + x, t = s - h;
    l += (h - (s - t)) + (x - t);
    h = s;
    mag += fabsf(x);
  }
  // += (vh + vl) p
  __device__ __forceinline__ void fma(float vh, float vl, float p) {
    const float q = vh * p;
    l += fmaf(vl, p, fmaf(vh, p, -q));
    add(q);
  }
  // float32 value, good unless false is returned (an infinity or NaN fails every comparison; mag is zero where every
  // term is, or underflows float32 altogether)
  __device__ __forceinline__ bool value(float& v) const {
    v = h + l;
    return (fabsf(v) >= mag * 0x1p-16f && fabsf(v) >= kPairMin && mag <= kPairMax) || mag == 0.0f;
  }
};

// NaN for a value outside the range: every sum with it is done in float64.
__global__ void spmm_pack_kernel(int64_t nnz, const int64_t* col, const double* val, float4* out) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nnz; k += (int64_t)gridDim.x * blockDim.x) {
    const double v = val[k];
    const float h = v == 0.0 || (fabs(v) >= kPairMin && fabs(v) <= kPairMax) ? (float)v : NAN;
    out[k] = make_float4(h, (float)(v - (double)h), __int_as_float((int)col[k]), 0.0f);
  }
}

kf_status spmm_pack(cudaStream_t s, int64_t nnz, const int64_t* col, const double* val, float4* out) {
  spmm_pack_kernel<<<(unsigned)std::min<int64_t>(ceil_div(nnz, 256), 4096), 256, 0, s>>>(nnz, col, val, out);
  note_launch();
  return launch_check("spmm_pack");
}

// The same sum in float64, as the kernels above form it: row[k] times F[k], p the column of P (its rows ld apart) or
// the row of W (ld 1).
__device__ __noinline__ double spmm_sum64(int64_t k0, int64_t k1, const int64_t* col, const double* val, const float* p,
                                          int64_t ld) {
  double acc = 0.0;
  for (int64_t k = k0; k < k1; ++k) acc = fma(val[k], (double)p[col[k] * ld], acc);
  return acc;
}

// W = F P, one block per row: four consecutive columns per thread, each entry's row of P read in 16-byte loads.
__global__ void __launch_bounds__(256) spmm_fp_packed_kernel(int64_t N, const int64_t* rowptr, const int64_t* col,
                                                             const double* val, const float4* F, const float* P,
                                                             int64_t ldp, float* W, int64_t ldw) {
  const int64_t i = blockIdx.x, k0 = rowptr[i], k1 = rowptr[i + 1];
  for (int64_t j = 4 * (int64_t)threadIdx.x; j < N; j += 4 * 256) {
    Pair acc[4];
    for (int64_t k = k0; k < k1; ++k) {
      const float4 f = F[k];
      const float4 p = *reinterpret_cast<const float4*>(P + (int64_t)__float_as_int(f.z) * ldp + j);
      acc[0].fma(f.x, f.y, p.x);
      acc[1].fma(f.x, f.y, p.y);
      acc[2].fma(f.x, f.y, p.z);
      acc[3].fma(f.x, f.y, p.w);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (j + e >= N) break;
      float v;
      if (!acc[e].value(v)) v = (float)spmm_sum64(k0, k1, col, val, P + j + e, ldp);
      W[i * ldw + j + e] = v;
    }
  }
}

// out = W F^T (+ Q): a block stages R rows of W in shared memory, so that the gathers at F's columns are shared
// loads and each entry of F is read once for R rows.
template <int R>
__global__ void __launch_bounds__(512) spmm_wft_packed_kernel(int64_t N, const int64_t* rowptr, const int64_t* col,
                                                              const double* val, const float4* F, const float* W,
                                                              int64_t ldw, float* out, int64_t ldo, int q_kind,
                                                              const double* q) {
  extern __shared__ __align__(16) float rows[];  // R x ldw
  const int64_t i0 = (int64_t)blockIdx.x * R;
  const int nr = (int)(N - i0 < R ? N - i0 : R);
  for (int64_t u = threadIdx.x; u < nr * (ldw / 4); u += 512)
    reinterpret_cast<float4*>(rows)[u] = reinterpret_cast<const float4*>(W + i0 * ldw)[u];
  __syncthreads();
  for (int64_t j = threadIdx.x; j < N; j += 512) {
    Pair acc[R];
    const int64_t k0 = rowptr[j], k1 = rowptr[j + 1];
    for (int64_t k = k0; k < k1; ++k) {
      const float4 f = F[k];
      const float* w = rows + __float_as_int(f.z);
#pragma unroll
      for (int r = 0; r < R; ++r) acc[r].fma(f.x, f.y, w[r * ldw]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (r >= nr) break;
      const int64_t i = i0 + r;
      const bool add_q = q_kind == 2 || (q_kind >= 0 && i == j);
      double qv = 0.0;
      if (add_q) {
        qv = q_kind == 0 ? q[0] : q_kind == 1 ? q[i] : q[i * N + j];
        const float h = (float)qv;
        acc[r].add(h);
        acc[r].add((float)(qv - (double)h));
      }
      float v;
      if (!acc[r].value(v)) {
        const double s = spmm_sum64(k0, k1, col, val, rows + r * ldw, 1);
        v = (float)(add_q ? s + qv : s);
      }
      out[i * ldo + j] = v;
    }
  }
}

template <int R>
kf_status launch_wft_packed(cudaStream_t s, int64_t N, const SpmmPacked& F, const float* W, int64_t ldw, float* out,
                            int64_t ldo, int q_kind, const double* q) {
  KF_CUDA_TRY(smem_limit_per_device((const void*)spmm_wft_packed_kernel<R>, 216 * 1024));
  spmm_wft_packed_kernel<R><<<(unsigned)ceil_div(N, R), 512, R * ldw * sizeof(float), s>>>(
      N, F.rowptr, F.col, F.val, F.pack, W, ldw, out, ldo, q_kind, q);
  note_launch();
  return launch_check("spmm_wft_packed");
}

// As many rows per block as keep two blocks on an SM, four at most while eight would leave SMs idle.
kf_status spmm_wft_packed(cudaStream_t s, int64_t N, const SpmmPacked& F, const float* W, int64_t ldw, float* out,
                          int64_t ldo, int q_kind, const double* q) {
  const int64_t row = ldw * (int64_t)sizeof(float);
  if (8 * row <= 108 * 1024 && N >= 8 * 304) return launch_wft_packed<8>(s, N, F, W, ldw, out, ldo, q_kind, q);
  if (4 * row <= 108 * 1024) return launch_wft_packed<4>(s, N, F, W, ldw, out, ldo, q_kind, q);
  if (2 * row <= 108 * 1024) return launch_wft_packed<2>(s, N, F, W, ldw, out, ldo, q_kind, q);
  if (row > 216 * 1024) return KF_ERR_ARG;
  return launch_wft_packed<1>(s, N, F, W, ldw, out, ldo, q_kind, q);
}

bool spmm_packed_ok(int64_t N, int64_t ld) { return N <= INT32_MAX && ld % 4 == 0 && ld * 4 <= 216 * 1024; }

kf_status spmm_fp_packed(cudaStream_t s, int64_t N, const SpmmPacked& F, const float* P, int64_t ldp, float* W, int64_t ldw) {
  if (N <= 0) return KF_OK;
  spmm_fp_packed_kernel<<<(unsigned)N, 256, 0, s>>>(N, F.rowptr, F.col, F.val, F.pack, P, ldp, W, ldw);
  note_launch();
  return launch_check("spmm_fp_packed");
}

kf_status spmm_fpft_packed(cudaStream_t s, int64_t N, const SpmmPacked& F, const float* P, int64_t ldp, float* W, int64_t ldw,
                           float* out, int64_t ldo, int q_kind, const double* q) {
  KF_TRY(spmm_fp_packed(s, N, F, P, ldp, W, ldw));
  return spmm_wft_packed(s, N, F, W, ldw, out, ldo, q_kind, q);
}

template kf_status spmm_fpft<double>(cudaStream_t, int64_t, const int64_t*, const int64_t*, const double*,
                                     const double*, int64_t, double*, int64_t, double*, int64_t, int,
                                     const double*);
template kf_status spmm_fpft<float>(cudaStream_t, int64_t, const int64_t*, const int64_t*, const double*,
                                    const float*, int64_t, float*, int64_t, float*, int64_t, int,
                                    const double*);
template kf_status spmm_pft<double>(cudaStream_t, int64_t, const int64_t*, const int64_t*, const double*,
                                    const double*, int64_t, double*, int64_t);
template kf_status spmm_pft<float>(cudaStream_t, int64_t, const int64_t*, const int64_t*, const double*,
                                   const float*, int64_t, float*, int64_t);

}  // namespace kfm
