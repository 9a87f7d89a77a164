// Cholesky factor and triangular inverse of a float32 matrix of up to kCholDirectMaxN rows in one launch: the
// leaves of the smoother-gain factorisation P_{t+1|t} = L L^T, W = L^{-1} (eqn 11).
//
// What bounds it: the chain of n pivots (about 200 cycles each) and, per 32-wide tile column, two trips through
// L2 (the inverse of the diagonal tile to the panel below it, the panel to the next diagonal tile).  As a
// recursion of launches a matrix of 1024 rows took eight 128-wide leaves on one SM each (30 us) and about 40
// small products (5 to 23 us), about 0.5 ms together; this launch takes 0.24 ms (1501 rows: 0.43 ms).
//
// Layout: 32 x 32 tiles, a CTA per tile of L and of W, in dataflow order with a flag per tile.
//   L(i, j), i > j: starts from A(i, j), subtracts L(i, k) L(j, k)^T for k < j, then multiplies by D_j^T
//   (D_j = L_jj^{-1});  diagonal tiles factor and invert theirs after the subtractions;
//   W(i, j), i > j: sums L(i, k) W(k, j) for j <= k < i and multiplies by -D_i;  W(j, j) = D_j.
// Tickets go by tile column j of L, then row j of W, so that every CTA waits only for lower tickets and the
// launch progresses however many CTAs are resident.  Waits are bounded; they end when the status word reports a
// failure.  Products are float32 fused multiply-adds in a fixed order: deterministic; sums over tiles carry their
// rounding errors, which keeps the inverse as accurate as with the split-bf16 products of the recursion (relative
// error at n = 700, cond 100: 9.6e-7, and 2.2e-6 by recursion).
#include "ops.cuh"
#include "tc_ptx.cuh"

namespace kfm {

namespace {

constexpr int kCdThreads = 256;  // thread: row tid / 8, columns 4 (tid mod 8) .. + 3 of the CTA's tile
constexpr int kPad = 36;         // 16-byte aligned rows, 8 rows apart in different banks

struct CdArgs {
  int n, T;
  float* L;
  int64_t ldl;
  float* W;
  int64_t ldw;
  int* flags;  // ticket, then T x T: [i T + j] for L(i, j) (i > j), D_i and W(i, i) (i == j); [j T + i] for W(i, j)
  int* status;
  int step, base;
};

__device__ __forceinline__ int cd_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// The CTA waits for a tile; false when the wait expired or another tile failed.
__device__ __forceinline__ bool cd_wait(const int* flag, const CdArgs& a) {
  bool ok = true;
  if (threadIdx.x == 0 && cd_acquire(flag) == 0) {
    const uint64_t t0 = globaltimer();
    for (int n = 1; cd_acquire(flag) == 0; ++n) {
      if ((n & 15) == 0) {
        if (status_failed(a.status)) {
          ok = false;
          break;
        }
        if (globaltimer() - t0 > WAIT_NS) {
          status_set(a.status, KF_ERR_TIMEOUT, a.step, 23);
          ok = false;
          break;
        }
      }
    }
  }
  return __syncthreads_and(ok);
}

__device__ __forceinline__ void cd_publish(int* flag) {
  __syncthreads();
  if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(flag) : "memory");
}

// The thread's four elements of tile (i, j) of X; zero outside the n x n matrix.
__device__ __forceinline__ float4 cd_load(const float* X, int64_t ld, int n, int i, int j, int r, int c) {
  const int gi = 32 * i + r, gj = 32 * j + c;
  if (gi >= n) return make_float4(0.f, 0.f, 0.f, 0.f);
  const float* p = X + (int64_t)gi * ld + gj;
  if (gj + 4 <= n) return *reinterpret_cast<const float4*>(p);
  float v[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) v[e] = gj + e < n ? p[e] : 0.0f;
  return make_float4(v[0], v[1], v[2], v[3]);
}

__device__ __forceinline__ void cd_store(float* X, int64_t ld, int n, int i, int j, int r, int c, const float (&v)[4]) {
  const int gi = 32 * i + r, gj = 32 * j + c;
  if (gi >= n) return;
  float* p = X + (int64_t)gi * ld + gj;
  if (gj + 4 <= n) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (gj + e < n) p[e] = v[e];
  }
}

// acc[e] += sum_k A[r][k] B[k][c + e] for tiles in shared memory (A by rows, B by its rows k).
__device__ __forceinline__ void cd_mul(const float (*A)[kPad], const float (*B)[kPad], int r, int c, float (&acc)[4]) {
#pragma unroll
  for (int k = 0; k < 32; k += 4) {
    const float4 a4 = *reinterpret_cast<const float4*>(&A[r][k]);
    const float av[4] = {a4.x, a4.y, a4.z, a4.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float4 b = *reinterpret_cast<const float4*>(&B[k + e][c]);
      acc[0] = fmaf(av[e], b.x, acc[0]);
      acc[1] = fmaf(av[e], b.y, acc[1]);
      acc[2] = fmaf(av[e], b.z, acc[2]);
      acc[3] = fmaf(av[e], b.w, acc[3]);
    }
  }
}

// total += part per element, the rounding errors kept beside it (Knuth's two-sum): a sum over many tiles stays at
// the accuracy of one tile's.
__device__ __forceinline__ void cd_add(const float (&part)[4], float (&total)[4], float (&low)[4]) {
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float sum = total[e] + part[e], t = sum - total[e];
    low[e] += (total[e] - (sum - t)) + (part[e] - t);
    total[e] = sum;
  }
}

struct CdSmem {
  float A[32][kPad], B[32][kPad];
  float col[2][kPad];  // a finished column of the diagonal tile, and its 1 / pivot in [32]
  int fail;
};

// Diagonal tile in s.A (by rows): warp 0 factors it (lane = row, the row in registers), warp 1 forms the inverse one
// column behind (lane = column of the inverse); on return s.A holds L and s.B the inverse, both by rows.
__device__ void cd_factor(CdSmem& s, const CdArgs& a, int tile) {
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int m = min(32, a.n - 32 * tile);
  if (warp == 0) {
    float r[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) r[k] = lane < m && k < m ? s.A[lane][k] : (lane == k ? 1.0f : 0.0f);
    int bad = -1;
    float d = __shfl_sync(0xffffffffu, r[0], 0);
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      if (bad < 0 && !(d > 0.0f && d < INFINITY)) bad = j;
      float q = rsqrtf(d);
      q = q * (1.5f - 0.5f * d * q * q);  // one Newton step: about 1 ulp
      const float l = lane > j ? r[j] * q : (lane == j ? d * q : 0.0f);
      // the next pivot ahead of this column's round trip through shared memory
      if (j < 31) d = __shfl_sync(0xffffffffu, fmaf(-l, l, r[j + 1]), j + 1);
      float* col = s.col[j & 1];
      col[lane] = l;
      if (lane == 0) col[32] = q;
      asm volatile("bar.sync 1, 64;" ::: "memory");
      r[j] = l;
#pragma unroll
      for (int g = (j + 1) / 4; g < 8; ++g) {
        const float4 v = reinterpret_cast<const float4*>(col)[g];
        const float ve[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (4 * g + e > j) r[4 * g + e] = fmaf(-l, ve[e], r[4 * g + e]);
      }
    }
    if (lane == 0) {
      s.fail = bad >= 0;
      if (bad >= 0) status_set(a.status, KF_ERR_NOT_PD, a.step, a.base + 32 * tile + bad);
    }
#pragma unroll
    for (int k = 0; k < 32; ++k) s.A[lane][k] = k <= lane ? r[k] : 0.0f;
  } else if (warp == 1) {
    float x[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) x[i] = i == lane ? 1.0f : 0.0f;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      asm volatile("bar.sync 1, 64;" ::: "memory");
      const float* col = s.col[j & 1];
      const float xj = x[j] * col[32];
      x[j] = xj;
#pragma unroll
      for (int g = (j + 1) / 4; g < 8; ++g) {
        const float4 v = reinterpret_cast<const float4*>(col)[g];
        const float ve[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (4 * g + e > j) x[4 * g + e] = fmaf(-ve[e], xj, x[4 * g + e]);
      }
    }
#pragma unroll
    for (int i = 0; i < 32; ++i) s.B[i][lane] = i >= lane ? x[i] : 0.0f;
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kCdThreads) chol_direct_kernel(const CdArgs a) {
  __shared__ __align__(16) CdSmem s;
  __shared__ int ticket_s;
  if (threadIdx.x == 0) {
    ticket_s = status_failed(a.status) ? -1 : atomicAdd(a.flags, 1);
    s.fail = 0;
  }
  __syncthreads();
  if (ticket_s < 0) return;
  // ticket -> (column j of L: tiles i = j .. T-1; then row j of W: tiles 0 .. j-1): T tickets per j
  const int j = ticket_s / a.T, u = ticket_s % a.T;
  const int T = a.T, n = a.n;
  const int r = threadIdx.x / 8, c = 4 * (threadIdx.x % 8);
  int* fl = a.flags + 1;
  auto put = [&](float (*dst)[kPad], const float4& v) { *reinterpret_cast<float4*>(&dst[r][c]) = v; };
  auto put_t = [&](float (*dst)[kPad], const float4& v) {
    dst[c][r] = v.x;
    dst[c + 1][r] = v.y;
    dst[c + 2][r] = v.z;
    dst[c + 3][r] = v.w;
  };
  float total[4] = {0.f, 0.f, 0.f, 0.f}, low[4] = {0.f, 0.f, 0.f, 0.f};
  if (u < T - j) {
    // ---- L(i, j)
    const int i = j + u;
    const float4 a0 = cd_load(a.L, a.ldl, n, i, j, r, c);
    for (int k = 0; k < j; ++k) {
      if (!cd_wait(fl + i * T + k, a)) return;
      const float4 x = cd_load(a.L, a.ldl, n, i, k, r, c);
      float4 y = x;
      if (i != j) {
        if (!cd_wait(fl + j * T + k, a)) return;
        y = cd_load(a.L, a.ldl, n, j, k, r, c);
      }
      put(s.A, x);
      put_t(s.B, y);
      __syncthreads();
      float part[4] = {0.f, 0.f, 0.f, 0.f};
      cd_mul(s.A, s.B, r, c, part);
      cd_add(part, total, low);
      __syncthreads();
    }
    put(s.A, make_float4((a0.x - total[0]) - low[0], (a0.y - total[1]) - low[1], (a0.z - total[2]) - low[2],
                         (a0.w - total[3]) - low[3]));
    __syncthreads();
    if (i == j) {
      cd_factor(s, a, j);
      if (s.fail) return;
      float d[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) d[e] = s.B[r][c + e];
      cd_store(a.W, a.ldw, n, j, j, r, c, d);
      cd_publish(fl + j * T + j);
#pragma unroll
      for (int e = 0; e < 4; ++e)  // the lower triangle of L
        if (c + e <= r && 32 * j + r < n) a.L[(int64_t)(32 * j + r) * a.ldl + 32 * j + c + e] = s.A[r][c + e];
      return;
    }
    if (!cd_wait(fl + j * T + j, a)) return;
    put_t(s.B, cd_load(a.W, a.ldw, n, j, j, r, c));  // (D_j)^T
    __syncthreads();
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    cd_mul(s.A, s.B, r, c, acc);
    cd_store(a.L, a.ldl, n, i, j, r, c, acc);
    cd_publish(fl + i * T + j);
    return;
  }
  // ---- W(i, jw) with i = j
  const int i = j, jw = u - (T - j);
  for (int k = jw; k < i; ++k) {
    if (!cd_wait(fl + i * T + k, a)) return;                     // L(i, k)
    const float4 x = cd_load(a.L, a.ldl, n, i, k, r, c);
    if (!cd_wait(k == jw ? fl + k * T + k : fl + jw * T + k, a)) return;  // W(k, jw)
    const float4 y = cd_load(a.W, a.ldw, n, k, jw, r, c);
    put(s.A, x);
    put(s.B, y);
    __syncthreads();
    float part[4] = {0.f, 0.f, 0.f, 0.f};
    cd_mul(s.A, s.B, r, c, part);
    cd_add(part, total, low);
    __syncthreads();
  }
  if (!cd_wait(fl + i * T + i, a)) return;  // D_i
  put(s.A, cd_load(a.W, a.ldw, n, i, i, r, c));
  put(s.B, make_float4(-(total[0] + low[0]), -(total[1] + low[1]), -(total[2] + low[2]), -(total[3] + low[3])));
  __syncthreads();
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  cd_mul(s.A, s.B, r, c, acc);
  cd_store(a.W, a.ldw, n, i, jw, r, c, acc);
  cd_publish(fl + jw * T + i);
}

}  // namespace

kf_status chol_inverse_direct(cudaStream_t s, int n, float* L, int64_t ldl, float* W, int64_t ldw, void* scratch,
                              int* status, int step, int base) {
  if (n < 1 || n > kCholDirectMaxN || !L || !W || !scratch) return KF_ERR_ARG;
  if (ldl % 4 || ldw % 4 || ((reinterpret_cast<uintptr_t>(L) | reinterpret_cast<uintptr_t>(W)) & 15)) return KF_ERR_ARG;
  CdArgs a;
  a.n = n;
  a.T = (int)ceil_div(n, 32);
  a.L = L;
  a.ldl = ldl;
  a.W = W;
  a.ldw = ldw;
  a.flags = static_cast<int*>(scratch);
  a.status = status;
  a.step = step;
  a.base = base;
  KF_CUDA_TRY(cudaMemsetAsync(scratch, 0, chol_direct_scratch(n), s));
  chol_direct_kernel<<<(unsigned)(a.T * a.T), kCdThreads, 0, s>>>(a);
  note_launch();
  return launch_check("chol_direct");
}

size_t chol_direct_scratch(int n) {
  const int T = (int)ceil_div(n, 32);
  return (size_t)(1 + T * T) * sizeof(int);
}

}  // namespace kfm
