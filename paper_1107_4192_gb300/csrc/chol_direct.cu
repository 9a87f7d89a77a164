// Cholesky factor and triangular inverse of a float32 matrix of up to kCholDirectMaxN rows in one launch: the
// leaves of the smoother-gain factorisation P_{t+1|t} = L L^T, W = L^{-1} (eqn 11).
//
// What bounds it: the chain of n pivots (6.1 us per tile column: about 200 cycles per pivot, and the trip of the
// diagonal tile's inverse through L2 to the tile below it), and from about 1200 rows on the tiles' loads.  As a
// recursion of launches a matrix of 1024 rows took eight 128-wide leaves on one SM each (30 us) and about 40
// small products (5 to 23 us), about 0.5 ms together; this launch takes 0.21 ms (n = 128: 25 us, 512: 97 us, 1281:
// 0.29 ms, 1501: 0.38 ms).  With the diagonal tiles on CTAs of their own, a trip through L2 more per column, and a
// look at two flags before each tile it was 0.24 ms, and 0.43 ms for 1501 rows.  Subtracting a column's products one
// column later, behind the next pivot, gave nothing (0.21 and 0.39 ms).
//
// Layout: 32 x 32 tiles, a CTA per tile of L and of W, in dataflow order with a flag per tile.
//   L(i, j), i > j: starts from A(i, j), subtracts L(i, k) L(j, k)^T for k < j, then multiplies by D_j^T
//   (D_j = L_jj^{-1});  the CTA of L(j + 1, j) goes on with diagonal tile j + 1, which it factors and inverts;
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

// Tiles k, k + 1, .. of two rows of flags: waits for both flags of tile k and returns how many tiles up to k1 are ready
// in a row (at most 32; 0 when the wait expired or another tile failed).  One look at the flags for a run of tiles: a
// CTA that starts behind the others passes the finished columns at the pace of its loads.
__device__ __forceinline__ int cd_ready(const int* f, const int* g, int k, int k1, int* count, const CdArgs& a) {
  if (threadIdx.x < 32) {
    const int kk = k + (int)threadIdx.x;
    const uint64_t t0 = globaltimer();
    int run = 0;
    for (int n = 1; run == 0; ++n) {
      int ready = 0;
      if (kk < k1) {
        const int x = cd_acquire(f + kk), y = cd_acquire(g + kk);
        ready = x != 0 && y != 0;
      }
      run = __ffs(~__ballot_sync(0xffffffffu, ready)) - 1;
      if (run < 0) run = 32;
      if (run == 0 && (n & 15) == 0) {
        int stop = 0;
        if (threadIdx.x == 0) {
          stop = status_failed(a.status);
          if (!stop && globaltimer() - t0 > WAIT_NS) {
            status_set(a.status, KF_ERR_TIMEOUT, a.step, 23);
            stop = 1;
          }
        }
        if (__shfl_sync(0xffffffffu, stop, 0)) break;
      }
    }
    if (threadIdx.x == 0) *count = run;
  }
  __syncthreads();
  return *count;
}

struct CdSmem {
  float A[2][32][kPad], B[2][32][kPad], C[2][32][kPad];
  float col[32][kPad];  // the finished columns of the diagonal tile, each with its 1 / pivot in [32]
  int fail, run;
};

// Diagonal tile in s.A[0] (by rows): warp 0 factors it (lane = row, the row in registers), warp 1 forms the inverse four
// columns behind (lane = column of the inverse); on return s.A[0] holds L and s.B[0] the inverse, both by rows.  Warp 0
// announces every fourth column at a barrier of its own and waits for nothing.  Not inlined: with the caller's
// registers live the columns spill.
__device__ __noinline__ void cd_factor(CdSmem& s, const CdArgs& a, int tile) {
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int m = min(32, a.n - 32 * tile);
  if (warp == 0) {
    float r[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) r[k] = lane < m && k < m ? s.A[0][lane][k] : (lane == k ? 1.0f : 0.0f);
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
      float* col = s.col[j];
      col[lane] = l;
      if (lane == 0) col[32] = q;
      __syncwarp();
      if (j % 4 == 3) asm volatile("bar.arrive %0, 64;" ::"r"(1 + j / 4) : "memory");
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
    for (int k = 0; k < 32; ++k) s.A[0][lane][k] = k <= lane ? r[k] : 0.0f;
  } else if (warp == 1) {
    float x[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) x[i] = i == lane ? 1.0f : 0.0f;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      if (j % 4 == 0) asm volatile("bar.sync %0, 64;" ::"r"(1 + j / 4) : "memory");
      const float* col = s.col[j];
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
    for (int i = 0; i < 32; ++i) s.B[0][i][lane] = i >= lane ? x[i] : 0.0f;
  }
  __syncthreads();
}

// Two CTAs per SM: with three the columns of a diagonal tile spill (1024 rows 0.23 ms).
__global__ void __launch_bounds__(kCdThreads, 2) chol_direct_kernel(const CdArgs a) {
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
  auto minus = [](const float4& v, const float (&t)[4], const float (&l)[4]) {
    return make_float4((v.x - t[0]) - l[0], (v.y - t[1]) - l[1], (v.z - t[2]) - l[2], (v.w - t[3]) - l[3]);
  };
  if (u < T - j) {
    // ---- L(i, j); the CTA of L(j + 1, j) goes on with diagonal tile j + 1
    const int i = j + u;
    if (u == 0 && j > 0) return;  // factored by the CTA of L(j, j - 1)
    const bool next = u == 1;
    if (u == 0) {
      put(s.A[0], cd_load(a.L, a.ldl, n, 0, 0, r, c));
      __syncthreads();
    } else {
      const float4 a0 = cd_load(a.L, a.ldl, n, i, j, r, c);
      const float4 d0 = next ? cd_load(a.L, a.ldl, n, i, i, r, c) : a0;
      float dtotal[4] = {0.f, 0.f, 0.f, 0.f}, dlow[4] = {0.f, 0.f, 0.f, 0.f};
      for (int k = 0; k < j;) {
        const int end = k + cd_ready(fl + i * T, fl + j * T, k, j, &s.run, a);
        if (end == k) return;
        float4 x = cd_load(a.L, a.ldl, n, i, k, r, c), y = cd_load(a.L, a.ldl, n, j, k, r, c);
#pragma unroll 1
        for (; k < end; ++k) {
          const int b = k & 1;
          put(s.A[b], x);
          put_t(s.B[b], y);
          if (next) put_t(s.C[b], x);
          __syncthreads();
          if (k + 1 < end) {
            x = cd_load(a.L, a.ldl, n, i, k + 1, r, c);
            y = cd_load(a.L, a.ldl, n, j, k + 1, r, c);
          }
          float part[4] = {0.f, 0.f, 0.f, 0.f};
          cd_mul(s.A[b], s.B[b], r, c, part);
          cd_add(part, total, low);
          if (next) {
            float dpart[4] = {0.f, 0.f, 0.f, 0.f};
            cd_mul(s.A[b], s.C[b], r, c, dpart);
            cd_add(dpart, dtotal, dlow);
          }
        }
      }
      __syncthreads();
      put(s.A[0], minus(a0, total, low));
      if (!cd_wait(fl + j * T + j, a)) return;
      put_t(s.B[0], cd_load(a.W, a.ldw, n, j, j, r, c));  // (D_j)^T
      __syncthreads();
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
      cd_mul(s.A[0], s.B[0], r, c, acc);
      cd_store(a.L, a.ldl, n, i, j, r, c, acc);
      if (!next) {
        cd_publish(fl + i * T + j);
        return;
      }
      __syncthreads();
      const float4 l = make_float4(acc[0], acc[1], acc[2], acc[3]);
      put(s.A[0], l);
      put_t(s.B[0], l);
      __syncthreads();
      float part[4] = {0.f, 0.f, 0.f, 0.f};
      cd_mul(s.A[0], s.B[0], r, c, part);
      cd_add(part, dtotal, dlow);
      __syncthreads();
      put(s.A[0], minus(d0, dtotal, dlow));
      __syncthreads();
      // L(i, j) published by a warp that has no part in the factorisation
      if (threadIdx.x == kCdThreads - 1)
        asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(fl + i * T + j) : "memory");
    }
    cd_factor(s, a, i);
    if (s.fail) return;
    float d[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) d[e] = s.B[0][r][c + e];
    cd_store(a.W, a.ldw, n, i, i, r, c, d);
    cd_publish(fl + i * T + i);
#pragma unroll
    for (int e = 0; e < 4; ++e)  // the lower triangle of L
      if (c + e <= r && 32 * i + r < n) a.L[(int64_t)(32 * i + r) * a.ldl + 32 * i + c + e] = s.A[0][r][c + e];
    return;
  }
  // ---- W(i, jw) with i = j
  const int i = j, jw = u - (T - j);
  for (int k = jw; k < i;) {
    const int end = k + cd_ready(fl + i * T, fl + jw * T, k, i, &s.run, a);  // L(i, k) and W(k, jw)
    if (end == k) return;
    float4 x = cd_load(a.L, a.ldl, n, i, k, r, c), y = cd_load(a.W, a.ldw, n, k, jw, r, c);
#pragma unroll 1
    for (; k < end; ++k) {
      const int b = k & 1;
      put(s.A[b], x);
      put(s.B[b], y);
      __syncthreads();
      if (k + 1 < end) {
        x = cd_load(a.L, a.ldl, n, i, k + 1, r, c);
        y = cd_load(a.W, a.ldw, n, k + 1, jw, r, c);
      }
      float part[4] = {0.f, 0.f, 0.f, 0.f};
      cd_mul(s.A[b], s.B[b], r, c, part);
      cd_add(part, total, low);
    }
  }
  __syncthreads();
  if (!cd_wait(fl + i * T + i, a)) return;  // D_i
  put(s.A[0], cd_load(a.W, a.ldw, n, i, i, r, c));
  put(s.B[0], make_float4(-(total[0] + low[0]), -(total[1] + low[1]), -(total[2] + low[2]), -(total[3] + low[3])));
  __syncthreads();
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  cd_mul(s.A[0], s.B[0], r, c, acc);
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
