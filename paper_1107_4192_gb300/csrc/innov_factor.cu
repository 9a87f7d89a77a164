// Cholesky factor of the innovation covariance (eqn 8), its inverse and the solve of the innovation
// vector, S = L L^T, L^{-1} and L^{-1} nu, float64, in one launch.  The float64 path factors and inverts
// P_{t+1|t} (eqn 11) with it too, up to kInnovFactorMaxM sources.
//
// What bounds it: one warp's float64 instruction occupies its SM sub-partition for 64 cycles whatever
// the number of active lanes (measured; 19 cycles per instruction and SM when all four are busy), so
// the factorisation is a chain of m pivots (square root, reciprocal, scaled column: about 900 cycles
// each alone, 1300 beside the tile's updates and inverse) and every product has to be spread over many
// SMs.  Measured: m = 384 0.36 ms, m = 306 0.30 ms, m = 128 0.117 ms, m = 64 0.058 ms (0.9 us per
// pivot; 900 cycles are 0.43 us); as a sequence of launches of block kernels (32-wide leaves of one
// warp, 64 x 64 product tiles on one SM each) 1.87 ms and 0.32 ms at m = 306 and 64.
//
// Layout: 32-wide tiles, T = ceil(m / 32).  One warp per row of S (lane = column of the tile) does the
// row's panel products and updates in global dataflow order, one CTA per diagonal tile factors and
// inverts it, one CTA per row of L^{-1} forms it from the right, one warp does nu as an additional
// row below S.  Work is handed out by a ticket, and every task waits only on tasks with lower
// tickets (a row, for its own tile, on the rows above it alone: the diagonal tile is lower triangular),
// so the launch makes progress however many CTAs are resident.  Waits are bounded (2 s, then
// KF_ERR_TIMEOUT), and end when the status word reports a failure; the last CTA to finish clears the
// flags for the next launch.
//
// Every element gets the operations of the blocked right-looking algorithm of chol.cu with 32-wide
// blocks (potrf and trsm_right) in the same order: a sum over the 32 columns of a block from zero in
// increasing order, subtracted once; so L, L^{-1} and L^{-1} nu have the same bits (compared through
// kfx_innovation_factor).
#include "flag_ptx.cuh"
#include "ops.cuh"
#include "tc_ptx.cuh"

namespace kfm {

namespace {

constexpr int kRowsPerCta = 4;      // row tasks: one warp per SM sub-partition
constexpr int kIfThreads = 256;     // diagonal tiles use seven warps, the other tasks four
constexpr uint64_t kIfWaitNs = WAIT_NS;

struct IfArgs {
  int m, T;
  double* S;
  int64_t lds;
  double* dinv;   // T blocks of 32 x 32: inverses of the diagonal blocks
  double* Linv;   // m x m (row stride m), or null
  double* nu;     // m, or null
  double* W;      // L and the updated diagonal tiles, row stride 32 T
  double* Dt;     // the same, pairs of columns interleaved: D[c][kk] at ((kk / 2) 32 + c) 2 + kk mod 2
  int* flags;     // ticket, done, diag ready [T], diag rows updated [T], panel rows done [T x T]
  int* status;
  int step;
};

struct DiagTile {
  double A[32][33];   // A[k][i]: column k of the tile being factored; on output L[k][i] = L_ik
  double X[32][33];   // X[i][c]: rows of the inverse
  double q[32];       // 1 / L_jj
  int fail;
};
// The other tasks' shared memory: a row CTA holds kRowsPerCta rows of 32 T values; a row of L^{-1} its 32 T
// values X (as they become final) and T ready flags.

// Rows of tile i whose panel k is done, a bit per row.
__device__ __forceinline__ int* rows_word(const IfArgs& a, int k, int i) { return a.flags + 2 + 2 * a.T + k * a.T + i; }

// One warp waits until *flag has reached want (a count), or holds all of want's bits (BITS); false when the wait
// expired or another task failed.
template <bool BITS = false>
__device__ __forceinline__ bool wait_flag(const int* flag, int want, const IfArgs& a, int lane, int sleep_ns) {
  auto reached = [&](int v) { return BITS ? (v & want) == want : v >= want; };
  int ok = 1;
  if (lane == 0) {
    if (!reached(ld_acquire(flag))) {
      const uint64_t t0 = globaltimer();
      for (int n = 1;; ++n) {
        if (reached(ld_acquire(flag))) break;
        if ((n & 15) == 0) {
          if (status_failed(a.status)) { ok = 0; break; }
          if (globaltimer() - t0 > kIfWaitNs) {
            status_set(a.status, KF_ERR_TIMEOUT, a.step, 21);
            ok = 0;
            break;
          }
        }
        if (sleep_ns) __nanosleep(sleep_ns);
      }
    }
  }
  ok = __shfl_sync(0xffffffffu, ok, 0);
  __syncwarp();  // orders the other lanes' reads after lane 0's acquire; the exchange alone does not
  return ok != 0;
}

__device__ __forceinline__ double half_of(double x) {  // x / 2 for a normal x, without the float64 unit
  return __longlong_as_double(__double_as_longlong(x) - (1ll << 52));
}

// l = sqrt(d) and q = 1 / l, both rounded to nearest, by all lanes of a warp together: a float32
// estimate of 1 / sqrt(d), one Newton step for it and for sqrt(d) (the same instruction on even and
// odd lanes), then one correction each from an exact residual (fused multiply-add), which leaves an
// error of about 2^-94 before the last rounding (Markstein's scheme; checked bit for bit against
// correctly rounded square roots and reciprocals through kfx_innovation_factor).  Seven dependent float64 instructions instead of about fifteen.
// Pivots outside 2^+-100 (or not positive) take the library functions.
__device__ __forceinline__ void pivot_warp(double d, int lane, double& q, double& l) {
  const int ex = (__double2hiint(d) >> 20) & 0xfff;  // sign and exponent
  if (ex < 1023 - 100 || ex > 1023 + 100) {
    l = sqrt(d);
    q = 1.0 / l;
    return;
  }
  const float df = (float)d;
  float yf = rsqrtf(df);
  yf = fmaf(0.5f * yf, fmaf(-df * yf, yf, 1.0f), yf);
  const double y = (double)yf;
  const double g = __dmul_rn(d, y);
  const double r = __fma_rn(-g, y, 1.0);
  const double b = (lane & 1) ? g : y;
  const double t = __fma_rn(half_of(b), r, b);
  const double q0 = __shfl_sync(0xffffffffu, t, 0), l0 = __shfl_sync(0xffffffffu, t, 1);
  const double e = __fma_rn(-l0, l0, d);
  l = __fma_rn(e, half_of(q0), l0);
  if ((__double_as_longlong(l) & 0xFFFFFFFFFFFFFll) == 0xFFFFFFFFFFFFFll) {  // the scheme's one exception
    q = 1.0 / l;
    return;
  }
  const double e2 = __fma_rn(-l, q0, 1.0);
  q = __fma_rn(e2, q0, q0);
}

// Diagonal tile: warp 0 runs the pivot chain alone on its sub-partition; warps 1-3 hold the tile's
// columns in registers (lane = row, column k on warp 1 + k mod 3), and hand column j + 1 and the
// diagonal element after it to warp 0 first; warps 5-7 hold the inverse (lane = column, row i on warp
// 5 + i mod 3), one step behind.  Everything but the step's float64 instructions is unrolled and
// loaded ahead: with the tile's elements packed densely over the threads instead (fewer instructions,
// each behind a predicate and its own loads) a column took 1370 cycles.
__device__ void factor_tile(DiagTile& s, const IfArgs& a, int tile, int warp, int lane) {
  const int n = min(32, a.m - 32 * tile);
  const int ldw = 32 * a.T;
  if (threadIdx.x == 0) s.fail = 0;
  const int want = n;
  const bool ok = wait_flag(a.flags + 2 + a.T + tile, want, a, lane, 0);
  if (!__syncthreads_and(ok)) return;
  for (int e = threadIdx.x; e < 1024; e += kIfThreads) {
    const int i = e / 32, k = e % 32;
    double v = i == k ? 1.0 : 0.0;
    if (i < n && k < n) v = k <= i ? a.W[(int64_t)(32 * tile + i) * ldw + 32 * tile + k] : 0.0;
    s.A[k][i] = v;
    s.X[i][k] = 0.0;
  }
  __syncthreads();
  constexpr int kAll = 7 * 32, kColBar = 4 * 32, kInvBar = 3 * 32;
  if (warp == 0) {
    double d = s.A[0][0];
    int bad = -1;
    for (int j = 0; j < 32; ++j) {
      double q, l;
      if (bad < 0 && !(d > 0.0 && d < INFINITY)) bad = j;
      pivot_warp(d, lane, q, l);
      if (j > 0) bar_sync(3 + (j & 1), kColBar);  // column j and the diagonal element of column j + 1
      const double li = lane > j ? __dmul_rn(s.A[j][lane], q) : (lane == j ? l : 0.0);
      if (j < 31) {
        const double dn = s.A[j + 1][j + 1];
        const double lj = __shfl_sync(0xffffffffu, li, j + 1);
        d = __fma_rn(-lj, lj, dn);
      }
      s.A[j][lane] = li;
      if (lane == 0) s.q[j] = q;
      __syncwarp();
      bar_arrive(1 + (j & 1), kAll);
    }
    if (lane == 0 && bad >= 0) {
      s.fail = 1;
      status_set(a.status, KF_ERR_NOT_PD, a.step, 32 * tile + bad);
    }
  } else if (warp < 4) {
    const int w = warp - 1;
    double r[11];  // column 3 sl + w
#pragma unroll
    for (int sl = 0; sl < 11; ++sl) r[sl] = s.A[min(3 * sl + w, 31)][lane];
#pragma unroll
    for (int j = 0; j < 31; ++j) {
      bar_sync(1 + (j & 1), kAll);  // column j of L
      const double li = -s.A[j][lane];
      double lk[11];
#pragma unroll
      for (int sl = (j + 1) / 3; sl < 11; ++sl) lk[sl] = s.A[j][min(3 * sl + w, 31)];
      const int c1 = j + 1, c2 = j + 2;
      if (w == c1 % 3) {
        r[c1 / 3] = __fma_rn(li, lk[c1 / 3], r[c1 / 3]);
        s.A[c1][lane] = r[c1 / 3];
      } else if (c2 < 32 && w == c2 % 3) {
        r[c2 / 3] = __fma_rn(li, lk[c2 / 3], r[c2 / 3]);
        if (lane == c2) s.A[c2][lane] = r[c2 / 3];
      }
      __syncwarp();
      bar_arrive(3 + (c1 & 1), kColBar);
#pragma unroll
      for (int sl = c1 / 3; sl < 11; ++sl) {
        // columns above j + 2, and this warp's one if it is not among those two (all warp-uniform)
        const int k = 3 * sl + w;
        if (k > c2 && k < 32) r[sl] = __fma_rn(li, lk[sl], r[sl]);
      }
    }
    bar_sync(1 + (31 & 1), kAll);
  } else if (warp > 4) {
    const int w = warp - 5;
    double x[11];  // row 3 sl + w
#pragma unroll
    for (int sl = 0; sl < 11; ++sl) x[sl] = lane == 3 * sl + w ? 1.0 : 0.0;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      bar_sync(1 + (k & 1), kAll);  // column k of L and 1 / L_kk
      double lv[11];
#pragma unroll
      for (int sl = k / 3; sl < 11; ++sl) lv[sl] = -s.A[k][min(3 * sl + w, 31)];
      if (w == k % 3) s.X[k][lane] = __dmul_rn(x[k / 3], s.q[k]);
      bar_sync(5, kInvBar);
      const double xk = s.X[k][lane];
#pragma unroll
      for (int sl = k / 3; sl < 11; ++sl) {
        const int i = 3 * sl + w;
        if (i > k && i < 32) x[sl] = __fma_rn(lv[sl], xk, x[sl]);
      }
    }
  }
  __syncthreads();
  if (s.fail) return;
  // the rows below wait for Dt; L and the row-ordered inverse follow with a second count
#pragma unroll
  for (int u = 0; u < 512 / kIfThreads; ++u) {
    const int e = threadIdx.x + u * kIfThreads, c = e % 32, kk = 2 * (e / 32);
    reinterpret_cast<double2*>(a.Dt + (int64_t)tile * 1024)[e] = make_double2(s.X[c][kk], s.X[c][kk + 1]);
  }
  __syncthreads();
  if (threadIdx.x == 0) red_release(a.flags + 2 + tile, 1);
  for (int e = threadIdx.x; e < 1024; e += kIfThreads) {
    const int i = e / 32, c = e % 32;
    a.dinv[(int64_t)tile * 1024 + e] = s.X[i][c];
    if (i < n && c <= i) a.S[(int64_t)(32 * tile + i) * a.lds + 32 * tile + c] = s.A[c][i];
  }
  __syncthreads();
  if (threadIdx.x == 0) red_release(a.flags + 2 + tile, 1);
}

// Wait of a row CTA's four warps: warp 0 polls for all (one poll per warp slowed the data down), and the barrier
// itself carries its result: a flag in shared memory could already be the next wait's when a late warp reads it, and
// that warp would leave the others at their barrier for good.
template <bool BITS = false>
__device__ __forceinline__ bool wait_flag_rows(const int* flag, int want, const IfArgs& a, int warp, int lane, int sleep_ns) {
  const bool failed = warp == 0 && !wait_flag<BITS>(flag, want, a, lane, sleep_ns);
  return !bar_or(6, 32 * kRowsPerCta, failed);
}

// Four rows of one tile of S, a row per warp (or the innovation as row m, warp 0): for each panel k left
// of the rows' diagonal tile, L[r, k] = A[r, k] L_kk^{-T}, then A[r, i] -= L[r, k] L[i, k]^T for the
// tiles i > k of the row.
__device__ void row_task(double* row, const IfArgs& a, bool is_nu, int r, int warp, int lane) {
  const bool live = is_nu ? warp == 0 : r < a.m;
  const int tr = is_nu ? a.T : r / 32, ldw = 32 * a.T;
  const int ncols = live ? (is_nu ? a.m : min(a.m, 32 * (tr + 1))) : 0;
  const int last = is_nu ? a.T - 1 : tr;  // last column tile of the row
  const int* diag_ready = a.flags + 2;
  int bad = -1;
  for (int j = lane; j < 32 * (last + 1); j += 32) {
    const double v = j < ncols ? (is_nu ? a.nu[j] : a.S[(int64_t)r * a.lds + j]) : 0.0;
    if (is_nu && bad < 0 && !isfinite(v)) bad = j;
    row[j] = v;
  }
  __syncwarp();
  for (int k = 0; k < tr; ++k) {
    if (!wait_flag_rows(diag_ready + k, 1, a, warp, lane, 20)) return;
    const double2* D = reinterpret_cast<const double2*>(a.Dt + (int64_t)k * 1024) + lane;
    double2 dv[16];  // row `lane` of L_kk^{-1}
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) dv[kk] = ld2(D + 32 * kk);
    if (live) {
      double acc = 0.0;
#pragma unroll
      for (int kk = 0; kk < 16; ++kk) {
        acc = __fma_rn(row[32 * k + 2 * kk], dv[kk].x, acc);
        acc = __fma_rn(row[32 * k + 2 * kk + 1], dv[kk].y, acc);
      }
      __syncwarp();
      row[32 * k + lane] = acc;
      if (!is_nu) {
        a.W[(int64_t)r * ldw + 32 * k + lane] = acc;
        __syncwarp();
        if (lane == 0) or_release(rows_word(a, k, tr), (int)(1u << (r & 31)));
        a.S[(int64_t)r * a.lds + 32 * k + lane] = acc;
      }
      __syncwarp();
    }
    for (int i = k + 1; i <= last; ++i) {
      // the tile's rows; of the rows' own tile those up to the CTA's last one (r - warp is its first)
      const int rows = min(min(32, a.m - 32 * i), i == tr ? (r - warp) % 32 + kRowsPerCta : 32);
      if (!wait_flag_rows<true>(rows_word(a, k, i), rows == 32 ? -1 : (1 << rows) - 1, a, warp, lane, 0)) return;
      if (!live) continue;
      const int c = 32 * i + lane;
      // rows of L beyond m do not exist, and those below r do not matter to it: their lanes read the tile's first row
      // and drop the result
      const bool mine = c < a.m && c <= r;
      const double2* Lc = reinterpret_cast<const double2*>(a.W + (int64_t)(mine ? c : 32 * i) * ldw + 32 * k);
      double2 lv[16];
#pragma unroll
      for (int kk = 0; kk < 16; ++kk) lv[kk] = ld2(Lc + kk);
      double s = 0.0;
#pragma unroll
      for (int kk = 0; kk < 16; ++kk) {
        s = __fma_rn(row[32 * k + 2 * kk], lv[kk].x, s);
        s = __fma_rn(row[32 * k + 2 * kk + 1], lv[kk].y, s);
      }
      if (mine) row[c] = __dsub_rn(row[c], s);
    }
    __syncwarp();
  }
  if (!live) return;
  if (is_nu) {
    for (int j = lane; j < a.m; j += 32) a.nu[j] = row[j];
    // a non-finite innovation is reported after the factor, which has succeeded at this point
    if (bad >= 0) status_set(a.status, KF_ERR_NUMERIC, a.step, bad);
  } else {
    a.W[(int64_t)r * ldw + 32 * tr + lane] = row[32 * tr + lane];
    __syncwarp();
    if (lane == 0) red_release(a.flags + 2 + a.T + tr, 1);
  }
}

// Row r of L^{-1}, four warps: X_k for the row's tiles k = tr .. 0 with
// X_j = (0 - X_tr L[tr, j] - .. - X_{j+1} L[j+1, j]) L_jj^{-1}; warp w owns the tiles j = w mod 4 and
// applies the X_k that are ready while it waits for the last one.  Of tile j it needs the second count: the rows of
// tile tr have waited for the first alone, which does not cover dinv.
__device__ void inverse_row(double* B, int* ready_flags, const IfArgs& a, int r, int warp, int lane) {
  const int tr = r / 32, ldw = 32 * a.T;
  if (!wait_flag(a.flags + 2 + tr, 2, a, lane, 100)) return;
  double* out = a.Linv + (int64_t)r * a.m;
  volatile int* ready = ready_flags;
  for (int j = tr - 1 - ((tr - 1 - warp) & 3); j >= 0; j -= 4) {
    if (!wait_flag(a.flags + 2 + j, 2, a, lane, 0)) return;
    const double* D = a.dinv + (int64_t)j * 1024 + lane;
    double b = 0.0;
    double dv[32];
#pragma unroll
    for (int kk = 0; kk < 32; ++kk) dv[kk] = D[32 * kk];
    for (int k = tr; k > j; --k) {
      const int nk = min(32, a.m - 32 * k);
      const double* L = a.W + (int64_t)(32 * k) * ldw + 32 * j + lane;
      double lv[32];
#pragma unroll
      for (int kk = 0; kk < 32; ++kk) lv[kk] = kk < nk ? L[(int64_t)kk * ldw] : 0.0;
      const double* X;
      if (k == tr) {
        X = a.dinv + (int64_t)tr * 1024 + 32 * (r - 32 * tr);
      } else {
        int ok = 1;
        if (lane == 0 && !ready[k]) {
          const uint64_t t0 = globaltimer();
          while (!ready[k]) {
            if (status_failed(a.status)) {  // another warp of the row may have stopped at it
              ok = 0;
              break;
            }
            if (globaltimer() - t0 > kIfWaitNs) {
              status_set(a.status, KF_ERR_TIMEOUT, a.step, 22);
              ok = 0;
              break;
            }
          }
        }
        if (!__shfl_sync(0xffffffffu, ok, 0)) return;
        __syncwarp();
        __threadfence_block();
        X = B + 32 * k;
      }
      double acc = 0.0;
#pragma unroll
      for (int kk = 0; kk < 32; ++kk)
        if (kk < nk) acc = __fma_rn(X[kk], lv[kk], acc);
      b = __dsub_rn(b, acc);
    }
    B[32 * j + lane] = b;
    __syncwarp();
    double acc = 0.0;
#pragma unroll
    for (int kk = 0; kk < 32; ++kk) acc = __fma_rn(B[32 * j + kk], dv[kk], acc);
    __syncwarp();
    B[32 * j + lane] = acc;
    __threadfence_block();
    __syncwarp();
    if (lane == 0) ready[j] = 1;
    out[32 * j + lane] = acc;
  }
  // the diagonal tile's part, and the zeros above the diagonal
  for (int c = 32 * tr + threadIdx.x; c < a.m; c += 128)
    out[c] = c < 32 * (tr + 1) ? a.dinv[(int64_t)tr * 1024 + 32 * (r - 32 * tr) + c - 32 * tr] : 0.0;
}

__global__ void __launch_bounds__(kIfThreads) innovation_factor_kernel(const IfArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* rows = reinterpret_cast<double*>(smem_raw);
  int* ready = reinterpret_cast<int*>(rows + 32 * a.T);
  __shared__ int ticket_s;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (threadIdx.x == 0) ticket_s = status_failed(a.status) ? -1 - atomicAdd(a.flags, 1) : atomicAdd(a.flags, 1);
  for (int e = threadIdx.x; e < a.T; e += kIfThreads) ready[e] = 0;
  __syncthreads();
  const int ticket = ticket_s;
  // tickets: per tile its row CTAs, then its diagonal tile; then the innovation; then the rows of L^{-1}
  const int full = 32 / kRowsPerCta + 1;
  const int last_rows = a.m - 32 * (a.T - 1), last_units = (last_rows + kRowsPerCta - 1) / kRowsPerCta + 1;
  const int nfac = full * (a.T - 1) + last_units;
  if (ticket >= 0) {
    if (ticket < nfac) {
      const int tile = min(ticket / full, a.T - 1), u = ticket - tile * full;
      const int units = tile == a.T - 1 ? last_units : full;
      if (u == units - 1) {
        factor_tile(*reinterpret_cast<DiagTile*>(smem_raw), a, tile, warp, lane);
      } else if (warp < kRowsPerCta) {
        row_task(rows + warp * 32 * a.T, a, false, 32 * tile + kRowsPerCta * u + warp, warp, lane);
      }
    } else if (a.nu && ticket == nfac) {
      if (warp < kRowsPerCta) row_task(rows + warp * 32 * a.T, a, true, a.m, warp, lane);
    } else if (warp < 4) {
      const int r = ticket - nfac - (a.nu ? 1 : 0);
      inverse_row(rows, ready, a, r, warp, lane);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    ticket_s = atomicAdd(a.flags + 1, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (ticket_s) {  // every other CTA has finished: clear the flags for the next launch
    __threadfence();
    for (int e = threadIdx.x; e < 2 + 2 * a.T + a.T * a.T; e += kIfThreads) a.flags[e] = 0;
  }
}

}  // namespace

size_t innovation_factor_flags(int64_t m) {
  const int64_t T = ceil_div(m, 32);
  return (size_t)(2 + 2 * T + T * T);
}

kf_status innovation_factor(cudaStream_t s, int m, double* S, int64_t lds, double* dinv, double* Linv, double* nu,
                            double* W, double* Dt, int* flags, int* status, int step) {
  if (m < 1 || m > kInnovFactorMaxM || !S || !dinv || !W || !Dt || !flags) return KF_ERR_ARG;
  if ((reinterpret_cast<uintptr_t>(W) | reinterpret_cast<uintptr_t>(Dt)) & 15) return KF_ERR_ARG;
  IfArgs a;
  a.m = m;
  a.T = (int)ceil_div(m, 32);
  a.S = S;
  a.lds = lds;
  a.dinv = dinv;
  a.Linv = Linv;
  a.nu = nu;
  a.W = W;
  a.Dt = Dt;
  a.flags = flags;
  a.status = status;
  a.step = step;
  const int full = 32 / kRowsPerCta + 1;
  const int last_units = (int)ceil_div(m - 32 * (a.T - 1), kRowsPerCta) + 1;
  const int grid = full * (a.T - 1) + last_units + (nu ? 1 : 0) + (Linv ? m : 0);
  const size_t smem = std::max(sizeof(DiagTile), (size_t)kRowsPerCta * 32 * a.T * sizeof(double));
  static_assert(kRowsPerCta >= 2, "a row of the inverse and its flags fit");
  KF_CUDA_TRY(smem_limit_per_device((const void*)innovation_factor_kernel,
                                    kRowsPerCta * (kInnovFactorMaxM + 32) * (int)sizeof(double)));
  innovation_factor_kernel<<<grid, kIfThreads, smem, s>>>(a);
  note_launch();
  return launch_check("innovation_factor");
}

}  // namespace kfm
