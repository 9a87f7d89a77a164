// The one-launch factorisation of the innovation covariance (its source is appended to SOURCE by the test) on the
// CPU: factor, inverse and innovation solve of a random S under many schedules, with poisoned work space.
//   argv: m  seeds  resident CTAs  bad pivot (-1: none)  hold back after a release, after a barrier (chances)
#include "host_cuda.h"

namespace emu { Scheduler sched; }

enum { KF_OK = 0, KF_ERR_NOT_PD = 2, KF_ERR_NUMERIC = 3, KF_ERR_TIMEOUT = 7 };
namespace kfm {
constexpr uint64_t WAIT_NS = 2000000000ull;
constexpr int kInnovFactorMaxM = 1536;
inline bool status_failed(const int* st) { return *(volatile const int*)st != 0; }
inline void status_set(int* st, int code, int step, int index) {
  if (*st == 0) {
    st[0] = code;
    st[1] = step;
    st[2] = index;
  }
}
inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }
}  // namespace kfm

#include SOURCE

using namespace kfm;

int main(int argc, char** argv) {
  const int m = atoi(argv[1]), seeds = atoi(argv[2]), resident = atoi(argv[3]), bad = atoi(argv[4]);
  emu::sched.hold_release = atof(argv[5]);
  emu::sched.hold_barrier = atof(argv[6]);
  const int T = (int)ceil_div(m, 32), ldw = 32 * T;
  uint64_t r = 88172645463325252ull;
  auto uni = [&]() {
    r ^= r << 13;
    r ^= r >> 7;
    r ^= r << 17;
    return (double)(r >> 11) * 0x1p-53 - 0.5;
  };
  std::vector<double> G((size_t)m * m), S0((size_t)m * m), nu0(m);
  for (double& g : G) g = uni();
  for (int i = 0; i < m; ++i)
    for (int j = 0; j < m; ++j) {
      double s = i == j ? 1.0 + 0.01 * i : 0.0;
      for (int k = 0; k < m; ++k) s += G[(size_t)i * m + k] * G[(size_t)j * m + k];
      S0[(size_t)i * m + j] = s;
    }
  for (double& v : nu0) v = uni();
  if (bad >= 0)
    for (int j = 0; j < m; ++j) S0[(size_t)bad * m + j] = S0[(size_t)j * m + bad] = 0.0;
  // reference in extended precision
  std::vector<long double> L((size_t)m * m, 0.0L), X((size_t)m * m, 0.0L), y(m);
  if (bad < 0)
    for (int i = 0; i < m; ++i) {
      for (int j = 0; j <= i; ++j) {
        long double s = S0[(size_t)i * m + j];
        for (int k = 0; k < j; ++k) s -= L[(size_t)i * m + k] * L[(size_t)j * m + k];
        L[(size_t)i * m + j] = i == j ? sqrtl(s) : s / L[(size_t)j * m + j];
      }
      long double s = nu0[i];
      for (int k = 0; k < i; ++k) s -= L[(size_t)i * m + k] * y[k];
      y[i] = s / L[(size_t)i * m + i];
      for (int c = 0; c <= i; ++c) {
        long double t = i == c ? 1.0L : 0.0L;
        for (int k = c; k < i; ++k) t -= L[(size_t)i * m + k] * X[(size_t)k * m + c];
        X[(size_t)i * m + c] = t / L[(size_t)i * m + i];
      }
    }
  std::vector<int> flags(innovation_factor_flags(m), 0);
  const double nan = NAN;
  for (int seed = 1; seed <= seeds; ++seed) {
    std::vector<double> S = S0, nu = nu0, Linv((size_t)m * m, nan), dinv((size_t)T * 1024, nan);
    std::vector<double> W((size_t)m * ldw + 2, nan), Dt((size_t)T * 1024 + 2, nan);
    int status[4] = {0, 0, 0, 0};
    auto align = [](double* p) { return (double*)(((uintptr_t)p + 15) & ~(uintptr_t)15); };
    IfArgs a;
    a.m = m;
    a.T = T;
    a.S = S.data();
    a.lds = m;
    a.dinv = dinv.data();
    a.Linv = Linv.data();
    a.nu = nu.data();
    a.W = align(W.data());
    a.Dt = align(Dt.data());
    a.flags = flags.data();
    a.status = status;
    a.step = 5;
    const int full = 32 / kRowsPerCta + 1, last = (int)ceil_div(m - 32 * (T - 1), kRowsPerCta) + 1;
    const int grid = full * (T - 1) + last + 1 + m;
    const size_t smem = std::max(sizeof(DiagTile), (size_t)kRowsPerCta * 32 * T * sizeof(double));
    emu::sched.seed = 0x9E3779B97F4A7C15ull * seed + 1;
    if (!emu::sched.launch(grid, kIfThreads, smem, resident, [&] { innovation_factor_kernel(a); })) {
      printf("seed %d: deadlock\n", seed);
      return 1;
    }
    for (int f : flags)
      if (f) {
        printf("seed %d: flags left behind\n", seed);
        return 1;
      }
    if (bad >= 0) {
      if (status[0] != KF_ERR_NOT_PD || status[1] != 5 || status[2] != bad) {
        printf("seed %d: status %d step %d index %d\n", seed, status[0], status[1], status[2]);
        return 1;
      }
      continue;
    }
    if (status[0]) {
      printf("seed %d: status %d index %d\n", seed, status[0], status[2]);
      return 1;
    }
    double worst = 0;
    for (int i = 0; i < m; ++i) {
      for (int j = 0; j < m; ++j) {
        const double dx = fabs((double)(Linv[(size_t)i * m + j] - X[(size_t)i * m + j]));
        const double dl = j <= i ? fabs((double)(S[(size_t)i * m + j] - L[(size_t)i * m + j])) : 0.0;
        if (!(dx <= 1e-12) || !(dl <= 1e-12 * m)) {
          printf("seed %d: row %d column %d: L %g (%g) inverse %g (%g)\n", seed, i, j, S[(size_t)i * m + j],
                 (double)L[(size_t)i * m + j], Linv[(size_t)i * m + j], (double)X[(size_t)i * m + j]);
          return 1;
        }
        worst = std::max(worst, dx);
      }
      if (!(fabs((double)(nu[i] - y[i])) <= 1e-12)) {
        printf("seed %d: nu[%d]\n", seed, i);
        return 1;
      }
    }
    if (seed == seeds) printf("worst %g, %lld steps\n", worst, (long long)emu::sched.steps);
  }
  return 0;
}
