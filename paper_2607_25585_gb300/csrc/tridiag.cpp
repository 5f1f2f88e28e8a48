// Host half of FTLM (Eqs. 4-5 of arxiv 2607.25585): the tridiagonal
// eigenproblem of every Lanczos run and the Boltzmann sums.
//
// The eigenproblem uses the implicit QL iteration with shifts for symmetric
// tridiagonal matrices (Bowdler, Martin, Reinsch and Wilkinson, Numer. Math.
// 11, 1968).  The sums need only two rows of the eigenvector matrix U:
// U_0n (the weight <n|r>) and sum_j conj(p_j) U_jn (= <r|O|n>), so instead of
// accumulating the whole of U the plane rotations are applied to those row
// vectors only: O(M^2) per run instead of O(M^3).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <functional>
#include <limits>
#include <string>
#include <thread>
#include <utility>
#include <vector>

#include "ftlm_internal.h"

namespace ftlm {

namespace {

// sqrt(a^2 + b^2): the plain formula where the squares can neither overflow
// nor underflow, the library's careful hypot elsewhere
inline double norm2(double a, double b) {
  const double m = std::max(std::fabs(a), std::fabs(b));
  if (m < 1e150 && m > 1e-150) return std::sqrt(a * a + b * b);
  return std::hypot(a, b);
}

// Estimated cost of one run's eigenproblem with `rows` rotated rows, and of one
// (temperature, Ritz value) term of the sums, in nanoseconds (measured on the
// Grace cores: 16 us for 24 rows, 190 us for 100; 4 ns a term).
double ql_ns(int m, int rows) { return 1.7 * m * m * (8.0 + 1.2 * rows); }
constexpr double kTermNs = 4.0;

// Eigenvalues of tridiag(d, e) (d[0..m-1], e[0..m-2] off-diagonal) with the
// rotations applied to the rows z[k][0..m-1], k < nz.  Returns false if the
// iteration does not converge.
bool ql_implicit(int m, double* d, double* e_in, int nz, double** z) {
  std::vector<double> e(m, 0.0);
  for (int i = 0; i + 1 < m; ++i) e[i] = e_in[i];
  const double eps = std::numeric_limits<double>::epsilon();
  for (int l = 0; l < m; ++l) {
    int iter = 0;
    while (true) {
      int mm = l;
      for (; mm < m - 1; ++mm) {
        const double dd = std::fabs(d[mm]) + std::fabs(d[mm + 1]);
        if (std::fabs(e[mm]) <= eps * dd) break;
      }
      if (mm == l) break;
      if (++iter > 100) return false;
      // shift from the leading 2x2 block
      double g = (d[l + 1] - d[l]) / (2.0 * e[l]);
      double r = norm2(g, 1.0);
      g = d[mm] - d[l] + e[l] / (g + (g >= 0 ? r : -r));
      double s = 1.0, c = 1.0, p = 0.0;
      int i = mm - 1;
      bool deflated = false;
      for (; i >= l; --i) {
        const double f = s * e[i], b = c * e[i];
        r = norm2(f, g);
        e[i + 1] = r;
        if (r == 0.0) {  // underflow: split the matrix here
          d[i + 1] -= p;
          e[mm] = 0.0;
          deflated = true;
          break;
        }
        s = f / r;
        c = g / r;
        g = d[i + 1] - p;
        r = (d[i] - g) * s + 2.0 * c * b;
        p = s * r;
        d[i + 1] = g + p;
        g = c * r - b;
        for (int k = 0; k < nz; ++k) {
          const double zi = z[k][i], zi1 = z[k][i + 1];
          z[k][i + 1] = s * zi + c * zi1;
          z[k][i] = c * zi - s * zi1;
        }
      }
      if (deflated) continue;
      d[l] -= p;
      e[l] = g;
      e[mm] = 0.0;
    }
  }
  return true;
}

// fn(i) for i in [0, n), each exactly once, on the caller's thread and as many
// others as the work pays for: starting and joining a thread costs some 60 us,
// so each gets at least 200 us of `total_ns` (ten eigenproblems of 24 rows and
// their sums, 0.2 ms on one thread, took 0.4 ms on six and 1.5 ms on ten and more).
// false: an item threw (out of memory).
bool parallel_for(int n, double total_ns, const std::function<void(int)>& fn) {
  const int hw = (int)std::max(1u, std::thread::hardware_concurrency());
  const int nth = std::min({n, hw, 32, 1 + (int)std::min(1e6, total_ns / 200e3)});
  std::atomic<int> next{0};
  std::atomic<bool> ok{true};
  auto work = [&]() {
    try {
      for (int i; (i = next.fetch_add(1)) < n;) fn(i);
    } catch (...) {
      ok = false;
    }
  };
  std::vector<std::thread> pool;
  try {
    for (int k = 1; k < nth; ++k) pool.emplace_back(work);
  } catch (...) {  // fewer threads: the others take the remaining items
  }
  work();
  for (auto& t : pool) t.join();
  return ok;
}

// One run's eigenproblem: its Ritz values, the weights' row U_0n and the rows Re, Im
// of sum_j conj(p_j) U_jn.
// (In the system's one block: four vectors a run, allocated by one thread and freed by
// another, took 0.5 ms of a batch of 24 systems of 48 vectors.)
struct Ritz {
  double *eps = nullptr, *w0 = nullptr, *qr = nullptr, *qi = nullptr;
  int m = 0;
};

// null, or what is wrong with run r
const char* solve_run(const HostSums& s, int r, Ritz& run) {
  const int m = s.M_eff[r];
  auto at = [&](int j) { return r * s.run + j * s.step; };
  run.m = m;
  for (int j = 0; j < m; ++j) run.eps[j] = s.alpha[at(j)];
  std::vector<double> e(m > 1 ? m - 1 : 1, 0.0);
  for (int j = 0; j + 1 < m; ++j) e[j] = s.beta[at(j)];
  std::fill(run.w0, run.w0 + m, 0.0);
  run.w0[0] = 1.0;
  for (int j = 0; j < m; ++j) {  // conj(p_j)
    run.qr[j] = s.p[2 * at(j)];
    run.qi[j] = -s.p[2 * at(j) + 1];
  }
  for (int j = 0; j < m; ++j)
    if (!std::isfinite(run.eps[j]) || (j + 1 < m && !std::isfinite(e[j]))) return "non-finite Lanczos coefficient in run ";
  double* rows[3] = {run.w0, run.qr, run.qi};
  return ql_implicit(m, run.eps, e.data(), 3, rows) ? nullptr : "tridiagonal eigensolver did not converge (run ";
}

// the results at temperature t, from the solved runs in order
void sum_runs(const HostSums& s, const std::vector<Ritz>& runs, double E0, int t) {
  const double b = 1.0 / s.T[t];
  double z = 0.0, e1 = 0.0, orr = 0.0, oi = 0.0;
  std::vector<double> ws;  // the weights, for the variance
  ws.reserve((size_t)s.R * s.M);
  for (const Ritz& run : runs)
    for (int n = 0; n < run.m; ++n) {
      const double boltz = std::exp(-b * (run.eps[n] - E0));
      const double w = run.w0[n] * run.w0[n] * boltz;
      ws.push_back(w);
      z += w;
      e1 += w * run.eps[n];
      orr += boltz * run.w0[n] * run.qr[n];
      oi += boltz * run.w0[n] * run.qi[n];
    }
  const double Em = e1 / z;
  double var = 0.0;
  const double* w = ws.data();
  for (const Ritz& run : runs)
    for (int n = 0; n < run.m; ++n) var += *w++ * (run.eps[n] - Em) * (run.eps[n] - Em);
  ftlm_result* res = s.res;
  if (res->lnZ) res->lnZ[t] = std::log(s.dim / s.R * z) - b * E0;
  if (res->E) res->E[t] = Em;
  if (res->C) res->C[t] = b * b * var / z;
  if (res->M_B) res->M_B[t] = -s.g * orr / z;
  if (res->M_B_imag) res->M_B_imag[t] = -s.g * oi / z;
}
// the coefficients to the caller's arrays
void store_runs(const HostSums& s) {
  const ftlm_result& o = *s.res;
  for (int r = 0; r < s.R; ++r) {
    if (o.M_eff) o.M_eff[r] = s.M_eff[r];
    for (int j = 0; j < s.M; ++j) {
      const size_t to = (size_t)r * s.M + j, at = r * s.run + j * s.step;
      if (o.alpha) o.alpha[to] = s.alpha[at];
      if (o.beta) o.beta[to] = s.beta[at];
      if (o.p) {
        o.p[2 * to] = s.p[2 * at];
        o.p[2 * to + 1] = s.p[2 * at + 1];
      }
    }
  }
}

}  // namespace

// All systems' eigenproblems, then all their temperatures, as one list of items: a
// batch of two long runs keeps as many threads busy as a batch of many short ones
// (2 x 64 vectors of 200 steps: a thread a system took 52 ms).  An item is as many of a
// system's eigenproblems, or temperatures, as make 50 us: one of 8 steps takes 1 us, and
// the threads would spend as long passing each other the counters (24 systems of 48
// vectors: 0.7 ms more).  A temperature's item comes after every eigenproblem's, so
// those that it may have to wait for are being solved on other threads.
void host_sums_many(std::vector<HostSums>& sums) {
  struct Work {
    std::vector<double> block;  // [R][4][M]
    std::vector<Ritz> runs;
    std::vector<const char*> bad;
    std::atomic<int> left{0};
    std::atomic<bool> memory{false};
    double E0 = std::numeric_limits<double>::infinity();
  };
  const int n = (int)sums.size();
  std::vector<Work> work(n);
  struct Item {
    int k, from, to;  // system; its runs, or its temperatures
  };
  std::vector<Item> solve, sum;
  auto divide = [](std::vector<Item>& items, int k, int count, double each_ns) {
    const int step = (int)std::min<double>(count, std::max(1.0, 50e3 / each_ns));
    for (int i = 0; i < count; i += step) items.push_back({k, i, std::min(count, i + step)});
  };
  double ns = 0.0;
  for (int k = 0; k < n; ++k) {
    HostSums& s = sums[k];
    s.status = FTLM_ERR_INVALID_ARG;
    if (s.R < 1 || s.M < 1 || !s.M_eff || !s.alpha || !s.beta || !s.p || !s.T || s.nT < 1 || !s.res || !(s.dim > 0)) {
      s.msg = "ftlm_sums: invalid arguments";
      continue;
    }
    s.msg.clear();
    for (int t = 0; t < s.nT; ++t)
      if (!(s.T[t] > 0.0) || !std::isfinite(s.T[t])) s.msg = "temperatures must be positive and finite";
    for (int r = 0; r < s.R && s.msg.empty(); ++r)
      if (s.M_eff[r] < 1 || s.M_eff[r] > s.M) s.msg = "M_eff out of range";
    if (!s.msg.empty()) continue;
    s.status = FTLM_OK;
    work[k].block.resize((size_t)4 * s.R * s.M);
    work[k].runs.resize(s.R);
    for (int r = 0; r < s.R; ++r) {
      double* b = work[k].block.data() + (size_t)4 * r * s.M;
      work[k].runs[r] = {b, b + s.M, b + 2 * s.M, b + 3 * s.M, 0};
    }
    work[k].bad.assign(s.R, nullptr);
    work[k].left = s.R;
    divide(solve, k, s.R, ql_ns(s.M, 3));
    divide(sum, k, s.nT, kTermNs * s.M * s.R);
    ns += s.R * (ql_ns(s.M, 3) + kTermNs * s.M * s.nT);
  }
  parallel_for((int)(solve.size() + sum.size()), ns, [&](int i) {
    if (i < (int)solve.size()) {
      const Item it = solve[i];
      Work& w = work[it.k];
      try {
        for (int r = it.from; r < it.to; ++r) w.bad[r] = solve_run(sums[it.k], r, w.runs[r]);
      } catch (...) {
        w.memory = true;
      }
      if (w.left.fetch_sub(it.to - it.from) == it.to - it.from) {  // the system's last: its lowest Ritz value
        for (const Ritz& run : w.runs)
          for (int n = 0; n < run.m; ++n) w.E0 = std::min(w.E0, run.eps[n]);
        w.left.store(-1);
      }
      return;
    }
    const Item it = sum[i - solve.size()];
    Work& w = work[it.k];
    while (w.left.load() >= 0) std::this_thread::yield();
    for (const char* b : w.bad)
      if (b || w.memory) return;
    if (it.from == 0 && sums[it.k].store) store_runs(sums[it.k]);
    try {
      for (int t = it.from; t < it.to; ++t) sum_runs(sums[it.k], w.runs, w.E0, t);
    } catch (...) {
      w.memory = true;
    }
  });
  for (int k = 0; k < n; ++k) {
    HostSums& s = sums[k];
    if (s.status != FTLM_OK) continue;
    if (work[k].memory) {
      s.status = FTLM_ERR_OUT_OF_MEMORY;
      s.msg = "out of host memory";
      continue;
    }
    for (int r = 0; r < s.R && s.status == FTLM_OK; ++r)
      if (const char* b = work[k].bad[r]) {
        s.status = FTLM_ERR_NUMERICAL;
        s.msg = b + std::to_string(r) + (std::strchr(b, '(') ? ")" : "");
      }
    if (s.status == FTLM_OK) s.res->E0 = work[k].E0;
  }
}

ftlm_status host_sums(int R, int M, const int* M_eff, const double* alpha, const double* beta, const double* p,
                      double dim, double g, const double* T, int nT, ftlm_result* res, std::string& msg) {
  std::vector<HostSums> one(1);
  one[0] = {R, M, M_eff, alpha, beta, p, (size_t)std::max(0, M), 1, false, dim, g, T, nT, res};
  host_sums_many(one);
  msg = one[0].msg;
  return one[0].status;
}

// Symmetric FTLM for O = u.S, Eqs. (E-2-G), (E-2-H): per run,
//   num_r = sum_{m,n} e^{-beta (eps_m + eps_n)/2} U_0m <m|O|n> U_0n = y^T O y,
//   y_i = sum_n U_in e^{-beta eps_n / 2} U_0n,
// with O_ij = <v_i|O|v_j> in the Lanczos basis (<m|O|n> = (U^T O U)_mn, U real),
// den_r = sum_n e^{-beta eps_n} U_0n^2; both shifted by E0, the lowest Ritz value
// over all runs.  Omat[r][i][j] (complex, row-major, M x M per run).  The whole
// of U is accumulated here: O(M^3) per run.
ftlm_status host_sums_sym(int R, int M, const int* M_eff, const double* alpha, const double* beta,
                          const double* Omat, double g, const double* T, int nT, double* MB_sym, double* MB_sym_imag,
                          std::string& msg) {
  if (R < 1 || M < 1 || !M_eff || !alpha || !beta || !Omat || !T || nT < 1) {
    msg = "sFTLM sums: invalid arguments";
    return FTLM_ERR_INVALID_ARG;
  }
  struct Run {
    int m = 0;
    std::vector<double> eps, U;  // U[k * m + n] = U_kn
  };
  std::vector<Run> runs(R);
  for (int r = 0; r < R; ++r)
    if (M_eff[r] < 1 || M_eff[r] > M) {
      msg = "M_eff out of range";
      return FTLM_ERR_INVALID_ARG;
    }
  std::vector<int> bad(R, 0);
  const bool solved = parallel_for(R, R * ql_ns(M, M), [&](int r) {
    Run& run = runs[r];
    const int m = run.m = M_eff[r];
    run.eps.assign(alpha + (size_t)r * M, alpha + (size_t)r * M + m);
    std::vector<double> e(m > 1 ? m - 1 : 1, 0.0);
    for (int j = 0; j + 1 < m; ++j) e[j] = beta[(size_t)r * M + j];
    run.U.assign((size_t)m * m, 0.0);
    std::vector<double*> rows(m);
    for (int k = 0; k < m; ++k) {
      run.U[(size_t)k * m + k] = 1.0;
      rows[k] = run.U.data() + (size_t)k * m;
    }
    if (!ql_implicit(m, run.eps.data(), e.data(), m, rows.data())) bad[r] = 1;
  });
  if (!solved) return msg = "out of host memory", FTLM_ERR_OUT_OF_MEMORY;
  double E0 = std::numeric_limits<double>::infinity();
  for (int r = 0; r < R; ++r) {
    if (bad[r]) {
      msg = "tridiagonal eigensolver did not converge (run " + std::to_string(r) + ")";
      return FTLM_ERR_NUMERICAL;
    }
    for (double v : runs[r].eps) E0 = std::min(E0, v);
  }
  const bool summed = parallel_for(nT, 3.0 * nT * R * M * M, [&](int t) {
    const double b = 1.0 / T[t];
    double den = 0.0, nre = 0.0, nim = 0.0;
    for (int r = 0; r < R; ++r) {
      const Run& run = runs[r];
      const int m = run.m;
      std::vector<double> x(m), y(m, 0.0);
      for (int n = 0; n < m; ++n) {
        const double h = std::exp(-0.5 * b * (run.eps[n] - E0));
        x[n] = h * run.U[n];  // U_0n
        den += h * h * run.U[n] * run.U[n];
      }
      for (int i = 0; i < m; ++i) {
        double acc = 0.0;
        for (int n = 0; n < m; ++n) acc += run.U[(size_t)i * m + n] * x[n];
        y[i] = acc;
      }
      const double* O = Omat + (size_t)r * M * M * 2;
      for (int i = 0; i < m; ++i)
        for (int j = 0; j < m; ++j) {
          const double w = y[i] * y[j];
          nre += w * O[((size_t)i * M + j) * 2];
          nim += w * O[((size_t)i * M + j) * 2 + 1];
        }
    }
    MB_sym[t] = -g * nre / den;
    if (MB_sym_imag) MB_sym_imag[t] = -g * nim / den;
  });
  if (!summed) return msg = "out of host memory", FTLM_ERR_OUT_OF_MEMORY;
  return FTLM_OK;
}

}  // namespace ftlm
