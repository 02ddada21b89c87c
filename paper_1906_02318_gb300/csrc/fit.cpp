// fit_model: least-squares fit of the lifted operator (Sec. IV-A), and the
// sparsity-promoting selection of its basis (Sec. IV-A, V-C.3).
//
// K = argmin sum_m || Psi(x_{m+1}, u_m) - K Psi(x_m, u_m) ||^2.  With the lifted
// snapshots as rows of X (m x n) and Y (m x n) this is X K^T ~= Y, solved by
// Householder QR of X in float64 (no normal equations, so the conditioning of X
// is not squared).  The fit runs once per model, offline, on the host.
#include <math.h>
#include <sched.h>

#include <algorithm>
#include <atomic>
#include <condition_variable>
#include <functional>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include "basis.h"
#include "internal.h"

namespace mpmi {

// One lifted row; a constant KIND folds feature_split's switch away.
template <int KIND>
static void lift_row(const double* x, const double* u, double* out) {
  double p[kMaxP] = {0, 0, 0};
  monomials64(KIND, u, p);
  const int ai = angle_index(KIND);
  const double s = ai >= 0 ? sin(x[ai]) : 0.0, c = ai >= 0 ? cos(x[ai]) : 0.0;
#pragma GCC unroll 32
  for (int j = 0; j < BasisTraits<KIND>::N; ++j) {
    double a, b[kMaxP];
    feature_split<double>(KIND, j, x, s, c, &a, b);
    double v = a;
    for (int k = 0; k < kMaxP; ++k)
      if (b[k] != 0.0) v += p[k] * b[k];
    out[j] = v;
  }
}

typedef void (*LiftFn)(const double*, const double*, double*);
static LiftFn lift_of(int kind) {
  switch (kind) {
    case kBot: return lift_row<kBot>;
    case kCar: return lift_row<kCar>;
    case kLin11: return lift_row<kLin11>;
    case kLin22: return lift_row<kLin22>;
    default: return lift_row<kLin41>;
  }
}

// Column-major lifted snapshots: X[j * m + i] = Psi_j(x_i, u_i), Y likewise for
// (x_next_i, u_i).
static void lift_pairs(int kind, int n, int nx, int nu, const double* x, const double* u,
                       const double* xn, int64_t m, std::vector<double>* X,
                       std::vector<double>* Y) {
  X->assign((size_t)m * n, 0.0);
  Y->assign((size_t)m * n, 0.0);
  std::vector<double> row(n);
  const LiftFn lift = lift_of(kind);
  for (int64_t i = 0; i < m; ++i) {
    lift(x + i * nx, u + i * nu, row.data());
    for (int j = 0; j < n; ++j) (*X)[(size_t)j * m + i] = row[j];
    lift(xn + i * nx, u + i * nu, row.data());
    for (int j = 0; j < n; ++j) (*Y)[(size_t)j * m + i] = row[j];
  }
}

// ---- least squares by Householder QR in row blocks --------------------------------
// The rows [A | B] are taken in blocks of kFitRows, each block is reduced to its
// triangle [R | Q^T B], and triangles are stacked kFitMerge at a time and reduced
// again until one is left (tall-skinny QR; every reduction is a Householder QR, so
// the conditioning is that of the plain one).  A block of the race car's 60 columns
// is 123 KB and stays in a core's cache, where the whole matrix (2 x 5 MB at m = 20000)
// was read and written twice per reflection.  Blocks are shared by a few threads; what
// each block computes, and the order of the merges and of the sums, does not depend on
// their number.  GB300 host (16 cores): race car, m = 20000 42.9 ms one column at a time,
// 2.0 ms now (14 threads); m = 500 0.93 -> 0.40 ms and balance bot, m = 5000 1.6 ->
// 0.78 ms on the calling thread alone.
constexpr int kFitRows = 256, kFitMerge = 8;

// d[c] = sum over rows i >= i0 of M[i][k] M[i][c], c >= k.
static void column_dots(const double* __restrict M, int rows, int i0, int k, int W,
                        double* __restrict d) {
  for (int c = k; c < W; ++c) d[c] = 0.0;
  for (int i = i0; i < rows; ++i) {
    const double* r = M + (size_t)i * W;
    const double s = r[k];
    for (int c = k; c < W; ++c) d[c] += s * r[c];
  }
}

// Householder QR of the first p columns of M (rows x W, row-major), applied to all W:
// afterwards M[k][k .. W) holds row k of [R | Q^T B] for k < min(p, rows).  One pass
// over the rows per reflection: it applies reflection k and gathers column k + 1's
// products with the columns after it, which give the next norm and the next factors.
// The loops run along a row, so they vectorise without reordering any sum.  d, f: W
// values of scratch each.
static void house_rows(double* __restrict M, int rows, int p, int W, double* __restrict d,
                       double* __restrict f) {
  column_dots(M, rows, 0, 0, W, d);
  for (int k = 0; k < p && k + 1 < rows; ++k) {
    double* rk = M + (size_t)k * W;
    const double norm2 = d[k];
    if (norm2 == 0.0) {  // nothing to reflect; the caller judges the rank
      if (k + 1 < p) column_dots(M, rows, k + 1, k + 1, W, d);
      continue;
    }
    const double norm = sqrt(norm2);
    const double alpha = rk[k] > 0 ? -norm : norm;
    // v = column - alpha e_k; v^T v = 2 (norm2 - alpha M[k][k])
    const double vtv = 2.0 * (norm2 - alpha * rk[k]), vk = rk[k] - alpha;
    for (int c = k + 1; c < W; ++c) f[c] = 2.0 * (d[c] - alpha * rk[c]) / vtv;
    rk[k] = alpha;
    for (int c = k + 1; c < W; ++c) {
      rk[c] -= f[c] * vk;
      d[c] = 0.0;
    }
    if (k + 1 == W) continue;
    const int n1 = k + 1;
    int i = k + 1;
    for (; i + 4 <= rows; i += 4) {
      double* __restrict r0 = M + (size_t)i * W;
      double* __restrict r1 = r0 + W;
      double* __restrict r2 = r1 + W;
      double* __restrict r3 = r2 + W;
      const double v0 = r0[k], v1 = r1[k], v2 = r2[k], v3 = r3[k];
      const double s0 = r0[n1] - f[n1] * v0, s1 = r1[n1] - f[n1] * v1;
      const double s2 = r2[n1] - f[n1] * v2, s3 = r3[n1] - f[n1] * v3;
      for (int c = n1; c < W; ++c) {
        const double fc = f[c];
        const double m0 = r0[c] - fc * v0, m1 = r1[c] - fc * v1;
        const double m2 = r2[c] - fc * v2, m3 = r3[c] - fc * v3;
        r0[c] = m0;
        r1[c] = m1;
        r2[c] = m2;
        r3[c] = m3;
        d[c] += (s0 * m0 + s1 * m1) + (s2 * m2 + s3 * m3);
      }
    }
    for (; i < rows; ++i) {
      double* __restrict r = M + (size_t)i * W;
      const double v = r[k], s = r[n1] - f[n1] * v;
      for (int c = n1; c < W; ++c) {
        const double m = r[c] - f[c] * v;
        r[c] = m;
        d[c] += s * m;
      }
    }
  }
}

// Rows [R | Q^T B] of a reduced block: min(p, rows) of them, zeros left of the diagonal.
static int take_triangle(const double* M, int rows, int p, int W, double* out) {
  const int nr = rows < p ? rows : p;
  for (int k = 0; k < nr; ++k)
    for (int c = 0; c < W; ++c) out[(size_t)k * W + c] = c < k ? 0.0 : M[(size_t)k * W + c];
  return nr;
}

// Threads that take numbered tasks from a counter: run(n, fn) returns when fn(i, thread)
// is done for i = 0 .. n - 1 (fn must not throw).  The threads live as long as the
// object; where one cannot be started the others do its share.
class FitTeam {
 public:
  explicit FitTeam(int threads) {
    for (int i = 1; i < threads; ++i) {
      try {
        team_.emplace_back([this, i] { work(i); });
      } catch (...) {
        break;
      }
    }
  }
  ~FitTeam() {
    {
      std::lock_guard<std::mutex> lock(mu_);
      stop_ = true;
    }
    start_.notify_all();
    for (auto& t : team_) t.join();
  }
  int size() const { return 1 + (int)team_.size(); }
  void run(int n, const std::function<void(int, int)>& fn) {
    if (team_.empty() || n <= 1) {
      for (int i = 0; i < n; ++i) fn(i, 0);
      return;
    }
    {
      std::lock_guard<std::mutex> lock(mu_);
      fn_ = &fn;
      n_ = n;
      next_ = 0;
      busy_ = (int)team_.size();
      ++round_;
    }
    start_.notify_all();
    take(fn, n, 0);
    std::unique_lock<std::mutex> lock(mu_);
    done_.wait(lock, [this] { return busy_ == 0; });
  }

 private:
  void take(const std::function<void(int, int)>& fn, int n, int thread) {
    for (int i = next_++; i < n; i = next_++) fn(i, thread);
  }
  void work(int thread) {
    unsigned long seen = 0;
    std::unique_lock<std::mutex> lock(mu_);
    while (true) {
      start_.wait(lock, [&] { return stop_ || round_ != seen; });
      if (stop_) return;
      seen = round_;
      const std::function<void(int, int)>* fn = fn_;
      const int n = n_;
      lock.unlock();
      take(*fn, n, thread);
      lock.lock();
      if (--busy_ == 0) done_.notify_one();
    }
  }
  std::vector<std::thread> team_;
  std::mutex mu_;
  std::condition_variable start_, done_;
  const std::function<void(int, int)>* fn_ = nullptr;
  std::atomic<int> next_{0};
  int n_ = 0, busy_ = 0;
  unsigned long round_ = 0;
  bool stop_ = false;
};

// CPUs that the calling thread may run on: a caller with a narrower affinity mask (taskset,
// a container's CPU set, sched_setaffinity) gets no more threads than it has CPUs.
static int usable_cpus() {
  cpu_set_t set;
  if (sched_getaffinity(0, sizeof(set), &set) == 0) return CPU_COUNT(&set);
  return (int)std::thread::hardware_concurrency();
}

// Threads for a fit of m rows with p regressors and q targets: one per 8 MFLOP (about
// a millisecond), at most sixteen.
static int fit_threads(int64_t m, int p, int q) {
  const int64_t work = m * p * (p + 2 * q) / 4000000;
  return (int)std::max<int64_t>(1, std::min<int64_t>(std::min(usable_cpus(), 16), work));
}

// Least squares A W ~= B (A: m x p, B: m x q).  fill(i0, rows, dst): rows [A | B] i0 ..
// i0 + rows - 1, row-major, into dst (must not throw).  W (p x q) row-major.
static int qr_lstsq(FitTeam* team, int64_t m, int p, int q,
                    const std::function<void(int64_t, int, double*)>& fill,
                    std::vector<double>* Wout, std::string* err) {
  const int W = p + q;
  const int stack = std::max(kFitRows, kFitMerge * p);  // most rows of a reduction
  int n = (int)((m + kFitRows - 1) / kFitRows);
  std::vector<double> tri((size_t)n * p * W), next((size_t)((n + kFitMerge - 1) / kFitMerge) * p * W);
  std::vector<int> rows(n), rows_next((n + kFitMerge - 1) / kFitMerge);
  // per thread: the rows being reduced and two vectors of scratch
  const size_t per = (size_t)(stack + 2) * W;
  std::vector<double> work(per * team->size());
  team->run(n, [&](int b, int thread) {
    double* M = &work[per * thread];
    const int64_t i0 = (int64_t)b * kFitRows;
    const int nr = (int)std::min<int64_t>(kFitRows, m - i0);
    fill(i0, nr, M);
    house_rows(M, nr, p, W, M + (size_t)stack * W, M + (size_t)(stack + 1) * W);
    rows[b] = take_triangle(M, nr, p, W, &tri[(size_t)b * p * W]);
  });
  while (n > 1) {
    const int groups = (n + kFitMerge - 1) / kFitMerge;
    team->run(groups, [&](int g, int thread) {
      double* M = &work[per * thread];
      int nr = 0;
      for (int b = g * kFitMerge; b < n && b < (g + 1) * kFitMerge; ++b) {
        std::copy_n(&tri[(size_t)b * p * W], (size_t)rows[b] * W, M + (size_t)nr * W);
        nr += rows[b];
      }
      house_rows(M, nr, p, W, M + (size_t)stack * W, M + (size_t)(stack + 1) * W);
      rows_next[g] = take_triangle(M, nr, p, W, &next[(size_t)g * p * W]);
    });
    tri.swap(next);
    rows.swap(rows_next);
    n = groups;
  }
  const double* R = tri.data();
  double rmax = 0.0;
  for (int k = 0; k < p; ++k) rmax = fmax(rmax, fabs(R[(size_t)k * W + k]));
  for (int k = 0; k < p; ++k) {
    const double r = fabs(R[(size_t)k * W + k]);
    if (!(r > 0.0) || r <= 1e-13 * rmax) {
      *err = "fit: lifted data is rank deficient";
      return MPMI_E_INVALID_ARG;
    }
  }
  // back substitution R W = Q^T B
  Wout->assign((size_t)p * q, 0.0);
  for (int i = p - 1; i >= 0; --i) {
    double* wi = &(*Wout)[(size_t)i * q];
    for (int c = 0; c < q; ++c) wi[c] = R[(size_t)i * W + p + c];
    for (int j = i + 1; j < p; ++j) {
      const double r = R[(size_t)i * W + j];
      const double* wj = &(*Wout)[(size_t)j * q];
      for (int c = 0; c < q; ++c) wi[c] -= r * wj[c];
    }
    for (int c = 0; c < q; ++c) wi[c] /= R[(size_t)i * W + i];
  }
  return MPMI_OK;
}

// Held input features: the exact least-squares solution of their rows is the
// unit row (their target column is their regressor column), which the solver
// returns up to rounding; set it exactly.
static void set_held_rows(int kind, int n, std::vector<double>* K) {
  for (int c = 0; c < n; ++c)
    if (held_feature(kind, c))
      for (int k = 0; k < n; ++k) (*K)[(size_t)c * n + k] = k == c ? 1.0 : 0.0;
}

// ||X K^T - Y||_F / ||Y||_F over the predicted features `rows` (all if empty).
static double fit_residual(const std::vector<double>& X, const std::vector<double>& Y,
                           const std::vector<double>& K, int64_t m, int n,
                           const std::vector<unsigned char>& keep) {
  double num = 0.0, den = 0.0;
  for (int c = 0; c < n; ++c) {
    if (!keep.empty() && !keep[c]) continue;
    const double* kc = &K[(size_t)c * n];
    for (int64_t i = 0; i < m; ++i) {
      double pred = 0.0;
      for (int k = 0; k < n; ++k) pred += X[(size_t)k * m + i] * kc[k];
      const double y = Y[(size_t)c * m + i];
      num += (pred - y) * (pred - y);
      den += y * y;
    }
  }
  return den > 0 ? sqrt(num / den) : 0.0;
}

int fit_householder(int kind, const double* x, const double* u, const double* xn,
                    int64_t m, std::vector<double>* K, double* residual, std::string* err) {
  int n, nx, nu, np;
  kind_dims(kind, &n, &nx, &nu, &np);
  if (m < n) {
    *err = "fit_model: need at least n transitions";
    return MPMI_E_INVALID_ARG;
  }
  const LiftFn lift = lift_of(kind);
  // targets: the free features (the held ones' rows of K are set below)
  std::vector<int> free_rows;
  for (int c = 0; c < n; ++c)
    if (!held_feature(kind, c)) free_rows.push_back(c);
  const int q = (int)free_rows.size(), W = n + q;
  const int64_t blocks = (m + kFitRows - 1) / kFitRows;
  FitTeam team(fit_threads(m, n, q));
  std::vector<double> Wt;
  const int rc = qr_lstsq(
      &team, m, n, q,
      [&](int64_t i0, int rows, double* dst) {
        double y[32];
        for (int64_t i = i0; i < i0 + rows; ++i, dst += W) {
          lift(x + i * nx, u + i * nu, dst);
          lift(xn + i * nx, u + i * nu, y);
          for (int c = 0; c < q; ++c) dst[n + c] = y[free_rows[c]];
        }
      },
      &Wt, err);
  if (rc != MPMI_OK) return rc;
  // K = W^T on the free rows
  K->assign((size_t)n * n, 0.0);
  for (int r = 0; r < n; ++r)
    for (int c = 0; c < q; ++c) (*K)[(size_t)free_rows[c] * n + r] = Wt[(size_t)r * q + c];
  set_held_rows(kind, n, K);
  if (!residual) return MPMI_OK;
  // ||X K^T - Y||_F / ||Y||_F, summed per block, then over the blocks in order
  std::vector<double> KT((size_t)n * n), part(2 * (size_t)blocks);
  for (int r = 0; r < n; ++r)
    for (int k = 0; k < n; ++k) KT[(size_t)k * n + r] = (*K)[(size_t)r * n + k];
  team.run((int)blocks, [&](int b, int) {
    double X[32], Y[32], pred[32], num[32] = {0}, den[32] = {0};
    const int64_t end = std::min<int64_t>(m, (int64_t)(b + 1) * kFitRows);
    for (int64_t i = (int64_t)b * kFitRows; i < end; ++i) {
      lift(x + i * nx, u + i * nu, X);
      lift(xn + i * nx, u + i * nu, Y);
      for (int c = 0; c < n; ++c) pred[c] = 0.0;
      for (int k = 0; k < n; ++k)
        for (int c = 0; c < n; ++c) pred[c] += X[k] * KT[(size_t)k * n + c];
      for (int c = 0; c < n; ++c) {
        num[c] += (pred[c] - Y[c]) * (pred[c] - Y[c]);
        den[c] += Y[c] * Y[c];
      }
    }
    double ns = 0.0, ds = 0.0;
    for (int c = 0; c < n; ++c) {
      ns += num[c];
      ds += den[c];
    }
    part[2 * (size_t)b] = ns;
    part[2 * (size_t)b + 1] = ds;
  });
  double num = 0.0, den = 0.0;
  for (int64_t b = 0; b < blocks; ++b) {
    num += part[2 * (size_t)b];
    den += part[2 * (size_t)b + 1];
  }
  *residual = den > 0 ? sqrt(num / den) : 0.0;
  return MPMI_OK;
}

// ---- sparsity-promoting basis selection -----------------------------------
// Sparsity-promoting DMD (Jovanovic, Schmid & Nichols 2014) has two stages: an
// l1-type penalised least squares solved by ADMM, then an unpenalised refit
// ("polishing") on the surviving terms.  Applied here to the lifted regression
// X W ~= Y (W = K^T) with one group per candidate feature j (row W[j, :], its
// influence on every predicted feature), on unit-RMS scaled A = X D^-1 and
// B = Y E^-1:
//   minimise (1/m) ||A V - B||_F^2 + gamma sum_{j in C} ||V[j, :]||_2
// ADMM (split V = Z, penalty rho, scaled dual U):
//   V <- (2/m A^T A + rho I)^-1 (2/m A^T B + rho (Z - U))   (Cholesky, once)
//   Z[j] <- max(0, 1 - (gamma/rho) / ||(V + U)[j]||) (V + U)[j]  for j in C,
//   Z[j] <- (V + U)[j] otherwise;   U <- U + V - Z.
// Candidates C: every feature but the state and the held ones.  The support is
// {j : Z[j] != 0} plus every feature outside C; polishing refits on its columns.
static int cholesky(std::vector<double>* G, int n) {
  for (int j = 0; j < n; ++j) {
    double d = (*G)[(size_t)j * n + j];
    for (int k = 0; k < j; ++k) d -= (*G)[(size_t)j * n + k] * (*G)[(size_t)j * n + k];
    if (!(d > 0.0)) return MPMI_E_INVALID_ARG;
    const double l = sqrt(d);
    (*G)[(size_t)j * n + j] = l;
    for (int i = j + 1; i < n; ++i) {
      double s = (*G)[(size_t)i * n + j];
      for (int k = 0; k < j; ++k) s -= (*G)[(size_t)i * n + k] * (*G)[(size_t)j * n + k];
      (*G)[(size_t)i * n + j] = s / l;
    }
  }
  return MPMI_OK;
}

// Solves L L^T v = b in place (L lower, row-major n x n).
static void chol_solve(const std::vector<double>& L, int n, double* b) {
  for (int i = 0; i < n; ++i) {
    double s = b[i];
    for (int k = 0; k < i; ++k) s -= L[(size_t)i * n + k] * b[k];
    b[i] = s / L[(size_t)i * n + i];
  }
  for (int i = n - 1; i >= 0; --i) {
    double s = b[i];
    for (int k = i + 1; k < n; ++k) s -= L[(size_t)k * n + i] * b[k];
    b[i] = s / L[(size_t)i * n + i];
  }
}

int fit_sparse(int kind, const double* x, const double* u, const double* xn, int64_t m,
               double gamma, double rho, int iters, std::vector<double>* K,
               std::vector<unsigned char>* support, double* residual, std::string* err) {
  int n, nx, nu, np;
  kind_dims(kind, &n, &nx, &nu, &np);
  if (m < n) {
    *err = "fit_sparse: need at least n transitions";
    return MPMI_E_INVALID_ARG;
  }
  std::vector<double> X, Y;
  lift_pairs(kind, n, nx, nu, x, u, xn, m, &X, &Y);
  // unit-RMS scaling of regressors and targets
  std::vector<double> A = X, B = Y;
  for (int j = 0; j < n; ++j) {
    for (std::vector<double>* M : {&A, &B}) {
      double* col = &(*M)[(size_t)j * m];
      double ss = 0.0;
      for (int64_t i = 0; i < m; ++i) ss += col[i] * col[i];
      double s = sqrt(ss / (double)m);
      if (s == 0.0) s = 1.0;
      for (int64_t i = 0; i < m; ++i) col[i] /= s;
    }
  }
  std::vector<unsigned char> cand(n, 0);
  for (int j = nx; j < n; ++j) cand[j] = held_feature(kind, j) ? 0 : 1;
  // G = 2/m A^T A + rho I (row-major), AtB = 2/m A^T B (row-major, n x n)
  std::vector<double> G((size_t)n * n), AtB((size_t)n * n);
  for (int a = 0; a < n; ++a) {
    for (int b = 0; b < n; ++b) {
      double g = 0.0, h = 0.0;
      const double* ca = &A[(size_t)a * m];
      const double* cb = &A[(size_t)b * m];
      const double* yb = &B[(size_t)b * m];
      for (int64_t i = 0; i < m; ++i) {
        g += ca[i] * cb[i];
        h += ca[i] * yb[i];
      }
      G[(size_t)a * n + b] = 2.0 / (double)m * g + (a == b ? rho : 0.0);
      AtB[(size_t)a * n + b] = 2.0 / (double)m * h;
    }
  }
  if (cholesky(&G, n) != MPMI_OK) {
    *err = "fit_sparse: normal matrix not positive definite";
    return MPMI_E_INVALID_ARG;
  }
  std::vector<double> Z((size_t)n * n, 0.0), U((size_t)n * n, 0.0), V((size_t)n * n),
      col(n);
  for (int it = 0; it < iters; ++it) {
    // V = G^-1 (AtB + rho (Z - U)), one right-hand side per target column
    for (int c = 0; c < n; ++c) {
      for (int r = 0; r < n; ++r)
        col[r] = AtB[(size_t)r * n + c] + rho * (Z[(size_t)r * n + c] - U[(size_t)r * n + c]);
      chol_solve(G, n, col.data());
      for (int r = 0; r < n; ++r) V[(size_t)r * n + c] = col[r];
    }
    for (int r = 0; r < n; ++r) {
      double nrm2 = 0.0;
      for (int c = 0; c < n; ++c) {
        const double pv = V[(size_t)r * n + c] + U[(size_t)r * n + c];
        nrm2 += pv * pv;
      }
      const double nrm = sqrt(nrm2);
      double f = 1.0;
      if (cand[r]) {
        f = nrm > 0.0 ? 1.0 - (gamma / rho) / nrm : 0.0;
        if (f < 0.0) f = 0.0;
      }
      for (int c = 0; c < n; ++c) {
        const double pv = V[(size_t)r * n + c] + U[(size_t)r * n + c];
        Z[(size_t)r * n + c] = f * pv;
      }
    }
    for (size_t i = 0; i < U.size(); ++i) U[i] += V[i] - Z[i];
  }
  support->assign(n, 1);
  std::vector<int> cols;
  for (int r = 0; r < n; ++r) {
    if (cand[r]) {
      bool nz = false;
      for (int c = 0; c < n; ++c) nz = nz || Z[(size_t)r * n + c] != 0.0;
      (*support)[r] = nz ? 1 : 0;
    }
    if ((*support)[r]) cols.push_back(r);
  }
  // polishing: least squares on the support's columns of X
  const int p = (int)cols.size();
  std::vector<double> W;
  FitTeam team(fit_threads(m, p, n));
  const int rc = qr_lstsq(
      &team, m, p, n,
      [&](int64_t i0, int rows, double* dst) {
        for (int64_t i = i0; i < i0 + rows; ++i, dst += p + n) {
          for (int a = 0; a < p; ++a) dst[a] = X[(size_t)cols[a] * m + i];
          for (int c = 0; c < n; ++c) dst[p + c] = Y[(size_t)c * m + i];
        }
      },
      &W, err);
  if (rc != MPMI_OK) return rc;
  K->assign((size_t)n * n, 0.0);
  for (int a = 0; a < p; ++a)
    for (int c = 0; c < n; ++c) (*K)[(size_t)c * n + cols[a]] = W[(size_t)a * n + c];
  for (int r = 0; r < n; ++r)
    if (!(*support)[r])
      for (int c = 0; c < n; ++c) (*K)[(size_t)r * n + c] = 0.0;
  set_held_rows(kind, n, K);
  if (residual) *residual = fit_residual(X, Y, *K, m, n, *support);
  return MPMI_OK;
}

}  // namespace mpmi
