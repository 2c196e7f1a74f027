// Smoothed-aggregation algebraic multigrid for the pressure projection's
// Poisson matrix and for the elliptic relaxation (sec. 3.2 solves both by
// Jacobi-preconditioned conjugate gradients; a multigrid V-cycle as the
// preconditioner cuts the iterations from hundreds or thousands to tens
// while the solution stays that of the same linear system).  The Poisson
// matrix depends on the mesh only: its hierarchy is built once.  The
// relaxation matrices change with the statistics: the prolongations come
// once from the stiffness matrix, the level matrices are recomputed on the
// device at every solve (the second half of this file).
//
// Hierarchy (host, FP64, once): plain aggregation of the strongly connected
// unknowns (relative to each row's strongest connection), tentative
// prolongation by the constant vector (the null space of the pure-Neumann
// matrix), smoothed prolongation P = (I - w_p D^-1 A) P_tent with w_p =
// 4 / (3 rho), rho a bound of the eigenvalues of D^-1 A,
// Galerkin coarse matrices A_c = P^T A P, down to a dense coarsest matrix
// whose inverse (for a singular matrix with constant null space the
// regularised (A_c + mean(diag) 1 1^T / n_c)^-1, which solves every
// compatible right-hand side exactly) is applied directly.
//
// One V-cycle with one damped-Jacobi sweep (W = w_s D^-1) before and after
// the coarse correction is, per level,
//   M^-1 b = (2 W - W A W) b + Q M_c^-1 Q^T b,   Q = (I - W A) P,
// so the device runs two sweeps per level, "down" (x = W b and
// b_c = Q^T b) and "up" (z = x + W (b - A x) + Q e_c), and one dense
// matrix-vector product on the coarsest level (cycle.cuh: the sweeps of the
// lower levels, or of a small system's whole solve, in one kernel).  The cycle is symmetric, as
// the conjugate-gradient method needs.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <new>
#include <system_error>
#include <thread>
#include <type_traits>
#include <vector>

#include <cooperative_groups.h>

#include "amg.cuh"
#include "cycle.cuh"

namespace pdfgb {

namespace {

struct HCsr {
  int32_t n = 0, m = 0;
  std::vector<int32_t> rp, ci;
  std::vector<double> v;
};

HCsr transpose(const HCsr& A) {
  HCsr T;
  T.n = A.m;
  T.m = A.n;
  T.rp.assign(T.n + 1, 0);
  for (int32_t c : A.ci) T.rp[c + 1]++;
  for (int32_t i = 0; i < T.n; ++i) T.rp[i + 1] += T.rp[i];
  T.ci.resize(A.ci.size());
  T.v.resize(A.v.size());
  std::vector<int32_t> fill(T.rp.begin(), T.rp.end() - 1);
  for (int32_t i = 0; i < A.n; ++i)
    for (int32_t q = A.rp[i]; q < A.rp[i + 1]; ++q) {
      const int32_t d = fill[A.ci[q]]++;
      T.ci[d] = i;
      T.v[d] = A.v[q];
    }
  return T;  // columns ascending within each row
}

// f(lo, hi, chunk) over chunks of at least `grain` of the rows [0, n) on
// several host threads (the set-up runs at the first solve of a mesh, on its
// critical path).  A thread costs some 30 us to start: chunks of a matrix
// product or a plan (about a microsecond a row) from 512 rows, of a power
// iteration (20 ns a row) from 8,192.  Throws std::bad_alloc when a chunk did.
constexpr int kMaxChunks = 16;
int row_chunks(int32_t n, int32_t grain) {
  const int hw = (int)std::thread::hardware_concurrency();
  return std::max(1, std::min({kMaxChunks, hw > 0 ? hw : 1, n / grain}));
}
template <typename F>
void parallel_rows(int32_t n, F f, int32_t grain = 512) {
  const int c = row_chunks(n, grain);
  std::atomic<bool> failed{false};
  auto run = [&](int k) {
    try {
      f((int32_t)((int64_t)n * k / c), (int32_t)((int64_t)n * (k + 1) / c), k);
    } catch (...) {
      failed = true;
    }
  };
  std::thread th[kMaxChunks];
  int started = 1;
  for (; started < c; ++started) {
    try {
      th[started] = std::thread(run, started);
    } catch (const std::system_error&) {
      break;
    }
  }
  run(0);
  for (int k = started; k < c; ++k) run(k);  // (threads the system did not give)
  for (int k = 1; k < started; ++k) th[k].join();
  if (failed) throw std::bad_alloc();
}

// A matrix whose row i (n rows, m columns) is the sum of the terms that
// terms(i, add) gives by add(column, value), in that order; columns ascending.
template <typename F>
HCsr row_sums(int32_t n, int32_t m, F terms) {
  HCsr C;
  C.n = n;
  C.m = m;
  C.rp.assign(n + 1, 0);
  std::vector<int32_t> ci[kMaxChunks];
  std::vector<double> v[kMaxChunks];
  parallel_rows(n, [&](int32_t lo, int32_t hi, int k) {
    std::vector<int32_t> mark(m, -1), cols;
    std::vector<double> acc(m, 0.0);
    for (int32_t i = lo; i < hi; ++i) {
      cols.clear();
      terms(i, [&](int32_t j, double x) {
        if (mark[j] != i) { mark[j] = i; acc[j] = 0.0; cols.push_back(j); }
        acc[j] += x;
      });
      std::sort(cols.begin(), cols.end());
      for (int32_t j : cols) { ci[k].push_back(j); v[k].push_back(acc[j]); }
      C.rp[i + 1] = (int32_t)cols.size();
    }
  });
  for (int32_t i = 0; i < n; ++i) C.rp[i + 1] += C.rp[i];
  C.ci.reserve(C.rp[n]);
  C.v.reserve(C.rp[n]);
  for (int k = 0; k < kMaxChunks; ++k) {
    C.ci.insert(C.ci.end(), ci[k].begin(), ci[k].end());
    C.v.insert(C.v.end(), v[k].begin(), v[k].end());
  }
  return C;
}

// The same sums as lists: entry t of the matrix (rows rp, columns ci) is the
// sum of weight w[k] times another array's entry id[k], off[t] <= k < off[t + 1].
// terms(i, add) gives row i's terms by add(column, id, weight).
struct Plan {
  std::vector<int32_t> rp, ci, off, id;
  std::vector<double> w;
};
template <typename F>
Plan make_plan(int32_t n, int32_t m, F terms) {
  Plan P;
  P.rp.assign(n + 1, 0);
  std::vector<int32_t> ci[kMaxChunks], cnt[kMaxChunks], id[kMaxChunks];
  std::vector<double> w[kMaxChunks];
  parallel_rows(n, [&](int32_t lo, int32_t hi, int k) {
    std::vector<int32_t> mark(m, -1), num(m, 0), cols;
    for (int32_t i = lo; i < hi; ++i) {
      cols.clear();
      int32_t total = 0;
      terms(i, [&](int32_t j, int32_t, double) {
        if (mark[j] != i) { mark[j] = i; num[j] = 0; cols.push_back(j); }
        ++num[j];
        ++total;
      });
      std::sort(cols.begin(), cols.end());
      int32_t at = (int32_t)id[k].size();
      id[k].resize(at + total);
      w[k].resize(at + total);
      for (int32_t j : cols) {  // num[j]: the next place of column j's terms
        const int32_t c = num[j];
        ci[k].push_back(j);
        cnt[k].push_back(c);
        num[j] = at;
        at += c;
      }
      terms(i, [&](int32_t j, int32_t q, double x) {
        id[k][num[j]] = q;
        w[k][num[j]++] = x;
      });
      P.rp[i + 1] = (int32_t)cols.size();
    }
  });
  for (int32_t i = 0; i < n; ++i) P.rp[i + 1] += P.rp[i];
  P.off.assign(1, 0);
  P.off.reserve(P.rp[n] + 1);
  for (int k = 0; k < kMaxChunks; ++k) {
    P.ci.insert(P.ci.end(), ci[k].begin(), ci[k].end());
    P.id.insert(P.id.end(), id[k].begin(), id[k].end());
    P.w.insert(P.w.end(), w[k].begin(), w[k].end());
    for (int32_t c : cnt[k]) P.off.push_back(P.off.back() + c);
  }
  return P;
}

HCsr multiply(const HCsr& A, const HCsr& B) {
  return row_sums(A.n, B.m, [&](int32_t i, auto add) {
    for (int32_t q = A.rp[i]; q < A.rp[i + 1]; ++q) {
      const int32_t k = A.ci[q];
      const double a = A.v[q];
      for (int32_t t = B.rp[k]; t < B.rp[k + 1]; ++t) add(B.ci[t], a * B.v[t]);
    }
  });
}

std::vector<double> diagonal(const HCsr& A) {
  std::vector<double> d(A.n, 0.0);
  for (int32_t i = 0; i < A.n; ++i)
    for (int32_t q = A.rp[i]; q < A.rp[i + 1]; ++q)
      if (A.ci[q] == i) d[i] = A.v[q];
  return d;
}

// A bound of the eigenvalues of D^-1 A for the dampings: twelve power
// iterations times 1.15, at most Gershgorin's bound.  (kDamp over it stays
// below 2 / lambda_max while the iterations reach 0.73 lambda_max.)
double eigen_bound(const HCsr& A, const std::vector<double>& d) {
  std::vector<double> x(A.n), y(A.n);
  double gersh[kMaxChunks] = {}, sum[kMaxChunks] = {};
  for (int32_t i = 0; i < A.n; ++i) x[i] = 1.0 + (double)((i * 7919) % 101) / 101.0;
  double lam = 0.0, nx = 1.0;
  for (int it = 0; it < 12; ++it) {
    parallel_rows(A.n, [&](int32_t lo, int32_t hi, int k) {
      double s2 = 0.0, g = 0.0;
      for (int32_t i = lo; i < hi; ++i) {
        double s = 0.0, a = 0.0;
        for (int32_t q = A.rp[i]; q < A.rp[i + 1]; ++q) {
          s += A.v[q] * x[A.ci[q]];
          a += std::fabs(A.v[q]);
        }
        y[i] = s / (d[i] * nx);
        s2 += y[i] * y[i];
        g = std::max(g, a / d[i]);
      }
      sum[k] = s2;
      gersh[k] = g;
    }, 8192);
    double t = 0.0;
    for (double s : sum) t += s;
    if (!(t > 0.0)) break;
    nx = std::sqrt(t);  // (x = y / nx formed by the next product)
    lam = it > 0 ? nx : 0.0;
    std::swap(x, y);
  }
  const double g = *std::max_element(gersh, gersh + kMaxChunks);
  return lam > 0.0 ? std::min(g, 1.15 * lam) : g;
}

// Aggregates of strongly connected unknowns: seeds whose strong
// neighbourhood is free take it whole; leftovers join the aggregate they
// are most strongly connected to; what remains forms new aggregates.
// A connection is strong when -a_ij >= theta sqrt(m_i m_j), m_i the largest
// -a_ij of row i: relative to the row's strongest connection, so that on the
// channel's flat cells (couplings across the cell 40 times those along it)
// the coarsening follows the strong direction, and on isotropic cells takes
// all neighbours.  (|a_ij| >= 0.08 sqrt(a_ii a_jj) also took the jittered cells'
// middling couplings, and point smoothing then fails along the weak
// direction: 50 iterations to 1e-12 on the 100 x 200 channel against 20.)
std::vector<int32_t> aggregate(const HCsr& A, double theta, int32_t* n_agg) {
  const int32_t n = A.n;
  std::vector<double> m(n, 0.0);
  for (int32_t i = 0; i < n; ++i)
    for (int32_t q = A.rp[i]; q < A.rp[i + 1]; ++q)
      if (A.ci[q] != i) m[i] = std::max(m[i], -A.v[q]);
  auto strong = [&](int32_t i, int32_t q) {
    const int32_t j = A.ci[q];
    return j != i && A.v[q] < 0.0 && A.v[q] * A.v[q] >= theta * theta * m[i] * m[j];
  };
  std::vector<int32_t> agg(n, -1);
  int32_t na = 0;
  for (int32_t i = 0; i < n; ++i) {
    if (agg[i] >= 0) continue;
    bool free_nb = true;
    for (int32_t q = A.rp[i]; q < A.rp[i + 1] && free_nb; ++q)
      if (strong(i, q) && agg[A.ci[q]] >= 0) free_nb = false;
    if (!free_nb) continue;
    agg[i] = na;
    for (int32_t q = A.rp[i]; q < A.rp[i + 1]; ++q)
      if (strong(i, q)) agg[A.ci[q]] = na;
    ++na;
  }
  std::vector<int32_t> agg2 = agg;
  for (int32_t i = 0; i < n; ++i) {
    if (agg[i] >= 0) continue;
    double best = 0.0;
    for (int32_t q = A.rp[i]; q < A.rp[i + 1]; ++q)
      if (strong(i, q) && agg[A.ci[q]] >= 0 && std::fabs(A.v[q]) > best) {
        best = std::fabs(A.v[q]);
        agg2[i] = agg[A.ci[q]];
      }
  }
  for (int32_t i = 0; i < n; ++i) {
    if (agg2[i] >= 0) continue;
    agg2[i] = na;
    for (int32_t q = A.rp[i]; q < A.rp[i + 1]; ++q)
      if (strong(i, q) && agg2[A.ci[q]] < 0) agg2[A.ci[q]] = na;
    ++na;
  }
  *n_agg = na;
  return agg2;
}

template <typename T>
pdf_status up(T** dst, const std::vector<T>& src) {
  if (src.empty()) { *dst = nullptr; return PDF_OK; }
  cudaError_t e = cudaMalloc((void**)dst, src.size() * sizeof(T));
  if (e == cudaSuccess) e = cudaMemcpy(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice);
  return e == cudaSuccess ? PDF_OK : cuda_fail(e, "amg: upload");
}

pdf_status dev_vec(double** p, int64_t n) {
  cudaError_t e = cudaMalloc((void**)p, sizeof(double) * std::max<int64_t>(n, 1));
  return e == cudaSuccess ? PDF_OK : cuda_fail(e, "amg: allocation");
}

}  // namespace

void amg_free(Amg& G) {
  for (AmgLevel& L : G.lv) {
    cudaFree(L.a_rp); cudaFree(L.a_ci); cudaFree(L.a_v); cudaFree(L.w);
    cudaFree(L.q_rp); cudaFree(L.q_ci); cudaFree(L.q_v);
    cudaFree(L.s_rp); cudaFree(L.s_ci); cudaFree(L.s_v);
    cudaFree(L.b); cudaFree(L.x); cudaFree(L.z);
  }
  cudaFree(G.cinv); cudaFree(G.cb); cudaFree(G.cz);
  G = Amg();
}

// Damping of the Jacobi smoother over the bound of the largest eigenvalue of
// D^-1 A (below 2 / bound: the V-cycle stays positive definite).  5/3 needs
// about a tenth fewer iterations than the 4/3 of the prolongation's
// smoothing on the channel and obstacle meshes.
constexpr double kDamp = 5.0 / 3.0;

// The smoothed-aggregation hierarchy of A0 down to at most kCoarse
// unknowns: the level matrices As, prolongations Ps and the coarsest matrix;
// with_q: also Q = (I - W A) P and the smoother weights W of every level.
static pdf_status build_levels(HCsr A, int32_t kCoarse, bool with_q, std::vector<HCsr>& As, std::vector<HCsr>& Ps,
                               std::vector<HCsr>& Qs, std::vector<std::vector<double>>& Ws, HCsr& Afinal) {
  constexpr int32_t kMaxLevels = 12;
  double theta = 0.5;  // falls by 0.7 a level: the coarse matrices are denser and more isotropic
  while (A.n > kCoarse && (int32_t)As.size() < kMaxLevels) {
    const std::vector<double> d = diagonal(A);
    for (double x : d)
      if (!(x > 0.0)) return fail(PDF_EINVAL, "amg: non-positive diagonal");
    int32_t na = 0;
    std::vector<int32_t> agg = aggregate(A, theta, &na);
    // hardly any coarsening (few mutually strong connections): weaker ones count too
    for (double t = 0.5 * theta; na > 0.7 * A.n && t > 1e-3; t *= 0.5) agg = aggregate(A, t, &na);
    if (na >= A.n || na < 1) break;
    const double rho = eigen_bound(A, d);
    // P = (I - wp D^-1 A) P_tent
    const double wp = 4.0 / (3.0 * rho);
    const HCsr P = row_sums(A.n, na, [&](int32_t i, auto add) {
      add(agg[i], 1.0);
      for (int32_t q = A.rp[i]; q < A.rp[i + 1]; ++q) add(agg[A.ci[q]], -wp * A.v[q] / d[i]);
    });
    const HCsr AP = multiply(A, P);
    HCsr Ac = multiply(transpose(P), AP);
    if (with_q) {  // smoother W = ws D^-1 and Q = P - W A P
      const double ws = kDamp / rho;
      std::vector<double> W(A.n);
      for (int32_t i = 0; i < A.n; ++i) W[i] = ws / d[i];
      Qs.push_back(row_sums(A.n, na, [&](int32_t i, auto add) {
        for (int32_t q = P.rp[i]; q < P.rp[i + 1]; ++q) add(P.ci[q], P.v[q]);
        for (int32_t q = AP.rp[i]; q < AP.rp[i + 1]; ++q) add(AP.ci[q], -W[i] * AP.v[q]);
      }));
      Ws.push_back(std::move(W));
    }
    As.push_back(std::move(A));
    Ps.push_back(P);
    A = std::move(Ac);
    theta *= 0.7;
  }
  Afinal = std::move(A);
  return PDF_OK;
}

// Pressure systems of at most this many unknowns are solved by one cluster,
// unless some of them lie on the inflow or outflow.
constexpr int32_t kAmgWholeMax = 4096;
// The coarsest system of the kernels per sweep, and the size up to which it is
// the only one (the dense inverse is the preconditioner, one iteration is
// enough: 192 unknowns 145 us a call, by levels 335 us).
constexpr int32_t kAmgDense = 256;
static_assert(2 * kAmgDense <= kCyShared, "the coarsest vectors fit the shared memory of the levels");

static pdf_status amg_setup_host(int32_t n, const std::vector<int32_t>& rp, const std::vector<int32_t>& ci,
                                 const std::vector<double>& v, bool singular, Amg& G);

pdf_status amg_setup(int32_t n, const std::vector<int32_t>& rp, const std::vector<int32_t>& ci,
                     const std::vector<double>& v, bool singular, Amg& G) {
  try {
    return amg_setup_host(n, rp, ci, v, singular, G);
  } catch (const std::bad_alloc&) {
    amg_free(G);
    return fail(PDF_ENOMEM, "amg: host allocation");
  }
}

static pdf_status amg_setup_host(int32_t n, const std::vector<int32_t>& rp, const std::vector<int32_t>& ci,
                     const std::vector<double>& v, bool singular, Amg& G) {
  // Unknowns without couplings (rows of the unit matrix: inflow and outflow)
  // never coarsen.  They come on top of the coarsest size, or levels of little
  // but them are added in vain (80,000 unknowns with 800 such: six levels and
  // 8.1 ms a call against four and 3.3 ms), and they keep a system from the
  // cluster form, where every CTA takes the dense coarsest product for itself
  // (4,000 unknowns with 200 such: 1.70 ms against 1.08 ms; 40 and fewer:
  // equal).  In that form 256 coarsest unknowns took 18 us per cycle, so 64.
  int32_t single = 0;
  for (int32_t i = 0; i < n; ++i) {
    bool coupled = false;
    for (int32_t q = rp[i]; q < rp[i + 1]; ++q) coupled = coupled || (ci[q] != i && v[q] != 0.0);
    single += !coupled;
  }
  const bool whole = n <= kAmgDense || (n <= kAmgWholeMax && single == 0);
  const int32_t kCoarse = whole && n > kAmgDense ? 64 : kAmgDense + single;
  HCsr A0;
  A0.n = A0.m = n;
  A0.rp = rp;
  A0.ci = ci;
  A0.v = v;
  std::vector<HCsr> As, Ps, Qs;
  std::vector<std::vector<double>> Ws;
  HCsr A;
  pdf_status bs = build_levels(std::move(A0), kCoarse, true, As, Ps, Qs, Ws, A);
  if (bs != PDF_OK) return bs;
  // coarsest: regularised dense inverse (Gauss-Jordan with partial pivoting)
  const int32_t nc = A.n;
  std::vector<double> B((size_t)nc * nc, 0.0), Inv((size_t)nc * nc, 0.0);
  double dmean = 0.0;
  for (int32_t i = 0; i < nc; ++i)
    for (int32_t q = A.rp[i]; q < A.rp[i + 1]; ++q) {
      B[(size_t)i * nc + A.ci[q]] += A.v[q];
      if (A.ci[q] == i) dmean += A.v[q];
    }
  dmean = nc > 0 ? dmean / nc : 1.0;
  if (!(dmean > 0.0)) dmean = 1.0;
  if (singular)
    for (size_t k = 0; k < B.size(); ++k) B[k] += dmean / nc;
  for (int32_t i = 0; i < nc; ++i) Inv[(size_t)i * nc + i] = 1.0;
  for (int32_t c = 0; c < nc; ++c) {
    int32_t piv = c;
    for (int32_t r = c + 1; r < nc; ++r)
      if (std::fabs(B[(size_t)r * nc + c]) > std::fabs(B[(size_t)piv * nc + c])) piv = r;
    if (!(std::fabs(B[(size_t)piv * nc + c]) > 0.0)) return fail(PDF_EINVAL, "amg: singular coarse matrix");
    if (piv != c)
      for (int32_t k = 0; k < nc; ++k) {
        std::swap(B[(size_t)c * nc + k], B[(size_t)piv * nc + k]);
        std::swap(Inv[(size_t)c * nc + k], Inv[(size_t)piv * nc + k]);
      }
    const double s = 1.0 / B[(size_t)c * nc + c];
    for (int32_t k = 0; k < nc; ++k) { B[(size_t)c * nc + k] *= s; Inv[(size_t)c * nc + k] *= s; }
    for (int32_t r = 0; r < nc; ++r) {
      if (r == c) continue;
      const double f = B[(size_t)r * nc + c];
      if (f == 0.0) continue;
      for (int32_t k = 0; k < nc; ++k) {
        B[(size_t)r * nc + k] -= f * B[(size_t)c * nc + k];
        Inv[(size_t)r * nc + k] -= f * Inv[(size_t)c * nc + k];
      }
    }
  }
  // upload
  amg_free(G);
  pdf_status s = PDF_OK;
  for (size_t l = 0; l < As.size() && s == PDF_OK; ++l) {
    G.lv.emplace_back();
    AmgLevel& L = G.lv.back();
    L.n = As[l].n;
    L.nc = Qs[l].m;
    const HCsr S = transpose(Qs[l]);
    L.nnz_a = (int64_t)As[l].ci.size();
    L.nnz_q = (int64_t)Qs[l].ci.size();
    if ((s = up(&L.a_rp, As[l].rp)) != PDF_OK || (s = up(&L.a_ci, As[l].ci)) != PDF_OK ||
        (s = up(&L.a_v, As[l].v)) != PDF_OK || (s = up(&L.w, Ws[l])) != PDF_OK ||
        (s = up(&L.q_rp, Qs[l].rp)) != PDF_OK || (s = up(&L.q_ci, Qs[l].ci)) != PDF_OK ||
        (s = up(&L.q_v, Qs[l].v)) != PDF_OK || (s = up(&L.s_rp, S.rp)) != PDF_OK ||
        (s = up(&L.s_ci, S.ci)) != PDF_OK || (s = up(&L.s_v, S.v)) != PDF_OK)
      break;
    if (l > 0 && ((s = dev_vec(&L.b, L.n)) != PDF_OK || (s = dev_vec(&L.z, L.n)) != PDF_OK)) break;
    s = dev_vec(&L.x, L.n);
  }
  G.nc = nc;
  G.whole = whole && nc <= kAmgDense;
  if (s == PDF_OK) s = up(&G.cinv, Inv);
  if (s == PDF_OK) s = dev_vec(&G.cb, nc);
  if (s == PDF_OK) s = dev_vec(&G.cz, nc);
  if (s != PDF_OK) amg_free(G);
  return s;
}

// ------------------------------------------------------------------ device

// Rows of the coarse levels hold tens to hundreds of entries: a group of
// kG lanes shares a row (strided over its entries, then a shuffle sum).
constexpr int kG = 8;

__device__ __forceinline__ double group_sum(double v) {
#pragma unroll
  for (int o = kG / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o, kG);
  return v;
}

// x = W b on the level's rows (one thread per row); b_c = Q^T b on the
// coarse rows (kG lanes per row; blocks past the first nbx).  Skipped when
// *done is set.
__global__ void __launch_bounds__(256) k_amg_down(int32_t n, int32_t nc, int32_t nbx, const double* __restrict__ w,
                                                  const int32_t* __restrict__ s_rp, const int32_t* __restrict__ s_ci,
                                                  const double* __restrict__ s_v, const double* __restrict__ b,
                                                  double* __restrict__ x, double* __restrict__ bc,
                                                  const int32_t* __restrict__ done) {
  if (*done) return;
  if ((int32_t)blockIdx.x < nbx) {
    const int32_t i = blockIdx.x * 256 + threadIdx.x;
    if (i < n) x[i] = w[i] * b[i];
  } else {
    const int32_t J = ((blockIdx.x - nbx) * 256 + threadIdx.x) / kG, g = threadIdx.x % kG;
    double s = 0.0;
    if (J < nc)
      for (int32_t q = s_rp[J] + g; q < s_rp[J + 1]; q += kG) s += s_v[q] * b[s_ci[q]];
    s = group_sum(s);
    if (J < nc && g == 0) bc[J] = s;
  }
}

// Coarsest level: z = Inv b, one warp per row.
__global__ void __launch_bounds__(256) k_amg_coarse(int32_t nc, const double* __restrict__ inv,
                                                    const double* __restrict__ b, double* __restrict__ z,
                                                    const int32_t* __restrict__ done) {
  if (*done) return;
  const int32_t row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= nc) return;
  double s = 0.0;
  for (int32_t k = lane; k < nc; k += 32) s += inv[(int64_t)row * nc + k] * b[k];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) z[row] = s;
}

// z = x + W (b - A x) + Q e_c on the finest level (kF lanes per row), the
// block partials of b . z to part, and in the last block to finish their
// sum: *rz_old = *rz, *rz = sum (counter returns to 0).  More lanes per row
// shorten the gather chains but multiply the blocks, which costs more on
// this level's 10^5 rows than it saves, so one.
constexpr int kF = 1;

__global__ void __launch_bounds__(256) k_amg_up(int32_t n, const int32_t* __restrict__ a_rp,
                                                const int32_t* __restrict__ a_ci, const double* __restrict__ a_v,
                                                const double* __restrict__ w, const int32_t* __restrict__ q_rp,
                                                const int32_t* __restrict__ q_ci, const double* __restrict__ q_v,
                                                const double* __restrict__ b, const double* __restrict__ x,
                                                const double* __restrict__ ec, double* __restrict__ z,
                                                double* __restrict__ part, int32_t* __restrict__ counter,
                                                double* __restrict__ rz, double* __restrict__ rz_old,
                                                const int32_t* __restrict__ done) {
  if (*done) return;
  const int32_t i = (blockIdx.x * 256 + threadIdx.x) / kF, g = threadIdx.x % kF;
  double ax = 0.0, qe = 0.0;
  if (i < n) {
    for (int32_t q = a_rp[i] + g; q < a_rp[i + 1]; q += kF) ax += a_v[q] * x[a_ci[q]];
    for (int32_t q = q_rp[i] + g; q < q_rp[i + 1]; q += kF) qe += q_v[q] * ec[q_ci[q]];
  }
#pragma unroll
  for (int o = kF / 2; o > 0; o >>= 1) {
    ax += __shfl_xor_sync(0xffffffffu, ax, o, kF);
    qe += __shfl_xor_sync(0xffffffffu, qe, o, kF);
  }
  double bz = 0.0;
  if (i < n && g == 0) {
    const double bi = b[i];
    const double zi = x[i] + w[i] * (bi - ax) + qe;
    z[i] = zi;
    bz = bi * zi;
  }
  __shared__ double sh[8];
  __shared__ bool last;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) bz += __shfl_xor_sync(0xffffffffu, bz, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = bz;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int k = 0; k < 8; ++k) t += sh[k];
    part[blockIdx.x] = t;
    __threadfence();
    last = atomicAdd(counter, 1) == (int32_t)gridDim.x - 1;
    if (last) *counter = 0;
  }
  __syncthreads();
  if (!last) return;
  double t = 0.0;
  for (int32_t k = threadIdx.x; k < (int32_t)gridDim.x; k += 256) t += __ldcg(part + k);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int k = 0; k < 8; ++k) v += sh[k];
    *rz_old = *rz;
    *rz = v;
  }
}

// The same with kG lanes per row (coarse levels, no partials).
__global__ void __launch_bounds__(256) k_amg_up_g(int32_t n, const int32_t* __restrict__ a_rp,
                                                  const int32_t* __restrict__ a_ci, const double* __restrict__ a_v,
                                                  const double* __restrict__ w, const int32_t* __restrict__ q_rp,
                                                  const int32_t* __restrict__ q_ci, const double* __restrict__ q_v,
                                                  const double* __restrict__ b, const double* __restrict__ x,
                                                  const double* __restrict__ ec, double* __restrict__ z,
                                                  const int32_t* __restrict__ done) {
  if (*done) return;
  const int32_t i = (blockIdx.x * 256 + threadIdx.x) / kG, g = threadIdx.x % kG;
  double ax = 0.0, qe = 0.0;
  if (i < n) {
    for (int32_t q = a_rp[i] + g; q < a_rp[i + 1]; q += kG) ax += a_v[q] * x[a_ci[q]];
    for (int32_t q = q_rp[i] + g; q < q_rp[i + 1]; q += kG) qe += q_v[q] * ec[q_ci[q]];
  }
  ax = group_sum(ax);
  qe = group_sum(qe);
  if (i < n && g == 0) z[i] = x[i] + w[i] * (b[i] - ax) + qe;
}

// The levels, level 0's right-hand side r.
static Cycle<double, 1> amg_cycle(const Amg& G, const double* r, int first, int ctas) {
  Cycle<double, 1> C;
  C.L = (int)G.lv.size();
  C.first = first;
  C.nc = G.nc;
  C.cinv = G.cinv;
  for (int l = 0; l < C.L; ++l) {
    const AmgLevel& V = G.lv[l];
    CyLevel<double, 1>& D = C.lv[l];
    D.n = V.n; D.nc = V.nc; D.nnz_a = V.nnz_a; D.nnz_q = V.nnz_q;
    D.a_rp = V.a_rp; D.a_ci = V.a_ci; D.q_rp = V.q_rp; D.q_ci = V.q_ci; D.s_rp = V.s_rp; D.s_ci = V.s_ci;
    D.a[0] = V.a_v; D.q[0] = V.q_v; D.s[0] = V.s_v; D.w[0] = V.w;
    D.b = l == 0 ? const_cast<double*>(r) : V.b;
    D.x = V.x;
    D.z = V.z;
  }
  cy_plan(C, ctas);
  return C;
}

// The line between the two forms: one cluster against kernels per sweep, whole
// projection calls of 20 particles per element: 748 against 960 us at 760
// unknowns, 1,020 against 1,038 at 3,520, 1,326 against 1,170 at 6,930 (one
// component on eight SMs is FP64-bound there).  For the same reason the large
// form keeps a kernel per sweep on every level: a cluster for the levels
// below 3,000 unknowns made it 4 % slower.
pdf_status amg_solve(const Amg& G, const AmgSystem& A, int32_t it_end, cudaStream_t st) {
  const int ctas = cy_ctas(A.n);
  CySys<1> S;
  S.n = A.n;
  S.rp = A.rp; S.ci = A.ci; S.wall = nullptr;
  S.a[0] = A.val;
  S.x = A.x; S.r = A.r; S.p = A.p; S.q = A.q;
  S.rr = A.rr; S.rz = A.rz; S.tol2 = A.tol2;
  S.iters = A.iters; S.state = A.done;
  S.on = 0; S.off = 1;
  const Cycle<double, 1> C = amg_cycle(G, nullptr, 0, ctas);
  cudaError_t e = cudaSuccess;
  PDF_KERNEL("k_press_pcg", st, e = (cy_launch_pcg<kAmgWholeMax, double, 1>(1, ctas, st, S, C, it_end)));
  return e == cudaSuccess ? PDF_OK : cuda_fail(e, "k_press_pcg");
}

pdf_status amg_apply(const Amg& G, const double* r, double* z, double* part, int32_t* counter, double* rz,
                     double* rz_old, const int32_t* done, cudaStream_t st) {
  const int32_t L = (int32_t)G.lv.size();
  // down: level l's right-hand side is r (l = 0) or lv[l].b
  for (int32_t l = 0; l < L; ++l) {
    const AmgLevel& V = G.lv[l];
    const double* b = l == 0 ? r : V.b;
    double* bc = l + 1 < L ? G.lv[l + 1].b : G.cb;
    const int32_t nbx = (V.n + 255) / 256, nbc = (int32_t)(((int64_t)V.nc * kG + 255) / 256);
    PDF_KERNEL("k_amg_down", st, k_amg_down<<<nbx + nbc, 256, 0, st>>>(V.n, V.nc, nbx, V.w, V.s_rp, V.s_ci, V.s_v, b,
                                                                        V.x, bc, done));
  }
  if (L == 0) {
    PDF_KERNEL("k_amg_coarse", st, k_amg_coarse<<<(G.nc + 7) / 8, 256, 0, st>>>(G.nc, G.cinv, r, z, done));
    return PDF_OK;
  }
  PDF_KERNEL("k_amg_coarse", st, k_amg_coarse<<<(G.nc + 7) / 8, 256, 0, st>>>(G.nc, G.cinv, G.cb, G.cz, done));
  for (int32_t l = L - 1; l >= 0; --l) {
    const AmgLevel& V = G.lv[l];
    const double* b = l == 0 ? r : V.b;
    const double* ec = l + 1 < L ? G.lv[l + 1].z : G.cz;
    double* out = l == 0 ? z : V.z;
    if (l == 0)
      PDF_KERNEL("k_amg_up", st, k_amg_up<<<(int32_t)(((int64_t)V.n * kF + 255) / 256), 256, 0, st>>>(
                                     V.n, V.a_rp, V.a_ci, V.a_v, V.w, V.q_rp, V.q_ci, V.q_v, b, V.x, ec, out, part,
                                     counter, rz, rz_old, done));
    else
      PDF_KERNEL("k_amg_up", st, k_amg_up_g<<<(int32_t)(((int64_t)V.n * kG + 255) / 256), 256, 0, st>>>(
                                     V.n, V.a_rp, V.a_ci, V.a_v, V.w, V.q_rp, V.q_ci, V.q_v, b, V.x, ec, out, done));
  }
  return PDF_OK;
}

// ------------------------------------------------------------- persistent PCG

constexpr int kMaxLv = 12;

struct PcgLevel {
  int32_t n, nc;
  const int32_t *a_rp, *a_ci, *q_rp, *q_ci, *s_rp, *s_ci;
  const double *a_v, *w, *q_v, *s_v;
  double *b, *x, *z;
};

struct PcgArgs {
  int32_t n, L, nc;
  const int32_t *rp, *ci;
  const double* val;
  double *x, *r, *z, *p, *q, *scal, *part;
  int32_t* ctl;
  const double* cinv;
  double *cb, *cz;
  PcgLevel lv[kMaxLv];
};

// Sum over the block of v; the result in every thread.
__device__ __forceinline__ double block_sum_all(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
#pragma unroll
  for (int i = 0; i < 8; ++i) t += sh[i];
  __syncthreads();
  return t;
}

// Sum of the grid's block partials, in block order: identical in every block.
__device__ __forceinline__ double grid_total(const double* part, double* sh) {
  double t = 0.0;
  for (int32_t i = threadIdx.x; i < (int32_t)gridDim.x; i += 256) t += __ldcg(part + i);
  return block_sum_all(t, sh);
}

__global__ void __launch_bounds__(256) k_amg_pcg(PcgArgs A) {
  namespace cg = cooperative_groups;
  cg::grid_group grid = cg::this_grid();
  __shared__ double sh[8];
  const int32_t tid = blockIdx.x * 256 + threadIdx.x, nthr = gridDim.x * 256;
  const int32_t gl = tid / kG, lane_g = threadIdx.x % kG, ngrp = nthr / kG;
  double* part0 = A.part;
  double* part1 = A.part + gridDim.x;
  double* part2 = A.part + 2 * gridDim.x;
  int32_t it = A.ctl[kPcgIters];
  const int32_t max_it = A.ctl[kPcgMaxIt];
  bool done = A.ctl[kPcgDone] != 0;
  double rz = A.scal[kPcgRz], rz_old = A.scal[kPcgRzOld], rr = A.scal[kPcgRr], pq = 0.0;
  const double tol2 = A.scal[kPcgTol2];
  while (!done) {
    // z = M^-1 r: down the levels
    for (int l = 0; l < A.L; ++l) {
      const PcgLevel& V = A.lv[l];
      const double* b = l == 0 ? A.r : V.b;
      double* bc = l + 1 < A.L ? A.lv[l + 1].b : A.cb;
      for (int32_t i = tid; i < V.n; i += nthr) V.x[i] = V.w[i] * b[i];
      for (int32_t J0 = 0; J0 < V.nc; J0 += ngrp) {
        const int32_t J = J0 + gl;
        double s = 0.0;
        if (J < V.nc)
          for (int32_t k = V.s_rp[J] + lane_g; k < V.s_rp[J + 1]; k += kG) s += V.s_v[k] * b[V.s_ci[k]];
#pragma unroll
        for (int o = kG / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o, kG);
        if (J < V.nc && lane_g == 0) bc[J] = s;
      }
      grid.sync();
    }
    // coarsest level, one warp per row
    {
      const double* b = A.L > 0 ? A.cb : A.r;
      double* zc = A.L > 0 ? A.cz : A.z;
      const int32_t w = tid >> 5, lane = threadIdx.x & 31, nw = nthr >> 5;
      for (int32_t row0 = 0; row0 < A.nc; row0 += nw) {
        const int32_t row = row0 + w;
        double s = 0.0;
        if (row < A.nc)
          for (int32_t k = lane; k < A.nc; k += 32) s += A.cinv[(int64_t)row * A.nc + k] * b[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (row < A.nc && lane == 0) zc[row] = s;
      }
      grid.sync();
    }
    // up the levels; the finest one also gives r . z
    double bz = 0.0;
    for (int l = A.L - 1; l >= 0; --l) {
      const PcgLevel& V = A.lv[l];
      const double* b = l == 0 ? A.r : V.b;
      const double* ec = l + 1 < A.L ? A.lv[l + 1].z : A.cz;
      double* out = l == 0 ? A.z : V.z;
      if (l == 0) {
        for (int32_t i = tid; i < V.n; i += nthr) {
          double ax = 0.0, qe = 0.0;
          for (int32_t k = V.a_rp[i]; k < V.a_rp[i + 1]; ++k) ax += V.a_v[k] * V.x[V.a_ci[k]];
          for (int32_t k = V.q_rp[i]; k < V.q_rp[i + 1]; ++k) qe += V.q_v[k] * ec[V.q_ci[k]];
          const double zi = V.x[i] + V.w[i] * (b[i] - ax) + qe;
          out[i] = zi;
          bz += b[i] * zi;
        }
      } else {
        for (int32_t i0 = 0; i0 < V.n; i0 += ngrp) {
          const int32_t i = i0 + gl;
          double ax = 0.0, qe = 0.0;
          if (i < V.n) {
            for (int32_t k = V.a_rp[i] + lane_g; k < V.a_rp[i + 1]; k += kG) ax += V.a_v[k] * V.x[V.a_ci[k]];
            for (int32_t k = V.q_rp[i] + lane_g; k < V.q_rp[i + 1]; k += kG) qe += V.q_v[k] * ec[V.q_ci[k]];
          }
#pragma unroll
          for (int o = kG / 2; o > 0; o >>= 1) {
            ax += __shfl_xor_sync(0xffffffffu, ax, o, kG);
            qe += __shfl_xor_sync(0xffffffffu, qe, o, kG);
          }
          if (i < V.n && lane_g == 0) out[i] = V.x[i] + V.w[i] * (b[i] - ax) + qe;
        }
      }
      if (l > 0) grid.sync();
    }
    if (A.L == 0)
      for (int32_t i = tid; i < A.n; i += nthr) bz += A.r[i] * A.z[i];
    {
      const double t = block_sum_all(bz, sh);
      if (threadIdx.x == 0) part0[blockIdx.x] = t;
    }
    grid.sync();
    // beta; p = z + beta p and q = K z + beta q (= K p by the recurrence,
    // so no barrier between them); p . q
    rz_old = rz;
    rz = grid_total(part0, sh);
    const double beta = rz_old != 0.0 ? rz / rz_old : 0.0;
    double s_pq = 0.0;
    for (int32_t i = tid; i < A.n; i += nthr) {
      double kz = 0.0;
      for (int32_t k = A.rp[i]; k < A.rp[i + 1]; ++k) kz += A.val[k] * A.z[A.ci[k]];
      const double pv = A.z[i] + beta * A.p[i];
      const double qv = kz + beta * A.q[i];
      A.p[i] = pv;
      A.q[i] = qv;
      s_pq += pv * qv;
    }
    {
      const double t = block_sum_all(s_pq, sh);
      if (threadIdx.x == 0) part1[blockIdx.x] = t;
    }
    grid.sync();
    pq = grid_total(part1, sh);
    const double alpha = pq > 0.0 ? rz / pq : 0.0;
    double s_rr = 0.0;
    for (int32_t i = tid; i < A.n; i += nthr) {
      A.x[i] += alpha * A.p[i];
      const double rv = A.r[i] - alpha * A.q[i];
      A.r[i] = rv;
      s_rr += rv * rv;
    }
    {
      const double t = block_sum_all(s_rr, sh);
      if (threadIdx.x == 0) part2[blockIdx.x] = t;
    }
    grid.sync();
    rr = grid_total(part2, sh);
    ++it;
    done = rr <= tol2 || it >= max_it || !(pq > 0.0);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    A.scal[kPcgRr] = rr;
    A.scal[kPcgRz] = rz;
    A.scal[kPcgRzOld] = rz_old;
    A.scal[kPcgPq] = pq;
    A.ctl[kPcgIters] = it;
    A.ctl[kPcgDone] = 1;
  }
}

pdf_status amg_pcg(const Amg& G, int32_t n, const int32_t* rp, const int32_t* ci, const double* val, double* x,
                   double* r, double* z, double* p, double* q, double* scal, int32_t* ctl, double* part,
                   int32_t part_cap, cudaStream_t st) {
  if ((int)G.lv.size() > kMaxLv) return fail(PDF_EINVAL, "amg_pcg: too many levels");
  int dev = 0, coop = 0, sms = 0, per_sm = 0;
  PDF_CUDA(cudaGetDevice(&dev));
  PDF_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
  PDF_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  PDF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_amg_pcg, 256, 0));
  if (!coop || per_sm < 1) return fail(PDF_EINVAL, "amg_pcg: no cooperative launch");
  // at most one row per thread on the finest level, at most the resident grid
  int blocks = std::min<int64_t>((int64_t)sms * per_sm, ((int64_t)n + 255) / 256);
  blocks = std::max(1, std::min(blocks, part_cap / 3));
  PcgArgs A;
  std::memset(&A, 0, sizeof(A));
  A.n = n;
  A.L = (int32_t)G.lv.size();
  A.nc = G.nc;
  A.rp = rp; A.ci = ci; A.val = val;
  A.x = x; A.r = r; A.z = z; A.p = p; A.q = q; A.scal = scal; A.part = part; A.ctl = ctl;
  A.cinv = G.cinv; A.cb = G.cb; A.cz = G.cz;
  for (int l = 0; l < A.L; ++l) {
    const AmgLevel& V = G.lv[l];
    A.lv[l] = PcgLevel{V.n, V.nc, V.a_rp, V.a_ci, V.q_rp, V.q_ci, V.s_rp, V.s_ci,
                       V.a_v, V.w, V.q_v, V.s_v, V.b, V.x, V.z};
  }
  void* args[] = {&A};
  cudaError_t le = cudaSuccess;
  PDF_KERNEL("k_amg_pcg", st,
             le = cudaLaunchCooperativeKernel((const void*)k_amg_pcg, dim3(blocks), dim3(256), args, 0, st));
  if (le != cudaSuccess) return cuda_fail(le, "amg_pcg: cooperative launch");
  return PDF_OK;
}

// ------------------------------------------------------- relaxation multigrid

namespace {

template <typename T>
pdf_status up_vec(T** dst, const std::vector<T>& src) {
  cudaError_t e = cudaMalloc((void**)dst, std::max<size_t>(src.size(), 1) * sizeof(T));
  if (e == cudaSuccess && !src.empty())
    e = cudaMemcpy(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice);
  return e == cudaSuccess ? PDF_OK : cuda_fail(e, "relax multigrid: upload");
}

template <typename T>
pdf_status zeros(T** p, int64_t n) {
  cudaError_t e = cudaMalloc((void**)p, sizeof(T) * std::max<int64_t>(n, 1));
  if (e == cudaSuccess) e = cudaMemset(*p, 0, sizeof(T) * std::max<int64_t>(n, 1));
  return e == cudaSuccess ? PDF_OK : cuda_fail(e, "relax multigrid: allocation");
}

}  // namespace

void relax_amg_free(RelaxAmg& G) {
  for (RxLevel& L : G.lv) {
    cudaFree(L.a_rp); cudaFree(L.a_ci); cudaFree(L.a_dpos); cudaFree(L.q_rp); cudaFree(L.q_ci);
    cudaFree(L.s_rp); cudaFree(L.s_ci); cudaFree(L.s_perm); cudaFree(L.ap_off); cudaFree(L.ap_qa);
    cudaFree(L.ap_pv); cudaFree(L.c_off); cudaFree(L.c_tap); cudaFree(L.c_pv); cudaFree(L.q_pin);
    cudaFree(L.q_row); cudaFree(L.mem);
  }
  cudaFree(G.c_rp); cudaFree(G.c_ci);
  for (int v = 0; v < kRxVar; ++v) cudaFree(G.c_v[v]);
  cudaFree(G.cinv); cudaFree(G.r32); cudaFree(G.omega); cudaFree(G.gpart);
  cudaFree(G.upart);
  G = RelaxAmg();
}

static pdf_status relax_amg_setup_host(int32_t n, const std::vector<int32_t>& rp, const std::vector<int32_t>& ci,
                                       const std::vector<double>& kv, RelaxAmg& G);

pdf_status relax_amg_setup(int32_t n, const std::vector<int32_t>& rp, const std::vector<int32_t>& ci,
                           const std::vector<double>& kv, RelaxAmg& G) {
  try {
    return relax_amg_setup_host(n, rp, ci, kv, G);
  } catch (const std::bad_alloc&) {
    relax_amg_free(G);
    return fail(PDF_ENOMEM, "relax multigrid: host allocation");
  }
}

static pdf_status relax_amg_setup_host(int32_t n, const std::vector<int32_t>& rp, const std::vector<int32_t>& ci,
                                       const std::vector<double>& kv, RelaxAmg& G) {
  HCsr K;
  K.n = K.m = n;
  K.rp = rp;
  K.ci = ci;
  K.v = kv;
  std::vector<HCsr> As, Ps, Qs;
  std::vector<std::vector<double>> Ws;
  HCsr Afinal;
  pdf_status s = build_levels(std::move(K), 64, false, As, Ps, Qs, Ws, Afinal);
  if (s != PDF_OK) return s;
  if ((int)As.size() > kRxMaxLv) return fail(PDF_EINVAL, "relax multigrid: too many levels");
  relax_amg_free(G);
  // the pattern of every level's matrix follows from the plans: level 0 is
  // the relaxation pattern, level l + 1 that of P_l^T (A_l P_l)
  std::vector<int32_t> a_rp = rp, a_ci = ci;
  int32_t na = n;
  for (size_t l = 0; l < As.size() && s == PDF_OK; ++l) {
    const HCsr& P = Ps[l];
    G.lv.emplace_back();
    RxLevel& L = G.lv.back();
    L.n = na;
    L.nc = P.m;
    L.nnz_a = (int64_t)a_ci.size();
    // diagonal positions
    std::vector<int32_t> dpos(na, -1);
    for (int32_t i = 0; i < na; ++i)
      for (int32_t q = a_rp[i]; q < a_rp[i + 1]; ++q)
        if (a_ci[q] == i) dpos[i] = q;
    for (int32_t i = 0; i < na; ++i)
      if (dpos[i] < 0) return fail(PDF_EINVAL, "relax multigrid: missing diagonal");
    // plan of A P: per row, the (A entry, P value) pairs of each column
    const Plan ap = make_plan(na, P.m, [&](int32_t i, auto add) {
      for (int32_t q = a_rp[i]; q < a_rp[i + 1]; ++q) {
        const int32_t j = a_ci[q];
        for (int32_t t = P.rp[j]; t < P.rp[j + 1]; ++t) add(P.ci[t], q, P.v[t]);
      }
    });
    const std::vector<int32_t>&q_rp = ap.rp, &q_ci = ap.ci;
    const int64_t nap = (int64_t)q_ci.size();
    std::vector<int32_t> q_row(nap);
    std::vector<double> q_pin(nap, 0.0);  // P at each position (both rows ascending)
    for (int32_t i = 0; i < na; ++i) {
      int32_t t = P.rp[i];
      for (int32_t k = q_rp[i]; k < q_rp[i + 1]; ++k) {
        q_row[k] = i;
        while (t < P.rp[i + 1] && P.ci[t] < q_ci[k]) ++t;
        if (t < P.rp[i + 1] && P.ci[t] == q_ci[k]) q_pin[k] = P.v[t];
      }
    }
    L.nnz_ap = nap;
    L.ap_terms = (int64_t)ap.id.size();
    // S = Q^T with the permutation of the entries
    std::vector<int32_t> s_rp(P.m + 1, 0), s_ci(nap), s_perm(nap);
    for (int64_t t = 0; t < nap; ++t) s_rp[q_ci[t] + 1]++;
    for (int32_t J = 0; J < P.m; ++J) s_rp[J + 1] += s_rp[J];
    {
      std::vector<int32_t> fill(s_rp.begin(), s_rp.end() - 1);
      for (int32_t i = 0; i < na; ++i)
        for (int32_t t = q_rp[i]; t < q_rp[i + 1]; ++t) {
          const int32_t d = fill[q_ci[t]]++;
          s_ci[d] = i;
          s_perm[d] = t;
        }
    }
    // plan of the next matrix, P^T (A P): coarse entry (I, J) sums P_iI (A P)_iJ
    const HCsr Pt = transpose(P);
    Plan nx = make_plan(P.m, P.m, [&](int32_t I, auto add) {
      for (int32_t k = Pt.rp[I]; k < Pt.rp[I + 1]; ++k) {
        const int32_t i = Pt.ci[k];
        for (int32_t t = q_rp[i]; t < q_rp[i + 1]; ++t) add(q_ci[t], t, Pt.v[k]);
      }
    });
    L.c_terms = (int64_t)nx.id.size();
    if ((s = up_vec(&L.a_rp, a_rp)) != PDF_OK || (s = up_vec(&L.a_ci, a_ci)) != PDF_OK ||
        (s = up_vec(&L.a_dpos, dpos)) != PDF_OK || (s = up_vec(&L.q_rp, q_rp)) != PDF_OK ||
        (s = up_vec(&L.q_ci, q_ci)) != PDF_OK || (s = up_vec(&L.s_rp, s_rp)) != PDF_OK ||
        (s = up_vec(&L.s_ci, s_ci)) != PDF_OK || (s = up_vec(&L.s_perm, s_perm)) != PDF_OK ||
        (s = up_vec(&L.ap_off, ap.off)) != PDF_OK || (s = up_vec(&L.ap_qa, ap.id)) != PDF_OK ||
        (s = up_vec(&L.ap_pv, ap.w)) != PDF_OK || (s = up_vec(&L.c_off, nx.off)) != PDF_OK ||
        (s = up_vec(&L.c_tap, nx.id)) != PDF_OK || (s = up_vec(&L.c_pv, nx.w)) != PDF_OK ||
        (s = up_vec(&L.q_pin, q_pin)) != PDF_OK || (s = up_vec(&L.q_row, q_row)) != PDF_OK)
      break;
    // the values and vectors, cleared, in one allocation (one each per array made
    // the first solve on 3,200 nodes 12.5 -> 13.3 ms)
    size_t bytes = 0;
    auto place = [&](auto** p, int64_t n) {  // (an offset until the base is known)
      *p = reinterpret_cast<std::remove_reference_t<decltype(*p)>>(bytes);
      bytes += ((size_t)n * sizeof(**p) + 255) & ~(size_t)255;
    };
    auto arrays = [&](auto put) {
      put(&L.ap_v, kRxVar * nap);
      for (int v = 0; v < kRxVar; ++v) {
        put(&L.a_v[v], L.nnz_a);
        put(&L.a_f[v], L.nnz_a);
        put(&L.q_f[v], nap);
        put(&L.s_f[v], nap);
        put(&L.w_f[v], (int64_t)na);
        put(&L.w_v[v], (int64_t)na);
      }
      put(&L.x, 9 * (int64_t)na);
      if (l > 0) {
        put(&L.b, 9 * (int64_t)na);
        put(&L.z, 9 * (int64_t)na);
      }
    };
    arrays(place);
    if ((s = zeros(&L.mem, (int64_t)bytes)) != PDF_OK) break;
    arrays([&](auto** p, int64_t) {
      *p = reinterpret_cast<std::remove_reference_t<decltype(*p)>>(L.mem + reinterpret_cast<uintptr_t>(*p));
    });
    a_rp = std::move(nx.rp);
    a_ci = std::move(nx.ci);
    na = P.m;
  }
  if (s == PDF_OK && na > 64) s = fail(PDF_EINVAL, "relax multigrid: coarsest level above 64 unknowns");
  if (s == PDF_OK && G.lv.size() < 2 && !relax_mg_whole(n))
    s = fail(PDF_EINVAL, "relax multigrid: fewer than two levels");  // (the large form needs two)
  if (s == PDF_OK) {
    G.nc = na;
    G.nnz_c = (int64_t)a_ci.size();
    s = up_vec(&G.c_rp, a_rp);
    if (s == PDF_OK) s = up_vec(&G.c_ci, a_ci);
    for (int v = 0; v < kRxVar && s == PDF_OK; ++v) s = zeros(&G.c_v[v], G.nnz_c);
    if (s == PDF_OK) s = zeros(&G.cinv, (int64_t)kRxVar * na * na);
    if (s == PDF_OK) s = zeros(&G.r32, 9 * (int64_t)n);
    if (s == PDF_OK) s = zeros(&G.omega, kRxVar * kRxMaxLv);
    G.gblocks = (int32_t)std::min<int64_t>(1024, ((int64_t)n + 255) / 256);
    if (s == PDF_OK) s = zeros(&G.gpart, (int64_t)kRxVar * G.gblocks);
    if (s == PDF_OK) s = zeros(&G.upart, 9 * (((int64_t)n + 255) / 256));
  }
  if (s != PDF_OK) relax_amg_free(G);
  return s;
}

// Per-variant pointers of one level, for the kernels.
struct RxVals {
  const double* a[kRxVar];
  double4_32a* ap;         // A P, the four variants of an entry side by side
  double* an[kRxVar];  // the next level's matrix values
  float *af[kRxVar], *qf[kRxVar], *sf[kRxVar], *wf[kRxVar];
  double* w[kRxVar];
};

// (A P)[t] for the four variants (each thread all four: the plan's indices
// are loaded once).  The four values of an entry are stored side by side:
// k_rx_next gathers them, and from four arrays each gather moved four sectors
// of 32 bytes for 32 bytes used.  G lanes per entry (the group's own part of
// the terms, then a butterfly): one thread per entry was a chain of dependent
// loads, up to hundreds of terms long on the coarsest levels, with few blocks.
// 79,600 unknowns, four levels: k_rx_ap 355 -> 336 us, k_rx_next 403 -> 283 us
// (eight lanes everywhere 402 and 372: the FP64 sums across the lanes); 760
// unknowns, three levels: 55 -> 27 and 66 -> 25 us.
// Entries from which one thread each is enough, and mean terms above which an
// entry takes a warp.
constexpr int64_t kRxThreads = 65536, kRxMany = 64;
// The G lanes' sums of four values; lanes 0 to 3 end with one value each, of
// variant rx_variant.  (Each stage halves the values a lane carries: four FP64
// additions a lane where a butterfly of all four takes twelve.)
template <int G>
__device__ __forceinline__ double rx_group_sum(const double s[kRxVar]) {
  static_assert(kRxVar == 4, "four variants");
  const uint32_t m = G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u) << (threadIdx.x & 31 & ~(G - 1));
  const bool b0 = threadIdx.x & 1, b1 = threadIdx.x & 2;
  const double r0 = (b0 ? s[2] : s[0]) + __shfl_xor_sync(m, b0 ? s[0] : s[2], 1);
  const double r1 = (b0 ? s[3] : s[1]) + __shfl_xor_sync(m, b0 ? s[1] : s[3], 1);
  double q = (b1 ? r1 : r0) + __shfl_xor_sync(m, b1 ? r0 : r1, 2);
#pragma unroll
  for (int o = 4; o < G; o <<= 1) q += __shfl_xor_sync(m, q, o);
  return q;
}
__device__ __forceinline__ int rx_variant(int lane) { return 2 * (lane & 1) + ((lane >> 1) & 1); }
template <int G>
__global__ void __launch_bounds__(256) k_rx_ap(int64_t nnz_ap, const int32_t* __restrict__ off,
                                               const int32_t* __restrict__ qa, const double* __restrict__ pv,
                                               RxVals V) {
  const int lane = threadIdx.x & (G - 1);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x / G;
  for (int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / G; t < nnz_ap; t += stride) {
    double s[kRxVar] = {0.0, 0.0, 0.0, 0.0};
    const int32_t end = off[t + 1];
    for (int32_t k = off[t] + lane; k < end; k += G) {
      const int32_t q = qa[k];
      const double w = pv[k];
#pragma unroll
      for (int v = 0; v < kRxVar; ++v) s[v] += V.a[v][q] * w;
    }
    if constexpr (G == 1) {
      V.ap[t] = make_double4_32a(s[0], s[1], s[2], s[3]);
    } else {
      const double x = rx_group_sum<G>(s);
      if (lane < kRxVar) reinterpret_cast<double*>(V.ap + t)[rx_variant(lane)] = x;
    }
  }
}

// Gershgorin bound of D^-1 A per variant: block partial maxima.
__global__ void __launch_bounds__(256) k_rx_gersh(int32_t n, const int32_t* __restrict__ rp,
                                                  const int32_t* __restrict__ dpos, RxVals V,
                                                  double* __restrict__ part) {
  const int v = blockIdx.y;
  const double* a = V.a[v];
  double m = 0.0;
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int32_t q = rp[i]; q < rp[i + 1]; ++q) s += fabs(a[q]);
    m = fmax(m, s / a[dpos[i]]);
  }
  __shared__ double sh[8];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int k = 0; k < 8; ++k) t = fmax(t, sh[k]);
    part[(int64_t)v * gridDim.x + blockIdx.x] = t;
  }
}

// (a warp per variant)
__global__ void __launch_bounds__(32 * kRxVar) k_rx_omega(const double* __restrict__ part, int32_t nb, int level,
                                                          double* __restrict__ omega) {
  const int v = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double m = 0.0;
  for (int32_t b = lane; b < nb; b += 32) m = fmax(m, part[(int64_t)v * nb + b]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) omega[v * kRxMaxLv + level] = m > 0.0 ? kDamp / m : 0.0;
}

// The smoother weights W = omega / a_ii (FP64 and FP32) and the FP32 copy
// of the level matrix.
__global__ void k_rx_cast(int32_t n, int64_t nnz_a, const int32_t* __restrict__ dpos,
                          const double* __restrict__ omega, int level, RxVals V) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nnz_a; t += (int64_t)gridDim.x * blockDim.x) {
    const int32_t d = t < n ? dpos[t] : 0;
#pragma unroll
    for (int v = 0; v < kRxVar; ++v) {
      V.af[v][t] = (float)V.a[v][t];
      if (t < n) {
        const double w = omega[v * kRxMaxLv + level] / V.a[v][d];
        V.w[v][t] = w;
        V.wf[v][t] = (float)w;
      }
    }
  }
}

// Q = P - W (A P); S = Q^T; the next level's matrix.
__global__ void k_rx_q(int64_t nnz_ap, const double* __restrict__ pin, const int32_t* __restrict__ row, RxVals V) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nnz_ap; t += (int64_t)gridDim.x * blockDim.x) {
    const int32_t i = row[t];
    const double p = pin[t];
    const double4_32a ap = V.ap[t];
    const double x[kRxVar] = {ap.x, ap.y, ap.z, ap.w};
#pragma unroll
    for (int v = 0; v < kRxVar; ++v) V.qf[v][t] = (float)(p - V.w[v][i] * x[v]);
  }
}

__global__ void k_rx_s(int64_t nnz_ap, const int32_t* __restrict__ perm, RxVals V) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nnz_ap; t += (int64_t)gridDim.x * blockDim.x) {
    const int32_t k = perm[t];
#pragma unroll
    for (int v = 0; v < kRxVar; ++v) {
      V.sf[v][t] = V.qf[v][k];
    }
  }
}

template <int G>
__global__ void __launch_bounds__(256) k_rx_next(int64_t nnz_n, const int32_t* __restrict__ off,
                                                 const int32_t* __restrict__ tap, const double* __restrict__ pv,
                                                 RxVals V) {
  const int lane = threadIdx.x & (G - 1);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x / G;
  for (int64_t c = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / G; c < nnz_n; c += stride) {
    double s[kRxVar] = {0.0, 0.0, 0.0, 0.0};
    const int32_t end = off[c + 1];
#pragma unroll 4
    for (int32_t k = off[c] + lane; k < end; k += G) {
      const double4_32a q = V.ap[tap[k]];
      const double w = pv[k];
      s[0] += q.x * w;
      s[1] += q.y * w;
      s[2] += q.z * w;
      s[3] += q.w * w;
    }
    if constexpr (G == 1) {
#pragma unroll
      for (int v = 0; v < kRxVar; ++v) V.an[v][c] = s[v];
    } else {
      const double x = rx_group_sum<G>(s);
      const int v = rx_variant(lane);
      double* o = v == 0 ? V.an[0] : (v == 1 ? V.an[1] : (v == 2 ? V.an[2] : V.an[3]));
      if (lane < kRxVar) o[c] = x;
    }
  }
}

// Inverses of the four coarsest matrices (symmetric positive definite, at
// most 64 unknowns), one block each: symmetric Gauss-Jordan sweeps on the
// lower triangle, which the threads hold in registers.  The FP64 pipe of one
// SM bounds it (an update of 2,080 entries, 0.6 us, per sweep): 106 us for a
// coarsest level of some 60 unknowns, against 432 us for the elimination of
// the full matrix beside the unit matrix in global memory.
constexpr int kCoarseMax = 64;
constexpr int kCoarsePer = (kCoarseMax * (kCoarseMax + 1) / 2 + 255) / 256;
__global__ void __launch_bounds__(256) k_rx_coarse_inv(int32_t nc, const int32_t* __restrict__ rp,
                                                       const int32_t* __restrict__ ci, RxVals V,
                                                       float* __restrict__ cinv) {
  __shared__ double tri[kCoarseMax * (kCoarseMax + 1) / 2];
  __shared__ double col[2][kCoarseMax], scaled[kCoarseMax], inv[2];
  const int v = blockIdx.x, n_tri = nc * (nc + 1) / 2;
  for (int k = threadIdx.x; k < n_tri; k += 256) tri[k] = 0.0;
  __syncthreads();
  for (int i = threadIdx.x; i < nc; i += 256)
    for (int32_t q = rp[i]; q < rp[i + 1]; ++q)
      if (ci[q] <= i) tri[i * (i + 1) / 2 + ci[q]] = V.an[v][q];
  __syncthreads();
  double a[kCoarsePer];
  int row[kCoarsePer], at[kCoarsePer];  // entry (row, at), at <= row
#pragma unroll
  for (int k = 0; k < kCoarsePer; ++k) {
    const int e = threadIdx.x + 256 * k;
    int i = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
    if ((i + 1) * (i + 2) / 2 <= e) ++i;
    if (i * (i + 1) / 2 > e) --i;
    row[k] = e < n_tri ? i : -1;
    at[k] = e - i * (i + 1) / 2;
    a[k] = e < n_tri ? tri[e] : 0.0;
  }
  // column c (= row c) and the reciprocal of its pivot, by the threads that
  // have just formed them; two buffers, so that a sweep needs two barriers
  auto publish = [&](int k, int c) {
    if (row[k] == c) {
      col[c & 1][at[k]] = a[k];
      if (at[k] == c) inv[c & 1] = 1.0 / a[k];
    } else if (at[k] == c && row[k] > c) {
      col[c & 1][row[k]] = a[k];
    }
  };
#pragma unroll
  for (int k = 0; k < kCoarsePer; ++k) publish(k, 0);
  for (int c = 0; c < nc; ++c) {
    __syncthreads();
    const double* x = col[c & 1];
    const double d = inv[c & 1];
    if (threadIdx.x < nc) scaled[threadIdx.x] = x[threadIdx.x] * d;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kCoarsePer; ++k) {
      if (256 * k >= n_tri) break;
      if (row[k] < 0) continue;
      if (row[k] == c) a[k] = at[k] == c ? -d : scaled[at[k]];
      else if (at[k] == c) a[k] = scaled[row[k]];
      else a[k] -= scaled[row[k]] * x[at[k]];
      publish(k, c + 1);
    }
  }
  // the sweeps leave the negative inverse
#pragma unroll
  for (int k = 0; k < kCoarsePer; ++k) {
    if (row[k] < 0) continue;
    const float x = (float)-a[k];
    float* o = cinv + (int64_t)v * nc * nc;
    o[(int64_t)row[k] * nc + at[k]] = x;
    o[(int64_t)at[k] * nc + row[k]] = x;
  }
}

static int rx_lanes(int64_t entries, int64_t terms) {
  return terms > kRxMany * entries ? 32 : (entries >= kRxThreads ? 1 : 8);
}
static int rx_blocks(int64_t n) { return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 4096)); }

pdf_status relax_amg_update(RelaxAmg& G, cudaStream_t st) {
  const int L = (int)G.lv.size();
  for (int l = 0; l < L; ++l) {
    RxLevel& V = G.lv[l];
    RxVals R;
    R.ap = reinterpret_cast<double4_32a*>(V.ap_v);
    for (int v = 0; v < kRxVar; ++v) {
      R.a[v] = V.a_v[v];
      R.an[v] = l + 1 < L ? G.lv[l + 1].a_v[v] : G.c_v[v];
      R.af[v] = V.a_f[v];
      R.qf[v] = V.q_f[v];
      R.sf[v] = V.s_f[v];
      R.wf[v] = V.w_f[v];
      R.w[v] = V.w_v[v];
    }
    const int64_t nnz_n = l + 1 < L ? G.lv[l + 1].nnz_a : G.nnz_c;
    const int ga = rx_lanes(V.nnz_ap, V.ap_terms);
    void (*ap)(int64_t, const int32_t*, const int32_t*, const double*, RxVals) =
        ga == 1 ? k_rx_ap<1> : (ga == 8 ? k_rx_ap<8> : k_rx_ap<32>);
    PDF_KERNEL("k_rx_ap", st, ap<<<rx_blocks(ga * V.nnz_ap), 256, 0, st>>>(V.nnz_ap, V.ap_off, V.ap_qa, V.ap_pv, R));
    const int gb = std::min<int>(G.gblocks, rx_blocks(V.n));
    PDF_KERNEL("k_rx_gersh", st, k_rx_gersh<<<dim3(gb, kRxVar), 256, 0, st>>>(V.n, V.a_rp, V.a_dpos, R, G.gpart));
    PDF_KERNEL("k_rx_omega", st, k_rx_omega<<<1, 32 * kRxVar, 0, st>>>(G.gpart, gb, l, G.omega));
    PDF_KERNEL("k_rx_cast", st, k_rx_cast<<<rx_blocks(V.nnz_a), 256, 0, st>>>(V.n, V.nnz_a, V.a_dpos, G.omega, l, R));
    PDF_KERNEL("k_rx_q", st, k_rx_q<<<rx_blocks(V.nnz_ap), 256, 0, st>>>(V.nnz_ap, V.q_pin, V.q_row, R));
    PDF_KERNEL("k_rx_s", st, k_rx_s<<<rx_blocks(V.nnz_ap), 256, 0, st>>>(V.nnz_ap, V.s_perm, R));
    const int gn = rx_lanes(nnz_n, V.c_terms);
    void (*next)(int64_t, const int32_t*, const int32_t*, const double*, RxVals) =
        gn == 1 ? k_rx_next<1> : (gn == 8 ? k_rx_next<8> : k_rx_next<32>);
    PDF_KERNEL("k_rx_next", st, next<<<rx_blocks(gn * nnz_n), 256, 0, st>>>(nnz_n, V.c_off, V.c_tap, V.c_pv, R));
  }
  RxVals R;
  R.ap = nullptr;
  for (int v = 0; v < kRxVar; ++v) {
    R.a[v] = nullptr;
    R.af[v] = R.qf[v] = R.sf[v] = R.wf[v] = nullptr;
    R.w[v] = nullptr;
    R.an[v] = G.c_v[v];
  }
  PDF_KERNEL("k_rx_coarse_inv", st, k_rx_coarse_inv<<<kRxVar, 256, 0, st>>>(G.nc, G.c_rp, G.c_ci, R, G.cinv));
  return PDF_OK;
}

}  // namespace pdfgb

