// Smoothed-aggregation multigrid preconditioner (host setup, device cycle).
#pragma once
#include <vector>

#include "common.cuh"

namespace pdfgb {

struct AmgLevel {
  int32_t n = 0, nc = 0;  // rows of this level, of the next one
  int64_t nnz_a = 0, nnz_q = 0;
  int32_t *a_rp = nullptr, *a_ci = nullptr;  // the level's matrix A
  double* a_v = nullptr;
  double* w = nullptr;                       // damped Jacobi weights w_s / a_ii
  int32_t *q_rp = nullptr, *q_ci = nullptr;  // Q = (I - W A) P, n x nc
  double* q_v = nullptr;
  int32_t *s_rp = nullptr, *s_ci = nullptr;  // Q^T, nc x n
  double* s_v = nullptr;
  double *b = nullptr, *x = nullptr, *z = nullptr;  // right-hand side (l > 0), pre-smoothed, result (l > 0)
};

struct Amg {
  std::vector<AmgLevel> lv;
  int32_t nc = 0;           // coarsest size
  double* cinv = nullptr;   // [nc][nc] regularised inverse of the coarsest matrix
  double *cb = nullptr, *cz = nullptr;
  bool whole = false;       // solved by one cluster in one launch (amg_solve)
};

// Builds the hierarchy of the symmetric CSR matrix (n rows, columns
// sorted; positive definite, or with singular = true positive semi-definite
// with the constants as null space) and uploads it.
pdf_status amg_setup(int32_t n, const std::vector<int32_t>& rp, const std::vector<int32_t>& ci,
                     const std::vector<double>& v, bool singular, Amg& G);
void amg_free(Amg& G);
// z = M^-1 r (one V-cycle).  When the hierarchy has a level, the finest
// up-sweep also forms r . z (block partials in part, finished by the last
// block through *counter, which it resets): *rz_old = *rz, *rz = r . z;
// else the caller forms it.  Every kernel returns at once when *done is set.
pdf_status amg_apply(const Amg& G, const double* r, double* z, double* part, int32_t* counter, double* rz,
                     double* rz_old, const int32_t* done, cudaStream_t st);

// The whole preconditioned conjugate-gradient solve of a system of n
// unknowns by one cluster in one launch, up to iteration it_end (*done = 1 at
// r.r <= *tol2 or a breakdown), for hierarchies with G.whole.
struct AmgSystem {
  int32_t n = 0;
  const int32_t *rp = nullptr, *ci = nullptr;
  const double* val = nullptr;
  double *x = nullptr, *r = nullptr, *p = nullptr, *q = nullptr, *rr = nullptr, *rz = nullptr, *tol2 = nullptr;
  int32_t *iters = nullptr, *done = nullptr;
};
pdf_status amg_solve(const Amg& G, const AmgSystem& A, int32_t it_end, cudaStream_t st);

// The whole preconditioned conjugate-gradient iteration for the CSR matrix
// (n rows; rp, ci, val) in one persistent cooperative kernel, the phases
// separated by grid-wide barriers.  Entry state (as left by the caller's
// initialisation): x, r = b - A x, p = q = 0, scal[kPcgRz] = scal[kPcgRzOld] = 1,
// scal[kPcgTol2] = the stopping threshold on r.r, ctl[kPcgDone/Iters/MaxIt].
// On return x, r, scal[kPcgRr], ctl[kPcgIters] and ctl[kPcgDone] = 1 (the
// caller tells convergence from r.r <= tol2).  part: 3 x grid doubles.
// Returns PDF_EINVAL when the device cannot launch it cooperatively (the
// caller then runs the separate kernels).
enum { kPcgDone = 0, kPcgIters = 1, kPcgMaxIt = 2 };
enum { kPcgPq = 0, kPcgRz = 1, kPcgRr = 2, kPcgRzOld = 6, kPcgTol2 = 7 };
pdf_status amg_pcg(const Amg& G, int32_t n, const int32_t* rp, const int32_t* ci, const double* val, double* x,
                   double* r, double* z, double* p, double* q, double* scal, int32_t* ctl, double* part,
                   int32_t part_cap, cudaStream_t st);

// ---------------------------------------------------------------------------
// The relaxation's multigrid: the prolongations of the smoothed-aggregation
// hierarchy of the stiffness matrix K (fixed per mesh), applied to the
// relaxation matrices M + K_{L^2} of the current statistics, whose Galerkin
// coarse matrices, smoothers and Q = (I - W A) P are recomputed on the
// device at every solve through precomputed plans.  Four operators
// ("variants"): the C_xi classes of wp_11, wp_22, wp_33 with their Dirichlet
// rows (no-slip nodes) and the off-diagonal components (walls and no-slip
// nodes).  Fixed unknowns carry identity rows and columns.
constexpr int kRxVar = 4;
constexpr int kRxMaxLv = 12;

struct RxLevel {
  int32_t n = 0, nc = 0;
  int64_t nnz_a = 0, nnz_ap = 0;
  int32_t *a_rp = nullptr, *a_ci = nullptr, *a_dpos = nullptr;  // A_l and its diagonal positions
  int32_t *q_rp = nullptr, *q_ci = nullptr;                      // pattern of A_l P_l = pattern of Q_l
  int32_t *s_rp = nullptr, *s_ci = nullptr, *s_perm = nullptr;   // Q_l^T: S[t] = Q[s_perm[t]]
  int32_t *ap_off = nullptr, *ap_qa = nullptr;                   // (A P)[t] = sum a[ap_qa] * ap_pv
  double* ap_pv = nullptr;
  int32_t *c_off = nullptr, *c_tap = nullptr;                    // A_{l+1}[c] = sum c_pv * (A P)[c_tap]
  double* c_pv = nullptr;
  double* q_pin = nullptr;                                       // P at each (A P) position, else 0
  int32_t* q_row = nullptr;
  double* a_v[kRxVar] = {};
  double* ap_v = nullptr;  // [nnz_ap][kRxVar]
  int64_t ap_terms = 0, c_terms = 0;  // terms of the two plans
  double* w_v[kRxVar] = {};  // smoother weights W = omega / a_ii
  // FP32 copies for the cycle: A, Q, S and W
  float *a_f[kRxVar] = {}, *q_f[kRxVar] = {}, *s_f[kRxVar] = {}, *w_f[kRxVar] = {};
  float *b = nullptr, *x = nullptr, *z = nullptr;                // [9][n] (b, z for l > 0; level 0's b is r32)
  char* mem = nullptr;  // the allocation of the arrays from a_v on (A P too)
};

struct RelaxAmg {
  std::vector<RxLevel> lv;
  int32_t nc = 0;
  int64_t nnz_c = 0;
  int32_t *c_rp = nullptr, *c_ci = nullptr;  // the coarsest matrix
  double* c_v[kRxVar] = {};
  float* cinv = nullptr;                     // [kRxVar][nc][nc]
  float* r32 = nullptr;                      // [9][n] FP32 residual, the finest level's b
  double *omega = nullptr, *gpart = nullptr; // [kRxVar][kRxMaxLv], Gershgorin partial maxima
  int32_t gblocks = 0;
  double* upart = nullptr;                   // [9][blocks of the finest up-sweep], r . z partials
};

// Device scalars (9 components each) and control words of the relaxation's
// conjugate gradients.
enum { kRPq = 0, kRRz = 9, kRRr = 18, kRBb = 27, kRTol2 = 36, kRAlpha = 45, kRBeta = 54 };
enum { kRDone = 0, kRIt = 1, kRMaxIt = 2, kRCntClose = 3, kRCntUp0 = 4, kRCntSpmv = 8, kRCntUpd = 17, kRActive = 26,
       kRIters = 35 };

// The nine components' systems (the matrices are the hierarchy's finest
// ones, on the pattern rp / ci) and the iteration's vectors
// ([9][n] each), as the caller's initialisation leaves them: x, r = b - A x,
// scal (r.r, the thresholds), ctl (active components, max_it).  wall[i]
// marks fixed unknowns (2 for every component; 1 for the off-diagonal
// components c != 0, 4, 8).  part: 18 doubles per 256 unknowns.
struct RxSystem {
  int32_t n = 0;
  const int32_t *rp = nullptr, *ci = nullptr;
  const uint8_t* wall = nullptr;
  double *x = nullptr, *r = nullptr, *z = nullptr, *p = nullptr, *q = nullptr, *part = nullptr, *scal = nullptr;
  int32_t* ctl = nullptr;
};

// Plans from the hierarchy of K (n unknowns, CSR rp / ci / kv), coarsest
// level at most 64 unknowns.
pdf_status relax_amg_setup(int32_t n, const std::vector<int32_t>& rp, const std::vector<int32_t>& ci,
                           const std::vector<double>& kv, RelaxAmg& G);
void relax_amg_free(RelaxAmg& G);
// The finest matrix values of variant v, on the relaxation pattern: filled
// by the caller before relax_amg_update.
inline double* relax_amg_level0(RelaxAmg& G, int v) { return G.lv.empty() ? G.c_v[v] : G.lv[0].a_v[v]; }
// The Galerkin matrices, smoother weights, Q and S of every level and the
// inverses of the coarsest matrices of the four variants, from the finest
// values (fixed unknowns with their diagonal only).
pdf_status relax_amg_update(RelaxAmg& G, cudaStream_t st);
// The conjugate gradients preconditioned by one V-cycle per iteration
// (relax_pcg.cu); component c uses variant 0, 1, 2 for c = 0, 4, 8 and 3
// otherwise.  The cycle runs in FP32 (level matrices and vectors), the
// rest in FP64.  relax_mg_whole: whether a system of n unknowns runs its whole
// solve up to iteration it_end in one launch (relax_mg_solve, which leaves
// scal[kRRr], ctl[kRIters] and ctl[kRActive], 0 for the converged components) or by relax_mg_begin (the first
// z = M^-1 r) and chunks of relax_mg_iterations (kernels that return at once
// when ctl[kRDone] is set).
bool relax_mg_whole(int32_t n);
pdf_status relax_mg_solve(const RelaxAmg& G, const RxSystem& A, int32_t it_end, cudaStream_t st);
pdf_status relax_mg_begin(const RelaxAmg& G, const RxSystem& A, cudaStream_t st);
pdf_status relax_mg_iterations(const RelaxAmg& G, const RxSystem& A, int k, cudaStream_t st);

}  // namespace pdfgb
