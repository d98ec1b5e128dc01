// Device kernels of the two-site DMRG hot path and their launch wrappers.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace gbdmrg {

// One contribution C += alpha * op(A) * op(B) to an output block.
//   A: m x k row-major (lda) unless GT_TA: then A is stored k x m (A^T used)
//   B: n x k row-major (ldb)   (C = A B^T)  unless GT_BN: stored k x n (C = A B)
enum : int { GT_TA = 1, GT_BN = 2 };
struct GemmTerm {
  const double* A;
  const double* B;
  int lda, ldb, k, flags;
  double alpha;
};
// One output block: C (m x n, row-major ldc) = beta*C + sum_{t in [t0,t1)} terms
struct GemmTask {
  double* C;
  int ldc, m, n;
  int beta;
  int t0, t1;
};
// One tile of an output block.  A block of m rows is cut into gemm_parts(m, cap) nearly
// equal row ranges (no range longer than cap, lengths differing by at most one), and its
// columns likewise.  rows, cols: the first row or column in the low 24 bits, the length
// (at most 64) above them.
struct GemmTile {
  int task, rows, cols;
};

// tile edges of the FP64 grouped GEMM (the largest row or column count of a tile)
constexpr int GEMM_CAPS[3] = {8, 16, 32};
inline int gemm_parts(int n, int cap) { return (n + cap - 1) / cap; }
// range i of the `parts` ranges of n (n < 2^24)
inline int gemm_range(int n, int parts, int i) {
  const int a = (int)((long)n * i / parts), b = (int)((long)n * (i + 1) / parts);
  return a | (b - a) << 24;
}
// The edge for a launch whose blocks are at most max_dim in either direction, given the
// number of tiles ntiles[i] it has with each GEMM_CAPS[i]: see launch_gemm.
int gemm_pick_cap(int max_dim, const long ntiles[3]);

// Linear combination of operators with a common block layout:
//   out_j[e] = sum_{t in [c0_j, c1_j)} coef_t * in_t[e],  e < nnz_j
struct ComboOut {
  double* out;
  long nnz;
  int t0, t1;
};
struct ComboTerm {
  const double* in;
  double coef;
};

// Copy of a 2-D sub-block: dst[i*ldd + j] = alpha * src[i*lds + j] (or src[j*lds + i] if trans)
struct CopyJob {
  const double* src;
  double* dst;
  int rows, cols, lds, ldd, trans;
  double alpha;
};

// number of kernel launches issued by this library (all launch wrappers)
long launch_count();
// adds kernel launches made outside this file to the count
void count_launches(long n);

// cap: the tile edge the tiles were cut with (one of GEMM_CAPS), or 64: then every listed
// tile is taken by four thread blocks, one per quarter (a list of a quarter of the length).
// Every B is read b_shift elements and every C written c_shift elements further than its
// descriptor says (a plan made for one vector serves any).
void launch_gemm(const GemmTile* d_tiles, int ntiles, const GemmTask* d_tasks,
                 const GemmTerm* d_terms, int cap, cudaStream_t s, long b_shift = 0, long c_shift = 0);
void launch_combo(const ComboOut* d_outs, int nouts, long max_nnz, const ComboTerm* d_terms,
                  cudaStream_t s);
void launch_copy(const CopyJob* d_jobs, int njobs, int max_elems, cudaStream_t s);
void launch_fill(double* p, long n, double v, cudaStream_t s);

// vector ops (FP64, length n)
// y = a x + b y (b == 0: y is only written)
void launch_axpby(long n, double a, const double* x, double b, double* y, cudaStream_t s);
// Workspace of the reductions below: partial sums of up to DOT_MAX dots over DOT_BLOCKS blocks
// and a counter (zero before the first use; every launch leaves it at zero).  One launch
// at a time may use it.
constexpr int DOT_MAX = 49, DOT_BLOCKS = 304;
struct DotWork {
  double* part;  // DOT_MAX * DOT_BLOCKS
  unsigned* count;
};
// dots[j] = <V_j, x> for j < m, V row-major [m][n]; result written to d_out[m] (deterministic)
// and, where G is given, to row and column `col` of G
void launch_multidot(const double* V, long ldv, int m, const double* x, long n, DotWork w, double* d_out,
                     cudaStream_t s, double* G = nullptr, int ldg = 0, int col = 0);
// t = r / (theta - diag), |denominator| clamped to >= eps
void launch_precond(long n, const double* r, const double* diag, double theta, double eps,
                    double* t, cudaStream_t s);
// diagonal extraction: out[i * ldo + col] = coef * A[i*(lda+1)]  for i < rows
struct DiagJob {
  const double* A;
  double* out;
  int rows, lda, ldo;
  double coef;
};
void launch_diag_extract(const DiagJob* d_jobs, int njobs, int max_rows, cudaStream_t s);

// Davidson on the device (FP64).  Rayleigh-Ritz: lowest eigenpair of the symmetric
// part of the m x m projected matrix G (m <= 48) by parallel cyclic Jacobi in one
// thread block; eigenvalue to scal[0] (NaN where it does not converge in max_sweeps sweeps),
// eigenvector to y[0..m).  false (nothing launched) if m is outside [1, RR_MAX_SUB]
constexpr int RR_MAX_SUB = 48, JAC_SWEEPS = 60;
// Eigen-decompositions of symmetric d x d matrices (row-major, d <= EIGH_MAX), one thread block
// each: w the eigenvalues in ascending order, row i of G the eigenvector of w[i]; *info is set to
// 1 (and w to NaN) if the matrix is not finite or does not converge in max_sweeps sweeps
constexpr int EIGH_MAX = 32;
struct EighJob {
  double* G;
  double* w;
  int* info;
  int d;
};
void launch_eigh(const EighJob* d_jobs, int njobs, cudaStream_t s, int max_sweeps = JAC_SWEEPS);
bool launch_rr(const double* G, int ldg, int m, double* y, double* scal, cudaStream_t s, int max_sweeps = JAC_SWEEPS);
// One Davidson iteration's vectors from the subspace V, its sigma vectors S and the Ritz
// coefficients c: x = sum_j c_j V_j, hx = sum_j c_j S_j, r = hx - theta x (theta on device), the
// diagonal correction t = r / (theta - diag) with |denominator| >= eps, and *rr = |r|^2
void launch_ritz(const double* V, const double* S, long ldv, int m, const double* d_c, long n, const double* d_theta,
                 const double* diag, double eps, double* x, double* hx, double* r, double* t, DotWork w, double* rr,
                 cudaStream_t s);
// t -= sum_j c[j] V_j (c on device), then dots[j] = <V_j, t>
void launch_project(const double* V, long ldv, int m, const double* d_c, long n, double* t, DotWork w, double* dots,
                    cudaStream_t s);
// t -= sum_j c[j] V_j (c on device), then *tt = |t|^2
void launch_project_norm(const double* V, long ldv, int m, const double* d_c, long n, double* t, DotWork w, double* tt,
                         cudaStream_t s);
// y = x / sqrt(*nrm2)
void launch_scale_rsqrt(long n, const double* x, const double* d_nrm2, double* y, cudaStream_t s);
// G[0] = theta / xn2
void launch_restart_g(double* G, const double* d_theta, const double* d_xn2, cudaStream_t s);

}  // namespace gbdmrg
