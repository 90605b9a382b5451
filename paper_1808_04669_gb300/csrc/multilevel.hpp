// Multilevel preconditioner for the condensed facet system S lam = g of eq. (12)
// (Sec. 2.4) on meshes without the lattice structure (walls, perturbed or
// unstructured meshes), built once per mesh on the host. The paper factorises
// this system directly (Sec. 4); here it is solved by PCG, and block Jacobi
// alone needs O(1/h) iterations.
//
// Levels (finest first):
//   p-levels on the facet space: all k+1 Legendre modes of each facet, then modes
//   {0, 1} (k >= 2), then mode 0 (the facet-constant multipliers). Each is the
//   facet stencil of S restricted to its leading modes (the Galerkin operator of
//   the injection), applied matrix-free; transfers keep or add the leading modes.
//   h-levels: smoothed aggregation on the mode-0 operator (a zero-row-sum M-matrix:
//   its kernel is the constant multiplier). Aggregates from strong connections,
//   tentative prolongator from the near-null vector carried down the levels (so
//   the kernel stays exact on every level), one Jacobi smoothing step of the
//   prolongator, Galerkin coarse operators R A P with R = P^T.
//   The coarsest operator (<= kMLCoarseMax rows) is applied through its dense
//   pseudo-inverse (one grid-wide phase, where every further level would take
//   four or five).
// Smoothing: Chebyshev polynomials of degree 2 in B A with B the block-Jacobi
// inverse, on [lmax / 4, 1.1 lmax], lmax estimated by Lanczos (from CG
// coefficients). Pre- and post-smoothing use the same polynomial, so one V-cycle
// is a symmetric positive semi-definite preconditioner.
#pragma once

#include <cstdint>
#include <string>
#include <vector>

#include "setup.hpp"

namespace dgdf {

constexpr int kMLMaxLevels = 16;

// Layout of the solver kernel's operator tables (ml_operator_table). Rows of three values are
// padded to four (one 16-byte access); the class stride is 16 bytes past a multiple of 128, so that
// lanes of different classes hit different shared-memory banks.
#ifdef __CUDACC__
#define DGDF_HD __host__ __device__
#else
#define DGDF_HD
#endif
DGDF_HD constexpr int ml_row_stride(int nl) { return nl == 3 ? 4 : nl; }
// lanes a facet row of bs values takes, each ml_modes consecutive values of it
DGDF_HD constexpr int ml_lanes(int bs) { return bs == 1 ? 1 : bs == 2 || bs == 6 ? 2 : 4; }
DGDF_HD constexpr int ml_modes(int bs) { return bs == 6 ? 3 : 1; }
DGDF_HD constexpr int ml_class_stride(int nl, int nb, int word) {
  const int used = (nb + 1) * nl * ml_row_stride(nl) + 8;
  return (used * word + 127 - 16) / 128 * (128 / word) + 16 / word;
}
constexpr int kMLCoarseMax = 1024;

struct CsrHost {
  int n_rows = 0, n_cols = 0;
  std::vector<int32_t> rp, ci;
  std::vector<double> v;
};

// A sparse matrix in sliced rows for the device: a slice is the 32 / G rows of one warp, G lanes
// a row; slice s holds its entries step by step at [32 (ptr[s] + step) + lane], lane = row-in-slice
// G + p % G for the row's entry p = step G + p % G, short rows padded by zeros (column 0).
struct SellHost {
  int n_rows = 0, G = 1;
  std::vector<int32_t> ptr, ci;
  std::vector<double> v;
};

struct MLHostLevel {
  bool stencil = false;       // operator: the facet stencil on the first bs modes (else the CSR matrix A)
  int bs = 1;                 // values per row
  int n = 0;                  // rows (facets on stencil levels)
  std::vector<double> binv;   // stencil: [n_stencil][bs][bs] inverses of the own sub-blocks; CSR: [n] 1 / a_ii
  CsrHost A;                  // CSR levels
  bool inject = false;        // transfer to the next level keeps its leading modes (facet rows on both)
  CsrHost P, R;               // otherwise: prolongation [n x n_next] and restriction R = P^T
  int n_next = 0, bs_next = 1;
  double lmax = 0.0;          // estimate of the largest eigenvalue of B A
  double cheb[3] = {0, 0, 0}; // Chebyshev(2) coefficients c0 = 1 / theta, c1 = rho1 rho0, c2 = 2 rho1 / delta
  // one operator down and one up in place of the level's smoothing, residual and transfer phases
  // (fuse_levels): b_next = D b and x = U [b; x_next]
  bool fused = false;
  SellHost D, U;
};

struct MLHost {
  std::vector<MLHostLevel> lv;   // smoothing levels, finest first
  int nc = 0;                    // rows of the coarsest level
  std::vector<double> cpinv;     // [nc][nc] pseudo-inverse of the coarsest operator
};

// Fused operators of the levels with one value per row. With N b the Chebyshev(2) smoothing of
// A x = b from zero (N = ((1 + c1) c0 + c2) B - c2 c0 B A B), such a level of the V-cycle is
//   down: b_next = P^T (I - A N) b                       = D b
//   up:   x = N b + P x_next, then smoothed once more    = (2 N - N A N) b + D^T x_next
// so it takes two phases of sparse rows instead of five or six, of 3 us each with their barriers.
// The rows are longer (A's stencil to the third power). A level is fused while its operators hold at
// most kMLFuseFill times the entries of A (M2 once, D twice) and kMLFuseBytes in the V-cycle's
// precision (word = bytes a value), or goes into the dense operator (below), and only together with
// every coarser level. On triangles the ratio is 8 to 9 and the fused level wins (128^2 box, 49408
// rows: 10 us instead of 18); on the faces of tetrahedra it is 13 to 20, and its scattered rows lose
// (16^3 cubes, 49152 rows: 35 us instead of 20). Then the coarsest dense operator takes in the last fused level while that has at most
// dense_max rows: pinv <- 2 N - N A N + D^T pinv D. Results are those of the V-cycle up to rounding.
// grid_threads: threads of the solver's grid (lanes a row).
constexpr double kMLFuseBytes = 64e6;
constexpr double kMLFuseFill = 11.0;
void fuse_levels(MLHost& ml, int word, int dense_max, int grid_threads);

// Per-class operator tables of the solver kernel (class_tables = true): for each stencil class its
// nb blocks [nb][nl][rs], the block-Jacobi inverse of all modes [nl][rs], of the leading two modes
// [2][2] and of mode 0 (then 3 words of padding), rs = ml_row_stride(nl), classes ml_class_stride
// apart. Otherwise (more classes than a block can hold) one set a facet, transposed so that the
// lanes of a warp read consecutive words: [nb][nl (column)][facet][lanes x modes], then the three
// inverses [nl][facet][lanes x modes], [2][facet][2], [facet].
std::vector<double> ml_operator_table(bool class_tables, int nl, int nb, int n_cls, int n, const int32_t* cls,
                                      const double* blocks, int word);

// Builds the hierarchy from hm's facet stencil. Returns 0 or a dg_status code.
int build_multilevel(const HostMesh& hm, MLHost& ml, std::string& err);

// The same hierarchy from an assembled operator A0 (CSR, nl values per face, face-major): level 0
// keeps all modes and transfers to the face-constant multipliers (mode 0) by injection, then
// smoothed aggregation as above with point-Jacobi smoothing. Level 0 smooths with block Jacobi
// on its face stencil when cls (stencil class per face) and cls_binv ([class][nl][nl] inverses of
// the own blocks) are given (a stencil level, applied by the device through the level's own
// stencil pointers; the host V-cycle does not take it), else with point Jacobi on the CSR rows.
// Used for the face system of the three-dimensional path.
int build_multilevel_csr(const CsrHost& A0, int nl, const int32_t* cls, const std::vector<double>* cls_binv,
                         MLHost& ml, std::string& err);

// A block stencil operator as CSR: row block f couples to itself and to nbr[f][0..nb) through
// blocks[cls[f]][1 + nb][nl][nl] (slot 0 its own block); duplicate columns are merged.
CsrHost stencil_csr(int n, int nl, int nb, const int32_t* cls, const int32_t* nbr, const double* blocks);

// z = M r for one V-cycle, on the host (the reference of the device kernel);
// r and z hold n_facet (k+1) values.
void multilevel_apply_host(const HostMesh& hm, const MLHost& ml, const double* r, double* z);

}  // namespace dgdf
