// Direct solve of a small periodic coarse stencil by cyclic reduction over lattice lines
// (coarsest_lines.cu), with the dense LU of the same matrix behind it.
#pragma once

#include <vector>

#include "common.cuh"

namespace mg {

// one level of the reduction: a ring of r lines of b dofs; line p couples to p +- 1 (mod r)
struct LineLevel {
  int r = 0, K = 0, E = 0;  // lines, kept (even positions), eliminated (odd positions)
  Cx<double> *D = nullptr, *R = nullptr, *L = nullptr;        // [r] blocks: self, next, previous (r <= 2: R holds both)
  Cx<double> *Dinv = nullptr, *WL = nullptr, *WR = nullptr;   // [E]: D^-1, D^-1 L, D^-1 R (r = 1: Dinv of the last line)
  long long rhs = 0, y = 0, x = 0;                            // offsets of the level's vectors in the workspace
  long long w_jobs = 0, u_jobs = 0;                           // first product of the level in the job list
  int n_w = 0, n_u = 0;
};

// C = I1 + I2 + sgn (A1 B1 + A2 B2) on b x b row-major blocks (null terms left out). band_a / band_b: the
// left / right factors' entries (i, k) vanish where |i - k| (cyclic in b) exceeds it; -1: full.
struct LineJob {
  Cx<double> *C;
  const Cx<double> *I1, *I2, *A1, *B1, *A2, *B2;
  double sgn;
  int band_a, band_b;
};

struct LineSolver {
  int N = 0, L0 = 0, L1 = 0, n = 0;
  int axis = 1, Q = 0, b = 0;  // line coordinate (1: lines along x0, one per x1), sites per line, dofs per line
  bool planned = false;
  enum class Kind { kNone, kLines, kDense };
  Kind kind = Kind::kNone;     // the factors in use; none before the first factorisation and after a failed one
  Kind last = Kind::kNone;     // of the last factorisation that succeeded: what a captured graph may hold
  std::vector<LineLevel> lv;
  std::vector<LineJob> jobs;
  DevBuf<Cx<double>> mem, tmp, pinv, chk;
  DevBuf<LineJob> jobs_dev;
  DevBuf<Cx<double>> LU;
  DevBuf<int> ipiv, info;      // info[0]: singular pivot seen
  DevBuf<double> berr;         // backward error of the check
};

// entries of the vector workspace that line_solve needs per right-hand side (shared between the
// solvers of one lattice; at least n, for the dense path)
long long line_work_size(Geo2 g, int N);
// Factors the 5-point stencil Y[j][dir][col][row] + shift (nine = false) or the 9-point stencil
// Y[j][o][row][col] (nine = true). work: workspace of one right-hand side. Synchronises s.
// Returns true when the kind of factors is another than at the last success (a graph captured with those is
// stale; a failure in between changes nothing about it); fails with MG_ERR_NAN ("... zero pivot at column k") on a singular matrix.
bool line_factor(LineSolver &f, const Cx<double> *Y, Geo2 g, int N, bool nine, double shift, Cx<double> *work,
                 cudaStream_t s, const char *what);
// x_v = A^{-1} b_v for nvec vectors of stride n (b and x may be equal); work: nvec workspaces. Fails with
// MG_ERR_STATE where the last factorisation failed.
void line_solve(const LineSolver &f, const Cx<double> *b, Cx<double> *x, int nvec, Cx<double> *work, cudaStream_t s);

}  // namespace mg
