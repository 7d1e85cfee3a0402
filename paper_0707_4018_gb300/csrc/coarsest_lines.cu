// Exact solve on a small coarsest level (paper: the coarsest level of the V-cycle is solved
// exactly): cyclic reduction over lattice lines, FP64.
//
// The coarse operator couples a site to its nearest neighbours (the normal equations' 9-point
// stencil: the diagonal ones too), so the dofs of one lattice line couple only to the two
// neighbouring lines: the matrix is a periodic block tridiagonal ring of r lines with b = Q N dofs
// each (Q: the shorter extent). One level eliminates every second line,
//     x_e = D_e^-1 (b_e - L_e x_prev - R_e x_next),
// which leaves a ring of half the lines with full b x b blocks; log2 r levels end in one line.
//
// GB300's FP64 rate (about 1 TFLOP/s, two multiply-adds per clock and SM) bounds this, not memory:
// the dense factorisation of n = 2048 dofs is 23 GFLOP and its triangular solves are a chain of
// 2048 steps; the ring of 16 lines x 128 dofs takes 1.8 GFLOP and a chain of 4 levels.
// Measured at n = 2048 (16 x 16 sites, N = 8): one solve 68 us (dense triangular solves: 3.4 ms);
// a 64^2 two-level FP64 setup and solve, 5 factorisations and 64 solves, 29.9 ms (dense: 524 ms), 22.8 with the
// other kernels of that path as they are now.
//
//  * D_e^-1: Gauss-Jordan over 16 x 16 sub-blocks, a CTA per 16 x 16 tile and line, one launch per
//    sub-block column; the CTA that finishes the next pivot block inverts it (partial pivoting
//    inside the sub-block), so no launch waits for an inversion of its own;
//  * every product: 16 x 16 tiles, one output per thread, so that even the last levels (a handful
//    of products) fill the chip;
//  * solve: a warp per row over all lines of the level, three launches per level.
//
// Pivots stay inside a 16 x 16 sub-block, which the near-positive Wilson operators do not mind
// but an arbitrary matrix may: every factorisation is followed by a solve for a fixed vector whose
// componentwise backward error must stay below kBackward; otherwise (and for rings of fewer than
// three lines) the dense LU with partial pivoting takes over. The bound is what that LU gives itself: on the same
// vector and the operators of 64^2 and smaller lattices at the couplings' masses the reduction has 3e-16 to 9.5e-16
// (n = 96 to 2048), the LU 7e-16 to 2.8e-15. Where the operator is indefinite (m = -1, -1.7) the reduction reaches
// 1.2e-12 and the LU 7.8e-15.
#include <algorithm>
#include <cmath>
#include <string>
#include <utility>

#include "coarsest_lines.h"
#include "kernels.h"

namespace mg {

namespace {

constexpr int kT = 16;                // tile edge
constexpr int kGridY = 65535;         // lines or products of one launch: the most that a grid's second extent takes
constexpr double kBackward = 2e-15;   // largest accepted |b - A x| / (|A| |x| + |b|), entry by entry

// position of dof i of line p in a level-0 vector (site-major); compact levels: axis 1
struct LineMap {
  int axis, L0, N, b;
  __device__ __forceinline__ long long at(int p, int i) const {
    if (axis == 1) return (long long)p * b + i;
    const int q = i / N;
    return ((long long)p + (long long)L0 * q) * N + (i - q * N);
  }
};

// blocks of the finest ring's lines p0, p0 + 1, ... from the stencil: which = 0 (self), 1 (next line), 2 (previous line)
__global__ void line_blocks_kernel(const Cx<double> *__restrict__ Y, Cx<double> *__restrict__ D,
                                   Cx<double> *__restrict__ R, Cx<double> *__restrict__ L, int L0, int L1, int N,
                                   int axis, int Q, int b, int p0, bool nine, double shift) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= (long long)b * b) return;
  const int i = (int)(t / b), k = (int)(t - (long long)i * b);
  const int p = p0 + blockIdx.y, which = blockIdx.z;
  const int q = i / N, a = i - q * N, qq = k / N, c = k - qq * N;
  const long long j = axis == 1 ? (long long)q + (long long)L0 * p : (long long)p + (long long)L0 * q;
  Cx<double> v = mk(0.0, 0.0);
  const int nd = nine ? 9 : 5;
  for (int d = 0; d < nd; ++d) {
    int o0, o1;
    if (nine) {
      o0 = d % 3 - 1;
      o1 = d / 3 - 1;
    } else {
      o0 = d == 1 ? 1 : d == 2 ? -1 : 0;
      o1 = d == 3 ? 1 : d == 4 ? -1 : 0;
    }
    const int dp = axis == 1 ? o1 : o0, dq = axis == 1 ? o0 : o1;
    if (dp != (which == 0 ? 0 : which == 1 ? 1 : -1)) continue;
    if ((q + dq + Q) % Q != qq) continue;
    v = v + (nine ? Y[((j * 9 + d) * N + a) * N + c] : Y[((j * 5 + d) * N + c) * N + a]);
  }
  if (which == 0 && i == k) v.re += shift;
  Cx<double> *out = which == 0 ? D : which == 1 ? R : L;
  out[(long long)p * b * b + t] = v;
}

// Inverse of the m x m block in `a` by 256 threads (thread = element), partial pivoting, result in `a`;
// *info = 1 on a pivot that is zero or not finite. A chain of m steps: warp 0 picks the pivot from the
// entries' FP32 magnitudes (one integer maximum; which of two nearly equal rows leads does not matter),
// inverts it and scales the pivot row, then every element is updated into the other buffer, so a step
// is two barriers and 16 x 16 complex multiply-adds. 11 us; with exact norms, a division by every
// thread's element and in-place updates 33 us.
__device__ __forceinline__ void invert_tile(Cx<double> (*a)[kT + 1], int m, int *info) {
  __shared__ Cx<double> other[kT][kT + 1], lead[kT];
  __shared__ Cx<double> dinv;
  __shared__ int piv[kT];
  const int i = threadIdx.x / kT, j = threadIdx.x % kT;
  const bool in = i < m && j < m;
  Cx<double>(*src)[kT + 1] = a, (*dst)[kT + 1] = other;
  for (int s = 0; s < m; ++s) {
    __syncthreads();
    if (threadIdx.x < 32) {
      const int lane = threadIdx.x;
      unsigned int key = 0u;
      if (lane >= s && lane < m)
        key = (__float_as_uint(fmaxf(fabsf((float)src[lane][s].re), fabsf((float)src[lane][s].im))) & ~15u) |
              (unsigned int)(15 - lane);
      key = __reduce_max_sync(0xffffffffu, key);
      const int p = 15 - (int)(key & 15u);
      const Cx<double> pv = src[p][s];
      const double inv = 1.0 / norm2(pv);
      const Cx<double> d = mk(pv.re * inv, -pv.im * inv);
      if (lane == 0) {
        piv[s] = p;
        dinv = d;
        if (!(inv > 0.0) || !isfinite(inv)) *info = 1;
      }
      if (lane < m) lead[lane] = src[p][lane] * d;
    }
    __syncthreads();
    if (in) {
      const int p = piv[s];
      const int row = i == s ? p : i == p ? s : i;  // rows s and p change places
      const Cx<double> as = src[row][s];
      Cx<double> v;
      if (i == s) {
        v = j == s ? dinv : lead[j];
      } else if (j == s) {
        v = as * dinv;
        v = mk(-v.re, -v.im);
      } else {
        v = src[row][j];
        cmac(v, mk(-as.re, -as.im), lead[j]);
      }
      dst[i][j] = v;
    }
    Cx<double>(*t)[kT + 1] = src;
    src = dst;
    dst = t;
  }
  // the row exchanges undone as column exchanges, last first: column j of the result
  __syncthreads();
  Cx<double> v = mk(0.0, 0.0);
  if (in) {
    int c = j;
    for (int s = 0; s < m; ++s) {  // where column j comes from: the exchanges in forward order
      const int p = piv[s];
      c = c == s ? p : c == p ? s : c;
    }
    v = src[i][c];
  }
  __syncthreads();
  if (in) a[i][j] = v;
  __syncthreads();
}

// inverse of the first pivot block of every line to be inverted
__global__ void __launch_bounds__(kT *kT) gj_first_kernel(const Cx<double> *__restrict__ src, long long stride, int b,
                                                          Cx<double> *__restrict__ pinv, int *info) {
  __shared__ Cx<double> a[kT][kT + 1];
  const int i = threadIdx.x / kT, j = threadIdx.x % kT, m = b < kT ? b : kT;
  src += blockIdx.x * stride;
  a[i][j] = i < m && j < m ? src[(long long)i * b + j] : mk(0.0, 0.0);
  invert_tile(a, m, info);
  pinv[((long long)blockIdx.x * 2) * kT * kT + threadIdx.x] = a[i][j];
}

// one Gauss-Jordan step over the 16 columns of sub-block k: dst = the matrix after the step.
// Bound by FP64 issue: 2 x 16^3 complex multiply-adds per tile, 8 us on an SM of its own.
__global__ void __launch_bounds__(kT *kT) gj_step_kernel(const Cx<double> *__restrict__ src, long long sstride,
                                                         Cx<double> *__restrict__ dst, long long dstride, int b, int k,
                                                         Cx<double> *__restrict__ pinv, int *info) {
  __shared__ Cx<double> P[kT][kT + 1], A[kT][kT + 1], B[kT][kT + 1];
  const int nt = (b + kT - 1) / kT;
  const int tr = blockIdx.x / nt, tc = blockIdx.x - tr * nt;
  const int i = threadIdx.x / kT, j = threadIdx.x % kT;
  const int r0 = tr * kT, c0 = tc * kT, k0 = k * kT;
  src += blockIdx.y * sstride;
  dst += blockIdx.y * dstride;
  pinv += (long long)blockIdx.y * 2 * kT * kT;
  auto get = [&](int r, int c) { return r < b && c < b ? src[(long long)r * b + c] : mk(0.0, 0.0); };
  P[i][j] = pinv[(k & 1) * kT * kT + threadIdx.x];
  A[i][j] = get(r0 + i, k0 + j);  // column panel
  B[i][j] = get(k0 + i, c0 + j);  // row panel
  Cx<double> v = tr == k || tc == k ? mk(0.0, 0.0) : get(r0 + i, c0 + j);
  __syncthreads();
  if (tr == k && tc == k) {
    v = P[i][j];
  } else if (tc == k) {
#pragma unroll
    for (int q = 0; q < kT; ++q) cmac(v, mk(-A[i][q].re, -A[i][q].im), P[q][j]);
  } else {
    Cx<double> t = mk(0.0, 0.0);
#pragma unroll
    for (int q = 0; q < kT; ++q) cmac(t, P[i][q], B[q][j]);
    if (tr == k) {
      v = t;
    } else {
      __syncthreads();
      B[i][j] = t;
      __syncthreads();
#pragma unroll
      for (int q = 0; q < kT; ++q) cmac(v, mk(-A[i][q].re, -A[i][q].im), B[q][j]);
    }
  }
  if (r0 + i < b && c0 + j < b) dst[(long long)(r0 + i) * b + c0 + j] = v;
  if (tr == k + 1 && tc == k + 1) {  // the next pivot block is final: invert it for the next launch
    __syncthreads();
    A[i][j] = v;
    invert_tile(A, b - r0 < kT ? b - r0 : kT, info);
    pinv[((k + 1) & 1) * kT * kT + threadIdx.x] = A[i][j];
  }
}

// whether 16 x 16 tiles whose first indexes differ by d can hold an entry within `band` (cyclic in b)
__device__ __forceinline__ bool in_band(int d, int b, int band) {
  const int lo = min(abs(d), min(abs(d - b), abs(d + b)));
  return lo - (kT - 1) <= band || b - (kT - 1) <= band;
}

// the block products of one level, at the FP64 rate. The couplings of the finest ring connect a site to
// the site(s) of the next line beside it: their products take 3 of 8 tiles at most (16 x 16 sites, N = 8:
// 1.2 instead of 1.9 ms of products per factorisation)
__global__ void __launch_bounds__(kT *kT) line_product_kernel(const LineJob *__restrict__ jobs, int b) {
  __shared__ Cx<double> A[kT][kT + 1], B[kT][kT + 1];
  const LineJob job = jobs[blockIdx.y];
  const int nt = (b + kT - 1) / kT;
  const int tr = blockIdx.x / nt, tc = blockIdx.x - tr * nt;
  const int i = threadIdx.x / kT, j = threadIdx.x % kT;
  const int r = tr * kT + i, c = tc * kT + j;
  const bool in = r < b && c < b;
  Cx<double> acc = mk(0.0, 0.0);
  for (int half = 0; half < 2; ++half) {
    const Cx<double> *Am = half ? job.A2 : job.A1, *Bm = half ? job.B2 : job.B1;
    if (Am == nullptr) continue;
    for (int k0 = 0; k0 < b; k0 += kT) {
      // tiles outside a factor's band hold zeros
      if (job.band_a >= 0 && !in_band(k0 - tr * kT, b, job.band_a)) continue;
      if (job.band_b >= 0 && !in_band(k0 - tc * kT, b, job.band_b)) continue;
      __syncthreads();
      A[i][j] = r < b && k0 + j < b ? Am[(long long)r * b + k0 + j] : mk(0.0, 0.0);
      B[i][j] = k0 + i < b && c < b ? Bm[(long long)(k0 + i) * b + c] : mk(0.0, 0.0);
      __syncthreads();
#pragma unroll
      for (int q = 0; q < kT; ++q) cmac(acc, A[i][q], B[q][j]);
    }
  }
  if (!in) return;
  const long long e = (long long)r * b + c;
  Cx<double> v = mk(job.sgn * acc.re, job.sgn * acc.im);
  if (job.I1 != nullptr) v = v + job.I1[e];
  if (job.I2 != nullptr) v = v + job.I2[e];
  job.C[e] = v;
}

// acc[v] += (row of M) . x_v, a warp per row; x_v(c) = x[v stride + map(p, c)]
template <int NR>
__device__ __forceinline__ void row_dot(Cx<double> (&acc)[NR], const Cx<double> *__restrict__ Mrow,
                                        const Cx<double> *__restrict__ x, long long stride, int nv, LineMap map, int p,
                                        int b, int lane) {
  for (int c = lane; c < b; c += 32) {
    const Cx<double> m = Mrow[c];
    const Cx<double> *xc = x + map.at(p, c);
#pragma unroll
    for (int v = 0; v < NR; ++v)
      if (v < nv) cmac(acc[v], m, xc[v * stride]);
  }
}

template <int NR>
__device__ __forceinline__ void warp_sum(Cx<double> (&acc)[NR]) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int v = 0; v < NR; ++v) {
      acc[v].re += __shfl_xor_sync(0xffffffffu, acc[v].re, o);
      acc[v].im += __shfl_xor_sync(0xffffffffu, acc[v].im, o);
    }
}

// what one launch of the solve does with the rows of a level
enum class Stage { kInverse, kReduce, kBack };

struct StageArgs {
  LineLevel lv;
  int b;
  LineMap in, out;             // maps of the level's right-hand side and solution
  const Cx<double> *rhs;       // level right-hand side
  Cx<double> *y;               // D_e^-1 rhs_e
  Cx<double> *next;            // kReduce: the next level's right-hand side
  const Cx<double> *xc;        // kBack: the next level's solution
  Cx<double> *x;               // kBack (and kInverse on the last line): this level's solution
  long long s_rhs, s_ws, s_x;  // vector strides
  int nvec;
};

template <Stage S, int NR>
__global__ void __launch_bounds__(256) line_stage_kernel(StageArgs g) {
  const int w = (int)((blockIdx.x * 256 + threadIdx.x) >> 5), lane = threadIdx.x & 31, b = g.b;
  const LineLevel &lv = g.lv;
  const int rows = (S == Stage::kInverse ? (lv.r == 1 ? 1 : lv.E) : S == Stage::kReduce ? lv.K : lv.r) * b;
  if (w >= rows) return;
  const int v0 = blockIdx.y * NR, nv = g.nvec - v0 < NR ? g.nvec - v0 : NR;
  const int p = w / b, i = w - p * b;
  const long long b2 = (long long)b * b, ro = (long long)i * b;
  const LineMap cm{1, 0, 1, b};  // compact vectors
  const Cx<double> *rhs = g.rhs + v0 * g.s_rhs;
  Cx<double> *y = g.y + v0 * g.s_ws;
  Cx<double> acc[NR];
#pragma unroll
  for (int v = 0; v < NR; ++v) acc[v] = mk(0.0, 0.0);
  if (S == Stage::kInverse) {
    row_dot<NR>(acc, lv.Dinv + p * b2 + ro, rhs, g.s_rhs, nv, g.in, lv.r == 1 ? 0 : 2 * p + 1, b, lane);
    warp_sum<NR>(acc);
    if (lane == 0) {
#pragma unroll
      for (int v = 0; v < NR; ++v)
        if (v < nv) {
          if (lv.r == 1)
            g.x[(v0 + v) * g.s_x + g.out.at(0, i)] = acc[v];
          else
            y[v * g.s_ws + w] = acc[v];
        }
    }
  } else if (S == Stage::kReduce) {
    const int pos = 2 * p;
    const int right = pos + 1 < lv.r ? p : -1;
    const int left = lv.r == 2 ? -1 : p > 0 ? p - 1 : lv.r % 2 == 0 ? lv.E - 1 : -1;
    if (right >= 0) row_dot<NR>(acc, lv.R + pos * b2 + ro, y, g.s_ws, nv, cm, right, b, lane);
    if (left >= 0) row_dot<NR>(acc, lv.L + pos * b2 + ro, y, g.s_ws, nv, cm, left, b, lane);
    warp_sum<NR>(acc);
    if (lane == 0) {
#pragma unroll
      for (int v = 0; v < NR; ++v)
        if (v < nv) g.next[(v0 + v) * g.s_ws + w] = rhs[v * g.s_rhs + g.in.at(pos, i)] - acc[v];
    }
  } else {
    const Cx<double> *xc = g.xc + v0 * g.s_ws;
    Cx<double> *x = g.x + v0 * g.s_x;
    if (p % 2 == 0) {  // a kept line
      if (lane < nv) x[lane * g.s_x + g.out.at(p, i)] = xc[lane * g.s_ws + (long long)(p / 2) * b + i];
      return;
    }
    const int e = p / 2;
    row_dot<NR>(acc, lv.WL + e * b2 + ro, xc, g.s_ws, nv, cm, e, b, lane);
    if (lv.r > 2) row_dot<NR>(acc, lv.WR + e * b2 + ro, xc, g.s_ws, nv, cm, (e + 1) % lv.K, b, lane);
    warp_sum<NR>(acc);
    if (lane == 0) {
#pragma unroll
      for (int v = 0; v < NR; ++v)
        if (v < nv) x[v * g.s_x + g.out.at(p, i)] = y[v * g.s_ws + (long long)e * b + i] - acc[v];
    }
  }
}

// the check's right-hand side: entries of modulus about 1 without structure
__global__ void check_vector_kernel(Cx<double> *x, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  unsigned int h = (unsigned int)i * 2654435761u;
  h ^= h >> 15;
  h *= 2246822519u;
  h ^= h >> 13;
  x[i] = mk((double)(h & 0xffff) / 32768.0 - 1.0, (double)(h >> 16) / 32768.0 - 1.0);
}

// largest |b - A x| / (|A| |x| + |b|) over the rows, a warp per row of the finest ring
__global__ void __launch_bounds__(256) check_kernel(LineLevel lv, int b, LineMap map, const Cx<double> *__restrict__ x,
                                                    const Cx<double> *__restrict__ rhs, double *worst) {
  const int w = (int)((blockIdx.x * 256 + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (w >= lv.r * b) return;
  const int p = w / b, i = w - p * b;
  Cx<double> acc = mk(0.0, 0.0);
  double mag = 0.0;
  for (int which = 0; which < 3; ++which) {
    const Cx<double> *M = (which == 0 ? lv.D : which == 1 ? lv.R : lv.L) + ((long long)p * b + i) * b;
    const int q = which == 0 ? p : which == 1 ? (p + 1) % lv.r : (p + lv.r - 1) % lv.r;
    for (int c = lane; c < b; c += 32) {
      const Cx<double> m = M[c], xv = x[map.at(q, c)];
      cmac(acc, m, xv);
      mag += sqrt(norm2(m) * norm2(xv));
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    acc.re += __shfl_xor_sync(0xffffffffu, acc.re, o);
    acc.im += __shfl_xor_sync(0xffffffffu, acc.im, o);
    mag += __shfl_xor_sync(0xffffffffu, mag, o);
  }
  if (lane == 0) {
    const Cx<double> bv = rhs[map.at(p, i)], d = bv - acc;
    const double e = sqrt(norm2(d)) / (mag + sqrt(norm2(bv)));
    // a value that is not a number counts as the worst one
    const unsigned long long bits = __double_as_longlong(e <= 1e300 ? e : 1e300);
    atomicMax(reinterpret_cast<unsigned long long *>(worst), bits);
  }
}

// the axis whose lines are shorter (fewer dofs per line), as (axis, Q, ring length)
void line_shape(Geo2 g, int &axis, int &Q, int &r) {
  axis = g.L0 <= g.L1 ? 1 : 0;
  Q = axis == 1 ? g.L0 : g.L1;
  r = axis == 1 ? g.L1 : g.L0;
}

// ring lengths of the reduction, and the offsets of its vectors
std::vector<LineLevel> line_levels(int r, int b, long long *ws) {
  std::vector<LineLevel> lv;
  long long off = 0;
  for (;;) {
    LineLevel l;
    l.r = r;
    l.K = (r + 1) / 2;
    l.E = r / 2;
    l.rhs = off;
    l.x = off + (long long)r * b;
    l.y = off + 2LL * r * b;
    off += (2LL * r + l.E) * b;
    lv.push_back(l);
    if (r == 1) break;
    r = l.K;
  }
  *ws = off;
  return lv;
}

// The plan is made aside and taken over whole: solvers of batched masses are planned inside a solve, and an
// allocation that fails there must leave the solver as one that was never planned.
void line_plan(LineSolver &solver, Geo2 g, int N, bool nine, cudaStream_t s) {
  if (solver.planned) return;
  LineSolver f;
  f.N = N;
  f.L0 = g.L0;
  f.L1 = g.L1;
  f.n = (int)(g.nsites * N);
  int r = 0;
  line_shape(g, f.axis, f.Q, r);
  f.b = f.Q * N;
  f.info.alloc(1);
  f.planned = true;
  if (r < 3) {
    pool_ready();
    solver = std::move(f);
    return;
  }
  long long ws = 0;
  f.lv = line_levels(r, f.b, &ws);
  const long long b2 = (long long)f.b * f.b;
  long long blocks = 0;
  for (const LineLevel &l : f.lv) blocks += 3LL * l.r + 3LL * (l.r == 1 ? 1 : l.E);
  f.mem.alloc((size_t)(blocks * b2));
  f.tmp.alloc((size_t)(std::max(f.lv[0].E, 1) * b2));
  f.pinv.alloc((size_t)std::max(f.lv[0].E, 1) * 2 * kT * kT);
  f.chk.alloc((size_t)2 * f.n);
  f.berr.alloc(1);
  Cx<double> *q = f.mem.p;
  auto take = [&](long long k) {
    Cx<double> *at = q;
    q += k * b2;
    return at;
  };
  for (LineLevel &l : f.lv) {
    l.D = take(l.r);
    l.R = take(l.r);
    l.L = take(l.r);
    const int e = l.r == 1 ? 1 : l.E;
    l.Dinv = take(e);
    l.WL = take(e);
    l.WR = take(e);
  }
  // the products of every level (see the file comment; r = 2 keeps both couplings in R)
  for (size_t k = 0; k + 1 < f.lv.size(); ++k) {
    LineLevel &l = f.lv[k];
    const LineLevel &c = f.lv[k + 1];
    const int band = k > 0 ? -1 : nine ? 2 * N - 1 : N - 1;  // of the couplings L and R
    l.w_jobs = (long long)f.jobs.size();
    for (int e = 0; e < l.E; ++e) {
      const Cx<double> *di = l.Dinv + e * b2;
      f.jobs.push_back({l.WL + e * b2, nullptr, nullptr, di, (l.r == 2 ? l.R : l.L) + (2 * e + 1) * b2, nullptr,
                        nullptr, 1.0, -1, band});
      if (l.r > 2)
        f.jobs.push_back({l.WR + e * b2, nullptr, nullptr, di, l.R + (2 * e + 1) * b2, nullptr, nullptr, 1.0, -1,
                          band});
    }
    l.n_w = (int)(f.jobs.size() - l.w_jobs);
    l.u_jobs = (long long)f.jobs.size();
    for (int a = 0; a < l.K; ++a) {
      const int pos = 2 * a;
      const int right = pos + 1 < l.r ? a : -1;
      const int left = l.r == 2 ? -1 : a > 0 ? a - 1 : l.r % 2 == 0 ? l.E - 1 : -1;
      const Cx<double> *Ra = l.R + pos * b2, *La = l.L + pos * b2;
      LineJob d{c.D + a * b2, l.D + pos * b2, nullptr, nullptr, nullptr, nullptr, nullptr, -1.0, band, -1};
      if (right >= 0) {
        d.A1 = Ra;
        d.B1 = l.WL + right * b2;
      }
      if (left >= 0) {
        d.A2 = La;
        d.B2 = l.WR + left * b2;
      }
      f.jobs.push_back(d);
      if (l.K == 1) continue;
      // couplings of the kept line to the next and to the previous kept line
      LineJob n{c.R + a * b2, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, -1.0, band, -1};
      LineJob v{c.L + a * b2, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, -1.0, band, -1};
      if (right >= 0) {
        n.A1 = Ra;
        n.B1 = l.WR + right * b2;
      } else {
        n.I1 = Ra;
      }
      LineJob &p = l.K == 2 ? n : v;  // two lines: both couplings go to the same line
      if (left >= 0) {
        p.A2 = La;
        p.B2 = l.WL + left * b2;
      } else {
        p.I2 = La;
      }
      f.jobs.push_back(n);
      if (l.K > 2) f.jobs.push_back(v);
    }
    l.n_u = (int)(f.jobs.size() - l.u_jobs);
  }
  f.jobs_dev.alloc(f.jobs.size());
  pool_ready();
  MG_CUDA(cudaMemcpyAsync(f.jobs_dev.p, f.jobs.data(), f.jobs.size() * sizeof(LineJob), cudaMemcpyHostToDevice, s));
  solver = std::move(f);
}

// Dinv of `count` blocks at src (stride in entries)
void line_inverse(LineSolver &f, const Cx<double> *src, long long stride, int count, Cx<double> *Dinv, cudaStream_t s) {
  const int b = f.b, nt = (b + kT - 1) / kT;
  const long long b2 = (long long)b * b;
  gj_first_kernel<<<count, kT * kT, 0, s>>>(src, stride, b, f.pinv.p, f.info.p);
  MG_LAUNCHED();
  for (int k = 0; k < nt; ++k) {
    Cx<double> *dst = (nt - 1 - k) % 2 == 0 ? Dinv : f.tmp.p;
    for (int c = 0; c < count; c += kGridY) {
      gj_step_kernel<<<dim3(nt * nt, std::min(count - c, kGridY)), kT * kT, 0, s>>>(
          src + c * stride, stride, dst + c * b2, b2, b, k, f.pinv.p + (long long)c * 2 * kT * kT, f.info.p);
      MG_LAUNCHED();
    }
    src = dst;
    stride = b2;
  }
}

void line_products(const LineSolver &f, long long first, int count, cudaStream_t s) {
  const int nt = (f.b + kT - 1) / kT;
  for (int c = 0; c < count; c += kGridY) {
    line_product_kernel<<<dim3(nt * nt, std::min(count - c, kGridY)), kT * kT, 0, s>>>(f.jobs_dev.p + first + c, f.b);
    MG_LAUNCHED();
  }
}

template <Stage S>
void launch_stage(const StageArgs &a, int rows, cudaStream_t s) {
  const unsigned int gx = (unsigned int)((rows + 7) / 8);
  if (a.nvec == 1)
    line_stage_kernel<S, 1><<<gx, 256, 0, s>>>(a);
  else
    line_stage_kernel<S, 4><<<dim3(gx, (a.nvec + 3) / 4), 256, 0, s>>>(a);
  MG_LAUNCHED();
}

void line_reduce_solve(const LineSolver &f, const Cx<double> *b, Cx<double> *x, int nvec, Cx<double> *work,
                       cudaStream_t s) {
  const LineMap outer{f.axis, f.L0, f.N, f.b}, compact{1, 0, 1, f.b};
  const LineLevel &last = f.lv.back();
  const long long ws = last.rhs + (2LL * last.r + last.E) * f.b;  // workspace of one right-hand side
  auto args = [&](size_t k) {
    const LineLevel &l = f.lv[k];
    StageArgs a;
    a.lv = l;
    a.b = f.b;
    a.nvec = nvec;
    a.in = a.out = k == 0 ? outer : compact;
    a.rhs = k == 0 ? b : work + l.rhs;
    a.s_rhs = k == 0 ? f.n : ws;
    a.x = k == 0 ? x : work + l.x;
    a.s_x = k == 0 ? f.n : ws;
    a.y = work + l.y;
    a.s_ws = ws;
    a.next = k + 1 < f.lv.size() ? work + f.lv[k + 1].rhs : nullptr;
    a.xc = k + 1 < f.lv.size() ? work + f.lv[k + 1].x : nullptr;
    return a;
  };
  for (size_t k = 0; k + 1 < f.lv.size(); ++k) {
    const StageArgs a = args(k);
    launch_stage<Stage::kInverse>(a, a.lv.E * f.b, s);
    launch_stage<Stage::kReduce>(a, a.lv.K * f.b, s);
  }
  launch_stage<Stage::kInverse>(args(f.lv.size() - 1), f.b, s);
  for (size_t k = f.lv.size() - 1; k-- > 0;) {
    const StageArgs a = args(k);
    launch_stage<Stage::kBack>(a, a.lv.r * f.b, s);
  }
}

// cyclic reduction and its check; false: use the dense LU
bool line_try(LineSolver &f, const Cx<double> *Y, bool nine, double shift, Cx<double> *work, cudaStream_t s) {
  if (f.lv.empty()) return false;
  const long long b2 = (long long)f.b * f.b;
  MG_CUDA(cudaMemsetAsync(f.info.p, 0, sizeof(int), s));
  MG_CUDA(cudaMemsetAsync(f.berr.p, 0, sizeof(double), s));
  LineLevel &t = f.lv[0];
  for (int p = 0; p < t.r; p += kGridY) {
    line_blocks_kernel<<<dim3(grid_for(b2, 256), std::min(t.r - p, kGridY), 3), 256, 0, s>>>(
        Y, t.D, t.R, t.L, f.L0, f.L1, f.N, f.axis, f.Q, f.b, p, nine, shift);
    MG_LAUNCHED();
  }
  for (size_t k = 0; k < f.lv.size(); ++k) {
    LineLevel &l = f.lv[k];
    if (l.r == 1) {
      line_inverse(f, l.D, b2, 1, l.Dinv, s);
      break;
    }
    line_inverse(f, l.D + b2, 2 * b2, l.E, l.Dinv, s);
    line_products(f, l.w_jobs, l.n_w, s);
    line_products(f, l.u_jobs, l.n_u, s);
  }
  check_vector_kernel<<<grid_for(f.n, 256), 256, 0, s>>>(f.chk.p, f.n);
  MG_LAUNCHED();
  line_reduce_solve(f, f.chk.p, f.chk.p + f.n, 1, work, s);
  check_kernel<<<grid_for((long long)f.n * 32, 256), 256, 0, s>>>(t, f.b, LineMap{f.axis, f.L0, f.N, f.b},
                                                                   f.chk.p + f.n, f.chk.p, f.berr.p);
  MG_LAUNCHED();
  int info = 0;
  double err = 0.0;
  MG_CUDA(cudaMemcpyAsync(&info, f.info.p, sizeof(int), cudaMemcpyDeviceToHost, s));
  MG_CUDA(cudaMemcpyAsync(&err, f.berr.p, sizeof(double), cudaMemcpyDeviceToHost, s));
  MG_CUDA(cudaStreamSynchronize(s));
  return info == 0 && err <= kBackward;
}

}  // namespace

long long line_work_size(Geo2 g, int N) {
  int axis, Q, r;
  line_shape(g, axis, Q, r);
  long long ws = 0;
  (void)line_levels(r, Q * N, &ws);
  return std::max(ws, (long long)g.nsites * N);
}

bool line_factor(LineSolver &f, const Cx<double> *Y, Geo2 g, int N, bool nine, double shift, Cx<double> *work,
                 cudaStream_t s, const char *what) {
  f.kind = LineSolver::Kind::kNone;
  line_plan(f, g, N, nine, s);
  const bool lines = line_try(f, Y, nine, shift, work, s);
  if (!lines) {
    if (f.ipiv.p == nullptr) {  // the later of the two: both are there or both are made
      f.LU.alloc((size_t)f.n * f.n);
      f.ipiv.alloc((size_t)f.n);
      pool_ready();
    }
    if (nine)
      launch_dense_from_stencil9(Y, f.LU.p, g, N, s);
    else
      launch_dense_from_stencil(Y, f.LU.p, g, N, s, shift);
    lu_factor(f.LU.p, f.n, f.ipiv.p, f.info.p, s);
    int info = 0;
    MG_CUDA(cudaMemcpyAsync(&info, f.info.p, sizeof(int), cudaMemcpyDeviceToHost, s));
    MG_CUDA(cudaStreamSynchronize(s));
    if (info != 0) fail(MG_ERR_NAN, std::string(what) + ": zero pivot at column " + std::to_string(info - 1));
  }
  const LineSolver::Kind was = f.last;
  f.kind = f.last = lines ? LineSolver::Kind::kLines : LineSolver::Kind::kDense;
  return was != LineSolver::Kind::kNone && was != f.last;
}

void line_solve(const LineSolver &f, const Cx<double> *b, Cx<double> *x, int nvec, Cx<double> *work, cudaStream_t s) {
  if (f.kind == LineSolver::Kind::kNone) fail(MG_ERR_STATE, "the coarsest level has no factors: factoring it failed");
  if (f.kind == LineSolver::Kind::kLines) {
    line_reduce_solve(f, b, x, nvec, work, s);
    return;
  }
  for (int v = 0; v < nvec; ++v)
    lu_solve_ws(f.LU.p, f.ipiv.p, f.n, b + (long long)v * f.n, x + (long long)v * f.n, work, s);
}

}  // namespace mg
