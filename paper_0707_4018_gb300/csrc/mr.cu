// Fused minimum-residual (MR) smoothing kernels (paper: the relaxation steps
// of the V-cycle; MR with under-relaxation omega as the relaxation method).
//
// One MR iteration is  alpha = omega <A r, r> / |A r|^2,  x += alpha r,
// r -= alpha A r. Unfused, that is three kernels (apply, reduce, update). Here
// an iteration is one kernel: it reads the previous r and A r, forms
// r_new = r - alpha A r on the fly at the neighbours it needs, updates x and r
// at its own site, applies A to r_new and publishes its block's sums of
// <A r_new, r_new> and |A r_new|^2. nu MR iterations cost nu + 1 launches.
//
// Reductions are finished by the consumer: every block of the next launch sums
// the previous launch's block partials itself, in one fixed order (so every
// block, and every run, forms the same alpha), while its own loads of r, A r
// and the operator are already in flight. The producer has no tail (no fence,
// ticket or last block), which matters because these small levels are latency-
// bound. Partials alternate between two buffers; r and A r alternate between
// two buffers too, so no thread overwrites a value another thread still reads.
// Sums are in the vectors' precision.
#include "kernels.h"
#include "mr.cuh"
#include "stencil8.cuh"
#include "wilson.cuh"

namespace mg {

// ---- fine Wilson level: one thread per site ----
template <typename R, bool STEP, bool LOOP>
__global__ void __launch_bounds__(256) mr_wilson_kernel(const Cx<R> *__restrict__ U, const Cx<R> *r_old,
                                                        const Cx<R> *Ar_old, const R *part_in, int nb_in,
                                                        double omega, Cx<R> *x, int x_init, Cx<R> *r_new,
                                                        Cx<R> *Ar_new, int L0, int L1, R diag, R *part_out,
                                                        const double *shift) {
  __shared__ R sh[32 * 3];
  if (shift != nullptr) diag += (R)shift[blockIdx.y];
  const long long V = (long long)L0 * L1;
  {  // vector blockIdx.y of the batch (stride 2 V); partials per vector
    const long long off = blockIdx.y * 2 * V;
    r_old += off;
    if (STEP) {
      Ar_old += off;
      x += off;
      r_new += off;
      part_in += 3LL * nb_in * blockIdx.y;
    }
    Ar_new += off;
    part_out += 3LL * gridDim.x * blockIdx.y;
  }
  const Cx<R> z = mk((R)0, (R)0);
  Cx<R> alpha = z;
  R v[3] = {(R)0, (R)0, (R)0};
  // every block makes its first pass (alpha is a block-wide sum), then strides on
  const long long sb = blockIdx.x * (long long)blockDim.x;
  long long s0 = sb;
  do {
    const long long s = s0 + threadIdx.x;
    // issue every load of the site first; alpha (a reduction) overlaps with them
    const bool live = s < V;
    Cx<R> rv[10], av[10];  // self, +0, +1, -0, -1 (two spin components each)
    Cx<R> xa = z, xb = z, ux0 = z, ux1 = z, ub0 = z, ub1 = z;
#pragma unroll
    for (int k = 0; k < 10; ++k) rv[k] = av[k] = z;
    if (live) {
      const int x1 = (int)(s / L0), x0 = (int)(s - (long long)x1 * L0);
      const long long row = (long long)x1 * L0;
      const long long nbr[5] = {s, row + (x0 + 1 == L0 ? 0 : x0 + 1), (x1 + 1 == L1 ? 0 : row + L0) + x0,
                                row + (x0 == 0 ? L0 - 1 : x0 - 1),
                                (x1 == 0 ? (long long)(L1 - 1) * L0 : row - L0) + x0};
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        rv[2 * k] = r_old[2 * nbr[k]];
        rv[2 * k + 1] = r_old[2 * nbr[k] + 1];
        if (STEP) {
          av[2 * k] = Ar_old[2 * nbr[k]];
          av[2 * k + 1] = Ar_old[2 * nbr[k] + 1];
        }
      }
      if (STEP && !x_init) {
        xa = x[2 * s];
        xb = x[2 * s + 1];
      }
      const Pair<R> ux = reinterpret_cast<const Pair<R> *>(U)[s];
      ux0 = ux.a;
      ux1 = ux.b;
      ub0 = U[2 * nbr[3] + 0];
      ub1 = U[2 * nbr[4] + 1];
    }
    if (STEP && (!LOOP || s0 == sb))
      alpha = mr_alpha<R>(part_in, nb_in, omega, sh);  // all threads of the block
    if (live) {
      const Cx<R> ma = mk(-alpha.re, -alpha.im);
      Cx<R> w[10];
#pragma unroll
      for (int k = 0; k < 10; ++k) w[k] = STEP ? mr_step(rv[k], av[k], ma) : rv[k];
      if (STEP) {
        cmac(xa, alpha, rv[0]);
        cmac(xb, alpha, rv[1]);
        x[2 * s] = xa;
        x[2 * s + 1] = xb;
        r_new[2 * s] = w[0];
        r_new[2 * s + 1] = w[1];
      }
      const Cx<R> p0 = w[0], p1 = w[1];
      const Cx<R> t1 = ux0 * (w[2] - w[3]);                    // +0: (1 - s1) U psi(x+0)
      const Cx<R> t2 = cmul_conj(ub0, w[6] + w[7]);            // -0: (1 + s1) U^* psi(x-0)
      const Cx<R> t3 = ux1 * (w[4] + times_i(w[5]));           // +1: (1 - s2) U psi(x+1)
      const Cx<R> t4 = cmul_conj(ub1, w[8] - times_i(w[9]));   // -1: (1 + s2) U^* psi(x-1)
      const Cx<R> hu = mk(t1.re + t2.re + t3.re + t4.re, t1.im + t2.im + t3.im + t4.im);
      const Cx<R> hl = mk(-t1.re + t2.re + t3.im - t4.im, -t1.im + t2.im - t3.re + t4.re);
      const R h = (R)0.5;
      const Cx<R> a0 = mk(diag * p0.re - h * hu.re, diag * p0.im - h * hu.im);
      const Cx<R> a1 = mk(diag * p1.re - h * hl.re, diag * p1.im - h * hl.im);
      Ar_new[2 * s] = a0;
      Ar_new[2 * s + 1] = a1;
      v[0] += a0.re * p0.re + a0.im * p0.im + a1.re * p1.re + a1.im * p1.im;
      v[1] += a0.re * p0.im - a0.im * p0.re + a1.re * p1.im - a1.im * p1.re;
      v[2] += a0.re * a0.re + a0.im * a0.im + a1.re * a1.re + a1.im * a1.im;
    }
    s0 += gridDim.x * (long long)blockDim.x;
  } while (LOOP && s0 < V);
  mr_publish<R>(v, part_out, sh);
}

// ---- coarse stencil level in FP64, N = 8: a warp per site, four threads per row ----
// Thread q of a row takes 10 of the 40 (direction, column) terms. FP64 issue bounds it (an instruction holds the SM's
// pipe for 16 cycles), so nothing is worked out twice: the 40 source entries r - alpha A r are formed once per warp,
// in shared memory, beside the blocks' loads; the four lanes of a row share the update's components and the three
// sums. 69 FP64 instructions per site; accumulating Y r and Y (A r) to have the products before alpha took 120.
// 64^2 sites, one vector: 26.4 us an iteration, 44.1 before; without the step 16.7, 22.9 before.
template <bool STEP, bool LOOP>
__global__ void __launch_bounds__(256) mr_stencil8_kernel(const Cx<double> *__restrict__ Y, const Cx<double> *r_old,
                                                          const Cx<double> *Ar_old, const double *part_in, int nb_in,
                                                          double omega, Cx<double> *x, int x_init, Cx<double> *r_new,
                                                          Cx<double> *Ar_new, int L0, int L1, double *part_out,
                                                          const double *shift) {
  using C = Cx<double>;
  __shared__ double sh[32 * 3];
  __shared__ C ws[8][40];
  {
    const long long off = blockIdx.y * (long long)L0 * L1 * 8;
    r_old += off;
    if (STEP) {
      Ar_old += off;
      x += off;
      r_new += off;
      part_in += 3LL * nb_in * blockIdx.y;
    }
    Ar_new += off;
    part_out += 3LL * gridDim.x * blockIdx.y;
  }
  const int lane = threadIdx.x & 31, row = lane >> 2, q = lane & 3;
  C *w = ws[threadIdx.x >> 5];
  const long long sites = (long long)L0 * L1, jb = blockIdx.x * 8LL;
  const C z = mk(0.0, 0.0);
  C alpha = z;
  double sum = 0.0;  // lane q: <A r, r> re, im, |A r|^2, none
  long long j0 = jb;
  do {
    const long long j = j0 + (threadIdx.x >> 5);
    const bool live = j < sites;  // uniform over the warp
    const long long i = j * 8 + row;
    C y[10], wr[2], wa[2], rself = z;
    double xc = 0.0;
#pragma unroll
    for (int u = 0; u < 2; ++u) wr[u] = wa[u] = z;
    if (live) {
      const int x1 = (int)(j / L0), x0 = (int)(j - (long long)x1 * L0);
      const long long rowo = (long long)x1 * L0;
      const long long xp0 = rowo + (x0 + 1 == L0 ? 0 : x0 + 1);
      const long long xm0 = rowo + (x0 == 0 ? L0 - 1 : x0 - 1);
      const long long xp1 = (x1 + 1 == L1 ? 0 : rowo + L0) + x0;
      const long long xm1 = (x1 == 0 ? (long long)(L1 - 1) * L0 : rowo - L0) + x0;
      // source entries: lane = 8 direction + column for directions 0 to 3, lanes 0 to 7 those of direction 4
      const int dir = lane >> 3, col = lane & 7;
      const long long e0 = (dir == 0 ? j : dir == 1 ? xp0 : dir == 2 ? xm0 : xp1) * 8 + col, e1 = xm1 * 8 + col;
      wr[0] = r_old[e0];
      if (STEP) wa[0] = Ar_old[e0];
      if (lane < 8) {
        wr[1] = r_old[e1];
        if (STEP) wa[1] = Ar_old[e1];
      }
      if (STEP && q < 2) {
        rself = r_old[i];
        if (!x_init) xc = reinterpret_cast<const double *>(x + i)[q];
      }
#pragma unroll
      for (int u = 0; u < 10; ++u) {
        const int term = q * 10 + u;
        y[u] = Y[(j * 5 + (term >> 3)) * 64 + (term & 7) * 8 + row];
      }
    }
    if (STEP && (!LOOP || j0 == jb)) alpha = mr_alpha<double>(part_in, nb_in, omega, sh);  // all threads of the block
    if (live) {
      const C ma = mk(-alpha.re, -alpha.im);
      if (LOOP) __syncwarp();  // the site before is done with
      w[lane] = STEP ? mr_step(wr[0], wa[0], ma) : wr[0];
      if (lane < 8) w[32 + lane] = STEP ? mr_step(wr[1], wa[1], ma) : wr[1];
      __syncwarp();
      C acc = z;
#pragma unroll
      for (int u = 0; u < 10; ++u) cmac(acc, y[u], w[q * 10 + u]);
#pragma unroll
      for (int o = 1; o < 4; o <<= 1) {
        acc.re += __shfl_xor_sync(0xffffffffu, acc.re, o);
        acc.im += __shfl_xor_sync(0xffffffffu, acc.im, o);
      }
      const C self = w[row];
      if (STEP && q < 2) {
        xc = fma(alpha.re, q == 0 ? rself.re : rself.im, xc);
        xc = fma(q == 0 ? -alpha.im : alpha.im, q == 0 ? rself.im : rself.re, xc);
        reinterpret_cast<double *>(x + i)[q] = xc;
        if (q == 0) r_new[i] = self;
      }
      if (shift != nullptr) {
        const double sv = shift[blockIdx.y];
        acc.re = fma(sv, self.re, acc.re);
        acc.im = fma(sv, self.im, acc.im);
      }
      if (q == 0) Ar_new[i] = acc;
      const double p0 = q == 0 ? self.re : q == 1 ? self.im : q == 2 ? acc.re : 0.0;
      const double p1 = q == 0 ? self.im : q == 1 ? -self.re : q == 2 ? acc.im : 0.0;
      sum = fma(acc.re, p0, sum);
      sum = fma(acc.im, p1, sum);
    }
    j0 += gridDim.x * 8LL;
  } while (LOOP && j0 < sites);
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  mr_publish_lanes<double>(sum, part_out, sh);
}

// ---- the same in FP32: a warp per site and VB vectors, the site's blocks loaded once for them ----
template <bool STEP, bool LOOP, int VB>
__global__ void __launch_bounds__(256) mr_stencil8_f32_kernel(const Cx<float> *__restrict__ Y, const Cx<float> *r_old,
                                                              const Cx<float> *Ar_old, const float *part_in,
                                                              int nb_in, double omega, Cx<float> *x, int x_init,
                                                              Cx<float> *r_new, Cx<float> *Ar_new, int L0, int L1,
                                                              float *part_out, const double *shift, int nvec) {
  __shared__ float sh[32 * 3 * VB];
  __shared__ float2 s_alpha[VB];
  const Lane8 l;
  const int sites = L0 * L1, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int v0 = blockIdx.y * VB;
  const long long ld = (long long)sites * 8;
  float sums[3 * VB];
#pragma unroll
  for (int k = 0; k < 3 * VB; ++k) sums[k] = 0.f;
  int j = blockIdx.x * 8 + warp;
  bool first = true;
  do {
    const bool live = j < sites;  // uniform over the warp
    const Site8 st(live ? j : 0, L0, L1);
    float4 y[5];
    load_blocks8(Y, st.nb[0], l, y);
    if (STEP && first) {
      // step lengths: warp w sums the partials of vector v0 + w (one vector: the whole block), while
      // the blocks of the first site are on their way
      if (VB == 1) {
        const Cx<float> a = mr_alpha<float>(part_in + 3LL * nb_in * v0, nb_in, omega, sh);
        if (threadIdx.x == 0) s_alpha[0] = make_float2(a.re, a.im);
      } else if (warp < VB && v0 + warp < nvec) {
        const float *part = part_in + 3LL * nb_in * (v0 + warp);
        float t[3] = {0.f, 0.f, 0.f};
        for (int b = lane; b < nb_in; b += 32) {
#pragma unroll
          for (int k = 0; k < 3; ++k) t[k] += __ldcg(part + 3 * b + k);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) t[k] += __shfl_xor_sync(0xffffffffu, t[k], o);
        if (lane == 0)
          s_alpha[warp] = t[2] > 0.f ? make_float2((float)omega * t[0] / t[2], (float)omega * t[1] / t[2])
                                     : make_float2(0.f, 0.f);
      }
      __syncthreads();
    }
    first = false;
    if (live) {
#pragma unroll
      for (int u = 0; u < VB; ++u) {
        const int v = v0 + u;
        if (VB > 1 && v >= nvec) break;
        const long long off = v * ld;
        float2 w[5];
#pragma unroll
        for (int d = 0; d < 5; ++d) w[d] = load_col8(r_old + off, st.nb[d], l.q);
        const float2 rs = load_col8(r_old + off, j, l.row);
        float2 self = rs;
        if (STEP) {
          const float2 al = s_alpha[u];
#pragma unroll
          for (int d = 0; d < 5; ++d) {
            const float2 a = load_col8(Ar_old + off, st.nb[d], l.q);
            w[d].x -= al.x * a.x - al.y * a.y;
            w[d].y -= al.x * a.y + al.y * a.x;
          }
          const float2 a = load_col8(Ar_old + off, j, l.row);
          self.x -= al.x * a.x - al.y * a.y;
          self.y -= al.x * a.y + al.y * a.x;
          if (l.writes) {
            const long long e = (off + (long long)j * 8 + l.row) * 2 + l.im;
            float *xp = reinterpret_cast<float *>(x) + e;
            const float dx = l.im ? al.x * rs.y + al.y * rs.x : al.x * rs.x - al.y * rs.y;
            *xp = x_init ? dx : *xp + dx;
            reinterpret_cast<float *>(r_new)[e] = l.im ? self.y : self.x;
          }
        }
        float k = stencil8(y, w, l);
        const float own = l.im ? self.y : self.x, other = l.im ? -self.x : self.y;
        if (shift != nullptr) k = fmaf((float)shift[v], own, k);
        if (l.writes) {
          reinterpret_cast<float *>(Ar_new)[(off + (long long)j * 8 + l.row) * 2 + l.im] = k;
          sums[3 * u] = fmaf(k, own, sums[3 * u]);
          sums[3 * u + 1] = fmaf(k, other, sums[3 * u + 1]);
          sums[3 * u + 2] = fmaf(k, k, sums[3 * u + 2]);
        }
      }
    }
    j += gridDim.x * 8;
  } while (LOOP && j - warp < sites);
  block_reduce<3 * VB, float>(sums, sh);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int u = 0; u < VB; ++u) {
      if (VB > 1 && v0 + u >= nvec) break;
#pragma unroll
      for (int k = 0; k < 3; ++k) part_out[3LL * (gridDim.x * (long long)(v0 + u) + blockIdx.x) + k] = sums[3 * u + k];
    }
  }
}

// ---- coarse stencil level, any N: one thread per (site, row) ----
template <typename R, bool STEP>
__global__ void __launch_bounds__(256) mr_stencil_kernel(const Cx<R> *__restrict__ Y, const Cx<R> *r_old,
                                                         const Cx<R> *Ar_old, const R *part_in, int nb_in,
                                                         double omega, Cx<R> *x, int x_init, Cx<R> *r_new,
                                                         Cx<R> *Ar_new, int L0, int L1, int N, R *part_out,
                                                         const double *shift) {
  __shared__ R sh[32 * 3];
  {
    const long long off = blockIdx.y * (long long)L0 * L1 * N;
    r_old += off;
    if (STEP) {
      Ar_old += off;
      x += off;
      r_new += off;
      part_in += 3LL * nb_in * blockIdx.y;
    }
    Ar_new += off;
    part_out += 3LL * gridDim.x * blockIdx.y;
  }
  Cx<R> alpha = mk((R)0, (R)0);
  if (STEP) alpha = mr_alpha<R>(part_in, nb_in, omega, sh);  // all threads of the block
  const Cx<R> ma = mk(-alpha.re, -alpha.im);
  R v[3] = {(R)0, (R)0, (R)0};
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < (long long)L0 * L1 * N;
       t += gridDim.x * (long long)blockDim.x) {
    const long long j = t / N;
    const int row = (int)(t - j * N);
    auto src = [&](long long k) { return STEP ? mr_step(r_old[k], Ar_old[k], ma) : r_old[k]; };
    const int x1 = (int)(j / L0), x0 = (int)(j - (long long)x1 * L0);
    const long long rowo = (long long)x1 * L0;
    long long nb[5];
    nb[0] = j;
    nb[1] = rowo + (x0 + 1 == L0 ? 0 : x0 + 1);
    nb[2] = rowo + (x0 == 0 ? L0 - 1 : x0 - 1);
    nb[3] = (x1 + 1 == L1 ? 0 : rowo + L0) + x0;
    nb[4] = (x1 == 0 ? (long long)(L1 - 1) * L0 : rowo - L0) + x0;
    const Cx<R> self = src(t);
    if (STEP) {
      Cx<R> xv = x_init ? mk((R)0, (R)0) : x[t];
      cmac(xv, alpha, r_old[t]);
      x[t] = xv;
      r_new[t] = self;
    }
    Cx<R> acc = mk((R)0, (R)0);
#pragma unroll
    for (int dir = 0; dir < 5; ++dir) {
      const Cx<R> *Yd = Y + (j * 5 + dir) * (long long)N * N + row;
      const long long base = nb[dir] * N;
      for (int col = 0; col < N; ++col) cmac(acc, Yd[(long long)col * N], src(base + col));
    }
    if (shift != nullptr) {
      const R sv = (R)shift[blockIdx.y];
      acc.re = fma(sv, self.re, acc.re);
      acc.im = fma(sv, self.im, acc.im);
    }
    Ar_new[t] = acc;
    v[0] += acc.re * self.re + acc.im * self.im;
    v[1] += acc.re * self.im - acc.im * self.re;
    v[2] += acc.re * acc.re + acc.im * acc.im;
  }
  mr_publish<R>(v, part_out, sh);
}

// x (+)= alpha r for the last MR iteration; with r_out, also the final residual
// r_out = r_old - alpha A r_old (= b - A x; r_out may be r_old)
template <typename R>
__global__ void mr_last_kernel(const Cx<R> *r_old, const Cx<R> *Ar_old, const R *part_in, int nb_in, double omega,
                               Cx<R> *__restrict__ x, int x_init, Cx<R> *r_out, long long n) {
  __shared__ R sh[32 * 3];
  r_old += blockIdx.y * n;
  x += blockIdx.y * n;
  Ar_old += blockIdx.y * n;
  if (r_out != nullptr) r_out += blockIdx.y * n;
  const Cx<R> alpha = mr_alpha<R>(part_in + 3LL * nb_in * blockIdx.y, nb_in, omega, sh);
  const Cx<R> malpha = mk(-alpha.re, -alpha.im);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const Cx<R> ri = r_old[i];
    Cx<R> xv = x_init ? mk((R)0, (R)0) : x[i];
    cmac(xv, alpha, ri);
    x[i] = xv;
    if (r_out != nullptr) r_out[i] = mr_step(ri, Ar_old[i], malpha);
  }
}

// ---------------------------------------------------------------------------
template <typename R>
int mr_grid(const OpDesc<R> &op) {
  const long long units = op.wilson ? op.geo.nsites : op.geo.nsites * (op.N == 8 ? 32 : op.N);
  const int threads = op.wilson ? site_threads(units) : 256;
  return mr_blocks((units + threads - 1) / threads);
}

template <typename R>
void launch_mr_iteration(const OpDesc<R> &op, bool step, const Cx<R> *r_old, const Cx<R> *Ar_old, const R *part_in,
                         double omega, Cx<R> *x, bool x_init, Cx<R> *r_new, Cx<R> *Ar_new, R *part_out,
                         long long part_capacity, cudaStream_t s, int nvec) {
  const int threads = op.wilson ? site_threads(op.geo.nsites) : 256;
  if (nvec > 128) fail(MG_ERR_UNSUPPORTED, "MR batch larger than 128 vectors");
  const int nb = mr_grid(op);
  if (3LL * nb * nvec > part_capacity) fail(MG_ERR_STATE, "MR reduction workspace too small");
  const dim3 grid(nb, nvec);
  const int xi = step && x_init ? 1 : 0;
  const long long units = op.wilson ? op.geo.nsites : op.geo.nsites * (op.N == 8 ? 32 : op.N);
  const bool loop = (long long)nb * threads < units;  // the blocks stride
  auto wilson = [&](auto kernel) {
    kernel<<<grid, threads, 0, s>>>(op.U, r_old, Ar_old, part_in, nb, omega, x, xi, r_new, Ar_new, op.geo.L0,
                                    op.geo.L1, (R)op.diag, part_out, op.shift);
  };
  auto stencil8 = [&](auto kernel) {
    kernel<<<grid, threads, 0, s>>>(op.Y, r_old, Ar_old, part_in, nb, omega, x, xi, r_new, Ar_new, op.geo.L0,
                                    op.geo.L1, part_out, op.shift);
  };
  auto stencil = [&](auto kernel) {
    kernel<<<grid, threads, 0, s>>>(op.Y, r_old, Ar_old, part_in, nb, omega, x, xi, r_new, Ar_new, op.geo.L0,
                                    op.geo.L1, op.N, part_out, op.shift);
  };
  if (op.wilson) {
    if (loop)
      step ? wilson(mr_wilson_kernel<R, true, true>) : wilson(mr_wilson_kernel<R, false, true>);
    else
      step ? wilson(mr_wilson_kernel<R, true, false>) : wilson(mr_wilson_kernel<R, false, false>);
  } else if (op.N == 8) {
    if constexpr (sizeof(R) == 4) {
      // four vectors per block where that still leaves two blocks per SM
      const int vb = nvec > 1 && (long long)nb * ((nvec + 3) / 4) >= 304 ? 4 : 1;
      auto run = [&](auto kernel) {
        kernel<<<dim3(nb, (nvec + vb - 1) / vb), threads, 0, s>>>(op.Y, r_old, Ar_old, part_in, nb, omega, x, xi,
                                                                  r_new, Ar_new, op.geo.L0, op.geo.L1, part_out,
                                                                  op.shift, nvec);
      };
      if (vb == 4)
        loop ? (step ? run(mr_stencil8_f32_kernel<true, true, 4>) : run(mr_stencil8_f32_kernel<false, true, 4>))
             : (step ? run(mr_stencil8_f32_kernel<true, false, 4>) : run(mr_stencil8_f32_kernel<false, false, 4>));
      else
        loop ? (step ? run(mr_stencil8_f32_kernel<true, true, 1>) : run(mr_stencil8_f32_kernel<false, true, 1>))
             : (step ? run(mr_stencil8_f32_kernel<true, false, 1>) : run(mr_stencil8_f32_kernel<false, false, 1>));
    } else {
      if (loop)
        step ? stencil8(mr_stencil8_kernel<true, true>) : stencil8(mr_stencil8_kernel<false, true>);
      else
        step ? stencil8(mr_stencil8_kernel<true, false>) : stencil8(mr_stencil8_kernel<false, false>);
    }
  } else {
    step ? stencil(mr_stencil_kernel<R, true>) : stencil(mr_stencil_kernel<R, false>);
  }
  MG_LAUNCHED();
}

template <typename R>
void launch_mr_last(const OpDesc<R> &op, const Cx<R> *r_old, const Cx<R> *Ar_old, const R *part_in, double omega,
                    Cx<R> *x, bool x_init, Cx<R> *r_out, long long n, cudaStream_t s, int nvec) {
  mr_last_kernel<R><<<dim3((unsigned int)mr_blocks((n + 255) / 256), nvec), 256, 0, s>>>(
      r_old, Ar_old, part_in, mr_grid(op), omega, x, x_init ? 1 : 0, r_out, n);
  MG_LAUNCHED();
}

#define MG_INST_MR(R)                                                                                              \
  template int mr_grid<R>(const OpDesc<R> &);                                                                     \
  template void launch_mr_iteration<R>(const OpDesc<R> &, bool, const Cx<R> *, const Cx<R> *, const R *, double,  \
                                       Cx<R> *, bool, Cx<R> *, Cx<R> *, R *, long long, cudaStream_t, int);        \
  template void launch_mr_last<R>(const OpDesc<R> &, const Cx<R> *, const Cx<R> *, const R *, double, Cx<R> *,     \
                                  bool, Cx<R> *, long long, cudaStream_t, int);
MG_INST_MR(double)
MG_INST_MR(float)
#undef MG_INST_MR

}  // namespace mg
